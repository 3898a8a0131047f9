// Per-layer immediate eviction (IKV_EVICT_LAYER): every layer folds its Eq. 1 score
// into a state indexed by token position and shared by all layers, then keeps the
// budget's highest-utility tokens among those it holds (Appendix "Layer scoring",
// each layer's hook acting at once).  A live position that a layer does not hold gets
// score 0 there, so Eq. 4 multiplies it by alpha.
//
// No layer's eviction changes another layer's inputs within a step: a layer attends
// its own rows, and its update reads only the tokens it held before the step's
// evictions.  So after all attention (and the stored per-layer scores), one pass over
// token positions walks the layers in order -- the state as each layer saw it is that
// layer's utility for its slot of the position -- and every layer is then selected
// and compacted at once by the step's usual kernels (rows = batch x layers).
#include "ikv_internal.cuh"

namespace ikv {

__device__ unsigned int g_layer_error = 0;  // bit 2: no free slot; bit 3: next_pos reached pos_cap

namespace {

constexpr int kBeginThreads = 1024;

// The live positions (held by some layer) as bits, set by one thread per (sequence,
// layer, slot) into the cleared bitmap.  Nothing is evicted between here and the fold,
// so with the new token's bit (set by the begin kernel) this is the fold's live set.
constexpr int kMarkThreads = 256;
__global__ void __launch_bounds__(kMarkThreads) layer_mark_kernel(const LayerArgs a) {
    pdl_wait();
    const int b = blockIdx.z, l = blockIdx.y;
    const int j = blockIdx.x * kMarkThreads + threadIdx.x;
    if (j >= a.len[b]) return;
    const int p = a.pos[((int64_t)b * a.layers + l) * a.cap + j];
    if (p >= 0 && p < a.pos_cap) atomicOr(a.live + (int64_t)b * a.live_words + (p >> 5), 1u << (p & 31));
}

// One CTA per sequence: the new token's state (0, or the mean over the live positions),
// its live bit and position in every layer's row, then len and next_pos advanced.
__global__ void __launch_bounds__(kBeginThreads) layer_begin_kernel(const LayerArgs a) {
    pdl_wait();
    __shared__ float red[2][kBeginThreads / 32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int b = blockIdx.x;
    const int L = a.len[b];
    const int S = a.start ? a.start[b] : 0;
    const int np = a.next_pos[b];
    float *m = a.m + (int64_t)b * a.pos_cap;
    uint32_t *bits = a.live + (int64_t)b * a.live_words;
    if (S + L >= a.cap || np >= a.pos_cap) {
        if (tid == 0) {
            a.slot[b] = -1;
            atomicOr(&g_layer_error, S + L >= a.cap ? 4u : 8u);
        }
        return;
    }
    float init = 0.f;
    if (a.init_mean) {
        float sum = 0.f, cnt = 0.f;
        for (int p = tid; p < np; p += kBeginThreads)
            if ((bits[p >> 5] >> (p & 31)) & 1u) {
                sum += m[p];
                cnt += 1.f;
            }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            sum += __shfl_xor_sync(0xffffffffu, sum, o);
            cnt += __shfl_xor_sync(0xffffffffu, cnt, o);
        }
        if (lane == 0) red[0][warp] = sum, red[1][warp] = cnt;
        __syncthreads();
        float ts = 0.f, tc = 0.f;
        for (int w = 0; w < kBeginThreads / 32; ++w) ts += red[0][w], tc += red[1][w];
        init = tc > 0.f ? ts / tc : 0.f;
    }
    __syncthreads();  // every thread has read len / next_pos and the bits
    for (int l = tid; l < a.layers; l += kBeginThreads) a.pos[((int64_t)b * a.layers + l) * a.cap + L] = np;
    if (tid == 0) {
        bits[np >> 5] |= 1u << (np & 31);  // the new token is live too
        m[np] = init;
        a.slot[b] = L;
        a.next_pos[b] = np + 1;
        a.len[b] = L + 1;
    }
}

// inv[b][l][pos[b][l][j]] = j for every slot j < len[b] of every layer
constexpr int kInvThreads = 256;
__global__ void __launch_bounds__(kInvThreads) layer_inverse_kernel(const LayerArgs a) {
    pdl_wait();
    const int b = blockIdx.z, l = blockIdx.y;
    const int j = blockIdx.x * kInvThreads + threadIdx.x;
    if (j >= a.len[b]) return;
    const int p = a.pos[((int64_t)b * a.layers + l) * a.cap + j];
    if (p >= 0 && p < a.pos_cap) a.inv[((int64_t)b * a.layers + l) * a.pos_cap + p] = j;
}

// LG lanes per live token position p (held by some layer), each for up to NB consecutive
// layers: at every eligible layer of a refresh step m <- alpha m + (1 - alpha) s, s the
// layer's pooled score of p if it holds p, else 0; each layer holding p gets m as its
// utility of p's slot.  The final m is stored.  Dead positions are left as they are.
// A lane folds its layers from zero; the lanes of a position compose those affine maps in
// layer order (shuffles), which gives each the m that enters its layers.  Bound by the
// instructions of a lane's chain: one lane walking 32 layers took 12 us at 32 layers x 3.3k
// slots, its loads batched however (a step 116.8 us, 110.8 this way).
constexpr int kFoldThreads = 256;
template <int LG, int NB>
__global__ void __launch_bounds__(kFoldThreads) layer_fold_kernel(const LayerArgs a) {
    pdl_wait();
    constexpr int PP = 32 / LG;  // positions per warp
    const int lane = threadIdx.x & 31;
    const int grp = lane / PP, sub = lane % PP;
    const int b = blockIdx.y;
    const int p = (blockIdx.x * (kFoldThreads / 32) + (threadIdx.x >> 5)) * PP + sub;
    const bool on = p < a.next_pos[b] && p < a.pos_cap &&
                    ((__ldg(a.live + (int64_t)b * a.live_words + (p >> 5)) >> (p & 31)) & 1u);
    if (!__any_sync(0xffffffffu, on)) return;
    const int L = a.len[b];
    float *mp = a.m + (int64_t)b * a.pos_cap + p;
    float m = on ? *mp : 0.f;
    const int per = (a.layers + LG - 1) / LG;
    const int l0 = grp * per, l1 = min(l0 + per, a.layers);
    const int64_t row0 = (int64_t)b * a.layers + l0;
    // the lane's slot lookups, then their checks and scores, all issued before use
    int j[NB];
    const int32_t *ip = a.inv + row0 * a.pos_cap + p;
#pragma unroll
    for (int u = 0; u < NB; ++u, ip += a.pos_cap) j[u] = on && l0 + u < l1 ? __ldg(ip) : -1;
    uint32_t held = 0u, elig = 0u;
    const int32_t *pp = a.pos + row0 * a.cap;
#pragma unroll
    for (int u = 0; u < NB; ++u, pp += a.cap)
        if (j[u] >= 0 && j[u] < L && __ldg(pp + j[u]) == p) held |= 1u << u;
    float sc[NB];
    if (a.scoring) {
        int k = 0;  // eligible layers before the lane's
        for (int l = 0; l < l0; l += 32)
            k += __popc(a.elig_bits[l >> 5] & (l0 - l >= 32 ? ~0u : (1u << (l0 - l)) - 1u));
        const float *sp = a.sbuf + ((int64_t)b * a.n_elig + k) * a.lstride;
#pragma unroll
        for (int u = 0; u < NB; ++u) {
            const int l = l0 + u;
            sc[u] = 0.f;
            if (l < l1 && ((a.elig_bits[l >> 5] >> (l & 31)) & 1u)) {
                elig |= 1u << u;
                if ((held >> u) & 1u) sc[u] = __ldg(sp + j[u]);
                sp += a.lstride;
            }
        }
    }
    const float beta = 1.f - a.alpha;
    float f = 1.f, c = 0.f;  // the lane's layers: m -> f m + c
#pragma unroll
    for (int u = 0; u < NB; ++u)
        if ((elig >> u) & 1u) {
            c = a.alpha * c + beta * sc[u];
            f *= a.alpha;
        }
#pragma unroll
    for (int g = 0; g < LG - 1; ++g) {
        const float fg = __shfl_sync(0xffffffffu, f, g * PP + sub), cg = __shfl_sync(0xffffffffu, c, g * PP + sub);
        if (g < grp) m = fg * m + cg;
    }
    float *up = a.util + row0 * a.cap;
#pragma unroll
    for (int u = 0; u < NB; ++u, up += a.cap) {
        if ((elig >> u) & 1u) m = a.alpha * m + beta * sc[u];
        if ((held >> u) & 1u) up[j[u]] = m;
    }
    if (on && grp == LG - 1) *mp = m;
}

template <int LG, int NB>
cudaError_t launch_fold(const LayerArgs &a, int32_t max_pos, cudaStream_t st) {
    constexpr int kPos = kFoldThreads / LG;  // positions of a CTA
    return launch_k(layer_fold_kernel<LG, NB>, dim3((max_pos + kPos - 1) / kPos, a.batch), dim3(kFoldThreads), 0, st, a);
}

}  // namespace

cudaError_t launch_layer_begin(const LayerArgs &a, int32_t max_len, cudaStream_t st) {
    if (max_len > 0) {
        cudaError_t e = launch_k(layer_mark_kernel, dim3((max_len + kMarkThreads - 1) / kMarkThreads, a.layers, a.batch),
                                 dim3(kMarkThreads), 0, st, a);
        note_launch();
        if (e != cudaSuccess) return e;
    }
    cudaError_t e = launch_k(layer_begin_kernel, dim3(a.batch), dim3(kBeginThreads), 0, st, a);
    note_launch();
    return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t launch_layer_fold(const LayerArgs &a, int32_t max_len, int32_t max_pos, cudaStream_t st) {
    if (max_len <= 0 || max_pos <= 0) return cudaSuccess;
    cudaError_t e = launch_k(layer_inverse_kernel, dim3((max_len + kInvThreads - 1) / kInvThreads, a.layers, a.batch),
                             dim3(kInvThreads), 0, st, a);
    note_launch();
    if (e != cudaSuccess) return e;
    // lanes per position for at most eight layers each (16 beyond 256 layers)
    e = a.layers <= 32 ? launch_fold<4, 8>(a, max_pos, st)
        : a.layers <= 64 ? launch_fold<8, 8>(a, max_pos, st)
        : a.layers <= 128 ? launch_fold<16, 8>(a, max_pos, st)
                          : launch_fold<32, 16>(a, max_pos, st);
    note_launch();
    return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t read_clear_layer_error(unsigned int *v) {
    unsigned int z = 0;
    cudaError_t e = cudaMemcpyFromSymbol(v, g_layer_error, sizeof(*v));
    if (e == cudaSuccess) e = cudaMemcpyToSymbol(g_layer_error, &z, sizeof(z));
    return e;
}

}  // namespace ikv
