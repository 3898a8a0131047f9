// Split-K grouped-query decode attention that also emits per-token logits.
//
// One CTA handles (split s, kv head g, sequence b, layer l): the G query heads
// of KV head g against cache slots [s*split, min((s+1)*split, len[b])).
// K/V rows stream through shared memory in 64-token tiles (cp.async, 16-byte
// chunks, XOR-swizzled by row so both the token-major QK reads and the
// dim-major PV reads are bank-conflict free).  QK: each warp owns a quarter of
// the head dimension and two tokens per lane; partial dot products meet in
// shared memory.  Softmax is online per head in the log2 domain (the query is
// pre-scaled by log2(e)/sqrt(d)); each tile's logits are written out for the
// Eq. 1 score pass.  PV: each thread owns one 16-byte column chunk of V for all
// G heads over a strided subset of the tile's tokens.  The split's running
// (max, sum) and unnormalised output go to the workspace; combine_kernel merges
// splits, writes the output and the per-head log-sum-exp.
#include "ikv_internal.cuh"

namespace ikv {
namespace {

__device__ __forceinline__ void cp_async16(void *smem, const void *gmem) {
    const uint32_t s = static_cast<uint32_t>(__cvta_generic_to_shared(smem));
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(s), "l"(gmem) : "memory");
}
// the same, or 16 zero bytes (nothing read) when !in
__device__ __forceinline__ void cp_async16_zfill(void *smem, const void *gmem, bool in) {
    const uint32_t s = static_cast<uint32_t>(__cvta_generic_to_shared(smem));
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(s), "l"(gmem), "r"(in ? 16 : 0) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory"); }

template <typename T>
struct Chunk;
template <>
struct Chunk<__nv_bfloat16> {
    static constexpr int kElems = 8;
    __device__ __forceinline__ static void load(const uint4 &c, float *x) {
        const uint32_t w[4] = {c.x, c.y, c.z, c.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            x[2 * i] = __uint_as_float(w[i] << 16);
            x[2 * i + 1] = __uint_as_float(w[i] & 0xFFFF0000u);
        }
    }
    __device__ __forceinline__ static void store(void *p, int64_t idx, float v) {
        reinterpret_cast<__nv_bfloat16 *>(p)[idx] = __float2bfloat16_rn(v);
    }
    __device__ __forceinline__ static float read(const void *p, int64_t idx) {
        return __bfloat162float(reinterpret_cast<const __nv_bfloat16 *>(p)[idx]);
    }
};
template <>
struct Chunk<float> {
    static constexpr int kElems = 4;
    __device__ __forceinline__ static void load(const uint4 &c, float *x) {
        x[0] = __uint_as_float(c.x);
        x[1] = __uint_as_float(c.y);
        x[2] = __uint_as_float(c.z);
        x[3] = __uint_as_float(c.w);
    }
    __device__ __forceinline__ static void store(void *p, int64_t idx, float v) {
        reinterpret_cast<float *>(p)[idx] = v;
    }
    __device__ __forceinline__ static float read(const void *p, int64_t idx) {
        return reinterpret_cast<const float *>(p)[idx];
    }
};

__device__ __forceinline__ float warp_max(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}
__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

template <typename T, int D, int G>
struct AttendCfg {
    static constexpr int TT = kTileTokens;
    static constexpr int kRowBytes = D * (int)sizeof(T);
    static constexpr int CPR = kRowBytes / 16;             // 16-byte chunks per row
    static constexpr int EPC = Chunk<T>::kElems;          // elements per chunk
    static constexpr int QCH = CPR / 4;                   // chunks per warp in QK
    static constexpr int NTG = kAttendThreads / CPR;      // token groups in PV
    static constexpr int kTileBytes = TT * kRowBytes;
    static constexpr int kStageBytes = 2 * kTileBytes;    // K + V
    static constexpr int NSTAGE = kStageBytes <= 32768 ? 3 : 2;
    static constexpr int GP = (G + 3) / 4 * 4;
    static constexpr int kStageArea = NSTAGE * kStageBytes;
    static constexpr int kObufBytes = NTG * G * D * 4;
    static_assert(kObufBytes <= kStageArea, "output reduction must fit in the stage area");
    static_assert(CPR >= 8 && CPR % 4 == 0, "row must be >= 8 chunks");
    // float regions after the stage area
    static constexpr int kQ = 0;                          // G*D
    static constexpr int kRed = kQ + G * D;               // 4*G*TT
    static constexpr int kZ = kRed + 4 * G * TT;          // G*TT
    static constexpr int kP = kZ + G * TT;                // TT*GP
    static constexpr int kM = kP + TT * GP;               // G
    static constexpr int kL = kM + GP;                    // G
    static constexpr int kC = kL + GP;                    // G
    static constexpr int kFloats = kC + GP;
    static constexpr int kSmemBytes = kStageArea + kFloats * 4;
};

template <typename T, int D, int G, bool LOGITS>
__global__ void __launch_bounds__(kAttendThreads, 2) attend_split_kernel(const AttendArgs a) {
    using C = AttendCfg<T, D, G>;
    pdl_wait();
    extern __shared__ __align__(128) unsigned char smem[];
    float *fs = reinterpret_cast<float *>(smem + C::kStageArea);
    float *q_s = fs + C::kQ;
    float *red = fs + C::kRed;
    float *zt = fs + C::kZ;
    float *p_s = fs + C::kP;
    float *m_run = fs + C::kM;
    float *l_run = fs + C::kL;
    float *corr_s = fs + C::kC;

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int s = blockIdx.x, g = blockIdx.y;
    const int b = blockIdx.z % a.batch, li = blockIdx.z / a.batch;
    const int l = a.layer0 + li;
    const int L = a.len[b];
    const int S0 = a.pv.start_of(b);
    const int32_t *prow = a.pos ? a.pos + ((int64_t)b * a.rows_per_seq + (a.rows_per_seq == 1 ? 0 : g)) * a.cap : nullptr;
    const int t0 = s * a.split_tokens;
    if (t0 >= L) return;
    const int t1 = min(t0 + a.split_tokens, L);
    const int H = a.q_heads;
    const int n_tiles = (t1 - t0 + C::TT - 1) / C::TT;

    const unsigned char *kbase = reinterpret_cast<const unsigned char *>(a.k);
    const unsigned char *vbase = reinterpret_cast<const unsigned char *>(a.v);

    auto issue_tile = [&](int tile) {
        unsigned char *st = smem + (tile % C::NSTAGE) * C::kStageBytes;
        const int base = t0 + tile * C::TT;
#pragma unroll
        for (int it = 0; it < C::TT * C::CPR / kAttendThreads; ++it) {
            const int idx = it * kAttendThreads + tid;
            const int j = idx / C::CPR, c = idx % C::CPR;
            const int tok = base + j;
            if (tok < t1) {
                const int64_t row = a.pv.row_phys(b, l, g, S0 + tok);
                const int off = j * C::kRowBytes + ((c ^ (j & 7)) << 4);
                cp_async16(st + off, kbase + row * C::kRowBytes + c * 16);
                cp_async16(st + C::kTileBytes + off, vbase + row * C::kRowBytes + c * 16);
            }
        }
    };

    // prologue: start the first tiles before touching anything else
#pragma unroll
    for (int i = 0; i < C::NSTAGE - 1; ++i) {
        if (i < n_tiles) issue_tile(i);
        cp_async_commit();
    }

    // query of the G heads, pre-scaled into the log2 domain
    const int64_t qoff = (((int64_t)li * a.batch + b) * H + (int64_t)g * G) * D;
    for (int i = tid; i < G * D; i += kAttendThreads) q_s[i] = Chunk<T>::read(a.q, qoff + i) * a.scale_log2;
    if (tid < G) {
        m_run[tid] = -INFINITY;
        l_run[tid] = 0.f;
    }

    float o[G][C::EPC];
#pragma unroll
    for (int h = 0; h < G; ++h)
#pragma unroll
        for (int e = 0; e < C::EPC; ++e) o[h][e] = 0.f;

    const int pc = tid % C::CPR;   // PV column chunk
    const int tg = tid / C::CPR;   // PV token group

    for (int tile = 0; tile < n_tiles; ++tile) {
        __syncthreads();  // previous tile's PV done with its stage and with p_s
        if (tile + C::NSTAGE - 1 < n_tiles) issue_tile(tile + C::NSTAGE - 1);
        cp_async_commit();
        cp_async_wait<C::NSTAGE - 1>();
        __syncthreads();

        const unsigned char *Ks = smem + (tile % C::NSTAGE) * C::kStageBytes;
        const unsigned char *Vs = Ks + C::kTileBytes;
        const int tbase = t0 + tile * C::TT;
        const int nv = min(C::TT, t1 - tbase);

        // ---- QK: warp owns chunks [warp*QCH, (warp+1)*QCH), lane owns tokens lane, lane+32
        {
            float acc0[G], acc1[G];
#pragma unroll
            for (int h = 0; h < G; ++h) acc0[h] = acc1[h] = 0.f;
            const int j0 = lane, j1 = lane + 32;
#pragma unroll
            for (int qc = 0; qc < C::QCH; ++qc) {
                const int c = warp * C::QCH + qc;
                float x0[C::EPC], x1[C::EPC];
                Chunk<T>::load(*reinterpret_cast<const uint4 *>(Ks + j0 * C::kRowBytes + ((c ^ (j0 & 7)) << 4)), x0);
                Chunk<T>::load(*reinterpret_cast<const uint4 *>(Ks + j1 * C::kRowBytes + ((c ^ (j1 & 7)) << 4)), x1);
#pragma unroll
                for (int h = 0; h < G; ++h) {
                    const float4 *qp = reinterpret_cast<const float4 *>(q_s + h * D + c * C::EPC);
#pragma unroll
                    for (int e4 = 0; e4 < C::EPC / 4; ++e4) {
                        const float4 qv = qp[e4];
                        acc0[h] = fmaf(qv.x, x0[4 * e4 + 0], acc0[h]);
                        acc0[h] = fmaf(qv.y, x0[4 * e4 + 1], acc0[h]);
                        acc0[h] = fmaf(qv.z, x0[4 * e4 + 2], acc0[h]);
                        acc0[h] = fmaf(qv.w, x0[4 * e4 + 3], acc0[h]);
                        acc1[h] = fmaf(qv.x, x1[4 * e4 + 0], acc1[h]);
                        acc1[h] = fmaf(qv.y, x1[4 * e4 + 1], acc1[h]);
                        acc1[h] = fmaf(qv.z, x1[4 * e4 + 2], acc1[h]);
                        acc1[h] = fmaf(qv.w, x1[4 * e4 + 3], acc1[h]);
                    }
                }
            }
#pragma unroll
            for (int h = 0; h < G; ++h) {
                red[(warp * G + h) * C::TT + j0] = acc0[h];
                red[(warp * G + h) * C::TT + j1] = acc1[h];
            }
        }
        __syncthreads();

        // ---- logits of this tile (log2 domain), masked tail and dead slots (-inf)
        for (int idx = tid; idx < G * C::TT; idx += kAttendThreads) {
            const int h = idx / C::TT, j = idx % C::TT;
            float z = red[(0 * G + h) * C::TT + j] + red[(1 * G + h) * C::TT + j] + red[(2 * G + h) * C::TT + j] +
                      red[(3 * G + h) * C::TT + j];
            if (j < nv) {
                if (prow && prow[tbase + j] < 0) z = -INFINITY;
                if (LOGITS)
                    a.logits[((((int64_t)b * a.sc_layers + a.sc_layer0 + li) * H) + g * G + h) * (int64_t)a.lstride +
                             tbase + j] = z;
            } else {
                z = -INFINITY;
            }
            zt[h * C::TT + j] = z;
        }
        __syncthreads();

        // ---- online softmax per head
        for (int h = warp; h < G; h += kAttendThreads / 32) {
            const float za = zt[h * C::TT + lane], zb = zt[h * C::TT + lane + 32];
            const float mx = warp_max(fmaxf(za, zb));
            const float m_old = m_run[h];
            const float m_new = fmaxf(m_old, mx);
            const float m_ref = m_new == -INFINITY ? 0.f : m_new;  // every slot so far dead: nothing to scale
            const float corr = exp2f(m_old - m_ref);
            const float pa = exp2f(za - m_ref), pb = exp2f(zb - m_ref);
            const float sum = warp_sum(pa + pb);
            p_s[lane * C::GP + h] = pa;
            p_s[(lane + 32) * C::GP + h] = pb;
            __syncwarp();
            if (lane == 0) {
                l_run[h] = l_run[h] * corr + sum;
                m_run[h] = m_new;
                corr_s[h] = corr;
            }
        }
        __syncthreads();

        // ---- PV
        {
#pragma unroll
            for (int h = 0; h < G; ++h) {
                const float cr = corr_s[h];
#pragma unroll
                for (int e = 0; e < C::EPC; ++e) o[h][e] *= cr;
            }
            for (int j = tg; j < nv; j += C::NTG) {
                float xv[C::EPC];
                Chunk<T>::load(*reinterpret_cast<const uint4 *>(Vs + j * C::kRowBytes + ((pc ^ (j & 7)) << 4)), xv);
                float p[C::GP];
#pragma unroll
                for (int h4 = 0; h4 < C::GP / 4; ++h4) {
                    const float4 pv = reinterpret_cast<const float4 *>(p_s + j * C::GP)[h4];
                    p[4 * h4] = pv.x;
                    p[4 * h4 + 1] = pv.y;
                    p[4 * h4 + 2] = pv.z;
                    p[4 * h4 + 3] = pv.w;
                }
#pragma unroll
                for (int h = 0; h < G; ++h)
#pragma unroll
                    for (int e = 0; e < C::EPC; ++e) o[h][e] = fmaf(p[h], xv[e], o[h][e]);
            }
        }
    }

    // ---- reduce the PV token groups, write the split partial
    cp_async_wait<0>();
    __syncthreads();
    float *obuf = reinterpret_cast<float *>(smem);
#pragma unroll
    for (int h = 0; h < G; ++h)
#pragma unroll
        for (int e = 0; e < C::EPC; ++e) obuf[(tg * G + h) * D + pc * C::EPC + e] = o[h][e];
    __syncthreads();
    const int64_t pbase = (((int64_t)b * a.n_layers + li) * H + (int64_t)g * G) * a.n_splits;
    for (int idx = tid; idx < G * D; idx += kAttendThreads) {
        const int h = idx / D, e = idx % D;
        float acc = 0.f;
#pragma unroll
        for (int t = 0; t < C::NTG; ++t) acc += obuf[(t * G + h) * D + e];
        a.part_o[((pbase + (int64_t)h * a.n_splits) + s) * D + e] = acc;
    }
    if (tid < G) {
        a.part_ml[((pbase + (int64_t)tid * a.n_splits) + s) * 2 + 0] = m_run[tid];
        a.part_ml[((pbase + (int64_t)tid * a.n_splits) + s) * 2 + 1] = l_run[tid];
    }
}

// What the CTAs of a (sequence, layer, kv head) unit do once a CTA has its split's result:
// P partial softmaxes over disjoint tokens, obuf [P][G][D] unnormalised outputs and mlbuf
// [P][GP][2] (max, sum) in shared memory, merged into the split's (max, sum, output).  A
// unit of one split is final and goes straight to out and lse2; otherwise the split goes to
// the workspace and the unit's last CTA to arrive (counter only, no waiting) merges them.
// Entered by every thread of the CTA; obuf is reused.
template <typename T, int D, int GP, int P>
__device__ __forceinline__ void finish_split(const AttendArgs &a, float *obuf, float *mlbuf, int G, int s,
                                             int ns_active, int b, int li, int g) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int H = a.q_heads;
    const int64_t hrow = ((int64_t)li * a.batch + b) * H + (int64_t)g * G;           // out rows
    const int64_t lrow = ((int64_t)b * a.sc_layers + a.sc_layer0 + li) * H + (int64_t)g * G;  // lse2
    const int64_t pbase = (((int64_t)b * a.n_layers + li) * H + (int64_t)g * G) * a.n_splits;
    for (int idx = tid; idx < G * D; idx += kAttendThreads) {
        const int h = idx / D, e = idx % D;
        float M = -INFINITY;
#pragma unroll
        for (int w = 0; w < P; ++w) M = fmaxf(M, mlbuf[(w * GP + h) * 2]);
        const float ref = M == -INFINITY ? 0.f : M;
        float acc = 0.f, sum = 0.f;
#pragma unroll
        for (int w = 0; w < P; ++w) {
            const float f = exp2f(mlbuf[(w * GP + h) * 2] - ref);
            sum += mlbuf[(w * GP + h) * 2 + 1] * f;
            acc += obuf[(w * G + h) * D + e] * f;
        }
        if (ns_active == 1) {
            Chunk<T>::store(a.out, (hrow + h) * D + e, sum > 0.f ? acc / sum : 0.f);
            if (e == 0) a.lse2[lrow + h] = sum > 0.f ? M + log2f(sum) : -INFINITY;
        } else {
            const int64_t at = pbase + (int64_t)h * a.n_splits + s;
            a.part_o[at * D + e] = acc;
            if (e == 0) {
                a.part_ml[at * 2] = M;
                a.part_ml[at * 2 + 1] = sum;
            }
        }
    }
    if (ns_active == 1) return;
    __shared__ int last;
    const int64_t unit = ((int64_t)b * a.n_layers + li) * a.pv.kv_heads + g;
    __syncthreads();
    if (tid == 0) last = arrive_acq_rel(a.arrivals + unit) == ns_active - 1;
    __syncthreads();
    if (!last) return;
    if (tid == 0) a.arrivals[unit] = 0;
    // warp w merges heads w, w + 4, ...: the (max, sum) pairs give each split's weight, then
    // every lane sums D / 32 output dims over the splits, eight loads in flight
    constexpr int E = D / 32;
    float *wq = obuf + warp * kMaxSplits;
    for (int h = warp; h < G; h += kAttendThreads / 32) {
        const float2 *ml = reinterpret_cast<const float2 *>(a.part_ml) + pbase + (int64_t)h * a.n_splits;
        const float *po = a.part_o + (pbase + (int64_t)h * a.n_splits) * D + lane * E;
        float mv[kMaxSplits / 32], lv[kMaxSplits / 32], M = -INFINITY;
#pragma unroll
        for (int k = 0; k < kMaxSplits / 32; ++k) {
            const int q = lane + 32 * k;
            const float2 x = q < ns_active ? __ldcg(ml + q) : make_float2(-INFINITY, 0.f);
            mv[k] = x.x;
            lv[k] = x.y;
            M = fmaxf(M, x.x);
        }
        M = warp_max(M);
        const float ref = M == -INFINITY ? 0.f : M;
        float W = 0.f;
#pragma unroll
        for (int k = 0; k < kMaxSplits / 32; ++k) {
            const float f = exp2f(mv[k] - ref);
            W += lv[k] * f;
            wq[lane + 32 * k] = f;
        }
        W = warp_sum(W);
        __syncwarp();
        float acc[E];
#pragma unroll
        for (int e = 0; e < E; ++e) acc[e] = 0.f;
        for (int q0 = 0; q0 < ns_active; q0 += 8) {
            float ov[8][E];
#pragma unroll
            for (int j = 0; j < 8; ++j)
#pragma unroll
                for (int e = 0; e < E; ++e) ov[j][e] = q0 + j < ns_active ? __ldcg(po + (int64_t)(q0 + j) * D + e) : 0.f;
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const float f = q0 + j < ns_active ? wq[q0 + j] : 0.f;
#pragma unroll
                for (int e = 0; e < E; ++e) acc[e] += f * ov[j][e];
            }
        }
#pragma unroll
        for (int e = 0; e < E; ++e)
            Chunk<T>::store(a.out, (hrow + h) * D + lane * E + e, W > 0.f ? acc[e] / W : 0.f);
        if (lane == 0) a.lse2[lrow + h] = W > 0.f ? M + log2f(W) : -INFINITY;
        __syncwarp();
    }
}

// A sequence without slots: output 0, log-sum-exp -inf (written by its first split's CTA).
template <typename T>
__device__ __forceinline__ void store_empty(const AttendArgs &a, int G, int D, int b, int li, int g) {
    const int64_t hrow = ((int64_t)li * a.batch + b) * a.q_heads + (int64_t)g * G;
    for (int i = threadIdx.x; i < G * D; i += kAttendThreads) Chunk<T>::store(a.out, hrow * D + i, 0.f);
    if ((int)threadIdx.x < G)
        a.lse2[((int64_t)b * a.sc_layers + a.sc_layer0 + li) * a.q_heads + (int64_t)g * G + threadIdx.x] = -INFINITY;
}

// fp32 K/V.  HBM bound: a K and V byte costs G / 4 FMAs, half an SM's rate at G = 8.  Every
// warp is on its own: it takes every fourth group of 8 (d = 128) or 16 (d = 64) tokens of
// the split through its own cp.async ring and keeps its own online softmax, so the loop has
// no block barrier, and each lane reads back the 16 bytes of each row that it copied itself.
// A lane's partial dot products of 8 tokens x G heads are summed over the row's lanes by a
// halving exchange (one shuffle a value instead of five), which leaves each lane with the
// logits it exponentiates; the probabilities go through a few hundred bytes of shared memory
// to the P.V products.  8 warps an SM (two CTAs) keep 128 KB in flight.  Measured, a whole
// step of b = 4, 8 layers, 16 / 4 heads of 128, 2048 tokens (269 MB, 39.7 us at the copy
// rate): 185.1 -> 76.9 us against attend_split_kernel, which ran one CTA of four warps an
// SM with five block barriers per 64-token tile; tiny steps save the combine launch.
template <int D, int G>
struct F32Cfg {
    static constexpr int GP = G == 7 ? 8 : G;
    static constexpr int RL = D / 4;              // lanes of a row (16 bytes each)
    static constexpr int RPI = 32 / RL;           // rows a warp reads at once
    static constexpr int T = 8;                   // tokens per group and row slot
    static constexpr int TW = T * RPI;            // tokens per warp and group
    static constexpr int kRowB = D * 4;
    static constexpr int kStageB = 2 * TW * kRowB;
    static constexpr int NST = 3;
    static constexpr int kWarps = kAttendThreads / 32;
    static constexpr int kRing = kWarps * NST * kStageB;
    static constexpr int P = kWarps * RPI;        // independent softmaxes of a CTA
    static constexpr int N = T * GP;              // logits of a group per row slot
    static constexpr int VPL = N > RL ? N / RL : 1;   // logits a lane ends up with
    static constexpr int DUP = N < RL ? RL / N : 1;   // lanes holding the same logit
    static constexpr int kPw = RPI * (T + 1) * GP;    // floats per warp: probabilities, rescales
    static constexpr int kSmemBytes = kRing + (kWarps * kPw + 2 * P * GP) * 4;
    static_assert(P * G * D * 4 <= kRing && kWarps * kMaxSplits * 4 <= kRing, "the merge reuses the ring");
};

template <int D, int G>
__global__ void __launch_bounds__(kAttendThreads, 2) attend_f32_kernel(const AttendArgs a) {
    using C = F32Cfg<D, G>;
    constexpr int GP = C::GP, T = C::T, TW = C::TW, NST = C::NST, VPL = C::VPL, DUP = C::DUP;
    pdl_wait();
    extern __shared__ __align__(128) unsigned char smem[];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int s = blockIdx.x, g = blockIdx.y;
    const int b = blockIdx.z % a.batch, li = blockIdx.z / a.batch;
    const int l = a.layer0 + li;
    const int L = a.len[b];
    const int S0 = a.pv.start_of(b);
    const int t0 = s * a.split_tokens;
    if (t0 >= L) {
        if (s == 0) store_empty<float>(a, G, D, b, li, g);
        return;
    }
    const int t1 = min(t0 + a.split_tokens, L);
    const int ns_active = min((L + a.split_tokens - 1) / a.split_tokens, a.n_splits);
    const int32_t *prow = a.pos ? a.pos + ((int64_t)b * a.rows_per_seq + (a.rows_per_seq == 1 ? 0 : g)) * a.cap : nullptr;
    const int groups = (t1 - t0 + TW - 1) / TW;
    const int mine = groups > warp ? (groups - warp + C::kWarps - 1) / C::kWarps : 0;
    unsigned char *ring = smem + warp * NST * C::kStageB;
    float *p_s = reinterpret_cast<float *>(smem + C::kRing) + warp * C::kPw;
    float *c_s = p_s + C::RPI * T * GP;
    float *mlbuf = reinterpret_cast<float *>(smem + C::kRing) + C::kWarps * C::kPw;
    const int half = lane / C::RL, lr = lane % C::RL;

    const unsigned char *kb = reinterpret_cast<const unsigned char *>(a.k) + lr * 16;
    const unsigned char *vb = reinterpret_cast<const unsigned char *>(a.v) + lr * 16;
    // pool row of token lane % TW of the warp's group j (-1 past the split), one per lane;
    // looked up one group ahead of its use, so the block table's latency is off the path
    auto lookup = [&](int j) -> int64_t {
        const int tok = t0 + (warp + C::kWarps * j) * TW + lane % TW;
        return j < mine && tok < t1 ? a.pv.row_phys(b, l, g, S0 + tok) : -1;
    };
    auto issue = [&](int j, int64_t row) {
        unsigned char *st = ring + (j % NST) * C::kStageB + half * T * C::kRowB + lr * 16;
#pragma unroll
        for (int t = 0; t < T; ++t) {
            const int64_t r = __shfl_sync(0xffffffffu, row, half * T + t);
            const int64_t at = (r < 0 ? 0 : r) * C::kRowB;
            cp_async16_zfill(st + t * C::kRowB, kb + at, r >= 0);
            cp_async16_zfill(st + (TW + t) * C::kRowB, vb + at, r >= 0);
        }
    };
#pragma unroll
    for (int i = 0; i < NST - 1; ++i) {
        issue(i, lookup(i));
        cp_async_commit();
    }
    int64_t row_next = lookup(NST - 1);

    float q[G][4];  // the lane's four dims of each head, pre-scaled into the log2 domain
    const float *qg = reinterpret_cast<const float *>(a.q) + (((int64_t)li * a.batch + b) * a.q_heads + (int64_t)g * G) * D;
#pragma unroll
    for (int h = 0; h < G; ++h) {
        const float4 x = *reinterpret_cast<const float4 *>(qg + h * D + lr * 4);
        q[h][0] = x.x * a.scale_log2;
        q[h][1] = x.y * a.scale_log2;
        q[h][2] = x.z * a.scale_log2;
        q[h][3] = x.w * a.scale_log2;
    }
    float o[G][4];
#pragma unroll
    for (int h = 0; h < G; ++h)
#pragma unroll
        for (int e = 0; e < 4; ++e) o[h][e] = 0.f;
    // after the exchange the lane holds logits x0 .. x0 + VPL - 1 of the group's T x GP
    // (head-major), all of one head
    const int x0 = lr / DUP * VPL, hx = x0 / T, tx = x0 % T;
    const bool first_copy = lr % DUP == 0;
    float m_run = -INFINITY, l_run = 0.f;
    float *lg = a.logits && hx < G
                    ? a.logits + ((((int64_t)b * a.sc_layers + a.sc_layer0 + li) * a.q_heads) + (int64_t)g * G + hx) *
                                     (int64_t)a.lstride
                    : nullptr;
    // bit j: logit x0 + j of the warp's group i is a valid, live token; fetched a group ahead
    auto live_of = [&](int i) -> uint32_t {
        uint32_t bits = 0u;
        const int tok = t0 + (warp + C::kWarps * i) * TW + half * T + tx;
#pragma unroll
        for (int j = 0; j < VPL; ++j)
            if (i < mine && hx < G && tok + j < t1 && (!prow || __ldg(prow + tok + j) >= 0)) bits |= 1u << j;
        return bits;
    };
    uint32_t live_next = live_of(0);

    for (int i = 0; i < mine; ++i) {
        if (i + NST - 1 < mine) issue(i + NST - 1, row_next);
        cp_async_commit();
        row_next = lookup(i + NST);
        const uint32_t live = live_next;
        live_next = live_of(i + 1);
        cp_async_wait<NST - 1>();
        const unsigned char *st = ring + (i % NST) * C::kStageB + half * T * C::kRowB + lr * 16;
        float z[C::N];
#pragma unroll
        for (int t = 0; t < T; ++t) {
            const float4 k = *reinterpret_cast<const float4 *>(st + t * C::kRowB);
#pragma unroll
            for (int h = 0; h < GP; ++h)
                z[h * T + t] = h < G ? fmaf(q[h % G][3], k.w, fmaf(q[h % G][2], k.z, fmaf(q[h % G][1], k.y, q[h % G][0] * k.x)))
                                     : 0.f;
        }
        // halving exchange over the row's lanes: each step sums pairs of lanes and leaves
        // each with half of the values; plain butterflies once one value is left
        int n = C::N;
#pragma unroll
        for (int off = C::RL / 2; off > 0; off >>= 1) {
            if (n > 1) {
                n >>= 1;
                const bool up = lr & off;
#pragma unroll
                for (int j = 0; j < C::N / 2; ++j)
                    if (j < n) {
                        const float keep = up ? z[j + n] : z[j], send = up ? z[j] : z[j + n];
                        z[j] = keep + __shfl_xor_sync(0xffffffffu, send, off);
                    }
            } else {
                z[0] += __shfl_xor_sync(0xffffffffu, z[0], off);
            }
        }
        const int tok = t0 + (warp + C::kWarps * i) * TW + half * T + tx;
        float mx = -INFINITY;
#pragma unroll
        for (int j = 0; j < VPL; ++j) {
            z[j] = (live >> j) & 1u ? z[j] : -INFINITY;
            if (lg && first_copy && tok + j < t1) lg[tok + j] = z[j];
            mx = fmaxf(mx, z[j]);
        }
#pragma unroll
        for (int off = DUP; off < T * DUP / VPL; off <<= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, off));
        const float m_new = fmaxf(m_run, mx);
        const float ref = m_new == -INFINITY ? 0.f : m_new;  // every token so far dead: nothing to scale
        const float corr = exp2f(m_run - ref);
        const bool moved = __any_sync(0xffffffffu, m_new != m_run);
        m_run = m_new;
        float sum = 0.f;
#pragma unroll
        for (int j = 0; j < VPL; ++j) {
            const float p = exp2f(z[j] - ref);
            sum += p;
            if (first_copy) p_s[(half * T + tx + j) * GP + hx] = p;
        }
        l_run = l_run * corr + sum;
        if (first_copy && tx == 0) c_s[half * GP + hx] = corr;
        __syncwarp();
        if (moved) {
#pragma unroll
            for (int h = 0; h < G; ++h) {
                const float cr = c_s[half * GP + h];
#pragma unroll
                for (int e = 0; e < 4; ++e) o[h][e] *= cr;
            }
        }
#pragma unroll
        for (int t = 0; t < T; ++t) {
            const float4 v = *reinterpret_cast<const float4 *>(st + (TW + t) * C::kRowB);
#pragma unroll
            for (int h = 0; h < G; ++h) {
                const float p = p_s[(half * T + t) * GP + h];
                o[h][0] = fmaf(p, v.x, o[h][0]);
                o[h][1] = fmaf(p, v.y, o[h][1]);
                o[h][2] = fmaf(p, v.z, o[h][2]);
                o[h][3] = fmaf(p, v.w, o[h][3]);
            }
        }
        __syncwarp();  // the next group rewrites p_s and c_s
    }
#pragma unroll
    for (int off = DUP; off < T * DUP / VPL; off <<= 1) l_run += __shfl_xor_sync(0xffffffffu, l_run, off);
    cp_async_wait<0>();
    __syncthreads();  // every warp is done with its ring: the outputs go there
    float *obuf = reinterpret_cast<float *>(smem);
    const int part = warp * C::RPI + half;
    if (first_copy && tx == 0) {
        mlbuf[(part * GP + hx) * 2] = m_run;
        mlbuf[(part * GP + hx) * 2 + 1] = l_run;
    }
#pragma unroll
    for (int h = 0; h < G; ++h)
        *reinterpret_cast<float4 *>(obuf + (part * G + h) * D + lr * 4) = make_float4(o[h][0], o[h][1], o[h][2], o[h][3]);
    __syncthreads();
    finish_split<float, D, GP, C::P>(a, obuf, mlbuf, G, s, ns_active, b, li, g);
}

template <typename T>
__global__ void __launch_bounds__(128) combine_kernel(const CombineArgs a) {
    pdl_wait();
    const int h = blockIdx.x;
    const int b = blockIdx.y % a.batch, li = blockIdx.y / a.batch;
    const int D = a.head_dim;
    const int L = a.len[b];
    const int ns = min((L + a.split_tokens - 1) / a.split_tokens, a.n_splits);
    const int64_t pbase = (((int64_t)b * a.n_layers + li) * a.q_heads + h) * a.n_splits;
    const float *ml = a.part_ml + pbase * 2;
    float M = -INFINITY;
    for (int s = 0; s < ns; ++s) M = fmaxf(M, ml[2 * s]);
    const float Mref = M == -INFINITY ? 0.f : M;  // splits whose slots are all dead carry -inf
    float wsum = 0.f;
    for (int s = 0; s < ns; ++s) wsum += ml[2 * s + 1] * exp2f(ml[2 * s] - Mref);
    const float inv = wsum > 0.f ? 1.f / wsum : 0.f;
    const int64_t obase = (((int64_t)li * a.batch + b) * a.q_heads + h) * D;
    for (int e = threadIdx.x; e < D; e += blockDim.x) {
        float acc = 0.f;
        for (int s = 0; s < ns; ++s) acc += a.part_o[(pbase + s) * D + e] * exp2f(ml[2 * s] - Mref);
        Chunk<T>::store(a.out, obase + e, acc * inv);
    }
    if (a.lse2 && threadIdx.x == 0)
        a.lse2[((int64_t)b * a.sc_layers + a.sc_layer0 + li) * a.q_heads + h] = wsum > 0.f ? M + log2f(wsum) : -INFINITY;
}

template <typename T, int D, int G>
cudaError_t launch_attend_t(const AttendArgs &a, cudaStream_t st) {
    using C = AttendCfg<T, D, G>;
    dim3 grid(a.n_splits, a.pv.kv_heads, a.batch * a.n_layers);
    if (a.logits) {
        auto k = attend_split_kernel<T, D, G, true>;
        cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, C::kSmemBytes);
        if (e != cudaSuccess) return e;
        { cudaError_t le = launch_k(k, grid, dim3(kAttendThreads), C::kSmemBytes, st, a); if (le != cudaSuccess) return le; }
    } else {
        auto k = attend_split_kernel<T, D, G, false>;
        cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, C::kSmemBytes);
        if (e != cudaSuccess) return e;
        { cudaError_t le = launch_k(k, grid, dim3(kAttendThreads), C::kSmemBytes, st, a); if (le != cudaSuccess) return le; }
    }
    note_launch();
    return cudaGetLastError();
}

template <int D, int G>
cudaError_t launch_attend_f32_g(const AttendArgs &a, cudaStream_t st) {
    constexpr int smem = F32Cfg<D, G>::kSmemBytes;
    auto k = attend_f32_kernel<D, G>;
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    e = launch_k(k, dim3(a.n_splits, a.pv.kv_heads, a.batch * a.n_layers), dim3(kAttendThreads), smem, st, a);
    note_launch();
    return e != cudaSuccess ? e : cudaGetLastError();
}
template <int D>
cudaError_t launch_attend_f32(const AttendArgs &a, int group, cudaStream_t st) {
    switch (group) {
        case 1: return launch_attend_f32_g<D, 1>(a, st);
        case 2: return launch_attend_f32_g<D, 2>(a, st);
        case 4: return launch_attend_f32_g<D, 4>(a, st);
        case 7: return launch_attend_f32_g<D, 7>(a, st);
        case 8: return launch_attend_f32_g<D, 8>(a, st);
        default: return cudaErrorInvalidValue;
    }
}

template <typename T, int D>
cudaError_t launch_attend_d(const AttendArgs &a, int group, cudaStream_t st) {
    switch (group) {
        case 1: return launch_attend_t<T, D, 1>(a, st);
        case 2: return launch_attend_t<T, D, 2>(a, st);
        case 4: return launch_attend_t<T, D, 4>(a, st);
        case 7: return launch_attend_t<T, D, 7>(a, st);
        case 8: return launch_attend_t<T, D, 8>(a, st);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace

cudaError_t launch_attend(const AttendArgs &a, int dtype, int head_dim, int group, cudaStream_t st) {
    if (dtype == IKV_BF16) {
        if (head_dim == 128) return launch_attend_d<__nv_bfloat16, 128>(a, group, st);
        if (head_dim == 64) return launch_attend_d<__nv_bfloat16, 64>(a, group, st);
    } else {
        if (head_dim == 128) return launch_attend_f32<128>(a, group, st);
        if (head_dim == 64) return launch_attend_f32<64>(a, group, st);
    }
    return cudaErrorInvalidValue;
}

cudaError_t launch_combine(const CombineArgs &a, int dtype, cudaStream_t st) {
    dim3 grid(a.q_heads, a.batch * a.n_layers);
    if (dtype == IKV_BF16)
        { cudaError_t le = launch_k(combine_kernel<__nv_bfloat16>, grid, dim3(128), 0, st, a); if (le != cudaSuccess) return le; }
    else
        { cudaError_t le = launch_k(combine_kernel<float>, grid, dim3(128), 0, st, a); if (le != cudaSuccess) return le; }
    note_launch();
    return cudaGetLastError();
}

}  // namespace ikv
