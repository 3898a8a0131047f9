// Split-K grouped-query decode attention that also emits per-token logits, for the shapes
// the TMA / tcgen05 kernel of attend_tc.cu does not take: fp32 caches, 64-dim heads, page
// sizes that do not tile 128 rows, pools past its 32-bit row coordinates.
//
// One CTA of four warps handles (split s, kv head g, sequence b, layer l): the G query heads
// of KV head g against cache slots [s*split, min((s+1)*split, len[b])).  Each warp streams its
// own share of the tokens through a private cp.async ring and keeps its own online softmax
// in the log2 domain; the logits are written out for the Eq. 1 score pass.  The warps'
// results meet in shared memory once, at the end; a unit of several splits is merged by its
// last CTA to arrive.
#include "book.cuh"

namespace ikv {

__device__ unsigned int g_attend_error = 0;  // bit 2: an append found no free slot (start + len = cap)

namespace {

// 16 bytes to shared memory, the first n of them (0 or 16) from gmem and the rest zeros
__device__ __forceinline__ void cp_async16_n(uint32_t smem, const void *gmem, uint32_t n) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(smem), "l"(gmem), "r"(n) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory"); }

// What the CTAs of a (sequence, layer, kv head) unit do once a CTA has its split's result:
// P partial softmaxes over disjoint tokens, obuf [P][G][D] unnormalised outputs and mlbuf
// [P][GP][2] (max, sum) in shared memory, merged into the split's (max, sum, output).  A
// unit of one split is final and goes straight to out and lse2; otherwise the split goes to
// the workspace and the unit's last CTA to arrive (counter only, no waiting) merges them.
// Entered by every thread of the CTA; obuf is reused.
template <typename T, int D, int GP, int P>
__device__ __forceinline__ void finish_split(const AttendArgs &a, float *obuf, float *mlbuf, int G, int s,
                                             int ns_active, int b, int li, int g) {
    const int tid = threadIdx.x, warp = tid >> 5;
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
            store_as(static_cast<T *>(a.out) + (hrow + h) * D + e, sum > 0.f ? acc / sum : 0.f);
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
    if (ns_active == 1 || !a.arrivals) return;  // without counters the caller merges later
    __shared__ int last;
    const int64_t unit = ((int64_t)b * a.n_layers + li) * a.pv.kv_heads + g;
    __syncthreads();
    if (tid == 0) last = arrive_acq_rel(a.arrivals + unit) == ns_active - 1;
    __syncthreads();
    if (!last) return;
    if (tid == 0) a.arrivals[unit] = 0;
    for (int h = warp; h < G; h += kAttendThreads / 32)
        merge_head<D / 32>(reinterpret_cast<const float2 *>(a.part_ml) + pbase + (int64_t)h * a.n_splits,
                           a.part_o + (pbase + (int64_t)h * a.n_splits) * D, ns_active, obuf + warp * kMaxSplits,
                           static_cast<T *>(a.out) + (hrow + h) * D, a.lse2 + lrow + h);
}

// The new token's K and V rows of (layer, KV head) from k_new / v_new into pool row `row`, and the
// V row's norm into *vnorm (or null), by one warp.
template <typename T, int D>
__device__ __forceinline__ void store_new_rows(const AttendArgs &a, int64_t unit, int64_t row, float *vnorm) {
    constexpr int kChunks = D * (int)sizeof(T) / 16, E = 16 / (int)sizeof(T);
    const int lane = threadIdx.x & 31;
    float sq = 0.f;
    for (int c = lane; c < kChunks; c += 32) {
        const uint4 k = reinterpret_cast<const uint4 *>(a.k_new)[unit * kChunks + c];
        const uint4 v = reinterpret_cast<const uint4 *>(a.v_new)[unit * kChunks + c];
        reinterpret_cast<uint4 *>(const_cast<void *>(a.k))[row * kChunks + c] = k;
        reinterpret_cast<uint4 *>(const_cast<void *>(a.v))[row * kChunks + c] = v;
        const T *x = reinterpret_cast<const T *>(&v);
#pragma unroll
        for (int e = 0; e < E; ++e) sq += static_cast<float>(x[e]) * static_cast<float>(x[e]);
    }
    if (vnorm) {
        sq = warp_sum(sq);
        if (lane == 0) *vnorm = sqrtf(sq);
    }
}

// A sequence without slots: output 0, log-sum-exp -inf (written by its first split's CTA).
template <typename T>
__device__ __forceinline__ void store_empty(const AttendArgs &a, int G, int D, int b, int li, int g) {
    const int64_t hrow = ((int64_t)li * a.batch + b) * a.q_heads + (int64_t)g * G;
    for (int i = threadIdx.x; i < G * D; i += kAttendThreads) store_as(static_cast<T *>(a.out) + hrow * D + i, 0.f);
    if ((int)threadIdx.x < G)
        a.lse2[((int64_t)b * a.sc_layers + a.sc_layer0 + li) * a.q_heads + (int64_t)g * G + threadIdx.x] = -INFINITY;
}

// N consecutive floats of shared memory, N * 4 bytes aligned (16 at most)
template <int N>
__device__ __forceinline__ void load_vec(const float *p, float (&x)[N]) {
    if constexpr (N == 1) {
        x[0] = *p;
    } else if constexpr (N == 2) {
        const float2 y = *reinterpret_cast<const float2 *>(p);
        x[0] = y.x;
        x[1] = y.y;
    } else {
#pragma unroll
        for (int i = 0; i < N / 4; ++i) {
            const float4 y = reinterpret_cast<const float4 *>(p)[i];
            x[4 * i] = y.x;
            x[4 * i + 1] = y.y;
            x[4 * i + 2] = y.z;
            x[4 * i + 3] = y.w;
        }
    }
}

// fp32 K/V.  HBM bound: a K and V byte costs G / 4 FMAs, half an SM's rate at G = 8.  Every
// warp is on its own: it takes every fourth group of T (d = 128) or 2 T (d = 64) tokens of
// the split through its own cp.async ring and keeps its own online softmax, so the loop has
// no block barrier, and each lane reads back the 16 bytes of each row that it copied itself.
// A lane's partial dot products of T tokens x G heads are summed over the row's lanes by a
// halving exchange (one shuffle a value instead of five), which leaves each lane with the
// logits it exponentiates; the probabilities go through a few hundred bytes of shared memory
// to the P.V products.  Measured, a whole step of b = 4, 8 layers, 16 / 4 heads of 128, 2048
// tokens (269 MB, 39.7 us at the copy rate): 185.1 -> 76.9 us against a kernel of one CTA of
// four warps an SM with five block barriers per 64-token tile.  Warps hide the rest, not deep
// rings: two CTAs of three stages an SM 72.7 us, three of two stages 61.8 (G = 4; four of
// T = 4 and three stages 65.4); at G = 8, whose logits of 8 tokens fill the registers, two
// CTAs 89.8 us, three with T = 4 and four stages 81.4.
template <int D, int G>
struct F32Cfg {
    static constexpr int GP = G == 7 ? 8 : G;
    static constexpr int RL = D / 4;              // lanes of a row (16 bytes each)
    static constexpr int RPI = 32 / RL;           // rows a warp reads at once
    static constexpr int T = G <= 4 ? 8 : 4;      // tokens per group and row slot
    static constexpr int TW = T * RPI;            // tokens per warp and group
    static constexpr int kRowB = D * 4;
    static constexpr int kStageB = 2 * TW * kRowB;
    static constexpr int NST = G <= 4 ? 2 : 4;
    static constexpr int kWarps = kAttendThreads / 32;
    static constexpr int kRing = kWarps * NST * kStageB;
    static constexpr int P = kWarps * RPI;        // independent softmaxes of a CTA
    static constexpr int N = T * GP;              // logits of a group per row slot
    static constexpr int VPL = N > RL ? N / RL : 1;   // logits a lane ends up with
    static constexpr int DUP = N < RL ? RL / N : 1;   // lanes holding the same logit
    static constexpr int kPw = (RPI * (T + 1) * GP + 3) / 4 * 4;  // floats per warp: probabilities, rescales
    static constexpr int kSmemBytes = kRing + (kWarps * kPw + 2 * P * GP) * 4;
    static_assert(P * G * D * 4 <= kRing && kWarps * kMaxSplits * 4 <= kRing, "the merge reuses the ring");
};

template <int D, int G>
__global__ void __launch_bounds__(kAttendThreads, kF32CtasPerSm) attend_f32_kernel(const AttendArgs a) {
    using C = F32Cfg<D, G>;
    constexpr int GP = C::GP, T = C::T, TW = C::TW, NST = C::NST, VPL = C::VPL, DUP = C::DUP;
    pdl_wait();
    extern __shared__ __align__(128) unsigned char smem[];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // 1-D grid: the bookkeeping CTAs, if any, then splits, kv heads, sequences, layers
    int bid = blockIdx.x;
    if (a.book.on) {
        const int books = a.batch * a.rows_per_seq;
        if (bid < books) {
            book_row<kAttendThreads>(a.book, a.len, a.pv.start, a.cap, a.rows_per_seq, bid, &g_attend_error,
                                     reinterpret_cast<uint32_t *>(smem), C::kRing / 4);
            return;
        }
        bid -= books;
    }
    const int s = bid % a.n_splits;
    bid /= a.n_splits;
    const int g = bid % a.pv.kv_heads;
    bid /= a.pv.kv_heads;
    const int b = bid % a.batch, li = bid / a.batch;
    const int l = a.layer0 + li;
    const int L0 = a.len[b];
    const int S0 = a.pv.start_of(b);
    const bool grown = a.book.on && S0 + L0 < a.cap;
    const int L = L0 + (grown ? 1 : 0);
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
    // the new token's slot (-1: none): its rows come from k_new / v_new, not from the pool
    const int t_new = a.book.on ? (grown ? L0 : -1) : a.k_new ? a.slot[b] : -1;
    const int64_t unit = ((int64_t)li * a.batch + b) * a.pv.kv_heads + g;
    const unsigned char *kn = reinterpret_cast<const unsigned char *>(a.k_new) + unit * C::kRowB + lr * 16;
    const unsigned char *vn = reinterpret_cast<const unsigned char *>(a.v_new) + unit * C::kRowB + lr * 16;
    // pool row of token lane % TW of the warp's group j (kNoRow past the split, kNewRow the new
    // token; a row index fits 32 bits: rows are 256 bytes at least), one per lane; looked up one
    // group ahead of its use, so the block table's latency is off the path
    constexpr uint32_t kNoRow = ~0u, kNewRow = ~0u - 1u;
    auto lookup = [&](int j) -> uint32_t {
        const int tok = t0 + (warp + C::kWarps * j) * TW + lane % TW;
        return j < mine && tok < t1 ? tok == t_new ? kNewRow : (uint32_t)a.pv.row_phys(b, l, g, S0 + tok) : kNoRow;
    };
    const uint32_t ring_u = static_cast<uint32_t>(__cvta_generic_to_shared(ring)) + half * T * C::kRowB + lr * 16;
    auto issue = [&](int stage, uint32_t row) {
        const uint32_t st = ring_u + stage * C::kStageB;
#pragma unroll
        for (int t = 0; t < T; ++t) {
            const uint32_t r = __shfl_sync(0xffffffffu, row, half * T + t);
            const uint32_t n = r == kNoRow ? 0u : 16u;
            const uint64_t at = (uint64_t)(r >= kNewRow ? 0u : r) * C::kRowB;
            cp_async16_n(st + t * C::kRowB, r == kNewRow ? kn : kb + at, n);
            cp_async16_n(st + (TW + t) * C::kRowB, r == kNewRow ? vn : vb + at, n);
        }
    };
#pragma unroll
    for (int i = 0; i < NST - 1; ++i) {
        issue(i, lookup(i));
        cp_async_commit();
    }
    uint32_t row_next = lookup(NST - 1);
    if (warp == 0 && t_new >= t0 && t_new < t1)  // into the cache, for later steps
        store_new_rows<float, D>(a, unit, a.pv.row_phys(b, l, g, S0 + t_new),
                                 a.vnorm ? a.vnorm + (((int64_t)l * a.batch + b) * a.pv.kv_heads + g) * a.cap + t_new : nullptr);

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
            if (i < mine && hx < G && tok + j < t1 && (!prow || tok + j == t_new || __ldg(prow + tok + j) >= 0)) bits |= 1u << j;
        return bits;
    };
    uint32_t live_next = live_of(0);

    int stage = 0;
    for (int i = 0; i < mine; ++i) {
        if (i + NST - 1 < mine) issue(stage == 0 ? NST - 1 : stage - 1, row_next);
        cp_async_commit();
        row_next = lookup(i + NST);
        const uint32_t live = live_next;
        live_next = live_of(i + 1);
        cp_async_wait<NST - 1>();
        const unsigned char *st = ring + stage * C::kStageB + half * T * C::kRowB + lr * 16;
        stage = stage == NST - 1 ? 0 : stage + 1;
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
            float pt[GP];
            load_vec<GP>(p_s + (half * T + t) * GP, pt);
#pragma unroll
            for (int h = 0; h < G; ++h) {
                const float p = pt[h];
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

// bf16 K/V (head_dim 64, and the 128-dim shapes the TMA kernel of attend_tc.cu does not
// take).  HBM bound; mma.sync keeps the arithmetic (32 m16n8k16 per 16 tokens of 64 dims)
// under half of the stream's time.  As in the fp32 kernel every warp runs alone: its own
// ring of 16-token stages, its own online softmax over every fourth group of the split, no
// block barrier.  The heads are the M rows: S = Q K^T leaves each lane four logits of one
// head, which are the A operand of O += P V as they stand.  Rows 8-15 of that operand would
// be padding (a group has at most 8 heads); they carry the second of three bf16 terms whose
// sum is the fp32 probability bit for bit (8 + 8 + 8 mantissa bits), and one more product
// adds the third, so P loses nothing to the tensor cores' operand type. Measured, a whole step of
// b = 8, 16 layers, 32 / 8 heads of 64, 2048 tokens (539 MB, 79.5 us at the copy rate):
// 222.4 -> 128.5 us against the CUDA-core kernel with its block barriers; 128 dims in
// 48-token pages 271 -> 208 us when 32 tokens, not 16, came to share the row look-ups and
// the registers left room for 16 warps an SM.  The two halves of a block are a rolled loop
// at 64 dims (unrolled, 128 registers spill 48 bytes: 122.4 us a step against 118.8) and
// unrolled at 128 (255 registers, no spill: 206.3 us against 207.4).  What is left: the
// ramp of each CTA (length, table, rows: three dependent loads) and 1.7 waves of CTAs.
__device__ __forceinline__ void ldsm_x4(uint32_t addr, uint32_t (&r)[4]) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr)
                 : "memory");
}
__device__ __forceinline__ void ldsm_x4_trans(uint32_t addr, uint32_t (&r)[4]) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr)
                 : "memory");
}
__device__ __forceinline__ void mma_16x8x16(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                            uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, "
        "%2, %3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
// x and y to bf16 (packed), and what that leaves of them
__device__ __forceinline__ uint32_t take_bf16(float &x, float &y) {
    const __nv_bfloat162 t = __floats2bfloat162_rn(x, y);
    x -= __low2float(t);
    y -= __high2float(t);
    return *reinterpret_cast<const uint32_t *>(&t);
}

template <int D>
struct Bf16Cfg {
    static constexpr int GP = 8;                 // heads of the M rows 0-7
    static constexpr int TW = 16;                // tokens of a stage; a warp's block is two stages
    static constexpr int kRowB = D * 2;
    static constexpr int RL = kRowB / 16;        // lanes of a row (16 bytes each)
    static constexpr int RPI = 32 / RL;          // rows a warp copies at once
    static constexpr int kStageB = 2 * TW * kRowB;
    static constexpr int NST = 3;
    static constexpr int kWarps = kAttendThreads / 32;
    static constexpr int kRing = kWarps * NST * kStageB;
    static constexpr int kSmemBytes = kRing + 2 * kWarps * GP * 4;
    static constexpr int kCtasPerSm = D == 64 ? kBf16D64CtasPerSm : kBf16D128CtasPerSm;
    static_assert(kWarps * GP * D * 4 <= kRing && kWarps * kMaxSplits * 4 <= kRing, "the merge reuses the ring");
    static_assert(kCtasPerSm * (kSmemBytes + 1024) <= 227 * 1024, "resident CTAs");
};

template <int D>
__global__ void __launch_bounds__(kAttendThreads, Bf16Cfg<D>::kCtasPerSm) attend_bf16_kernel(const AttendArgs a) {
    using C = Bf16Cfg<D>;
    constexpr int TW = C::TW, NST = C::NST;
    pdl_wait();
    extern __shared__ __align__(128) unsigned char smem[];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // 1-D grid: the bookkeeping CTAs, if any, then splits, kv heads, sequences, layers
    int bid = blockIdx.x;
    if (a.book.on) {
        const int books = a.batch * a.rows_per_seq;
        if (bid < books) {
            book_row<kAttendThreads>(a.book, a.len, a.pv.start, a.cap, a.rows_per_seq, bid, &g_attend_error,
                                     reinterpret_cast<uint32_t *>(smem), C::kRing / 4);
            return;
        }
        bid -= books;
    }
    const int s = bid % a.n_splits;
    bid /= a.n_splits;
    const int g = bid % a.pv.kv_heads;
    bid /= a.pv.kv_heads;
    const int b = bid % a.batch, li = bid / a.batch;
    const int l = a.layer0 + li;
    const int G = a.q_heads / a.pv.kv_heads;
    const int L0 = a.len[b];
    const int S0 = a.pv.start_of(b);
    const bool grown = a.book.on && S0 + L0 < a.cap;
    const int L = L0 + (grown ? 1 : 0);
    const int t0 = s * a.split_tokens;
    if (t0 >= L) {
        if (s == 0) store_empty<__nv_bfloat16>(a, G, D, b, li, g);
        return;
    }
    const int t1 = min(t0 + a.split_tokens, L);
    const int ns_active = min((L + a.split_tokens - 1) / a.split_tokens, a.n_splits);
    const int32_t *prow = a.pos ? a.pos + ((int64_t)b * a.rows_per_seq + (a.rows_per_seq == 1 ? 0 : g)) * a.cap : nullptr;
    const uint32_t ring = static_cast<uint32_t>(__cvta_generic_to_shared(smem)) + warp * NST * C::kStageB;
    float *mlbuf = reinterpret_cast<float *>(smem + C::kRing);

    // The warp takes every fourth 32-token block of the split, from tok0 on.  Lane i looks up
    // the pool row of the block's token i (a row index fits 32 bits: rows are 128 bytes at
    // least; ~0 past the split) and its liveness, two blocks and one block ahead of their use.
    int tok0 = t0 + warp * 32;
    constexpr int kStride = C::kWarps * 32;
    const int64_t page0 = (int64_t)l * a.pv.num_pages;
    const int32_t *table = a.pv.block_table + (int64_t)b * a.pv.max_pages;
    // the new token's slot (-1: none): its rows come from k_new / v_new, not from the pool
    const int t_new = a.book.on ? (grown ? L0 : -1) : a.k_new ? a.slot[b] : -1;
    constexpr uint32_t kNewRow = ~0u - 1u;
    auto lookup = [&](int base) -> uint32_t {
        const int tok = base + lane;
        if (tok >= t1) return ~0u;
        if (tok == t_new) return kNewRow;
        const int phys = S0 + tok;
        const int lp = a.pv.page_shift >= 0 ? phys >> a.pv.page_shift : phys / a.pv.page_size;
        return (uint32_t)(((page0 + table[lp]) * a.pv.kv_heads + g) * a.pv.page_size + (phys - lp * a.pv.page_size));
    };
    auto alive = [&](int base) -> bool {
        const int tok = base + lane;
        return tok < t1 && (!prow || tok == t_new || __ldg(prow + tok) >= 0);
    };
    // 16-byte chunk c of a row lies at c ^ (row % 8): the eight rows an ldmatrix reads at one
    // chunk fall into different banks
    const int cr = lane / C::RL, cc = lane % C::RL;
    const unsigned char *kb = reinterpret_cast<const unsigned char *>(a.k) + cc * 16;
    const unsigned char *vb = reinterpret_cast<const unsigned char *>(a.v) + cc * 16;
    const int64_t unit = ((int64_t)li * a.batch + b) * a.pv.kv_heads + g;
    const unsigned char *kn = reinterpret_cast<const unsigned char *>(a.k_new) + unit * C::kRowB + cc * 16;
    const unsigned char *vn = reinterpret_cast<const unsigned char *>(a.v_new) + unit * C::kRowB + cc * 16;
    auto issue = [&](int stage, int half, uint32_t rows) {
        const uint32_t st = ring + stage * C::kStageB + cr * C::kRowB;
#pragma unroll
        for (int t = 0; t < TW; t += C::RPI) {
            const uint32_t r = __shfl_sync(0xffffffffu, rows, half * TW + t + cr);
            const uint32_t n = r == ~0u ? 0u : 16u;
            const uint64_t at = (uint64_t)(r >= kNewRow ? 0u : r) * C::kRowB;
            const uint32_t dst = st + t * C::kRowB + ((cc ^ ((t + cr) & 7)) << 4);
            cp_async16_n(dst, r == kNewRow ? kn : kb + at, n);
            cp_async16_n(dst + TW * C::kRowB, r == kNewRow ? vn : vb + at, n);
        }
        cp_async_commit();
    };
    {
        const uint32_t rows = lookup(tok0);
        issue(0, 0, rows);
        issue(1, 1, rows);
    }
    uint32_t rows_next = lookup(tok0 + kStride);
    uint32_t live = __ballot_sync(0xffffffffu, alive(tok0));
    if (warp == 0 && t_new >= t0 && t_new < t1)  // into the cache, for later steps
        store_new_rows<__nv_bfloat16, D>(a, unit, a.pv.row_phys(b, l, g, S0 + t_new),
                                         a.vnorm ? a.vnorm + (((int64_t)l * a.batch + b) * a.pv.kv_heads + g) * a.cap + t_new
                                                 : nullptr);

    // the lane's head (M row) and its tokens tq, tq + 1, tq + 8, tq + 9 of a stage
    const int h = lane >> 2, tq = (lane & 3) * 2;
    uint32_t qa[D / 16][2];
    {
        const __nv_bfloat16 *qg = reinterpret_cast<const __nv_bfloat16 *>(a.q) +
                                  (((int64_t)li * a.batch + b) * a.q_heads + (int64_t)g * G + h) * D + tq;
#pragma unroll
        for (int k = 0; k < D / 16; ++k) {
            qa[k][0] = h < G ? *reinterpret_cast<const uint32_t *>(qg + k * 16) : 0u;
            qa[k][1] = h < G ? *reinterpret_cast<const uint32_t *>(qg + k * 16 + 8) : 0u;
        }
    }
    float *lg = a.logits && h < G
                    ? a.logits + ((((int64_t)b * a.sc_layers + a.sc_layer0 + li) * a.q_heads) + (int64_t)g * G + h) *
                                     (int64_t)a.lstride + tq
                    : nullptr;
    // ldmatrix row addresses: K as B (tokens x dims), V transposed (dims x tokens)
    const int mat = lane >> 3, mr = lane & 7;
    const uint32_t k_row = (uint32_t)(((mat >> 1) * 8 + mr) * C::kRowB), k_c = mat & 1;
    const uint32_t v_row = (uint32_t)((TW + (mat & 1) * 8 + mr) * C::kRowB), v_c = mat >> 1;

    float o[D / 8][4];
#pragma unroll
    for (int n = 0; n < D / 8; ++n)
#pragma unroll
        for (int e = 0; e < 4; ++e) o[n][e] = 0.f;
    float m_run = -INFINITY, l_run = 0.f;
    int stage = 0;  // ring stage of the next 16 tokens

    for (; tok0 < t1; tok0 += kStride) {
        const uint32_t rows = rows_next;
        rows_next = lookup(tok0 + 2 * kStride);
        const bool alive_next = alive(tok0 + kStride);
#pragma unroll (D == 64 ? 1 : 2)
        for (int half = 0; half < 2; ++half) {
            __syncwarp();  // the stage about to be refilled was read in the previous round
            issue(stage == 0 ? NST - 1 : stage - 1, half, rows);
            cp_async_wait<NST - 1>();
            __syncwarp();  // every lane's copies of this stage have landed
            const uint32_t st = ring + stage * C::kStageB;
            stage = stage == NST - 1 ? 0 : stage + 1;
            float sc[2][4];
#pragma unroll
            for (int n = 0; n < 2; ++n)
#pragma unroll
                for (int e = 0; e < 4; ++e) sc[n][e] = 0.f;
#pragma unroll
            for (int k = 0; k < D / 16; ++k) {
                uint32_t kf[4];
                ldsm_x4(st + k_row + (((2 * k + k_c) ^ mr) << 4), kf);
                mma_16x8x16(sc[0], qa[k][0], 0u, qa[k][1], 0u, kf[0], kf[1]);
                mma_16x8x16(sc[1], qa[k][0], 0u, qa[k][1], 0u, kf[2], kf[3]);
            }
            const uint32_t lv = h < G ? live >> (half * TW + tq) : 0u;  // bits 0, 1, 8, 9: the lane's tokens
            float z[4];
#pragma unroll
            for (int j = 0; j < 4; ++j)
                z[j] = (lv >> ((j >> 1) * 8 + (j & 1))) & 1u ? sc[j >> 1][j & 1] * a.scale_log2 : -INFINITY;
            if (lg) {
                const int x = tok0 + half * TW;
#pragma unroll
                for (int n = 0; n < 2; ++n) {
                    if (x + n * 8 + tq + 1 < t1)
                        *reinterpret_cast<float2 *>(lg + x + n * 8) = make_float2(z[2 * n], z[2 * n + 1]);
                    else if (x + n * 8 + tq < t1)
                        lg[x + n * 8] = z[2 * n];
                }
            }
            float mx = fmaxf(fmaxf(z[0], z[1]), fmaxf(z[2], z[3]));
            mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
            mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
            const float m_new = fmaxf(m_run, mx);
            const float ref = m_new == -INFINITY ? 0.f : m_new;  // every token so far dead: nothing to scale
            if (__any_sync(0xffffffffu, m_new != m_run)) {
                const float corr = exp2f(m_run - ref);
                l_run *= corr;
#pragma unroll
                for (int n = 0; n < D / 8; ++n)
#pragma unroll
                    for (int e = 0; e < 4; ++e) o[n][e] *= corr;
            }
            m_run = m_new;
            float p[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) p[j] = exp2f(z[j] - ref);
            l_run += (p[0] + p[1]) + (p[2] + p[3]);
            const uint32_t h0 = take_bf16(p[0], p[1]), h1 = take_bf16(p[2], p[3]);
            const uint32_t m0 = take_bf16(p[0], p[1]), m1 = take_bf16(p[2], p[3]);
            const uint32_t l0 = take_bf16(p[0], p[1]), l1 = take_bf16(p[2], p[3]);
#pragma unroll
            for (int n = 0; n < D / 16; ++n) {
                uint32_t vf[4];
                ldsm_x4_trans(st + v_row + (((2 * n + v_c) ^ mr) << 4), vf);
                mma_16x8x16(o[2 * n], h0, m0, h1, m1, vf[0], vf[1]);
                mma_16x8x16(o[2 * n + 1], h0, m0, h1, m1, vf[2], vf[3]);
                mma_16x8x16(o[2 * n], 0u, l0, 0u, l1, vf[0], vf[1]);
                mma_16x8x16(o[2 * n + 1], 0u, l0, 0u, l1, vf[2], vf[3]);
            }
        }
        live = __ballot_sync(0xffffffffu, alive_next);
    }
    l_run += __shfl_xor_sync(0xffffffffu, l_run, 1);
    l_run += __shfl_xor_sync(0xffffffffu, l_run, 2);
    cp_async_wait<0>();
    __syncthreads();  // every warp is done with its ring: the outputs go there
    float *obuf = reinterpret_cast<float *>(smem);
    if ((lane & 3) == 0) {
        mlbuf[(warp * C::GP + h) * 2] = m_run;
        mlbuf[(warp * C::GP + h) * 2 + 1] = l_run;
    }
    if (h < G) {
#pragma unroll
        for (int n = 0; n < D / 8; ++n) {
            // an infinite V makes the first term's sum infinite and the others' NaN (0 x inf)
            const float x = isfinite(o[n][0]) ? o[n][0] + o[n][2] : o[n][0];
            const float y = isfinite(o[n][1]) ? o[n][1] + o[n][3] : o[n][1];
            *reinterpret_cast<float2 *>(obuf + (warp * G + h) * D + n * 8 + tq) = make_float2(x, y);
        }
    }
    __syncthreads();
    finish_split<__nv_bfloat16, D, C::GP, C::kWarps>(a, obuf, mlbuf, G, s, ns_active, b, li, g);
}

dim3 attend_grid(const AttendArgs &a) {
    return dim3((unsigned)a.n_splits * a.pv.kv_heads * a.batch * a.n_layers + (a.book.on ? a.batch * a.rows_per_seq : 0));
}

template <int D, int G>
cudaError_t launch_attend_f32_g(const AttendArgs &a, cudaStream_t st) {
    constexpr int smem = F32Cfg<D, G>::kSmemBytes;
    auto k = attend_f32_kernel<D, G>;
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    e = launch_k(k, attend_grid(a), dim3(kAttendThreads), smem, st, a);
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

template <int D>
cudaError_t launch_attend_bf16(const AttendArgs &a, cudaStream_t st) {
    constexpr int smem = Bf16Cfg<D>::kSmemBytes;
    cudaError_t e = cudaFuncSetAttribute(attend_bf16_kernel<D>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    e = launch_k(attend_bf16_kernel<D>, attend_grid(a), dim3(kAttendThreads), smem,
                 st, a);
    note_launch();
    return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace

cudaError_t launch_attend(const AttendArgs &a, int dtype, int head_dim, int group, cudaStream_t st) {
    if (dtype == IKV_BF16) {
        if (head_dim == 128) return launch_attend_bf16<128>(a, st);
        if (head_dim == 64) return launch_attend_bf16<64>(a, st);
    } else {
        if (head_dim == 128) return launch_attend_f32<128>(a, group, st);
        if (head_dim == 64) return launch_attend_f32<64>(a, group, st);
    }
    return cudaErrorInvalidValue;
}

cudaError_t read_clear_attend_error(unsigned int *v) {
    unsigned int z = 0;
    cudaError_t e = cudaMemcpyFromSymbol(v, g_attend_error, sizeof(*v));
    if (e == cudaSuccess) e = cudaMemcpyToSymbol(g_attend_error, &z, sizeof(z));
    return e;
}

}  // namespace ikv
