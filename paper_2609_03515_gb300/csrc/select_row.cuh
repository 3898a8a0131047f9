// Budgeted selection of one utility row, by a CTA or by a cluster of CTAs that share the row;
// used by the select kernel and by the score pass, whose last CTA of a row selects that row
// at once.  See select.cu.
#pragma once
#include "ikv_internal.cuh"

namespace ikv {
namespace {

__device__ __forceinline__ uint32_t ord_key(float f) {
    uint32_t u = __float_as_uint(f);
    if ((u & 0x7FFFFFFFu) > 0x7F800000u) return 1u;  // NaN: below every number (-inf maps to 0x007FFFFF)
    if ((u & 0x7FFFFFFFu) == 0u) u = 0u;              // -0.0 == +0.0
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
constexpr uint32_t kDeadKey = 0u;  // dead slots: below every live key, never kept

// thread-block cluster: barrier over every thread of the cluster (release / acquire), and
// loads from the shared memory of the cluster's CTA `rank` at the address of `p` in this one
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t cluster_addr(const void *p, int rank) {
    uint32_t ra;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;"
                 : "=r"(ra)
                 : "r"(static_cast<uint32_t>(__cvta_generic_to_shared(p))), "r"(rank));
    return ra;
}
__device__ __forceinline__ float ld_cluster(const float *p, int rank) {
    float v;
    asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(cluster_addr(p, rank)) : "memory");
    return v;
}
__device__ __forceinline__ uint32_t ld_cluster(const uint32_t *p, int rank) {
    uint32_t v;
    asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(cluster_addr(p, rank)) : "memory");
    return v;
}
__device__ __forceinline__ unsigned long long ld_cluster(const unsigned long long *p, int rank) {
    unsigned long long v;
    asm volatile("ld.shared::cluster.u64 %0, [%1];" : "=l"(v) : "r"(cluster_addr(p, rank)) : "memory");
    return v;
}

constexpr int kSelMaxCtas = 8;  // CTAs that share a row (portable cluster size)

constexpr int kSelSlots = 3072;  // slots a CTA should have to be worth a cluster's barriers

// The selection of utility row r by a CTA of NT threads (CL false), or by up to `ctas` CTAs of a
// cluster, of which this one is the `rank`-th (CL), entered by all of their threads.  CTA `rank`
// owns a contiguous share of the row's slots and keeps their keys in keys[0, keys_cap) (shared
// memory) when they fit; otherwise every sweep reads the row again, a few loads in flight a
// thread.  L: the row's slots in use.  A row too short for the whole cluster is shared by fewer of
// its CTAs, down to one, and the others leave (a cluster barrier waits for no thread that has).
template <int NT, bool CL>
__device__ __forceinline__ void select_row(int rank, int ctas, int r, int L, int32_t cap, const float *util, int32_t rps,
                                           const int32_t *__restrict__ budget, int32_t *pos, int32_t *keep,
                                           int32_t *keep_len, DeferArgs df, uint32_t *keys, int keys_cap) {
    static_assert(NT % 32 == 0 && NT <= 1024, "whole warps");
    constexpr int NW = NT / 32;
    constexpr int U = NT == 256 ? 4 : 8;  // keys a thread has in flight
    constexpr int DT = NT < 256 ? NT : 256;                   // threads of the digit scan,
    constexpr int DPT = (256 + DT - 1) / DT;                  // and the digits each of them holds
    static_assert(DT % 32 == 0, "whole warps");
    __shared__ uint32_t hist[2][256];
    __shared__ uint32_t warp_a[NW], warp_b[NW];
    __shared__ unsigned long long warp_min[NW], s_min;
    __shared__ uint32_t s_digit, s_above, s_live, s_gt, s_eq;
    __shared__ bool s_whole;

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int b = r / rps;
    const int B = max(budget[b], 0);
    const int S = df.start ? df.start[b] : 0;
    const int C = CL ? max(1, min(ctas, L / kSelSlots)) : 1;
    if (CL && rank >= C) return;
    const int seg = (L + C - 1) / C;
    const int lo = min(rank * seg, L), hi = min(lo + seg, L);
    const bool cached = hi - lo <= keys_cap;
    const float *u = util + (int64_t)r * cap;
    int32_t *pr = pos ? pos + (int64_t)r * cap : nullptr;
    int32_t *kp = keep + (int64_t)r * cap;
    // (through L2: in the score pass other CTAs of the same launch wrote the utilities)
    // slots i0, i0 + step, ... : their keys from the row, kDeadKey from `end` on (those load the last
    // slot: with a branch around each load they went out one by one, 2.2 us a batch of eight)
    auto load_keys = [&](int i0, int step, int end, uint32_t (&key)[U]) {
        float x[U];
        int32_t p[U];
#pragma unroll
        for (int k = 0; k < U; ++k) x[k] = __ldcg(u + min(i0 + k * step, end - 1));
        if (pr) {
#pragma unroll
            for (int k = 0; k < U; ++k) p[k] = __ldcg(pr + min(i0 + k * step, end - 1));
        } else {
#pragma unroll
            for (int k = 0; k < U; ++k) p[k] = 0;
        }
#pragma unroll
        for (int k = 0; k < U; ++k) key[k] = i0 + k * step < end && p[k] >= 0 ? ord_key(x[k]) : kDeadKey;
    };
    // the same, from shared memory when they are there
    auto get_keys = [&](int i0, int step, int end, uint32_t (&key)[U]) {
        if (cached) {
#pragma unroll
            for (int k = 0; k < U; ++k) key[k] = i0 + k * step < end ? keys[i0 + k * step - lo] : kDeadKey;
        } else {
            load_keys(i0, step, end, key);
        }
    };
    auto sync_all = [&]() {
        if (CL && C > 1) cluster_sync();
        else __syncthreads();
    };
    auto peer = [&](const auto *p, int c) { return CL && C > 1 ? ld_cluster(p, c) : *p; };
    constexpr int kPeers = CL ? kSelMaxCtas : 1;

    // one sweep: the live count and the lowest (key, highest slot) among the live slots,
    // which is the victim whenever exactly one slot must go
    uint32_t cnt = 0u;
    unsigned long long best = ~0ull;
    for (int i0 = lo + tid; i0 < hi; i0 += NT * U) {
        uint32_t key[U];
        load_keys(i0, NT, hi, key);
#pragma unroll
        for (int k = 0; k < U; ++k) {
            const int i = i0 + k * NT;
            if (cached && i < hi) keys[i - lo] = key[k];
            if (key[k] == kDeadKey) continue;
            ++cnt;
            const unsigned long long v = ((unsigned long long)key[k] << 32) | (uint32_t)(~(uint32_t)i);
            best = v < best ? v : best;
        }
    }
    for (int i = tid; i < 512; i += NT) (&hist[0][0])[i] = 0u;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long y = __shfl_xor_sync(0xffffffffu, best, o);
        best = y < best ? y : best;
        cnt += __shfl_xor_sync(0xffffffffu, cnt, o);
    }
    if (lane == 0) {
        warp_min[warp] = best;
        warp_a[warp] = cnt;
    }
    __syncthreads();
    if (warp == 0) {
        best = lane < NW ? warp_min[lane] : ~0ull;
        cnt = lane < NW ? warp_a[lane] : 0u;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const unsigned long long y = __shfl_xor_sync(0xffffffffu, best, o);
            best = y < best ? y : best;
            cnt += __shfl_xor_sync(0xffffffffu, cnt, o);
        }
        if (lane == 0) {
            s_min = best;
            s_live = cnt;
        }
    }
    sync_all();
    // (remote loads are issued together, here and below: one round trip, not C)
    int n_live = 0;
    best = ~0ull;
    {
        uint32_t live[kPeers];
        unsigned long long low[kPeers];
#pragma unroll
        for (int c = 0; c < kPeers; ++c) {
            live[c] = c < C ? peer(&s_live, c) : 0u;
            low[c] = c < C ? peer(&s_min, c) : ~0ull;
        }
#pragma unroll
        for (int c = 0; c < kPeers; ++c) {
            n_live += (int)live[c];
            best = low[c] < best ? low[c] : best;
        }
    }
    const int kept = min(n_live, B);
    if (n_live == B + 1 && B > 0 && pr && df.max_holes > 0 && L - B <= df.max_holes && S + L < df.cap) {
        // deferred compaction (the rule the compaction kernels apply): the victim is
        // only marked dead, and keep_len < 0 tells compaction that nothing moves
        if (rank == 0 && tid == 0) {
            const int ev = (int)(~(uint32_t)(best & 0xFFFFFFFFull));
            if (df.later) kp[0] = ev;
            else pr[ev] = -1;
            keep_len[r] = -1 - B;
        }
        if (CL && C > 1) cluster_sync();  // a CTA may not leave while another reads its shared memory
        return;
    }
    if (rank == 0 && tid == 0) keep_len[r] = kept;
    if (n_live == L && kept >= L - 1) {  // no dead slot, at most one to go: no counting needed
        const int ev = kept == L ? L : (int)(~(uint32_t)(best & 0xFFFFFFFFull));
        if (kept > 0)
            for (int i = lo + tid; i < hi; i += NT)
                if (i != ev) kp[i < ev ? i : i - 1] = i;
    } else if (kept > 0) {
        // theta: the kept-th largest key.  Everything above it is kept, and of the slots equal
        // to it the lowest ones.  All live slots kept: every live key is above the dead one.
        // One slot too many: the lowest live key.
        uint32_t theta = n_live <= B ? kDeadKey : (uint32_t)(best >> 32);
        if (n_live > B + 1) {
            // MSB-first radix select on the keys (dead slots carry the lowest one, and more than
            // B live keys lie above it, so theta is live and no dead slot is ever kept).  The
            // CTAs' histograms are summed by every CTA; two buffers, one barrier a digit.
            uint32_t prefix = 0u, mask = 0u, k = (uint32_t)B;
#pragma unroll 1
            for (int pass = 0; pass < 4; ++pass) {
                const int shift = 24 - 8 * pass;
                uint32_t *h = hist[pass & 1];
                for (int i0 = lo + tid; i0 < hi; i0 += NT * U) {
                    uint32_t key[U];
                    get_keys(i0, NT, hi, key);
#pragma unroll
                    for (int q = 0; q < U; ++q)
                        if (i0 + q * NT < hi && (key[q] & mask) == prefix) atomicAdd(&h[(key[q] >> shift) & 0xFFu], 1u);
                }
                sync_all();
                // (every CTA is past its reads of the other buffer)
                // inclusive counts from the top digit down: thread t holds digits from 255 - t DPT down
                uint32_t v[DPT], x = 0u;
                if (tid < DT) {
#pragma unroll
                    for (int q = 0; q < DPT; ++q) {
                        const int d = 255 - (tid * DPT + q);
                        v[q] = 0u;
                        if (d < 0) continue;
                        hist[(pass & 1) ^ 1][d] = 0u;
                        uint32_t w[kPeers];
#pragma unroll
                        for (int c = 0; c < kPeers; ++c) w[c] = c < C ? peer(&h[d], c) : 0u;
#pragma unroll
                        for (int c = 0; c < kPeers; ++c) v[q] += w[c];
                        x += v[q];
                    }
#pragma unroll
                    for (int o = 1; o < 32; o <<= 1) {
                        const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
                        if (lane >= o) x += y;
                    }
                    if (lane == 31) warp_a[warp] = x;
                }
                __syncthreads();
                if (tid < DT) {
                    uint32_t incl = x;
                    for (int w = 0; w < warp; ++w) incl += warp_a[w];
#pragma unroll
                    for (int q = DPT - 1; q >= 0; --q) {  // incl: through digit q of the thread's
                        if (incl - v[q] < k && incl >= k) {  // exactly one digit satisfies this
                            s_digit = 255u - (uint32_t)(tid * DPT + q);
                            s_above = incl - v[q];
                            s_whole = incl == k;
                        }
                        incl -= v[q];
                    }
                }
                __syncthreads();
                k -= s_above;
                prefix |= s_digit << shift;
                mask |= 0xFFu << shift;
                // every key of the digit's bin is kept (short rows: after two digits, as a rule):
                // the cut runs just below the bin, the remaining digits do not matter
                if (s_whole && prefix != 0u) {
                    prefix -= 1u;
                    break;
                }
            }
            theta = prefix;
        }
        // each warp owns a contiguous part of the segment: its counts above and at theta, the
        // counts before it, then its kept slots in ascending order
        const int part = (seg + NT - 1) / NT * 32;
        const int wlo = min(lo + warp * part, hi), whi = min(wlo + part, hi);
        uint32_t gt = 0u, eq = 0u;
        for (int i0 = wlo + lane; i0 < whi; i0 += 32 * U) {
            uint32_t key[U];
            get_keys(i0, 32, whi, key);
#pragma unroll
            for (int q = 0; q < U; ++q) {
                gt += key[q] > theta;
                eq += key[q] == theta && key[q] != kDeadKey;
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            gt += __shfl_xor_sync(0xffffffffu, gt, o);
            eq += __shfl_xor_sync(0xffffffffu, eq, o);
        }
        __syncthreads();  // warp_a is free
        if (lane == 0) {
            warp_a[warp] = gt;
            warp_b[warp] = eq;
        }
        __syncthreads();
        if (warp == 0) {  // exclusive over the warps
            uint32_t g = lane < NW ? warp_a[lane] : 0u, e = lane < NW ? warp_b[lane] : 0u;
            const uint32_t g0 = g, e0 = e;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t yg = __shfl_up_sync(0xffffffffu, g, o), ye = __shfl_up_sync(0xffffffffu, e, o);
                if (lane >= o) {
                    g += yg;
                    e += ye;
                }
            }
            if (lane < NW) {
                warp_a[lane] = g - g0;
                warp_b[lane] = e - e0;
            }
            if (lane == NW - 1) {
                s_gt = g;
                s_eq = e;
            }
        }
        sync_all();
        uint32_t gt_all = 0u, gt_run = warp_a[warp], eq_run = warp_b[warp];
        {
            uint32_t g[kPeers], e[kPeers];
#pragma unroll
            for (int c = 0; c < kPeers; ++c) {
                g[c] = c < C ? peer(&s_gt, c) : 0u;
                e[c] = c < C ? peer(&s_eq, c) : 0u;
            }
#pragma unroll
            for (int c = 0; c < kPeers; ++c) {
                gt_all += g[c];
                if (c < rank) {
                    gt_run += g[c];
                    eq_run += e[c];
                }
            }
        }
        const uint32_t need_eq = (uint32_t)kept - gt_all;  // theta-valued slots that survive
        const uint32_t below = (1u << lane) - 1u;
        for (int i0 = wlo; i0 < whi; i0 += 32 * U) {
            uint32_t key[U];
            get_keys(i0 + lane, 32, whi, key);
#pragma unroll
            for (int q = 0; q < U; ++q) {
                if (i0 + 32 * q >= whi) break;
                const bool is_gt = key[q] > theta, is_eq = key[q] == theta && key[q] != kDeadKey;
                const uint32_t mg = __ballot_sync(0xffffffffu, is_gt), me = __ballot_sync(0xffffffffu, is_eq);
                const uint32_t e = eq_run + __popc(me & below);
                if (is_gt || (is_eq && e < need_eq))
                    kp[gt_run + __popc(mg & below) + min(e, need_eq)] = i0 + 32 * q + lane;
                gt_run += __popc(mg);
                eq_run += __popc(me);
            }
        }
    }
    if (CL && C > 1) cluster_sync();  // a CTA may not leave while another reads its shared memory
}

}  // namespace
}  // namespace ikv
