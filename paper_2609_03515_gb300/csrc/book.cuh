// The bookkeeping of a step's append, done by extra CTAs of its attention launch.
#pragma once
#include "merge.cuh"
#include "select_row.cuh"

namespace ikv {
namespace {

// One CTA of NT threads appends sequence b's new token: its position, its utility (0, or the mean
// over the live slots of its row), next_pos, and len1[b] = the length with it, which the step's later
// kernels read; len[b] itself is left to the compaction, because the attention CTAs that run
// beside this one work from it (slot len[b] is the new token's, live whatever pos still says
// there).  No room: len1[b] = len[b] and bit 2 of *err.  With k.select it then selects the
// sequence's rows, hidden behind the attention (a kernel of its own after it cost 5 us a step);
// keys, keys_cap: the CTA's shared memory for their keys.
template <int NT>
__device__ __noinline__ void book_sequence(const BookArgs &k, const int32_t *len, const int32_t *start, int32_t cap,
                                           int32_t rows_per_seq, int b, unsigned int *err, uint32_t *keys, int keys_cap) {
    constexpr int NW = NT / 32, U = 8;
    __shared__ float scratch[2][NW];
    const int tid = threadIdx.x;
    const int L = len[b];
    const bool room = (start ? start[b] : 0) + L < cap;
    if (room) {
        for (int rr = 0; rr < rows_per_seq; ++rr) {
            const int64_t row = ((int64_t)b * rows_per_seq + rr) * cap;
            float init = 0.f;
            if (k.init_mean && L > 0) {
                float s = 0.f, c = 0.f;
                for (int i0 = tid; i0 < L; i0 += NT * U) {
                    float m[U];
                    int32_t p[U];
#pragma unroll
                    for (int u = 0; u < U; ++u) {
                        const int i = i0 + u * NT;
                        m[u] = i < L ? k.ema[row + i] : 0.f;
                        p[u] = i < L ? (k.dead_slots ? k.pos[row + i] : 0) : -1;
                    }
#pragma unroll
                    for (int u = 0; u < U; ++u)
                        if (p[u] >= 0) {  // the mean over live slots only
                            s += m[u];
                            c += 1.f;
                        }
                }
                s = warp_sum(s);
                c = warp_sum(c);
                if ((tid & 31) == 0) {
                    scratch[0][tid >> 5] = s;
                    scratch[1][tid >> 5] = c;
                }
                __syncthreads();
                s = c = 0.f;
                for (int w = 0; w < NW; ++w) {
                    s += scratch[0][w];
                    c += scratch[1][w];
                }
                __syncthreads();
                init = c > 0.f ? s / c : 0.f;
            }
            if (tid == 0) {
                k.ema[row + L] = init;
                k.pos[row + L] = k.next_pos[b];
            }
        }
    }
    if (tid == 0) {
        if (room) k.next_pos[b] += 1;
        else atomicOr(err, 4u);  // the token was not stored; ikv_device_status reports it
        k.len1[b] = L + (room ? 1 : 0);
    }
    if (!k.select) return;
    __syncthreads();  // the new token's utility and position
    for (int rr = 0; rr < rows_per_seq; ++rr) {
        select_row<NT>(0, 1, b * rows_per_seq + rr, L + (room ? 1 : 0), cap, k.ema, rows_per_seq, k.budget,
                       k.dead_slots ? k.pos : nullptr, k.keep, k.keep_len, k.df, keys, keys_cap);
        __syncthreads();  // its shared memory is reused
    }
}

}  // namespace
}  // namespace ikv
