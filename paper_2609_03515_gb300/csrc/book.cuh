// The bookkeeping of a step's append, done by extra CTAs of its attention launch.
#pragma once
#include "merge.cuh"
#include "select_row.cuh"

namespace ikv {
namespace {

// One CTA of NT threads appends the new token to utility row r: its position and its utility (0, or
// the mean over the row's live slots).  The last CTA of sequence b's rows counts next_pos[b] up, once
// all of them have read it, and leaves len1[b] = the length with the token, which the step's later
// kernels read; len[b] itself is left to the compaction, because the attention CTAs that run
// beside this one work from it (slot len[b] is the new token's, live whatever pos still says
// there).  No room: len1[b] = len[b] and bit 2 of *err.  With k.select it then selects the
// row, hidden behind the attention (a kernel of its own after it costs 3 us a step);
// keys, keys_cap: the CTA's shared memory for its keys.  A CTA a row: one CTA taking a
// sequence's eight rows in turn lasted longer than the attention of 3277 slots (32 layers
// 104 us a step against 69, 2 layers 68.6 against 11.9).
template <int NT>
__device__ __noinline__ void book_row(const BookArgs &k, const int32_t *len, const int32_t *start, int32_t cap,
                                      int32_t rows_per_seq, int r, unsigned int *err, uint32_t *keys, int keys_cap) {
    constexpr int NW = NT / 32, U = 8;
    __shared__ float scratch[2][NW];
    const int tid = threadIdx.x;
    const int b = r / rows_per_seq;
    const int L = len[b];
    const bool room = (start ? start[b] : 0) + L < cap;
    const int64_t row = (int64_t)r * cap;
    if (room) {
        float init = 0.f;
        if (k.init_mean && L > 0) {
            float s = 0.f, c = 0.f;
            // (slots past L load the last one and count for nothing: with a branch around the loads
            // they went out one by one, 80 us for a row of 65536 slots)
            const float *m = k.ema + row;
            const int32_t *p = k.dead_slots ? k.pos + row : nullptr;
            for (int i0 = tid; i0 < L; i0 += NT * U) {
                float x[U];
                int32_t alive[U];
#pragma unroll
                for (int u = 0; u < U; ++u) x[u] = m[min(i0 + u * NT, L - 1)];
                if (p) {
#pragma unroll
                    for (int u = 0; u < U; ++u) alive[u] = p[min(i0 + u * NT, L - 1)];
                } else {
#pragma unroll
                    for (int u = 0; u < U; ++u) alive[u] = 0;
                }
#pragma unroll
                for (int u = 0; u < U; ++u)
                    if (i0 + u * NT < L && alive[u] >= 0) {  // the mean over live slots only
                        s += x[u];
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
            init = c > 0.f ? s / c : 0.f;
        }
        if (tid == 0) {
            k.ema[row + L] = init;
            k.pos[row + L] = k.next_pos[b];
        }
    }
    if (tid == 0 && (rows_per_seq == 1 || arrive_acq_rel(k.done + b) == rows_per_seq - 1)) {
        if (rows_per_seq > 1) k.done[b] = 0;
        if (room) k.next_pos[b] += 1;
        else atomicOr(err, 4u);  // the token was not stored; ikv_device_status reports it
        k.len1[b] = L + (room ? 1 : 0);
    }
    if (!k.select) return;
    __syncthreads();  // the new token's utility and position
    select_row<NT, false>(0, 1, r, L + (room ? 1 : 0), cap, k.ema, rows_per_seq, k.budget, k.dead_slots ? k.pos : nullptr,
                   k.keep, k.keep_len, k.df, keys, keys_cap);
}

}  // namespace
}  // namespace ikv
