// Budgeted selection: keep the B highest utilities of a row (Sec. 3: evict the
// lowest m whenever the cache exceeds B).
//
// A row is taken by one CTA of 256 to 1024 threads, or shared by a cluster of up to eight of 512,
// which load it once and keep its keys in shared memory.  Utilities map to order-preserving
// 32-bit keys (sign-flipped IEEE bits; -0.0 folded onto +0.0; NaN -> 1, below
// every number).  Dead slots (pos < 0, deferred compaction) get key 0: below
// every live key, never kept, not counted against B.  General case: an
// MSB-first radix select with 8-bit digits (four passes over the keys, shared-memory
// histograms, summed across the cluster through distributed shared memory)
// finds the exact B-th largest key theta; one more sweep writes the kept slots in
// ascending order (per-warp ballots after one exchange of counts), keeping the lowest
// slots among keys equal to theta.  Steady-state case, one live slot too many:
// the first sweep finds theta, the lowest key, itself (among equal keys the
// highest slot goes).  The result depends only on the fp32 values, so it is
// bit-exact against any correct sort.
//
// Bound by latency, not by the few hundred kilobytes it touches: a chain of barriers.  One
// 1024-thread CTA a row, re-reading the row from L2 in every pass and scanning twice per 1024
// slots, took 41 us for 32 rows of 16385 slots and 124 us for one of 32769; clusters of four and
// eight take 15 us.  A row's CTAs follow its length, not its capacity, as many as have 3072 slots
// each (one row of 3277 slots in 33024: 4.4 us with eight CTAs, 3.7 with one; of 16384: 4.7
// with five), and a launch takes no more CTAs than SMs (32 rows of 16384 slots with four CTAs each
// 4.9 us, with eight 7.3; 128 rows of 8000 with one 4.6, with two 6.9).
#include "select_row.cuh"

namespace ikv {
namespace {

constexpr int kSelKeysMax = 48 * 1024;  // keys a CTA keeps in shared memory

template <int NT, bool CL>
__global__ void __launch_bounds__(NT, NT == 1024 ? 1 : 2)
    select_kernel(int32_t cap, const float *util, const int32_t *__restrict__ len, int32_t rps,
                  const int32_t *__restrict__ budget, int32_t *pos, int32_t *keep, int32_t *keep_len, DeferArgs df,
                  int32_t ctas, int32_t keys_cap) {
    extern __shared__ uint32_t keys[];
    pdl_wait();
    const int r = CL ? blockIdx.x / ctas : blockIdx.x;
    select_row<NT, CL>(CL ? blockIdx.x % ctas : 0, ctas, r, len[r / rps], cap, util, rps, budget, pos, keep, keep_len,
                       df, keys, keys_cap);
}

}  // namespace

SelectPlan select_plan(int64_t rows, int32_t max_len, int sms) {
    SelectPlan p;
    // the largest cluster that leaves every CTA some slots of the longest row and every CTA an SM
    int C = kSelMaxCtas;
    while (C > 1 && (rows * C > sms || (int64_t)C * kSelSlots > max_len)) C >>= 1;
    const int seg = (max_len + C - 1) / C;
    p.ctas = C;
    // threads for about one batch of eight keys each: more warps would issue the same predicated
    // batches for nothing (one row of 1096 slots: 14.3 us with 1024 threads, 8.2 with 256)
    p.threads = C == 1 && seg <= 2048 ? 256 : C > 1 || seg <= 4608 ? 512 : 1024;
    // (shorter rows of the launch have fewer CTAs, of up to twice kSelSlots slots each)
    const int keys = C > 1 && seg < 2 * kSelSlots ? 2 * kSelSlots : seg;
    p.keys = keys < kSelKeysMax ? keys : kSelKeysMax;
    return p;
}

cudaError_t launch_select(int32_t rows, int32_t cap, int32_t max_len, const float *util, const int32_t *len,
                          int32_t rows_per_seq, const int32_t *budget, int32_t *pos, int32_t *keep, int32_t *keep_len,
                          const DeferArgs &df, int sms, cudaStream_t st) {
    if (rows <= 0) return cudaSuccess;
    const SelectPlan p = select_plan(rows, max_len, sms);
    const int C = p.ctas, nt = p.threads;
    auto kernel = C > 1          ? select_kernel<512, true>
                  : nt == 256    ? select_kernel<256, false>
                  : nt == 512    ? select_kernel<512, false>
                                 : select_kernel<1024, false>;
    const size_t smem = (size_t)p.keys * sizeof(uint32_t);
    // the limit is the process's, so every call writes the same value: with a call's own size, a
    // small selection on another thread could lower it between this and the launch
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         kSelKeysMax * (int)sizeof(uint32_t));
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)C * (unsigned)rows);
    cfg.blockDim = dim3(nt);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    int n = 0;
    if (C > 1) {
        attr[n].id = cudaLaunchAttributeClusterDimension;
        attr[n].val.clusterDim.x = C;
        attr[n].val.clusterDim.y = 1;
        attr[n].val.clusterDim.z = 1;
        ++n;
    }
    if (pdl_enabled()) {
        attr[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[n].val.programmaticStreamSerializationAllowed = 1;
        ++n;
    }
    cfg.attrs = attr;
    cfg.numAttrs = n;
    e = cudaLaunchKernelEx(&cfg, kernel, cap, util, len, rows_per_seq, budget, pos, keep, keep_len, df, C, p.keys);
    note_launch();
    return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace ikv
