// Where a selection over arrays reads its configs from: the distinct metric arrays a call touches,
// the bound that goes with each, and the order-preserving keys made of them.  Shared by the
// one-launch kernels over materialised metrics (select_coop.cu) and by the fused form's kernels over
// its compact sample (select_stream.cu).
#pragma once
#include "select_sink.cuh"

namespace guide {

static constexpr u32 ROW = 64;                  // configs per warp-wide load (32 lanes x 2)
static constexpr int MAX_ARR = 6;               // distinct arrays a call can touch

// one metric array with the role it plays in this call
struct Arr {
    const double *p;
    double bound;
    int cmp;          // 0: no bound, 1: value <= bound, 2: value >= bound
    int neg;          // used as a metric through its negation (throughput)
};

__device__ __forceinline__ bool within(const Arr &a, double v) {
    // no bound, value <= bound, or value >= bound; written so that a NaN fails an active bound
    return a.cmp == 0 || (a.cmp == 1 ? v <= a.bound : v >= a.bound);
}

__device__ __forceinline__ u64 metric_key(const Arr &a, double v) { return enc(a.neg ? 0.0 - v : v); }

__device__ __forceinline__ void pair_min(u64 &key, u64 &idx, u64 okey, u64 oidx) {
    if (okey < key || (okey == key && oidx < idx)) { key = okey; idx = oidx; }
}

}  // namespace guide
