// The end of a CTA's fixed-order FP64 sum: one value per thread, in shared memory.
#pragma once

namespace evx {

// Sum of red[0 .. n) (n >= 1, a value per thread of a CTA of n threads), for the threads
// tid < min(n, 32); thread 0 gets it. A CTA may have fewer than 32 threads (the z passes
// shrink theirs while a grid is short): then only those lanes exist and only they shuffle.
__device__ __forceinline__ double first_warp_sum(const double* red, int n, int tid) {
    const int live = n < 32 ? n : 32;
    const unsigned lanes = live == 32 ? 0xffffffffu : (1u << live) - 1u;
    double t = 0.0;
    for (int i = tid; i < n; i += 32) t += red[i];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const double u = __shfl_down_sync(lanes, t, o);
        if (tid + o < live) t += u;
    }
    return t;
}

}  // namespace evx
