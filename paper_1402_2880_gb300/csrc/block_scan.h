// Exclusive sum of one int per thread over a CTA.
#pragma once

namespace sscf {

// Two shuffle scans and two barriers, for whole warps (one thread adding up the
// CTA's counts in shared memory took 7 us of the 10.8 of the closure's labels, 1024
// threads). part: 33 ints of shared memory, in use by nothing else; part[32] is the
// total afterwards.
__device__ __forceinline__ int block_scan(int v, int* part) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, n_warps = blockDim.x >> 5;
    int inc = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += u;
    }
    if (lane == 31) part[warp] = inc;
    __syncthreads();
    if (warp == 0) {
        const int c = lane < n_warps ? part[lane] : 0;
        int run = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int u = __shfl_up_sync(0xffffffffu, run, o);
            if (lane >= o) run += u;
        }
        part[lane] = run - c;
        if (lane == 31) part[32] = run;
    }
    __syncthreads();
    return inc - v + part[warp];
}

}  // namespace sscf
