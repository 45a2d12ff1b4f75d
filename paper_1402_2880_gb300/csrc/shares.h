// Sums over all atom pairs of a cluster, split for the FP64 pipe: one warp takes
// 32 atoms (blockIdx.x) and share blockIdx.y of gridDim.y of the atoms they
// couple to; the shares are added in order afterwards.
#pragma once

namespace sscf {

// atoms of a share (at least) and shares (at most). A warp's FP64 instructions take 64 clocks each
// whatever else its quarter of an SM does, so small clusters are spread thin (648 atoms, shares of 64
// and of 16: 48 and 21 us)
constexpr int kShareAtoms = 16;
constexpr int kMaxShares = 64;

// the atoms [b0, b1) of this CTA's share of [lo, hi)
__device__ __forceinline__ void share_range(int lo, int hi, int& b0, int& b1) {
    const int per = (hi - lo + (int)gridDim.y - 1) / (int)gridDim.y;
    b0 = min(hi, lo + (int)blockIdx.y * per);
    b1 = min(hi, b0 + per);
}

}  // namespace sscf
