// H_W(mu) = gamma5 D_W(mu) (Sec. 1 of the paper) in FP64, eight lanes per site and field: one
// lane per hop (direction nu = 0..3, forward or backward).
//
// What bounds it: the FP64 pipe.  An SM executes two FP64 operations per cycle, half a one in each
// of its four sub-partitions, so a warp's FP64 instruction takes 64 cycles of its sub-partition
// whatever its active lanes, and a site costs about 900 of them.  With a thread per site a 4^4
// lattice is eight warps of 900; with a lane per hop it is 64 warps of 114.  Measured, us per
// launch, thread per site -> lane per hop: 4^4 x 1 field 31.3 -> 6.5, 6^4 x 1 32.5 -> 6.8,
// 7x6x9x8 x 3 32.8 -> 18.9, 10^4 x 12 206 -> 189 (FP64 pipe 92 % busy), where natural-order
// fields also save the 24 us of packing and unpacking.  A row of the link per warp (45 instructions)
// took the 4^4 solve from 5.80 to 4.69 ms (361 of its 1,000 launches are stencils).
#include "hops.cuh"

namespace sgn {

cudaError_t launch_hw_f64(double2* out, const double2* in, const double2* U, int nrhs, const StencilParams& p,
                          const int* skip, cudaStream_t st, bool nat) {
    // a row of the link per warp where that shortens the busiest sub-partition's work: 45 FP64
    // instructions for each of three times the warps, against 111
    const int64_t warps = (p.vol + 3) / 4 * nrhs, pipes = 4 * 152;
    if (45 * ((3 * warps + pipes - 1) / pipes) < 111 * ((warps + pipes - 1) / pipes))
        return hops::launch<double, double2, true>(out, in, U, nrhs, p, skip, st, nat);
    return hops::launch<double, double2, false>(out, in, U, nrhs, p, skip, st, nat);
}

}  // namespace sgn
