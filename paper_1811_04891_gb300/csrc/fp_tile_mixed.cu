// fp_tile_mixed.cu -- the mixed form's tile kernels, for n = FP_N GLL points
// per direction.  Compiled without contraction of separate multiplies and
// adds: a pair takes the same steps in k_newton_tile<n, TILE_MIXED> and in
// the TILE_PHASE32 / TILE_FINAL sequence, and with every fused multiply-add
// written out the kernels round alike, so that a find's results do not depend
// on how many points share the call.  (1 % of the time; the FP64 form has one
// kernel for both passes and keeps contraction.)  The digits' layout is here
// too: fragments made on the fly are to have its bits.
#include "fp_common.cuh"
#include "fp_internal.h"
#include "fp_tile_launch.cuh"

#ifndef FP_N
#error "FP_N: GLL points per direction"
#endif

namespace fpg {

#define FP_CAT2(a, b) a##b
#define FP_CAT(a, b) FP_CAT2(a, b)

cudaError_t FP_CAT(newton_tile_mixed_, FP_N)(const FindArgs& a, const NewtonArgs& na, int64_t npairs, const BasisTab& tab,
                                             int block, unsigned grid, cudaStream_t s)
{
    return newton_tile<FP_N, true>(a, na, npairs, tab, block, grid, s);
}

cudaError_t FP_CAT(digits_mixed_, FP_N)(int64_t E, const double* coords, ElemBox* boxes, unsigned char* dig,
                                        const BasisTab& tab, cudaStream_t s)
{
    return digits_form<FP_N, true>(E, coords, boxes, dig, tab, s);
}

int FP_CAT(tile_fit_mixed_, FP_N)(int block) { return tile_fit<FP_N, TILE_MIXED>(block); }

}  // namespace fpg
