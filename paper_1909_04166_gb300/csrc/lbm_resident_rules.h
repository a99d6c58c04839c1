// Rules of the resident step kernel (lbm_resident.cu) that need no GPU to evaluate: plain C++ that
// the kernel, its launches and the CPU tests share.
#pragma once

#ifdef __CUDACC__
#define CMLBM_RULE __host__ __device__ __forceinline__
#else
#define CMLBM_RULE inline
#endif

namespace cmlbm {

// The carry row holds what the last row of a round pushed north, planes 2, 5 and 6 of the row above
// it, which the next round, whose first row that is, copies into place while it pushes.  Two words of
// such a row come from nowhere in the round before: plane 5 of the first column beside a no-slip
// left side and plane 6 of the last one beside a no-slip right side are bounced back there by the
// row's own node, in the round of the copy, so the carry does not fill them.  (A free-slip side
// mirrors populations 6 and 5 of the row below into the same words: those are carried.)
CMLBM_RULE bool carry_fills(int plane, int column, int width, bool noslip_left, bool noslip_right)
{
    return !(noslip_left && plane == 5 && column == 0) &&
           !(noslip_right && plane == 6 && column == width - 1);
}

}  // namespace cmlbm
