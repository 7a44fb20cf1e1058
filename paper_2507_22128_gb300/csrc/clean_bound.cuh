// The lower bound of the next CLEAN peak that the cleaned peak itself leaves
// (k_msclean, k_minor.cu): a tile whose bound from above lies below it is not
// updated.  Plain C++, so that it can be checked against the loop's arithmetic on
// the host.
#pragma once

#ifdef __CUDACC__
#define RIX_CLEAN_FN __host__ __device__ __forceinline__
#else
#define RIX_CLEAN_FN inline
#endif

namespace rix {

// A peak of candidate value v, cleaned with `gain`, keeps (1 - gain) v up to the
// rounding of amp = gain R / P and of R - amp P, a few 2^-24 of v itself: no
// longer small beside the remainder when the gain is near 1.  Negative there,
// which bounds nothing and updates every tile.
RIX_CLEAN_FN float clean_keep(float v, double gain) { return v * (float)((1.0 - gain) * 0.9999 - 1e-6); }

}  // namespace rix
