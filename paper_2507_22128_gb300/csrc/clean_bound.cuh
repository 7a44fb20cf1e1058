// Rules of the ms-CLEAN loops (k_minor.cu): which of them a call takes, its CTAs,
// and the lower bound of the next peak that the cleaned peak itself leaves.  Plain
// C++, so that they can be checked on the host.
#pragma once

#include <cstdint>

#ifdef __CUDACC__
#define RIX_CLEAN_FN __host__ __device__ __forceinline__
#else
#define RIX_CLEAN_FN inline
#endif

namespace rix {

// The lower bound: a tile whose bound from above lies below it is not updated.  A
// peak of candidate value v, cleaned with `gain`, keeps (1 - gain) v up to the
// rounding of amp = gain R / P and of R - amp P, a few 2^-24 of v itself: no
// longer small beside the remainder when the gain is near 1.  Negative there,
// which bounds nothing and updates every tile.
RIX_CLEAN_FN float clean_keep(float v, double gain) { return v * (float)((1.0 - gain) * 0.9999 - 1e-6); }

// Whether a minor cycle updates its tiles lazily (k_msclean) or all at every
// iteration (k_msclean_sweep).  The lazy form's bounds, and the candidates of a few
// long tiles instead of a pixel per thread, cost about two microseconds per
// iteration, which it earns back where a sweep is bound by memory.  Microseconds
// per iteration, lazy / sweep, one and three scales: FP32 512^2 7.4 / 5.1 and 9.2 /
// 6.1, 1024^2 11.0 / 8.1 and 13.4 / 10.7, 2048^2 18.3 / 15.5 and 25 / 34 (two
// scales 21 / 25), 4096^2 one and four 48 / 79 and 85 / 201; FP64 256^2 9.3 / 6.0
// and 10.3 / 6.6, 512^2 11.0 / 7.9 and 14.8 / 10.3, 1024^2 17.8 / 13.5 and 24.1 /
// 22.7, 2048^2 28 / 35 and 49 / 72.
inline bool clean_lazy(bool fp64, int n, int ns) { return n > 2048 || (n == 2048 && (fp64 || ns > 1)); }

// CTAs per SM of the loop, at most: two for a sweep, which leave room for another
// partition's or job's loop and make the barrier cheaper, four where it is bound
// by memory and wants the loads in flight, and for the lazy form.  Two / four,
// microseconds per iteration of one loop and of two jobs' at once, three scales:
// FP64 512^2 10.3 / 13.2 and 17.8 / 26.4, 1024^2 22.7 / 24.8 and 43 / 50; FP32 512^2
// 6.1 / 7.0 and 12.3 / 14.1, 1024^2 11.8 / 10.7; one scale at 1024^2 8.1 / 8.3, at
// 2048^2 22.3 / 15.8; FP64 1024^2 with four scales 28.2 / 28.9, with six 46 / 37.
inline int clean_ctas_per_sm(bool fp64, int n, int ns, bool lazy) {
  return lazy || (int64_t)n * n * ns >= (int64_t)(fp64 ? 5 : 2) * 1024 * 1024 ? 4 : 2;
}

}  // namespace rix
