// Hand-written FFT stages (the F, F^dagger of Eq. 2 and the padded
// convolutions of the minor cycles): tables and the pieces shared by the row
// and column passes (k_fft_rows_*.cu, k_fft_cols_*.cu; fft_engine.cuh).
//
// Every transform maps between a real M x M image, centred on an L x L grid
// (L = M or 2 M; pixel offset a' = a - M/2 sits at grid index a' mod L,
// multiplied by (-1)^(a'+b') so that spectrum index j holds frequency
// j - L/2), and the window [lo, lo + S)^2 of its spectrum, stored u-major:
// spec[ju][jv].  A 2D transform is two passes over HBM:
//   rows    a CTA transforms a batch of image rows and writes the window
//           columns only, transposed (T);
//   columns a CTA transforms a batch of window columns and writes the window
//           rows contiguously.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <vector>

#include "rix_internal.cuh"
#include "fft_engine.cuh"

namespace rix {
namespace {

// screen[p][pix] = corr[pix] * exp(-2 pi i (w0 + p dw) nm1[pix]), formed as
// the row passes form it (wscreen).  n - 1 and corr are even in both
// coordinates: one thread per quadrant pixel of a plane forms the phase (FP64)
// once for the up to four pixels that share it.
template <typename R>
__global__ void k_screen_table(int M, int nplanes, double w0, double dw, const R* __restrict__ corr,
                               const double* __restrict__ nm1, cplx<R>* __restrict__ screen) {
  const int h = M / 2;
  const int64_t q = (int64_t)(h + 1) * (h + 1), npix = (int64_t)M * M;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < q * nplanes;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int p = (int)(i / q);
    const int r = (int)(i - p * q), b = r / (h + 1), c = r - b * (h + 1);
    const int64_t pix = (int64_t)b * M + c;
    const cplx<R> e = wscreen<R, -1>(w0 + p * dw, nm1[pix]);
    const R f = corr[pix];
    const cplx<R> z = cmake<cplx<R>>(e.x * f, e.y * f);
    cplx<R>* s = screen + p * npix;
    const int bm = M - b, cm = M - c;     // the mirrors of h - b and h - c
    const bool mb = b > 0 && b < h, mc = c > 0 && c < h;
    s[pix] = z;
    if (mc) s[(int64_t)b * M + cm] = z;
    if (mb) s[(int64_t)bm * M + c] = z;
    if (mb && mc) s[(int64_t)bm * M + cm] = z;
  }
}

// img = (accumulate ? img : 0) + sum over g < G of part[g]
template <typename R>
__global__ void k_sum_groups(R* __restrict__ img, const R* __restrict__ part, int G, int64_t n, int accumulate) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    R v = accumulate ? img[i] : R(0);
    for (int g = 0; g < G; ++g) v += part[(int64_t)g * n + i];
    img[i] = v;
  }
}

}  // namespace

template <typename R>
int fft_max_len() {
  return 1 << kMaxLogL<R>;
}
template int fft_max_len<float>();
template int fft_max_len<double>();

// roots of every power of two up to kTwMax: exp(-2 pi i k / 2^j) at 2^j + k
int fft_init_twiddles(Ctx* ctx) {
  std::vector<double2> t64(2 * kTwMax);
  std::vector<float2> t32(2 * kTwMax);
  for (int j = 0; j <= kTwLog; ++j)
    for (int k = 0; k < (1 << j); ++k) {
      const double ang = 2.0 * M_PI * (double)((int64_t)k << (kTwLog - j)) / (double)kTwMax;
      t64[(1 << j) + k] = make_double2(std::cos(ang), -std::sin(ang));
      t32[(1 << j) + k] = make_float2((float)t64[(1 << j) + k].x, (float)t64[(1 << j) + k].y);
    }
  RIX_TRY(ctx->tw64.alloc(ctx, 2 * kTwMax * sizeof(double2)));
  RIX_TRY(ctx->tw32.alloc(ctx, 2 * kTwMax * sizeof(float2)));
  RIX_CUDA(cudaMemcpy(ctx->tw64.p, t64.data(), 2 * kTwMax * sizeof(double2), cudaMemcpyHostToDevice));
  RIX_CUDA(cudaMemcpy(ctx->tw32.p, t32.data(), 2 * kTwMax * sizeof(float2), cudaMemcpyHostToDevice));
  return RIX_OK;
}

template <typename R>
int build_screen_table(const Ctx* ctx, const XformGeom& g, cplx<R>* screen, cudaStream_t st) {
  if (g.mode != kFacPhase || !g.corr || !g.nm1 || g.M <= 0 || g.nplanes <= 0)
    return set_error(RIX_EINVAL, "screen table needs a w-stacked geometry");
  const int64_t npix = (int64_t)g.M * g.M;
  const int blocks = (int)std::min<int64_t>(ceil_div(npix * g.nplanes, 4 * 256), (int64_t)ctx->num_sms * 16);
  ::rix::note_launch();
  k_screen_table<R><<<blocks, 256, 0, st>>>(g.M, g.nplanes, g.w0, g.dw, static_cast<const R*>(g.corr), g.nm1,
                                            screen);
  RIX_LAUNCH_CHECK();
  return RIX_OK;
}
template <typename R>
int sum_groups(const Ctx* ctx, R* img, const R* parts, int G, int64_t n, int accumulate, cudaStream_t st) {
  ::rix::note_launch();
  k_sum_groups<R><<<(int)std::min<int64_t>(ceil_div(n, 256), (int64_t)ctx->num_sms * 8), 256, 0, st>>>(
      img, parts, G, n, accumulate);
  RIX_LAUNCH_CHECK();
  return RIX_OK;
}

#define RIX_FFT_INST(R)                                                                              \
  template int build_screen_table<R>(const Ctx*, const XformGeom&, cplx<R>*, cudaStream_t);           \
  template int sum_groups<R>(const Ctx*, R*, const R*, int, int64_t, int, cudaStream_t);
RIX_FFT_INST(float)
RIX_FFT_INST(double)

}  // namespace rix
