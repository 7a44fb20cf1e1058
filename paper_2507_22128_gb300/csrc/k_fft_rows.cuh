// The row passes (see fft_engine.cuh).
#pragma once

#include <algorithm>

#include "fft_engine.cuh"

namespace rix {

template <typename R>
int fwd_rows(const Ctx* ctx, const XformGeom& g, const R* img, cplx<R>* T, cudaStream_t st) {
  RIX_TRY(check_rows<R>(g, false));
  if constexpr (sizeof(R) == 4) {
    if (g.M != g.L)
      return with_log<kMinLogF + 1, kMaxLogL<R>>(g.logL, [&](auto ll) {
        using X = PadRows<decltype(ll)::value>;
        return x_launch<X>(k_pad_rows<decltype(ll)::value>, dim3((unsigned)ceil_div(g.M, X::NB), (unsigned)g.nplanes),
                           st, x_args(g), img, T, twiddles<R>(ctx));
      });
  }
  return with_plane_shape<R>(g, [&](auto lf, auto e) {
    using X = Xf<R, decltype(lf)::value, decltype(e)::value, false>;
    return x_launch<X>(k_fwd_rows<R, decltype(lf)::value, decltype(e)::value>,
                       dim3((unsigned)(g.M / X::NB), (unsigned)g.nplanes), st, x_args(g), img, T, twiddles<R>(ctx));
  });
}

// The planes of one row batch are summed by one CTA.  With many planes and
// few row batches the grid ends in a nearly empty wave; split the planes into
// G groups (grid rows) when that takes fewer plane-transforms per SM slot,
// each group summing into its own image, and add the G images after.  At most
// max_groups groups (a divisor of the plane count).
template <typename R>
int inv_rows_groups(const Ctx* ctx, const XformGeom& g, int max_groups) {
  const int P = g.nplanes;
  if (P <= 1 || max_groups <= 1) return 1;
  auto pick = [&](auto kern, int threads, size_t smem, int nb) -> int {
    if (smem > 48 * 1024) RIX_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    int per_sm = 0;
    RIX_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, threads, smem));
    const int64_t slots = (int64_t)ctx->num_sms * std::max(per_sm, 1);
    const int64_t rowb = g.M / nb;
    double best = 1e300;
    int G = 1;
    for (int c = 1; c <= P && c <= 16 && c <= max_groups; c *= 2) {
      if (P % c) continue;
      const double cost = (double)ceil_div(rowb * c, slots) * (P / c) + 0.1 * c;   // + the group sum
      if (cost < best) { best = cost; G = c; }
    }
    return G;
  };
  if constexpr (sizeof(R) == 4) {
    if (g.M != g.L)
      return with_log<kMinLogF + 1, kMaxLogL<R>>(g.logL, [&](auto ll) {
        using X = CropRows<decltype(ll)::value>;
        return pick(k_crop_rows<decltype(ll)::value>, X::T, X::kSmem, X::NB);
      });
  }
  return with_plane_shape<R>(g, [&](auto lf, auto e) {
    using X = Xf<R, decltype(lf)::value, decltype(e)::value, false>;
    return pick(k_inv_rows<R, decltype(lf)::value, decltype(e)::value>, X::T, X::kSmem, X::NB);
  });
}

template <typename R>
int inv_rows(const Ctx* ctx, const XformGeom& g0, const cplx<R>* T, R* img, double scale, int accumulate,
             cudaStream_t st, R* group_buf, int max_groups) {
  RIX_TRY(check_rows<R>(g0, true));
  XformGeom g = g0;
  const int P = g.nplanes;
  const int G = inv_rows_groups<R>(ctx, g, max_groups < 0 ? 16 : max_groups);
  if (G < 0) return G;
  const int64_t n = (int64_t)g.M * g.M;
  // the group images: the caller's buffer, else a stream-ordered temporary
  // released on every way out
  struct StreamFree {
    void* p = nullptr;
    cudaStream_t s;
    ~StreamFree() {
      if (p) cudaFreeAsync(p, s);
    }
  } part{nullptr, st};
  R* out = img;
  if (G > 1) {
    out = group_buf;
    if (!out) {
      if (malloc_async(&part.p, (size_t)G * n * sizeof(R), st) != cudaSuccess) {
        part.p = nullptr;
        cudaGetLastError();
        return set_error(RIX_ENOMEM, "plane-group images (%zu bytes)", (size_t)G * n * sizeof(R));
      }
      out = static_cast<R*>(part.p);
    }
  }
  g.pg = P / G;
  const int acc = G > 1 ? 0 : accumulate;
  auto launch = [&]() -> int {
    if constexpr (sizeof(R) == 4) {
      if (g.M != g.L)
        return with_log<kMinLogF + 1, kMaxLogL<R>>(g.logL, [&](auto ll) {
          using X = CropRows<decltype(ll)::value>;
          return x_launch<X>(k_crop_rows<decltype(ll)::value>, dim3((unsigned)ceil_div(g.M, X::NB), (unsigned)G), st,
                             x_args(g), T, out, scale, acc, twiddles<R>(ctx));
        });
    }
    return with_plane_shape<R>(g, [&](auto lf, auto e) {
      using X = Xf<R, decltype(lf)::value, decltype(e)::value, false>;
      return x_launch<X>(k_inv_rows<R, decltype(lf)::value, decltype(e)::value>,
                         dim3((unsigned)(g.M / X::NB), (unsigned)G), st, x_args(g), T, out, scale, acc,
                         twiddles<R>(ctx));
    });
  };
  RIX_TRY(launch());
  if (G > 1) return sum_groups<R>(ctx, img, out, G, n, accumulate, st);
  return RIX_OK;
}

#define RIX_FFT_ROWS_INST(R)                                                                             \
  template int fwd_rows<R>(const Ctx*, const XformGeom&, const R*, cplx<R>*, cudaStream_t);              \
  template int inv_rows<R>(const Ctx*, const XformGeom&, const cplx<R>*, R*, double, int, cudaStream_t, R*, int); \
  template int inv_rows_groups<R>(const Ctx*, const XformGeom&, int);

}  // namespace rix
