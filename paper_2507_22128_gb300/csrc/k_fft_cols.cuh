// The column passes (see fft_engine.cuh).
#pragma once

#include "fft_engine.cuh"

namespace rix {

template <typename R>
int fwd_cols(const Ctx* ctx, const XformGeom& g, const cplx<R>* T, cplx<R>* spec, cudaStream_t st) {
  RIX_TRY(check_geom<R>(g));
  if constexpr (sizeof(R) == 4) {
    if (g.M != g.L)
      return with_log<kMinLogF + 1, kMaxLogL<R>>(g.logL, [&](auto ll) {
        using X = PadCols<decltype(ll)::value>;
        return x_launch<X>(k_pad_cols<decltype(ll)::value>,
                           dim3((unsigned)ceil_div(g.S, X::NB * X::CPT), (unsigned)g.nplanes), st, x_args(g), T, spec,
                           twiddles<R>(ctx));
      });
  }
  return with_plane_shape<R>(g, [&](auto lf, auto e) {
    using X = Xf<R, decltype(lf)::value, decltype(e)::value, true>;
    return x_launch<X>(k_fwd_cols<R, decltype(lf)::value, decltype(e)::value>,
                       dim3((unsigned)ceil_div(g.S, X::NB), (unsigned)g.nplanes), st, x_args(g), T, spec,
                       twiddles<R>(ctx));
  });
}

template <typename R>
int inv_cols(const Ctx* ctx, const XformGeom& g, const cplx<R>* spec, int op, const void* tab, cplx<R>* T,
             cudaStream_t st) {
  RIX_TRY(check_geom<R>(g));
  if constexpr (sizeof(R) == 4) {
    if (g.M != g.L)
      return with_log<kMinLogF + 1, kMaxLogL<R>>(g.logL, [&](auto ll) {
        using X = PadCols<decltype(ll)::value>;
        return x_launch<X>(k_crop_cols<decltype(ll)::value>,
                           dim3((unsigned)ceil_div(g.S, X::NB * X::CPT), (unsigned)g.nplanes), st, x_args(g), spec, op,
                           tab, T, twiddles<R>(ctx));
      });
  }
  return with_plane_shape<R>(g, [&](auto lf, auto e) {
    using X = Xf<R, decltype(lf)::value, decltype(e)::value, true>;
    return x_launch<X>(k_inv_cols<R, decltype(lf)::value, decltype(e)::value>,
                       dim3((unsigned)ceil_div(g.S, X::NB), (unsigned)g.nplanes), st, x_args(g), spec, op, tab, T,
                       twiddles<R>(ctx));
  });
}

template <typename R>
int conv_cols(const Ctx* ctx, const XformGeom& g, const cplx<R>* Tin, int op, const void* tab, cplx<R>* Tout,
              cudaStream_t st) {
  RIX_TRY(check_geom<R>(g));
  if (g.lo != 0 || g.nplanes != 1 || 2 * g.M != g.L)
    return set_error(RIX_EINVAL, "conv_cols needs a zero-padded plane and a window starting at 0");
  return with_log<kMinLogF, kMaxLogL<R> - 1>(g.logL - 1, [&](auto lf) {
    using X = Xf<R, decltype(lf)::value, 2, true>;
    return x_launch<X>(k_conv_cols<R, decltype(lf)::value>, dim3((unsigned)ceil_div(g.S, X::NB)), st, x_args(g), Tin,
                       op, tab, Tout, twiddles<R>(ctx));
  });
}

#define RIX_FFT_COLS_INST(R)                                                                             \
  template int fwd_cols<R>(const Ctx*, const XformGeom&, const cplx<R>*, cplx<R>*, cudaStream_t);        \
  template int inv_cols<R>(const Ctx*, const XformGeom&, const cplx<R>*, int, const void*, cplx<R>*, cudaStream_t); \
  template int conv_cols<R>(const Ctx*, const XformGeom&, const cplx<R>*, int, const void*, cplx<R>*, cudaStream_t);

}  // namespace rix
