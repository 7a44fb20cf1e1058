// Device-side building blocks of the FFT stages: in-register DFTs, twiddles
// and phase screens.  Included by the translation units that launch them
// (each gets its own copy in an anonymous namespace).
#pragma once

#include <cuda_runtime.h>

#include <type_traits>

#include "rix_internal.cuh"

namespace rix {
namespace {

constexpr int kFftThreads = 256;

// Ping-pong CTAs hold kFftThreads * kPingPongVals complex values per buffer.
template <typename R> constexpr int kPingPongVals = std::is_same<R, float>::value ? 16 : 8;

__host__ __device__ constexpr int padi(int i) { return i + (i >> 4); }
__host__ __device__ constexpr int padded_len(int L) { return L + (L >> 4); }

// cos / sin of 2 pi m / 16
__device__ constexpr double kCos16[16] = {1.0, 0.92387953251128674, 0.70710678118654752, 0.38268343236508978,
                                          0.0, -0.38268343236508978, -0.70710678118654752, -0.92387953251128674,
                                          -1.0, -0.92387953251128674, -0.70710678118654752, -0.38268343236508978,
                                          0.0, 0.38268343236508978, 0.70710678118654752, 0.92387953251128674};
__device__ constexpr double kSin16[16] = {0.0, 0.38268343236508978, 0.70710678118654752, 0.92387953251128674,
                                          1.0, 0.92387953251128674, 0.70710678118654752, 0.38268343236508978,
                                          0.0, -0.38268343236508978, -0.70710678118654752, -0.92387953251128674,
                                          -1.0, -0.92387953251128674, -0.70710678118654752, -0.38268343236508978};

// exp(DIR * 2 pi i m / N) for N | 16
template <int N, int DIR, typename C>
__device__ __forceinline__ C wconst(int m) {
  const int k = (m * (16 / N)) & 15;
  return cmake<C>(kCos16[k], DIR * kSin16[k]);
}

template <int DIR, typename C>
__device__ __forceinline__ C rot90(C a) {   // a * exp(DIR i pi / 2)
  C r;
  if (DIR < 0) { r.x = a.y; r.y = -a.x; } else { r.x = -a.y; r.y = a.x; }
  return r;
}

template <int DIR, typename C>
__device__ __forceinline__ void dft4(C& a0, C& a1, C& a2, C& a3) {
  const C t0 = a0 + a2, t1 = a0 - a2, t2 = a1 + a3, t3 = rot90<DIR>(a1 - a3);
  a0 = t0 + t2; a2 = t0 - t2; a1 = t1 + t3; a3 = t1 - t3;
}

// in-register DFT of size RAD, natural order in and out
template <int RAD, int DIR, typename C>
__device__ __forceinline__ void dft(C* v) {
  if constexpr (RAD == 2) {
    const C t = v[0]; v[0] = t + v[1]; v[1] = t - v[1];
  } else if constexpr (RAD == 4) {
    dft4<DIR>(v[0], v[1], v[2], v[3]);
  } else if constexpr (RAD == 8) {
    // n = 2 n1 + n2: length-4 DFTs over n1, twiddle W8^(n2 k1), length-2 over n2
    dft4<DIR>(v[0], v[2], v[4], v[6]);
    dft4<DIR>(v[1], v[3], v[5], v[7]);
    C o[8];
#pragma unroll
    for (int k1 = 0; k1 < 4; ++k1) {
      const C a = v[2 * k1];
      const C b = k1 ? cmul(v[2 * k1 + 1], wconst<8, DIR, C>(k1)) : v[2 * k1 + 1];
      o[k1] = a + b;
      o[k1 + 4] = a - b;
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] = o[i];
  } else {
    static_assert(RAD == 16, "radix");
    // n = 4 n1 + n2: length-4 DFTs over n1, twiddle W16^(n2 k1), length-4 over n2
#pragma unroll
    for (int n2 = 0; n2 < 4; ++n2) dft4<DIR>(v[n2], v[4 + n2], v[8 + n2], v[12 + n2]);
    C y[16];
#pragma unroll
    for (int k1 = 0; k1 < 4; ++k1)
#pragma unroll
      for (int n2 = 0; n2 < 4; ++n2) {
        const C t = v[4 * k1 + n2];
        y[4 * k1 + n2] = (n2 * k1) ? cmul(t, wconst<16, DIR, C>(n2 * k1)) : t;
      }
#pragma unroll
    for (int k1 = 0; k1 < 4; ++k1) {
      dft4<DIR>(y[4 * k1], y[4 * k1 + 1], y[4 * k1 + 2], y[4 * k1 + 3]);
#pragma unroll
      for (int k2 = 0; k2 < 4; ++k2) v[k1 + 4 * k2] = y[4 * k1 + k2];
    }
  }
}

// v[r] *= w^r, w = exp(DIR 2 pi i k / 2^m), 2^m = p RAD and k < p: w, w^4 and
// w^8 come from the FP64-accurate table, the other powers from at most three
// products of them (a few ulp), instead of RAD - 1 dependent table loads.  The
// table holds the roots of every power of two, exp(-2 pi i k / 2^j) at
// 2^j + k, so w^4 and w^8 are the k-th roots of 2^(m-2) and 2^(m-3) and the
// lanes of a warp, which hold consecutive k, read consecutive entries (from
// one table of the longest length, k 2^(14-m) apart, each load touched up to
// 16 cache lines).
template <typename R, int DIR, int RAD>
__device__ __forceinline__ void apply_twiddles(cplx<R>* v, const cplx<R>* __restrict__ tw, int k, int m) {
  using C = cplx<R>;
  C w[RAD];
  auto ld = [&](int j) {
    C t = tw[(1 << j) + k];
    if (DIR > 0) t.y = -t.y;
    return t;
  };
  w[1] = ld(m);
  if constexpr (RAD >= 4) {
    w[2] = cmul(w[1], w[1]);
    w[3] = cmul(w[2], w[1]);
  }
  if constexpr (RAD >= 8) {
    w[4] = ld(m - 2);
#pragma unroll
    for (int r = 5; r < 8; ++r) w[r] = cmul(w[4], w[r - 4]);
  }
  if constexpr (RAD >= 16) {
    w[8] = ld(m - 3);
#pragma unroll
    for (int r = 9; r < 16; ++r) w[r] = cmul(w[8], w[r - 8]);
  }
#pragma unroll
  for (int r = 1; r < RAD; ++r) v[r] = cmul(v[r], w[r]);
}

// ---------------------------------------------------------------- factors ----
template <typename R> __device__ __forceinline__ void sincos_pi(R x, R* s, R* c);
template <> __device__ __forceinline__ void sincos_pi<float>(float x, float* s, float* c) { sincospif(x, s, c); }
template <> __device__ __forceinline__ void sincos_pi<double>(double x, double* s, double* c) { sincospi(x, s, c); }

// exp(DIR 2 pi i w_p (n-1)) with the phase argument formed and reduced in FP64
template <typename R, int DIR>
__device__ __forceinline__ cplx<R> wscreen(double wp, double nm1) {
  const double ph = wp * nm1;
  const double fr = ph - rint(ph);
  R s, c;
  sincos_pi<R>((R)(2.0 * fr), &s, &c);
  return cmake<cplx<R>>(c, DIR * s);
}

// exp(DIR 2 pi i w (n-1)) in FP32 with w = wh + wl and n - 1 = m.x + m.y held as
// pairs of floats (48 bits): the leading product is reduced to a fraction of a turn
// exactly; what it lost to rounding (up to 2^-24 of its turns) and the two cross
// products are added in FP32.  Left out are 2^-24 of those additions and wl m.y,
// 2^-48 of the turns: below the rounding of the result to float up to some
// thousand turns.  Eight FP32 operations instead of five FP64 ones at 1/64 of
// their rate
template <int DIR>
__device__ __forceinline__ float2 wscreen_ff(float wh, float wl, float2 m) {
  const float p = __fmul_rn(wh, m.x);
  float e = __fmaf_rn(wh, m.x, -p);
  e = __fmaf_rn(wh, m.y, e);
  e = __fmaf_rn(wl, m.x, e);
  const float fr = (p - rintf(p)) + e;
  float s, c;
  sincospif(2.0f * fr, &s, &c);
  return make_float2(c, DIR * s);
}

// ------------------------------------------------------ host-side setup ----
template <typename R>
const cplx<R>* twiddles(const Ctx* ctx) {
  return std::is_same<R, float>::value ? static_cast<const cplx<R>*>(ctx->tw32.p)
                                       : static_cast<const cplx<R>*>(ctx->tw64.p);
}

}  // namespace
}  // namespace rix
