// Row and column passes of the 2D transforms between a real M x M image and
// the window [lo, lo + S)^2 of its L x L spectrum (k_fft.cu describes the
// conventions), with every length fixed at compile time.
//
// Zero padding and cropping are not transformed (but for k_pad_rows and
// k_pad_cols): with L = 2 M the L-point
// transform of M centred values is two M-point transforms,
//   X[2k + e] = sum_n (x[n] w_L^(e n)) w_M^(k n),            e = 0, 1,
// and the M cropped outputs of an L-point inverse transform are
//   x[n] = y_0[n] + w_L^(-n) y_1[n],  y_e = F_M^-1 X[2k + e],
// n the centred offset -M/2 .. M/2 - 1 (held at n mod M).  M = L is the single
// transform e = 0.
//
// A thread carries V = 16 values (fewer in FP64 at short lengths) in registers
// through every pass: global memory
// -> registers -> first pass, one shared-memory exchange between passes, last
// pass -> registers -> global memory.
//
// The intermediate T[j][b] (window column j, image row b) is stored in blocks
// of four columns, [j / 4][b][j % 4]: a row pass, which holds few rows, then
// writes and reads whole 32-byte sectors, and a column pass, whose threads
// run over its columns first, reads and writes contiguous memory.  With the
// plain [j][b] layout a row pass of one 8192-point row moved a 32-byte sector
// for every 8-byte value.
//
// Measured per launch on the outer uv partition of a 4096^2 job (32 planes,
// FP32, 8.6 GB in and out of each pass, 1.27 ms at the copy bandwidth), before
// (run-time radices, [j][b], 8-byte runs, twiddles 2^(14 - m) entries apart)
// and after: forward rows 12.3 -> 3.1 ms, forward columns 8.6 -> 2.8, inverse
// columns 8.5 -> 3.0, inverse rows 18.2 -> 3.5; of a 1024^2 job (16 planes)
// 195 -> 69, 142 -> 57, 146 -> 59 and 289 -> 84 us.  Instruction issue and
// shared-memory wavefronts bound them now (60-70 % each).
#pragma once

#include "fft_ct.cuh"

namespace rix {
namespace {

constexpr int kTBlk = 4;   // window columns per block of T

__host__ __device__ __forceinline__ int64_t t_index(int j, int b, int M) {
  return ((int64_t)(j >> 2) * M + b) * kTBlk + (j & (kTBlk - 1));
}
static_assert(kTBlk == 4, "t_index");
// moving j by a multiple dj of kTBlk moves t_index by dj M
// complex values of one plane of T for a window of S columns
__host__ __device__ __forceinline__ int64_t t_plane(int S, int M) {
  return (int64_t)((S + kTBlk - 1) / kTBlk) * kTBlk * M;
}

struct XArgs {
  int M, L, lo, S, nplanes, mode, herm;
  const void* corr;
  const double* nm1;
  const float2* nm1f;   // n - 1 as pairs of floats (FP32 inverse rows), or null
  double w0, dw;
  const void* screen;   // tabulated corr x phase screen per plane, or null
  int pg;               // inverse rows: planes per grid row y
};

// Transforms of up to 2^kFewLogF points take fewer values per thread in FP64 (4, from
// 2^8 on 8): the double-precision pipe takes a warp's instruction in 16 cycles or
// more, so the 1,200 instructions of a thread with 16 values were 10 us of every pass
// over a small image, however few its rows.  ms-CLEAN cycle of 20 components, four
// partitions, 16 values / fewer: 32^2 3.1 / 1.6 ms, 128^2 3.8 / 1.8, 256^2 4.2 / 3.0,
// 512^2 6.7 / 6.2.
constexpr int kFewLogF = 9;

// One transform length F = 2^LOGF, E = L / F sub-transforms; rows, or columns
// with the thread index running over the CTA's columns first.
//   T       F / 4 threads between 64 (short lengths: more CTAs for small
//           images) and 256 (512 above 4096), 16 values each; 128 threads
//           with V = 4 or 8
//   kCtas   CTAs per SM that the registers (WARPS in all) and the shared
//           memory are sized for; one in FP64, whose rate of 1/64 of FP32
//           leaves nothing for more warps to hide
//   kPing   two exchange buffers (one barrier per exchange) where they fit
template <typename R, int LOGF, int E, bool COLS, int WARPS = 24>
struct Xf {
  static constexpr int F = 1 << LOGF;
  static constexpr bool kF32 = sizeof(R) == 4;
  static constexpr int V = kF32 || LOGF > kFewLogF ? 16 : LOGF < 8 ? 4 : 8;
  static constexpr int MLR = V == 16 ? 4 : V == 8 ? 3 : 2;   // log2 of the largest radix
  static constexpr int kMaxT = F > 4096 ? 512 : 256;
  static constexpr int kWant = F / 4 < 64 ? 64 : F / 4;
  static constexpr int T = V < 16 ? 128 : kWant < kMaxT ? kWant : kMaxT;
  static constexpr int NB = T * V / F;                 // rows (columns) per CTA
  static constexpr int PADF = padded_len(F);
  static constexpr int kBuf = NB * PADF;               // complex values of an exchange buffer
  // CTAs per SM the registers and the shared memory are set for
  static constexpr int kCtas = kF32 ? WARPS * 32 / T : 1;
  static constexpr size_t kStash = (size_t)(E == 2 ? T * V : 0) * 2 * sizeof(R);
  static constexpr bool kPing = kF32 && kCtas * (2 * kBuf * 2 * sizeof(R) + kStash) <= 220 * 1024;
  static constexpr size_t kSmem = (size_t)(kPing ? 2 : 1) * kBuf * 2 * sizeof(R) + kStash;
  static constexpr int NP = ct_npass(LOGF, MLR);
  static constexpr int LRL = ct_lr(LOGF, NP - 1, MLR); // radix of the last pass
  static constexpr int IPRL = F >> LRL;
  static constexpr int LR0 = ct_lr(LOGF, 0, MLR);
  static constexpr int IPR0 = F >> LR0;
  // item `it` of the thread in a pass with 2^LR legs: row (column) c and the
  // position i of leg 0; leg r sits at i + r IPR.  Slot s = it 2^LR + r.
  template <int LR>
  static __device__ __forceinline__ void item(int tid, int it, int& c, int& i) {
    constexpr int IPR = F >> LR;
    const int g = tid + it * T;
    if constexpr (COLS) {
      c = g % NB;
      i = g / NB;
    } else {
      c = g / IPR;
      i = g % IPR;
    }
  }
  template <int LR>
  static __device__ __forceinline__ void slot(int tid, int s, int& c, int& pos) {
    constexpr int RAD = 1 << LR, IPR = F >> LR;
    item<LR>(tid, s / RAD, c, pos);
    pos += (s % RAD) * IPR;
  }
  // a position's place in the exchange buffer
  static constexpr int kPosStride = COLS ? NB : 1;
  static __device__ __forceinline__ int addr(int c, int pos) {
    if constexpr (COLS) return padi(pos) * NB + c;
    else return c * PADF + padi(pos);
  }
};

// Offset of the pixel at position i + r IPR of a centred, zero-padded
// transform of length L from the one at i (legs ct_outer only: i < IPR does
// not carry past the fold at L / 2).
template <int LR, int L>
__host__ __device__ constexpr int fold(int r) {
  return r < (1 << LR) / 2 ? r * (L >> LR) + L / 4 : r * (L >> LR) + L / 4 - L;
}

// Pass PS and the ones after it of the NB transforms held in v (slots of pass
// PS on entry, of the last pass on return).  par: the exchange buffer of the
// next exchange (ping-pong); without ping-pong every exchange waits until the
// buffer has been read.
template <class X, typename R, int DIR, int LOGF, int PS, bool kPad = false>
__device__ __forceinline__ void xf_passes(cplx<R> (&v)[X::V], cplx<R>* buf, int& par, const cplx<R>* __restrict__ tw,
                                          int tid) {
  using C = cplx<R>;
  constexpr int LR = ct_lr(LOGF, PS, X::MLR), LOGP = ct_logp(LOGF, PS, X::MLR);
  constexpr int RAD = 1 << LR, IPR = X::F >> LR, P = 1 << LOGP, K = X::V / RAD;
#pragma unroll
  for (int it = 0; it < K; ++it) {
    C* w = v + it * RAD;
    if constexpr (LOGP > 0) {
      int c, pos;
      X::template slot<LR>(tid, it * RAD, c, pos);
      const int k = pos & (P - 1);
      if constexpr (sizeof(R) == 4) {
        if (k) apply_twiddles<R, DIR, RAD>(w, tw, k, LOGP + LR);
      } else {
        // FP64: every twiddle from the table (forming powers costs four
        // double-precision operations each)
#pragma unroll
        for (int r = 1; r < RAD; ++r) {
          C t = tw[(1 << (LOGP + LR)) + r * k];
          if (DIR > 0) t.y = -t.y;
          w[r] = cmul(w[r], t);
        }
      }
    }
    if constexpr (kPad && PS == 0) dft_zin<RAD, DIR>(w);   // the centred input's zero half is not read
    else dft<RAD, DIR>(w);
  }
  if constexpr (PS + 1 < X::NP) {
    constexpr int LRN = ct_lr(LOGF, PS + 1, X::MLR);
    constexpr int RADN = 1 << LRN, IPRN = X::F >> LRN, KN = X::V / RADN, PST = X::kPosStride;
    // padi is linear over multiples of 16 and inside one group of 16
    constexpr bool kLin16 = (P % 16) == 0;
    constexpr bool kLinSmall = (P * RAD <= 16) && (16 % (P * RAD) == 0);
    C* b = X::kPing ? buf + par * X::kBuf : buf;
    if constexpr (X::kPing) par ^= 1;
    else __syncthreads();
#pragma unroll
    for (int it = 0; it < K; ++it) {
      int c, i;
      X::template item<LR>(tid, it, c, i);
      const int k = i & (P - 1);
      const int o = ((i - k) << LR) + k;
      C* d = b + X::addr(c, o);
#pragma unroll
      for (int r = 0; r < RAD; ++r) {
        if constexpr (kLin16) d[r * (P + P / 16) * PST] = v[it * RAD + r];
        else if constexpr (kLinSmall) d[r * P * PST] = v[it * RAD + r];
        else b[X::addr(c, o + r * P)] = v[it * RAD + r];
      }
    }
    __syncthreads();
#pragma unroll
    for (int it = 0; it < KN; ++it) {
      int c, i;
      X::template item<LRN>(tid, it, c, i);
      const C* d = b + X::addr(c, i);
#pragma unroll
      for (int r = 0; r < RADN; ++r) {
        if constexpr ((IPRN % 16) == 0) v[it * RADN + r] = d[r * (IPRN + IPRN / 16) * PST];
        else v[it * RADN + r] = b[X::addr(c, i + r * IPRN)];
      }
    }
    xf_passes<X, R, DIR, LOGF, PS + 1, kPad>(v, buf, par, tw, tid);
  }
}

// The thread index, opaque to the compiler: formed once per trip of a loop over
// transforms, it keeps the loop's addresses and twiddles from being hoisted
// out of the loop into registers (300 bytes of spills in k_inv_rows).
__device__ __forceinline__ int opaque_tid() {
  int t = threadIdx.x;
  asm volatile("" : "+r"(t));
  return t;
}

// The E sub-transforms: v holds e = 0's inputs, stash (the thread's own 16
// slots, T apart) e = 1's; on return v holds the last one's outputs and
// stash, with E = 2, the first one's.
template <class X, typename R, int DIR, int LOGF, int E>
__device__ __forceinline__ void xf_run(cplx<R> (&v)[X::V], cplx<R>* buf, cplx<R>* stash, int& par,
                                       const cplx<R>* __restrict__ tw) {
#pragma unroll 1
  for (int e = 0;; ++e) {
    xf_passes<X, R, DIR, LOGF, 0>(v, buf, par, tw, opaque_tid());
    if (e == E - 1) break;
#pragma unroll
    for (int s = 0; s < X::V; ++s) {
      const cplx<R> t = stash[s * X::T];
      stash[s * X::T] = v[s];
      v[s] = t;
    }
  }
}

// w_L^(DIR a) of the centred offset a at position n of an F-point transform
template <typename R, int LOGF, int DIR>
__device__ __forceinline__ cplx<R> half_twiddle(const cplx<R>* __restrict__ tw, int n) {
  constexpr int F = 1 << LOGF;
  const int a = n < F / 2 ? n : n - F;
  cplx<R> t = tw[2 * F + (a & (2 * F - 1))];
  if (DIR > 0) t.y = -t.y;
  return t;
}

// 16-byte (FP64: two 16-byte) access of a pair of complex values
template <typename C>
__device__ __forceinline__ void xld_pair(const C* p, C& a, C& b) {
  if constexpr (sizeof(C) == 8) {
    const float4 w = *reinterpret_cast<const float4*>(p);
    a.x = w.x; a.y = w.y; b.x = w.z; b.y = w.w;
  } else {
    a = p[0];
    b = p[1];
  }
}
template <typename C>
__device__ __forceinline__ void xst_pair(C* p, const C& a, const C& b) {
  if constexpr (sizeof(C) == 8) {
    *reinterpret_cast<float4*>(p) = make_float4(a.x, a.y, b.x, b.y);
  } else {
    p[0] = a;
    p[1] = b;
  }
}

template <typename R>
__device__ __forceinline__ cplx<R> xspec_op(int op, cplx<R> x, const void* tab, int64_t k) {
  if (op == kOpMulReal) return x * static_cast<const R*>(tab)[k];
  if (op == kOpMulCplx) return cmul(x, static_cast<const cplx<R>*>(tab)[k]);
  return x;
}

#define RIX_X_SMEM                                                   \
  extern __shared__ __align__(16) unsigned char smem_raw[];          \
  C* buf = reinterpret_cast<C*>(smem_raw);                           \
  C* stash = buf + (X::kPing ? 2 : 1) * X::kBuf + threadIdx.x;       \
  int par = 0, tid = threadIdx.x;

// ---------------------------------------------------------------- kernels ----
// image rows -> window columns of their spectra (T); grid (M / NB, planes)
template <typename R, int LOGF, int E>
__global__ void __launch_bounds__((Xf<R, LOGF, E, false>::T), (Xf<R, LOGF, E, false>::kCtas))
    k_fwd_rows(XArgs a, const R* __restrict__ img, cplx<R>* __restrict__ T, const cplx<R>* __restrict__ tw) {
  using C = cplx<R>;
  using X = Xf<R, LOGF, E, false>;
  constexpr int M = X::F;
  RIX_X_SMEM
  const int p = blockIdx.y, b0 = blockIdx.x * X::NB;
  const R* corr = static_cast<const R*>(a.corr);
  const C* scr = a.mode == kFacPhase && a.screen ? static_cast<const C*>(a.screen) + (int64_t)p * M * M : nullptr;
  const double wp = a.w0 + p * a.dw;
  C v[X::V];
#pragma unroll
  for (int s = 0; s < X::V; ++s) {
    int c, n;
    X::template slot<X::LR0>(tid, s, c, n);
    const int aa = (n + M / 2) & (M - 1), b = b0 + c;
    const int64_t pix = (int64_t)b * M + aa;
    R x = img[pix];
    if ((aa + b) & 1) x = -x;
    if (scr) {
      v[s] = scr[pix] * x;
    } else {
      if (a.mode != kFacNone) x *= corr[pix];
      if (a.mode == kFacPhase) v[s] = wscreen<R, -1>(wp, a.nm1[pix]) * x;
      else v[s] = cmake<C>(x, 0.0);
    }
  }
  if constexpr (E == 2) {
#pragma unroll
    for (int s = 0; s < X::V; ++s) {
      int c, n;
      X::template slot<X::LR0>(tid, s, c, n);
      stash[s * X::T] = cmul(v[s], half_twiddle<R, LOGF, -1>(tw, n));
    }
  }
  xf_run<X, R, -1, LOGF, E>(v, buf, stash, par, tw);
  C* Tp = T + (int64_t)p * t_plane(a.S, M);
#pragma unroll
  for (int s = 0; s < X::V; ++s) {
    int c, k;
    X::template slot<X::LRL>(tid, s, c, k);
    const int b = b0 + c, j = E * k - a.lo;
    if constexpr (E == 2) {
      const C v0 = stash[s * X::T];
      if ((a.lo & 1) == 0) {
        // an odd S leaves the pair's second value in the block's padding
        if (j >= 0 && j < a.S) xst_pair(Tp + t_index(j, b, M), v0, v[s]);
      } else {
        if (j >= 0 && j < a.S) Tp[t_index(j, b, M)] = v0;
        if (j + 1 >= 0 && j + 1 < a.S) Tp[t_index(j + 1, b, M)] = v[s];
      }
    } else {
      if (j >= 0 && j < a.S) Tp[t_index(j, b, M)] = v[s];
    }
  }
}

// The forward passes of a zero-padded plane in FP32 as one L-point transform
// whose first pass skips the zero half.  A residual v - G^dagger F x is small
// beside both terms, so its relative difference is a thousand times the
// transform's rounding: this plan (radices, twiddles, order of operations) is
// the one the FP32 model planes have always been formed with, and keeps the
// major cycle's residual bit for bit up to the gridder, which the two half
// transforms would not (1.7e-4 - 4.9e-4 of a residual at the noise level).
// 32 warps per SM (64 registers): the passes alternate between loads, two to
// three exchanges and stores, and at 16 warps issued on 44 % of the cycles
// (68 % at 32).
constexpr int kPadWarps = 32;

template <int LOGL>
using PadRows = Xf<float, LOGL, 1, false, kPadWarps>;

template <int LOGL>
__global__ void __launch_bounds__((PadRows<LOGL>::T), (PadRows<LOGL>::kCtas))
    k_pad_rows(XArgs a, const float* __restrict__ img, float2* __restrict__ T, const float2* __restrict__ tw) {
  using R = float;
  using C = float2;
  using X = PadRows<LOGL>;
  constexpr int L = X::F, M = L / 2;
  RIX_X_SMEM
  const int p = blockIdx.y, b0 = blockIdx.x * X::NB;
  const R* corr = static_cast<const R*>(a.corr);
  const C* scr = a.mode == kFacPhase && a.screen ? static_cast<const C*>(a.screen) + (int64_t)p * M * M : nullptr;
  const double wp = a.w0 + p * a.dw;
  constexpr int RAD0 = 1 << X::LR0, RADL = 1 << X::LRL;
  C v[16];
#pragma unroll
  for (int it = 0; it < 16 / RAD0; ++it) {
    int c, i;
    X::template item<X::LR0>(tid, it, c, i);
    const int64_t pix0 = (int64_t)(b0 + c) * M + i;
    const bool odd = (i + b0 + c) & 1;   // the fold and the legs are even
#pragma unroll
    for (int r = 0; r < RAD0; ++r) {
      if (!ct_outer<RAD0>(r)) continue;
      const int64_t pix = pix0 + fold<X::LR0, L>(r);
      R x = img[pix];
      if (odd) x = -x;
      C& z = v[it * RAD0 + r];
      if (scr) {
        z = scr[pix] * x;
      } else {
        if (a.mode != kFacNone) x *= corr[pix];
        if (a.mode == kFacPhase) z = wscreen<R, -1>(wp, a.nm1[pix]) * x;
        else z = cmake<C>(x, 0.0);
      }
    }
  }
  xf_passes<X, R, -1, LOGL, 0, true>(v, buf, par, tw, tid);
  (void)stash;
  C* Tp = T + (int64_t)p * t_plane(a.S, M);
#pragma unroll
  for (int it = 0; it < 16 / RADL; ++it) {
    int c, i;
    X::template item<X::LRL>(tid, it, c, i);
    const int j0 = i - a.lo;
    C* o = Tp + t_index(j0, b0 + c, M);
#pragma unroll
    for (int r = 0; r < RADL; ++r)
      if ((unsigned)(j0 + r * X::IPRL) < (unsigned)a.S) o[(int64_t)r * X::IPRL * M] = v[it * RADL + r];
  }
}

// CPT columns per thread: the CTA reads CPT adjacent columns of T together and
// transforms them in turn, the waiting ones' inputs in shared memory.
template <int LOGL>
struct PadCols : Xf<float, LOGL, 1, true, kPadWarps> {
  using B = Xf<float, LOGL, 1, true, kPadWarps>;
  static constexpr int CPT = B::NB >= kTBlk ? 1 : 2;
  static constexpr size_t kStash = (size_t)(CPT - 1) * 8 * B::T * sizeof(float2);
  static constexpr bool kPing = B::kCtas * (2 * B::kBuf * sizeof(float2) + kStash) <= 220 * 1024;
  static constexpr size_t kSmem = (size_t)(kPing ? 2 : 1) * B::kBuf * sizeof(float2) + kStash;
};

template <int LOGL>
__global__ void __launch_bounds__((PadCols<LOGL>::T), (PadCols<LOGL>::kCtas))
    k_pad_cols(XArgs a, const float2* __restrict__ T, float2* __restrict__ spec, const float2* __restrict__ tw) {
  using R = float;
  using C = float2;
  using X = PadCols<LOGL>;
  constexpr int L = X::F, M = L / 2, CPT = X::CPT, RAD0 = 1 << X::LR0;
  RIX_X_SMEM
  const int p = blockIdx.y, j0 = blockIdx.x * X::NB * CPT;
  const C* Tp = T + (int64_t)p * t_plane(a.S, M);
  constexpr int RADL = 1 << X::LRL;
  C v[16];
  int live = 0;   // the slot's place among the ones that hold data
#pragma unroll
  for (int it = 0; it < 16 / RAD0; ++it) {
    int c, i;
    X::template item<X::LR0>(tid, it, c, i);
    const int j = j0 + c * CPT;
    const C* src = Tp + t_index(j, i, M);
#pragma unroll
    for (int r = 0; r < RAD0; ++r) {
      if (!ct_outer<RAD0>(r)) continue;
      C x[CPT];
#pragma unroll
      for (int q = 0; q < CPT; ++q) x[q] = make_float2(0.f, 0.f);
      if (j < a.S) {
        // a second column past S is the block's padding: read, not stored
        const C* e = src + fold<X::LR0, L>(r) * kTBlk;
        if constexpr (CPT == 1) x[0] = e[0];
        else xld_pair(e, x[0], x[1]);
      }
      v[it * RAD0 + r] = x[0];
#pragma unroll
      for (int q = 1; q < CPT; ++q) stash[((q - 1) * 8 + live) * X::T] = x[q];
      ++live;
    }
  }
  C* sp = spec + (int64_t)p * a.S * a.S;
#pragma unroll 1
  for (int q = 0; q < CPT; ++q) {
    tid = opaque_tid();
    if (CPT > 1 && q > 0) {
      int k = 0;
#pragma unroll
      for (int s = 0; s < 16; ++s)
        if (ct_outer<RAD0>(s % RAD0)) v[s] = stash[((q - 1) * 8 + k++) * X::T];
    }
    xf_passes<X, R, -1, LOGL, 0, true>(v, buf, par, tw, tid);
#pragma unroll
    for (int it = 0; it < 16 / RADL; ++it) {
      int c, i;
      X::template item<X::LRL>(tid, it, c, i);
      const int j = j0 + c * CPT + q, i0 = i - a.lo;
      C* o = sp + (int64_t)j * a.S + i0;
#pragma unroll
      for (int r = 0; r < RADL; ++r)
        if (j < a.S && (unsigned)(i0 + r * X::IPRL) < (unsigned)a.S) o[r * X::IPRL] = v[it * RADL + r];
    }
  }
}

// window columns (T) -> window rows of the spectrum; grid (ceil(S / NB), planes)
template <typename R, int LOGF, int E>
__global__ void __launch_bounds__((Xf<R, LOGF, E, true>::T), (Xf<R, LOGF, E, true>::kCtas))
    k_fwd_cols(XArgs a, const cplx<R>* __restrict__ T, cplx<R>* __restrict__ spec, const cplx<R>* __restrict__ tw) {
  using C = cplx<R>;
  using X = Xf<R, LOGF, E, true>;
  constexpr int M = X::F;
  RIX_X_SMEM
  const int p = blockIdx.y, j0 = blockIdx.x * X::NB;
  const C* Tp = T + (int64_t)p * t_plane(a.S, M);
  C v[X::V];
#pragma unroll
  for (int s = 0; s < X::V; ++s) {
    int c, n;
    X::template slot<X::LR0>(tid, s, c, n);
    const int j = j0 + c;
    v[s] = j < a.S ? Tp[t_index(j, (n + M / 2) & (M - 1), M)] : cmake<C>(0.0, 0.0);
  }
  if constexpr (E == 2) {
#pragma unroll
    for (int s = 0; s < X::V; ++s) {
      int c, n;
      X::template slot<X::LR0>(tid, s, c, n);
      stash[s * X::T] = cmul(v[s], half_twiddle<R, LOGF, -1>(tw, n));
    }
  }
  xf_run<X, R, -1, LOGF, E>(v, buf, stash, par, tw);
  C* sp = spec + (int64_t)p * a.S * a.S;
  const bool even = ((a.lo | a.S) & 1) == 0;
#pragma unroll
  for (int s = 0; s < X::V; ++s) {
    int c, k;
    X::template slot<X::LRL>(tid, s, c, k);
    const int j = j0 + c, i = E * k - a.lo;
    if (j >= a.S) continue;
    C* o = sp + (int64_t)j * a.S + i;
    if constexpr (E == 2) {
      const C v0 = stash[s * X::T];
      if (even) {
        if (i >= 0 && i < a.S) xst_pair(o, v0, v[s]);
      } else {
        if (i >= 0 && i < a.S) o[0] = v0;
        if (i + 1 >= 0 && i + 1 < a.S) o[1] = v[s];
      }
    } else {
      if (i >= 0 && i < a.S) o[0] = v[s];
    }
  }
}

// window rows of op(spec) -> image rows per window column (T)
template <typename R, int LOGF, int E>
__global__ void __launch_bounds__((Xf<R, LOGF, E, true>::T), (Xf<R, LOGF, E, true>::kCtas))
    k_inv_cols(XArgs a, const cplx<R>* __restrict__ spec, int op, const void* tab, cplx<R>* __restrict__ T,
               const cplx<R>* __restrict__ tw) {
  using C = cplx<R>;
  using X = Xf<R, LOGF, E, true>;
  constexpr int M = X::F;
  RIX_X_SMEM
  const int p = blockIdx.y, j0 = blockIdx.x * X::NB;
  const C* sp = spec + (int64_t)p * a.S * a.S;
  const C zero = cmake<C>(0.0, 0.0);
  const bool even = ((a.lo | a.S) & 1) == 0;
  C v[X::V];
#pragma unroll
  for (int s = 0; s < X::V; ++s) {
    int c, k;
    X::template slot<X::LR0>(tid, s, c, k);
    const int j = j0 + c, i = E * k - a.lo;
    const int64_t q = (int64_t)j * a.S + i;
    C x0 = zero, x1 = zero;
    if (j < a.S) {
      if constexpr (E == 2) {
        if (even) {
          if (i >= 0 && i < a.S) {
            xld_pair(sp + q, x0, x1);
            x0 = xspec_op<R>(op, x0, tab, q);
            x1 = xspec_op<R>(op, x1, tab, q + 1);
          }
        } else {
          if (i >= 0 && i < a.S) x0 = xspec_op<R>(op, sp[q], tab, q);
          if (i + 1 >= 0 && i + 1 < a.S) x1 = xspec_op<R>(op, sp[q + 1], tab, q + 1);
        }
      } else {
        if (i >= 0 && i < a.S) x0 = xspec_op<R>(op, sp[q], tab, q);
      }
    }
    v[s] = x0;
    if constexpr (E == 2) stash[s * X::T] = x1;
  }
  xf_run<X, R, +1, LOGF, E>(v, buf, stash, par, tw);
  C* Tp = T + (int64_t)p * t_plane(a.S, M);
#pragma unroll
  for (int s = 0; s < X::V; ++s) {
    int c, n;
    X::template slot<X::LRL>(tid, s, c, n);
    const int j = j0 + c;
    C z = v[s];
    if constexpr (E == 2) z = stash[s * X::T] + cmul(z, half_twiddle<R, LOGF, +1>(tw, n));
    if (j < a.S) Tp[t_index(j, (n + M / 2) & (M - 1), M)] = z;
  }
}

// window columns: F, op, F^-1 (the spectrum's full length L per column, window
// columns lo = 0 .. S - 1); grid ceil(S / NB).  Each sub-transform's spectrum
// X[2k + e] is multiplied and transformed back before the next is formed.
template <typename R, int LOGF>
__global__ void __launch_bounds__((Xf<R, LOGF, 2, true>::T), (Xf<R, LOGF, 2, true>::kCtas))
    k_conv_cols(XArgs a, const cplx<R>* __restrict__ Tin, int op, const void* tab, cplx<R>* __restrict__ Tout,
                const cplx<R>* __restrict__ tw) {
  using C = cplx<R>;
  using X = Xf<R, LOGF, 2, true>;
  constexpr int M = X::F, L = 2 * M;
  RIX_X_SMEM
  const int j0 = blockIdx.x * X::NB;
  C v[X::V];
#pragma unroll
  for (int s = 0; s < X::V; ++s) {
    int c, n;
    X::template slot<X::LR0>(tid, s, c, n);
    const int j = j0 + c;
    v[s] = j < a.S ? Tin[t_index(j, (n + M / 2) & (M - 1), M)] : cmake<C>(0.0, 0.0);
    stash[s * X::T] = cmul(v[s], half_twiddle<R, LOGF, -1>(tw, n));
  }
  // the exchange buffer between a forward and an inverse transform (the last
  // pass's slots are not the first pass's)
#pragma unroll 1
  for (int e = 0;; ++e) {
    tid = opaque_tid();
    xf_passes<X, R, -1, LOGF, 0>(v, buf, par, tw, tid);
    C* b = X::kPing ? buf + par * X::kBuf : buf;
    if constexpr (X::kPing) par ^= 1;
    else __syncthreads();
#pragma unroll
    for (int s = 0; s < X::V; ++s) {
      int c, k;
      X::template slot<X::LRL>(tid, s, c, k);
      const int j = j0 + c;
      C x = v[s];
      if (j < a.S) x = xspec_op<R>(op, x, tab, (int64_t)j * L + 2 * k + e);
      b[X::addr(c, k)] = x;
    }
    __syncthreads();
#pragma unroll
    for (int s = 0; s < X::V; ++s) {
      int c, k;
      X::template slot<X::LR0>(tid, s, c, k);
      v[s] = b[X::addr(c, k)];
    }
    xf_passes<X, R, +1, LOGF, 0>(v, buf, par, tw, tid);
    if (e == 1) break;
    // the first pass's own slots hold e = 1's input; the last pass's results
    // of e = 0 take their place slot by slot
#pragma unroll
    for (int s = 0; s < X::V; ++s) {
      const C t = stash[s * X::T];
      stash[s * X::T] = v[s];
      v[s] = t;
    }
  }
#pragma unroll
  for (int s = 0; s < X::V; ++s) {
    int c, n;
    X::template slot<X::LRL>(tid, s, c, n);
    const int j = j0 + c;
    const C z = stash[s * X::T] + cmul(v[s], half_twiddle<R, LOGF, +1>(tw, n));
    if (j < a.S) Tout[t_index(j, (n + M / 2) & (M - 1), M)] = z;
  }
}

// image rows b0 .. b0 + NB: sum over the CTA's planes (blockIdx.y * pg ..) of
// Re(conj(factor) F^-1 T), into image blockIdx.y of the output.  a.herm: the
// window holds columns 0 .. L/2 of a Hermitian spectrum, column c > L/2 is the
// conjugate of column L - c.
template <typename R, int LOGF, int E>
__global__ void __launch_bounds__((Xf<R, LOGF, E, false>::T), (Xf<R, LOGF, E, false>::kCtas))
    k_inv_rows(XArgs a, const cplx<R>* __restrict__ T, R* __restrict__ img, double scale, int accumulate,
               const cplx<R>* __restrict__ tw) {
  using C = cplx<R>;
  using X = Xf<R, LOGF, E, false>;
  constexpr int M = X::F, L = E * M;
  RIX_X_SMEM
  const int b0 = blockIdx.x * X::NB;
  const int pb = blockIdx.y * a.pg, pe = min(pb + a.pg, a.nplanes);
  img += (int64_t)blockIdx.y * M * M;
  const R* corr = static_cast<const R*>(a.corr);
  const C zero = cmake<C>(0.0, 0.0);
  R acc[X::V];
#pragma unroll
  for (int s = 0; s < X::V; ++s) acc[s] = R(0);
#pragma unroll 1
  for (int p = pb; p < pe; ++p) {
    tid = opaque_tid();
    const C* Tp = T + (int64_t)p * t_plane(a.S, M);
    C v[X::V];
#pragma unroll
    for (int s = 0; s < X::V; ++s) {
      int c, k;
      X::template slot<X::LR0>(tid, s, c, k);
      const int b = b0 + c, j = E * k - a.lo;
      C x0 = zero, x1 = zero;
      if (E == 2 && (a.lo & 1) == 0 && !a.herm) {
        if (j >= 0 && j < a.S) {
          xld_pair(Tp + t_index(j, b, M), x0, x1);
          if (j + 1 >= a.S) x1 = zero;
        }
      } else {
        auto ld = [&](int jj) -> C {
          if (jj >= 0 && jj < a.S) return Tp[t_index(jj, b, M)];
          if (a.herm && jj > 0) {
            C t = Tp[t_index(L - jj, b, M)];
            t.y = -t.y;
            return t;
          }
          return zero;
        };
        x0 = ld(j);
        if constexpr (E == 2) x1 = ld(j + 1);
      }
      v[s] = x0;
      if constexpr (E == 2) stash[s * X::T] = x1;
    }
    const C* scr = a.mode == kFacPhase && a.screen ? static_cast<const C*>(a.screen) + (int64_t)p * M * M : nullptr;
    xf_run<X, R, +1, LOGF, E>(v, buf, stash, par, tw);
    const double wp = a.w0 + p * a.dw;
#pragma unroll
    for (int s = 0; s < X::V; ++s) {
      int c, n;
      X::template slot<X::LRL>(tid, s, c, n);
      const int64_t pix = (int64_t)(b0 + c) * M + ((n + M / 2) & (M - 1));
      C z = v[s];
      if constexpr (E == 2) z = stash[s * X::T] + cmul(z, half_twiddle<R, LOGF, +1>(tw, n));
      if (scr) {
        // Re(z conj(t)) with t = corr exp(-2 pi i w_p (n-1))
        const C t = scr[pix];
        acc[s] += z.x * t.x + z.y * t.y;
      } else if (a.mode == kFacPhase) {
        const C e = wscreen<R, +1>(wp, a.nm1[pix]);
        acc[s] += z.x * e.x - z.y * e.y;
      } else {
        acc[s] += z.x;
      }
    }
  }
#pragma unroll
  for (int s = 0; s < X::V; ++s) {
    int c, n;
    X::template slot<X::LRL>(tid, s, c, n);
    const int b = b0 + c, aa = (n + M / 2) & (M - 1);
    const int64_t pix = (int64_t)b * M + aa;
    R o = acc[s] * (R)scale;
    if ((aa + b) & 1) o = -o;
    if (a.mode != kFacNone && !a.screen) o *= corr[pix];
    img[pix] = accumulate ? img[pix] + o : o;
  }
}

// Rows of an FP32 zero-padded plane's inverse as one L-point transform whose
// last pass forms the cropped half only: 8 accumulators and no waiting
// sub-transform per thread, so twice the warps fit.  Grid and meaning as
// k_inv_rows.
template <int LOGL>
using CropRows = Xf<float, LOGL, 1, false, kPadWarps>;

template <int LOGL>
__global__ void __launch_bounds__((CropRows<LOGL>::T), (CropRows<LOGL>::kCtas))
    k_crop_rows(XArgs a, const float2* __restrict__ T, float* __restrict__ img, double scale, int accumulate,
                const float2* __restrict__ tw) {
  using R = float;
  using C = float2;
  using X = CropRows<LOGL>;
  constexpr int L = X::F, M = L / 2, RAD0 = 1 << X::LR0, RADL = 1 << X::LRL;
  RIX_X_SMEM
  (void)stash;
  const int b0 = blockIdx.x * X::NB;
  const int pb = blockIdx.y * a.pg, pe = min(pb + a.pg, a.nplanes);
  img += (int64_t)blockIdx.y * M * M;
  const R* corr = static_cast<const R*>(a.corr);
  R acc[16];
#pragma unroll
  for (int s = 0; s < 16; ++s) acc[s] = 0.f;
#pragma unroll 1
  for (int p = pb; p < pe; ++p) {
    tid = opaque_tid();
    const C* Tp = T + (int64_t)p * t_plane(a.S, M);
    C v[16];
#pragma unroll
    for (int it = 0; it < 16 / RAD0; ++it) {
      int c, i;
      X::template item<X::LR0>(tid, it, c, i);
      const int j0 = i - a.lo;
      const C* src = Tp + t_index(j0, b0 + c, M);
#pragma unroll
      for (int r = 0; r < RAD0; ++r) {
        const int j = j0 + r * X::IPR0;
        C& z = v[it * RAD0 + r];
        z = make_float2(0.f, 0.f);
        if ((unsigned)j < (unsigned)a.S) {
          z = src[(int64_t)r * X::IPR0 * M];
        } else if (a.herm && j > 0) {
          z = Tp[t_index(L - j, b0 + c, M)];
          z.y = -z.y;
        }
      }
    }
    xf_passes<X, R, +1, LOGL, 0>(v, buf, par, tw, tid);
    const double wp = a.w0 + p * a.dw;
    const float wh = (float)wp, wl = (float)(wp - (double)wh);
    const C* scr = a.mode == kFacPhase && a.screen ? static_cast<const C*>(a.screen) + (int64_t)p * M * M : nullptr;
#pragma unroll
    for (int it = 0; it < 16 / RADL; ++it) {
      int c, i;
      X::template item<X::LRL>(tid, it, c, i);
      const int64_t pix0 = (int64_t)(b0 + c) * M + i;
#pragma unroll
      for (int r = 0; r < RADL; ++r) {
        if (!ct_outer<RADL>(r)) continue;
        const int64_t pix = pix0 + fold<X::LRL, L>(r);
        const C z = v[it * RADL + r];
        R& o = acc[it * RADL + r];
        if (scr) {
          // Re(z conj(t)) with t = corr exp(-2 pi i w_p (n-1))
          const C t = scr[pix];
          o += z.x * t.x + z.y * t.y;
        } else if (a.mode == kFacPhase) {
          const C e = wscreen_ff<+1>(wh, wl, a.nm1f[pix]);
          o += z.x * e.x - z.y * e.y;
        } else {
          o += z.x;
        }
      }
    }
  }
#pragma unroll
  for (int it = 0; it < 16 / RADL; ++it) {
    int c, i;
    X::template item<X::LRL>(tid, it, c, i);
    const int64_t pix0 = (int64_t)(b0 + c) * M + i;
    const bool odd = (i + b0 + c) & 1;
#pragma unroll
    for (int r = 0; r < RADL; ++r) {
      if (!ct_outer<RADL>(r)) continue;
      const int64_t pix = pix0 + fold<X::LRL, L>(r);
      R o = acc[it * RADL + r] * (R)scale;
      if (odd) o = -o;
      if (a.mode != kFacNone && !a.screen) o *= corr[pix];
      img[pix] = accumulate ? img[pix] + o : o;
    }
  }
}

// The same for the columns; CPT adjacent columns per thread in turn (as
// k_pad_cols), the first ones' results kept in shared memory until they are
// written to T together.
template <int LOGL>
__global__ void __launch_bounds__((PadCols<LOGL>::T), (PadCols<LOGL>::kCtas))
    k_crop_cols(XArgs a, const float2* __restrict__ spec, int op, const void* tab, float2* __restrict__ T,
                const float2* __restrict__ tw) {
  using R = float;
  using C = float2;
  using X = PadCols<LOGL>;
  constexpr int L = X::F, M = L / 2, CPT = X::CPT, RAD0 = 1 << X::LR0, RADL = 1 << X::LRL;
  static_assert(CPT <= 2, "pairs of columns");
  RIX_X_SMEM
  const int p = blockIdx.y, j0 = blockIdx.x * X::NB * CPT;
  const C* sp = spec + (int64_t)p * a.S * a.S;
  C* Tp = T + (int64_t)p * t_plane(a.S, M);
#pragma unroll 1
  for (int q = 0; q < CPT; ++q) {
    tid = opaque_tid();
    C v[16];
#pragma unroll
    for (int it = 0; it < 16 / RAD0; ++it) {
      int c, i;
      X::template item<X::LR0>(tid, it, c, i);
      const int j = j0 + c * CPT + q, i0 = i - a.lo;
      const int64_t e0 = (int64_t)j * a.S + i0;
#pragma unroll
      for (int r = 0; r < RAD0; ++r)
        v[it * RAD0 + r] = j < a.S && (unsigned)(i0 + r * X::IPR0) < (unsigned)a.S
                               ? xspec_op<R>(op, sp[e0 + r * X::IPR0], tab, e0 + r * X::IPR0)
                               : make_float2(0.f, 0.f);
    }
    xf_passes<X, R, +1, LOGL, 0>(v, buf, par, tw, tid);
    int live = 0;
#pragma unroll
    for (int it = 0; it < 16 / RADL; ++it) {
      int c, i;
      X::template item<X::LRL>(tid, it, c, i);
      const int j = j0 + c * CPT;
      C* o = Tp + t_index(j, i, M);
#pragma unroll
      for (int r = 0; r < RADL; ++r) {
        if (!ct_outer<RADL>(r)) continue;
        const C z = v[it * RADL + r];
        if (CPT == 2 && q == 0) {
          stash[live * X::T] = z;
        } else if (j < a.S) {
          // a second column past S falls in the block's padding
          C* d = o + fold<X::LRL, L>(r) * kTBlk;
          if constexpr (CPT == 2) xst_pair(d, stash[live * X::T], z);
          else d[0] = z;
        }
        ++live;
      }
    }
  }
}

// ------------------------------------------------------------------- host ----
template <typename R>
constexpr int kMaxLogL = sizeof(R) == 4 ? 13 : 12;   // longest transform
constexpr int kMinLogF = 5;

inline XArgs x_args(const XformGeom& g) {
  XArgs a{};
  a.M = g.M; a.L = g.L; a.lo = g.lo; a.S = g.S; a.nplanes = g.nplanes; a.mode = g.mode; a.herm = g.herm;
  a.corr = g.corr; a.nm1 = g.nm1; a.nm1f = g.nm1f; a.w0 = g.w0; a.dw = g.dw; a.screen = g.screen;
  a.pg = g.pg > 0 ? g.pg : g.nplanes;
  return a;
}

template <typename R>
int check_geom(const XformGeom& g) {
  if ((1 << g.logL) != g.L || (g.M != g.L && 2 * g.M != g.L) || g.M < (1 << kMinLogF) || g.logL > kMaxLogL<R> ||
      g.lo < 0 || g.S <= 0 || g.lo + g.S > g.L || g.nplanes <= 0)
    return set_error(RIX_EINVAL, "bad transform geometry (M=%d L=%d lo=%d S=%d)", g.M, g.L, g.lo, g.S);
  return RIX_OK;
}

// ... and, for a row pass, the tables its pixel factors come from: the screen
// table, or corr with n - 1 in the form that the pass reads
template <typename R>
int check_rows(const XformGeom& g, bool inverse) {
  RIX_TRY(check_geom<R>(g));
  if (g.mode == kFacNone || (g.mode == kFacPhase && g.screen)) return RIX_OK;
  const bool pairs = sizeof(R) == 4 && inverse && g.M != g.L;
  if (!g.corr || (g.mode == kFacPhase && (pairs ? !g.nm1f : !g.nm1)))
    return set_error(RIX_EINVAL, "transform rows without their factor tables");
  return RIX_OK;
}

// calls f(LOGF) with the transform length's log2 as a compile-time constant
template <int LO, int HI, class Fn>
int with_log(int logf, const Fn& f) {
  if constexpr (LO <= HI) {
    if (logf == LO) return f(std::integral_constant<int, LO>{});
    return with_log<LO + 1, HI>(logf, f);
  } else {
    return set_error(RIX_EINVAL, "transform length 2^%d not supported", logf);
  }
}

// dispatch on (log2 of the sub-transform length, sub-transforms)
template <typename R, class Fn>
int with_shape(const XformGeom& g, const Fn& f) {
  if (g.M == g.L)
    return with_log<kMinLogF + 1, kMaxLogL<R>>(g.logL, [&](auto lf) { return f(lf, std::integral_constant<int, 1>{}); });
  return with_log<kMinLogF, kMaxLogL<R> - 1>(g.logL - 1, [&](auto lf) { return f(lf, std::integral_constant<int, 2>{}); });
}

// the same for the row and column passes, whose FP32 zero-padded planes go
// through k_pad_* and k_crop_*
template <typename R, class Fn>
int with_plane_shape(const XformGeom& g, const Fn& f) {
  if constexpr (sizeof(R) == 4)
    return with_log<kMinLogF + 1, kMaxLogL<R>>(g.logL, [&](auto lf) { return f(lf, std::integral_constant<int, 1>{}); });
  else
    return with_shape<R>(g, f);
}

template <class X, class K, class... Args>
int x_launch(K kern, dim3 grid, cudaStream_t st, Args... args) {
  if constexpr (X::kSmem > 48 * 1024)
    RIX_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)X::kSmem));
  timing_mark(kTimeFft, st, true);
  kern<<<grid, X::T, X::kSmem, st>>>(args...);
  ::rix::note_launch();
  timing_mark(kTimeFft, st, false);
  RIX_LAUNCH_CHECK();
  return RIX_OK;
}

}  // namespace
}  // namespace rix
