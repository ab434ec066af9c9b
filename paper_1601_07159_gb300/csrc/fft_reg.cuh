// Register-resident mixed-radix DFTs (radices 2, 3, 4, 5) for one thread.
//
// A thread holds a whole line of N complex values in registers and transforms
// it with a fully unrolled decimation-in-time recursion: N = R * M, R sub-DFTs
// of length M over the decimated inputs a[r + R m], twiddles w_N^{r k}, then a
// radix-R butterfly across r. All indices are compile-time constants after
// unrolling, so the values stay in registers and the twiddles come from the
// kernel's constant parameter bank (a table of w_NTOP^k = exp(-2 pi i k/NTOP)
// for k < NTOP, computed on the host in FP64 from sin/cos). Exact quarter
// turns (w = 1, -i, -1, i) are applied as swaps, not multiplications.
//
// This is the Poisson solver's transform (Sec. 2: each solve is
// O(N_g log N_g) with FFTs); the 3-D transform is built from these line
// transforms in pair_kernels.cu.
//
// Radix order, fixed per translation unit by ACE_RADIX_ORDER: 0 (default)
// takes a radix 4 first, then 2, 3, 5; 1 takes the odd radix (3, then 5)
// first when the length has one, so 48 = 3 x 16 instead of 4 x 12 (other
// twiddle sets, other instruction schedules). The code of each order sits in
// its own inline namespace, so instances of both orders link into one library.
#pragma once
#include <cuda_runtime.h>

#ifndef ACE_RADIX_ORDER
#define ACE_RADIX_ORDER 0
#endif
#if ACE_RADIX_ORDER == 0
#define ACE_RADIX_NS radix0
#elif ACE_RADIX_ORDER == 1
#define ACE_RADIX_NS radix1
#else
#error "ACE_RADIX_ORDER must be 0 or 1"
#endif

namespace ace {
inline namespace ACE_RADIX_NS {

template <typename R> struct cplx_t;
template <> struct cplx_t<float> { using type = float2; };
template <> struct cplx_t<double> { using type = double2; };
template <typename R> using cplx = typename cplx_t<R>::type;

template <typename T> __device__ __forceinline__ T cmk(decltype(T::x) x, decltype(T::x) y) {
  T r; r.x = x; r.y = y; return r;
}
// Sums and differences of FP32 values as one packed instruction on the (re, im)
// pair (the same rounding per component; the FP32 lane rate does not change, the
// issue slots halve). PK = false keeps two scalar additions (a kernel that
// measures faster with them asks for it). Products stay scalar: w x mixes the two
// halves, and the packed form needs as many instructions once the swap is counted.
template <bool PK = true, typename T> __device__ __forceinline__ T cadd(T a, T b) {
  if constexpr (PK && sizeof(T) == sizeof(float2)) return __fadd2_rn(a, b);
  else return cmk<T>(a.x + b.x, a.y + b.y);
}
template <bool PK = true, typename T> __device__ __forceinline__ T csub(T a, T b) {
  if constexpr (PK && sizeof(T) == sizeof(float2)) return __fadd2_rn(a, make_float2(-b.x, -b.y));
  else return cmk<T>(a.x - b.x, a.y - b.y);
}
template <typename T> __device__ __forceinline__ T cmul(T a, T b) {
  return cmk<T>(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
// conj(a) * b
template <typename T> __device__ __forceinline__ T cmulc(T a, T b) {
  return cmk<T>(a.x * b.x + a.y * b.y, a.x * b.y - a.y * b.x);
}
template <typename T> __device__ __forceinline__ T cscale(T a, decltype(T::x) s) { return cmk<T>(a.x * s, a.y * s); }
// a + s t
template <bool PK = true, typename T> __device__ __forceinline__ T caxpy(T a, decltype(T::x) s, T t) {
  if constexpr (PK && sizeof(T) == sizeof(float2)) return __ffma2_rn(t, make_float2(s, s), a);
  else return cmk<T>(a.x + s * t.x, a.y + s * t.y);
}
// acc + a b and acc + conj(a) b as four fused multiply-adds (accumulations)
template <typename T> __device__ __forceinline__ T cfma(T acc, T a, T b) {
  acc.x = fma(a.x, b.x, acc.x);
  acc.x = fma(-a.y, b.y, acc.x);
  acc.y = fma(a.x, b.y, acc.y);
  acc.y = fma(a.y, b.x, acc.y);
  return acc;
}
template <typename T> __device__ __forceinline__ T cfmac(T acc, T a, T b) {
  acc.x = fma(a.x, b.x, acc.x);
  acc.x = fma(a.y, b.y, acc.x);
  acc.y = fma(a.x, b.y, acc.y);
  acc.y = fma(-a.y, b.x, acc.y);
  return acc;
}
// multiply by -i (forward) or +i (inverse) -> "rotate by the forward quarter turn"
template <bool INV, typename T> __device__ __forceinline__ T rot_q(T a) {
  return INV ? cmk<T>(-a.y, a.x) : cmk<T>(a.y, -a.x);
}

template <typename R, int NTOP> struct TwTable { cplx<R> w[NTOP]; };

// w_N^e (forward sign), or its conjugate for the inverse transform, applied to x.
template <int N, int NTOP, bool INV, typename R>
__device__ __forceinline__ cplx<R> twiddle(cplx<R> x, int e, const TwTable<R, NTOP>& tw) {
  e %= N;
  if (e == 0) return x;
  if ((4 * e) % N == 0) {
    const int q = (4 * e) / N;             // quarter turns
    if (q == 1) return rot_q<INV>(x);
    if (q == 2) return cmk<cplx<R>>(-x.x, -x.y);
    return rot_q<!INV>(x);
  }
  const cplx<R> w = tw.w[e * (NTOP / N)];
  return INV ? cmk<cplx<R>>(x.x * w.x + x.y * w.y, x.y * w.x - x.x * w.y)   // x * conj(w)
             : cmul(x, w);
}

// The twiddle w_N^e (forward sign) or its conjugate as a value: exact for the
// quarter turns, from the table otherwise. With e a compile-time constant after
// unrolling this is a pair of constants.
template <int N, int NTOP, bool INV, typename R>
__device__ __forceinline__ cplx<R> twiddle_value(int e, const TwTable<R, NTOP>& tw) {
  e %= N;
  if (e == 0) return cmk<cplx<R>>(R(1), R(0));
  if ((4 * e) % N == 0) {
    const int q = (4 * e) / N;   // forward: -i, -1, +i
    if (q == 2) return cmk<cplx<R>>(R(-1), R(0));
    const R s = (q == 1) != INV ? R(-1) : R(1);
    return cmk<cplx<R>>(R(0), s);
  }
  const cplx<R> w = tw.w[e * (NTOP / N)];
  return INV ? cmk<cplx<R>>(w.x, -w.y) : w;
}

// s = a + w b and d = a - w b with w = w_N^e (conjugated for the inverse), as six
// fused operations: s by four, d = 2 a - s by two, instead of four for the
// product and four sums. The FP64 passes are bound by the FP64 pipe, so they
// gain what they save: passes A, B, C of a 64-pair tile 581, 488, 518 -> 545, 452,
// 483 us at 48^3 (FP32 pair additions are one packed instruction each).
// d carries s's rounding beside its own: line transforms of 8 to 96 points have 0.2 to 1.4 %
// more rms error (against long double, 1.0 to 3.5e-16) than with four sums, which the
// error of a build does not show (32^3, N = 27: 3.7 and 4.1e-16 before, 4.0 and 4.0e-16
// so, two sets of orbitals). d by its own four operations costs a build 5.5 %.
template <int N, int NTOP, bool INV, typename R>
__device__ __forceinline__ void tw_sum_diff(cplx<R> a, cplx<R> b, int e, const TwTable<R, NTOP>& tw, cplx<R>& s,
                                            cplx<R>& d) {
  e %= N;
  if ((4 * e) % N == 0) {
    const cplx<R> t = twiddle<N, NTOP, INV, R>(b, e, tw);
    s = cadd(a, t);
    d = csub(a, t);
    return;
  }
  const cplx<R> w = twiddle_value<N, NTOP, INV, R>(e, tw);
  s = cmk<cplx<R>>(fma(-w.y, b.y, fma(w.x, b.x, a.x)), fma(w.y, b.x, fma(w.x, b.y, a.y)));
  d = cmk<cplx<R>>(fma(R(2), a.x, -s.x), fma(R(2), a.y, -s.y));
}

template <int N> __host__ __device__ constexpr int first_radix() {
  if constexpr (ACE_RADIX_ORDER == 1 && N % 3 == 0 && N != 3) return 3;
  if constexpr (ACE_RADIX_ORDER == 1 && N % 5 == 0 && N != 5) return 5;
  return (N % 4 == 0 && N != 4) ? 4 : (N % 2 == 0 ? 2 : (N % 3 == 0 ? 3 : (N % 5 == 0 ? 5 : N)));
}

template <int N, int NTOP, bool INV, typename R, bool PK = true>
__device__ __forceinline__ void dft(cplx<R> (&a)[N], const TwTable<R, NTOP>& tw);

template <int NTOP, bool INV, typename R, bool PK>
__device__ __forceinline__ void bfly2(cplx<R> (&a)[2]) {
  const cplx<R> t = a[0];
  a[0] = cadd<PK>(t, a[1]);
  a[1] = csub<PK>(t, a[1]);
}

template <int NTOP, bool INV, typename R, bool PK>
__device__ __forceinline__ void bfly4(cplx<R> (&a)[4]) {
  const cplx<R> s02 = cadd<PK>(a[0], a[2]), d02 = csub<PK>(a[0], a[2]);
  const cplx<R> s13 = cadd<PK>(a[1], a[3]), d13 = rot_q<INV>(csub<PK>(a[1], a[3]));
  a[0] = cadd<PK>(s02, s13);
  a[2] = csub<PK>(s02, s13);
  a[1] = cadd<PK>(d02, d13);
  a[3] = csub<PK>(d02, d13);
}

// radix 3: X1,2 = a0 + c (a1 + a2) -/+ i s (a1 - a2) with w_3 = c - i s (forward)
template <int NTOP, bool INV, typename R, bool PK>
__device__ __forceinline__ void bfly3(cplx<R> (&a)[3], const TwTable<R, NTOP>& tw) {
  const cplx<R> w3 = tw.w[NTOP / 3];
  const R c = w3.x, s = -w3.y;
  const cplx<R> t = cadd<PK>(a[1], a[2]);
  const cplx<R> d = cscale(csub<PK>(a[1], a[2]), s);
  const cplx<R> u = caxpy<PK>(a[0], c, t);
  a[0] = cadd<PK>(a[0], t);
  const cplx<R> rd = rot_q<INV>(d);
  a[1] = cadd<false>(u, rd);   // scalar: s (a1 - a2) and the sum are one FMA each
  a[2] = csub<false>(u, rd);
}

// radix 5 with c1 = cos 2pi/5, c2 = cos 4pi/5, s1 = sin 2pi/5, s2 = sin 4pi/5
template <int NTOP, bool INV, typename R, bool PK>
__device__ __forceinline__ void bfly5(cplx<R> (&a)[5], const TwTable<R, NTOP>& tw) {
  const cplx<R> w1 = tw.w[NTOP / 5], w2 = tw.w[2 * NTOP / 5];
  const R c1 = w1.x, s1 = -w1.y, c2 = w2.x, s2 = -w2.y;
  const cplx<R> t1 = cadd<PK>(a[1], a[4]), t2 = cadd<PK>(a[2], a[3]);
  const cplx<R> t3 = csub<PK>(a[1], a[4]), t4 = csub<PK>(a[2], a[3]);
  const cplx<R> b1 = cmk<cplx<R>>(a[0].x + c1 * t1.x + c2 * t2.x, a[0].y + c1 * t1.y + c2 * t2.y);
  const cplx<R> b2 = cmk<cplx<R>>(a[0].x + c2 * t1.x + c1 * t2.x, a[0].y + c2 * t1.y + c1 * t2.y);
  const cplx<R> e1 = rot_q<INV>(cmk<cplx<R>>(s1 * t3.x + s2 * t4.x, s1 * t3.y + s2 * t4.y));
  const cplx<R> e2 = rot_q<INV>(cmk<cplx<R>>(s2 * t3.x - s1 * t4.x, s2 * t3.y - s1 * t4.y));
  a[0] = cadd<PK>(a[0], cadd<PK>(t1, t2));
  a[1] = cadd<PK>(b1, e1);
  a[4] = csub<PK>(b1, e1);
  a[2] = cadd<PK>(b2, e2);
  a[3] = csub<PK>(b2, e2);
}

template <int N, int NTOP, bool INV, typename R, bool PK>
__device__ __forceinline__ void dft(cplx<R> (&a)[N], const TwTable<R, NTOP>& tw) {
  static_assert(NTOP % N == 0, "sub-length must divide the table length");
  if constexpr (N == 1) {
    return;
  } else if constexpr (N == 2) {
    bfly2<NTOP, INV, R, PK>(a);
  } else if constexpr (N == 3) {
    bfly3<NTOP, INV, R, PK>(a, tw);
  } else if constexpr (N == 4) {
    bfly4<NTOP, INV, R, PK>(a);
  } else if constexpr (N == 5) {
    bfly5<NTOP, INV, R, PK>(a, tw);
  } else {
    constexpr int RX = first_radix<N>();
    static_assert(RX != N, "unsupported prime factor");
    constexpr int M = N / RX;
    cplx<R> sub[RX][M];
#pragma unroll
    for (int r = 0; r < RX; ++r)
#pragma unroll
      for (int m = 0; m < M; ++m) sub[r][m] = a[r + RX * m];
#pragma unroll
    for (int r = 0; r < RX; ++r) dft<M, NTOP, INV, R, PK>(sub[r], tw);
#pragma unroll
    for (int k = 0; k < M; ++k) {
      cplx<R> t[RX];
      if constexpr (sizeof(R) == 8 && (RX == 2 || RX == 4)) {   // FP64: twiddles fused into the butterfly
        if constexpr (RX == 2) {
          tw_sum_diff<N, NTOP, INV, R>(sub[0][k], sub[1][k], k, tw, t[0], t[1]);
        } else {
          cplx<R> s02, d02, s13, d13;
          tw_sum_diff<N, NTOP, INV, R>(sub[0][k], sub[2][k], 2 * k, tw, s02, d02);
          tw_sum_diff<N, NTOP, INV, R>(twiddle<N, NTOP, INV, R>(sub[1][k], k, tw), sub[3][k], 3 * k, tw, s13, d13);
          d13 = rot_q<INV>(d13);
          t[0] = cadd(s02, s13);
          t[2] = csub(s02, s13);
          t[1] = cadd(d02, d13);
          t[3] = csub(d02, d13);
        }
      } else {
#pragma unroll
        for (int r = 0; r < RX; ++r) t[r] = twiddle<N, NTOP, INV, R>(sub[r][k], r * k, tw);
        dft<RX, NTOP, INV, R, PK>(t, tw);
      }
#pragma unroll
      for (int q = 0; q < RX; ++q) a[k + M * q] = t[q];
    }
  }
}

// A whole line in one thread by a radix-2 step over the even and odd samples:
// the operations of the two-lane form (split_line_dft), in the same order, so
// the two give the same bits.
template <int N, bool INV, typename R>
__device__ __forceinline__ void line_dft2(cplx<R> (&a)[N], const TwTable<R, N>& tw) {
  constexpr int M = N / 2;
  cplx<R> e[M], o[M];
#pragma unroll
  for (int m = 0; m < M; ++m) {
    e[m] = a[2 * m];
    o[m] = a[2 * m + 1];
  }
  dft<M, N, INV, R>(e, tw);
  dft<M, N, INV, R>(o, tw);
#pragma unroll
  for (int k = 0; k < M; ++k) {
    const cplx<R> t = k == 0 ? o[k] : 4 * k == N ? rot_q<INV>(o[k]) : cmul(o[k], twiddle_value<N, N, INV, R>(k, tw));
    a[k] = cadd(e[k], t);
    a[k + M] = csub(e[k], t);
  }
}

}  // namespace ACE_RADIX_NS
}  // namespace ace
