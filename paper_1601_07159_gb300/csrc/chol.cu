// FP64 Cholesky factorisation of -M and the inverse of its factor (Sec. 3:
// -M = L L^*, then Xi = W L^{-*} of Eq. Wtilde), blocked so that the FP64 work
// spreads over many SMs (FP64 throughput per SM is low on this part).
//
// Blocks of NB = 16 columns (the diagonal blocks run on one SM each, so they
// are kept small; 32 measured slightly slower). For panel p (rows/cols
// [p0, p0 + nb)):
//   diag    one CTA: A_pp -> L_pp (status word on a non-finite or non-positive
//           pivot) and D_p = L_pp^{-1}; L_pp is stored in A, D_p in the diagonal
//           block of X.
//   panel   L_ip = A_ip D_p^*  for every row i below the panel (one CTA per 2
//           rows, in place: a CTA reads and writes only its own rows).
//   update  A_ik -= sum_l L_il conj(L_kl) over the panel columns l, for the
//           trailing lower triangle i >= k (8 x 8 output tiles).
// Then X = L^{-1} below the diagonal blocks by recursive doubling: with
// [[A, 0], [B, C]] the blocks of edge h = 16, 32, ... of L,
//   T = B A^{-1}, then X_B = -C^{-1} T
// for all pairs of a level at once: 2 log2(n / 16) launches.
// Finally LinvH[c][i] = conj(X_ic) (zero above the diagonal), so that
// Xi_k = sum_i W_i LinvH[i][k].
// FP64 issue bounds each of these kernels (about 1.7 multiply-adds per cycle and SM: 75
// cycles per warp instruction and SM quadrant), and at 128 orbitals and fewer its latency: outputs are
// spread over as many SMs as there are (2-row panels and 8 x 8 tiles in place of 16 rows
// and 16 x 16), sums are cut in parts that meet by shuffles, and dependent steps
// are few. Kernel times for 128 orbitals: 392 -> 239 us (diag 8 x 22.4 -> 14.2, panel 8.1 ->
// 4.9, update 8.2 -> 5.2, the inverse from 7 row steps of 12.9 to 3 levels of 16.0).
// Every kernel returns at once when the status word already holds a failure.
#include <cmath>

#include "ace_internal.h"

namespace ace {

namespace {

constexpr int NB = 16;   // panel width
constexpr int TT = 8;    // output tile edge of the FP64 tile products

__device__ __forceinline__ double2 zfma(double2 acc, double2 a, double2 b) {   // acc + a b
  acc.x = fma(a.x, b.x, acc.x);
  acc.x = fma(-a.y, b.y, acc.x);
  acc.y = fma(a.x, b.y, acc.y);
  acc.y = fma(a.y, b.x, acc.y);
  return acc;
}
__device__ __forceinline__ double2 zfmac(double2 acc, double2 a, double2 b) {  // acc + a conj(b)
  acc.x = fma(a.x, b.x, acc.x);
  acc.x = fma(a.y, b.y, acc.x);
  acc.y = fma(a.y, b.x, acc.y);
  acc.y = fma(-a.x, b.y, acc.y);
  return acc;
}

__global__ void neg_copy_kernel(const double2* __restrict__ M, long long count, double2* __restrict__ A) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < count) A[i] = make_double2(-M[i].x, -M[i].y);
}

// d positive and finite, from its words (a comparison of doubles costs as much as a
// multiply-add).
__device__ __forceinline__ bool positive_finite(double d) {
  const unsigned hi = (unsigned)__double2hiint(d);
  return hi < 0x7ff00000u && (hi | (unsigned)__double2loint(d)) != 0u;
}

// a - |u|^2 r, with one dependent operation after r where |u|^2 cannot leave the range of
// doubles (the larger component's exponent in [-480, 480)), else by products with u r.
__device__ __forceinline__ double minus_abs2(double a, double2 u, double r) {
  const int e = max(__double2hiint(u.x) & 0x7fffffff, __double2hiint(u.y) & 0x7fffffff) >> 20;
  if ((unsigned)(e - (1023 - 480)) < 960u) return fma(-fma(u.x, u.x, u.y * u.y), r, a);
  return fma(-u.y * r, u.y, fma(-u.x * r, u.x, a));
}

// Factor and invert the diagonal block of panel p (nb <= NB). The block is padded to
// NB with the identity, so every loop runs NB uniform steps.
// Elimination on unscaled columns, -M = L' D L'^*: step j subtracts
// (a_ij / d_j) conj(a_kj) from the trailing a_ik (i >= k > j) and (a_ij / d_j) x_jc from
// row i of X = L'^{-1} (c <= j, X starts as the identity): row i has i + 1
// elements in every step. So each lower-triangle element (i, k) has one thread, which
// holds a_ik in a register up to step k, where it is final, and x_ik from
// there on. A step reads column j of a and row j of x, published in shared memory by
// the step before (two buffers, one barrier a step). Warp PIV works ahead on the
// pivot: d_{j+1} = a_{j+1,j+1} - |a_{j+1,j}|^2 / d_j and its reciprocal, while the
// others do step j (with the pivot taken from its element's thread and the inverse
// formed afterwards, by recursive doubling, the kernel took 22.4 us; 14.2 so). What it
// leaves for a step (the pivot's reciprocal and verdict) lies in the word of that
// step's parity, which no thread reads before the barrier.
// At the end L_ik = a_ik / sqrt(d_k), and row i of X is divided by sqrt(d_i). Reciprocals
// and roots are CUDA's division and square root, correctly rounded.
constexpr int kTri = NB * (NB + 1) / 2;             // lower-triangle elements
constexpr int PIV = (kTri + 31) / 32;               // the pivot's warp, after the elements'
__global__ void __launch_bounds__((PIV + 1) * 32)
diag_kernel(double2* __restrict__ A, double2* __restrict__ X, int n, int p0, int nb, int* status) {
  __shared__ double2 col[2][NB], row[2][NB];        // a_ij (i > j) and x_jc (c <= j) of step j
  __shared__ double dg[2], rj[2];                   // a_{j+1,j+1} before step j, 1 / d_j
  __shared__ double dd[NB], y[NB];                  // d_j, then its root; 1 / sqrt(d_j)
  __shared__ int fail[2];                           // status code of pivot j at j & 1 (0: good)
  const int tid = threadIdx.x, w = tid >> 5;
  if (status[0] != 0) return;
  // element (i, k) of thread tid: rows in decreasing order, so that the elements of a
  // step are the first threads
  int i = NB - 1, k = tid;
  while (k > i && i >= 0) k -= i-- + 1;
  const bool elem = tid < kTri;
  double2 v = make_double2(0.0, 0.0);
  if (elem) {
    v = make_double2(i == k ? 1.0 : 0.0, 0.0);
    if (i < nb) v = A[(long long)(p0 + i) * n + p0 + k];
    if (k == 0) col[0][i] = v;
    if (i == 1 && k == 1) dg[0] = v.x;
  }
  auto pivot = [&](int j, double d) {               // lane 0 of warp PIV: check d_j, keep it and its reciprocal
    const bool ok = positive_finite(d);
    dd[j] = d;
    fail[j & 1] = ok ? 0 : isfinite(d) ? -2 : -3;
    if (ok) rj[j & 1] = 1.0 / d;
  };
  if (tid == 0) row[0][0] = make_double2(1.0, 0.0);
  __syncthreads();
  if (tid == PIV * 32) pivot(0, col[0][0].x);
  __syncthreads();
  double2 l = v;                                    // a_ik once it is final
  for (int j = 0; j < NB; ++j) {
    const int c = j & 1;
    // pivot j's word: written in the step before; this step writes the other one
    if (fail[c]) {
      if (tid == 0) {
        status[0] = fail[c];
        status[1] = p0 + j + 1;
      }
      return;
    }
    const double r = rj[c];
    if (w == PIV) {
      if (tid == PIV * 32 && j + 1 < NB) {
        const double2 u = col[c][j + 1];
        pivot(j + 1, minus_abs2(dg[c], u, r));
      }
    } else if (elem && i > j) {
      if (k == j) {                                 // a_ij is final: on to x_ij, which starts at zero
        l = v;
        v = make_double2(0.0, 0.0);
      }
      const double2 u = col[c][i];
      double2 z = k > j ? col[c][k] : row[c][k];
      if (k > j) z.y = -z.y;
      v = zfma(v, make_double2(-u.x * r, -u.y * r), z);
      if (k == j + 1) col[c ^ 1][i] = v;
      if (i == j + 1) row[c ^ 1][k] = k == i ? make_double2(1.0, 0.0) : v;
      if (i == j + 2 && k == i) dg[c ^ 1] = v.x;
    }
    __syncthreads();
  }
  if (tid < NB) {
    dd[tid] = sqrt(dd[tid]);
    y[tid] = 1.0 / dd[tid];
  }
  __syncthreads();
  if (!elem || i >= nb) return;
  const double yi = y[i], yk = y[k];
  const long long o = (long long)(p0 + i) * n + p0 + k;
  if (i == k) {
    A[o] = make_double2(dd[i], 0.0);
    X[o] = make_double2(yi, 0.0);
  } else {
    A[o] = make_double2(l.x * yk, l.y * yk);
    X[o] = make_double2(v.x * yi, v.y * yi);
  }
}

// L_ip = A_ip D_p^* for rows i in [r0, n): PR rows and all nb columns per CTA, four
// threads per output.
constexpr int PR = 2;
__global__ void __launch_bounds__(PR * NB * 4)
panel_kernel(double2* __restrict__ A, const double2* __restrict__ X, int n, int p0, int nb, int r0,
             const int* status) {
  __shared__ double2 rows[PR][NB + 1];
  __shared__ double2 d[NB][NB + 1];
  if (status[0] != 0) return;
  const int tid = threadIdx.x;
  const int i0 = r0 + blockIdx.x * PR;
  for (int e = tid; e < PR * NB; e += blockDim.x) {
    const int i = e / NB, k = e % NB;
    rows[i][k] = (i0 + i < n && k < nb) ? A[(long long)(i0 + i) * n + p0 + k] : make_double2(0.0, 0.0);
  }
  for (int e = tid; e < NB * NB; e += blockDim.x) {
    const int i = e / NB, k = e % NB;
    d[i][k] = (i < nb && k <= i) ? X[(long long)(p0 + i) * n + p0 + k] : make_double2(0.0, 0.0);
  }
  __syncthreads();
  const int part = tid & 3, c = (tid >> 2) % NB, i = (tid >> 2) / NB;
  double2 s = make_double2(0.0, 0.0);
#pragma unroll
  for (int k = 0; k < NB; k += 4) s = zfmac(s, rows[i][k + part], d[c][k + part]);   // sum_k A_ik conj(D_ck)
#pragma unroll
  for (int o = 1; o < 4; o *= 2) {
    s.x += __shfl_xor_sync(0xffffffffu, s.x, o);
    s.y += __shfl_xor_sync(0xffffffffu, s.y, o);
  }
  if (part == 0 && i0 + i < n && c < nb) A[(long long)(i0 + i) * n + p0 + c] = s;
}

// A_ik -= sum_{l in panel} L_il conj(L_kl), trailing lower triangle i >= k >= r0.
// Grid: one CTA per lower 8 x 8 tile (bi >= bk) of the trailing block, two threads
// per output.
__global__ void __launch_bounds__(2 * TT * TT)
update_kernel(double2* __restrict__ A, int n, int p0, int nb, int r0, const int* status) {
  __shared__ double2 li[TT][NB + 1];
  __shared__ double2 lk[TT][NB + 1];
  if (status[0] != 0) return;
  // bi (bi + 1) / 2 <= blockIdx.x < (bi + 1) (bi + 2) / 2
  int bi = (int)((sqrtf(8.f * (float)blockIdx.x + 1.f) - 1.f) * 0.5f);
  while (bi * (bi + 1) / 2 > (int)blockIdx.x) --bi;
  while ((bi + 1) * (bi + 2) / 2 <= (int)blockIdx.x) ++bi;
  const int bk = (int)blockIdx.x - bi * (bi + 1) / 2;
  const int i0 = r0 + bi * TT, k0 = r0 + bk * TT;
  const int tid = threadIdx.x;
  for (int e = tid; e < TT * NB; e += blockDim.x) {
    const int r = e / NB, c = e % NB;
    const bool okc = c < nb;
    li[r][c] = (okc && i0 + r < n) ? A[(long long)(i0 + r) * n + p0 + c] : make_double2(0.0, 0.0);
    lk[r][c] = (okc && k0 + r < n) ? A[(long long)(k0 + r) * n + p0 + c] : make_double2(0.0, 0.0);
  }
  __syncthreads();
  const int part = tid & 1, r = (tid >> 1) / TT, c = (tid >> 1) % TT;
  double2 s = make_double2(0.0, 0.0);
#pragma unroll
  for (int l = 0; l < NB; l += 2) s = zfmac(s, li[r][l + part], lk[c][l + part]);
  s.x += __shfl_xor_sync(0xffffffffu, s.x, 1);
  s.y += __shfl_xor_sync(0xffffffffu, s.y, 1);
  const int i = i0 + r, k = k0 + c;
  if (part != 0 || i >= n || k >= n || k > i) return;
  double2& out = A[(long long)i * n + k];
  out = make_double2(out.x - s.x, out.y - s.y);
}

// One product of a doubling level, for the pair blockIdx.z of blocks of edge h at rows
// and columns s = 2 h blockIdx.z; 8 x 8 outputs (r, c) per CTA, two threads each. The
// intermediate T(r, c) lies transposed in the unused upper triangle, at X(s + c, s + h + r).
//   FIRST:  T(r, c) = sum_{m >= c} L(s + h + r, s + m) X(s + m, s + c)
//   second: X(s + h + r, s + c) = -sum_{m <= r} X(s + h + r, s + h + m) T(m, c)
template <bool FIRST>
__global__ void __launch_bounds__(2 * TT * TT)
inv_level_kernel(const double2* __restrict__ A, double2* __restrict__ X, int n, int h, const int* status) {
  __shared__ double2 f[TT][NB + 1];                 // rows r of the left factor
  __shared__ double2 g[TT][NB + 1];                 // columns c of the right factor
  if (status[0] != 0) return;
  const int s = 2 * h * blockIdx.z, r0 = blockIdx.y * TT, c0 = blockIdx.x * TT, lo = s + h;
  if (lo + r0 >= n) return;
  const int tid = threadIdx.x, part = tid & 1, r = (tid >> 1) / TT, c = (tid >> 1) % TT;
  const int rows = min(h, n - lo);                  // of the pair's lower block
  const int m0 = FIRST ? c0 : 0, m1 = FIRST ? h : min(r0 + TT, rows);
  double2 acc = make_double2(0.0, 0.0);
  for (int m = m0; m < m1; m += NB) {
    for (int e = tid; e < TT * NB; e += blockDim.x) {
      const int q = e / NB, mm = m + e % NB;
      const bool okr = r0 + q < rows && mm < m1;
      double2 u = make_double2(0.0, 0.0);
      if (FIRST) {
        if (okr) u = A[(long long)(lo + r0 + q) * n + s + mm];
      } else {
        if (okr && mm <= r0 + q) u = X[(long long)(lo + r0 + q) * n + lo + mm];
      }
      f[q][e % NB] = u;
    }
    for (int e = tid; e < TT * NB; e += blockDim.x) {
      // FIRST: rows mm of X, contiguous over c; second: T transposed, contiguous over mm
      const int q = FIRST ? e % TT : e / NB, t = FIRST ? e / TT : e % NB, mm = m + t;
      double2 u = make_double2(0.0, 0.0);
      if (mm < m1) {
        if (FIRST) {
          if (mm >= c0 + q) u = X[(long long)(s + mm) * n + s + c0 + q];
        } else {
          u = X[(long long)(s + c0 + q) * n + lo + mm];
        }
      }
      g[q][t] = u;
    }
    __syncthreads();
#pragma unroll
    for (int t = 0; t < NB; t += 2) acc = zfma(acc, f[r][t + part], g[c][t + part]);
    __syncthreads();
  }
  acc.x += __shfl_xor_sync(0xffffffffu, acc.x, 1);
  acc.y += __shfl_xor_sync(0xffffffffu, acc.y, 1);
  if (part != 0 || r0 + r >= rows) return;
  if (FIRST) X[(long long)(s + c0 + c) * n + lo + r0 + r] = acc;
  else X[(long long)(lo + r0 + r) * n + s + c0 + c] = make_double2(-acc.x, -acc.y);
}

__global__ void linvh_kernel(const double2* __restrict__ X, int n, double* __restrict__ LinvH,
                             const int* status) {
  if (status[0] != 0) return;
  const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= (long long)n * n) return;
  const int c = (int)(e / n), i = (int)(e % n);
  double2 v = make_double2(0.0, 0.0);
  if (i >= c) v = X[(long long)i * n + c];
  LinvH[2 * e] = v.x;
  LinvH[2 * e + 1] = -v.y;
}

}  // namespace

void prepare_cholesky(int) {}

size_t cholesky_work_doubles(int n) { return (size_t)4 * n * n; }

int launch_cholesky_inv(const double* M, int n, double* work, double* LinvH, int* status, cudaStream_t st) {
  double2* A = reinterpret_cast<double2*>(work);
  double2* X = A + (size_t)n * n;
  int launches = 0;
  const long long nn = (long long)n * n;
  neg_copy_kernel<<<(unsigned)((nn + 255) / 256), 256, 0, st>>>(reinterpret_cast<const double2*>(M), nn, A);
  ++launches;
  for (int p0 = 0; p0 < n; p0 += NB) {
    const int nb = (p0 + NB <= n) ? NB : n - p0;
    diag_kernel<<<1, (PIV + 1) * 32, 0, st>>>(A, X, n, p0, nb, status);
    ++launches;
    const int r0 = p0 + nb;
    if (r0 >= n) break;
    const int rows = n - r0;
    panel_kernel<<<(rows + PR - 1) / PR, PR * NB * 4, 0, st>>>(A, X, n, p0, nb, r0, status);
    const int bt = (rows + TT - 1) / TT;
    update_kernel<<<bt * (bt + 1) / 2, 2 * TT * TT, 0, st>>>(A, n, p0, nb, r0, status);
    launches += 2;
  }
  for (int h = NB; h < n; h *= 2) {
    const dim3 grid(h / TT, h / TT, (n + h - 1) / (2 * h));
    inv_level_kernel<true><<<grid, 2 * TT * TT, 0, st>>>(A, X, n, h, status);
    inv_level_kernel<false><<<grid, 2 * TT * TT, 0, st>>>(A, X, n, h, status);
    launches += 2;
  }
  linvh_kernel<<<(unsigned)((nn + 255) / 256), 256, 0, st>>>(X, n, LinvH, status);
  return launches + 1;
}

__global__ void scale_kernel_f(float* x, long long count, float s) {
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < count; i += (long long)gridDim.x * blockDim.x)
    x[i] *= s;
}
__global__ void scale_kernel_d(double* x, long long count, double s) {
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < count; i += (long long)gridDim.x * blockDim.x)
    x[i] *= s;
}

// X *= s over the first ng elements of each of `count` vectors of stride ld
// (real and imaginary parts alike): one packed run when ld == ng.
void launch_scale(bool f64, bool real, void* X, long long count, long long ng, long long ld, double s,
                  cudaStream_t st) {
  const long long per = real ? 1 : 2;   // reals per element
  const long long runs = ld == ng ? 1 : count, run = (ld == ng ? count * ng : ng) * per;
  const unsigned grid = (unsigned)((run + 255) / 256 < 152 * 16 ? (run + 255) / 256 : 152 * 16);
  for (long long v = 0; v < runs; ++v) {
    if (f64) scale_kernel_d<<<grid, 256, 0, st>>>(static_cast<double*>(X) + v * ld * per, run, s);
    else scale_kernel_f<<<grid, 256, 0, st>>>(static_cast<float*>(X) + v * ld * per, run, (float)s);
  }
}

}  // namespace ace
