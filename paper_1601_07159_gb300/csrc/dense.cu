// Dense steps of the ACE construction and apply (Sec. 3):
//   M = dV Phi^* W  (Eq. ACEconstruct2)       -> gram + gram_reduce
//   -M = L L^*, L^{-1} (FP64)                  -> cholesky_inv
//   Xi = W L^{-*}    (Eq. Wtilde)              -> outer with C = L^{-*}
//   C = dV Xi^* psi, Y = -Xi C   (Eq. ACE)     -> gram + gram_reduce, outer
//   E_x reductions (Eq. EX / EX_ACE)           -> energy_reduce, trace in gram_reduce
//
// Arrays of vectors are orbital-major [count][N_g] (x fastest); small matrices
// are row-major FP64 (complex interleaved). The GEMMs run on CUDA cores in the
// vectors' precision with a deterministic split-K reduction in FP64.
#include <algorithm>
#include <cmath>

#include "ace_internal.h"
#include "fft_reg.cuh"

namespace ace {

// ---------------------------------------------------------------- gram
// part[s][a][b] = sum_{g in chunk s} conj(A[a][g]) B[b][g]   (complex, FP64 out)
constexpr int GT = 64;   // FP32 output tile edge
constexpr int GK = 16;   // FP32 K chunk per shared-memory stage

__global__ void __launch_bounds__(256)
gram_kernel(const float2* __restrict__ A, int na, const float2* __restrict__ B, int nb, long long ld, long long ng,
            double* __restrict__ part, long long chunk) {
  __shared__ float2 As[GK][GT + 1];
  __shared__ float2 Bs[GK][GT + 1];
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  const int a0 = blockIdx.x * GT, b0 = blockIdx.y * GT;
  const long long g_begin = (long long)blockIdx.z * chunk;
  const long long g_end = g_begin + chunk < ng ? g_begin + chunk : ng;
  // this thread's rows a0 + ty + 16 i (i < ni) and columns b0 + tx + 16 j (j < nj)
  // inside the matrix: small matrices do no work on the tile's padding
  const int ra = na - a0 - ty, rb = nb - b0 - tx;
  const int ni = ra <= 0 ? 0 : (ra + 15) / 16, nj = rb <= 0 ? 0 : (rb + 15) / 16;
  float2 acc[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = make_float2(0.f, 0.f);

  for (long long g0 = g_begin; g0 < g_end; g0 += GK) {
    // load 64 rows x 16 columns of A and B: 1024 elements each, 4 per thread
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int idx = threadIdx.x + 256 * e;
      const int row = idx >> 4, col = idx & 15;
      const long long g = g0 + col;
      float2 va = make_float2(0.f, 0.f), vb = va;
      if (g < g_end) {
        if (a0 + row < na) va = A[(long long)(a0 + row) * ld + g];
        if (b0 + row < nb) vb = B[(long long)(b0 + row) * ld + g];
      }
      As[col][row] = va;
      Bs[col][row] = vb;
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < GK; ++k) {
      float2 av[4], bv[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) av[i] = As[k][ty + 16 * i];
#pragma unroll
      for (int j = 0; j < 4; ++j) bv[j] = Bs[k][tx + 16 * j];
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (i < ni) {
#pragma unroll
          for (int j = 0; j < 4; ++j)
            if (j < nj) acc[i][j] = cadd<false>(acc[i][j], cmulc(av[i], bv[j]));
        }
    }
    __syncthreads();
  }
  double* out = part + (long long)blockIdx.z * na * nb * 2;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int a = a0 + ty + 16 * i;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int b = b0 + tx + 16 * j;
      if (a < na && b < nb) {
        out[2 * ((long long)a * nb + b)] = (double)acc[i][j].x;
        out[2 * ((long long)a * nb + b) + 1] = (double)acc[i][j].y;
      }
    }
  }
}

// FP64: bound by the FP64 pipe (about 1.7 DFMA per clock and SM), so the tile
// is chosen for the least padding, not for reuse: 8 x 8 outputs per block, one
// per thread, with the block's four groups of 64 threads taking every fourth
// point (their sums meet in a fixed order at the end). Products are fused
// multiply-adds, and real vectors take one per point instead of a complex
// product on zeros. 24^3 real, N = 8: 100 -> 6 us; 32^3 complex, N = 27: 693 ->
// 221 us (64 x 64 tiles, six FP64 operations per complex product before).
constexpr int GT64 = 8;    // output tile edge
constexpr int GK64 = 32;   // points per shared-memory stage
template <bool REAL>
__global__ void __launch_bounds__(256)
gram64_kernel(const void* __restrict__ A, int na, const void* __restrict__ B, int nb, long long ld, long long ng,
              double* __restrict__ part, long long chunk) {
  __shared__ double2 As[GT64][GK64 + 1];
  __shared__ double2 Bs[GT64][GK64 + 1];
  __shared__ double2 red[3][GT64 * GT64];
  const int kl = threadIdx.x >> 6, o = threadIdx.x & 63, ia = o >> 3, ib = o & 7;
  const int a0 = blockIdx.x * GT64, b0 = blockIdx.y * GT64;
  const long long g_begin = (long long)blockIdx.z * chunk;
  const long long g_end = g_begin + chunk < ng ? g_begin + chunk : ng;
  const bool work = a0 + (ia & 4) < na;                  // a warp holds four rows
  const double2 zero = make_double2(0.0, 0.0);
  auto load = [&](const void* X, int count, int x0, long long g0, int e) {   // element e of the 8 x 32 stage
    const int row = e / GK64;
    const long long g = g0 + e % GK64;
    if (x0 + row >= count || g >= g_end) return zero;
    const long long off = (long long)(x0 + row) * ld + g;
    if constexpr (REAL) return make_double2(static_cast<const double*>(X)[off], 0.0);
    else return static_cast<const double2*>(X)[off];
  };
  const int tid = threadIdx.x;
  double2 va = load(A, na, a0, g_begin, tid), vb = load(B, nb, b0, g_begin, tid);
  double2 acc = zero;
  for (long long g0 = g_begin; g0 < g_end; g0 += GK64) {
    As[tid / GK64][tid % GK64] = va;
    Bs[tid / GK64][tid % GK64] = vb;
    __syncthreads();
    if (g0 + GK64 < g_end) {                             // the next stage's loads run under the products
      va = load(A, na, a0, g0 + GK64, tid);
      vb = load(B, nb, b0, g0 + GK64, tid);
    }
    if (work) {
#pragma unroll
      for (int k = 0; k < GK64 / 4; ++k) {
        const double2 x = As[ia][4 * k + kl], y = Bs[ib][4 * k + kl];
        if constexpr (REAL) acc.x = fma(x.x, y.x, acc.x);
        else acc = cfmac(acc, x, y);
      }
    }
    __syncthreads();
  }
  if (kl > 0) red[kl - 1][o] = acc;
  __syncthreads();
  if (kl == 0 && a0 + ia < na && b0 + ib < nb) {
#pragma unroll
    for (int q = 0; q < 3; ++q) acc = cadd(acc, red[q][o]);
    double2* out = reinterpret_cast<double2*>(part) + (long long)blockIdx.z * na * nb;
    out[(long long)(a0 + ia) * nb + b0 + ib] = acc;
  }
}

namespace {
constexpr long long kGramBlocks64 = 4 * 152;   // FP64: four blocks per SM
constexpr long long kMaxGramSplits = 256;
long long gram_tiles(bool f64, int na, int nb) {
  const int edge = f64 ? GT64 : GT;
  return (long long)((na + edge - 1) / edge) * ((nb + edge - 1) / edge);
}
}  // namespace

int gram_splits(bool f64, long long ng, int na, int nb) {
  // ~1k-point chunks keep the partial sums short; small matrices on small grids
  // take shorter chunks so that the launch still covers one wave of SMs (FP64:
  // four blocks per SM, whose tiles are small)
  long long s = (ng + 1023) / 1024;
  const long long tiles = gram_tiles(f64, na, nb);
  const long long blocks = f64 ? kGramBlocks64 : 152;
  const long long wave = tiles > 0 ? (blocks + tiles - 1) / tiles : 1;
  const long long stage = f64 ? GK64 : GK;
  const long long max_s = (ng + stage - 1) / stage;   // at least one K stage per split
  if (s < wave) s = wave;
  if (s > max_s) s = max_s;
  if (s > kMaxGramSplits) s = kMaxGramSplits;
  if (s < 1) s = 1;
  return (int)s;
}

// Entries to hold the partial matrices: for FP64 a bound on gram_splits() na nb that
// never falls as na or nb grows (a workspace sized for the widest call serves every
// narrower one; the splits of 8 x 8 tiles halve as tiles double, so the product itself
// does). With na nb <= 64 tiles, na nb ceil(blocks / tiles) <= 64 (blocks + tiles).
size_t gram_part_entries(bool f64, long long ng, int na, int nb) {
  if (!f64) return (size_t)gram_splits(f64, ng, na, nb) * na * nb;
  const long long points = std::min((ng + 1023) / 1024, kMaxGramSplits);
  const long long wave = std::min(kMaxGramSplits * na * nb, 64 * (kGramBlocks64 + gram_tiles(f64, na, nb)));
  return (size_t)std::max(points * na * nb, wave);
}

void launch_gram(bool f64, bool real_in, const void* A, int na, const void* B, int nb, long long ld,
                 long long ng, double* part, int splits, cudaStream_t st) {
  const int edge = f64 ? GT64 : GT, stage = f64 ? GK64 : GK;
  long long chunk = (ng + splits - 1) / splits;
  chunk = (chunk + stage - 1) / stage * stage;
  const dim3 grid((na + edge - 1) / edge, (nb + edge - 1) / edge, splits);
  if (f64) {
    if (real_in) gram64_kernel<true><<<grid, 256, 0, st>>>(A, na, B, nb, ld, ng, part, chunk);
    else gram64_kernel<false><<<grid, 256, 0, st>>>(A, na, B, nb, ld, ng, part, chunk);
  } else {
    gram_kernel<<<grid, 256, 0, st>>>(static_cast<const float2*>(A), na, static_cast<const float2*>(B), nb, ld, ng,
                                      part, chunk);
  }
}

// out[a][b] = scale * sum_s part[s][a][b] (part: FP64 complex [splits][na][nb]);
// real_out -> imaginary parts dropped (real Gamma-point case). A block sums 32
// consecutive entries: warp y takes the splits s = y, y + 8, ..., with 16-byte
// loads coalesced across the warp, and the eight partial sums meet in shared
// memory in a fixed order, so the result does not depend on timing.
constexpr int kRedGroups = 8;
__global__ void __launch_bounds__(32 * kRedGroups)
gram_reduce_kernel(const double* __restrict__ part, int splits, int na, int nb, double scale, int real_out,
                   double* __restrict__ out) {
  __shared__ double2 red[kRedGroups][32];
  const int lane = threadIdx.x & 31, y = threadIdx.x >> 5;
  const long long total = (long long)na * nb;
  const long long idx = (long long)blockIdx.x * 32 + lane;
  const double2* p2 = reinterpret_cast<const double2*>(part);
  double2 acc = make_double2(0.0, 0.0);
  if (idx < total)
    for (int s = y; s < splits; s += kRedGroups) {
      const double2 v = p2[(long long)s * total + idx];
      acc.x += v.x;
      acc.y += v.y;
    }
  red[y][lane] = acc;
  __syncthreads();
  if (y != 0 || idx >= total) return;
  double re = 0.0, im = 0.0;
#pragma unroll
  for (int k = 0; k < kRedGroups; ++k) {
    re += red[k][lane].x;
    im += red[k][lane].y;
  }
  if (real_out) {
    out[idx] = scale * re;
  } else {
    out[2 * idx] = scale * re;
    out[2 * idx + 1] = scale * im;
  }
}

// out <- (out + out^*) / 2 for an n x n matrix, in place: the thread of entry
// (a, b) with a <= b writes both (a, b) and (b, a).
__global__ void hermitize_kernel(double* __restrict__ out, int n, int real_out) {
  const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= (long long)n * n) return;
  const int a = (int)(e / n), b = (int)(e % n);
  if (a > b) return;
  const long long ab = (long long)a * n + b, ba = (long long)b * n + a;
  if (real_out) {
    const double h = 0.5 * (out[ab] + out[ba]);
    out[ab] = h;
    out[ba] = h;
  } else {
    const double re = 0.5 * (out[2 * ab] + out[2 * ba]);
    const double im = 0.5 * (out[2 * ab + 1] - out[2 * ba + 1]);
    out[2 * ab] = re;
    out[2 * ab + 1] = im;
    out[2 * ba] = re;
    out[2 * ba + 1] = -im;
  }
}

// 1/2 Re of the sum of the first `count` diagonal entries of the n x n matrix m:
// one warp, lane l summing the entries l, l + 32, ..., then a fixed shuffle tree.
__global__ void trace_half_kernel(const double* __restrict__ m, int n, int count, int real, double* out) {
  if (blockIdx.x != 0 || threadIdx.x >= 32) return;
  const int lane = threadIdx.x;
  double s = 0.0;
  for (int k = lane; k < count; k += 32) s += real ? m[(long long)k * n + k] : m[2 * ((long long)k * n + k)];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
  if (lane == 0) *out = 0.5 * s;
}

__global__ void m_copy_kernel(const double* __restrict__ mc, int n, int real, double* __restrict__ out) {
  const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= (long long)n * n) return;
  if (real) {
    out[e] = mc[2 * e];
  } else {
    out[2 * e] = mc[2 * e];
    out[2 * e + 1] = mc[2 * e + 1];
  }
}

// M_out <- M (real part only for real orbitals), Ex_out <- 1/2 Re tr M; both
// nullable. Returns the number of kernels launched.
int launch_m_outputs(const double* Mc, int n, bool real, double* M_out, double* Ex_out, cudaStream_t st,
                     int n_trace) {
  int k = 0;
  if (M_out) {
    const long long nn = (long long)n * n;
    m_copy_kernel<<<(unsigned)((nn + 255) / 256), 256, 0, st>>>(Mc, n, real ? 1 : 0, M_out);
    ++k;
  }
  if (Ex_out) {
    trace_half_kernel<<<1, 32, 0, st>>>(Mc, n, n_trace < 0 ? n : n_trace, 0, Ex_out);
    ++k;
  }
  return k;
}

int launch_gram_reduce(const double* part, int splits, int na, int nb, double scale, bool hermitize,
                       bool real_out, double* out, double* out_trace_half, cudaStream_t st) {
  const long long total = (long long)na * nb;
  gram_reduce_kernel<<<(unsigned)((total + 31) / 32), 32 * kRedGroups, 0, st>>>(part, splits, na, nb, scale,
                                                                              real_out ? 1 : 0, out);
  int k = 1;
  if (hermitize) {   // na == nb
    hermitize_kernel<<<(unsigned)((total + 255) / 256), 256, 0, st>>>(out, na, real_out ? 1 : 0);
    ++k;
  }
  if (out_trace_half) {
    trace_half_kernel<<<1, 32, 0, st>>>(out, na, na, real_out, out_trace_half);
    ++k;
  }
  return k;
}

// ---------------------------------------------------------------- outer
// Out[b][g] = alpha * sum_k A[k][g] C[k][b]   (C: FP64 complex [nk][nb])
constexpr int OG = 128;  // g per block
constexpr int OB = 16;   // b per block
constexpr int OK = 16;   // k per stage

__global__ void __launch_bounds__(256)
outer_kernel(const float2* __restrict__ A, int nk, const double* __restrict__ C, int nb, long long ld, long long ng,
             float alpha, float2* __restrict__ Out) {
  __shared__ float2 As[OK][OG];
  __shared__ float2 Cs[OK][OB];
  const int tg = threadIdx.x & 63, tb = threadIdx.x >> 6;   // 64 x 4
  const long long g0 = (long long)blockIdx.x * OG;
  const int b0 = blockIdx.y * OB;
  // this thread's columns b0 + 4 tb + j (j < nj) inside the output (padded
  // warps skip the products)
  const int rbb = nb - b0 - 4 * tb;
  const int nj = rbb <= 0 ? 0 : (rbb < 4 ? rbb : 4);
  float2 acc[2][4];
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = make_float2(0.f, 0.f);
  for (int k0 = 0; k0 < nk; k0 += OK) {
    const int kmax = nk - k0 < OK ? nk - k0 : OK;
#pragma unroll
    for (int e = 0; e < (OK * OG) / 256; ++e) {
      const int idx = threadIdx.x + 256 * e;
      const int kk = idx / OG, gg = idx % OG;
      const long long g = g0 + gg;
      As[kk][gg] = (k0 + kk < nk && g < ng) ? A[(long long)(k0 + kk) * ld + g] : make_float2(0.f, 0.f);
    }
    {
      const int kk = threadIdx.x / OB, bb = threadIdx.x % OB;
      float2 c = make_float2(0.f, 0.f);
      if (k0 + kk < nk && b0 + bb < nb) {
        const long long o = 2 * ((long long)(k0 + kk) * nb + b0 + bb);
        c = make_float2((float)C[o], (float)C[o + 1]);
      }
      Cs[kk][bb] = c;
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < OK; ++k) {
      if (k >= kmax) break;
      float2 av[2], cv[4];
#pragma unroll
      for (int i = 0; i < 2; ++i) av[i] = As[k][tg + 64 * i];
#pragma unroll
      for (int j = 0; j < 4; ++j) cv[j] = Cs[k][tb * 4 + j];
#pragma unroll
      for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j)
          if (j < nj) acc[i][j] = cadd<false>(acc[i][j], cmul(av[i], cv[j]));
    }
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const long long g = g0 + tg + 64 * i;
    if (g >= ng) continue;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int b = b0 + tb * 4 + j;
      if (b < nb) Out[(long long)b * ld + g] = cscale(acc[i][j], alpha);
    }
  }
}

// FP64, bound by the FP64 pipe as the gram product: 64 points x 16 columns per
// block, one point x 4 columns per thread, fused multiply-adds (real vectors:
// one per term, C's real part), and with `upper` (C = L^{-*}, zero below the
// diagonal) only the terms k <= b of each four columns. 24^3 real, N = 8: 17 ->
// 6 us; 32^3 complex, N = 27: 378 -> 113 us.
constexpr int OG64 = 64;
template <bool REAL>
__global__ void __launch_bounds__(256)
outer64_kernel(const void* __restrict__ A, int nk, const double2* __restrict__ C, int nb, long long ld, long long ng,
               double alpha, int upper, void* __restrict__ Out) {
  __shared__ double2 As[OK][OG64];
  __shared__ double2 Cs[OK][OB];
  const int tg = threadIdx.x & 63, tb = threadIdx.x >> 6;   // 64 x 4
  const long long g0 = (long long)blockIdx.x * OG64, g = g0 + tg;
  const int b0 = blockIdx.y * OB, bt = b0 + 4 * tb;
  const int nj = nb - bt < 4 ? nb - bt : 4;
  const int kend = upper && b0 + OB < nk ? b0 + OB : nk;                  // of the block
  const int kthr = nj <= 0 ? 0 : upper && bt + 4 < nk ? bt + 4 : nk;      // of this thread (uniform in a warp)
  double2 acc[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) acc[j] = make_double2(0.0, 0.0);
  for (int k0 = 0; k0 < kend; k0 += OK) {
#pragma unroll
    for (int e = 0; e < (OK * OG64) / 256; ++e) {
      const int kk = (threadIdx.x >> 6) + 4 * e;
      double2 v = make_double2(0.0, 0.0);
      if (k0 + kk < kend && g < ng) {
        const long long o = (long long)(k0 + kk) * ld + g;
        if constexpr (REAL) v.x = static_cast<const double*>(A)[o];
        else v = static_cast<const double2*>(A)[o];
      }
      As[kk][tg] = v;
    }
    {
      const int kk = threadIdx.x / OB, bb = threadIdx.x % OB;
      Cs[kk][bb] = (k0 + kk < kend && b0 + bb < nb) ? C[(long long)(k0 + kk) * nb + b0 + bb] : make_double2(0.0, 0.0);
    }
    __syncthreads();
    const int km = kthr - k0 < OK ? kthr - k0 : OK;
    for (int k = 0; k < km; ++k) {
      const double2 x = As[k][tg];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        if (j < nj) {
          if constexpr (REAL) acc[j].x = fma(x.x, Cs[k][4 * tb + j].x, acc[j].x);
          else acc[j] = cfma(acc[j], x, Cs[k][4 * tb + j]);
        }
      }
    }
    __syncthreads();
  }
  if (g >= ng) return;
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    if (j >= nj) continue;
    const long long o = (long long)(bt + j) * ld + g;
    if constexpr (REAL) static_cast<double*>(Out)[o] = alpha * acc[j].x;
    else static_cast<double2*>(Out)[o] = cscale(acc[j], alpha);
  }
}

void launch_outer(bool f64, bool real_io, const void* A, int nk, const double* C, int nb,
                  long long ld, long long ng, double alpha, bool upper, void* Out, cudaStream_t st) {
  if (!f64) {
    const dim3 grid((unsigned)((ng + OG - 1) / OG), (nb + OB - 1) / OB);
    outer_kernel<<<grid, 256, 0, st>>>(static_cast<const float2*>(A), nk, C, nb, ld, ng, (float)alpha,
                                       static_cast<float2*>(Out));
    return;
  }
  const dim3 grid((unsigned)((ng + OG64 - 1) / OG64), (nb + OB - 1) / OB);
  const double2* c = reinterpret_cast<const double2*>(C);
  if (real_io) outer64_kernel<true><<<grid, 256, 0, st>>>(A, nk, c, nb, ld, ng, alpha, upper, Out);
  else outer64_kernel<false><<<grid, 256, 0, st>>>(A, nk, c, nb, ld, ng, alpha, upper, Out);
}

// Xi = W L^{-*} with FP64 arithmetic from FP32 vectors (the plain FP64 form
// of Eq. Wtilde for FP32 storage): A is complex FP32 [nk][ld], promoted
// exactly; C = L^{-*} is upper triangular, so the block of columns
// [b0, b0 + OB) takes k < b0 + OB only; Out is complex FP32 (rounded once) or
// FP64 [nb][ld].
template <typename OUT>
__global__ void __launch_bounds__(256)
outer_f64acc_kernel(const float2* __restrict__ A, int nk, const double* __restrict__ C, int nb, long long ld,
                    long long ng, OUT* __restrict__ Out) {
  __shared__ double2 As[OK][OG];
  __shared__ double2 Cs[OK][OB];
  const int tg = threadIdx.x & 63, tb = threadIdx.x >> 6;
  const long long g0 = (long long)blockIdx.x * OG;
  const int b0 = blockIdx.y * OB;
  const int rbb = nb - b0 - 4 * tb;
  const int nj = rbb <= 0 ? 0 : (rbb < 4 ? rbb : 4);
  const int kend = b0 + OB < nk ? b0 + OB : nk;   // C[k][b] = 0 for k > b
  double2 acc[2][4];
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = make_double2(0.0, 0.0);
  for (int k0 = 0; k0 < kend; k0 += OK) {
    const int kmax = kend - k0 < OK ? kend - k0 : OK;
#pragma unroll
    for (int e = 0; e < (OK * OG) / 256; ++e) {
      const int idx = threadIdx.x + 256 * e;
      const int kk = idx / OG, gg = idx % OG;
      const long long g = g0 + gg;
      double2 v = make_double2(0.0, 0.0);
      if (k0 + kk < kend && g < ng) {
        const float2 t = A[(long long)(k0 + kk) * ld + g];
        v = make_double2((double)t.x, (double)t.y);
      }
      As[kk][gg] = v;
    }
    {
      const int kk = threadIdx.x / OB, bb = threadIdx.x % OB;
      double2 c = make_double2(0.0, 0.0);
      if (k0 + kk < kend && b0 + bb < nb) {
        const long long o = 2 * ((long long)(k0 + kk) * nb + b0 + bb);
        c = make_double2(C[o], C[o + 1]);
      }
      Cs[kk][bb] = c;
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < OK; ++k) {
      if (k >= kmax) break;
      double2 av[2], cv[4];
#pragma unroll
      for (int i = 0; i < 2; ++i) av[i] = As[k][tg + 64 * i];
#pragma unroll
      for (int j = 0; j < 4; ++j) cv[j] = Cs[k][tb * 4 + j];
#pragma unroll
      for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j)
          if (j < nj) acc[i][j] = cadd(acc[i][j], cmul(av[i], cv[j]));
    }
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const long long g = g0 + tg + 64 * i;
    if (g >= ng) continue;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int b = b0 + tb * 4 + j;
      if (b >= nb) continue;
      OUT o;
      o.x = acc[i][j].x;
      o.y = acc[i][j].y;
      Out[(long long)b * ld + g] = o;
    }
  }
}

void launch_outer_f64acc(const void* A, int nk, const double* C, int nb, long long ld, long long ng, void* Out,
                         bool out_f64, cudaStream_t st) {
  const dim3 grid((unsigned)((ng + OG - 1) / OG), (nb + OB - 1) / OB);
  const float2* a = static_cast<const float2*>(A);
  if (out_f64) outer_f64acc_kernel<double2><<<grid, 256, 0, st>>>(a, nk, C, nb, ld, ng, static_cast<double2*>(Out));
  else outer_f64acc_kernel<float2><<<grid, 256, 0, st>>>(a, nk, C, nb, ld, ng, static_cast<float2*>(Out));
}

// Cholesky + inverse (FP64): chol.cu

// ---------------------------------------------------------------- reductions
__global__ void energy_reduce_kernel(const double* __restrict__ part, int count, double factor,
                                     double* out) {
  __shared__ double red[1024];
  double s = 0.0;
  for (int i = threadIdx.x; i < count; i += blockDim.x) s += part[i];
  red[threadIdx.x] = s;
  __syncthreads();
  for (int w = blockDim.x / 2; w > 0; w >>= 1) {
    if ((int)threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) *out = factor * red[0];
}

void launch_energy_reduce(const double* part, int count, double factor, double* out, cudaStream_t st) {
  energy_reduce_kernel<<<1, 1024, 0, st>>>(part, count, factor, out);
}

void launch_zero(void* p, size_t bytes, cudaStream_t st) { cudaMemsetAsync(p, 0, bytes, st); }

namespace {
// Uniform values in [-1, 1) from a splitmix64 hash of (seed, index): timing
// inputs for the autotuner (any values with -M positive definite will do).
__device__ __forceinline__ unsigned long long splitmix64(unsigned long long z) {
  z += 0x9E3779B97F4A7C15ull;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}
template <typename T>
__global__ void fill_random_kernel(T* x, long long count, unsigned long long seed) {
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < count; i += (long long)gridDim.x * blockDim.x) {
    const unsigned long long h = splitmix64(seed ^ splitmix64((unsigned long long)i));
    x[i] = (T)((double)(h >> 11) * (2.0 / 9007199254740992.0) - 1.0);
  }
}
}  // namespace

void launch_fill_random(void* x, long long count, bool f64, unsigned long long seed, cudaStream_t st) {
  const long long blocks = (count + 255) / 256;
  const unsigned grid = (unsigned)(blocks < 152 * 16 ? (blocks > 0 ? blocks : 1) : 152 * 16);
  if (f64) fill_random_kernel<double><<<grid, 256, 0, st>>>(static_cast<double*>(x), count, seed);
  else fill_random_kernel<float><<<grid, 256, 0, st>>>(static_cast<float*>(x), count, seed);
}

}  // namespace ace
