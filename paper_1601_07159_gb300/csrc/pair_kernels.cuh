// Pair FFT-Poisson solves: the hot loop of Eq. applyVX / Eq. W.
//
// For a batch of pairs (l, r) the 3-D solve v = F^-1[ K F[conj(x_l) y_r] ] on an
// n_x x n_y x n_z grid is split into three passes over the batch's spectrum
// scratch S, each a set of register-resident line FFTs (fft_reg.cuh), plus one
// accumulate pass:
//
//   pass A  (per z-plane)   rho = conj(x_l) y_r; FFT along y (thread = column x,
//                           coalesced loads), transpose through shared memory,
//                           FFT along x (thread = row ky); store S[z][kx][ky]
//                           (coalesced along ky). Blocks run z-plane major, so
//                           the pairs of a tile that read the same orbital
//                           plane run together and find it in L2.
//   pass B  (per pencil)    FFT along z, multiply by K(G)/N_g, inverse FFT along
//                           z, in place (thread = (kx, ky) pencil, coalesced);
//                           optionally the Parseval energy sum K |rho_hat|^2.
//   pass C  (per z-plane)   inverse FFT along x (thread = ky), transpose through
//                           shared memory, inverse FFT along y (thread = x);
//                           store v(z, y, x) in place (coalesced along x).
//   pass D  (per point)     Out_r -= x_l v and, for symmetric tiles,
//                           Out_l -= y_r conj(v); registers hold the tile's
//                           orbitals and accumulators, one read-modify-write of
//                           each output per tile, fixed summation order (full
//                           off-diagonal tiles: four threads per point, FP64 two).
// The plane passes are compiled per (n_x, n_y), the pencil pass per n_z (the
// pencil's (kx, ky) position is a run-time index), the accumulate pass once per
// precision; a grid n_x x n_y x n_z runs when its plane and its pencil length
// are compiled in. On cubic grids passes B and D use instances with the grid
// compiled in (strides and offsets folded into the instructions). At the
// larger edges a line is held by two lanes instead of one thread
// (split_line_dft): the plane passes when the longer plane edge is >= 96
// (FP64: >= 64), FP64 pass B from n_z = 64; FP32 pencils of 64 and 96 are
// spread over four warps (pass_b_quad_kernel).
//
// Real vectors (R64) pack two pairs into one complex solve: a slot holds
// rho_lr + i rho_lr' (decode_slot_real), the kernel being real and even keeps
// V_lr and V_lr' in the real and imaginary parts, and pass D splits them.
//
// Two ways to run a schedule of batches:
//  * four kernels per batch (pass_*_kernel), chained with programmatic
//    dependent launch, replayed from a CUDA graph (the default) or launched
//    eagerly (per-pass timing);
//  * one persistent launch (pair_engine_kernel, cubic grids): co-resident
//    blocks take tasks (one pass-A/C block of planes, one pass-B block of
//    pencils, one pass-D block of points) in schedule order from an atomic
//    queue and wait, with a bounded spin, on per-batch completion counters:
//    pass p of batch k needs all of pass p-1 of batch k, pass A of batch k
//    needs the last pass of batch k-1 (the scratch is reused). Tasks are taken
//    in increasing order by resident blocks, so every awaited task is already
//    running: no deadlock.
//
// Tiles within a batch touch disjoint outputs (the schedule guarantees it) and
// batches run in order, so the accumulation needs no atomics and the result is
// bitwise reproducible. The engine sums a full off-diagonal tile's left
// outputs in one thread, so the two modes agree to rounding.
#pragma once
#include "ace_internal.h"
#include "fft_reg.cuh"


namespace ace {
inline namespace ACE_RADIX_NS {   // radix order of this translation unit (fft_reg.cuh)

// Twiddle tables of a plane: one per axis, shared when the plane is square.
template <typename R, int NX, int NY> struct PlaneTw {
  TwTable<R, NX> x;
  TwTable<R, NY> y;
  __device__ __forceinline__ const TwTable<R, NX>& tx() const { return x; }
  __device__ __forceinline__ const TwTable<R, NY>& ty() const { return y; }
  void fill(const double* twx, const double* twy) {
    for (int k = 0; k < NX; ++k) { x.w[k].x = (R)twx[2 * k]; x.w[k].y = (R)twx[2 * k + 1]; }
    for (int k = 0; k < NY; ++k) { y.w[k].x = (R)twy[2 * k]; y.w[k].y = (R)twy[2 * k + 1]; }
  }
};
template <typename R, int N> struct PlaneTw<R, N, N> {
  TwTable<R, N> x;
  __device__ __forceinline__ const TwTable<R, N>& tx() const { return x; }
  __device__ __forceinline__ const TwTable<R, N>& ty() const { return x; }
  void fill(const double* twx, const double*) {
    for (int k = 0; k < N; ++k) { x.w[k].x = (R)twx[2 * k]; x.w[k].y = (R)twx[2 * k + 1]; }
  }
};

// Passes A and C: the pair's vectors, the scratch, nz z-planes per pair. Poisson
// solves (instances POIS) have the constant orbital 1 for X, which pass A leaves
// out, and their potentials are the result: pass C writes slot (l, r)'s to vector
// r of V instead of the scratch. (As run-time cases these cost pass C 10 % at 96^3.)
template <typename R, int NX, int NY> struct PlaneParams {
  const void* X;
  const void* Y;
  void* V;
  int* clear;              // status word that the first block of pass A resets (nullable)
  int packed;              // real vectors: two pairs per slot
  cplx<R>* S;
  long long ld;
  int nz;
  int npairs;
  const TileDesc* tiles;   // device table of the batch's tiles
  int ntiles;
  PlaneTw<R, NX, NY> tw;
};

// Pass B: pencils of NZ points at the nxy = n_x n_y positions (kx, ky) of a plane.
template <typename R, int NZ> struct PencilParams {
  cplx<R>* S;
  const R* Kt;             // K(G) alpha / N_g, folded [kz][kx][ky] over 0..n/2 per axis
  double* Epart;
  int npairs;
  int nx, ny, nxy;
  int khy, kzs;            // folded table: row length n_y/2 + 1, kz stride (n_x/2 + 1)(n_y/2 + 1)
  const TileDesc* tiles;
  int ntiles;
  int packed;              // real vectors: two pairs per slot (energy weights by decode_slot_real)
  TwTable<R, NZ> tw;
};

// Pass D: the tile's vectors and outputs, the pair potentials in S.
template <typename R> struct PointParams {
  const void* X;
  const void* Y;
  void* OutX;
  void* OutY;
  const cplx<R>* S;
  long long ld;
  long long ng;
  R scale;
  const TileDesc* tiles;
};

// Programmatic dependent launch (four-kernel mode): every pass is launched with
// programmatic stream serialisation, so its blocks take the slots that the
// previous pass's last blocks leave; griddep_wait() blocks until the previous
// grid has completed and its writes are visible (a no-op without the attribute).
// Pass A reads X and Y before it waits: none of the passes writes them. The kernel in
// front of a call's first pass A may have (an eager call on vectors that the
// caller's last kernel wrote), so that one is launched without the attribute
// (PairLaunch::lead).
// No pass triggers its dependents itself (griddepcontrol.launch_dependents): a
// trigger at the start of the blocks let the next pass's blocks pile up on the
// few SMs with free slots, where they waited and then ran, while the other SMs
// idled. Passes A-D of one 64-pair tile, trigger at the start -> at block exit:
// 96^3 715 -> 646 us, 64^3 183 -> 170, 48^3 58.6 -> 56, 256 pairs of 16^3 16 -> 12
// (without programmatic launch 656, 181, 66, 21).
__device__ __forceinline__ void griddep_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

template <typename Kern, typename... Args>
inline void launch_pdl(bool pdl, Kern kern, dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                       const Args&... args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = pdl ? 1 : 0;
  cudaLaunchKernelEx(&cfg, kern, args...);
}

// Loads and stores of data that other blocks of the same launch produce or
// consume (the pair scratch and the outputs, in the persistent engine) go
// through L2 (.cg): L1 is not coherent across SMs.
template <bool COH, typename T> __device__ __forceinline__ T ldx(const T* p) {
  if constexpr (COH) return __ldcg(p);
  else return *p;
}
template <bool COH, typename T> __device__ __forceinline__ void stx(T* p, T v) {
  if constexpr (COH) __stcg(p, v);
  else *p = v;
}

// Slot p of the batch -> tile index and (l, r) orbital indices.
__device__ __forceinline__ int decode_pair(const TileDesc* __restrict__ tiles, int ntiles, int p, int& l, int& r) {
  int t = 0;
  while (t + 1 < ntiles && tiles[t + 1].slot0 <= p) ++t;
  const TileDesc d = tiles[t];
  int q = p - d.slot0;
  if (d.kind == 1) {
    int li = 0, len = d.nl;
    while (q >= len) { q -= len; ++li; --len; }
    l = d.l0 + li;
    r = d.r0 + li + q;
  } else {
    l = d.l0 + q / d.nr;
    r = d.r0 + q % d.nr;
  }
  return t;
}

// Slot s of a batch of real vectors -> tile index and the slot's pairs (l, r)
// (real part) and (l, r2) (imaginary part; r2 < 0: none). Diagonal tile row
// li: the slot (l, l) alone, then (l, l + 1 + 2m), (l, l + 2 + 2m); other
// tiles: row li holds (l, r0 + 2m), (l, r0 + 2m + 1).
__device__ __forceinline__ int decode_slot_real(const TileDesc* __restrict__ tiles, int ntiles, int s, int& l,
                                                int& r, int& r2) {
  int t = 0;
  while (t + 1 < ntiles && tiles[t + 1].slot0 <= s) ++t;
  const TileDesc d = tiles[t];
  int q = s - d.slot0;
  if (d.kind == 1) {
    int li = 0, len = 1 + d.nl / 2;
    while (q >= len) { q -= len; ++li; len = 1 + (d.nl - li) / 2; }
    l = d.l0 + li;
    r = q == 0 ? l : l + 2 * q - 1;
    r2 = (q != 0 && r + 1 < d.l0 + d.nl) ? r + 1 : -1;
  } else {
    const int w = (d.nr + 1) / 2;
    l = d.l0 + q / w;
    r = d.r0 + 2 * (q % w);
    r2 = r + 1 < d.r0 + d.nr ? r + 1 : -1;
  }
  return t;
}

// Energy weight of slot p: 1 for the diagonal pair (l, l), 2 otherwise (the
// pair and its mirror (r, l)).
__device__ __forceinline__ double slot_weight(const TileDesc* __restrict__ tiles, int ntiles, int p, bool real) {
  int l, r, r2;
  if (real) decode_slot_real(tiles, ntiles, p, l, r, r2);
  else decode_pair(tiles, ntiles, p, l, r);
  return l == r ? 1.0 : 2.0;
}

template <typename R, bool REAL>
__device__ __forceinline__ cplx<R> load_vec(const void* base, long long idx) {
  if constexpr (REAL) {
    return cmk<cplx<R>>(static_cast<const R*>(base)[idx], R(0));
  } else {
    return static_cast<const cplx<R>*>(base)[idx];
  }
}

// The kernel table is folded (K depends on |G|^2 only): index k of an axis of
// n points and n - k share an entry. kfold(k) = min(k, n - k).
template <int N> __host__ __device__ __forceinline__ constexpr int kfold(int k) { return k <= N / 2 ? k : N - k; }
__host__ __device__ __forceinline__ int kfold_rt(int k, int n) { return k <= n / 2 ? k : n - k; }
// Plane geometry seen by the pencil pass: compile-time for cubic grids
// (CUBE: n_x = n_y = n_z, so strides and table offsets fold into the
// instructions), read from the parameters otherwise.
template <typename R, int NZ, bool CUBE> struct PencilGeom {
  int nx, ny, nxy, khy, kzs;
  __device__ __forceinline__ explicit PencilGeom(const PencilParams<R, NZ>& P) {
    if constexpr (CUBE) {
      nx = NZ; ny = NZ; nxy = NZ * NZ; khy = NZ / 2 + 1; kzs = (NZ / 2 + 1) * (NZ / 2 + 1);
    } else {
      nx = P.nx; ny = P.ny; nxy = P.nxy; khy = P.khy; kzs = P.kzs;
    }
  }
  // offset of the (kx, ky) pencil f = kx n_y + ky in the folded table
  __device__ __forceinline__ int kt_pencil(int f) const {
    const int kx = f / ny, ky = f - kx * ny;
    return kfold_rt(kx, nx) * khy + kfold_rt(ky, ny);
  }
};

template <int NX, int NY> constexpr int kMaxLine = NX > NY ? NX : NY;

// Items (pair, z-plane) per CTA of the whole-line plane kernels: about 128
// threads (two planes of 48 or 64, five of 24), so that several independent
// blocks share an SM and one block's loads run under another's transforms;
// about 256 threads left one or two blocks per SM that loaded, transformed and
// stored together (a 64-pair tile, passes A + C: 24^3 8.3 -> 7.3, 32^3 6.0 ->
// 5.0, 36^3 7.3 -> 6.6 ps per pair point; FP64 24^3 242 -> 170). At most 96 KB.
template <typename R, int NX, int NY> __host__ __device__ constexpr int plane_items() {
  constexpr int ML = kMaxLine<NX, NY>;
  constexpr int by_threads = (128 / ML) > 0 ? (128 / ML) : 1;
  constexpr int by_smem = (96 * 1024) / (NY * (NX + 1) * (int)sizeof(cplx<R>));
  constexpr int v = by_threads < by_smem ? by_threads : by_smem;
  return v > 0 ? v : 1;
}
// Whole-line planes that transform their lines radix 2 first: FP32 planes whose
// longer edge is at least 48 (results equal to the bit to the two-lane form).
template <typename R, int NX, int NY> constexpr bool kLine2 =
    sizeof(R) == 4 && kMaxLine<NX, NY> >= 48 && NX % 4 == 0 && NY % 4 == 0;

// Blocks per SM those kernels are compiled for: FP32 lines need about 2 ML + 28
// registers (the line itself and the butterflies' temporaries), and more blocks
// would spill; FP64 two.
template <typename R, int NX, int NY> __host__ __device__ constexpr int plane_blocks() {
  constexpr int ML = kMaxLine<NX, NY>;
  constexpr int warps = (ML * plane_items<R, NX, NY>() + 31) / 32;
  constexpr int v = 65536 / (32 * warps * (2 * ML + 28));
  return sizeof(R) == 4 ? (v < 1 ? 1 : v > 8 ? 8 : v) : 2;
}
constexpr int kEngineThreads = 256;
template <typename R, int N> __host__ __device__ constexpr int engine_items() {
  // items per plane task of the engine: all 256 threads, <= 200 KB of planes
  constexpr int by_threads = (kEngineThreads / N) > 0 ? (kEngineThreads / N) : 1;
  constexpr int by_smem = (200 * 1024) / (N * (N + 1) * (int)sizeof(cplx<R>));
  constexpr int v = by_threads < by_smem ? by_threads : by_smem;
  return v > 0 ? v : 1;
}

// ---------------------------------------------------------------- pass bodies
// A whole line in registers: radix 2 first (LINE2) or by the radix order.
template <int N, bool INV, bool LINE2, typename R>
__device__ __forceinline__ void line_dft(cplx<R> (&a)[N], const TwTable<R, N>& tw) {
  if constexpr (LINE2) line_dft2<N, INV, R>(a, tw);
  else dft<N, N, INV, R>(a, tw);
}
// Pass A on virtual block `vb` (IPB plane items, thread tid = ty * max(NX, NY) + tx).
template <typename R, int NX, int NY, bool REAL, bool COH, int IPB, bool PDL, bool LINE2, bool POIS>
__device__ __forceinline__ void body_a(const PlaneParams<R, NX, NY>& P, const TileDesc* tiles, int ntiles,
                                       int npairs, cplx<R>* smem, long long vb, int tid) {
  constexpr int ML = kMaxLine<NX, NY>;
  const int tx = tid % ML, ty = tid / ML;
  cplx<R>* buf = smem + ty * NY * (NX + 1);
  const long long item = vb * IPB + ty;
  const bool active = ty < IPB && item < (long long)npairs * P.nz;
  int p = 0, z = 0, l = 0, r = 0, r2 = -1;
  if (active) {   // z-plane major: the pairs of a tile that share an orbital plane run together
    z = (int)(item / npairs);
    p = (int)(item % npairs);
    if constexpr (REAL) decode_slot_real(tiles, ntiles, p, l, r, r2);
    else decode_pair(tiles, ntiles, p, l, r);
  }
  if (active && tx < NX) {
    cplx<R> a[NY];
    const long long xo = (long long)l * P.ld + (long long)z * NX * NY + tx;
    const long long yo = (long long)r * P.ld + (long long)z * NX * NY + tx;
    if constexpr (REAL) {                     // x_l (y_r + i y_r2)
      const R* Xr = static_cast<const R*>(P.X);
      const R* Yr = static_cast<const R*>(P.Y);
      const bool two = r2 >= 0;
      const long long y2o = (long long)(two ? r2 : r) * P.ld + (long long)z * NX * NY + tx;
#pragma unroll
      for (int y = 0; y < NY; ++y) {
        const R xv = POIS ? R(1) : Xr[xo + y * NX];
        a[y] = cmk<cplx<R>>(xv * Yr[yo + y * NX], two ? xv * Yr[y2o + y * NX] : R(0));
      }
    } else {
#pragma unroll
      for (int y = 0; y < NY; ++y) {
        const cplx<R> xv = POIS ? cmk<cplx<R>>(R(1), R(0)) : load_vec<R, REAL>(P.X, xo + y * NX);
        const cplx<R> yv = load_vec<R, REAL>(P.Y, yo + y * NX);
        a[y] = cmulc(xv, yv);                 // conj(x_l) * y_r
      }
    }
    line_dft<NY, false, LINE2, R>(a, P.tw.ty());   // along y, column x = tx
#pragma unroll
    for (int k = 0; k < NY; ++k) buf[k * (NX + 1) + tx] = a[k];
  }
  __syncthreads();
  if (active && tx < NY) {
    cplx<R> b[NX];
#pragma unroll
    for (int x = 0; x < NX; ++x) b[x] = buf[tx * (NX + 1) + x];
    line_dft<NX, false, LINE2, R>(b, P.tw.tx());   // along x, row ky = tx
    if constexpr (PDL) {
      griddep_wait();                         // the previous batch's pass D still reads S
      if (P.clear && vb == 0 && tid == 0) P.clear[0] = P.clear[1] = 0;
    }
    cplx<R>* out = P.S + ((long long)p * P.nz + z) * NX * NY + tx;
#pragma unroll
    for (int kx = 0; kx < NX; ++kx) stx<COH>(out + kx * NY, b[kx]);
  }
}

// Pass B on virtual block `vb` of `nthr` pencils. mode 0: Poisson (forward z,
// K, inverse z); 1: energy only; 2: both. The energy partial of the block
// (mode != 0) is added to *eslot by thread 0 (one owner per slot).
template <typename R, int NZ, bool COH, bool CUBE>
__device__ __forceinline__ void body_b(const PencilParams<R, NZ>& P, const TileDesc* tiles, int ntiles, int npairs,
                                       int mode, long long vb, int tid, int nthr, double* red, double* eslot) {
  const PencilGeom<R, NZ, CUBE> G(P);
  const int nxy = G.nxy;
  const long long gid = vb * nthr + tid;
  const bool active = gid < (long long)npairs * nxy;
  double e = 0.0;
  if (active) {
    const int p = (int)(gid / nxy);
    const int f = (int)(gid % nxy);
    cplx<R>* s = P.S + (long long)p * NZ * nxy + f;
    cplx<R> a[NZ];
#pragma unroll
    for (int zz = 0; zz < NZ; ++zz) a[zz] = ldx<COH>(s + (long long)zz * nxy);
    dft<NZ, NZ, false, R>(a, P.tw);
    R acc = R(0);
    const R* kt = P.Kt + G.kt_pencil(f);
#pragma unroll
    for (int kz = 0; kz < NZ; ++kz) {
      const R k = kt[kfold<NZ>(kz) * G.kzs];
      if (mode != 0) acc += k * (a[kz].x * a[kz].x + a[kz].y * a[kz].y);
      a[kz] = cscale(a[kz], k);
    }
    if (mode != 0) e = slot_weight(tiles, ntiles, p, P.packed) * (double)acc;
    if (mode != 1) {
      dft<NZ, NZ, true, R>(a, P.tw);
#pragma unroll
      for (int zz = 0; zz < NZ; ++zz) stx<COH>(s + (long long)zz * nxy, a[zz]);
    }
  }
  if (mode != 0) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) e += __shfl_down_sync(0xffffffffu, e, o);
    if ((tid & 31) == 0) red[tid >> 5] = e;
    __syncthreads();
    if (tid == 0) {
      double s = 0.0;
      for (int w = 0; w < nthr / 32; ++w) s += red[w];
      *eslot += s;
    }
  }
}

// Where pass C leaves plane z of slot p: point i of the plane goes through store(i, v).
template <typename R, int NX, int NY, bool COH, bool POIS> struct PlaneOut {
  cplx<R>* c = nullptr;          // complex destination (the scratch or a vector of V)
  R *re = nullptr, *im = nullptr;   // real vectors of V (packed slots; im null: none)
  __device__ __forceinline__ PlaneOut(const PlaneParams<R, NX, NY>& P, int p, int z, cplx<R>* plane) {
    c = plane;
    if constexpr (POIS) {
      int l, r, r2 = -1;
      if (sizeof(R) == 8 && P.packed) {
        decode_slot_real(P.tiles, P.ntiles, p, l, r, r2);
        R* V = static_cast<R*>(P.V) + (long long)z * NX * NY;
        re = V + (long long)r * P.ld;
        im = r2 >= 0 ? V + (long long)r2 * P.ld : nullptr;
      } else {
        decode_pair(P.tiles, P.ntiles, p, l, r);
        c = static_cast<cplx<R>*>(P.V) + (long long)r * P.ld + (long long)z * NX * NY;
      }
    }
  }
  __device__ __forceinline__ void store(int i, cplx<R> v) const {
    if (sizeof(R) == 8 && POIS && re) {
      re[i] = v.x;
      if (im) im[i] = v.y;
    } else {
      stx<COH>(c + i, v);
    }
  }
};

// Pass C on virtual block `vb` (IPB plane items).
template <typename R, int NX, int NY, bool COH, int IPB, bool LINE2, bool POIS>
__device__ __forceinline__ void body_c(const PlaneParams<R, NX, NY>& P, int npairs, cplx<R>* smem, long long vb,
                                       int tid) {
  constexpr int ML = kMaxLine<NX, NY>;
  const int tx = tid % ML, ty = tid / ML;
  cplx<R>* buf = smem + ty * NY * (NX + 1);
  const long long item = vb * IPB + ty;
  const bool active = ty < IPB && item < (long long)npairs * P.nz;
  cplx<R>* plane = nullptr;
  int p = 0, z = 0;
  if (active) {
    p = (int)(item / P.nz);
    z = (int)(item % P.nz);
    plane = P.S + ((long long)p * P.nz + z) * NX * NY;
  }
  if (active && tx < NY) {
    cplx<R> b[NX];
#pragma unroll
    for (int kx = 0; kx < NX; ++kx) b[kx] = ldx<COH>(plane + kx * NY + tx);   // row ky = tx
    line_dft<NX, true, LINE2, R>(b, P.tw.tx());                              // inverse along x
#pragma unroll
    for (int x = 0; x < NX; ++x) buf[tx * (NX + 1) + x] = b[x];
  }
  __syncthreads();
  if (active && tx < NX) {
    cplx<R> a[NY];
#pragma unroll
    for (int ky = 0; ky < NY; ++ky) a[ky] = buf[ky * (NX + 1) + tx];  // column x = tx
    line_dft<NY, true, LINE2, R>(a, P.tw.ty());                       // inverse along y
    const PlaneOut<R, NX, NY, COH, POIS> out(P, p, z, plane);
#pragma unroll
    for (int y = 0; y < NY; ++y) out.store(y * NX + tx, a[y]);
  }
}

template <typename R, bool REAL, bool COH>
__device__ __forceinline__ void rmw_out(void* base, long long idx, cplx<R> acc, R scale) {
  if constexpr (REAL) {
    R* o = static_cast<R*>(base) + idx;
    stx<COH>(o, ldx<COH>(o) - scale * acc.x);
  } else {
    cplx<R>* o = static_cast<cplx<R>*>(base) + idx;
    const cplx<R> c = ldx<COH>(o);
    stx<COH>(o, cmk<cplx<R>>(c.x - scale * acc.x, c.y - scale * acc.y));
  }
}

// Full tiles (kTileMax orbitals per side): no runtime guards, so all loads of
// the tile's pair potentials can be issued back to back. v is read once, so it
// is loaded with the streaming (evict-first) hint.
template <typename R, bool REAL, bool COH, long long NGC>
__device__ __forceinline__ void d_full_diag(const PointParams<R>& P, const TileDesc& d,
                                            const cplx<R>* __restrict__ V, long long g) {
  const long long NG = NGC ? NGC : P.ng;
  constexpr int B = kTileMax;
  cplx<R> x[B], acc[B];
#pragma unroll
  for (int o = 0; o < B; ++o) {
    acc[o] = cmk<cplx<R>>(R(0), R(0));
    x[o] = load_vec<R, REAL>(P.X, (long long)(d.l0 + o) * P.ld + g);
  }
#pragma unroll
  for (int li = 0; li < B; ++li) {
#pragma unroll
    for (int ri = li; ri < B; ++ri) {
      const int q = li * B - li * (li - 1) / 2 + (ri - li);
      const cplx<R> v = __ldcs(V + (long long)q * NG);
      acc[ri] = cfma(acc[ri], x[li], v);
      if (ri != li) acc[li] = cfmac(acc[li], v, x[ri]);
    }
  }
#pragma unroll
  for (int o = 0; o < B; ++o) rmw_out<R, REAL, COH>(P.OutY, (long long)(d.l0 + o) * P.ld + g, acc[o], P.scale);
}

template <typename R, bool REAL, bool COH, long long NGC>
__device__ __forceinline__ void d_full_off(const PointParams<R>& P, const TileDesc& d,
                                           const cplx<R>* __restrict__ V, long long g) {
  const long long NG = NGC ? NGC : P.ng;
  constexpr int B = kTileMax;
  cplx<R> xl[B], yr[B], al[B], ar[B];
#pragma unroll
  for (int o = 0; o < B; ++o) {
    al[o] = cmk<cplx<R>>(R(0), R(0));
    ar[o] = al[o];
    xl[o] = load_vec<R, REAL>(P.X, (long long)(d.l0 + o) * P.ld + g);
    yr[o] = load_vec<R, REAL>(P.Y, (long long)(d.r0 + o) * P.ld + g);
  }
#pragma unroll
  for (int li = 0; li < B; ++li) {
#pragma unroll
    for (int ri = 0; ri < B; ++ri) {
      const cplx<R> v = __ldcs(V + (long long)(li * B + ri) * NG);
      ar[ri] = cfma(ar[ri], xl[li], v);
      al[li] = cfmac(al[li], v, yr[ri]);
    }
  }
#pragma unroll
  for (int o = 0; o < B; ++o) {
    rmw_out<R, REAL, COH>(P.OutY, (long long)(d.r0 + o) * P.ld + g, ar[o], P.scale);
    rmw_out<R, REAL, COH>(P.OutX, (long long)(d.l0 + o) * P.ld + g, al[o], P.scale);
  }
}

// Off-diagonal full tile with two threads per grid point: thread half h takes
// the right orbitals r0 + 4h .. r0 + 4h + 3 (its 32 of the tile's 64 pair
// potentials), so each thread holds half the state of d_full_off and a block
// keeps twice the loads in flight. Each warp covers 32 consecutive points of
// one half (coalesced). The left outputs' two partial sums (over the two
// halves of r) meet through shared memory and are added in a fixed order;
// thread h then updates Out_l for l0 + 4h .. l0 + 4h + 3 and Out_r for its r.
constexpr int kDSplitPts = 128;   // points per 256-thread block
template <typename R, bool REAL, long long NGC>
__device__ __forceinline__ void d_split_off(const PointParams<R>& P, const TileDesc& d, long long vbx, int tid,
                                            cplx<R>* xch) {
  const long long NG = NGC ? NGC : P.ng;
  constexpr int B = kTileMax, H = kTileMax / 2;
  const int h = (tid >> 5) & 1;
  const int pt = ((tid >> 6) << 5) | (tid & 31);
  const long long g = vbx * kDSplitPts + pt;
  const bool act = g < NG;
  const cplx<R>* V = P.S + (long long)d.slot0 * NG + g;
  cplx<R> xl[B], yr[H], al[B], ar[H];
#pragma unroll
  for (int o = 0; o < B; ++o) {
    al[o] = cmk<cplx<R>>(R(0), R(0));
    xl[o] = act ? load_vec<R, REAL>(P.X, (long long)(d.l0 + o) * P.ld + g) : al[o];
  }
#pragma unroll
  for (int o = 0; o < H; ++o) {
    ar[o] = al[o];
    yr[o] = act ? load_vec<R, REAL>(P.Y, (long long)(d.r0 + h * H + o) * P.ld + g) : al[o];
  }
  if (act) {
#pragma unroll
    for (int li = 0; li < B; ++li) {
#pragma unroll
      for (int ri = 0; ri < H; ++ri) {
        const cplx<R> v = __ldcs(V + (long long)(li * B + h * H + ri) * NG);
        ar[ri] = cfma(ar[ri], xl[li], v);
        al[li] = cfmac(al[li], v, yr[ri]);
      }
    }
  }
#pragma unroll
  for (int o = 0; o < H; ++o) xch[o * 256 + tid] = h ? al[o] : al[H + o];   // the partner's half
  __syncthreads();
  if (!act) return;
  const int partner = tid ^ 32;                                           // same point, other half
#pragma unroll
  for (int o = 0; o < H; ++o) {
    const cplx<R> own = h ? al[H + o] : al[o];
    const cplx<R> other = xch[o * 256 + partner];
    const cplx<R> lo = h ? other : own, hi = h ? own : other;              // r-half 0 first, then 1
    rmw_out<R, REAL, false>(P.OutX, (long long)(d.l0 + h * H + o) * P.ld + g, cadd(lo, hi), P.scale);
    rmw_out<R, REAL, false>(P.OutY, (long long)(d.r0 + h * H + o) * P.ld + g, ar[o], P.scale);
  }
}

// Off-diagonal full FP32 tile with four threads per grid point: thread (lh, rh)
// takes the left orbitals l0 + 4 lh .. + 3 and the right ones r0 + 4 rh .. + 3 (16
// of the tile's 64 pair potentials), so a thread has half the loads of d_split_off
// in flight at once and a tile has twice the threads: 64 potentials per thread
// pair left the launch of a 48^3 tile at 1.4 waves of blocks. The sums are those
// of d_split_off, in its order, to the bit: the right outputs' sums run over the
// left orbitals in turn, so the threads lh = 1 continue from the partial sums that
// lh = 0 leaves in shared memory (their potentials are in registers by then), and
// the left outputs add the two right halves' sums. Threads lh = 0 then update
// Out_l (4 rh .. 4 rh + 3), threads lh = 1 Out_r.
constexpr int kDQuadPts = 64;    // points per 256-thread block
template <typename R, long long NGC>
__device__ __forceinline__ void d_quad_off(const PointParams<R>& P, const TileDesc& d, long long vbx, int tid,
                                           cplx<R>* xch) {
  using C = cplx<R>;
  const long long NG = NGC ? NGC : P.ng;
  constexpr int B = kTileMax, H = kTileMax / 2;
  const int w = tid >> 5, rh = w & 1, lh = (w >> 1) & 1, pt = ((w >> 2) << 5) | (tid & 31);
  const long long g = vbx * kDQuadPts + pt;
  const bool act = g < NG;
  const C zero = cmk<C>(R(0), R(0));
  const C* V = P.S + (long long)(d.slot0 + lh * H * B + rh * H) * NG + g;
  const C* X = static_cast<const C*>(P.X) + (long long)(d.l0 + lh * H) * P.ld + g;
  const C* Y = static_cast<const C*>(P.Y) + (long long)(d.r0 + rh * H) * P.ld + g;
  // the output orbitals of this thread: Out_l for lh = 0, Out_r for lh = 1
  C* O = (lh ? static_cast<C*>(P.OutY) + (long long)d.r0 * P.ld : static_cast<C*>(P.OutX) + (long long)d.l0 * P.ld) +
         (long long)rh * H * P.ld + g;
  C v[H][H], xl[H], al[H], ar[H], out[H];
#pragma unroll
  for (int li = 0; li < H; ++li)
#pragma unroll
    for (int ri = 0; ri < H; ++ri) v[li][ri] = act ? __ldcs(V + (long long)(li * B + ri) * NG) : zero;
#pragma unroll
  for (int o = 0; o < H; ++o) {
    xl[o] = act ? X[(long long)o * P.ld] : zero;
    al[o] = zero;
    ar[o] = zero;
  }
#pragma unroll
  for (int ri = 0; ri < H; ++ri) {
    const C yr = act ? Y[(long long)ri * P.ld] : zero;
#pragma unroll
    for (int li = 0; li < H; ++li) al[li] = cfmac(al[li], v[li][ri], yr);
  }
#pragma unroll
  for (int o = 0; o < H; ++o) out[o] = act ? O[(long long)o * P.ld] : zero;
  // exchange, per point: [0, 4) the right sums so far of rh = 0, [4, 8) of rh = 1,
  // [8, 12) the left sums of (0, 1), [12, 16) of (1, 0), [16, 20) of (1, 1)
  C* xp = xch + pt;
  if (lh == 0) {
#pragma unroll
    for (int li = 0; li < H; ++li)
#pragma unroll
      for (int ri = 0; ri < H; ++ri) ar[ri] = cfma(ar[ri], xl[li], v[li][ri]);
#pragma unroll
    for (int o = 0; o < H; ++o) xp[(rh * H + o) * kDQuadPts] = ar[o];
  }
  if (lh | rh) {
#pragma unroll
    for (int o = 0; o < H; ++o) xp[((1 + 2 * lh + rh) * H + o) * kDQuadPts] = al[o];
  }
  __syncthreads();
  if (!act) return;
  if (lh == 0) {
#pragma unroll
    for (int o = 0; o < H; ++o) {
      const C lo = rh ? xp[(3 * H + o) * kDQuadPts] : al[o];
      const C hi = rh ? xp[(4 * H + o) * kDQuadPts] : xp[(2 * H + o) * kDQuadPts];
      ar[o] = cadd(lo, hi);
    }
  } else {
#pragma unroll
    for (int o = 0; o < H; ++o) ar[o] = xp[(rh * H + o) * kDQuadPts];
#pragma unroll
    for (int li = 0; li < H; ++li)
#pragma unroll
      for (int ri = 0; ri < H; ++ri) ar[ri] = cfma(ar[ri], xl[li], v[li][ri]);
  }
#pragma unroll
  for (int o = 0; o < H; ++o)
    O[(long long)o * P.ld] = cmk<C>(out[o].x - P.scale * ar[o].x, out[o].y - P.scale * ar[o].y);
}

// One-sided tile (V_X[Phi] Psi, Poisson solves) of complex vectors, two threads
// per grid point: half h takes the right orbitals r0 + 4h .. r0 + 4h + 3 and sums
// over the left ones in turn, four at a time, so that a thread has 16 potentials
// in flight (a batch is often one tile, and with one thread per point its launch
// held two blocks per SM with eight potentials in flight per thread): V_X of 61
// orbitals on 37 bands, 48x40x36: 1.43 -> 1.34 ms.
constexpr int kDRectPts = 128;   // points per 256-thread block
template <typename R, long long NGC>
__device__ __forceinline__ void d_rect(const PointParams<R>& P, const TileDesc& d, long long vbx, int tid) {
  using C = cplx<R>;
  const long long NG = NGC ? NGC : P.ng;
  constexpr int H = kTileMax / 2, U = 4;
  const int h = (tid >> 5) & 1, n = d.nr - h * H < H ? d.nr - h * H : H;   // right orbitals of this thread
  const long long g = vbx * kDRectPts + (((tid >> 6) << 5) | (tid & 31));
  if (g >= NG || n <= 0) return;
  const C* V = P.S + (long long)(d.slot0 + h * H) * NG + g;
  const C* X = static_cast<const C*>(P.X) + (long long)d.l0 * P.ld + g;
  C ar[H];
#pragma unroll
  for (int o = 0; o < H; ++o) ar[o] = cmk<C>(R(0), R(0));
  int li = 0;
  if (n == H) {
    for (; li + U <= d.nl; li += U) {
      C x[U], v[U][H];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        x[u] = X[(long long)(li + u) * P.ld];
#pragma unroll
        for (int o = 0; o < H; ++o) v[u][o] = __ldcs(V + (long long)((li + u) * d.nr + o) * NG);
      }
#pragma unroll
      for (int u = 0; u < U; ++u)
#pragma unroll
        for (int o = 0; o < H; ++o) ar[o] = cfma(ar[o], x[u], v[u][o]);
    }
  }
  for (; li < d.nl; ++li) {
    const C x = X[(long long)li * P.ld];
#pragma unroll
    for (int o = 0; o < H; ++o)
      if (o < n) ar[o] = cfma(ar[o], x, __ldcs(V + (long long)(li * d.nr + o) * NG));
  }
#pragma unroll
  for (int o = 0; o < H; ++o)
    if (o < n) rmw_out<R, false, false>(P.OutY, (long long)(d.r0 + h * H + o) * P.ld + g, ar[o], P.scale);
}

// Pass D (complex vectors) for point block `vbx` (nthr points) of tile `d`;
// NGC = N_g at compile time (cubic grids) or 0 (read from the parameters).
template <typename R, bool REAL, bool COH, bool FULL_OFF, long long NGC>
__device__ __forceinline__ void body_d_cplx(const PointParams<R>& P, const TileDesc& d, long long vbx, int tid,
                                            int nthr) {
  const long long NG = NGC ? NGC : P.ng;
  const long long g = vbx * nthr + tid;
  if (g >= NG) return;
  const cplx<R>* V = P.S + (long long)d.slot0 * NG + g;
  if (d.kind == 1 && d.nl == kTileMax) {
    d_full_diag<R, REAL, COH, NGC>(P, d, V, g);
  } else if (FULL_OFF && d.kind == 0 && d.nl == kTileMax && d.nr == kTileMax) {
    d_full_off<R, REAL, COH, NGC>(P, d, V, g);
  } else if (d.kind == 1) {
    cplx<R> x[kTileMax], acc[kTileMax];
#pragma unroll
    for (int o = 0; o < kTileMax; ++o) {
      acc[o] = cmk<cplx<R>>(R(0), R(0));
      x[o] = o < d.nl ? load_vec<R, REAL>(P.X, (long long)(d.l0 + o) * P.ld + g) : acc[o];
    }
    int q = 0;
#pragma unroll
    for (int li = 0; li < kTileMax; ++li) {
#pragma unroll
      for (int ri = li; ri < kTileMax; ++ri) {
        if (li < d.nl && ri < d.nl) {
          const cplx<R> v = ldx<COH>(V + (long long)q * NG);
          ++q;
          acc[ri] = cfma(acc[ri], x[li], v);
          if (ri != li) acc[li] = cfmac(acc[li], v, x[ri]);   // x_r conj(v)
        }
      }
    }
#pragma unroll
    for (int o = 0; o < kTileMax; ++o)
      if (o < d.nl) rmw_out<R, REAL, COH>(P.OutY, (long long)(d.l0 + o) * P.ld + g, acc[o], P.scale);
  } else if (d.kind == 0) {
    cplx<R> xl[kTileMax], yr[kTileMax], al[kTileMax], ar[kTileMax];
#pragma unroll
    for (int o = 0; o < kTileMax; ++o) {
      al[o] = cmk<cplx<R>>(R(0), R(0));
      ar[o] = al[o];
      xl[o] = o < d.nl ? load_vec<R, REAL>(P.X, (long long)(d.l0 + o) * P.ld + g) : al[o];
      yr[o] = o < d.nr ? load_vec<R, REAL>(P.Y, (long long)(d.r0 + o) * P.ld + g) : al[o];
    }
#pragma unroll
    for (int li = 0; li < kTileMax; ++li) {
#pragma unroll
      for (int ri = 0; ri < kTileMax; ++ri) {
        if (li < d.nl && ri < d.nr) {
          const cplx<R> v = ldx<COH>(V + (long long)(li * d.nr + ri) * NG);
          ar[ri] = cfma(ar[ri], xl[li], v);
          al[li] = cfmac(al[li], v, yr[ri]);
        }
      }
    }
#pragma unroll
    for (int o = 0; o < kTileMax; ++o) {
      if (o < d.nr) rmw_out<R, REAL, COH>(P.OutY, (long long)(d.r0 + o) * P.ld + g, ar[o], P.scale);
      if (o < d.nl) rmw_out<R, REAL, COH>(P.OutX, (long long)(d.l0 + o) * P.ld + g, al[o], P.scale);
    }
  } else {
    cplx<R> ar[kTileMax];
#pragma unroll
    for (int o = 0; o < kTileMax; ++o) ar[o] = cmk<cplx<R>>(R(0), R(0));
    for (int li = 0; li < d.nl; ++li) {
      const cplx<R> xv = load_vec<R, REAL>(P.X, (long long)(d.l0 + li) * P.ld + g);
#pragma unroll
      for (int ri = 0; ri < kTileMax; ++ri) {
        if (ri < d.nr) {
          const cplx<R> v = ldx<COH>(V + (long long)(li * d.nr + ri) * NG);
          ar[ri] = cfma(ar[ri], xv, v);
        }
      }
    }
#pragma unroll
    for (int o = 0; o < kTileMax; ++o)
      if (o < d.nr) rmw_out<R, REAL, COH>(P.OutY, (long long)(d.r0 + o) * P.ld + g, ar[o], P.scale);
  }
}

// ---- pass D for real vectors: a slot holds v = V_lr + i V_lr2 (decode_slot_real)
template <typename R, bool COH>
__device__ __forceinline__ void rmw_real(void* base, long long idx, R acc, R scale) {
  R* o = static_cast<R*>(base) + idx;
  stx<COH>(o, ldx<COH>(o) - scale * acc);
}
// full tiles read their potentials once, with the streaming hint
template <bool FULL, bool COH, typename T> __device__ __forceinline__ T ldv(const T* p) {
  if constexpr (FULL) return __ldcs(p);
  else return ldx<COH>(p);
}

// Diagonal tile: Out_l -= sum over its pairs; a pair (l, r != l) feeds both
// Out_r (x_l V_lr) and Out_l (x_r V_lr), the pair (l, l) Out_l once.
template <typename R, bool COH, bool FULL, long long NGC>
__device__ __forceinline__ void d_real_diag(const PointParams<R>& P, const TileDesc& d, const cplx<R>* V,
                                            long long g) {
  const long long NG = NGC ? NGC : P.ng;
  constexpr int B = kTileMax;
  const int n = FULL ? B : d.nl;
  const R* X = static_cast<const R*>(P.X);
  R x[B], acc[B];
#pragma unroll
  for (int o = 0; o < B; ++o) {
    acc[o] = R(0);
    x[o] = (FULL || o < n) ? X[(long long)(d.l0 + o) * P.ld + g] : R(0);
  }
  int q = 0;
#pragma unroll
  for (int li = 0; li < B; ++li) {
    if (FULL || li < n) {
      const cplx<R> v0 = ldv<FULL, COH>(V + (long long)q * NG);
      ++q;
      acc[li] += x[li] * v0.x;
#pragma unroll
      for (int ri = li + 1; ri < B; ri += 2) {
        if (FULL || ri < n) {
          const cplx<R> v = ldv<FULL, COH>(V + (long long)q * NG);
          ++q;
          acc[ri] += x[li] * v.x;
          acc[li] += v.x * x[ri];
          if (ri + 1 < B && (FULL || ri + 1 < n)) {
            acc[ri + 1] += x[li] * v.y;
            acc[li] += v.y * x[ri + 1];
          }
        }
      }
    }
  }
#pragma unroll
  for (int o = 0; o < B; ++o)
    if (FULL || o < n) rmw_real<R, COH>(P.OutY, (long long)(d.l0 + o) * P.ld + g, acc[o], P.scale);
}

// Off-diagonal tile of a symmetric schedule (one thread per point).
template <typename R, bool COH, bool FULL, long long NGC>
__device__ __forceinline__ void d_real_off(const PointParams<R>& P, const TileDesc& d, const cplx<R>* V,
                                           long long g) {
  const long long NG = NGC ? NGC : P.ng;
  constexpr int B = kTileMax, W2 = kTileMax / 2;
  const int nl = FULL ? B : d.nl, nr = FULL ? B : d.nr, w = FULL ? W2 : (d.nr + 1) / 2;
  const R* X = static_cast<const R*>(P.X);
  const R* Y = static_cast<const R*>(P.Y);
  R xl[B], yr[B], al[B], ar[B];
#pragma unroll
  for (int o = 0; o < B; ++o) {
    al[o] = R(0);
    ar[o] = R(0);
    xl[o] = (FULL || o < nl) ? X[(long long)(d.l0 + o) * P.ld + g] : R(0);
    yr[o] = (FULL || o < nr) ? Y[(long long)(d.r0 + o) * P.ld + g] : R(0);
  }
#pragma unroll
  for (int li = 0; li < B; ++li) {
#pragma unroll
    for (int m = 0; m < W2; ++m) {
      if ((FULL || li < nl) && (FULL || 2 * m < nr)) {
        const cplx<R> v = ldv<FULL, COH>(V + (long long)(li * w + m) * NG);
        ar[2 * m] += xl[li] * v.x;
        al[li] += v.x * yr[2 * m];
        if (FULL || 2 * m + 1 < nr) {
          ar[2 * m + 1] += xl[li] * v.y;
          al[li] += v.y * yr[2 * m + 1];
        }
      }
    }
  }
#pragma unroll
  for (int o = 0; o < B; ++o) {
    if (FULL || o < nr) rmw_real<R, COH>(P.OutY, (long long)(d.r0 + o) * P.ld + g, ar[o], P.scale);
    if (FULL || o < nl) rmw_real<R, COH>(P.OutX, (long long)(d.l0 + o) * P.ld + g, al[o], P.scale);
  }
}

// One-sided tile (V_X[Phi] Psi, Poisson solves): Out_r -= sum_l x_l V_lr.
template <typename R, bool COH, long long NGC>
__device__ __forceinline__ void d_real_rect(const PointParams<R>& P, const TileDesc& d, const cplx<R>* V,
                                            long long g) {
  const long long NG = NGC ? NGC : P.ng;
  constexpr int B = kTileMax, W2 = kTileMax / 2;
  const int w = (d.nr + 1) / 2;
  const R* X = static_cast<const R*>(P.X);
  R ar[B];
#pragma unroll
  for (int o = 0; o < B; ++o) ar[o] = R(0);
  for (int li = 0; li < d.nl; ++li) {
    const R xv = X[(long long)(d.l0 + li) * P.ld + g];
#pragma unroll
    for (int m = 0; m < W2; ++m) {
      if (2 * m < d.nr) {
        const cplx<R> v = ldx<COH>(V + (long long)(li * w + m) * NG);
        ar[2 * m] += xv * v.x;
        if (2 * m + 1 < d.nr) ar[2 * m + 1] += xv * v.y;
      }
    }
  }
#pragma unroll
  for (int o = 0; o < B; ++o)
    if (o < d.nr) rmw_real<R, COH>(P.OutY, (long long)(d.r0 + o) * P.ld + g, ar[o], P.scale);
}

// Full off-diagonal tile of real vectors with two threads per point, as
// d_split_off: half h takes the right orbitals r0 + 4h .. r0 + 4h + 3 (slots
// li * 4 + 2h, li * 4 + 2h + 1 of each row).
template <typename R, long long NGC>
__device__ __forceinline__ void d_split_off_real(const PointParams<R>& P, const TileDesc& d, long long vbx, int tid,
                                                 R* xch) {
  const long long NG = NGC ? NGC : P.ng;
  constexpr int B = kTileMax, H = kTileMax / 2, Q = H / 2;
  const int h = (tid >> 5) & 1;
  const int pt = ((tid >> 6) << 5) | (tid & 31);
  const long long g = vbx * kDSplitPts + pt;
  const bool act = g < NG;
  const cplx<R>* V = P.S + (long long)d.slot0 * NG + g;
  const R* X = static_cast<const R*>(P.X);
  const R* Y = static_cast<const R*>(P.Y);
  R xl[B], yr[H], al[B], ar[H];
#pragma unroll
  for (int o = 0; o < B; ++o) {
    al[o] = R(0);
    xl[o] = act ? X[(long long)(d.l0 + o) * P.ld + g] : R(0);
  }
#pragma unroll
  for (int o = 0; o < H; ++o) {
    ar[o] = R(0);
    yr[o] = act ? Y[(long long)(d.r0 + h * H + o) * P.ld + g] : R(0);
  }
  if (act) {
#pragma unroll
    for (int li = 0; li < B; ++li) {
#pragma unroll
      for (int m = 0; m < Q; ++m) {
        const cplx<R> v = __ldcs(V + (long long)(li * H + h * Q + m) * NG);
        ar[2 * m] += xl[li] * v.x;
        ar[2 * m + 1] += xl[li] * v.y;
        al[li] += v.x * yr[2 * m];
        al[li] += v.y * yr[2 * m + 1];
      }
    }
  }
#pragma unroll
  for (int o = 0; o < H; ++o) xch[o * 256 + tid] = h ? al[o] : al[H + o];   // the partner's half
  __syncthreads();
  if (!act) return;
  const int partner = tid ^ 32;
#pragma unroll
  for (int o = 0; o < H; ++o) {
    const R own = h ? al[H + o] : al[o];
    const R other = xch[o * 256 + partner];
    const R lo = h ? other : own, hi = h ? own : other;                    // r-half 0 first, then 1
    rmw_real<R, false>(P.OutX, (long long)(d.l0 + h * H + o) * P.ld + g, lo + hi, P.scale);
    rmw_real<R, false>(P.OutY, (long long)(d.r0 + h * H + o) * P.ld + g, ar[o], P.scale);
  }
}

// Pass D for point block `vbx` (nthr points) of tile `d`.
template <typename R, bool REAL, bool COH, bool FULL_OFF, long long NGC>
__device__ __forceinline__ void body_d(const PointParams<R>& P, const TileDesc& d, long long vbx, int tid,
                                       int nthr) {
  if constexpr (REAL) {
    const long long g = vbx * nthr + tid;
    if (g >= (NGC ? NGC : P.ng)) return;
    const cplx<R>* V = P.S + (long long)d.slot0 * (NGC ? NGC : P.ng) + g;
    if (d.kind == 1) {
      if (d.nl == kTileMax) d_real_diag<R, COH, true, NGC>(P, d, V, g);
      else d_real_diag<R, COH, false, NGC>(P, d, V, g);
    } else if (d.kind == 0) {
      if (FULL_OFF && d.nl == kTileMax && d.nr == kTileMax) d_real_off<R, COH, true, NGC>(P, d, V, g);
      else d_real_off<R, COH, false, NGC>(P, d, V, g);
    } else {
      d_real_rect<R, COH, NGC>(P, d, V, g);
    }
  } else {
    body_d_cplx<R, REAL, COH, FULL_OFF, NGC>(P, d, vbx, tid, nthr);
  }
}

// ---------------------------------------------------------------- four-kernel mode
template <typename R, int NX, int NY, bool REAL, bool POIS>
__global__ void __launch_bounds__(kMaxLine<NX, NY> * plane_items<R, NX, NY>(), plane_blocks<R, NX, NY>())
pass_a_kernel(const __grid_constant__ PlaneParams<R, NX, NY> P) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  body_a<R, NX, NY, REAL, false, plane_items<R, NX, NY>(), true, kLine2<R, NX, NY>, POIS>(
      P, P.tiles, P.ntiles, P.npairs, reinterpret_cast<cplx<R>*>(smem_raw), blockIdx.x, threadIdx.x);
}

// The two lanes of a line sit 16 apart: lanes 0-15 of a warp hold the even
// samples of 16 consecutive lines, lanes 16-31 the odd ones. A half-warp then
// touches 16 consecutive columns of one row (or one column of 16 consecutive
// padded rows), which are free of bank conflicts in the plane buffer and whole
// 128-byte lines in global memory; with neighbouring lanes sharing a line every
// access of the buffer was a two-way conflict (96^3, one 64-pair tile: A 220 ->
// 212, C 192 -> 188 us).
__device__ __forceinline__ int split_line(int tid) { return ((tid >> 5) << 4) | (tid & 15); }
__device__ __forceinline__ int split_half(int tid) { return (tid >> 4) & 1; }
template <typename T> __device__ __forceinline__ T shfl_pair(T v) {
  T r;
  r.x = __shfl_xor_sync(0xffffffffu, v.x, 16);
  r.y = __shfl_xor_sync(0xffffffffu, v.y, 16);
  return r;
}

// A length-N transform of a line held by two lanes (split_line): lane h
// holds the samples 2m + h in a[], and on return holds y[j] = Y[hN/4 + j] and
// y[N/4 + j] = Y[hN/4 + j + N/2] (the forward or inverse DFT, unnormalised):
// a DFT of N/2 per lane, the lane-1 twiddles w^{+-k}, one shuffle per value
// and the radix-2 combine (decimation in time).
// The halves are exchanged before the twiddles, so each lane multiplies only
// the H odd-half values of its own outputs (by w^j on lane 0, w^{H+j} on lane
// 1: two compile-time constants, selected).
template <typename R> __device__ __forceinline__ cplx<R> csel(bool c, cplx<R> a, cplx<R> b) {
  return cmk<cplx<R>>(c ? a.x : b.x, c ? a.y : b.y);
}
// The radix-2 step alone, on a[] already holding the half-length transform:
// each output goes to sink(j, Y) as soon as it is formed (y index j as in
// split_line_dft), so a caller that stores it right away frees the registers
// of a[j], a[H + j] within the loop instead of holding a second array.
template <int N, bool INV, typename R, typename Sink>
__device__ __forceinline__ void split_combine(const cplx<R> (&a)[N / 2], int h, const TwTable<R, N>& tw,
                                              Sink sink) {
  using C = cplx<R>;
  constexpr int H = N / 4;
#pragma unroll
  for (int j = 0; j < H; ++j) {
    const C recv = shfl_pair(h ? a[j] : a[H + j]);       // lane 0 gets O[j], lane 1 gets E[H + j]
    const C ev = h ? recv : a[j];                        // E[hH + j]
    const C od = h ? a[H + j] : recv;                    // O[hH + j]
    const C w = csel<R>(h, twiddle_value<N, N, INV, R>(H + j, tw), twiddle_value<N, N, INV, R>(j, tw));
    const C t = cmul(od, w);
    sink(j, cadd<false>(ev, t));
    sink(H + j, csub<false>(ev, t));
  }
}
template <int N, bool INV, typename R>
__device__ __forceinline__ void split_line_dft(cplx<R> (&a)[N / 2], cplx<R> (&y)[N / 2], int h,
                                               const TwTable<R, N>& tw) {
  dft<N / 2, N, INV, R, false>(a, tw);                     // E (lane 0) or O (lane 1)
  split_combine<N, INV, R>(a, h, tw, [&](int j, cplx<R> v) { y[j] = v; });
}
// Pass B for the large FP64 pencils (n_z >= 64), whose whole pencil per thread
// spills (FP32 pencils of 64 and 96 take the four-warp form, pass_b_quad_kernel):
// two lanes per z-pencil (split_line; 128 pencils per block). Lane h holds the samples z = 2m + h and transforms them with a DFT of
// N/2:
//   forward  Y[k] = E[k] + w^k O[k], Y[k + N/2] = E[k] - w^k O[k]
//            (E, O the half-length transforms of the even / odd samples,
//            w = exp(-2 pi i / N)); lane h keeps k in [hN/4, (h+1)N/4) and gets
//            the partner's half of E or w^k O by one shuffle per value;
//   inverse  x[2m] = IDFT(Y[k] + Y[k + N/2]), x[2m+1] = IDFT((Y[k] - Y[k + N/2]) w^-k)
//            over k < N/2; each lane forms its quarter of both sequences and
//            swaps the other lane's by shuffle; lane 0 transforms the first,
//            lane 1 the second.
// Lane roles are selected arithmetically (no divergent branches). At n_z = 48
// the shuffles cost more than the occupancy gains, so shorter pencils keep one
// thread per pencil.
constexpr int kBSplitPencils = 128;   // pencils per 256-thread block of the split pass B
// FP64 pencils of 64+ points need the whole register file of a thread: one
// block per SM. (For FP32 pencils of 96 this form spilled a few hundred bytes
// at two blocks per SM, still faster than one block without spills: 25.7 vs
// 31.7 ms of pass B per 96^3 build of 128 orbitals; the four-warp form takes
// 19.3 ms.)
template <typename R, int N> constexpr int kBSplitBlocks = sizeof(R) == 8 ? 1 : 2;
template <int NZ> constexpr bool kSplitPencil = NZ >= 64 && NZ % 4 == 0;

template <typename R, int NZ, bool CUBE>
__global__ void __launch_bounds__(256, kBSplitBlocks<R, NZ>)
pass_b_split_kernel(const __grid_constant__ PencilParams<R, NZ> P, int mode) {
  using C = cplx<R>;
  constexpr int N = NZ, M = N / 2, H = N / 4;
  static_assert(N % 4 == 0, "the split pass B halves a pencil twice");
  __shared__ double red[8];
  griddep_wait();
  const PencilGeom<R, NZ, CUBE> G(P);
  const int nxy = G.nxy;
  const int tid = threadIdx.x, h = split_half(tid);
  const long long gid = (long long)blockIdx.x * kBSplitPencils + split_line(tid);
  const bool active = gid < (long long)P.npairs * nxy;    // same for both lanes of a pencil
  const int p = active ? (int)(gid / nxy) : 0;
  const int f = active ? (int)(gid % nxy) : 0;
  C* s = P.S + (long long)p * N * nxy + f;
  const C zero = cmk<C>(R(0), R(0));
  C a[M];
#pragma unroll
  for (int m = 0; m < M; ++m) a[m] = active ? s[(long long)(2 * m + h) * nxy] : zero;
  C y[M];                                                  // y[j] = Y[hH + j], y[H + j] = Y[hH + j + M]
  split_line_dft<N, false, R>(a, y, h, P.tw);
  R acc = R(0);
  const R* kt = P.Kt + G.kt_pencil(f);
#pragma unroll
  for (int j = 0; j < M; ++j) {
    const int kz = h * H + (j < H ? j : j - H + M);
    const R k = kt[kfold<N>(kz) * G.kzs];
    if (mode != 0) acc += k * (y[j].x * y[j].x + y[j].y * y[j].y);
    y[j] = cscale(y[j], k);
  }
  double e = 0.0;
  if (mode != 0 && active) e = slot_weight(P.tiles, P.ntiles, p, P.packed) * (double)acc;
  if (mode != 1) {
#pragma unroll
    for (int j = 0; j < H; ++j) {                          // k = hH + j
      const C sum = cadd(y[j], y[H + j]);
      const C w = csel<R>(h, twiddle_value<N, N, true, R>(H + j, P.tw), twiddle_value<N, N, true, R>(j, P.tw));
      const C dif = cmul(csub(y[j], y[H + j]), w);
      const C recv = shfl_pair(h ? sum : dif);
      a[j] = h ? recv : sum;                               // lane 0: the sums, lane 1: the differences
      a[H + j] = h ? dif : recv;
    }
    dft<M, N, true, R>(a, P.tw);                           // x[2m + h] = a[m]
    if (active) {
#pragma unroll
      for (int m = 0; m < M; ++m) s[(long long)(2 * m + h) * nxy] = a[m];
    }
  }
  if (mode != 0) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) e += __shfl_down_sync(0xffffffffu, e, o);
    if ((tid & 31) == 0) red[tid >> 5] = e;
    __syncthreads();
    if (tid == 0) {
      double sum = 0.0;
      for (int w = 0; w < 8; ++w) sum += red[w];
      P.Epart[blockIdx.x] += sum;                          // one block per slot
    }
  }
}

// Planes whose passes use the two-lane line transforms (one plane per block):
// the lines that do not fit a thread's registers beside enough warps. A whole
// FP32 line of 64 needs 168 registers (three 128-thread blocks, 12 warps per
// SM) and still beats the two-lane form, whose selects and shuffles are 40 % of
// its instructions: 64^3 A 60.4 -> 51.8, C 59.4 -> 55.3 us per 64-pair tile,
// 48^3 25.6 -> 21.3 and 20.5 -> 18.4. At 96 (234 registers, six warps) it
// loses: A 207 -> 223, C 188 -> 213. FP64 lines take the two-lane form from 64,
// with one or two blocks per SM.
constexpr int kSplitMinEdge = 96;
constexpr int kSplitMinEdgeF64 = 64;
template <typename R, int NX, int NY> constexpr bool kSplitPlanes =
    NX % 4 == 0 && NY % 4 == 0 &&
    (sizeof(R) == 4 ? kMaxLine<NX, NY> >= kSplitMinEdge : kMaxLine<NX, NY> >= kSplitMinEdgeF64);
template <typename R, int NX, int NY> constexpr int kSplitBlocks =
    sizeof(R) == 8 && kMaxLine<NX, NY> >= 96 ? 1 : 2;
template <int NX, int NY> constexpr bool kSplitWarps = (2 * kMaxLine<NX, NY>) % 32 == 0;   // whole warps of line pairs
template <typename R, int NX, int NY> constexpr size_t kSplitSmem = (size_t)NY * (NX + 1) * sizeof(cplx<R>);

// frequency index held in y[j] by lane h
template <int N> __device__ __forceinline__ int split_index(int j, int h) {
  return h * (N / 4) + (j < N / 4 ? j : j - N / 4 + N / 2);
}

// Passes A and C with two lanes per line: one plane per block (2 max(n_x, n_y)
// threads), each pass's two line transforms by split_line_dft, the transpose
// through shared memory as in the one-thread-per-line form. Half the registers
// of a whole line per thread (which at 96^3 would need over 200), so more
// warps per SM hide the latency of the plane loads and stores. On a
// non-square plane the lanes past the shorter edge compute on zeros and store
// nothing, so every lane of a warp takes part in the shuffles. Scalar additions:
// with packed ones the 96-point passes measured 212 -> 207 (A) but 188 -> 207 us
// (C) per 64-pair tile.
template <typename R, int NX, int NY, bool REAL, bool POIS>
__global__ void __launch_bounds__(2 * kMaxLine<NX, NY>, kSplitBlocks<R, NX, NY>)
pass_a_split_kernel(const __grid_constant__ PlaneParams<R, NX, NY> P) {
  using C = cplx<R>;
  static_assert(kSplitWarps<NX, NY>, "a line's lanes share a warp");
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* buf = reinterpret_cast<C*>(smem_raw);
  const int tid = threadIdx.x, q = split_line(tid), h = split_half(tid);
  const long long item = blockIdx.x;                      // one (pair, z) plane per block, z-major:
  const int z = (int)(item / P.npairs), p = (int)(item % P.npairs);   // pairs sharing a plane run together
  int l, r, r2 = -1;
  if constexpr (REAL) decode_slot_real(P.tiles, P.ntiles, p, l, r, r2);
  else decode_pair(P.tiles, P.ntiles, p, l, r);
  const C zero = cmk<C>(R(0), R(0));
  {   // column x = q: samples y = 2m + h
    constexpr int M = NY / 2;
    const bool act = q < NX;
    C a[M];
    const long long xo = (long long)l * P.ld + (long long)z * NX * NY + q;
    const long long yo = (long long)r * P.ld + (long long)z * NX * NY + q;
    if constexpr (REAL) {                                  // x_l (y_r + i y_r2)
      const R* Xr = static_cast<const R*>(P.X);
      const R* Yr = static_cast<const R*>(P.Y);
      const bool two = r2 >= 0;
      const long long y2o = (long long)(two ? r2 : r) * P.ld + (long long)z * NX * NY + q;
#pragma unroll
      for (int m = 0; m < M; ++m) {
        const int yy = 2 * m + h;
        const R xv = !act ? R(0) : POIS ? R(1) : Xr[xo + yy * NX];
        a[m] = act ? cmk<C>(xv * Yr[yo + yy * NX], two ? xv * Yr[y2o + yy * NX] : R(0)) : zero;
      }
    } else {
#pragma unroll
      for (int m = 0; m < M; ++m) {
        const int yy = 2 * m + h;
        a[m] = act ? cmulc(POIS ? cmk<C>(R(1), R(0)) : load_vec<R, REAL>(P.X, xo + yy * NX),
                           load_vec<R, REAL>(P.Y, yo + yy * NX))
                   : zero;
      }
    }
    dft<M, NY, false, R, false>(a, P.tw.ty());            // along y
    split_combine<NY, false, R>(a, h, P.tw.ty(), [&](int j, C v) {
      if (act) buf[split_index<NY>(j, h) * (NX + 1) + q] = v;
    });
  }
  __syncthreads();
  {   // row ky = q: samples x = 2m + h
    constexpr int M = NX / 2;
    const bool act = q < NY;
    C a[M];
#pragma unroll
    for (int m = 0; m < M; ++m) a[m] = act ? buf[q * (NX + 1) + 2 * m + h] : zero;
    dft<M, NX, false, R, false>(a, P.tw.tx());            // along x
    griddep_wait();                                        // the previous batch's pass D still reads S
    if (P.clear && blockIdx.x == 0 && tid == 0) P.clear[0] = P.clear[1] = 0;
    C* out = P.S + ((long long)p * P.nz + z) * NX * NY + q;
    split_combine<NX, false, R>(a, h, P.tw.tx(), [&](int j, C v) {
      if (act) out[(long long)split_index<NX>(j, h) * NY] = v;
    });
  }
}

template <typename R, int NX, int NY, bool POIS>
__global__ void __launch_bounds__(2 * kMaxLine<NX, NY>, kSplitBlocks<R, NX, NY>)
pass_c_split_kernel(const __grid_constant__ PlaneParams<R, NX, NY> P) {
  using C = cplx<R>;
  static_assert(kSplitWarps<NX, NY>, "a line's lanes share a warp");
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* buf = reinterpret_cast<C*>(smem_raw);
  griddep_wait();
  const int tid = threadIdx.x, q = split_line(tid), h = split_half(tid);
  const long long item = blockIdx.x;
  const int p = (int)(item / P.nz), z = (int)(item % P.nz);
  C* plane = P.S + ((long long)p * P.nz + z) * NX * NY;
  const C zero = cmk<C>(R(0), R(0));
  {   // row ky = q of the spectrum: samples kx = 2m + h, inverse along x
    constexpr int M = NX / 2;
    const bool act = q < NY;
    C a[M];
#pragma unroll
    for (int m = 0; m < M; ++m) a[m] = act ? plane[(long long)(2 * m + h) * NY + q] : zero;
    dft<M, NX, true, R, false>(a, P.tw.tx());
    split_combine<NX, true, R>(a, h, P.tw.tx(), [&](int j, C v) {
      if (act) buf[q * (NX + 1) + split_index<NX>(j, h)] = v;   // row ky, column x
    });
  }
  __syncthreads();
  {   // column x = q: samples ky = 2m + h, inverse along y
    constexpr int M = NY / 2;
    const bool act = q < NX;
    C a[M];
#pragma unroll
    for (int m = 0; m < M; ++m) a[m] = act ? buf[(2 * m + h) * (NX + 1) + q] : zero;
    dft<M, NY, true, R, false>(a, P.tw.ty());
    const PlaneOut<R, NX, NY, false, POIS> out(P, p, z, plane);
    split_combine<NY, true, R>(a, h, P.tw.ty(), [&](int j, C v) {
      if (act) out.store(split_index<NY>(j, h) * NX + q, v);
    });
  }
}

// ---- four warps per 32 lines (pass B for FP32 pencils of 96)
// A length-N line transform (N = 4M, decimation in time by 4) is spread over
// four warps: the thread with phase h (warp-uniform) transforms the samples
// 4m + h (a DFT of M in registers) and multiplies by w_N^{hk}; after a block
// barrier the thread with phase h forms, for its M/4 frequencies k = hM/4 + j,
// the radix-4 combination Y[k + qM] = sum_h' (w_4)^{h'q} U_h'[k] (q = 0..3) of
// the four phases' values, read from shared memory. A thread holds a quarter of
// a line (M values) and needs no shuffles or lane-dependent selects (the phase
// is warp-uniform, so its twiddles are compile-time constants in one of four
// code paths). For the plane passes the same scheme measured slower than the
// two-lane form (six shared-memory accesses per point per pass: bound by the
// shared-memory pipe), so only pass B uses it.
template <int N, bool INV, typename R>
__device__ __forceinline__ void quad_sub_dft(cplx<R> (&a)[N / 4], int h, const TwTable<R, N>& tw) {
  constexpr int M = N / 4;
  dft<M, N, INV, R>(a, tw);
  if (h == 1) {
#pragma unroll
    for (int k = 1; k < M; ++k) a[k] = twiddle<N, N, INV, R>(a[k], k, tw);
  } else if (h == 2) {
#pragma unroll
    for (int k = 1; k < M; ++k) a[k] = twiddle<N, N, INV, R>(a[k], 2 * k, tw);
  } else if (h == 3) {
#pragma unroll
    for (int k = 1; k < M; ++k) a[k] = twiddle<N, N, INV, R>(a[k], 3 * k, tw);
  }
}

// The radix-4 step for one line whose value U_h'[k] sits at
// buf[base + (h'M + k) stride]: for j < M/4 and k = hM/4 + j,
// out[4j + q] = Y[k + qM].
template <int N, bool INV, typename R>
__device__ __forceinline__ void quad_combine(const cplx<R>* __restrict__ buf, int base, int stride, int h,
                                             cplx<R> (&out)[N / 4], const TwTable<R, N>& tw) {
  constexpr int M = N / 4, Q = M / 4;
#pragma unroll
  for (int j = 0; j < Q; ++j) {
    cplx<R> u[4];
#pragma unroll
    for (int hh = 0; hh < 4; ++hh) u[hh] = buf[base + (hh * M + h * Q + j) * stride];
    dft<4, N, INV, R>(u, tw);
#pragma unroll
    for (int q = 0; q < 4; ++q) out[4 * j + q] = u[q];
  }
}

// Pass B with four warps per 32 pencils (FP32 pencils of 64 and 96): warp h holds the
// samples z = 4m + h of its lane's pencil, transforms them (quad_sub_dft) and
// stores them to shared memory; after a barrier each thread forms the radix-4
// combination for its M/4 frequencies k = hM/4 + j, which gives it the 24
// spectrum values kz = k + qM (q = 0..3), multiplies them by K(G) (and sums
// the energy), and takes the inverse radix-4 step right away: for each of its k,
// Z_h'[k] = sum_q Y[k + qM] (w_4)^{-h'q} w_N^{-h'k}, h' = 0..3, written back to
// the same shared-memory places it read. After a second barrier warp h reads
// Z_h[k] for all k and an inverse DFT of M gives x[4m + h]. The 96-point pencil
// thus needs a quarter of it in registers per thread (no spills, where the
// two-lane form spills at two blocks per SM) and no shuffles.
constexpr int kQuadPencils = 32;   // pencils per 128-thread block of the four-warp pass B
// (At n_z = 48 the whole pencil per thread measured faster: 2.63 vs 2.84 ps per
// pair-point.)
template <typename R, int NZ> constexpr bool kQuadPencil = sizeof(R) == 4 && (NZ == 96 || NZ == 64);

// u[4j + h'] *= w_N^{-h'(HQ + j)} (inverse twiddles of warp phase H)
template <int N, int H, typename R>
__device__ __forceinline__ void quad_inv_twiddle(cplx<R> (&u)[N / 4], const TwTable<R, N>& tw) {
  constexpr int Q = N / 16;
#pragma unroll
  for (int j = 0; j < Q; ++j)
#pragma unroll
    for (int hp = 1; hp < 4; ++hp) u[4 * j + hp] = twiddle<N, N, true, R>(u[4 * j + hp], hp * (H * Q + j), tw);
}

template <typename R, int NZ, bool CUBE>
__global__ void __launch_bounds__(128, 5)
pass_b_quad_kernel(const __grid_constant__ PencilParams<R, NZ> P, int mode) {
  using C = cplx<R>;
  constexpr int N = NZ, M = N / 4, Q = M / 4, LP = kQuadPencils;
  static_assert(M % 4 == 0, "M / 4 frequencies per thread");
  __shared__ C buf[N * LP];                                // [phase h, k][pencil]
  __shared__ double red[4];
  griddep_wait();
  const PencilGeom<R, NZ, CUBE> G(P);
  const int nxy = G.nxy;
  const int h = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const long long gid = (long long)blockIdx.x * LP + lane;
  const bool active = gid < (long long)P.npairs * nxy;
  const int p = active ? (int)(gid / nxy) : 0;
  const int f = active ? (int)(gid % nxy) : 0;
  C* s = P.S + (long long)p * N * nxy + f;
  const C zero = cmk<C>(R(0), R(0));
  C a[M];
#pragma unroll
  for (int m = 0; m < M; ++m) a[m] = active ? s[(long long)(4 * m + h) * nxy] : zero;
  quad_sub_dft<N, false, R>(a, h, P.tw);
#pragma unroll
  for (int k = 0; k < M; ++k) buf[(h * M + k) * LP + lane] = a[k];
  __syncthreads();
  quad_combine<N, false, R>(buf, lane, LP, h, a, P.tw);    // a[4j + q] = Y[hQ + j + qM]
  R acc = R(0);
  const R* kt = P.Kt + G.kt_pencil(f);
#pragma unroll
  for (int j = 0; j < Q; ++j) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int kz = h * Q + j + q * M;
      const R kv = kt[kfold<N>(kz) * G.kzs];
      C& v = a[4 * j + q];
      if (mode != 0) acc += kv * (v.x * v.x + v.y * v.y);
      v = cscale(v, kv);
    }
  }
  if (mode != 1) {
#pragma unroll
    for (int j = 0; j < Q; ++j) {                          // inverse radix-4 over q: outputs by phase h'
      C u[4] = {a[4 * j], a[4 * j + 1], a[4 * j + 2], a[4 * j + 3]};
      dft<4, N, true, R>(u, P.tw);
#pragma unroll
      for (int hp = 0; hp < 4; ++hp) a[4 * j + hp] = u[hp];
    }
    if (h == 0) quad_inv_twiddle<N, 0, R>(a, P.tw);
    else if (h == 1) quad_inv_twiddle<N, 1, R>(a, P.tw);
    else if (h == 2) quad_inv_twiddle<N, 2, R>(a, P.tw);
    else quad_inv_twiddle<N, 3, R>(a, P.tw);
#pragma unroll
    for (int j = 0; j < Q; ++j)                            // the places quad_combine read
#pragma unroll
      for (int hp = 0; hp < 4; ++hp) buf[(hp * M + h * Q + j) * LP + lane] = a[4 * j + hp];
    __syncthreads();
#pragma unroll
    for (int k = 0; k < M; ++k) a[k] = buf[(h * M + k) * LP + lane];   // Z_h[k], k < M
    dft<M, N, true, R>(a, P.tw);                           // x[4m + h] = a[m]
    if (active) {
#pragma unroll
      for (int m = 0; m < M; ++m) s[(long long)(4 * m + h) * nxy] = a[m];
    }
  }
  if (mode != 0) {
    double e = active ? slot_weight(P.tiles, P.ntiles, p, P.packed) * (double)acc : 0.0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) e += __shfl_down_sync(0xffffffffu, e, o);
    if (lane == 0) red[h] = e;
    __syncthreads();
    if (threadIdx.x == 0) P.Epart[blockIdx.x] += red[0] + red[1] + red[2] + red[3];   // one block per slot
  }
}

// Blocks of 64 pencils, one per thread, so that a small call (one density on 48^3
// has 2304 pencils) spreads over the chip: nine blocks of 256 did not. 512
// threads per SM for FP32; FP64 pencils of 48 hold 96 doubles, so 256 (more would
// cap a thread at 128 registers and spill about 3 KB).
constexpr int kPencilThreads = 64;
template <typename R, int NZ, bool CUBE>
__global__ void __launch_bounds__(kPencilThreads, (sizeof(R) == 8 ? 256 : 512) / kPencilThreads)
pass_b_kernel(const __grid_constant__ PencilParams<R, NZ> P, int mode) {
  __shared__ double red[32];
  griddep_wait();
  body_b<R, NZ, false, CUBE>(P, P.tiles, P.ntiles, P.npairs, mode, blockIdx.x, threadIdx.x, blockDim.x, red,
                             mode != 0 ? P.Epart + blockIdx.x : nullptr);
}

template <typename R, int NX, int NY, bool POIS>
__global__ void __launch_bounds__(kMaxLine<NX, NY> * plane_items<R, NX, NY>(), plane_blocks<R, NX, NY>())
pass_c_kernel(const __grid_constant__ PlaneParams<R, NX, NY> P) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  griddep_wait();
  body_c<R, NX, NY, false, plane_items<R, NX, NY>(), kLine2<R, NX, NY>, POIS>(P, P.npairs, reinterpret_cast<cplx<R>*>(smem_raw), blockIdx.x,
                                                     threadIdx.x);
}

// The other tiles (diagonal, ragged, one-sided ones of real vectors): one thread
// per point, 256 points per block (beside tiles of smaller blocks in the same
// batch the upper blocks have no work). Not inlined, so that its larger register
// state does not spill into the full-tile path.
template <typename R, bool REAL, long long NGC>
__device__ __noinline__ void pass_d_other(const PointParams<R>& P, const TileDesc& d) {
  if ((long long)blockIdx.x * 256 >= (NGC ? NGC : P.ng)) return;
  body_d<R, REAL, false, false, NGC>(P, d, blockIdx.x, threadIdx.x, blockDim.x);
}

// Full off-diagonal tiles: FP32 four threads per grid point (d_quad_off) at three
// blocks per SM, FP64 two at two. Pass D waits on its loads, so what counts is
// that a thread issues them all at once: at four blocks (64 registers) the
// compiler splits them up, and where the spectrum does not fit L2 the pass took
// 47 us at 64^3 and 158 at 96^3 instead of 39 and 123. Two threads per point at
// four blocks took 49 and 150; 18.5 -> 16.4 at 48^3, 22.5 -> 18.4 at 32^3 (256 pairs).
// Points per block of a batch: the fewest that one of its tiles needs.
template <typename R> int d_points(const Batch& b, bool real) {
  int pts = 256;
  for (int t = 0; t < b.ntiles; ++t) {
    const TileDesc& d = b.t[t];
    if (d.kind == 0 && d.nl == kTileMax && d.nr == kTileMax) return sizeof(R) == 4 ? kDQuadPts : kDSplitPts;
    if (d.kind == 2 && !real) pts = kDRectPts;
  }
  return pts;
}
template <typename R, bool REAL, long long NGC>
__global__ void __launch_bounds__(256, sizeof(R) == 4 ? 3 : 2)
pass_d_kernel(const __grid_constant__ PointParams<R> P) {
  constexpr int B = kTileMax;
  __shared__ cplx<R> xch[sizeof(R) == 4 ? 5 * (B / 2) * kDQuadPts : (B / 2) * 256];
  griddep_wait();
  const TileDesc d = P.tiles[blockIdx.y];
  if (d.kind == 0 && d.nl == kTileMax && d.nr == kTileMax) {
    if constexpr (REAL) d_split_off_real<R, NGC>(P, d, blockIdx.x, threadIdx.x, reinterpret_cast<R*>(xch));
    else if constexpr (sizeof(R) == 4) d_quad_off<R, NGC>(P, d, blockIdx.x, threadIdx.x, xch);
    else d_split_off<R, REAL, NGC>(P, d, blockIdx.x, threadIdx.x, xch);
    return;
  }
  if constexpr (!REAL) {
    if (d.kind == 2) {
      d_rect<R, NGC>(P, d, blockIdx.x, threadIdx.x);
      return;
    }
  }
  pass_d_other<R, REAL, NGC>(P, d);
}

// ---------------------------------------------------------------- persistent engine
template <typename R, int N> struct EngineParams {
  PlaneParams<R, N, N> pl;      // npairs / ntiles unused: per batch from the table
  PencilParams<R, N> pe;
  PointParams<R> pt;
  const EngineBatch* batches;   // per batch: tiles, pairs, first task, tasks per pass
  int nbatches;
  int npasses;                  // 4 (Poisson) or 2 (energy only: A, B)
  long long ntasks;
  unsigned long long* head;     // task queue head
  unsigned* done;               // done[4 k + p]: finished tasks of pass p of batch k
  int* status;                  // plan status word: timeout -> ACE_ERR_TIMEOUT
  int mode;                     // 0: Poisson + accumulate; 1: energy only; 2: both
  unsigned spin_limit;          // polls before a dependent wait gives up
  unsigned wait_bias;           // added to every awaited count (0; a test hook)
};

__device__ __forceinline__ unsigned ld_acquire(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// A wait gives up after E.spin_limit polls (by default 2^22 sleeps of >= 256
// ns, about a second or more); the block then records ACE_ERR_TIMEOUT and
// leaves, and so do the blocks that wait on it, so the launch always ends. A
// block only ever waits before it starts a task, with nothing of its own in
// flight, so leaving is always safe. E.wait_bias > 0 (a test hook) asks for
// more finished tasks than a pass has, so that every dependent wait runs out.
template <typename R, int N, bool REAL>
__global__ void __launch_bounds__(kEngineThreads, 2)
pair_engine_kernel(const __grid_constant__ EngineParams<R, N> E) {
  constexpr int IPB = engine_items<R, N>();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ double red[32];
  __shared__ long long s_loc;
  __shared__ int s_batch, s_pass, s_stop;
  const int tid = threadIdx.x;
  cplx<R>* smem = reinterpret_cast<cplx<R>*>(smem_raw);
  for (;;) {
    if (tid == 0) {
      const long long t = (long long)atomicAdd(E.head, 1ull);
      int stop = 0, k = 0, pass = 0;
      long long loc = 0;
      if (t >= E.ntasks) {
        stop = 1;
      } else {
        int lo = 0, hi = E.nbatches - 1;   // last batch whose first task <= t
        while (lo < hi) {
          const int mid = (lo + hi + 1) >> 1;
          if (E.batches[mid].task0 <= t) lo = mid;
          else hi = mid - 1;
        }
        k = lo;
        const EngineBatch b = E.batches[k];
        loc = t - b.task0;
        while (loc >= b.n[pass]) { loc -= b.n[pass]; ++pass; }
        const unsigned* want = nullptr;
        unsigned target = 0;
        if (pass > 0) {
          want = E.done + kCtrStride * (4 * k + pass - 1);
          target = (unsigned)b.n[pass - 1] + E.wait_bias;
        } else if (k > 0) {
          want = E.done + kCtrStride * (4 * (k - 1) + E.npasses - 1);
          target = (unsigned)E.batches[k - 1].n[E.npasses - 1] + E.wait_bias;
        }
        if (want) {
          unsigned it = 0;
          while (ld_acquire(want) < target) {
            __nanosleep(it < 64 ? 32 : 256);
            if (++it > E.spin_limit) {
              E.status[0] = -6;   // ACE_ERR_TIMEOUT
              E.status[1] = (int)(t & 0x7fffffff);
              stop = 1;
              break;
            }
          }
        }
      }
      s_stop = stop;
      s_batch = k;
      s_pass = pass;
      s_loc = loc;
    }
    __syncthreads();
    if (s_stop) return;
    const int k = s_batch, pass = s_pass;
    const long long loc = s_loc;
    const EngineBatch& b = E.batches[k];
    const TileDesc* tiles = E.pl.tiles + b.toff;
    if (pass == 0) {
      body_a<R, N, N, REAL, true, IPB, false, false, false>(E.pl, tiles, b.ntiles, b.npairs, smem, loc, tid);
    } else if (pass == 1) {
      body_b<R, N, true, true>(E.pe, tiles, b.ntiles, b.npairs, E.mode, loc, tid, kEngineThreads, red,
                               E.mode != 0 ? E.pe.Epart + loc : nullptr);
    } else if (pass == 2) {
      body_c<R, N, N, true, IPB, false, false>(E.pl, b.npairs, smem, loc, tid);
    } else {
      const long long nvb = ((long long)N * N * N + kEngineThreads - 1) / kEngineThreads;
      const TileDesc d = tiles[loc / nvb];
      body_d<R, REAL, true, true, (long long)N * N * N>(E.pt, d, loc % nvb, tid, kEngineThreads);
    }
    __syncthreads();
    if (tid == 0) {
      __threadfence();
      atomicAdd(E.done + kCtrStride * (4 * k + pass), 1u);
    }
  }
}

// ---------------------------------------------------------------- host side
template <typename R, int NX, int NY>
void fill_plane(PlaneParams<R, NX, NY>& P, const PairLaunch& L, const Batch& b) {
  P.X = L.X;
  P.Y = L.Y;
  P.V = L.V;
  P.clear = L.clear;
  P.packed = L.real_io ? 1 : 0;
  P.S = static_cast<cplx<R>*>(L.S);
  P.ld = L.ld;
  P.nz = L.nz;
  P.npairs = b.npairs;
  P.tiles = L.dtiles;
  P.ntiles = b.ntiles;
  P.tw.fill(L.twx, L.twy);
}

template <typename R, int NZ>
void fill_pencil(PencilParams<R, NZ>& P, const PairLaunch& L, const Batch& b) {
  P.S = static_cast<cplx<R>*>(L.S);
  P.Kt = static_cast<const R*>(L.Kt);
  P.Epart = L.Epart;
  P.npairs = b.npairs;
  P.nx = L.nx;
  P.ny = L.ny;
  P.nxy = L.nx * L.ny;
  P.khy = L.ny / 2 + 1;
  P.kzs = (L.nx / 2 + 1) * (L.ny / 2 + 1);
  P.tiles = L.dtiles;
  P.ntiles = b.ntiles;
  P.packed = L.real_io ? 1 : 0;
  for (int k = 0; k < NZ; ++k) {
    P.tw.w[k].x = (R)L.twz[2 * k];
    P.tw.w[k].y = (R)L.twz[2 * k + 1];
  }
}

template <typename R>
void fill_point(PointParams<R>& P, const PairLaunch& L) {
  P.X = L.X;
  P.Y = L.Y;
  P.OutX = L.OutX;
  P.OutY = L.OutY;
  P.S = static_cast<const cplx<R>*>(L.S);
  P.ld = L.ld;
  P.ng = (long long)L.nx * L.ny * L.nz;
  P.scale = (R)L.scale;
  P.tiles = L.dtiles;
}

// Pass A (pass == 0) or C (pass == 2) of one batch, or (prepare_only) the
// kernels' shared-memory attributes, set once at plan creation on the plan's
// device, never during stream capture.
template <typename R, int NX, int NY, bool POIS>
void launch_plane_as(const PairLaunch& L, const Batch& b, int pass, cudaStream_t st) {
  constexpr bool F64 = sizeof(R) == 8, SPLIT = kSplitPlanes<R, NX, NY>;
  constexpr int IPB = SPLIT ? 1 : plane_items<R, NX, NY>();
  constexpr size_t smem = SPLIT ? kSplitSmem<R, NX, NY> : (size_t)IPB * NY * (NX + 1) * sizeof(cplx<R>);
  PlaneParams<R, NX, NY> P;
  if (!L.prepare_only) fill_plane<R, NX, NY>(P, L, b);
  const long long items = (long long)b.npairs * L.nz;
  const dim3 grid((unsigned)((items + IPB - 1) / IPB)), blk(kMaxLine<NX, NY> * (SPLIT ? 2 : IPB));
  auto run = [&](auto kern) {
    if (L.prepare_only) {
      cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
      cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
    } else {
      launch_pdl(!L.no_pdl && !(pass == 0 && L.lead), kern, grid, blk, smem, st, P);
    }
  };
  if constexpr (SPLIT) {
    if (pass == 2) run(pass_c_split_kernel<R, NX, NY, POIS>);
    else if (F64 && L.real_io) run(pass_a_split_kernel<R, NX, NY, F64, POIS>);
    else run(pass_a_split_kernel<R, NX, NY, false, POIS>);
  } else {
    if (pass == 2) run(pass_c_kernel<R, NX, NY, POIS>);
    else if (F64 && L.real_io) run(pass_a_kernel<R, NX, NY, F64, POIS>);
    else run(pass_a_kernel<R, NX, NY, false, POIS>);
  }
}
template <typename R, int NX, int NY>
bool launch_plane(const PairLaunch& L, const Batch& b, int pass, cudaStream_t st) {
  if (sizeof(R) != 8 && L.real_io) return false;
  if (L.prepare_only) {
    for (int q = 0; q <= 2; q += 2) {
      launch_plane_as<R, NX, NY, false>(L, b, q, st);
      launch_plane_as<R, NX, NY, true>(L, b, q, st);
    }
    return true;
  }
  if (L.V) launch_plane_as<R, NX, NY, true>(L, b, pass, st);
  else launch_plane_as<R, NX, NY, false>(L, b, pass, st);
  return true;
}

// Pass B of one batch (the compile-time geometry on cubic grids).
template <typename R, int NZ, bool CUBE>
void launch_pencil_as(const PencilParams<R, NZ>& P, const PairLaunch& L, long long pencils, cudaStream_t st) {
  if constexpr (kQuadPencil<R, NZ>) {
    const unsigned grid = (unsigned)((pencils + kQuadPencils - 1) / kQuadPencils);
    launch_pdl(!L.no_pdl, pass_b_quad_kernel<R, NZ, CUBE>, dim3(grid), dim3(128), 0, st, P, L.mode);
  } else if constexpr (kSplitPencil<NZ>) {
    const unsigned grid = (unsigned)((pencils + kBSplitPencils - 1) / kBSplitPencils);
    launch_pdl(!L.no_pdl, pass_b_split_kernel<R, NZ, CUBE>, dim3(grid), dim3(256), 0, st, P, L.mode);
  } else {
    const unsigned grid = (unsigned)((pencils + kPencilThreads - 1) / kPencilThreads);
    launch_pdl(!L.no_pdl, pass_b_kernel<R, NZ, CUBE>, dim3(grid), dim3(kPencilThreads), 0, st, P, L.mode);
  }
}
template <typename R, int NZ>
bool launch_pencil(const PairLaunch& L, const Batch& b, cudaStream_t st) {
  if (L.prepare_only) return true;
  PencilParams<R, NZ> P;
  fill_pencil<R, NZ>(P, L, b);
  const long long pencils = (long long)b.npairs * L.nx * L.ny;
  if (L.nx == NZ && L.ny == NZ) launch_pencil_as<R, NZ, true>(P, L, pencils, st);
  else launch_pencil_as<R, NZ, false>(P, L, pencils, st);
  return true;
}

// Pass D of one batch: NGC = N_g of a cubic grid compiled in, or 0 (any grid).
template <typename R, long long NGC>
bool launch_point(const PairLaunch& L, const Batch& b, cudaStream_t st) {
  if (L.prepare_only) return true;
  PointParams<R> P;
  fill_point<R>(P, L);
  if (NGC && P.ng != NGC) return false;
  const int pts = d_points<R>(b, L.real_io);
  const dim3 grid((unsigned)((P.ng + pts - 1) / pts), (unsigned)b.ntiles);
  if constexpr (sizeof(R) == 8) {
    if (L.real_io) {
      launch_pdl(!L.no_pdl, pass_d_kernel<R, true, NGC>, grid, dim3(256), 0, st, P);
      return true;
    }
  } else {
    if (L.real_io) return false;
  }
  launch_pdl(!L.no_pdl, pass_d_kernel<R, false, NGC>, grid, dim3(256), 0, st, P);
  return true;
}

// The persistent engine holds whole lines per thread; FP64 lines of 64 or more
// points do not fit, so those edges have no engine (plans fall back to the four
// kernels per batch).
template <typename R, int N> constexpr bool kEngineBuilt = !(sizeof(R) == 8 && N >= kSplitMinEdgeF64);

// Tasks per pass of a batch in the engine (A, B, C, D).
template <typename R, int N>
void engine_tasks(const Batch& b, int n[4]) {
  constexpr int IPB = engine_items<R, N>();
  n[0] = (int)(((long long)b.npairs * N + IPB - 1) / IPB);
  n[1] = (int)(((long long)b.npairs * N * N + kEngineThreads - 1) / kEngineThreads);
  n[2] = n[0];
  n[3] = (int)((((long long)N * N * N + kEngineThreads - 1) / kEngineThreads) * b.ntiles);
}

template <typename R, int N>
void engine_prepare(EngineInfo& info) {
  if constexpr (!kEngineBuilt<R, N>) {
    info = EngineInfo{};
    return;
  } else {
    constexpr int IPB = engine_items<R, N>();
    constexpr size_t smem = (size_t)IPB * N * (N + 1) * sizeof(cplx<R>);
    info.smem = smem;
    info.threads = kEngineThreads;
    int dev = 0, sms = 0, per = 0, occ = 1 << 30;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    auto one = [&](auto kern) {
      cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
      cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
      per = 0;
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kern, kEngineThreads, smem);
      if (per < occ) occ = per;
    };
    one(pair_engine_kernel<R, N, false>);
    if constexpr (sizeof(R) == 8) one(pair_engine_kernel<R, N, true>);
    info.blocks = occ > 0 ? occ * sms : 0;
  }
}

template <typename R, int N>
bool launch_engine(const PairLaunch& L, const EngineLaunch& EL, cudaStream_t st) {
  if constexpr (!kEngineBuilt<R, N>) {
    return false;
  } else {
    if (L.nx != N || L.ny != N || L.nz != N) return false;
    EngineParams<R, N> E;
    Batch none{};
    fill_plane<R, N, N>(E.pl, L, none);
    fill_pencil<R, N>(E.pe, L, none);
    fill_point<R>(E.pt, L);
    E.pl.tiles = EL.dtiles;
    E.pe.tiles = EL.dtiles;
    E.pt.tiles = EL.dtiles;
    E.batches = EL.batches;
    E.nbatches = EL.nbatches;
    E.npasses = L.mode == 1 ? 2 : 4;
    E.ntasks = EL.ntasks;
    E.head = EL.head;
    E.done = EL.done;
    E.status = EL.status;
    E.mode = L.mode;
    E.spin_limit = EL.spin_limit;
    E.wait_bias = EL.wait_bias;
    cudaLaunchConfig_t cfg{};
    long long blocks = EL.blocks;
    if (blocks > EL.ntasks) blocks = EL.ntasks;
    if (blocks < 1) return true;
    cfg.gridDim = dim3((unsigned)blocks);
    cfg.blockDim = dim3(kEngineThreads);
    cfg.dynamicSmemBytes = EL.smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeCooperative;   // all blocks co-resident (required by the waits)
    at[0].val.cooperative = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    if constexpr (sizeof(R) == 8) {
      if (L.real_io) {
        cudaLaunchKernelEx(&cfg, pair_engine_kernel<R, N, true>, E);
        return true;
      }
    }
    if (L.real_io) return false;
    cudaLaunchKernelEx(&cfg, pair_engine_kernel<R, N, false>, E);
    return true;
  }
}

}  // namespace ACE_RADIX_NS
}  // namespace ace
