// Tensor-core products of the ACE apply (Eq. ACE: C = dV Xi^* psi, Y = -Xi C) for
// complex FP32 vectors, on tcgen05 kind::f16 with FP16 operand pairs.
//
// FP32 accuracy from FP16 operands: a row or column of an operand is scaled by a power
// of two that puts its largest component in [2^14, 2^15), and a scaled value x is
// split x = hi + lo, hi = fp16(x), lo = fp16(x - hi) (round to nearest; the splitting
// of Markidis et al., "NVIDIA Tensor Core Programmability, Performance & Precision",
// 2018, with both parts scaled). hi and lo carry 22 to 23 bits of every value down to
// 2^-18 of the row's largest (lo is then a normal FP16 number) and below that an absolute
// error of 2^-40 of the largest. So what shares a scale matters: the gram product's
// rows and columns are vectors, scaled anew every 512 points; the outer product's rows
// are points (the largest value of any orbital there), so that V_ACE psi keeps its
// relative accuracy where every orbital is small, as in vacuum, and its columns are the
// bands' coefficients.
// Three products hi hi + hi lo + lo hi are kept; the dropped lo lo is below
// 2^-24. (The TF32 split of tc_gemm.cu truncates both parts and drops 2^-20.) A
// kind::f16 MMA does twice the work of a kind::tf32 one per cycle on half the
// shared-memory bytes, which is what bounds these products.
//
// As there, complex products are real ones on interleaved data: a tile of BB = TN/2
// complex columns is TN real MMA columns.
//   gram:  rows a, K' = 2 N_g; columns j < BB take B_b as stored (re, im), columns
//          BB + j take (im, -re).
//   outer: rows g, K' = 2 N; columns j < BB take (Re C, -Im C), BB + j (Im C, Re C).
//
// Pipeline (512 working threads, one CTA per SM, M = 128): K runs in chunks of 32 real terms.
// One thread keeps a ring of raw FP32 chunks filled by TMA, as deep as shared
// memory allows; every thread converts eight values of one row (A), or of one row of A and
// one of B, from the ring into an operand stage (K-major core matrices,
// conflict-free stores); one thread issues the chunk's MMAs and commits them to the
// stage's mbarrier. (Fetching with 16-byte cp.async by all threads took 157 us of the gram
// product below, 60 of them for issuing the copies; register prefetch held the TF32
// kernels at 33-41 % tensor activity.) The outer product's right operand is split once per
// call in the stage layout and arrives by one bulk copy per chunk. The accumulator
// restarts every kGroup chunks (24 MMAs: the tensor core's FP32
// accumulation truncates), alternating between two TMEM buffers; finished groups
// are added in FP32 registers while the next group's MMAs run. Every mbarrier wait
// is bounded, as in tc_gemm.cu.
//
// Measured, TF32 split -> this: 48^3, 128 orbitals, 192 bands: gram 169 -> 98 us, outer
// 188 -> 101 us, the sweep over the vectors for their maxima 44 us (6.5 TB/s), whole
// call 378 -> 281 us; 96^3, 1024 x 1536: 116 -> 68.7 ms (gram 37.5, outer 28.4, maxima 2.4).
// With the MMAs and the conversion switched off the 48^3 loops take 67 us (gram) and 95
// (outer, with a scale per value) (387 and 553 MB through L2, 5.8 TB/s): tile traffic
// bounds them, then the chain convert - fence - barrier - issue of a chunk. Relative error
// against FP64 at 48^3: 2.7e-6 -> 9.6e-7.
#include <cstdint>
#include <type_traits>
#include <cuda.h>
#include <cuda_fp16.h>

#include "ace_internal.h"
#include "tcgen05.cuh"

namespace ace {

namespace {

using tc::smem_u32;

constexpr int THREADS = 512;
constexpr int TM = 128;                 // rows per CTA (M of the MMA)
constexpr int KC = 32;                  // real K terms per chunk
constexpr int SBO = (KC * 2 / 16) * 128;   // bytes between 8-row groups of an operand tile
constexpr int kGroup = 4;               // chunks per accumulator group
constexpr unsigned kWaitLimit = 1u << 24;
constexpr int A_TILE = TM * KC * 2;     // one FP16 A tile (8 KB)

template <int TN> struct Tile {
  static_assert(TN == 64 || TN == 128 || TN == 192 || TN == 256, "MMA width");
  static constexpr int BB = TN / 2;                   // complex columns
  static constexpr int NH = TN / 8;                   // complex columns per thread (4 column groups of warps)
  static constexpr int B_TILE = TN * KC * 2;          // one FP16 B tile
  static constexpr int TMEM_COLS = TN == 64 ? 128 : TN == 128 ? 256 : 512;   // two accumulators, a power of two
  // instruction descriptor: D = F32, A = B = F16, both K-major, N = TN, M = 128
  static constexpr uint32_t IDESC = (1u << 4) | ((uint32_t)(TN >> 3) << 17) | ((uint32_t)(TM >> 4) << 24);
  // gram: stages of A_hi, A_lo, B_hi, B_lo and a raw ring of A and B rows
  static constexpr int G_STAGE = 2 * A_TILE + 2 * B_TILE;
  static constexpr int G_RAW = (TM + BB) * KC * 4;
  // The narrow tiles' chunks are short beside a block-wide barrier and the issue of their
  // MMAs: a warp of its own fetches and issues, and the working warps meet it on
  // mbarriers (16 x 24 vectors of 48^3, with one scale per vector: 38.0 us without, 35.6 us
  // with; 36.1 with the segments' scales). The wide ones need
  // the registers that a fifth warp per SM quadrant takes.
  static constexpr bool G_ISSUER = TN <= 128;
  static constexpr int G_THREADS = THREADS + (G_ISSUER ? 128 : 0);
  static constexpr int G_STAGES = TN == 64 ? 4 : TN == 256 ? 2 : 3;
  static constexpr int G_RING = TN == 64 ? 6 : TN == 128 ? 5 : TN == 192 ? 3 : 4;   // what 227 KB hold
  static constexpr int G_SMEM = G_STAGES * G_STAGE + G_RING * G_RAW + 1024 + 128;
  // outer: stages of A_hi, A_lo, a ring of right operands, a raw ring of A
  static constexpr int O_STAGE = 2 * A_TILE;
  static constexpr int O_B = 2 * B_TILE;
  static constexpr int O_RAW = TM * KC * 4;
  static constexpr int O_RING = TN == 64 ? 7 : TN == 128 ? 6 : 4;   // raw slots and right operands alike
  static constexpr int O_SMEM = 2 * O_STAGE + O_RING * (O_B + O_RAW) + 1024 + 128;
};

// byte offset of real K value k of row r in an operand tile
__device__ __forceinline__ int tile_off(int r, int k) {
  return (r >> 3) * SBO + (k >> 3) * 128 + (r & 7) * 16 + (k & 7) * 2;
}

// The power of two that takes a vector whose largest |component| has the bits `m`
// to [2^14, 2^15) (1 for zero and non-finite vectors), and its inverse.
__device__ __forceinline__ int scale_exp(unsigned m) {
  const int e = (int)(m >> 23);
  if (m == 0u || e == 255) return 0;
  return e < 15 ? 126 : 141 - e;          // tiny vectors: 2^126 keeps them far from overflow
}
__device__ __forceinline__ float exp2i(int e) { return __uint_as_float((unsigned)(e + 127) << 23); }   // |e| <= 126

// Further powers of two for a vector's values within one 512-point segment, from the
// biased exponents of the vector's and the segment's largest: in steps of 4, so that
// vectors without large variation stay in one unit, and at most 36, so that sums over
// all points in the units of two boosts stay below 2^123.
__device__ __forceinline__ int exp_scale(int e) { return e == 255 ? 0 : e < 15 ? 126 : 141 - e; }
__device__ __forceinline__ int boost(int ev, int es) {
  if (ev == 0 || ev == 255) return 0;
  return min((exp_scale(es) - exp_scale(ev)) & ~3, 36);
}

// one box of a 2D tensor map (x in floats, a multiple of 4; y a vector) to shared
// memory; coordinates past the tensor read zero and count as bytes on `bar`
__device__ __forceinline__ void load_box(void* dst, const CUtensorMap& map, int x, int y, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(
          smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(&map)), "r"(x), "r"(y), "r"(smem_u32(bar))
      : "memory");
}

// (re, im) -> (im, -re) of a pair of halves
__device__ __forceinline__ uint32_t swap_neg(uint32_t h) { return __byte_perm(h, h, 0x1032) ^ 0x80000000u; }

// two scaled values -> hi and lo halves
__device__ __forceinline__ void split2(float2 y, uint32_t& hi, uint32_t& lo) {
  const __half2 a = __float22half2_rn(y);
  const float2 b = __half22float2(a);
  const __half2 c = __float22half2_rn(__fadd2_rn(y, make_float2(-b.x, -b.y)));
  hi = *reinterpret_cast<const uint32_t*>(&a);
  lo = *reinterpret_cast<const uint32_t*>(&c);
}
// two complex values times s -> hi and lo halves
__device__ __forceinline__ void split4(const float4& u, float s, uint2& hi, uint2& lo) {
  split2(__fmul2_rn(make_float2(u.x, u.y), make_float2(s, s)), hi.x, lo.x);
  split2(__fmul2_rn(make_float2(u.z, u.w), make_float2(s, s)), hi.y, lo.y);
}

template <int TN>
__device__ __forceinline__ void mma_f16(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
      "l"(a), "l"(b), "r"(Tile<TN>::IDESC), "r"(accumulate)
      : "memory");
}

// the MMAs of one chunk: 2 K-steps x 3 products. Descriptors count 16-byte units, so
// the operands' are sums with constants: one thread issues, and the block's
// other warps wait for its warp.
template <int TN>
__device__ __forceinline__ void issue_chunk(uint32_t dtmem, uint32_t a, uint32_t b, bool first) {
  const uint64_t ah = tc::kmajor_desc(a, SBO), bh = tc::kmajor_desc(b, SBO);
  constexpr uint64_t LA = A_TILE / 16, LB = Tile<TN>::B_TILE / 16;
#pragma unroll
  for (uint64_t ks = 0; ks < KC / 16; ++ks) {
    const uint64_t o = ks * 16;   // two core matrices of 16 bytes along K
    mma_f16<TN>(dtmem, ah + o, bh + o, (first && ks == 0) ? 0u : 1u);
    mma_f16<TN>(dtmem, ah + o, bh + LB + o, 1u);
    mma_f16<TN>(dtmem, ah + LA + o, bh + o, 1u);
  }
}

// NH consecutive accumulator columns of this thread's lane, added into acc, at most
// 16 at a time (the sums already hold half of the registers)
template <int NH>
__device__ __forceinline__ void tmem_add(uint32_t taddr, float (&acc)[NH]) {
#pragma unroll
  for (int o = 0; o + 16 <= NH; o += 16) {
    uint32_t r[16];
    tc::tmem_ld16(taddr + (uint32_t)o, r);
    tc::tmem_wait_ld();
#pragma unroll
    for (int i = 0; i < 16; ++i) acc[o + i] += __uint_as_float(r[i]);
  }
  if constexpr (NH % 16 == 8) {
    uint32_t r[8];
    tc::tmem_ld8(taddr + (uint32_t)(NH - 8), r);
    tc::tmem_wait_ld();
#pragma unroll
    for (int i = 0; i < 8; ++i) acc[NH - 8 + i] += __uint_as_float(r[i]);
  }
}

// State of the chunk stream that both kernels run: operand stages, whose MMAs
// commit to bar[s]. Bit s of `phase` / `issued`: parity of, and a pending commit
// on, stage s; two bits per stage of `drain`: 1 + the TMEM buffer of a group that
// ends with that commit. (Every thread keeps its own copy.)
template <int TN> struct Stream {
  uint64_t* bar;
  uint32_t tmem, lane_col;
  unsigned phase = 0, issued = 0, drain = 0;
  float re[Tile<TN>::NH], im[Tile<TN>::NH];
  __device__ __forceinline__ void zero() {
#pragma unroll
    for (int i = 0; i < Tile<TN>::NH; ++i) re[i] = im[i] = 0.f;
  }
  // bounded wait for the MMAs of stage s, then the sums of a finished group, whose units
  // `units` gives the sums so far. VOTE: `units` exchanges values within the warp, so
  // that a lost wait has to take all its lanes along.
  template <bool VOTE, typename F> __device__ __forceinline__ bool settle(int s, F&& units) {
    const unsigned d = (drain >> (2 * s)) & 3u;
    bool done = tc::mbar_wait(&bar[s], (phase >> s) & 1u, kWaitLimit);
    if (VOTE && d) done = __all_sync(0xffffffffu, done);
    if (!done) return false;
    phase ^= 1u << s;
    issued &= ~(1u << s);
    if (d) {
      units();
      tc::fence_after_sync();
      const uint32_t t = tmem + lane_col + (uint32_t)(TN * (d - 1));
      tmem_add<Tile<TN>::NH>(t, re);
      tmem_add<Tile<TN>::NH>(t + Tile<TN>::BB, im);
      tc::fence_before_sync();
      drain &= ~(3u << (2 * s));
    }
    return true;
  }
};

template <int TN>
__device__ __forceinline__ uint32_t setup(uint64_t* bar, int nbar, uint32_t* slot, int nwarps = 0) {
  if (threadIdx.x == 0) {
    for (int i = 0; i < nbar; ++i) tc::mbar_init(&bar[i], 1);
    for (int i = 0; i < nwarps; ++i) tc::mbar_init(&bar[nbar + i], THREADS / 32);   // one arrival per working warp
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (threadIdx.x < 32) tc::tmem_alloc_warp(slot, Tile<TN>::TMEM_COLS);
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  return __shfl_sync(0xffffffffu, *slot, 0);   // the same register for the whole warp
}
template <int TN> __device__ __forceinline__ void teardown(uint32_t tmem) {
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  if (threadIdx.x < 32) tc::tmem_dealloc_warp(tmem, Tile<TN>::TMEM_COLS);
}

// Largest |component| (as float bits, which order like the values; NaN is skipped) of
// each vector, mx[0 .. na) for A and mx[na ..) for B, and of each point over the vectors
// of A, pt[g]; the biased exponent of each vector's largest in each segment, sx[segment *
// row + vector], with the vectors of B from `at_b` on. Grid: (ya parts of `per` vectors
// of A and then those of B, 512-point segments). A warp takes a segment of one vector at
// a time, eight 16-byte loads in flight a thread, and keeps the maxima of its points in
// registers; one sweep of the vectors, bound by memory.
constexpr int SEG = 512, kMaxPart = 64;
__global__ void __launch_bounds__(256)
maxima_kernel(const float2* __restrict__ A, int na, const float2* __restrict__ B, int nb, long long ld, long long ng,
              int per, int ya, unsigned* __restrict__ mx, unsigned* __restrict__ pt, unsigned char* __restrict__ sx,
              int row, int at_b) {
  __shared__ unsigned vm[kMaxPart];
  const bool first = (int)blockIdx.x < ya;               // a part of A
  const int count = first ? na : nb, v0 = ((int)blockIdx.x - (first ? 0 : ya)) * per;
  const int v1 = v0 + per < count ? v0 + per : count;
  const float2* X = first ? A : B;
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const long long n = ng / 2, i0 = (long long)blockIdx.y * (SEG / 2);   // float4 units: N_g is even on every grid
  int off[8];                                            // past the grid's end: its last points again
  float2 p[8];
#pragma unroll
  for (int u = 0; u < 8; ++u) {
    off[u] = i0 + lane + 32 * u < n ? lane + 32 * u : (int)(n - 1 - i0);
    p[u] = make_float2(0.f, 0.f);
  }
  for (int v = v0 + w; v < v1; v += 8) {
    const float4* x = reinterpret_cast<const float4*>(X + (long long)v * ld) + i0;
    float4 t[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) t[u] = x[off[u]];
    float m = 0.f;
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const float a = fmaxf(fabsf(t[u].x), fabsf(t[u].y)), b = fmaxf(fabsf(t[u].z), fabsf(t[u].w));
      p[u] = make_float2(fmaxf(p[u].x, a), fmaxf(p[u].y, b));
      m = fmaxf(m, fmaxf(a, b));
    }
    const unsigned r = __reduce_max_sync(0xffffffffu, __float_as_uint(m));
    if (lane == 0) vm[v - v0] = r;
  }
  __shared__ float2 red[8][SEG / 2];
  if (first) {
#pragma unroll
    for (int u = 0; u < 8; ++u) red[w][lane + 32 * u] = p[u];
  }
  __syncthreads();
  if ((int)threadIdx.x < v1 - v0) {
    const unsigned r = vm[threadIdx.x];
    const int v = v0 + threadIdx.x;
    atomicMax(mx + (first ? v : na + v), r);
    sx[(long long)blockIdx.y * row + (first ? v : at_b + v)] = (unsigned char)(r >> 23);
  }
  if (!first) return;
  const int i = threadIdx.x;
  float2 q = red[0][i];
#pragma unroll
  for (int k = 1; k < 8; ++k) q = make_float2(fmaxf(q.x, red[k][i].x), fmaxf(q.y, red[k][i].y));
  if (i0 + i < n) {
    atomicMax(pt + 2 * (i0 + i), __float_as_uint(q.x));
    atomicMax(pt + 2 * (i0 + i) + 1, __float_as_uint(q.y));
  }
}

// ---------------------------------------------------------------- gram
// part[s][a][b] = sum over the points of split s of conj(A_a) B_b, of the scaled
// vectors (FP32). Grid: (ceil(na / 128), ceil(nb / BB), splits); splits start at multiples of
// the 16 points of a chunk. A chunk's A and B boxes (128 bytes per row, in the
// 128-byte swizzle: 16-byte granule g of row r lies at g ^ (r & 7)) arrive by two TMA
// loads. Thread t owns row 8 (t / 32) + t % 8 and granules q and q + 4, q = (t / 8) % 4:
// its loads are conflict-free and its stores fill 128 contiguous bytes per 16 lanes.
// Scales are those of the vectors times each segment's boost, so that overlaps far below
// the vectors' largest values keep their accuracy: accumulator groups end where
// segments do, and when a segment's boosts differ from those of the sums so far, the
// sums are taken to its units first (a multiplication by a power of two). The split's
// sums are left in the units of the vectors. A segment's exponents arrive with its
// first chunk. Costs 5 of 98 us at 48^3, 128 x 192, 0.8 of 36 at 16 x 24.
template <int TN>
__global__ void __launch_bounds__(Tile<TN>::G_THREADS, 1)
gram16_kernel(const __grid_constant__ CUtensorMap A, int na, const __grid_constant__ CUtensorMap B, int nb, long long ng,
              const unsigned* __restrict__ mx, const unsigned char* __restrict__ sx, int row, int at_b,
              float2* __restrict__ part, long long chunk, int* status) {
  using T = Tile<TN>;
  constexpr int BB = T::BB, NH = T::NH, R = T::G_RING, ST = T::G_STAGES;
  extern __shared__ unsigned char smem_raw[];
  unsigned char* base = reinterpret_cast<unsigned char*>(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  unsigned char* ring = base + ST * T::G_STAGE;
  // barriers: ST for the MMAs of a stage, R for a landed chunk, ST for a stored stage
  uint64_t* bar = reinterpret_cast<uint64_t*>(ring + R * T::G_RAW);
  __shared__ volatile int s_fail;
  // biased exponents of the tile's 128 rows and BB columns: of the vectors' largest
  // values, and of their largest in the even and the odd segments
  __shared__ __align__(16) unsigned char s_ev[TM + BB], s_es[2][TM + BB];
  const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31;
  const int a0 = blockIdx.x * TM, b0 = blockIdx.y * BB;
  if (tid == 0) s_fail = 0;
  Stream<TN> S;
  S.bar = bar;
  constexpr bool IW = T::G_ISSUER;
  S.tmem = setup<TN>(bar, ST + R, reinterpret_cast<uint32_t*>(bar + 2 * ST + R), IW ? ST : 0);
  S.lane_col = ((uint32_t)(32 * (w & 3)) << 16) + (uint32_t)(NH * (w >> 2));

  const long long g_begin = (long long)blockIdx.z * chunk;
  const long long g_end = g_begin + chunk < ng ? g_begin + chunk : ng;
  const int nchunks = g_end > g_begin ? (int)((g_end - g_begin + KC / 2 - 1) / (KC / 2)) : 0;
  const int r = (w << 3) | (tid & 7), q = (tid >> 3) & 3;
  const bool arow = a0 + r < na, brow = r < BB && b0 + r < nb;
  const bool bthr = r < BB;                              // uniform in a warp
  constexpr int SC = 2 * SEG / KC, SG = SC / kGroup;     // chunks and groups per segment
  const unsigned c0 = (unsigned)(g_begin / (KC / 2));    // segments and groups count from the grid's first point
  auto group_start = [&](int c) { return c == 0 || (c0 + c) % kGroup == 0; };
  auto buffer = [&](int c) { return (int)((c0 + c) / kGroup & 1); };
  auto boost_of = [&](int i, int segment) { return boost(s_ev[i], s_es[segment & 1][i]); };
  auto fetch = [&](int c) {
    if (c < nchunks) {
      const int slot = c % R, x = (int)(2 * g_begin) + KC * c;
      uint64_t* fb = bar + ST + slot;
      unsigned char* d = ring + slot * T::G_RAW;
      const bool start = c == 0 || (c0 + c) % SC == 0;   // a segment: its exponents come with its first chunk
      tc::mbar_arrive_expect_tx(fb, (unsigned)(T::G_RAW + (start ? TM + BB : 0)));
      load_box(d, A, x, a0, fb);
      load_box(d + TM * KC * 4, B, x, b0, fb);
      if (start) {
        const int e = (int)((c0 + c) / SC);
        const unsigned char* src = sx + (long long)e * row;
        tc::bulk_g2s(s_es[e & 1], src + a0, TM, fb);
        tc::bulk_g2s(s_es[e & 1] + TM, src + at_b + b0, BB, fb);
      }
    }
  };
  if (IW && w >= THREADS / 32) {                         // ---- the issuing warp (and three idle ones)
    if (TN == 128) asm volatile("setmaxnreg.dec.sync.aligned.u32 24;");
    if (tid == THREADS) {
      int c = 0;
      for (int i = 0; i < R; ++i) fetch(i);
      for (; c < nchunks; ++c) {
        const int s = c % ST;
        // stored by all warps: also read from the ring, and the sums of the group that
        // last used this chunk's accumulator are drained (their stage came before)
        if (!tc::mbar_wait(bar + ST + R + s, (unsigned)(c / ST) & 1u, kWaitLimit)) break;
        tc::fence_after_sync();
        const uint32_t sa0 = smem_u32(base + s * T::G_STAGE);
        issue_chunk<TN>(S.tmem + (uint32_t)(TN * buffer(c)), sa0, sa0 + 2 * A_TILE, group_start(c));
        tc::mma_commit(&bar[s]);
        fetch(c + R);
      }
      if (c < nchunks) {                                 // a lost wait: the copies and MMAs in flight (bounded)
        s_fail = 1;
        for (int i = c; i < c + R && i < nchunks; ++i) tc::mbar_wait(bar + ST + i % R, (unsigned)(i / R) & 1u, 1u << 16);
        for (int i = c < ST ? 0 : c - ST; i < c; ++i) tc::mbar_wait(&bar[i % ST], (unsigned)(i / ST) & 1u, 1u << 16);
      }
    }
  } else {                                               // ---- the working warps
    if (TN == 128) asm volatile("setmaxnreg.inc.sync.aligned.u32 112;");   // 512 x 112 + 128 x 24 of 640 x 96 registers
    if (!IW && tid == 32)
      for (int c = 0; c < R - 1; ++c) fetch(c);
    if (tid < TM + BB) {
      const int v = tid < TM ? a0 + tid : na + b0 + tid - TM;
      s_ev[tid] = v < (tid < TM ? na : na + nb) ? (unsigned char)(mx[v] >> 23) : 0;
    }
    asm volatile("bar.sync 1, %0;" ::"n"(THREADS) : "memory");
    S.zero();
    // the sums so far into the units of `to` (< 0: of the vectors) from those of segment `from`
    const int lrow = 32 * (w & 3) + lane, lcol = NH * (w >> 2) + lane;   // this lane's row, and (lanes below NH) a column
    auto rescale = [&](int from, int to) {
      int db = -boost_of(lrow, from), dc = lane < NH ? -boost_of(TM + lcol, from) : 0;
      if (to >= 0) {
        db += boost_of(lrow, to);
        if (lane < NH) dc += boost_of(TM + lcol, to);
      }
      if (__any_sync(0xffffffffu, (db | dc) != 0)) {
#pragma unroll
        for (int j = 0; j < NH; ++j) {
          const float f = exp2i(db + __shfl_sync(0xffffffffu, dc, j));
          S.re[j] *= f;
          S.im[j] *= f;
        }
      }
    };
    unsigned group = c0 / kGroup;                          // the next group to add
    auto units = [&]() {
      if (group % SG == 0 && group > c0 / kGroup) rescale((int)(group / SG) - 1, (int)(group / SG));
      ++group;
    };
    int fresh = 0;                                         // chunks left in this segment
    float sa = 0.f, sb = 0.f;
    const int o = tile_off(r, 4 * q);
    constexpr int IM = (BB >> 3) * SBO;                    // rows BB ..: (im, -re)
    const int g0 = r * 128 + ((q ^ (r & 7)) << 4), g1 = g0 ^ 64;   // the granules in a raw tile
    bool ok = true;
    unsigned lphase = 0;                                   // parities of the landing barriers
    for (int c = 0; c < nchunks; ++c) {
      const int s = c % ST, slot = c % R;
      if (!IW && tid == 32) fetch(c + R - 1);               // into the slot that chunk c - 1 left
      if (!tc::mbar_wait(bar + ST + slot, (lphase >> slot) & 1u, kWaitLimit)) s_fail = 1;
      else lphase ^= 1u << slot;
      if (fresh-- == 0) {
        const int e = (int)((c0 + c) / SC);
        fresh = SC - 1 - (int)((c0 + c) % SC);
        if (arow) sa = exp2i(exp_scale(s_ev[r]) + boost_of(r, e));
        if (brow) sb = exp2i(exp_scale(s_ev[TM + r]) + boost_of(TM + r, e));
      }
      const unsigned char* raw = ring + slot * T::G_RAW;
      unsigned char* st = base + s * T::G_STAGE + o;
      uint2 ah[2], al[2], bh[2], bl[2];
      split4(*reinterpret_cast<const float4*>(raw + g0), sa, ah[0], al[0]);
      split4(*reinterpret_cast<const float4*>(raw + g1), sa, ah[1], al[1]);
      if (bthr) {
        split4(*reinterpret_cast<const float4*>(raw + TM * KC * 4 + g0), sb, bh[0], bl[0]);
        split4(*reinterpret_cast<const float4*>(raw + TM * KC * 4 + g1), sb, bh[1], bl[1]);
      }
      if (((S.issued >> s) & 1u) && !S.template settle<true>(s, units)) s_fail = 1;   // the MMAs of chunk c - ST read this stage
#pragma unroll
      for (int i = 0; i < 2; ++i) {                        // granule i: K values 4 q + 16 i ..
        *reinterpret_cast<uint2*>(st + i * 256) = ah[i];
        *reinterpret_cast<uint2*>(st + A_TILE + i * 256) = al[i];
      }
      if (bthr) {
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          unsigned char* b = st + 2 * A_TILE + i * 256;
          *reinterpret_cast<uint2*>(b) = bh[i];
          *reinterpret_cast<uint2*>(b + T::B_TILE) = bl[i];
          *reinterpret_cast<uint2*>(b + IM) = make_uint2(swap_neg(bh[i].x), swap_neg(bh[i].y));
          *reinterpret_cast<uint2*>(b + T::B_TILE + IM) = make_uint2(swap_neg(bl[i].x), swap_neg(bl[i].y));
        }
      }
      tc::fence_async_smem();
      const int buf = buffer(c);
      if constexpr (IW) {
        __syncwarp();
        if (lane == 0)
          asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar + ST + R + s)) : "memory");
        if (__any_sync(0xffffffffu, s_fail)) {           // the warp leaves as one
          ok = false;
          break;
        }
      } else {
        __syncthreads();
        if (s_fail) {
          ok = false;
          break;
        }
        if (tid == 0) {
          const uint32_t sa0 = smem_u32(base + s * T::G_STAGE);
          tc::fence_after_sync();
          issue_chunk<TN>(S.tmem + (uint32_t)(TN * buf), sa0, sa0 + 2 * A_TILE, group_start(c));
          tc::mma_commit(&bar[s]);
        }
      }
      S.issued |= 1u << s;
      if ((c0 + c) % kGroup == kGroup - 1 || c == nchunks - 1) S.drain |= (1u + (unsigned)buf) << (2 * s);
    }
    for (int i = 0; i < ST; ++i) {                         // the last commits, in chunk order
      const int s = (nchunks + i) % ST;
      if (((S.issued >> s) & 1u) && !S.template settle<true>(s, units)) s_fail = 1;
    }
    if (!IW && !ok)                                        // copies in flight (bounded)
      for (int i = 0; i < R; ++i) tc::mbar_wait(bar + ST + i, (lphase >> i) & 1u, 1u << 16);
    if (nchunks > 0) rescale((int)((c0 + nchunks - 1) / SC), -1);
    const int a = a0 + lrow, bq = b0 + NH * (w >> 2);
    if (ok && a < na) {
      float2* out = part + ((long long)blockIdx.z * na + a) * nb + bq;
#pragma unroll
      for (int j = 0; j < NH; ++j)
        if (bq + j < nb) out[j] = make_float2(S.re[j], S.im[j]);
    }
    if (!ok) s_fail = 1;
  }
  __syncthreads();
  if (s_fail && tid == 0) {
    status[0] = -6;   // ACE_ERR_TIMEOUT
    status[1] = -4;
  }
  teardown<TN>(S.tmem);
}

// (double)x in integer arithmetic (subnormal x gives zero): the hardware conversion
// set the time of the reduction below (1000 x 1500 coefficients of 12^3, 19 splits: 511 us
// with it, 289 us without, 79 us with the parts below fitted to the chip).
__device__ __forceinline__ double widen(float x) {
  const unsigned u = __float_as_uint(x), e = u & 0x7f800000u;
  unsigned hi = (u & 0x80000000u) | (((u & 0x7fffffffu) >> 3) + 0x38000000u);
  if (e == 0x7f800000u) hi |= 0x7ff00000u;
  return e ? __hiloint2double((int)hi, (int)(u << 29)) : 0.0;
}

// C[a][b] = dv sum_s part[s][a][b], of the scaled vectors (FP64 sums in a fixed order,
// rounded once: part y of `ways` takes the splits y, y + ways, ..., the parts meet in
// shared memory). FP64 additions bound it, so `ways` is no more than fills the chip.
// The scales enter in c_split_kernel.
__global__ void __launch_bounds__(256)
gram16_reduce_kernel(const float2* __restrict__ part, int splits, long long total, int ways, double dv,
                     float2* __restrict__ C) {
  __shared__ double2 red[256];
  const int tid = threadIdx.x, per = 256 / ways, y = tid / per;
  const long long idx = (long long)blockIdx.x * per + tid % per;
  double2 acc = make_double2(0.0, 0.0);
  if (idx < total) {
    const float2* p = part + y * total + idx;
    for (int s = y; s < splits; s += 5 * ways) {         // five loads in flight
      float2 v[5];
#pragma unroll
      for (int u = 0; u < 5; ++u)
        v[u] = s + u * ways < splits ? p[(long long)(s - y + u * ways) * total] : make_float2(0.f, 0.f);
#pragma unroll
      for (int u = 0; u < 5; ++u) {
        if (s + u * ways < splits) {
          acc.x += widen(v[u].x);
          acc.y += widen(v[u].y);
        }
      }
    }
  }
  if (ways > 1) {
    red[tid] = acc;
    __syncthreads();
    if (y != 0) return;
    for (int k = 1; k < ways; ++k) {
      acc.x += red[k * per + tid].x;
      acc.y += red[k * per + tid].y;
    }
  }
  if (idx < total) C[idx] = make_float2((float)(dv * acc.x), (float)(dv * acc.y));
}

// The outer product's right operand. With Xi_k = 2^-e_k X_k and psi_b = 2^-e_b P_b (X, P
// the scaled vectors, C their products), Y_b = -sum_k Xi_k (2^-e_k C_kb) 2^-e_b: column b of
// 2^-e_k C_kb, scaled by its own power of two 2^f to [2^14, 2^15), is split and written in the
// stage layout of (column tile bt, chunk c): [bt][c] holds B_hi, B_lo tiles of TN rows
// x 32 K. Eight columns per block (padding columns and rows are written as zeros).
// colexp[b] = -(f + e_b): the exponent that takes column b's products back.
template <int TN>
__global__ void __launch_bounds__(256)
c_split_kernel(const float2* __restrict__ C, int nk, int nb, int nch, const unsigned* __restrict__ mx,
               unsigned char* __restrict__ Bs, int* __restrict__ colexp) {
  using T = Tile<TN>;
  __shared__ int red[32][8];
  const int j8 = threadIdx.x & 7, kl = threadIdx.x >> 3;
  const int col = blockIdx.x * 8 + j8, bt = col / T::BB, j = col - bt * T::BB;
  // the largest biased exponent of 2^-e_k max(|re|, |im|)
  constexpr int kNone = -100000;
  int m = kNone;
  if (col < nb)
    for (int k = kl; k < nk; k += 32) {
      const float2 c = C[(long long)k * nb + col];
      const int e = (int)((max(__float_as_uint(c.x) & 0x7fffffffu, __float_as_uint(c.y) & 0x7fffffffu)) >> 23);
      if (e != 0) m = max(m, e - scale_exp(mx[k]));
    }
  red[kl][j8] = m;
  __syncthreads();
  for (int w = 16; w > 0; w >>= 1) {
    if (kl < w) red[kl][j8] = max(red[kl][j8], red[kl + w][j8]);
    __syncthreads();
  }
  const int f = red[0][j8] == kNone ? 0 : 141 - red[0][j8];
  if (kl == 0 && col < nb) colexp[col] = -(f + scale_exp(mx[nk + col]));
  for (int k = kl; k < nch * 16; k += 32) {
    float2 x = make_float2(0.f, 0.f);
    if (col < nb && k < nk) {
      const float2 c = C[(long long)k * nb + col];
      const int g = f - scale_exp(mx[k]);
      x = make_float2(ldexpf(c.x, g), ldexpf(c.y, g));
    }
    const __half2 hi = __float22half2_rn(x);
    const float2 b = __half22float2(hi);
    const __half2 lo = __float22half2_rn(make_float2(x.x - b.x, x.y - b.y));
    unsigned char* t = Bs + (size_t)(bt * nch + k / 16) * T::O_B;
    const int o = tile_off(j, 2 * (k % 16));
    constexpr int IM = (T::BB >> 3) * SBO;
    const __half2 v[2] = {hi, lo};
#pragma unroll
    for (int p = 0; p < 2; ++p) {                        // rows j: (re, -im), rows BB + j: (im, re)
      *reinterpret_cast<__half2*>(t + p * T::B_TILE + o) = __halves2half2(__low2half(v[p]), __hneg(__high2half(v[p])));
      *reinterpret_cast<__half2*>(t + p * T::B_TILE + o + IM) = __lowhigh2highlow(v[p]);
    }
  }
}

// ---------------------------------------------------------------- outer
// Out_b(g) = alpha sum_k A_k(g) C_kb. One CTA per SM runs its (column tile, 128-point)
// tiles, tile blockIdx.x + i gridDim.x in turn, as one stream of chunks, so that a
// tile's first loads and MMAs run under the previous tile's last ones and its
// stores. A chunk's 16 orbital rows (1 KB each, one TMA box) and its right operand (one
// bulk copy) arrive on one mbarrier, issued by one thread RING - 2 chunks ahead: its slots are
// those of chunk n - 2, whose MMAs have just ended. Thread t owns point t % 128 and
// orbitals 4 (t / 128) .. + 3 of each chunk. Row g is scaled by the power of two of the
// point's largest value, pt[g], which the stores take back with the column's.
template <int TN>
__global__ void __launch_bounds__(THREADS, 1)
outer16_kernel(const __grid_constant__ CUtensorMap A, int nb, long long ld, long long ng, float alpha,
               const unsigned* __restrict__ pt, const unsigned char* __restrict__ Bs, const int* __restrict__ colexp,
               int nch, float2* __restrict__ Out, int* status) {
  using T = Tile<TN>;
  constexpr int BB = T::BB, NH = T::NH, R = T::O_RING;
  extern __shared__ unsigned char smem_raw[];
  unsigned char* base = reinterpret_cast<unsigned char*>(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  unsigned char* bring = base + 2 * T::O_STAGE;
  unsigned char* ring = bring + R * T::O_B;
  uint64_t* bar = reinterpret_cast<uint64_t*>(ring + R * T::O_RAW);   // [0, 2): MMAs of a stage; then R: a chunk landed
  __shared__ int s_fail;
  const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31;
  if (tid == 0) s_fail = 0;
  Stream<TN> S;
  S.bar = bar;
  S.tmem = setup<TN>(bar, 2 + R, reinterpret_cast<uint32_t*>(bar + 2 + R));
  S.lane_col = ((uint32_t)(32 * (w & 3)) << 16) + (uint32_t)(NH * (w >> 2));
  S.zero();

  const int nbt = (nb + BB - 1) / BB;
  const int ntiles = nbt * (int)((ng + TM - 1) / TM);
  const int mine = blockIdx.x < (unsigned)ntiles ? (ntiles - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;
  const int total = mine * nch;                          // chunks of this CTA (< 2^31 on every supported grid)
  const int r = tid & 127, q = tid >> 7;
  // one thread: the copies of the next chunk (cursor fn: tile ft, chunk fc)
  int ft = blockIdx.x, fc = 0, fn = 0;
  auto fetch = [&]() {
    if (fn < total) {
      const int slot = fn % R, gt = ft / nbt, ct = ft - gt * nbt;
      uint64_t* fb = bar + 2 + slot;
      tc::mbar_arrive_expect_tx(fb, (unsigned)(T::O_B + T::O_RAW));
      load_box(ring + slot * T::O_RAW, A, 2 * TM * gt, fc * (KC / 2), fb);
      tc::bulk_g2s(bring + slot * T::O_B, Bs + ((size_t)ct * nch + fc) * T::O_B, T::O_B, fb);
      ++fn;
      if (++fc == nch) {
        fc = 0;
        ft += gridDim.x;
      }
    }
  };
  auto store_tile = [&](int tile) {                      // Out of a finished tile, from the sums; then zero them
    const int gt = tile / nbt;
    const long long g = (long long)gt * TM + 32 * (w & 3) + lane;
    const int bq = (tile - gt * nbt) * BB + NH * (w >> 2);
    if (g < ng) {
      float2* p = Out + (long long)bq * ld + g;
      const int* ce = colexp + bq;
      const int er = 127 - scale_exp(__ldg(pt + g));
#pragma unroll
      for (int j = 0; j < NH; ++j) {
        if (bq + j < nb) {
          // the exponent in two factors: it can leave FP32's range where the value does not
          const int e = er + __ldg(ce + j), e1 = max(1, min(254, e)), e2 = max(1, min(254, e - e1 + 127));
          const float f = alpha * __uint_as_float((unsigned)e1 << 23), h = __uint_as_float((unsigned)e2 << 23);
          *p = make_float2(h * (f * S.re[j]), h * (f * S.im[j]));
        }
        p += ld;
      }
    }
    S.zero();
  };

  if (tid == 32)
    for (int i = 0; i < R - 2; ++i) fetch();
  bool ok = true;
  int tile = blockIdx.x, c = 0, gi = 0;                  // current tile and chunk, group counter
  int due0 = -1, due1 = -1;                              // tile that ends with the pending commit of stage 0, 1
  unsigned lphase = 0;                                   // parities of the landing barriers
  auto finish = [&](int s) {                             // the pending commit of stage s, and the stores that it ends
    if (!S.template settle<false>(s, [] {})) {
      s_fail = 1;
      return;
    }
    const int t = s ? due1 : due0;
    if (t >= 0) {
      store_tile(t);
      if (s) due1 = -1;
      else due0 = -1;
    }
  };
  const int o = tile_off(r, 8 * q);
  auto point_max = [&](int t) {                          // of this thread's point in tile t
    const long long g = (long long)(t / nbt) * TM + r;
    return t < ntiles && g < ng ? __ldg(pt + g) : 0u;
  };
  unsigned pnext = point_max(tile);
  float sc = 0.f;
  for (int n = 0; n < total; ++n) {
    const int s = n & 1, slot = n % R;
    if (c == 0) {
      sc = exp2i(scale_exp(pnext));
      pnext = point_max(tile + (int)gridDim.x);
    }
    if ((S.issued >> s) & 1u) finish(s);                 // the MMAs of chunk n - 2
    if (tid == 32) fetch();                              // into the slots that chunk n - 2 left
    if (!tc::mbar_wait(bar + 2 + slot, (lphase >> slot) & 1u, kWaitLimit)) s_fail = 1;
    else lphase ^= 1u << slot;
    const float2* x = reinterpret_cast<const float2*>(ring + slot * T::O_RAW) + 4 * q * TM + r;
    uint32_t ah[4], al[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) split2(__fmul2_rn(x[i * TM], make_float2(sc, sc)), ah[i], al[i]);
    unsigned char* st = base + s * T::O_STAGE + o;
    *reinterpret_cast<uint4*>(st) = make_uint4(ah[0], ah[1], ah[2], ah[3]);
    *reinterpret_cast<uint4*>(st + A_TILE) = make_uint4(al[0], al[1], al[2], al[3]);
    tc::fence_async_smem();
    __syncthreads();
    if (s_fail) {
      ok = false;
      break;
    }
    const bool tile_last = c == nch - 1;
    const int buf = gi & 1;
    if (tid == 0) {
      tc::fence_after_sync();
      issue_chunk<TN>(S.tmem + (uint32_t)(TN * buf), smem_u32(base + s * T::O_STAGE), smem_u32(bring + slot * T::O_B),
                      c % kGroup == 0);
      tc::mma_commit(&bar[s]);
    }
    S.issued |= 1u << s;
    if (c % kGroup == kGroup - 1 || tile_last) {
      S.drain |= (1u + (unsigned)buf) << (2 * s);
      ++gi;
    }
    if (tile_last) {
      if (s) due1 = tile;
      else due0 = tile;
      tile += gridDim.x;
      c = 0;
    } else {
      ++c;
    }
  }
  if (ok) {                                              // the last two commits, in chunk order
    for (int i = 0; i < 2; ++i) {
      const int s = (total + i) & 1;
      if ((S.issued >> s) & 1u) finish(s);
    }
  } else {
    for (int s = 0; s < 2; ++s)
      if ((S.issued >> s) & 1u) S.template settle<false>(s, [] {});
    for (int i = 0; i < R; ++i)                          // copies in flight (bounded)
      tc::mbar_wait(bar + 2 + i, (lphase >> i) & 1u, 1u << 16);
  }
  __syncthreads();
  ok = ok && !s_fail;
  if (!ok && tid == 0) {
    status[0] = -6;   // ACE_ERR_TIMEOUT
    status[1] = -5;
  }
  teardown<TN>(S.tmem);
}

// MMA width for nb columns: the least work over the tiles, ties to the wider. A
// tile of TN columns converts its 128 A rows beside TN / 2 B rows and reads both, so
// it counts TN + 128 (48^3, 64 orbitals on 200 vectors: 7 tiles of 64 columns, the
// fewest MMA columns, 502 us; two of 256 254 us).
int width(int nb) {
  int best = 256;
  long long cost = -1;
  for (const int tn : {256, 192, 128, 64}) {
    const long long c = (long long)((nb + tn / 2 - 1) / (tn / 2)) * (tn + TM);
    if (cost < 0 || c < cost) {
      cost = c;
      best = tn;
    }
  }
  return best;
}

size_t align256(size_t x) { return (x + 255) & ~size_t(255); }

template <typename F> void by_width(int tn, F&& f) {
  if (tn == 256) f(std::integral_constant<int, 256>());
  else if (tn == 192) f(std::integral_constant<int, 192>());
  else if (tn == 128) f(std::integral_constant<int, 128>());
  else f(std::integral_constant<int, 64>());
}

// Split-K count of the gram product: fewest waves per split, within 2 % of full waves
// if that can be had (the fewest such splits: each adds partial sums), at most `cap`.
int splits_for(long long ng, int na, int nb, long long cap) {
  constexpr long long kSMs = 152, kMaxSplits = 1024;
  const int bb = width(nb) / 2;
  const long long tiles = (long long)((na + TM - 1) / TM) * ((nb + bb - 1) / bb);
  long long max_s = (ng + KC / 2 - 1) / (KC / 2);
  if (max_s > kMaxSplits) max_s = kMaxSplits;
  if (max_s > cap) max_s = cap;
  long long best = 1;
  double best_cost = (double)((tiles + kSMs - 1) / kSMs);
  for (long long waves = 1; best_cost > 1.02 * tiles / kSMs; ++waves) {   // the most splits of each wave count
    long long s = waves * kSMs / tiles;
    if (s < 1) continue;
    if (s > max_s) s = max_s;
    const double cost = (double)((tiles * s + kSMs - 1) / kSMs) / (double)s;
    if (cost < best_cost * 0.98) {
      best_cost = cost;
      best = s;
    }
    if (s == max_s) break;
  }
  return (int)best;
}

// Scratch layout: vector, point and segment maxima, column exponents, C, and the split
// sums, which the right operand overwrites once they are reduced. The splits are those that fit `budget`
// bytes: the plan's workspace holds what the TF32 products take, or `least` (one split)
// if that is more, and the maxima of the points and segments (`tables`) beside it.
struct Scratch {
  unsigned* mx;      // vector maxima
  unsigned* pt;      // point maxima
  unsigned char* sx; // segment exponents: rows of `row` bytes, Psi's from at_b on
  int row, at_b;
  int* colexp;
  unsigned char* Bs;
  float2* C;
  float2* part;
  int splits;
  size_t least, tables;
};
Scratch scratch(char* base, long long ng, int n, int nb, size_t budget) {
  Scratch s{};
  size_t off = 0;
  auto take = [&](size_t bytes) { char* r = base ? base + off : nullptr; off += align256(bytes); return r; };
  const int bb = width(nb) / 2;
  const size_t nbt = (size_t)(nb + bb - 1) / bb, nch = (size_t)(n + 15) / 16;
  s.mx = (unsigned*)take((size_t)(n + nb) * sizeof(unsigned));
  s.pt = (unsigned*)take((size_t)ng * sizeof(unsigned));   // behind mx: one memset clears both
  s.at_b = (n + TM - 1) / TM * TM;                       // rows of whole tiles: a tile's bytes come by bulk copies
  s.row = s.at_b + (int)(nbt * bb);
  const size_t bytes = (size_t)((ng + SEG - 1) / SEG) * s.row;
  s.sx = (unsigned char*)take(bytes);
  s.tables = align256((size_t)ng * sizeof(unsigned)) + align256(bytes);
  s.colexp = (int*)take((size_t)nb * sizeof(int));
  s.C = (float2*)take((size_t)n * nb * sizeof(float2));
  s.part = (float2*)take(0);
  s.Bs = (unsigned char*)s.part;
  const size_t one = (size_t)n * nb * sizeof(float2), bs = nbt * nch * (size_t)(2 * bb) * KC * 2 * 2;
  s.least = off - s.tables + align256(one > bs ? one : bs);
  if (s.least + s.tables <= budget) s.splits = splits_for(ng, n, nb, (long long)((budget - off) / one));
  return s;
}

using EncodeFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                              const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                              CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
EncodeFn encoder() {
  static const EncodeFn f = [] {
    void* e = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &e, 12000, cudaEnableDefault, &q) != cudaSuccess) {
      cudaGetLastError();   // no error of the plan's: the TF32 products serve
      e = nullptr;
    }
    return reinterpret_cast<EncodeFn>(e);
  }();
  return f;
}

// n vectors of ng complex values as a [n][2 ng] float tensor, in boxes of `rows` x `points`
bool vector_map(CUtensorMap* m, const float2* x, int n, long long ld, long long ng, int points, int rows, bool swizzle) {
  const cuuint64_t dim[2] = {(cuuint64_t)(2 * ng), (cuuint64_t)n}, stride[1] = {(cuuint64_t)(ld * (long long)sizeof(float2))};
  const cuuint32_t box[2] = {(cuuint32_t)(2 * points), (cuuint32_t)rows}, one[2] = {1, 1};
  return encoder()(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, const_cast<float2*>(x), dim, stride, box, one,
                   CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_NONE,
                   CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace

bool apply_tc_prepare() {
  if (!encoder()) return false;
  for (const int tn : {64, 128, 192, 256})
    by_width(tn, [](auto t) {
      constexpr int TN = decltype(t)::value;
      cudaFuncSetAttribute(gram16_kernel<TN>, cudaFuncAttributeMaxDynamicSharedMemorySize, Tile<TN>::G_SMEM);
      cudaFuncSetAttribute(outer16_kernel<TN>, cudaFuncAttributeMaxDynamicSharedMemorySize, Tile<TN>::O_SMEM);
    });
  return cudaGetLastError() == cudaSuccess;
}

// Six launches against four: the TF32 products of tc_gemm.cu are the faster on the
// smallest calls (graph replay, TF32 -> this: 24^3, 10 + 10 vectors 22.6 -> 23.3 us; 30 + 30
// 24.8 -> 24.0; 60 + 60 32.3 -> 30.7; 36^3, 4 + 4 42.7 -> 35.7). Above the line: 36^3, 16 +
// 24: 46.1 -> 36.6; 12^3, 500 + 700: 271 -> 136; 24^3, 100 + 100: 55.2 -> 48.2; 48^3, 4 + 2:
// 77.6 -> 58.5; 16 + 24: 85.6 -> 61.2; 1024 + 1: 922 -> 656; 96^3, 1 + 1: 524 -> 341. The line was
// drawn before the sweep for the maxima took 43 us in place of 48, and could lie lower.
bool apply_tc_faster(long long ng, int n, int nb) {
  return ng >= (1LL << 16) || ng * ((long long)n + nb) >= (7LL << 18);
}

size_t apply_tc_bytes(long long ng, int n, int nb, size_t tf32) {
  const Scratch s = scratch(nullptr, ng, n, nb, 0);
  const size_t b = tf32 > s.least ? tf32 : s.least;
  return apply_tc_faster(ng, n, nb) ? b + s.tables : b;
}

int launch_apply_tc(const void* Xi, int n, const void* Psi, int nb, long long ld, long long ng, double dv, void* Y,
                    void* ws, size_t budget, int* status, cudaStream_t st) {
  const Scratch s = scratch(static_cast<char*>(ws), ng, n, nb, budget);
  const float2 *x = static_cast<const float2*>(Xi), *psi = static_cast<const float2*>(Psi);
  if (s.splits < 1) return 0;
  CUtensorMap xg, qg, xo;                 // Xi and Psi of the gram product, Xi of the outer one
  if (!encoder() || !vector_map(&xg, x, n, ld, ng, KC / 2, TM, true) ||
      !vector_map(&qg, psi, nb, ld, ng, KC / 2, width(nb) / 2, true) || !vector_map(&xo, x, n, ld, ng, TM, KC / 2, false))
    return 0;
  cudaMemsetAsync(s.mx, 0, (size_t)(reinterpret_cast<char*>(s.pt + ng) - reinterpret_cast<char*>(s.mx)), st);
  // eight to 64 vectors per block (one to eight per warp), by what gives eight blocks per SM
  const long long segs = (ng + SEG - 1) / SEG;
  long long per = (segs * ((long long)n + nb) / (8 * 152) + 7) / 8 * 8;
  per = per < 8 ? 8 : per > kMaxPart ? kMaxPart : per;
  const int ya = (int)((n + per - 1) / per), yb = (int)((nb + per - 1) / per);
  maxima_kernel<<<dim3(ya + yb, (unsigned)segs), 256, 0, st>>>(x, n, psi, nb, ld, ng, (int)per, ya, s.mx, s.pt, s.sx, s.row, s.at_b);
  const int splits = s.splits, nch = (n + 15) / 16;
  long long chunk = (ng + splits - 1) / splits;
  chunk = (chunk + KC / 2 - 1) / (KC / 2) * (KC / 2);
  by_width(width(nb), [&](auto t) {
    constexpr int TN = decltype(t)::value;
    using T = Tile<TN>;
    const int nbt = (nb + T::BB - 1) / T::BB;
    gram16_kernel<TN><<<dim3((n + TM - 1) / TM, nbt, splits), T::G_THREADS, T::G_SMEM, st>>>(xg, n, qg, nb, ng, s.mx, s.sx,
                                                                                     s.row, s.at_b, s.part, chunk, status);
    const long long total = (long long)n * nb;
    int ways = 8;
    while (ways > 1 && (ways > splits || total * ways > 152LL * 2048)) ways /= 2;
    gram16_reduce_kernel<<<(unsigned)((total * ways + 255) / 256), 256, 0, st>>>(s.part, splits, total, ways, dv, s.C);
    c_split_kernel<TN><<<nbt * (T::BB / 8), 256, 0, st>>>(s.C, n, nb, nch, s.mx, s.Bs, s.colexp);
    const long long ntiles = (long long)nbt * ((ng + TM - 1) / TM);
    outer16_kernel<TN><<<(unsigned)(ntiles < 152 ? ntiles : 152), THREADS, T::O_SMEM, st>>>(
        xo, nb, ld, ng, -1.0f, s.pt, s.Bs, s.colexp, nch, static_cast<float2*>(Y), status);
  });
  return 5;
}

}  // namespace ace
