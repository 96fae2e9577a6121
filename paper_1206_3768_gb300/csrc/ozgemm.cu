// Split-BF16 tensor-core products for the Chebyshev filter (mixed-precision filter).
//
// A complex FP64 product C = Hs Y (Hs n x n Hermitian, Y n x m) is computed as the real
// product C^ = H^ Y^ of the 2n x 2n real embedding H^ (rows and columns interleaved as
// (re, im), so that Y^ and C^ are the complex column-major arrays read as real arrays)
// with the 2n x m real Y^.  Each operand is split into S "digit slices":
//
//     H^(r, k) = 2^{eA(r)} sum_s a_s(r, k) 2^{-7 s},   |a_1| <= 129, |a_{s>1}| <= 64
//     Y^(k, j) = 2^{eB(j)} sum_t b_t(k, j) 2^{-7 t}
//
// with power-of-two scales per (complex) row of Hs and per column of Y.  Every digit is an
// integer that bf16 holds exactly, every digit product is exact in FP32, and a K-chunk short
// enough that its sums stay below 2^24 accumulates EXACTLY in FP32 accumulators: 960 terms
// where a slice pair has an accumulator to itself (the mma.sync kernel), 384 to 960, by S,
// where the pairs of a level s + t share one (the tcgen05 kernel).  Chunks are scaled by 2^{-7(s+t)} (exact) and summed in double-float (FP32 pairs), and slice
// pairs with s + t <= S + 1 are kept.  The truncation error of the kept pairs is about
// 2^{-7S} relative to the row and column scales, so S = 7 gives FP64-level products and
// S = 3 about 1e-6, at 6 ... 28 tensor-core GEMMs per product instead of FP64 FMAs (which
// run 570x slower than bf16 mma.sync on this part).
#include <algorithm>
#include <cmath>
#include <cuda.h>
#include <cuda_bf16.h>
#include <cudaTypedefs.h>

#include <cstdlib>
#include <cstring>
#include <map>
#include <mutex>
#include <utility>
#include <vector>

#include "digit_plan.cuh"
#include "internal.cuh"

namespace {

// Programmatic dependent launch: a product is a chain of three or four short kernels, and the launch
// latency between them is a good part of a small one.  Each of them lets its successor start as
// soon as all its CTAs run (launch_dependents first) and waits for its own predecessor to have
// finished, with all its writes, before it touches memory (wait; it returns at once in an ordinary
// launch).  Since every kernel of the chain waits, the order of all reads and writes is that of
// the stream.
__device__ __forceinline__ void pdl_enter() {
  asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
  asm volatile("griddepcontrol.wait;\n" ::: "memory");
}

constexpr int OZ_BM = 128, OZ_BN = 64, OZ_BK = 64, OZ_THREADS = 256, OZ_STAGES = 3;
constexpr int OZ_BETA = 7;         // bits per digit slice
constexpr int OZ_CHUNK_KB = 15;    // k-blocks of 64 per exact FP32 chunk (960 terms: 960 * 129^2 < 2^24)
constexpr int OZ_MAX_PAIRS = 64;

struct OzPairs {
  int n;
  unsigned char s[OZ_MAX_PAIRS], t[OZ_MAX_PAIRS];
};

struct OzParams {
  int a_lower;             // A^ is the embedding of a lower-triangular matrix: skip zero k-blocks
  int c_lower;             // only the lower triangle of the complex result is needed
  const __nv_bfloat16* A;  // S_A slices, each Mp x Kp row-major
  const __nv_bfloat16* B;  // S_B slices, each Np x Kp (column j of B^ contiguous)
  int64_t sliceA, sliceB;  // elements per slice
  int Kp;                  // padded K (multiple of 64)
  int nkb;                 // k-blocks of 64 per pair
  int tiles_m;
  int splits;
  OzPairs pairs;
  double* part;            // splits x (Np x Mp) partials, column-major (ld Mp)
  int Mp, Np;
};

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(dst), "l"(src));
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;\n" ::"n"(N));
}

__device__ __forceinline__ void ldmatrix_x4(uint32_t addr, uint32_t& r0, uint32_t& r1, uint32_t& r2,
                                            uint32_t& r3) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
               : "r"(addr));
}

__device__ __forceinline__ void mma_bf16(float* c, const uint32_t* a, uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, "
      "{%8,%9}, {%0,%1,%2,%3};\n"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// byte offset of element (row, k) in a [rows][64] bf16 tile with 16-byte chunks XOR-swizzled
__device__ __forceinline__ uint32_t swz(int row, int k) {
  return (uint32_t)(row * 128 + ((((k >> 3) ^ (row & 7))) << 4) + ((k & 7) << 1));
}

// error-free addition of x into the double-float (hi, lo)
__device__ __forceinline__ void two_sum_acc(float& hi, float& lo, float x) {
  const float s = hi + x;
  const float bp = s - hi;
  const float err = (hi - (s - bp)) + (x - bp);
  hi = s;
  lo += err;
}

// the same for a sc, sc a power of two (so that a sc is exact)
__device__ __forceinline__ void two_sum_scaled(float& hi, float& lo, float a, float sc) {
  const float s = fmaf(a, sc, hi);
  const float bp = s - hi;
  const float err = (hi - (s - bp)) + fmaf(a, sc, -bp);
  hi = s;
  lo += err;
}

__global__ void __launch_bounds__(OZ_THREADS, 1) oz_gemm_kernel(const OzParams p) {
  extern __shared__ __align__(128) unsigned char smem[];
  unsigned char* sA = smem;                                    // stages x 128 x 64 bf16
  unsigned char* sB = smem + OZ_STAGES * OZ_BM * OZ_BK * 2;    // stages x 64 x 64 bf16
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int wm = warp & 3, wn = warp >> 2;
  const int tm = blockIdx.x % p.tiles_m, tn = blockIdx.x / p.tiles_m;
  const int m0 = tm * OZ_BM, n0 = tn * OZ_BN;
  if (p.c_lower && n0 > (m0 + OZ_BM - 1) / 2) return;
  const int nkb = p.a_lower ? min(p.nkb, m0 / OZ_BK + OZ_BM / OZ_BK) : p.nkb;

  const int total = p.pairs.n * nkb;
  const int per = (total + p.splits - 1) / p.splits;
  const int q0 = min(total, (int)blockIdx.y * per), q1 = min(total, q0 + per);

  float acc[2][4][4];
  float hi[2][4][4], lo[2][4][4];
#pragma unroll
  for (int a = 0; a < 2; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b)
#pragma unroll
      for (int c = 0; c < 4; ++c) acc[a][b][c] = hi[a][b][c] = lo[a][b][c] = 0.f;

  auto load_stage = [&](int q, int stage) {
    const int pr = q / nkb, kb = q - pr * nkb;
    const __nv_bfloat16* Ag = p.A + (int64_t)p.pairs.s[pr] * p.sliceA + (int64_t)m0 * p.Kp + kb * OZ_BK;
    const __nv_bfloat16* Bg = p.B + (int64_t)p.pairs.t[pr] * p.sliceB + (int64_t)n0 * p.Kp + kb * OZ_BK;
    const uint32_t sa = smem_u32(sA + stage * OZ_BM * OZ_BK * 2);
    const uint32_t sb = smem_u32(sB + stage * OZ_BN * OZ_BK * 2);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int idx = tid + i * OZ_THREADS;  // 0..1023
      const int row = idx >> 3, ch = idx & 7;
      cp_async16(sa + swz(row, ch * 8), Ag + (int64_t)row * p.Kp + ch * 8);
    }
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const int idx = tid + i * OZ_THREADS;  // 0..511
      const int row = idx >> 3, ch = idx & 7;
      cp_async16(sb + swz(row, ch * 8), Bg + (int64_t)row * p.Kp + ch * 8);
    }
  };

#pragma unroll
  for (int st = 0; st < OZ_STAGES - 1; ++st) {
    if (q0 + st < q1) load_stage(q0 + st, st);
    cp_async_commit();
  }

  for (int q = q0; q < q1; ++q) {
    const int stage = (q - q0) % OZ_STAGES;
    cp_async_wait<OZ_STAGES - 2>();
    __syncthreads();
    {
      const int qn = q + OZ_STAGES - 1;
      if (qn < q1) load_stage(qn, (qn - q0) % OZ_STAGES);
      cp_async_commit();
    }
    const uint32_t sa = smem_u32(sA + stage * OZ_BM * OZ_BK * 2);
    const uint32_t sb = smem_u32(sB + stage * OZ_BN * OZ_BK * 2);
#pragma unroll
    for (int kk = 0; kk < OZ_BK / 16; ++kk) {
      uint32_t af[2][4], bf[4][2];
#pragma unroll
      for (int mt = 0; mt < 2; ++mt) {
        const int row = wm * 32 + mt * 16 + (lane & 7) + ((lane >> 3) & 1) * 8;
        const int k = kk * 16 + (lane >> 4) * 8;
        ldmatrix_x4(sa + swz(row, k), af[mt][0], af[mt][1], af[mt][2], af[mt][3]);
      }
#pragma unroll
      for (int np = 0; np < 2; ++np) {
        const int row = wn * 32 + np * 16 + (lane & 7) + (lane >> 4) * 8;
        const int k = kk * 16 + ((lane >> 3) & 1) * 8;
        ldmatrix_x4(sb + swz(row, k), bf[2 * np][0], bf[2 * np][1], bf[2 * np + 1][0],
                    bf[2 * np + 1][1]);
      }
#pragma unroll
      for (int mt = 0; mt < 2; ++mt)
#pragma unroll
        for (int nt = 0; nt < 4; ++nt) mma_bf16(acc[mt][nt], af[mt], bf[nt][0], bf[nt][1]);
    }
    // drain the exact FP32 chunk at chunk ends, pair ends and the end of this CTA's range
    const int pr = q / nkb, kb = q - pr * nkb;
    if (((kb + 1) % OZ_CHUNK_KB) == 0 || kb == nkb - 1 || q == q1 - 1) {
      const float sc = ldexpf(1.0f, -OZ_BETA * (p.pairs.s[pr] + p.pairs.t[pr] + 2));
#pragma unroll
      for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b)
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            two_sum_acc(hi[a][b][c], lo[a][b][c], acc[a][b][c] * sc);
            acc[a][b][c] = 0.f;
          }
    }
  }
  cp_async_wait<0>();

  // partial (unscaled by the row/column exponents) -> p.part[split][col * Mp + row]
  double* P = p.part + (int64_t)blockIdx.y * p.Mp * p.Np;
#pragma unroll
  for (int mt = 0; mt < 2; ++mt)
#pragma unroll
    for (int nt = 0; nt < 4; ++nt) {
      const int r = m0 + wm * 32 + mt * 16 + (lane >> 2);
      const int c = n0 + wn * 32 + nt * 8 + 2 * (lane & 3);
      P[(int64_t)c * p.Mp + r] = (double)hi[mt][nt][0] + (double)lo[mt][nt][0];
      P[(int64_t)(c + 1) * p.Mp + r] = (double)hi[mt][nt][1] + (double)lo[mt][nt][1];
      P[(int64_t)c * p.Mp + r + 8] = (double)hi[mt][nt][2] + (double)lo[mt][nt][2];
      P[(int64_t)(c + 1) * p.Mp + r + 8] = (double)hi[mt][nt][3] + (double)lo[mt][nt][3];
    }
}

// Complex epilogue of the mma.sync kernel: C(i, j) = 2^{eA(i)+eB(j)} (sum_s P[s](2i, j), sum_s P[s](2i+1,
// j)), out = alpha C + beta Cin + gamma D (out may alias Cin or D element-wise), from FP64 partials.
__global__ void oz_mma_epilogue_kernel(const double* part, int splits, int Mp, int Np, const int* eA,
                                       const int* eB, int n, int m, double alpha, double beta,
                                       const zd* Cin, int64_t ldcin, double gamma, const zd* D,
                                       int64_t ldd, zd* out, int64_t ldo, int lower) {
  const int64_t total = (int64_t)n * m;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int i = (int)(e % n), j = (int)(e / n);
    if (lower && j > i) continue;
    double re = 0.0, im = 0.0;
    for (int s = 0; s < splits; ++s) {
      const double2 v = *reinterpret_cast<const double2*>(part + (int64_t)s * Mp * Np +
                                                          (int64_t)j * Mp + 2 * i);
      re += v.x;
      im += v.y;
    }
    // the kernel applied the slice-level scales 2^{-7(s+t)}; the row and column scales remain
    const int ex = eA[i] + eB[j];
    zd o = zmk(alpha * ldexp(re, ex), alpha * ldexp(im, ex));
    if (beta != 0.0) o = zadd(o, zscale(Cin[i + (int64_t)j * ldcin], beta));
    if (gamma != 0.0) o = zadd(o, zscale(D[i + (int64_t)j * ldd], gamma));
    out[i + (int64_t)j * ldo] = o;
  }
}

// ============================================================================ tcgen05 path
// The same digit products on the 5th-generation tensor cores (tcgen05.mma, bf16 inputs, FP32
// accumulators in tensor memory, operands staged by TMA).
//
// What bounds it: the tensor pipe needs 2 bytes of operand per 128 flops and tile row, and the
// path from L2 into an SM carries about 30 to 40 bytes a clock.  A kernel that brings in one A
// and one B tile for every slice pair (128 x 160 tile: 36 KB for 320 clocks of tensor work)
// is therefore held at 28 % of the tensor rate.  Here a K-block of 64 brings in every slice of
// both operands ONCE (S x 16 KB of A, S x 8 KB of B for a 64-column tile) and all S (S + 1) / 2
// pairs (s, t) are issued from shared memory: 168 KB for 3584 clocks at S = 7, a third of the
// bytes per flop.  Pairs of one level s + t carry the same scale 2^{-7 (s + t)} and add into
// one accumulator, so S levels x 64 columns fit the 512 columns of tensor memory; the A slice s
// meets several consecutive slices of B in ONE instruction of N = (levels of a group) x w
// columns (consecutive slices of B are consecutive rows of the stage, consecutive levels
// consecutive accumulator columns), which also reads the A tile from shared memory once for
// several pairs.  The groups are fixed (digit_plan.cuh): all instructions that add into a column
// have the same accumulator and shape, the condition under which they execute in issue order.
// Where a slice reaches a part of a group only, the other levels meet the zeros in front of
// slice 0 of B: at 7 slices 64 columns wide 31 slice products for 28, 4032 clocks a K-block.  (One
// instruction over all levels that a slice reaches, 3712 clocks, would overlap accumulators of
// different shapes, whose order nothing promises: filter of 20 steps at n = 9300, m = 320 58.6 ms,
// 61.0 with groups.)
// Exactness: |digit 1| <= 129 and the others <= 64, so level l adds at most 129^2 (l = 2) or
// 2 129 64 + (l - 3) 64^2 per k; a chunk of digit::chunk_blocks(S) K-blocks keeps every level below
// 2^24 and each chunk is exact in the FP32 accumulators.  Sixteen drain warps then add the
// levels into double-float sums (hi, lo) held in their registers, every level by two-sum: levels
// s + t >= 7 in the low word alone would lose what passes its 24 bits (sums of one level above
// 2^24; filter of 20 steps at n = 9300, m = 320 61.6 ms, 63.1 with two-sum for all).
// Regions: groups of levels are split into regions of at most 256 accumulator columns (columns 0
// and 256).  With one region (S w <= 256) chunks alternate between the two halves of tensor
// memory; with two, the first and the last K-block of a chunk issue region 0 (the larger
// products) and then region 1, so that draining region 0 overlaps the last products of region
// 1, and draining region 1 the first products of region 0 of the next chunk.
// Measured against the one-pair-per-stage kernel (Gauss form, 7 slices, one product): n = 9300,
// m = 320 6.1 -> 2.85 ms, 1.63 PFLOP/s of slice-pair flops (at the card's power cap: SM clock 2010
// to 2070 MHz); n = 5957, m = 37 0.82 -> 0.26 ms; with 5 slices n = 2600, m = 130 and fewer columns
// 0.15 -> 0.07 ms.
// Warp 0 issues TMA loads (a ring of A tiles and a ring of B stages), warp 1 issues MMAs, warps
// 2..17 drain: four warps per group of 32 tensor-memory lanes, warp h of a group owns the
// 8-column blocks h and h + 4 of the tile.  Every wait on an mbarrier is bounded; a wait that
// runs out sets DEV_TIMEOUT and the CTA unwinds (waiting, again bounded, for its own copies
// and MMAs) before freeing tensor memory.
constexpr int TC_BM = 128, TC_BK = 64;
constexpr int TC_W = digit::WIDEST;                        // widest column tile
constexpr int TC_REGION = digit::REGION;                   // accumulator columns of a region
constexpr int TC_DWQ = 4;                                  // drain warps per 32-lane quarter
constexpr int TC_THREADS = 64 + 32 * 4 * TC_DWQ;           // producer, MMA issuer, drain warps
constexpr int TC_MAX_A = 12, TC_MAX_B = 4;                 // ring depths
constexpr int TC_SMEM_BUDGET = 227 * 1024 - 1024 - 512;    // dynamic shared memory for the rings
constexpr int TC_A_BYTES = TC_BM * TC_BK * 2;              // 16 KB per A tile
static_assert(TC_BK == digit::BLOCK_K && TC_W % 16 == 0 && 8 * TC_W <= 2 * TC_REGION, "eight levels fit two regions");
constexpr long kMbarSpinLimit = 1L << 26;

struct TcParams {
  int a_lower, c_lower;                      // as in OzParams
  int b_tri;                                 // op(B) (complex) zero for k > j (1) or k < j (2)
  int S;                                     // slices (levels)
  int w;                                     // columns per tile (multiple of 16, <= TC_W)
  int group, zeros, U;                       // levels of a group, zero slices of B, levels of region 0
  int nkb, tiles_m, tiles_n, raster, splits, Mp, Np;
  int na, nb;                                // ring depths: A tiles, B stages
  int chunk_kb;                              // K-blocks per exact chunk
  int a_zslices, b_zslices;                  // slices between the products of the Gauss form
  double* part;
  int* status;
  long long spin_limit;                      // polls before a first-level wait gives up
  // Gauss form (nz = 3): blockIdx.z picks one of three real products whose operands follow
  // each other in the slice buffers and whose split partials follow each other in part
  // (splits x Mp x Np entries apart)
  int kfac;  // real k (and rows of A) per complex index: 2 in the embedding, 1 in the Gauss form
};

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(bar), "r"(count));
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(bar), "r"(bytes));
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
      " selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
// Bounded wait: false (with DEV_TIMEOUT set and the CTA's abort flag raised) if it ran out
// or another role of this CTA already gave up.
// The single-thread producer and MMA roles spin without back-off (their waits sit on the
// critical path); the drain warps back off after a while.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag,
                                          int* status, long long limit, bool backoff = false) {
  long long it = 0;
  while (!mbar_try(bar, parity)) {
    if (++it > limit) {
      *abort_flag = 1;
      atomicOr(status, DEV_TIMEOUT);
      return false;
    }
    if ((it & 255) == 0 && *abort_flag) return false;
    if (backoff && it > 1024) __nanosleep(64);
  }
  return true;
}

__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap* map, int x, int y, int z,
                                            uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];\n"
      ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(z), "r"(bar)
      : "memory");
}

// True for one lane of a converged warp.  The producer and the MMA issuer run under this
// election rather than under lane == 0: the tensor instructions take their operands from
// uniform registers, and a branch the compiler knows to be uniform issues them at 39 clocks
// each and a commit at about 100, against 53 and 250 (measured with N = 16).
__device__ __forceinline__ bool elect_one() {
  uint32_t r;
  asm volatile("{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.u32 %0, 1, 0, p;\n}\n" : "=r"(r));
  return r != 0;
}

// Shared-memory matrix descriptor: K-major operand, 128-byte swizzle, 8-row groups 1024 B apart.
__device__ __forceinline__ uint64_t sw128_desc(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);  // start address
  d |= (uint64_t)1 << 16;                     // leading byte offset (unused for this layout)
  d |= (uint64_t)(1024 >> 4) << 32;           // stride byte offset: 8 rows x 128 B
  d |= (uint64_t)1 << 46;                     // descriptor version
  d |= (uint64_t)2 << 61;                     // 128-byte swizzle
  return d;
}

// Instruction descriptor, kind::f16: FP32 accumulator, bf16 A and B, both K-major.
__device__ __forceinline__ uint32_t idesc_bf16(int M, int N) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ void tc_mma(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                       uint32_t accumulate) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n"
      ::"r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate));
}
__device__ __forceinline__ void tc_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n"
               ::"r"(bar) : "memory");
}
__device__ __forceinline__ void tc_fence_after() {
  asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
}
__device__ __forceinline__ void tc_fence_before() {
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
}

__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t* v) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];\n"
               : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
               : "r"(taddr));
}
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory"); }

// The MMA issuer's state: one elected thread walks the K-blocks of its CTA.
struct IssueArgs {
  uint32_t sA, sB, b_slice, b_stage;               // shared-memory addresses (sB: slice 0) and sizes
  uint32_t fullA, emptyA, fullB, emptyB, accf, acce;  // mbarriers
  uint32_t tmem;
  int w, NA, NB, kb_lo, kb_hi, chunk_kb;
  volatile int* abort_flag;
  int* status;
  long long spin_limit;
};
__device__ __noinline__ bool mbar_wait_slow(uint32_t bar, uint32_t parity, volatile int* abort_flag,
                                            int* status, long long limit) {
  return mbar_wait(bar, parity, abort_flag, status, limit);
}
__device__ __forceinline__ bool issue_wait(uint32_t bar, uint32_t parity, const IssueArgs& a) {
  return mbar_try(bar, parity) || mbar_wait_slow(bar, parity, a.abort_flag, a.status, a.spin_limit);
}
// Descriptors of one operand differ in their low word only (the start address).
__device__ __forceinline__ uint64_t desc_from(uint32_t lo, uint32_t hi) {
  uint64_t d;
  asm("mov.b64 %0, {%1, %2};\n" : "=l"(d) : "r"(lo), "r"(hi));
  return d;
}

// S slices, levels in groups of G.  A K-block is S waits, a group of four products for every slice and
// group of levels that it reaches, and S commits; the loops over slices and groups are unrolled
// because one thread issues all of it and its address arithmetic, not the tensor pipe, set the
// pace of a rolled loop (n = 9300, m = 320: 3.5 ms a product).
template <int S, int G>
__device__ __forceinline__ void issue_products(const IssueArgs& a) {
  constexpr int U = digit::region_levels(S, G, digit::widest_with(G));  // levels of region 0
  constexpr int NREG = S > U ? 2 : 1;
  const uint32_t desc_hi = (uint32_t)(sw128_desc(0) >> 32), desc_lo = (uint32_t)sw128_desc(0);
  const uint32_t idesc0 = idesc_bf16(TC_BM, 0), idesc_w = (uint32_t)(a.w >> 3) << 17;
  const uint32_t b_slice16 = a.b_slice >> 4;
  int chunk = 0, sa = 0, sb = 0;
  uint32_t pa = 0, pb = 0;
  for (int k0 = a.kb_lo; k0 < a.kb_hi; k0 += a.chunk_kb, ++chunk) {
    const int k1 = min(a.kb_hi, k0 + a.chunk_kb);
    for (int kb = k0; kb < k1; ++kb) {
      if (!issue_wait(a.fullB + 8 * sb, pb, a)) return;
      const uint32_t b_lo = desc_lo + ((a.sB + (uint32_t)sb * a.b_stage) >> 4);
      const bool first = kb == k0, last = kb == k1 - 1;
      // products of slice s into the groups of region `reg` that it reaches (the first product of
      // a chunk, s = 0, reaches every level of every group and overwrites it)
      auto group = [&](int s, int reg, uint32_t a_lo) -> bool {
        const uint32_t r = NREG == 2 ? (uint32_t)reg : (uint32_t)(chunk & 1);
        if (s == 0 && first) {
          // the region is free once the drain has finished its previous use
          const int use = NREG == 2 ? chunk : (chunk >> 1);
          if (use >= 1 && !issue_wait(a.acce + 8 * r, (use - 1) & 1, a)) return false;
          tc_fence_after();
        }
        const uint32_t keep = (s == 0 && first) ? 0u : 1u;
#pragma unroll
        for (int i = 0; i < digit::groups(S, G); ++i) {
          const digit::Product q = digit::product(S, G, U, s, i);
          if (q.region != reg || q.levels == 0) continue;
          const uint32_t idesc = idesc0 + (uint32_t)q.levels * idesc_w;
          const uint32_t d = a.tmem + r * TC_REGION + (uint32_t)(q.at * a.w);
          const uint32_t bl = b_lo + (uint32_t)q.first * b_slice16;
#pragma unroll
          for (int kk = 0; kk < TC_BK / 16; ++kk)  // 16 k = 32 bytes = 2 descriptor units
            tc_mma(d, desc_from(a_lo + 2 * kk, desc_hi), desc_from(bl + 2 * kk, desc_hi), idesc, kk ? 1u : keep);
        }
        return true;
      };
      int slot = sa;
      uint32_t ph = pa;
      auto next_slot = [&] {
        if (++slot == a.NA) {
          slot = 0;
          ph ^= 1;
        }
      };
      auto a_lo_of = [&](int sl) { return desc_lo + ((a.sA + (uint32_t)sl * TC_A_BYTES) >> 4); };
      if (NREG == 2 && (first || last)) {
        // the first and the last K-block of a chunk issue region 0 and then region 1 (see the
        // header); the A tiles below U stay until their second use
#pragma unroll
        for (int s = 0; s < U; ++s) {
          if (!issue_wait(a.fullA + 8 * slot, ph, a)) return;
          tc_fence_after();
          if (!group(s, 0, a_lo_of(slot))) return;
          next_slot();
        }
        if (last) tc_commit(a.accf);
        slot = sa;
        ph = pa;
#pragma unroll
        for (int s = 0; s < S; ++s) {
          if (s >= U) {
            if (!issue_wait(a.fullA + 8 * slot, ph, a)) return;
            tc_fence_after();
          }
          if (!group(s, 1, a_lo_of(slot))) return;
          tc_commit(a.emptyA + 8 * slot);
          next_slot();
        }
        if (last) tc_commit(a.accf + 8);
      } else {
        // the others slice by slice, which releases the A tiles earlier
#pragma unroll
        for (int s = 0; s < S; ++s) {
          if (!issue_wait(a.fullA + 8 * slot, ph, a)) return;
          tc_fence_after();
          const uint32_t al = a_lo_of(slot);
          if (s < U && !group(s, 0, al)) return;
          if (NREG == 2 && !group(s, 1, al)) return;
          tc_commit(a.emptyA + 8 * slot);
          next_slot();
        }
        if (NREG == 1 && last) tc_commit(a.accf + 8 * (chunk & 1));
      }
      tc_commit(a.emptyB + 8 * sb);
      sa = slot;
      pa = ph;
      if (++sb == a.NB) {
        sb = 0;
        pb ^= 1;
      }
    }
  }
}

__global__ void __launch_bounds__(TC_THREADS, 1)
    oz_gemm_tc_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                      const TcParams p) {
  extern __shared__ unsigned char tc_smem_raw[];
  const uintptr_t base = (reinterpret_cast<uintptr_t>(tc_smem_raw) + 1023) & ~(uintptr_t)1023;
  unsigned char* sA = reinterpret_cast<unsigned char*>(base);
  const int S = p.S, w = p.w, NA = p.na, NB = p.nb;
  // a B stage: the zero slices, then the S slices (all multiples of 2048 bytes)
  const uint32_t b_slice = (uint32_t)w * (TC_BK * 2), b_zeros = (uint32_t)p.zeros * b_slice;
  const uint32_t b_copy = (uint32_t)S * b_slice, b_stage = b_zeros + b_copy;
  unsigned char* sB = sA + NA * TC_A_BYTES;
  uint64_t* bars = reinterpret_cast<uint64_t*>(sB + NB * b_stage);
  // bars: fullA[NA], emptyA[NA], fullB[NB], emptyB[NB], accf[2], acce[2], done[1]
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * (NA + NB) + 5);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  // Tile order: groups of p.raster column tiles; within a group the column tiles of a row tile
  // are neighbours (they stream the same A slices at about the same time), row tiles follow.
  // With a lower-triangular A the row tiles with the longest k-range start first.
  int tm, tn;
  {
    const int per_group = p.tiles_m * p.raster;
    const int g = (int)blockIdx.x / per_group, r = (int)blockIdx.x - g * per_group;
    const int gw = min(p.raster, p.tiles_n - g * p.raster);
    tm = r / gw;
    tn = g * p.raster + (r - tm * gw);
    if (p.a_lower) tm = p.tiles_m - 1 - tm;
  }
  const int m0 = tm * TC_BM, n0 = tn * w;
  if (p.c_lower && n0 > (m0 + TC_BM - 1) / p.kfac) return;  // above the diagonal: not needed
  // nonzero k-blocks of the tile (k in real units, kfac per complex index): below
  // (m0 + 128) / 64 for a lower-triangular A (rows are in the same units); from kfac n0 / 64
  // for a lower-triangular B (zero for k < j); below kfac (n0 + w) / 64 for an
  // upper-triangular B (zero for k > j)
  int kb_first = 0, nkb = p.a_lower ? min(p.nkb, m0 / TC_BK + TC_BM / TC_BK) : p.nkb;
  if (p.b_tri == 2) kb_first = min(nkb, (p.kfac * n0) / TC_BK);
  if (p.b_tri == 1) nkb = min(nkb, (p.kfac * (n0 + w) + TC_BK - 1) / TC_BK);
  // split y takes the k-blocks [y per, (y + 1) per) of them
  const int per = (nkb - kb_first + p.splits - 1) / p.splits;
  const int kb_lo = min(nkb, kb_first + (int)blockIdx.y * per);
  const int kb_hi = min(nkb, kb_lo + per);
  const int U = p.U;  // levels of region 0
  const int nreg = S > U ? 2 : 1;

  const uint32_t sA_u = smem_u32(sA), sB_u = smem_u32(sB) + b_zeros;  // slice 0 of the first stage
  const uint32_t fullA = smem_u32(bars), emptyA = fullA + 8 * NA;
  const uint32_t fullB = emptyA + 8 * NA, emptyB = fullB + 8 * NB;
  const uint32_t accf0 = emptyB + 8 * NB, acce0 = accf0 + 16, done_bar = acce0 + 16;

  if (tid == 0) {
    for (int i = 0; i < NA; ++i) {
      mbar_init(fullA + 8 * i, 1);
      mbar_init(emptyA + 8 * i, 1);
    }
    for (int i = 0; i < NB; ++i) {
      mbar_init(fullB + 8 * i, 1);
      mbar_init(emptyB + 8 * i, 1);
    }
    for (int r = 0; r < 2; ++r) {
      mbar_init(accf0 + 8 * r, 1);
      mbar_init(acce0 + 8 * r, 4 * TC_DWQ);  // one arrival per drain warp
    }
    mbar_init(done_bar, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;\n" ::"r"(
        smem_u32(tmem_slot)));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n");
  }
  for (uint32_t x = tid; x < NB * (b_zeros >> 4); x += TC_THREADS) {
    const uint32_t stage = x / (b_zeros >> 4), at = x - stage * (b_zeros >> 4);
    *reinterpret_cast<uint4*>(sB + stage * b_stage + 16 * at) = make_uint4(0u, 0u, 0u, 0u);
  }
  asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");  // the tensor instructions read the zeros
  tc_fence_before();
  pdl_enter();  // set-up overlaps the end of the slicing; every thread waits before any copy or write
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  if (warp == 0) {
    // ------------------------------------------------------------ TMA producer
    if (elect_one()) {
      // ring positions kept incrementally (no division on this single-thread issue path)
      int ia = 0, ib = 0, sa = 0, sb = 0;
      uint32_t pa = 0, pb = 0;
      bool stop = false;
      const int az = (int)blockIdx.z * p.a_zslices, bz = (int)blockIdx.z * p.b_zslices;
      for (int kb = kb_lo; kb < kb_hi && !stop; ++kb) {
        if (ib >= NB && !mbar_wait(emptyB + 8 * sb, pb ^ 1, abort_flag, p.status, p.spin_limit)) break;
        mbar_expect_tx(fullB + 8 * sb, b_copy);
        tma_load_3d(sB_u + (uint32_t)sb * b_stage, &tmB, kb * TC_BK, n0, bz, fullB + 8 * sb);
        ++ib;
        if (++sb == NB) {
          sb = 0;
          pb ^= 1;
        }
        for (int s = 0; s < S; ++s) {
          if (ia >= NA && !mbar_wait(emptyA + 8 * sa, pa ^ 1, abort_flag, p.status, p.spin_limit)) {
            stop = true;
            break;
          }
          mbar_expect_tx(fullA + 8 * sa, TC_A_BYTES);
          tma_load_3d(sA_u + (uint32_t)sa * TC_A_BYTES, &tmA, kb * TC_BK, m0, az + s, fullA + 8 * sa);
          ++ia;
          if (++sa == NA) {
            sa = 0;
            pa ^= 1;
          }
        }
      }
      // on abort: let the copies already issued (the last NA tiles and NB stages) land before
      // the CTA can exit
      if (*abort_flag) {
        for (int j = max(0, ia - NA); j < ia; ++j) {
          long it = 0;
          while (!mbar_try(fullA + 8 * (j % NA), (j / NA) & 1) && ++it < kMbarSpinLimit) {}
        }
        for (int j = max(0, ib - NB); j < ib; ++j) {
          long it = 0;
          while (!mbar_try(fullB + 8 * (j % NB), (j / NB) & 1) && ++it < kMbarSpinLimit) {}
        }
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------ MMA issuer
    if (elect_one()) {
      IssueArgs ia;
      ia.sA = sA_u; ia.sB = sB_u; ia.b_slice = b_slice; ia.b_stage = b_stage;
      ia.fullA = fullA; ia.emptyA = emptyA; ia.fullB = fullB; ia.emptyB = emptyB;
      ia.accf = accf0; ia.acce = acce0;
      ia.tmem = tmem;
      ia.w = w; ia.NA = NA; ia.NB = NB; ia.kb_lo = kb_lo; ia.kb_hi = kb_hi; ia.chunk_kb = p.chunk_kb;
      ia.abort_flag = abort_flag; ia.status = p.status; ia.spin_limit = p.spin_limit;
      // one unrolled loop per (slices, levels of a group)
      switch (16 * p.group + S) {
        case 16 * 1 + 1: issue_products<1, 1>(ia); break;
        case 16 * 2 + 2: issue_products<2, 2>(ia); break;
        case 16 * 2 + 3: issue_products<3, 2>(ia); break;
        case 16 * 3 + 3: issue_products<3, 3>(ia); break;
        case 16 * 2 + 4: issue_products<4, 2>(ia); break;
        case 16 * 3 + 4: issue_products<4, 3>(ia); break;
        case 16 * 4 + 4: issue_products<4, 4>(ia); break;
        case 16 * 2 + 5: issue_products<5, 2>(ia); break;
        case 16 * 3 + 5: issue_products<5, 3>(ia); break;
        case 16 * 4 + 5: issue_products<5, 4>(ia); break;
        case 16 * 2 + 6: issue_products<6, 2>(ia); break;
        case 16 * 3 + 6: issue_products<6, 3>(ia); break;
        case 16 * 4 + 6: issue_products<6, 4>(ia); break;
        case 16 * 2 + 7: issue_products<7, 2>(ia); break;
        case 16 * 3 + 7: issue_products<7, 3>(ia); break;
        case 16 * 4 + 7: issue_products<7, 4>(ia); break;
        case 16 * 2 + 8: issue_products<8, 2>(ia); break;
        case 16 * 3 + 8: issue_products<8, 3>(ia); break;
        case 16 * 4 + 8: issue_products<8, 4>(ia); break;
        default: break;  // no other (S, w) is launched
      }
      // all MMAs issued by this thread are complete once done_bar fires
      tc_commit(done_bar);
      long it = 0;
      while (!mbar_try(done_bar, 0) && ++it < kMbarSpinLimit) {}
    }
  } else {
    // ------------------------------------------------------------ drain warps (2..17)
    // Thread (quarter, lane) of warp h (0..3 of its lane group) owns row 32 * quarter + lane of
    // the tile and the 8-column blocks h and h + 4.
    const int quarter = warp & 3, h = (warp - 2) >> 2, nblk = w >> 3;
    const uint32_t lane_base = tmem + ((uint32_t)(quarter * 32) << 16);
    float hi[2][8], lo[2][8];
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int q = 0; q < 8; ++q) hi[i][q] = lo[i][q] = 0.f;
    const int nchunks = kb_hi > kb_lo ? (kb_hi - kb_lo + p.chunk_kb - 1) / p.chunk_kb : 0;
    bool ok = true;
    for (int use = 0; use < nchunks * nreg && ok; ++use) {
      const int r = use & 1;  // regions alternate in both forms
      if (!mbar_wait(accf0 + 8 * r, (use >> 1) & 1, abort_flag, p.status, p.spin_limit, true)) {
        ok = false;
        break;
      }
      tc_fence_after();
      const int l0 = (nreg == 2 && r) ? U : 0, nl = l0 ? S - U : U;  // the levels of this region
      const uint32_t acc_base = lane_base + (uint32_t)(r * TC_REGION);
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const int blk = h + 4 * i;
        if (blk < nblk) {
          for (int l = 0; l < nl; l += 4) {
            uint32_t acc[4][8];
#pragma unroll
            for (int q = 0; q < 4; ++q)
              if (l + q < nl) tmem_ld8(acc_base + (uint32_t)((l + q) * w + 8 * blk), acc[q]);
            tmem_wait_ld();
#pragma unroll
            for (int q = 0; q < 4; ++q)
              if (l + q < nl) {
                // level l0 + l + q (0-based) carries 2^{-7 (level + 2)}
                const float sc = __int_as_float((127 - OZ_BETA * (l0 + l + q + 2)) << 23);
#pragma unroll
                for (int c = 0; c < 8; ++c) two_sum_scaled(hi[i][c], lo[i][c], __uint_as_float(acc[q][c]), sc);
              }
          }
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(acce0 + 8 * r);
    }
    if (ok && !*abort_flag) {
      // partial sums of this split as (hi, lo) pairs: P[split][col * Mp + row]
      float2* P = reinterpret_cast<float2*>(p.part) +
                  ((int64_t)blockIdx.z * p.splits + blockIdx.y) * p.Mp * p.Np;
      const int row = m0 + quarter * 32 + lane;
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const int blk = h + 4 * i;
        if (blk < nblk) {
#pragma unroll
          for (int c = 0; c < 8; ++c) {
            const int col = n0 + 8 * blk + c;
            if (col < p.Np) P[(int64_t)col * p.Mp + row] = make_float2(hi[i][c], lo[i][c]);
          }
        }
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 1) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;\n" ::"r"(tmem));
}

// ============================================================================ digit slices
// Digits come from integer operations on the bit patterns (an FP64 instruction occupies an SM
// quarter for 64 clocks).
//
// Key of |x|: its high word, the lowest bit set when the low word is not zero.  Keys order like
// the exponents and are zero for zero only, so a column's scale is a maximum of 32-bit words.
__device__ __forceinline__ unsigned abs_key(double x) {
  return ((unsigned)__double2hiint(x) & 0x7FFFFFFFu) | (__double2loint(x) != 0 ? 1u : 0u);
}
// smallest e with |x| < 2^e for every x of the maximal key (0 for zero)
__device__ __forceinline__ int exponent_of_key(unsigned key) {
  if (key == 0u) return 0;
  const int E = (int)(key >> 20);
  return (E ? E : 1) - 1022;
}
// Balanced digits of x (|x| < 2^e): y = |x| 2^{-e} rounded to 7S fractional bits is sum_k d_k 128^-k
// with d_2 .. d_S in [-64, 63] and d_1 in [0, 129]; the sign of x is applied to all.  Adding 64 at
// every place from the second on makes the places plain base-128 digits d_k + 64, so the word
// below holds all of them, place k at bit 7 (8 - k), without a carry chain.  Then |x - 2^e sum_k d_k
// 2^{-7k}| <= 2^{e-7S-1}, and the dropped slice pairs of a product carry digits of both signs (they
// largely cancel).  Every digit is exact in bf16.
struct DigitWord {
  unsigned long long z;
  unsigned sign;  // sign bit of x
};
__device__ __forceinline__ unsigned long long digit_centre(int S) {  // 64 at places 2 .. S
  unsigned long long c = 0;
#pragma unroll
  for (int k = 2; k <= 8; ++k)
    if (k <= S) c |= 64ull << (7 * (8 - k));
  return c;
}
__device__ __forceinline__ DigitWord digit_word(double x, int e, int S, unsigned long long centre) {
  const unsigned hi = (unsigned)__double2hiint(x);
  const int E = (int)((hi >> 20) & 0x7FFu);
  const unsigned long long mant =
      ((unsigned long long)((hi & 0xFFFFFu) | (E ? 0x100000u : 0u)) << 32) | (unsigned)__double2loint(x);
  const int sh = e - ((E ? E : 1) - 1075) - OZ_BETA * S;  // x = mant 2^(E - 1075); drop sh bits of it
  unsigned long long y;
  if (sh >= 1) y = sh <= 63 ? (mant + (1ull << (sh - 1))) >> sh : 0ull;  // round half up (magnitude)
  else y = mant << -sh;
  DigitWord w;
  w.z = (y << (OZ_BETA * (8 - S))) + centre;
  w.sign = hi & 0x80000000u;
  return w;
}
// bits of the FP32 value of digit k (1 ..): the place put into the significand of 2^23, less 2^23 (+ 64)
__device__ __forceinline__ unsigned digit_float_bits(const DigitWord& w, int k) {
  const unsigned u = k == 1 ? (unsigned)(w.z >> 49) : ((unsigned)(w.z >> (7 * (8 - k))) & 127u);
  return __float_as_uint(__uint_as_float(0x4B000000u | u) - (k == 1 ? 8388608.f : 8388672.f)) ^ w.sign;
}
// two neighbouring bf16 digits (the high halves of their FP32 values)
__device__ __forceinline__ unsigned digit_pair(const DigitWord& a, const DigitWord& b, int k) {
  return __byte_perm(digit_float_bits(a, k), digit_float_bits(b, k), 0x7632);
}
// digits of two neighbouring entries into S slices (out: 4-byte aligned)
__device__ __forceinline__ void store_digits(double a, double b, int e, int S, unsigned long long centre,
                                             __nv_bfloat16* out, int64_t slice) {
  const DigitWord wa = digit_word(a, e, S, centre), wb = digit_word(b, e, S, centre);
#pragma unroll
  for (int k = 1; k <= 8; ++k)
    if (k <= S) *reinterpret_cast<unsigned*>(out + (int64_t)(k - 1) * slice) = digit_pair(wa, wb, k);
}
// digits of two neighbouring complex entries, (re, im) interleaved (out: 8-byte aligned)
__device__ __forceinline__ void store_digits_ri(double ar, double ai, double br, double bi, int e, int S,
                                                unsigned long long centre, __nv_bfloat16* out, int64_t slice) {
  const DigitWord w0 = digit_word(ar, e, S, centre), w1 = digit_word(ai, e, S, centre);
  const DigitWord w2 = digit_word(br, e, S, centre), w3 = digit_word(bi, e, S, centre);
#pragma unroll
  for (int k = 1; k <= 8; ++k)
    if (k <= S)
      *reinterpret_cast<uint2*>(out + (int64_t)(k - 1) * slice) =
          make_uint2(digit_pair(w0, w1, k), digit_pair(w2, w3, k));
}

__device__ __forceinline__ unsigned warp_max(unsigned v) { return __reduce_max_sync(0xffffffffu, v); }

// Operand layouts.  Embedding (one part): B column j = (re, im) of column j interleaved; A rows 2i,
// 2i + 1 = [Re, -Im], [Im, Re] interleaved.  Gauss form (three real products instead of the 2n x 2n
// embedding): Hs Y = (Hr Yr - Hi Yi) + i ((Hr + Hi)(Yr + Yi) - Hr Yr - Hi Yi), parts re, im, re + im
// with a scale per row or column each, slices [part][s][row][k], scales [part][row].  The sums
// are formed in FP64 (one rounding) before the digits are taken.
enum { FORM_EMBED_B = 0, FORM_EMBED_A = 1, FORM_GAUSS = 2 };

// Entry k of column j of the operand: conjugated (rows of a Hermitian or of X^H), or its lower half
// (zero above the diagonal, half of the diagonal entry: the lower part L_h of Y = L_h + L_h^H).
struct ColumnSource {
  const zd* Y;
  int64_t ldy;
  int n, conj, lower_half;
  __device__ __forceinline__ zd at(int j, int k) const {
    if (k >= n) return zmk(0.0, 0.0);
    zd v = Y[k + (int64_t)j * ldy];
    if (conj) v.y = __hiloint2double(__double2hiint(v.y) ^ (int)0x80000000, __double2loint(v.y));
    if (lower_half) {
      if (k < j) v = zmk(0.0, 0.0);
      else if (k == j) v = zmk(0.5 * v.x, 0.5 * v.y);
    }
    return v;
  }
};

// Keys of the columns' parts: key[part * stride + j], raised by atomicMax (cleared before).  Grid:
// (row chunks, columns).
__global__ void oz_col_keys_kernel(const ColumnSource src, int parts, unsigned* key, int stride, int chunk) {
  pdl_enter();
  const int j = blockIdx.y, k1 = min(src.n, (int)(blockIdx.x + 1) * chunk);
  unsigned m0 = 0, m1 = 0, m2 = 0;
  for (int k = blockIdx.x * chunk + threadIdx.x; k < k1; k += blockDim.x) {
    const zd v = src.at(j, k);
    m0 = max(m0, abs_key(v.x));
    m1 = max(m1, abs_key(v.y));
    if (parts == 3) m2 = max(m2, abs_key(v.x + v.y));
  }
  if (parts == 1) m0 = max(m0, m1);
  m0 = warp_max(m0);
  m1 = warp_max(m1);
  m2 = warp_max(m2);
  if ((threadIdx.x & 31) == 0) {
    atomicMax(key + j, m0);
    if (parts == 3) {
      atomicMax(key + stride + j, m1);
      atomicMax(key + 2 * stride + j, m2);
    }
  }
}

// Slices of columns (B operands, and A operands whose rows are conjugated columns).  Grid: (row
// chunks, columns); each thread takes two neighbouring entries, so that a slice is written four
// (eight) bytes at a time.  The columns' keys come from the kernel above or from the epilogue
// that wrote the block; without them (key == nullptr, one chunk) the CTA scans its column first,
// which is cheaper when there are columns enough to fill the GPU (the second read hits L2).
// clear: the key words of the same columns that the next epilogue will raise.
template <int FORM>
__global__ void oz_slice_cols_kernel(const ColumnSource src, int S, __nv_bfloat16* out, int64_t slice,
                                     int64_t zstride, int Kp, int* e_out, int e_stride, const unsigned* key,
                                     unsigned* clear, int chunk) {
  pdl_enter();
  constexpr int parts = FORM == FORM_GAUSS ? 3 : 1;
  const int j = blockIdx.y, tid = threadIdx.x;
  unsigned kz[3] = {0, 0, 0};
  if (key) {
#pragma unroll
    for (int z = 0; z < parts; ++z) kz[z] = key[z * e_stride + j];
  } else {
    __shared__ unsigned sh[3][32];
    for (int k = tid; k < src.n; k += blockDim.x) {
      const zd v = src.at(j, k);
      kz[0] = max(kz[0], abs_key(v.x));
      kz[1] = max(kz[1], abs_key(v.y));
      if (parts == 3) kz[2] = max(kz[2], abs_key(v.x + v.y));
    }
    if (parts == 1) kz[0] = max(kz[0], kz[1]);
#pragma unroll
    for (int z = 0; z < parts; ++z) {
      const unsigned v = warp_max(kz[z]);
      if ((tid & 31) == 0) sh[z][tid >> 5] = v;
    }
    __syncthreads();
#pragma unroll
    for (int z = 0; z < parts; ++z) {
      unsigned v = sh[z][0];
      for (int w = 1; w < (int)(blockDim.x >> 5); ++w) v = max(v, sh[z][w]);
      kz[z] = v;
    }
  }
  int e[3];
#pragma unroll
  for (int z = 0; z < parts; ++z) e[z] = exponent_of_key(kz[z]);
  if (blockIdx.x == 0 && tid == 0) {
#pragma unroll
    for (int z = 0; z < parts; ++z) {
      e_out[z * e_stride + j] = e[z];
      if (clear) clear[z * e_stride + j] = 0u;
    }
  }
  const unsigned long long centre = digit_centre(S);
  const int k1 = min(src.n, (int)(blockIdx.x + 1) * chunk);
  for (int k = blockIdx.x * chunk + 2 * tid; k < k1; k += 2 * blockDim.x) {
    const zd u = src.at(j, k), v = src.at(j, k + 1);
    if (FORM == FORM_GAUSS) {
      __nv_bfloat16* o = out + (int64_t)j * Kp + k;
      store_digits(u.x, v.x, e[0], S, centre, o, slice);
      store_digits(u.y, v.y, e[1], S, centre, o + zstride, slice);
      store_digits(u.x + u.y, v.x + v.y, e[2], S, centre, o + 2 * zstride, slice);
    } else if (FORM == FORM_EMBED_B) {
      store_digits_ri(u.x, u.y, v.x, v.y, e[0], S, centre, out + (int64_t)j * Kp + 2 * k, slice);
    } else {
      __nv_bfloat16* o = out + (int64_t)(2 * j) * Kp + 2 * k;
      store_digits_ri(u.x, -u.y, v.x, -v.y, e[0], S, centre, o, slice);
      store_digits_ri(u.y, u.x, v.y, v.x, e[0], S, centre, o + Kp, slice);
    }
  }
}

// Keys of the ROWS of X (rows x cols, column-major) or of its conjugate: 32-row groups read column by
// column (coalesced), the columns shared out over blockIdx.y.
__global__ void oz_row_keys_kernel(const zd* X, int64_t ldx, int rows, int cols, int conj, int parts, unsigned* key,
                                   int stride) {
  pdl_enter();
  __shared__ unsigned red[3][8][32];
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;  // 32 x 8
  const int r = blockIdx.x * 32 + tx;
  unsigned m0 = 0, m1 = 0, m2 = 0;
  if (r < rows)
    for (int k = blockIdx.y * 8 + ty; k < cols; k += 8 * gridDim.y) {
      const zd v = X[r + (int64_t)k * ldx];
      m0 = max(m0, abs_key(v.x));
      m1 = max(m1, abs_key(v.y));
      if (parts == 3) m2 = max(m2, abs_key(conj ? v.x - v.y : v.x + v.y));
    }
  if (parts == 1) m0 = max(m0, m1);
  red[0][ty][tx] = m0;
  red[1][ty][tx] = m1;
  red[2][ty][tx] = m2;
  __syncthreads();
  if (ty < parts && r < rows) {
    unsigned m = red[ty][0][tx];
    for (int w = 1; w < 8; ++w) m = max(m, red[ty][w][tx]);
    atomicMax(key + ty * stride + r, m);
  }
}

// Slices of the ROWS of X (or of its conjugate): CTAs take one 32-row group and one range of columns
// each, 32 x 32 tiles transposed through shared memory, so that thin matrices still spread over
// the GPU; each thread writes two neighbouring entries.
template <int FORM>
__global__ void oz_slice_rows_kernel(const zd* X, int64_t ldx, int rows, int cols, int S, int conj,
                                     __nv_bfloat16* out, int64_t slice, int64_t zstride, int Kp, int* e_out,
                                     int e_stride, const unsigned* key, int chunk) {
  pdl_enter();
  constexpr int parts = FORM == FORM_GAUSS ? 3 : 1;
  __shared__ int ex[3][32];
  __shared__ zd tile[32][33];
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;  // 32 x 8
  const int r0 = blockIdx.x * 32;
  if (ty < parts) {
    const int e = r0 + tx < rows ? exponent_of_key(key[ty * e_stride + r0 + tx]) : 0;
    ex[ty][tx] = e;
    if (blockIdx.y == 0 && r0 + tx < rows) e_out[ty * e_stride + r0 + tx] = e;
  }
  const unsigned long long centre = digit_centre(S);
  const int k_end = min(cols, (int)(blockIdx.y + 1) * chunk);
  for (int k0 = blockIdx.y * chunk; k0 < k_end; k0 += 32) {
    for (int c = ty; c < 32; c += 8) {
      const int gr = r0 + tx, gk = k0 + c;  // read column gk, rows r0 .. r0 + 31 (coalesced)
      zd v = (gr < rows && gk < k_end) ? X[gr + (int64_t)gk * ldx] : zmk(0.0, 0.0);
      if (conj) v.y = __hiloint2double(__double2hiint(v.y) ^ (int)0x80000000, __double2loint(v.y));
      tile[c][tx] = v;
    }
    __syncthreads();
    for (int it = threadIdx.x; it < 512; it += 256) {  // row r0 + it / 16, columns k0 + 2 (it % 16) and the next
      const int rr = it >> 4, c = 2 * (it & 15), gr = r0 + rr, gk = k0 + c;
      if (gr >= rows || gk >= k_end) continue;
      const zd u = tile[c][rr], v = tile[c + 1][rr];
      if (FORM == FORM_GAUSS) {
        __nv_bfloat16* o = out + (int64_t)gr * Kp + gk;
        store_digits(u.x, v.x, ex[0][rr], S, centre, o, slice);
        store_digits(u.y, v.y, ex[1][rr], S, centre, o + zstride, slice);
        store_digits(u.x + u.y, v.x + v.y, ex[2][rr], S, centre, o + 2 * zstride, slice);
      } else if (FORM == FORM_EMBED_B) {
        store_digits_ri(u.x, u.y, v.x, v.y, ex[0][rr], S, centre, out + (int64_t)gr * Kp + 2 * gk, slice);
      } else {
        __nv_bfloat16* o = out + (int64_t)(2 * gr) * Kp + 2 * gk;
        store_digits_ri(u.x, -u.y, v.x, -v.y, ex[0][rr], S, centre, o, slice);
        store_digits_ri(u.y, u.x, v.y, v.x, ex[0][rr], S, centre, o + Kp, slice);
      }
    }
    __syncthreads();
  }
}

// ============================================================================ epilogue
// (h + l) 2^ex: the exponents are raised in the bit patterns, one FP64 addition is left (FP64
// conversions and ldexp cost several each, and the epilogue was bound by them).
__device__ __forceinline__ double widen_scaled(float x, int ex, bool& in_range) {
  const int f = __float_as_int(x), e = (f >> 23) & 0xFF;
  const int ne = e - 127 + 1023 + ex;
  if (e == 0) return 0.0;
  in_range = ne > 0 && ne < 2047;
  return __hiloint2double((f & 0x80000000) | (ne << 20) | ((f & 0x7FFFFF) >> 3), f << 29);
}
__device__ __forceinline__ double scaled_sum(float h, float l, int ex) {
  bool ok_h = true, ok_l = true;
  const double dh = widen_scaled(h, ex, ok_h), dl = widen_scaled(l, ex, ok_l);
  if (!(ok_h && ok_l)) return ldexp((double)h + (double)l, ex);  // near the ends of the FP64 range
  return dh + dl;
}

// out = alpha C + beta Cin + gamma D (out may alias Cin or D element-wise) from the split partials of
// the tensor-core kernel (double-float pairs, slice scales applied), each scaled by its row and
// column exponents.  NZ = 1: C(i, j) from rows 2i, 2i + 1 of the embedding; NZ = 3: C = P0 - P1 +
// i (P2 - P0 - P1) from the Gauss form's three products.  key (optional): the keys of the columns of
// out, for the slices of the next product (cleared before).  Grid: (row chunks, columns).
// What bounds it: 13 FP64 instructions an entry on large blocks (n = 9300, m = 320: 195 -> 113 us), the
// chain of loads on small ones, which is why the splits' loads are issued in groups.
constexpr int EPI_THREADS = 128;
template <int NZ>
__global__ void __launch_bounds__(EPI_THREADS)
    oz_epilogue_kernel(const float2* part, int splits, int Mp, int Np, const int* eA, const int* eB, int n,
                       double alpha, double beta, const zd* Cin, int64_t ldcin, double gamma, const zd* D,
                       int64_t ldd, zd* out, int64_t ldo, int lower, unsigned* key, int key_stride, int rows) {
  pdl_enter();
  const int64_t prod = (int64_t)Mp * Np, zst = splits * prod;
  const int i1 = min(n, (int)(blockIdx.x + 1) * rows), j = blockIdx.y;
  int eb[NZ];
#pragma unroll
  for (int z = 0; z < NZ; ++z) eb[z] = eB[z * Np + j];
  unsigned m0 = 0, m1 = 0, m2 = 0;
  for (int i = blockIdx.x * rows + threadIdx.x; i < i1; i += EPI_THREADS) {
    if (lower && j > i) continue;
    const zd cin = beta != 0.0 ? Cin[i + (int64_t)j * ldcin] : zmk(0.0, 0.0);
    const zd d = gamma != 0.0 ? D[i + (int64_t)j * ldd] : zmk(0.0, 0.0);
    zd o;
    if (NZ == 1) {
      float rh = 0.f, rl = 0.f, ih = 0.f, il = 0.f;
#pragma unroll 4
      for (int sp = 0; sp < splits; ++sp) {
        const float4 v = *reinterpret_cast<const float4*>(part + sp * prod + (int64_t)j * Mp + 2 * i);
        two_sum_acc(rh, rl, v.x);
        rl += v.y;
        two_sum_acc(ih, il, v.z);
        il += v.w;
      }
      const int ex = eA[i] + eb[0];
      o = zmk(alpha * scaled_sum(rh, rl, ex), alpha * scaled_sum(ih, il, ex));
    } else {
      double v[3];
#pragma unroll
      for (int z = 0; z < 3; ++z) {
        float h = 0.f, l = 0.f;
#pragma unroll 8
        for (int sp = 0; sp < splits; ++sp) {
          const float2 q = part[z * zst + sp * prod + (int64_t)j * Mp + i];
          two_sum_acc(h, l, q.x);
          l += q.y;
        }
        v[z] = scaled_sum(h, l, eA[z * Mp + i] + eb[NZ == 3 ? z : 0]);
      }
      o = zmk(alpha * (v[0] - v[1]), alpha * (v[2] - v[0] - v[1]));
    }
    if (beta != 0.0) o = zadd(o, zscale(cin, beta));
    if (gamma != 0.0) o = zadd(o, zscale(d, gamma));
    out[i + (int64_t)j * ldo] = o;
    if (key) {
      m0 = max(m0, abs_key(o.x));
      m1 = max(m1, abs_key(o.y));
      if (NZ == 3) m2 = max(m2, abs_key(o.x + o.y));
    }
  }
  if (key) {
    if (NZ == 1) m0 = max(m0, m1);
    m0 = warp_max(m0);
    m1 = warp_max(m1);
    m2 = warp_max(m2);
    if ((threadIdx.x & 31) == 0) {
      atomicMax(key + j, m0);
      if (NZ == 3) {
        atomicMax(key + key_stride + j, m1);
        atomicMax(key + 2 * key_stride + j, m2);
      }
    }
  }
}

int choose_oz_splits(int tiles, int total_kb, size_t cap_elems, int64_t tile_elems) {
  const int sms = sm_count();
  int best = 1;
  double best_cost = (double)((tiles + sms - 1) / sms);
  for (int S = 2; S <= 32; ++S) {
    if (total_kb / S < 4) break;
    if ((size_t)S * (size_t)tile_elems > cap_elems) break;
    const int64_t units = (int64_t)tiles * S;
    const double cost = (double)((units + sms - 1) / sms) / S + 0.004 * S;
    if (cost < best_cost * 0.97) { best_cost = cost; best = S; }
  }
  return best;
}

// Split count for the tcgen05 kernel: split y takes k-blocks [y per, (y + 1) per) of every
// tile.  Modelled time in clocks: a K-block costs its tensor work (digit::block_clocks) or its
// bytes at 36 per clock, a CTA about 5000 more (pipeline fill, last drain, partial
// sums), and the launch is that times the waves of one CTA per SM; every split adds a write
// and a read of the partial sums (16 bytes each, about 2800 bytes per clock over the GPU).
int choose_tc_splits(int tiles, int nz, int nkb, int S, int w, size_t cap_elems, int64_t prod_elems) {
  const int sms = sm_count();
  const double kb_cost = std::max((double)digit::block_clocks(S, w), S * (TC_A_BYTES + 128.0 * w) / 36.0);
  int best = 1;
  double best_cost = 1e300;
  for (int sp = 1; sp <= std::min(nkb, 64); ++sp) {
    if ((size_t)sp * (size_t)prod_elems > cap_elems) break;
    const int per = (nkb + sp - 1) / sp;
    const int64_t units = (int64_t)tiles * nz * sp;
    const double cost = (double)((units + sms - 1) / sms) * (per * kb_cost + 5000.0) +
                        16.0 * (double)sp * nz * (double)prod_elems / 2800.0;
    if (cost < best_cost * 0.999) { best_cost = cost; best = sp; }
  }
  return best;
}

}  // namespace

// ---------------------------------------------------------------------------- host side
// Autotuner of the tcgen05 kernel's split count: the best configuration measured for each
// product shape, shared by all contexts of the process (batch workers tune from several host
// threads) whose partial sums allow the same counts: max_splits, the most that a context could
// choose, is part of the key, so that no count is larger than the context has room for.  Environment variable CHFSI_OZ_AUTOTUNE=0 keeps the wave model's choice.
struct TuneKey {
  int Mp, Np, Kp, S, a_lower, c_lower, w, b_tri, nz, max_splits;
  bool operator<(const TuneKey& o) const {
    const int a[10] = {Mp, Np, Kp, S, a_lower, c_lower, w, b_tri, nz, max_splits};
    const int b[10] = {o.Mp, o.Np, o.Kp, o.S, o.a_lower, o.c_lower, o.w, o.b_tri, o.nz, o.max_splits};
    return std::lexicographical_compare(a, a + 10, b, b + 10);
  }
};
static std::mutex g_tune_mu;
static std::map<TuneKey, int> g_tune;
static bool tune_lookup(const TuneKey& k, int* splits) {
  std::lock_guard<std::mutex> lk(g_tune_mu);
  auto it = g_tune.find(k);
  if (it == g_tune.end()) return false;
  *splits = it->second;
  return true;
}
static void tune_store(const TuneKey& k, int splits) {
  std::lock_guard<std::mutex> lk(g_tune_mu);
  g_tune[k] = splits;
}
static bool oz_autotune() {
  static const bool v = [] {
    const char* e = std::getenv("CHFSI_OZ_AUTOTUNE");
    return !(e && std::strcmp(e, "0") == 0);
  }();
  return v;
}
// Product kernel: tcgen05 (default) or the mma.sync kernel, chosen once per process by the
// environment variable CHFSI_OZ_KERNEL ("tc" or "mma").
// The choices below are read once (thread-safe static initialisation: batch workers call
// the product from several host threads).
bool oz_use_tcgen05() {
  static const bool tc = [] {
    const char* v = std::getenv("CHFSI_OZ_KERNEL");
    return !(v && std::strcmp(v, "mma") == 0);
  }();
  return tc;
}
// 3-D bf16 tensor map over `slices` slices of `rows` rows of `inner` elements (row pitch
// `pitch`, slice pitch `slice` elements), boxes of 64 elements x box_rows rows x box_slices
// slices, 128-byte swizzle (the layout the tcgen05 descriptors expect).  inner and rows are the
// operand's true extents: the padding of K and of the last tile is filled with zeros by the
// copy, so the slice buffers need no clearing.
static bool encode_bf16_map(CUtensorMap* map, const void* ptr, int inner, int pitch, int rows, int64_t slice,
                            int slices, int box_rows, int box_slices) {
  static PFN_cuTensorMapEncodeTiled_v12000 encode = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    cudaDriverEntryPointQueryResult q;
    void* fn = nullptr;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q) ==
            cudaSuccess && q == cudaDriverEntryPointSuccess)
      encode = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(fn);
  });
  if (!encode) return false;
  cuuint64_t dims[3] = {(cuuint64_t)inner, (cuuint64_t)rows, (cuuint64_t)slices};
  cuuint64_t strides[2] = {(cuuint64_t)pitch * 2, (cuuint64_t)slice * 2};
  cuuint32_t box[3] = {(cuuint32_t)TC_BK, (cuuint32_t)box_rows, (cuuint32_t)box_slices};
  cuuint32_t estr[3] = {1, 1, 1};
  const CUresult r = encode(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(ptr), dims, strides,
                            box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                            CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS;
}
int oz_padded_k(int n) { return ((2 * n + OZ_BK - 1) / OZ_BK) * OZ_BK; }
int oz_padded_m(int n) { return ((2 * n + OZ_BM - 1) / OZ_BM) * OZ_BM; }
int oz_padded_n(int m) {
  return oz_use_tcgen05() ? ((m + 31) / 32) * 32 : ((m + OZ_BN - 1) / OZ_BN) * OZ_BN;
}

// ---- operands
#define CK_OZ(expr)                 \
  do {                              \
    cudaError_t e_ = (expr);        \
    if (e_ != cudaSuccess) return e_; \
  } while (0)

// Launch with programmatic stream serialization (see pdl_enter; kernels that call it only).
template <class... P, class... A>
static cudaError_t launch_chained(void (*kernel)(P...), dim3 grid, int block, size_t smem, cudaStream_t s,
                                  A... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, P(args)...);
  if (e == cudaSuccess) CHFSI_COUNT_LAUNCH();
  return e;
}

// Where a sliced operand goes: buffer, scales and layout.
struct SliceDst {
  __nv_bfloat16* ptr;
  int64_t slice, zstride;
  int Kp;
  int* e;
  int e_stride, form, S;
};

// Slices of `cols` columns (length n): keys from `key` if given, else scanned by the slicing CTA when
// there are two columns or more per SM, else by a kernel of their own over row chunks.
static cudaError_t slice_cols(const ColumnSource& src, int cols, const SliceDst& d, OzWorkspace& oz, cudaStream_t s,
                              const unsigned* key = nullptr, unsigned* clear = nullptr) {
  const int sms = sm_count();
  int chunk = src.n, gx = 1;
  if (key || cols < 2 * sms) {
    gx = std::max(1, std::min((src.n + 511) / 512, (6 * sms + cols - 1) / cols));
    chunk = ((src.n + gx - 1) / gx + 511) / 512 * 512;
    gx = (src.n + chunk - 1) / chunk;
    if (!key) {
      const int parts = d.form == FORM_GAUSS ? 3 : 1;
      CK_OZ(cudaMemsetAsync(oz.key[oz.key_cur], 0, sizeof(unsigned) * (size_t)parts * d.e_stride, s));
      CK_OZ(launch_chained(oz_col_keys_kernel, dim3(gx, cols), 256, 0, s, src, parts, oz.key[oz.key_cur], d.e_stride,
                           chunk));
      key = oz.key[oz.key_cur];
    }
  }
  const auto kernel = d.form == FORM_GAUSS     ? oz_slice_cols_kernel<FORM_GAUSS>
                      : d.form == FORM_EMBED_A ? oz_slice_cols_kernel<FORM_EMBED_A>
                                               : oz_slice_cols_kernel<FORM_EMBED_B>;
  return launch_chained(kernel, dim3(gx, cols), 256, 0, s, src, d.S, d.ptr, d.slice, d.zstride, d.Kp, d.e, d.e_stride,
                        key, clear, chunk);
}

// Slices of the rows of X (rows x cols) or of its conjugate: keys, then digits by (32-row group, column
// range) CTAs, about four CTAs per SM each.
static cudaError_t slice_rows(const zd* X, int64_t ldx, int rows, int cols, int conj, const SliceDst& d,
                              OzWorkspace& oz, cudaStream_t s) {
  const int groups = (rows + 31) / 32, kchunks = (cols + 31) / 32, parts = d.form == FORM_GAUSS ? 3 : 1;
  unsigned* key = oz.key[oz.key_cur];
  CK_OZ(cudaMemsetAsync(key, 0, sizeof(unsigned) * (size_t)parts * d.e_stride, s));
  const int gy = std::max(1, std::min(kchunks, (4 * sm_count() + groups - 1) / groups));
  CK_OZ(launch_chained(oz_row_keys_kernel, dim3(groups, gy), 256, 0, s, X, ldx, rows, cols, conj, parts, key,
                       d.e_stride));
  const int chunk = 32 * ((kchunks + gy - 1) / gy);
  const auto kernel = d.form == FORM_GAUSS     ? oz_slice_rows_kernel<FORM_GAUSS>
                      : d.form == FORM_EMBED_A ? oz_slice_rows_kernel<FORM_EMBED_A>
                                               : oz_slice_rows_kernel<FORM_EMBED_B>;
  return launch_chained(kernel, dim3(groups, (cols + chunk - 1) / chunk), 256, 0, s, X, ldx, rows, cols, d.S, conj,
                        d.ptr, d.slice, d.zstride, d.Kp, d.e, d.e_stride, key, chunk);
}

// op(A) (M x K) as the A operand.  op = OPC: row i of op(A) is the conjugated column i of X (K x M,
// contiguous); op = OPN: row i of X (M x K, strided).
static cudaError_t slice_a_into(OzA& a, int form, int op, const zd* X, int64_t ldx, int M, int K, int S,
                                OzWorkspace& oz, cudaStream_t s) {
  const SliceDst d{a.ptr, a.slice, (int64_t)S * a.slice, a.Kp, a.e, a.Mp, form, S};
  if (op == OPC) return slice_cols(ColumnSource{X, ldx, K, 1, 0}, M, d, oz, s);
  return slice_rows(X, ldx, M, K, 0, d, oz, s);
}
// op(B) (K x N) as the B operand.  op = OPN: column j of X (optionally its lower half); op = OPC: the
// conjugated row j of X (N x K).
static cudaError_t slice_b_into(OzB& b, int form, int op, const zd* X, int64_t ldx, int K, int N, int S,
                                int lower_half, OzWorkspace& oz, cudaStream_t s, const unsigned* key = nullptr,
                                unsigned* clear = nullptr) {
  const SliceDst d{b.ptr, b.slice, (int64_t)S * b.slice, b.Kp, b.e, b.Np, form, S};
  if (op == OPN) return slice_cols(ColumnSource{X, ldx, K, 0, lower_half}, N, d, oz, s, key, clear);
  return slice_rows(X, ldx, N, K, 1, d, oz, s);
}

static cudaError_t oz_slice_a(OzA& a, int op, const zd* X, int64_t ldx, int M, int K, int S, OzWorkspace& oz,
                              cudaStream_t s) {
  const int Kp = oz_padded_k(K), Mp = oz_padded_m(M);
  if (S > a.S_max || S < 1 || Kp > a.Kp_max || Mp > a.Mp_max || M <= 0 || K <= 0)
    return cudaErrorInvalidValue;
  a.S = S; a.M = M; a.K = K; a.Mp = Mp; a.Kp = Kp; a.nz = 1;
  a.slice = (int64_t)Mp * Kp;
  // zero the padding (rows >= 2M, columns >= 2K) that the mma.sync kernel reads
  if (!oz_use_tcgen05()) CK_OZ(cudaMemsetAsync(a.ptr, 0, sizeof(__nv_bfloat16) * (size_t)S * a.slice, s));
  return slice_a_into(a, FORM_EMBED_A, op, X, ldx, M, K, S, oz, s);
}

static cudaError_t oz_slice_b(OzB& b, int op, const zd* X, int64_t ldx, int K, int N, int S, int Kp, OzWorkspace& oz,
                              cudaStream_t s, int lower_half = 0, const unsigned* key = nullptr,
                              unsigned* clear = nullptr) {
  const int Np = oz_padded_n(N);
  if (Np > b.Np_max || Kp > b.Kp_max || S > b.S_max || S < 1 || N <= 0) return cudaErrorInvalidValue;
  b.S = S; b.N = N; b.Np = Np; b.Kp = Kp; b.nz = 1;
  b.slice = (int64_t)Np * Kp;
  // as in oz_slice_a
  if (!oz_use_tcgen05()) CK_OZ(cudaMemsetAsync(b.ptr, 0, sizeof(__nv_bfloat16) * (size_t)S * b.slice, s));
  return slice_b_into(b, FORM_EMBED_B, op, X, ldx, K, N, S, lower_half, oz, s, key, clear);
}

// out (M x N complex, M = a.M, N = b.N) = alpha op(A) op(B) + beta Cin + gamma D from the
// operands' slices, with the slice pairs (s, t), s + t <= S + 1.  a_lower: op(A) is lower
// triangular (zero k-blocks skipped); c_lower: only the lower triangle of out is written.
cudaError_t oz_product(const OzA& a, const OzB& b, int S, double alpha, double beta, const zd* Cin,
                       int64_t ldcin, double gamma, const zd* D, int64_t ldd, zd* out, int64_t ldo,
                       int a_lower, int c_lower, OzWorkspace& oz, cudaStream_t s,
                       cudaEvent_t ev_gemm_begin, cudaEvent_t ev_gemm_end, int b_tri, unsigned* key_out) {
  const int n = a.M, m = b.N, Kp = a.Kp, Mp = a.Mp, Np = b.Np;
  if (m <= 0 || n <= 0) return cudaSuccess;
  if (S > b.S || S > a.S || S < 1 || a.Kp != b.Kp || a.nz != b.nz) return cudaErrorInvalidValue;
  const int nz = a.nz;  // 3: Gauss form (tcgen05 path only)
  if (nz != 1 && (nz != 3 || !oz_use_tcgen05())) return cudaErrorInvalidValue;
  cudaError_t e = cudaSuccess;
  // Pairs (s, t) with s + t <= S + 1, grouped by the A slice s so that consecutive pairs
  // stream the same slice of the large operand (it stays in L2 between them).
  OzPairs pairs;
  pairs.n = 0;
  for (int si = 1; si <= S; ++si)
    for (int ti = 1; si + ti <= S + 1; ++ti) {
      pairs.s[pairs.n] = (unsigned char)(si - 1);
      pairs.t[pairs.n] = (unsigned char)(ti - 1);
      ++pairs.n;
    }
  int splits = 1;
  if (oz_use_tcgen05()) {
    TcParams tp;
    tp.a_lower = a_lower;
    tp.b_tri = b_tri;
    tp.c_lower = c_lower;
    tp.S = S;
    tp.nkb = Kp / OZ_BK;
    tp.tiles_m = Mp / TC_BM;
    tp.Mp = Mp;
    tp.Np = Np;
    tp.part = oz.part;
    tp.status = oz.status;
    tp.kfac = nz > 1 ? 1 : 2;
    tp.a_zslices = nz > 1 ? a.S : 0;
    tp.b_zslices = nz > 1 ? b.S : 0;
    tp.chunk_kb = digit::chunk_blocks(S);
    // first-level waits: the context's bound (a test hook) or the default; the waits that
    // let issued copies and MMAs finish after an abort always use the default
    tp.spin_limit = oz.wait_limit > 0 ? oz.wait_limit : kMbarSpinLimit;
    // column tiles: as few as cover the block, of equal width (rounded up to 16 columns).  The
    // A slices dominate a K-block's bytes, so fewer and wider tiles win over less padding
    tp.tiles_n = (m + TC_W - 1) / TC_W;
    tp.w = (((m + tp.tiles_n - 1) / tp.tiles_n + 15) / 16) * 16;
    // neighbouring CTAs share A: groups of up to 16 column tiles, so that the CTAs resident at
    // one time (152) cover about 10 row tiles x 16 column tiles of a wide product
    tp.raster = std::min(tp.tiles_n, 16);
    const int tiles = tp.tiles_m * tp.tiles_n;
    tp.group = digit::group_levels(S, tp.w);
    tp.zeros = digit::zero_slices(tp.group);
    tp.U = digit::region_levels(S, tp.group, tp.w);
    const int b_stage = (S + tp.zeros) * tp.w * TC_BK * 2;
    // rings: two B stages (more while a B stage is small against the A tiles of a K-block), the
    // rest of the shared memory for A tiles (at least the slices of region 0 stay resident)
    tp.nb = 2;
    while (tp.nb < TC_MAX_B && (tp.nb + 1) * b_stage + std::min(2 * S, TC_MAX_A) * TC_A_BYTES <= TC_SMEM_BUDGET)
      ++tp.nb;
    tp.na = std::min(TC_MAX_A, (TC_SMEM_BUDGET - tp.nb * b_stage) / TC_A_BYTES);
    if (tp.na < (S > tp.U ? tp.U + 1 : 2)) return cudaErrorInvalidValue;
    CUtensorMap mapA, mapB;
    const int kr = nz > 1 ? a.K : 2 * a.K;  // real k extent of both operands
    if (!encode_bf16_map(&mapA, a.ptr, kr, Kp, nz > 1 ? a.M : 2 * a.M, a.slice, nz * a.S, TC_BM, 1) ||
        !encode_bf16_map(&mapB, b.ptr, kr, Kp, m, b.slice, nz * b.S, tp.w, S))
      return cudaErrorInvalidValue;
    const size_t smem = 1024 + (size_t)tp.na * TC_A_BYTES + (size_t)tp.nb * b_stage + 512;
    // once per process (the library drives one device per process)
    static const cudaError_t tc_attr = cudaFuncSetAttribute(
        oz_gemm_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 1024 + TC_SMEM_BUDGET + 512);
    if (tc_attr != cudaSuccess) return tc_attr;
    auto launch = [&](int sp) -> cudaError_t {
      tp.splits = sp;
      return launch_chained(oz_gemm_tc_kernel, dim3(tiles, sp, nz), TC_THREADS, smem, s, mapA, mapB, tp);
    };
    // split count: the wave model's choice, or the fastest of a few candidates around it,
    // measured on the first product of each shape and kept for the process (autotuner)
    const size_t part_cap = oz.part_elems / (size_t)nz;  // partials of each of the nz products
    const int model_splits = choose_tc_splits(tiles, nz, tp.nkb, S, tp.w, part_cap, (int64_t)Mp * Np);
    splits = model_splits;
    const int max_splits = (int)std::min<size_t>(std::min(tp.nkb, 64), part_cap / ((size_t)Mp * Np));
    if (max_splits < 1) return cudaErrorInvalidValue;
    const TuneKey key{Mp, Np, Kp, S, a_lower, c_lower, tp.w, b_tri, nz, max_splits};
    if (oz_autotune() && !tune_lookup(key, &splits)) {
      cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
      if (cudaStreamIsCapturing(s, &cap) == cudaSuccess && cap == cudaStreamCaptureStatusNone) {
        std::vector<int> cand;
        for (int num : {2, 3, 4, 6, 8}) {  // model x {1/2, 3/4, 1, 3/2, 2}
          const int sp = std::max(1, std::min(max_splits, (model_splits * num + 2) / 4));
          if (std::find(cand.begin(), cand.end(), sp) == cand.end()) cand.push_back(sp);
        }
        cudaEvent_t t0, t1;
        if (cudaEventCreate(&t0) != cudaSuccess || cudaEventCreate(&t1) != cudaSuccess) return cudaGetLastError();
        float best_ms = 1e30f;
        for (const int c : cand) {
          cudaEventRecord(t0, s);
          e = launch(c);
          if (e != cudaSuccess) break;
          cudaEventRecord(t1, s);
          e = cudaEventSynchronize(t1);
          if (e != cudaSuccess) break;
          float ms = 0.f;
          cudaEventElapsedTime(&ms, t0, t1);
          if (ms < best_ms) { best_ms = ms; splits = c; }
        }
        cudaEventDestroy(t0);
        cudaEventDestroy(t1);
        if (e != cudaSuccess) return e;
        tune_store(key, splits);
      }
    }
    if (ev_gemm_begin) cudaEventRecord(ev_gemm_begin, s);
    e = launch(splits);
    if (ev_gemm_end) cudaEventRecord(ev_gemm_end, s);
    if (e != cudaSuccess) return e;
  } else {
    OzParams p;
    p.a_lower = a_lower;
    p.c_lower = c_lower;
    p.A = a.ptr;
    p.B = b.ptr;
    p.sliceA = a.slice;
    p.sliceB = b.slice;
    p.Kp = Kp;
    p.nkb = Kp / OZ_BK;
    p.tiles_m = Mp / OZ_BM;
    p.Mp = Mp;
    p.Np = Np;
    p.pairs = pairs;
    const int tiles = p.tiles_m * (Np / OZ_BN);
    p.splits = splits = choose_oz_splits(tiles, p.pairs.n * p.nkb, oz.part_elems, (int64_t)Mp * Np);
    p.part = oz.part;
    const size_t smem = (size_t)OZ_STAGES * (OZ_BM + OZ_BN) * OZ_BK * 2;
    static const cudaError_t mma_attr =
        cudaFuncSetAttribute(oz_gemm_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (mma_attr != cudaSuccess) return mma_attr;
    if (ev_gemm_begin) cudaEventRecord(ev_gemm_begin, s);
    oz_gemm_kernel<<<dim3(tiles, p.splits), OZ_THREADS, smem, s>>>(p);
    CHFSI_COUNT_LAUNCH();
    if (ev_gemm_end) cudaEventRecord(ev_gemm_end, s);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  if (!oz_use_tcgen05()) {
    const int64_t tot = (int64_t)n * m;
    const int blocks = (int)std::min<int64_t>(4 * sm_count(), (tot + 255) / 256);
    oz_mma_epilogue_kernel<<<blocks, 256, 0, s>>>(oz.part, splits, Mp, Np, a.e, b.e, n, m, alpha, beta, Cin, ldcin,
                                                  gamma, D, ldd, out, ldo, c_lower);
  } else {
    // 1024 rows a CTA, 128 (one per thread) while that leaves less than eight CTAs per SM
    const int rows = (int64_t)((n + 1023) / 1024) * m >= 8 * sm_count() ? 1024 : EPI_THREADS;
    const dim3 grid((n + rows - 1) / rows, m);
    return launch_chained(nz == 3 ? oz_epilogue_kernel<3> : oz_epilogue_kernel<1>, grid, EPI_THREADS, 0, s,
                          reinterpret_cast<const float2*>(oz.part), splits, Mp, Np, a.e, b.e, n, alpha, beta, Cin,
                          ldcin, gamma, D, ldd, out, ldo, c_lower, key_out, Np, rows);
  }
  CHFSI_COUNT_LAUNCH();
  return cudaGetLastError();
}

// Gauss form of the complex products (three real products, see the slicing kernels above):
// with the tcgen05 kernel, when the workspace allows it (the solver allows it for a
// well-conditioned B), unless environment variable CHFSI_OZ_GAUSS=0 keeps the embedding.
static bool oz_gauss(const OzWorkspace& oz) {
  static const bool v = [] {
    const char* e = std::getenv("CHFSI_OZ_GAUSS");
    return !(e && std::atoi(e) == 0);
  }();
  return v && oz.gauss && oz_use_tcgen05();
}

// The Gauss-form operands: slices of the real part, the imaginary part and their sum, a scale per row
// (A) or column (B) of each.
static cudaError_t oz_slice_a3(OzA& a, int op, const zd* X, int64_t ldx, int M, int K, int S, OzWorkspace& oz,
                               cudaStream_t s) {
  const int Mp = ((M + TC_BM - 1) / TC_BM) * TC_BM, Kp = ((K + OZ_BK - 1) / OZ_BK) * OZ_BK;
  if (S > a.S_max || S < 1 || M <= 0 || K <= 0 || Mp > a.Mp_max ||
      (int64_t)3 * S * Mp * Kp > (int64_t)a.S_max * a.Mp_max * a.Kp_max)
    return cudaErrorInvalidValue;
  a.S = S; a.M = M; a.K = K; a.Mp = Mp; a.Kp = Kp; a.nz = 3;
  a.slice = (int64_t)Mp * Kp;
  return slice_a_into(a, FORM_GAUSS, op, X, ldx, M, K, S, oz, s);
}

static cudaError_t oz_slice_b3(OzB& b, int op, const zd* X, int64_t ldx, int K, int N, int S, int Kp, OzWorkspace& oz,
                               cudaStream_t s, int lower_half, const unsigned* key = nullptr,
                               unsigned* clear = nullptr) {
  const int Np = oz_padded_n(N);
  if (S > b.S_max || S < 1 || N <= 0 || K <= 0 || Np > b.Np_max ||
      (int64_t)3 * S * Np * Kp > b.elems)
    return cudaErrorInvalidValue;
  b.S = S; b.N = N; b.Np = Np; b.Kp = Kp; b.nz = 3;
  b.slice = (int64_t)Np * Kp;
  return slice_b_into(b, FORM_GAUSS, op, X, ldx, K, N, S, lower_half, oz, s, key, clear);
}

// ---- the Hermitian matrix of the filter (its slices stay in oz.H for the whole problem)
cudaError_t oz_slice_hermitian(const zd* Hs, int64_t ldh, int n, int S, OzWorkspace& oz,
                               cudaStream_t s) {
  if (oz_gauss(oz)) return oz_slice_a3(oz.H, OPC, Hs, ldh, n, n, S, oz, s);
  return oz_slice_a(oz.H, OPC, Hs, ldh, n, n, S, oz, s);
}

// out(n x m) = alpha Hs Y + beta Cin + gamma D with Hs given by its slices in oz.H and Y
// sliced here into S slices.  In a chain of products whose Y is the previous one's out (or its
// first columns), keys_out of one and keys_in of the next hand the columns' scales on: the epilogue
// that writes a block also finds them, which saves the next product a pass over it.
cudaError_t oz_filter_product(const zd* Y, int64_t ldy, int n, int m, int S, double alpha,
                              double beta, const zd* Cin, int64_t ldcin, double gamma, const zd* D,
                              int64_t ldd, zd* out, int64_t ldo, OzWorkspace& oz, cudaStream_t s,
                              cudaEvent_t ev_gemm_begin, cudaEvent_t ev_gemm_end, bool keys_in, bool keys_out) {
  if (m <= 0) return cudaSuccess;
  if (S > oz.H.S || S < 1 || oz.H.M != n) return cudaErrorInvalidValue;
  if (!oz_use_tcgen05()) keys_in = keys_out = false;
  // keys of Y in buffer key_cur; the slicing clears the other buffer for the epilogue.  The keys'
  // stride is the padded width of the product that left them: one of another width scans Y again
  unsigned* clear = nullptr;
  const unsigned* key = nullptr;
  if (keys_in && oz.key_np == oz_padded_n(m)) key = oz.key[oz.key_cur];
  if (keys_out) {
    clear = oz.key[1 - oz.key_cur];
    if (!key) CK_OZ(cudaMemsetAsync(clear, 0, sizeof(unsigned) * 3 * (size_t)oz_padded_n(m), s));
  }
  cudaError_t e = oz.H.nz == 3 ? oz_slice_b3(oz.B, OPN, Y, ldy, n, m, S, oz.H.Kp, oz, s, 0, key, key ? clear : nullptr)
                               : oz_slice_b(oz.B, OPN, Y, ldy, n, m, S, oz.H.Kp, oz, s, 0, key, key ? clear : nullptr);
  if (e != cudaSuccess) return e;
  e = oz_product(oz.H, oz.B, S, alpha, beta, Cin, ldcin, gamma, D, ldd, out, ldo, 0, 0, oz, s,
                 ev_gemm_begin, ev_gemm_end, 0, clear);
  if (keys_out) {
    oz.key_cur = 1 - oz.key_cur;
    oz.key_np = oz_padded_n(m);
  }
  return e;
}

// General product with split operands: C = alpha op(A) op(B) + beta Cin + gamma D,
// op(A) M x K, op(B) K x N.  Uses the scratch operand buffers (not oz.H).
cudaError_t oz_gemm(int opA, const zd* A, int64_t lda, int opB, const zd* B, int64_t ldb, int M, int N,
                    int K, int S, double alpha, double beta, const zd* Cin, int64_t ldcin, double gamma,
                    const zd* D, int64_t ldd, zd* C, int64_t ldc, int a_lower, int c_lower,
                    OzWorkspace& oz, cudaStream_t s, int b_tri, int b_lower_half) {
  const bool g3 = oz_gauss(oz);
  CK_OZ(g3 ? oz_slice_a3(oz.X, opA, A, lda, M, K, S, oz, s) : oz_slice_a(oz.X, opA, A, lda, M, K, S, oz, s));
  CK_OZ(g3 ? oz_slice_b3(oz.B, opB, B, ldb, K, N, S, oz.X.Kp, oz, s, b_lower_half)
           : oz_slice_b(oz.B, opB, B, ldb, K, N, S, oz.X.Kp, oz, s, b_lower_half));
  return oz_product(oz.X, oz.B, S, alpha, beta, Cin, ldcin, gamma, D, ldd, C, ldc, a_lower, c_lower, oz,
                    s, nullptr, nullptr, b_tri);
}

int64_t oz_pair_count(int S) { return (int64_t)S * (S + 1) / 2; }

static cudaError_t alloc_a(OzA& a, int n_max, int S_max) {
  a.S_max = S_max;
  a.Kp_max = oz_padded_k(n_max);
  a.Mp_max = oz_padded_m(n_max);
  cudaError_t e = cudaMalloc((void**)&a.ptr, sizeof(__nv_bfloat16) * (size_t)S_max * a.Mp_max * a.Kp_max);
  if (e != cudaSuccess) return e;
  return cudaMalloc((void**)&a.e, sizeof(int) * (size_t)3 * a.Mp_max);  // 3 scale sets (Gauss form)
}

cudaError_t oz_alloc(OzWorkspace& oz, int n_max, int blk_max, int S_max) {
  cudaError_t e = alloc_a(oz.H, n_max, S_max);
  if (e != cudaSuccess) return e;
  e = alloc_a(oz.X, n_max, S_max);
  if (e != cudaSuccess) return e;
  // B operands: blocks of up to blk_max columns, and n_max columns for the reduction
  const int cols = std::max(n_max, blk_max);
  oz.B.S_max = S_max;
  oz.B.Kp_max = oz_padded_k(n_max);
  // covers both kernels' paddings
  oz.B.Np_max = ((std::max(cols, TC_W) + OZ_BN - 1) / OZ_BN) * OZ_BN;
  // the Gauss form holds three K x N parts (K padded to 64 complex entries) per slice, the
  // embedding one 2K-row part
  const int64_t kp1 = ((n_max + OZ_BK - 1) / OZ_BK) * OZ_BK;
  oz.B.elems = std::max<int64_t>((int64_t)S_max * oz.B.Np_max * oz.B.Kp_max,
                                 (int64_t)3 * S_max * oz.B.Np_max * kp1);
  e = cudaMalloc((void**)&oz.B.ptr, sizeof(__nv_bfloat16) * (size_t)oz.B.elems);
  if (e != cudaSuccess) return e;
  e = cudaMalloc((void**)&oz.B.e, sizeof(int) * (size_t)3 * oz.B.Np_max);
  if (e != cudaSuccess) return e;
  for (int k = 0; k < 2; ++k) {
    e = cudaMalloc((void**)&oz.key[k], sizeof(unsigned) * (size_t)3 * std::max(oz.B.Np_max, oz.H.Mp_max));
    if (e != cudaSuccess) return e;
  }
  const int np_blk = ((blk_max + OZ_BN - 1) / OZ_BN) * OZ_BN;
  const size_t mp = (size_t)oz_padded_m(n_max);
  const size_t mp1 = (size_t)((n_max + TC_BM - 1) / TC_BM) * TC_BM;  // rows of a Gauss-form product
  // split partials: 32 splits of a block product, one split of an n x n product (three of
  // them in the Gauss form)
  oz.part_elems = std::max({(size_t)32 * mp * np_blk, mp * oz.B.Np_max, (size_t)3 * mp1 * oz.B.Np_max});
  return cudaMalloc((void**)&oz.part, sizeof(double) * oz.part_elems);
}

void oz_free(OzWorkspace& oz) {
  void* ptrs[] = {oz.H.ptr, oz.H.e, oz.X.ptr, oz.X.e, oz.B.ptr, oz.B.e, oz.part,
                  oz.key[0], oz.key[1]};
  for (void* q : ptrs)
    if (q) cudaFree(q);
  oz = OzWorkspace{};
}
