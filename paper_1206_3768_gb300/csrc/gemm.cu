// Complex FP64 GEMM for every dense product of the solver (filter steps, reduction to
// standard form, Gram matrices, basis rotations).
//
// On sm_103a the FP64 pipe issues two fused multiply-adds per clock per SM (about
// 1 TFLOP/s for the chip; a warp's instruction takes 64 clocks of its SM quarter), so a
// complex GEMM is bound by FP64 issue, not by memory, and a small one by how many SMs it
// reaches.  The kernel therefore spends its effort on (1) fewer FMAs per complex product --
// the 3M form
//   Re = Ar Br - Ai Bi,  Im = (Ar + Ai)(Br + Bi) - Ar Br - Ai Bi
// with the operand sums formed once per shared-memory tile, i.e. 3 real FMAs per
// complex multiply-add instead of 4 -- and (2) load balance over the 152 SMs: the tile
// (64 x 32, 32 x 16 or 16 x 8) and the number of K splits are chosen together so that the
// SMs get equal work (choose_shape), and triangular operands skip the k-tiles that are
// known to be zero.
#include <algorithm>
#include <vector>

#include "internal.cuh"

namespace {

constexpr int NT = 128;  // four warps: one per quarter of an SM

// Tile of (16 R) x (8 R) outputs, R x R per thread, BK k-steps per shared-memory stage.
template <int R>
struct Tile {
  static constexpr int BM = 16 * R, BN = 8 * R, BK = R == 1 ? 32 : 16;
};

struct Params {
  GemmDesc g;
  int splits;
  int tiles_m;
  zd* part;  // splits x (M x N) partial sums, ld = M; nullptr when splits == 1
};

template <int R>
__device__ __forceinline__ void tile_k_range(const GemmDesc& g, int i0, int j0, int& klo,
                                             int& khi) {
  constexpr int BM = Tile<R>::BM, BN = Tile<R>::BN, BK = Tile<R>::BK;
  klo = 0;
  khi = g.K;
  if (g.triA == 1) khi = min(khi, i0 + BM);
  if (g.triA == 2) klo = max(klo, i0);
  if (g.triB == 1) khi = min(khi, j0 + BN);
  if (g.triB == 2) klo = max(klo, j0);
  klo = (klo / BK) * BK;
}

template <int OPA, int OPB, int R>
__global__ void __launch_bounds__(NT) zgemm3m_kernel(const Params p) {
  constexpr int BM = Tile<R>::BM, BN = Tile<R>::BN, BK = Tile<R>::BK;
  __shared__ double As[3][BK][BM];
  __shared__ double Bs[3][BK][BN];
  const GemmDesc& g = p.g;
  const int tid = threadIdx.x;
  const int tm = blockIdx.x % p.tiles_m, tn = blockIdx.x / p.tiles_m;
  const int i0 = tm * BM, j0 = tn * BN;
  if (g.lowerC && j0 > i0 + BM - 1) return;

  int klo, khi;
  tile_k_range<R>(g, i0, j0, klo, khi);
  const int nkt = khi > klo ? (khi - klo + BK - 1) / BK : 0;
  const int per = (nkt + p.splits - 1) / p.splits;
  const int kt0 = min(nkt, blockIdx.y * per), kt1 = min(nkt, kt0 + per);

  const int tx = tid & 15, ty = tid >> 4;  // rows tx + 16 r, cols ty + 8 c
  double t1[R][R], t2[R][R], t3[R][R];
#pragma unroll
  for (int r = 0; r < R; ++r)
#pragma unroll
    for (int c = 0; c < R; ++c) t1[r][c] = t2[r][c] = t3[r][c] = 0.0;

  for (int kt = kt0; kt < kt1; ++kt) {
    const int k0 = klo + kt * BK;
    // ---- A tile: op(A)(i0+i, k0+k), i < BM, k < BK
#pragma unroll
    for (int s = 0; s < BM * BK / NT; ++s) {
      const int x = tid + s * NT;
      int i, k;
      if (OPA == OPN) { i = x % BM; k = x / BM; }
      else            { k = x % BK; i = x / BK; }
      const int gi = i0 + i, gk = k0 + k;
      zd v = zmk(0.0, 0.0);
      if (gi < g.M && gk < g.K) {
        if (OPA == OPN) v = g.A[gi + (int64_t)gk * g.lda];
        else { v = g.A[gk + (int64_t)gi * g.lda]; v.y = -v.y; }
      }
      As[0][k][i] = v.x;
      As[1][k][i] = v.y;
      As[2][k][i] = v.x + v.y;
    }
    // ---- B tile: op(B)(k0+k, j0+j), k < BK, j < BN
#pragma unroll
    for (int s = 0; s < BN * BK / NT; ++s) {
      const int x = tid + s * NT;
      int k, j;
      if (OPB == OPN) { k = x % BK; j = x / BK; }
      else            { j = x % BN; k = x / BN; }
      const int gj = j0 + j, gk = k0 + k;
      zd v = zmk(0.0, 0.0);
      if (gj < g.N && gk < g.K) {
        if (OPB == OPN) v = g.B[gk + (int64_t)gj * g.ldb];
        else { v = g.B[gj + (int64_t)gk * g.ldb]; v.y = -v.y; }
      }
      Bs[0][k][j] = v.x;
      Bs[1][k][j] = v.y;
      Bs[2][k][j] = v.x + v.y;
    }
    __syncthreads();
#pragma unroll 4
    for (int kk = 0; kk < BK; ++kk) {
      double br[R], bi[R], bs[R];
#pragma unroll
      for (int c = 0; c < R; ++c) {
        br[c] = Bs[0][kk][ty + 8 * c];
        bi[c] = Bs[1][kk][ty + 8 * c];
        bs[c] = Bs[2][kk][ty + 8 * c];
      }
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const double ar = As[0][kk][tx + 16 * r];
        const double ai = As[1][kk][tx + 16 * r];
        const double as = As[2][kk][tx + 16 * r];
#pragma unroll
        for (int c = 0; c < R; ++c) {
          t1[r][c] = fma(ar, br[c], t1[r][c]);
          t2[r][c] = fma(ai, bi[c], t2[r][c]);
          t3[r][c] = fma(as, bs[c], t3[r][c]);
        }
      }
    }
    __syncthreads();
  }

  // ---- epilogue
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int gi = i0 + tx + 16 * r;
    if (gi >= g.M) continue;
#pragma unroll
    for (int c = 0; c < R; ++c) {
      const int gj = j0 + ty + 8 * c;
      if (gj >= g.N) continue;
      const zd acc = zmk(t1[r][c] - t2[r][c], t3[r][c] - t1[r][c] - t2[r][c]);
      if (p.splits > 1) {
        p.part[(int64_t)blockIdx.y * g.M * g.N + gi + (int64_t)gj * g.M] = acc;
        continue;
      }
      if (g.lowerC && gi < gj) continue;
      zd out = zscale(acc, g.alpha);
      if (g.beta != 0.0) out = zadd(out, zscale(g.Cin[gi + (int64_t)gj * g.ldcin], g.beta));
      if (g.gamma != 0.0) out = zadd(out, zscale(g.D[gi + (int64_t)gj * g.ldd], g.gamma));
      g.C[gi + (int64_t)gj * g.ldc] = out;
    }
  }
}

// Sum the split-K partials in split order (deterministic) and apply the epilogue.
__global__ void zgemm_splitk_epilogue(const Params p) {
  const GemmDesc& g = p.g;
  const int64_t total = (int64_t)g.M * g.N;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int gi = (int)(e % g.M), gj = (int)(e / g.M);
    if (g.lowerC && gi < gj) continue;
    zd acc = zmk(0.0, 0.0);
#pragma unroll 4
    for (int s = 0; s < p.splits; ++s) acc = zadd(acc, p.part[(int64_t)s * total + e]);
    zd out = zscale(acc, g.alpha);
    if (g.beta != 0.0) out = zadd(out, zscale(g.Cin[gi + (int64_t)gj * g.ldcin], g.beta));
    if (g.gamma != 0.0) out = zadd(out, zscale(g.D[gi + (int64_t)gj * g.ldd], g.gamma));
    g.C[gi + (int64_t)gj * g.ldc] = out;
  }
}

// Scale-only path for K == 0 (alpha * 0 + beta Cin + gamma D).
__global__ void zgemm_k0(const GemmDesc g) {
  const int64_t total = (int64_t)g.M * g.N;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int gi = (int)(e % g.M), gj = (int)(e / g.M);
    if (g.lowerC && gi < gj) continue;
    zd out = zmk(0.0, 0.0);
    if (g.beta != 0.0) out = zadd(out, zscale(g.Cin[gi + (int64_t)gj * g.ldcin], g.beta));
    if (g.gamma != 0.0) out = zadd(out, zscale(g.D[gi + (int64_t)gj * g.ldd], g.gamma));
    g.C[gi + (int64_t)gj * g.ldc] = out;
  }
}

}  // namespace

int sm_count() {
  static const int cached = [] {
    int dev = 0, n = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    return n > 0 ? n : 1;
  }();
  return cached;
}

// Tile size R and number of K splits of a product, by modelled clocks: a CTA's k-step issues 3 R^2
// FMAs per thread, 64 clocks each for a warp, and the CTAs of an SM share its quarters, so a launch
// takes ceil(CTAs / SMs) times a CTA's steps; a split launch adds the epilogue kernel and its pass
// over the partials.  Larger tiles are preferred where they are equal (fewer loads and operand
// sums per FMA).  Measured against 64 x 32 tiles only: Gram products and rotations of the n = 512
// sequence (at most 30 columns) 66 -> 12 and 56 -> 11 us (one tile split 16 ways reached 16 SMs),
// filter step n = 1024, m = 64 408 -> 365 us (608 CTAs of 4 unequal k-tiles before), 128 x 128 x 128
// 103 -> 28 us.
// A sum is split at least every CHAIN to 2 CHAIN terms where that takes at most 64 splits and the
// partials have room (above K = 8192 the pieces are K / 64 long; a triangular operand counts half
// its K, so its longest sums are in pieces twice as long): the rounding of a serial sum grows with
// the root of its length, and up to n = 1300 a filter step with the splits that balance alone would
// choose was up to 1.3 times further from the exact one than with the former tile's many splits
// (with these 0.92 to 1.04 times, at the same speed within 1 %).
constexpr int CHAIN = 64;
struct Shape {
  int R, splits, tiles_m, tiles_n;
};
static Shape choose_shape(const GemmDesc& g, size_t cap) {
  const int sms = sm_count();
  const int64_t MN = (int64_t)g.M * g.N;
  Shape best{4, 1, 0, 0};
  double best_cost = 1e300;
  for (int R : {4, 2, 1}) {
    const int bm = 16 * R, bn = 8 * R, bk = R == 1 ? 32 : 16;
    const int tm = (g.M + bm - 1) / bm, tn = (g.N + bn - 1) / bn;
    int64_t active = (int64_t)tm * tn;
    if (g.lowerC) {
      active = 0;
      for (int t = 0; t < tn; ++t) active += std::max(0, tm - t * bn / bm);  // tiles with i0 + bm - 1 >= j0
    }
    // typical k-tiles per tile (triangular operands halve it on average)
    int nkt = (g.K + bk - 1) / bk;
    if (g.triA || g.triB) nkt = std::max(1, nkt / 2);
    const double step = bk * 3.0 * R * R * 64.0 * (R == 4 ? 1.0 : R == 2 ? 1.02 : 1.06);
    const int room = (int)std::min<size_t>(64, cap / (size_t)MN);
    const int fewest = std::max(1, std::min({nkt, room, nkt * bk / CHAIN}));
    for (int S = fewest; S <= std::min(nkt, 64); ++S) {
      if (S > 1 && (size_t)S * (size_t)MN > cap) break;
      const int per = (nkt + S - 1) / S;
      const double waves = (double)((active * S + sms - 1) / sms);
      const double cost = waves * (per * step + 1500.0) + (S > 1 ? 5000.0 + 16.0 * S * MN / 2000.0 : 0.0);
      if (cost < best_cost * 0.98) {
        best_cost = cost;
        best = Shape{R, S, tm, tn};
      }
    }
  }
  return best;
}

template <int R>
static void launch_zgemm(const Params& p, dim3 grid, cudaStream_t stream) {
  const GemmDesc& g = p.g;
  if (g.opA == OPN && g.opB == OPN) zgemm3m_kernel<OPN, OPN, R><<<grid, NT, 0, stream>>>(p);
  else if (g.opA == OPN && g.opB == OPC) zgemm3m_kernel<OPN, OPC, R><<<grid, NT, 0, stream>>>(p);
  else if (g.opA == OPC && g.opB == OPN) zgemm3m_kernel<OPC, OPN, R><<<grid, NT, 0, stream>>>(p);
  else zgemm3m_kernel<OPC, OPC, R><<<grid, NT, 0, stream>>>(p);
}

cudaError_t zgemm_run(const GemmDesc& g, Workspace& ws, cudaStream_t stream) {
  if (g.M <= 0 || g.N <= 0) return cudaSuccess;
  if (g.K <= 0) {
    zgemm_k0<<<std::min<int64_t>(1024, ((int64_t)g.M * g.N + 255) / 256), 256, 0, stream>>>(g);
    CHFSI_COUNT_LAUNCH();
    return cudaGetLastError();
  }
  Params p;
  p.g = g;
  const Shape sh = choose_shape(g, ws.splitk_elems);
  p.tiles_m = sh.tiles_m;
  p.splits = sh.splits;
  p.part = p.splits > 1 ? ws.splitk : nullptr;
  const dim3 grid(sh.tiles_m * sh.tiles_n, p.splits);
  if (sh.R == 4) launch_zgemm<4>(p, grid, stream);
  else if (sh.R == 2) launch_zgemm<2>(p, grid, stream);
  else launch_zgemm<1>(p, grid, stream);
  CHFSI_COUNT_LAUNCH();
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  if (p.splits > 1) {
    const int64_t total = (int64_t)g.M * g.N;
    const int blocks = (int)std::min<int64_t>(4 * sm_count(), (total + 255) / 256);
    zgemm_splitk_epilogue<<<blocks, 256, 0, stream>>>(p);
    CHFSI_COUNT_LAUNCH();
    e = cudaGetLastError();
  }
  return e;
}
