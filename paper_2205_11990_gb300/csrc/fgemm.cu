// FP64 contractions on the FMA pipe: the small and middle-sized products of the
// sweeps (the large ones are sliced over the tensor cores, ozgemm.cu).
//
// GB300 takes two FP64 FMAs per SM and clock, so such a product runs at the rate of
// the SMs it occupies and of the multiplications it does not waste: a 16 x 16 tile
// costs 1 us per 16 of K on its SM, a 64 x 64 one 16 us.  Tiles of 64, 32 or 16
// and up to eight K slices are chosen to finish first by that count (fma_plan);
// rows and columns of a tile beyond the matrix are skipped by whole warps.  The K
// slices of a tile are the CTAs of one cluster, which add their partial products
// through distributed shared memory in a fixed order: no scratch and no second
// launch.  Each slice's sum runs in ascending k.
#include <cuda_runtime.h>

#include <algorithm>
#include <climits>
#include <cmath>

#include <cooperative_groups.h>

#include "common.cuh"

namespace cg = cooperative_groups;

namespace vp {
namespace {

constexpr int kFT = 256, kMaxSlices = 8;

struct FmaJob {
  TcOperand a, b;
  int M, N, K, kslice;
  double alpha;
  double* C;
  int ldc;
};

// element (row r, index k) of an operand of the given kind (TcOperand)
template <int KIND>
__device__ __forceinline__ double operand(const TcOperand& o, int r, int k) {
  if constexpr (KIND == 0) return o.p[(size_t)r * o.ld + k];
  if constexpr (KIND == 1) return o.p[(size_t)k * o.ld + r];
  return r <= k ? o.p[(size_t)k * o.ld + r] : 0.0;
}

template <int KA, int KB, int TILE>
__device__ __forceinline__ void fma_tile(const FmaJob& j, int bx, int by, int slice, int nslices) {
  constexpr int R = TILE / 16;
  __shared__ double As[16][TILE + 1];
  __shared__ double Bs[16][TILE + 1];
  __shared__ double P[TILE <= 32 ? TILE * TILE : 1];  // partial products (K slices: tiles up to 32)
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const int row0 = bx * TILE, col0 = by * TILE;
  // an upper-triangular A is zero for k below its first row
  const int kbeg = KA == 2 ? max(slice * j.kslice, row0) : slice * j.kslice, kend = min(j.K, slice * j.kslice + j.kslice);
  // rows and columns this warp has (warp w: rows 2 w, 2 w + 1 of every 16)
  const int wrow = (tid >> 5) * 2;
  double acc[R][R] = {};
  double ra[R], rb[R];
  // consecutive threads read consecutive addresses of each operand
  auto load = [&](int k0) {
#pragma unroll
    for (int u = 0; u < R; ++u) {
      const int e = tid + kFT * u;
      const int r = KA == 0 ? e / 16 : e % TILE, ka = KA == 0 ? e % 16 : e / TILE;
      ra[u] = row0 + r < j.M && k0 + ka < kend ? operand<KA>(j.a, row0 + r, k0 + ka) : 0.0;
      const int c = KB == 0 ? e / 16 : e % TILE, kb = KB == 0 ? e % 16 : e / TILE;
      rb[u] = col0 + c < j.N && k0 + kb < kend ? operand<KB>(j.b, col0 + c, k0 + kb) : 0.0;
    }
  };
  load(kbeg);
  for (int k0 = kbeg; k0 < kend; k0 += 16) {
#pragma unroll
    for (int u = 0; u < R; ++u) {
      const int e = tid + kFT * u;
      if (KA == 0) As[e % 16][e / 16] = ra[u]; else As[e / TILE][e % TILE] = ra[u];
      if (KB == 0) Bs[e % 16][e / 16] = rb[u]; else Bs[e / TILE][e % TILE] = rb[u];
    }
    __syncthreads();
    if (k0 + 16 < kend) load(k0 + 16);
    const int kn = min(16, kend - k0);
#pragma unroll 4
    for (int kk = 0; kk < kn; ++kk) {
      double av[R], bv[R];
#pragma unroll
      for (int i = 0; i < R; ++i) av[i] = As[kk][ty + 16 * i];
#pragma unroll
      for (int i = 0; i < R; ++i) bv[i] = Bs[kk][tx + 16 * i];
#pragma unroll
      for (int i = 0; i < R; ++i)
        if (row0 + 16 * i + wrow < j.M)
#pragma unroll
          for (int c = 0; c < R; ++c)
            if (col0 + 16 * c < j.N) acc[i][c] = fma(av[i], bv[c], acc[i][c]);
    }
    __syncthreads();
  }
  if (nslices == 1) {
#pragma unroll
    for (int i = 0; i < R; ++i)
#pragma unroll
      for (int c = 0; c < R; ++c) {
        const int r = row0 + ty + 16 * i, q = col0 + tx + 16 * c;
        if (r < j.M && q < j.N) j.C[(size_t)r * j.ldc + q] = j.alpha * acc[i][c];
      }
    return;
  }
  if constexpr (TILE <= 32) {
    cg::cluster_group cl = cg::this_cluster();
#pragma unroll
    for (int i = 0; i < R; ++i)
#pragma unroll
      for (int c = 0; c < R; ++c) P[(ty + 16 * i) * TILE + tx + 16 * c] = acc[i][c];
    cl.sync();
    for (int e = slice * kFT + tid; e < TILE * TILE; e += nslices * kFT) {
      const int r = row0 + e / TILE, q = col0 + e % TILE;
      if (r >= j.M || q >= j.N) continue;
      double part[kMaxSlices];
#pragma unroll
      for (int s = 0; s < kMaxSlices; ++s) part[s] = s < nslices ? *cl.map_shared_rank(P + e, s) : 0.0;
      double sum = 0.0;
#pragma unroll
      for (int s = 0; s < kMaxSlices; s += 2) sum += part[s] + part[s + 1];
      j.C[(size_t)r * j.ldc + q] = j.alpha * sum;
    }
    cl.sync();  // every partial product read before its CTA ends
  }
}

// blockIdx.x: tile, down a column of tiles first (as one number: along y there would be
// too few blocks for 16-wide tiles of a million columns); blockIdx.z: job x K slice (the
// slices of a tile are one cluster)
template <int KA, int KB, int TILE>
__global__ void __launch_bounds__(kFT) kb_gemm_fma(const __grid_constant__ Pack<FmaJob> pk, int zs) {
  follow();
  const FmaJob& j = pk.a[blockIdx.z / zs];
  const int down = (j.M + TILE - 1) / TILE, bx = blockIdx.x % down, by = blockIdx.x / down;
  if (by >= (j.N + TILE - 1) / TILE) return;  // the whole cluster
  fma_tile<KA, KB, TILE>(j, bx, by, blockIdx.z % zs, zs);
}

struct FmaPlan {
  int tile, slices, kslice;
};

// The tile and the K slices that finish first: CTAs per SM times the FMAs of one,
// two a clock, plus ~300 clocks a K step and ~1500 for a cluster's meeting; on a
// tie the smaller tile (8 x 8 x 16 took 34 us as one 64 tile, 26 as one of 16).
// Shape and device only.  (Whole vp_gemm calls on GB300, about 20 us of them the
// call itself, in us with split K through scratch and tiles of 32 and 64 / as it is
// here: 64 x 64 x 16 45.8 / 26.7, 512 x 4 x 2 45.0 / 24.3, 524288 x 4 x 2 959 /
// 102.)
FmaPlan fma_plan(const vp_ctx* ctx, int M, int N, int K) {
  FmaPlan best{16, 1, std::max(K, 1)};
  double least = 1e30;
  for (int tile : {16, 32, 64}) {
    const double tiles = (double)((M + tile - 1) / tile) * ((N + tile - 1) / tile);
    for (int sl : {1, 2, 4, 8}) {
      if (sl > 1 && (tile > 32 || K < 32 * sl)) break;
      const int ks = ((K + sl - 1) / sl + 15) / 16 * 16;
      const int used = std::max(1, (K + ks - 1) / ks);
      if (used != sl) continue;
      const double waves = std::ceil(tiles * sl / ctx->num_sms);
      // a tile no wider than the matrix computes only the 16-blocks it has
      const double rows = std::min(tile, (M + 15) / 16 * 16), cols = std::min(tile, (N + 15) / 16 * 16);
      const double t = waves * std::max(K, 16) / sl * (rows * cols / 2 + 300.0 / 16) + (sl > 1 ? 1500.0 : 0.0);
      if (t < 0.95 * least) {
        least = t;
        best = {tile, sl, sl > 1 ? ks : std::max(K, 1)};
      }
    }
  }
  return best;
}

template <int KA, int KB, int TILE>
int launch_group(vp_ctx* ctx, cudaStream_t st, const std::vector<FmaJob>& jobs, int zs) {
  for (size_t i0 = 0; i0 < jobs.size(); i0 += kMaxBatch) {
    const int nb = (int)std::min<size_t>(kMaxBatch, jobs.size() - i0);
    Pack<FmaJob> pk{};
    long long tiles = 1;
    for (int i = 0; i < nb; ++i) {
      pk.a[i] = jobs[i0 + i];
      tiles = std::max(tiles, (long long)((pk.a[i].M + TILE - 1) / TILE) * ((pk.a[i].N + TILE - 1) / TILE));
    }
    if (tiles > INT_MAX) return fail(ctx, VP_ECAPACITY, "gemm: too large");
    VP_TRY((launch_after(ctx, "gemm", kb_gemm_fma<KA, KB, TILE>, dim3((unsigned)tiles, 1, nb * zs), dim3(kFT), 0, st,
                         zs > 1 ? dim3(1, 1, zs) : kNoCluster, pk, zs)));
  }
  return VP_OK;
}

template <int KA, int KB>
int launch_kind(vp_ctx* ctx, cudaStream_t st, const std::vector<FmaJob>& jobs, int tile, int zs) {
  if (tile == 64) return launch_group<KA, KB, 64>(ctx, st, jobs, zs);
  if (tile == 32) return launch_group<KA, KB, 32>(ctx, st, jobs, zs);
  return launch_group<KA, KB, 16>(ctx, st, jobs, zs);
}

}  // namespace

int blaunch_fma_gemm(vp_ctx* ctx, cudaStream_t st, const std::vector<OzGemm>& v) {
  std::vector<FmaJob> jobs[3][3][4];  // [layout][tile 16 / 32 / 64][1, 2, 4, 8 slices]
  for (const OzGemm& g : v) {
    if (g.N > kGemmMaxN) return fail(ctx, VP_ECAPACITY, "gemm: N too large");
    const FmaPlan pl = fma_plan(ctx, g.M, g.N, g.K);
    const int kind = g.a.kind == 2 ? 2 : g.b.kind == 0 ? 1 : 0;
    const int ti = pl.tile == 64 ? 2 : pl.tile == 32 ? 1 : 0;
    const int si = pl.slices == 1 ? 0 : pl.slices == 2 ? 1 : pl.slices == 4 ? 2 : 3;
    jobs[kind][ti][si].push_back({g.a, g.b, g.M, g.N, g.K, pl.kslice, g.alpha, g.C, g.ldc});
  }
  for (int ti = 0; ti < 3; ++ti)
    for (int si = 0; si < 4; ++si) {
      const int tile = 16 << ti, zs = 1 << si;
      if (!jobs[0][ti][si].empty()) VP_TRY((launch_kind<0, 1>(ctx, st, jobs[0][ti][si], tile, zs)));
      if (!jobs[1][ti][si].empty()) VP_TRY((launch_kind<0, 0>(ctx, st, jobs[1][ti][si], tile, zs)));
      if (!jobs[2][ti][si].empty()) VP_TRY((launch_kind<2, 1>(ctx, st, jobs[2][ti][si], tile, zs)));
    }
  return VP_OK;
}

}  // namespace vp
