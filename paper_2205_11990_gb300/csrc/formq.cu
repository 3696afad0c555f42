// Q = H_0 ... H_{p-1} [I_p; 0] of a factored matrix, in double words (SI
// "Canonicalization and Compression").
//
// The columns of Q are independent; each is a chain over the reflectors, and one
// reflector at a time (a dot product, a warp's sum, an update) that chain waited on
// its own reductions: 0.7-1.1 us a reflector with the column in registers, 4.5-8 us
// above 512 rows, where it went through L2.  Here four reflectors are applied at
// once, H_4s ... H_4s+3 = I - V T V^T with V's four columns: four products of the
// column, one reduction for all of them, T (from the reflectors' own products,
// formed once beside the conversion to double words) and one update, with the
// column and the rows of V in registers.  W warps hold a column, eight rows a lane,
// and the columns of a block share V's panels through shared memory, the next panel
// in flight while one is applied.  Rows above a panel are neither loaded nor
// touched.  The arithmetic of a column depends on the factor's shape only.
//
// Measured on GB300 (event-timed, in a sweep, best of five; before: one reflector at a
// time): 1024 x 528 391 us (2891), 1456 x 348 244 (2894), 1056 x 184 122 (1154), 448 x 168
// 93 (153), 128 x 128 31 (106), 64 x 64 19 (36).
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "common.cuh"
#include "dw.cuh"
#include "dwsum.cuh"

namespace vp {
namespace {

constexpr int kFB = 4;            // reflectors applied at once
constexpr int kFqShared = 2048;   // rows up to which two panels fit shared memory
constexpr int kFqMaxRows = 4096;  // beyond: columns in global memory

struct FqArgs {
  const double* A;  // factored: reflectors below the diagonal
  const double* tau;
  int m, p;
  dw* V;  // m x 4 np, np = ceil(p / 4): reflectors, zero above the diagonal
  dw* T;  // 16 per panel: T_{qr} at 4 q + r (q <= r), zero below
  dw* scratch;
  double* Q;
  const int* rows;
};

__device__ __forceinline__ int panels(int p) { return (p + kFB - 1) / kFB; }

// Panel blockIdx.x of the reflectors as double words, and its T.
__global__ void __launch_bounds__(256) kb_formq_prep(const __grid_constant__ Pack<FqArgs> pk) {
  follow();
  const FqArgs& a = pk.a[blockIdx.y];
  __shared__ dw part[8][8];
  const int m = a.m, p = a.p, s = blockIdx.x, j0 = kFB * s;
  if (s >= panels(p)) return;  // the whole block
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  dw_acc acc[8];  // v_q . v_r, q < r: (01)(02)(03)(12)(13)(23)
  for (int i = tid; i < m; i += 256) {
    dw v[kFB];
#pragma unroll
    for (int q = 0; q < kFB; ++q) {
      const int j = j0 + q;
      v[q] = j < p && i > j ? dw_from_scaled(a.A[(size_t)j * m + i], 0) : dw{j < p && i == j ? 1.0f : 0.0f, 0.0f};
      a.V[(size_t)j * m + i] = v[q];
    }
    dw_dot_step(acc[0], v[0], v[1]);
    dw_dot_step(acc[1], v[0], v[2]);
    dw_dot_step(acc[2], v[0], v[3]);
    dw_dot_step(acc[3], v[1], v[2]);
    dw_dot_step(acc[4], v[1], v[3]);
    dw_dot_step(acc[5], v[2], v[3]);
  }
  dw val[8];
#pragma unroll
  for (int e = 0; e < 8; ++e) val[e] = {acc[e].s, acc[e].c};
  const dw w = warp_sums<8>(val, lane);
  if ((lane & 3) == 0) part[warp][lane >> 2] = w;
  __syncthreads();
  if (tid != 0) return;
  dw g[6], t[kFB];
#pragma unroll
  for (int e = 0; e < 6; ++e) {
    dw x = part[0][e];
#pragma unroll
    for (int u = 1; u < 8; ++u) x = acc_add(x, part[u][e]);
    g[e] = norm2(x);
  }
#pragma unroll
  for (int q = 0; q < kFB; ++q) t[q] = j0 + q < p ? dw_from_scaled(a.tau[j0 + q], 0) : dw{0.f, 0.f};
  // T_{qq} = tau_q; column r above it: -tau_r T_{0..r-1, 0..r-1} (V^T v_r)
  const dw t01 = dw_neg(dw_mul(t[1], dw_mul(t[0], g[0])));
  const dw t12 = dw_neg(dw_mul(t[2], dw_mul(t[1], g[3])));
  const dw t02 = dw_neg(dw_mul(t[2], dw_add(dw_mul(t[0], g[1]), dw_mul(t01, g[3]))));
  const dw t23 = dw_neg(dw_mul(t[3], dw_mul(t[2], g[5])));
  const dw t13 = dw_neg(dw_mul(t[3], dw_add(dw_mul(t[1], g[4]), dw_mul(t12, g[5]))));
  const dw t03 = dw_neg(dw_mul(t[3], dw_add(dw_add(dw_mul(t[0], g[2]), dw_mul(t01, g[4])), dw_mul(t02, g[5]))));
  const dw z = {0.f, 0.f};
  const dw T[16] = {t[0], t01, t02, t03, z, t[1], t12, t13, z, z, t[2], t23, z, z, z, t[3]};
#pragma unroll
  for (int e = 0; e < 16; ++e) a.T[16 * s + e] = T[e];
}

// 16 bytes from global to shared memory, asynchronously.
__device__ __forceinline__ void copy16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}

// NC columns a block, W warps each, row 32 (warp + W r) + lane, r < R (m <= 32 W R).
// Block 0 has the last columns, whose chains are the longest.
template <int W, int R, int NC>
__global__ void __launch_bounds__(32 * W * NC, W * NC <= 8 ? 2 : 1) kb_formq(const __grid_constant__ Pack<FqArgs> pk) {
  follow();
  constexpr int T = 32 * W * NC;
  const FqArgs& a = pk.a[blockIdx.y];
  extern __shared__ double qsm[];
  __shared__ dw part[W * NC][kFB];
  __shared__ __align__(16) dw Ts[2][16];
  const int m = a.m, p = a.p, groups = (p + NC - 1) / NC;
  if ((int)blockIdx.x >= groups) return;  // the whole block
  const int tid = threadIdx.x, lane = tid & 31, cl = tid / (32 * W), wc = (tid >> 5) % W;
  const int k0 = (groups - 1 - blockIdx.x) * NC, k = k0 + cl;
  dw* Vs = reinterpret_cast<dw*>(qsm);  // two panels of 4 m
  dw c[R];
#pragma unroll
  for (int r = 0; r < R; ++r) c[r] = {32 * (wc + W * r) + lane == k ? 1.0f : 0.0f, 0.0f};
  constexpr bool SHARED = 32 * W * R <= kFqShared;
  auto fetch = [&](int s) {  // (a panel is a multiple of 32 bytes)
    if constexpr (!SHARED) return;
    const dw* src = a.V + (size_t)kFB * s * m;
    dw* dst = Vs + (size_t)(s & 1) * kFB * m;
    for (int e = 2 * tid; e < kFB * m; e += 2 * T) copy16(dst + e, src + e);
    if (tid < 8) copy16(&Ts[s & 1][2 * tid], a.T + 16 * s + 2 * tid);
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  const int top = min(k0 + NC, p) - 1;
  fetch(top / kFB);
  for (int s = top / kFB; s >= 0; --s) {
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();  // panel s in place, and the other buffer no longer read
    if (s > 0) fetch(s - 1);
    const dw* v = SHARED ? Vs + (size_t)(s & 1) * kFB * m : a.V + (size_t)kFB * s * m;
    const dw* t = SHARED ? Ts[s & 1] : a.T + 16 * s;
    auto live = [&](int r) { return 32 * (wc + W * r) < m && 32 * (wc + W * r) + 31 >= kFB * s; };
    dw vv[R][kFB];
    dw_acc acc[kFB];
#pragma unroll
    for (int r = 0; r < R; ++r) {
      if (!live(r)) continue;
      const int i = 32 * (wc + W * r) + lane;
#pragma unroll
      for (int q = 0; q < kFB; ++q) {
        vv[r][q] = i < m ? v[(size_t)q * m + i] : dw{0.f, 0.f};
        dw_dot_step(acc[q], vv[r][q], c[r]);
      }
    }
    dw val[kFB];
#pragma unroll
    for (int q = 0; q < kFB; ++q) val[q] = {acc[q].s, acc[q].c};
    dw S = warp_sums<kFB>(val, lane);  // lane / 8: q
    if constexpr (W > 1) {
      if ((lane & 7) == 0) part[cl * W + wc][lane >> 3] = S;
      __syncthreads();
      S = {0.f, 0.f};
#pragma unroll
      for (int u = 0; u < (W + 7) / 8; ++u) {
        const int w = (lane & 7) + 8 * u;
        if (w < W) S = acc_add(S, part[cl * W + w][lane >> 3]);
      }
#pragma unroll
      for (int o = (W < 8 ? W : 8) / 2; o >= 1; o >>= 1) S = acc_add(S, shfl_xor_dw(S, o));
    }
    S = norm2(S);
    // w = T (V^T c): row lane mod 4 in each lane
    dw_acc wa;
#pragma unroll
    for (int r = 0; r < kFB; ++r) dw_dot_step(wa, t[(lane & 3) * kFB + r], shfl_dw(S, 8 * r));
    const dw wl = dw_acc_value(wa);
    dw w[kFB];
#pragma unroll
    for (int q = 0; q < kFB; ++q) w[q] = shfl_dw(wl, q);
#pragma unroll
    for (int r = 0; r < R; ++r) {
      if (!live(r)) continue;
      float hi = c[r].hi, lo = c[r].lo;
#pragma unroll
      for (int q = 0; q < kFB; ++q) fnma_acc(hi, lo, w[q], vv[r][q]);
      c[r] = fast_two_sum(hi, lo);
    }
  }
  if (k >= p) return;
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int i = 32 * (wc + W * r) + lane;
    if (i < m) a.Q[(size_t)(a.rows ? a.rows[i] : i) * p + k] = dw_to_scaled(c[r], 0);
  }
}

// More than kFqMaxRows rows: a warp per column, the column in global memory, one
// reflector at a time.
__global__ void kb_formq_long(const __grid_constant__ Pack<FqArgs> pk) {
  follow();
  const FqArgs& a = pk.a[blockIdx.y];
  const int lane = threadIdx.x & 31, m = a.m;
  const int k = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (k >= a.p) return;
  dw* q = a.scratch + (size_t)k * m;
  for (int i = lane; i < m; i += 32) q[i] = (i == k) ? dw{1.0f, 0.0f} : dw{0.0f, 0.0f};
  __syncwarp();
  for (int j = k; j >= 0; --j) {
    const dw t = a.T[16 * (j / kFB) + 5 * (j % kFB)];
    if (t.hi == 0.f) continue;
    const dw* v = a.V + (size_t)j * m;
    dw_acc acc;
    for (int i = j + lane; i < m; i += 32) dw_dot_step(acc, v[i], q[i]);
    const dw w = dw_mul(dw_warp_sum(dw_acc_value(acc)), t);
    for (int i = j + lane; i < m; i += 32) q[i] = dw_add(q[i], dw_neg(dw_mul(w, v[i])));
    __syncwarp();
  }
  for (int i = lane; i < m; i += 32) a.Q[(size_t)(a.rows ? a.rows[i] : i) * a.p + k] = dw_to_scaled(q[i], 0);
}

dw* align16(double* p) { return reinterpret_cast<dw*>((reinterpret_cast<uintptr_t>(p) + 15) & ~uintptr_t(15)); }

template <int W, int R, int NC>
int launch_formq(vp_ctx* ctx, cudaStream_t st, const std::vector<FqArgs>& v) {
  constexpr bool shared = 32 * W * R <= kFqShared;
  static AttrOnce at;
  if (!v.empty() && shared)
    VP_TRY(at.ensure(ctx, (const void*)kb_formq<W, R, NC>, 2 * kFB * 32 * W * R * (int)sizeof(dw), false));
  for (size_t i0 = 0; i0 < v.size(); i0 += kMaxBatch) {
    const int nb = (int)std::min<size_t>(kMaxBatch, v.size() - i0);
    Pack<FqArgs> pk{};
    int gx = 1, mm = 1;
    for (int i = 0; i < nb; ++i) {
      pk.a[i] = v[i0 + i];
      gx = std::max(gx, (pk.a[i].p + NC - 1) / NC);
      mm = std::max(mm, pk.a[i].m);
    }
    VP_TRY((launch_after(ctx, "formq", kb_formq<W, R, NC>, dim3(gx, nb), dim3(32 * W * NC),
                         shared ? 2 * kFB * (size_t)mm * sizeof(dw) : 0, st, kNoCluster, pk)));
  }
  return VP_OK;
}

}  // namespace

int blaunch_formq(vp_ctx* ctx, cudaStream_t st, const std::vector<FormQJob>& v) {
  std::vector<FqArgs> all, by[8], beyond;
  for (const FormQJob& j : v) {
    const int p = std::min(j.m, j.n);
    if (p <= 0) continue;
    const size_t np = (p + kFB - 1) / kFB;
    // T and V on 16-byte boundaries, as their asynchronous copies need, whatever the
    // allocator's alignment
    VP_TRY(reserve(ctx, *j.v, (size_t)j.m * kFB * np + 16 * np + 1));
    FqArgs a{j.A, j.tau, j.m, p, nullptr, align16(j.v->p), nullptr, j.Q, j.rows};
    a.V = a.T + 16 * np;
    if (j.m > kFqMaxRows) {
      VP_TRY(reserve(ctx, *j.scratch, (size_t)j.m * p));
      a.scratch = reinterpret_cast<dw*>(j.scratch->p);
      beyond.push_back(a);
    } else {
      by[j.m <= 32 ? 0 : j.m <= 64 ? 1 : j.m <= 128 ? 2 : j.m <= 256 ? 3 : j.m <= 512 ? 4 : j.m <= 1024 ? 5 : j.m <= 2048 ? 6 : 7].push_back(a);
    }
    all.push_back(a);
  }
  for (size_t i0 = 0; i0 < all.size(); i0 += kMaxBatch) {
    const int nb = (int)std::min<size_t>(kMaxBatch, all.size() - i0);
    Pack<FqArgs> pk{};
    int gx = 1;
    for (int i = 0; i < nb; ++i) {
      pk.a[i] = all[i0 + i];
      gx = std::max(gx, (pk.a[i].p + kFB - 1) / kFB);
    }
    VP_TRY((launch_after(ctx, "formq_prep", kb_formq_prep, dim3(gx, nb), dim3(256), 0, st, kNoCluster, pk)));
  }
  VP_TRY((launch_formq<1, 1, 4>(ctx, st, by[0])));
  VP_TRY((launch_formq<1, 2, 4>(ctx, st, by[1])));
  VP_TRY((launch_formq<1, 4, 4>(ctx, st, by[2])));
  VP_TRY((launch_formq<2, 4, 4>(ctx, st, by[3])));
  VP_TRY((launch_formq<2, 8, 4>(ctx, st, by[4])));
  VP_TRY((launch_formq<4, 8, 4>(ctx, st, by[5])));
  VP_TRY((launch_formq<8, 8, 2>(ctx, st, by[6])));
  VP_TRY((launch_formq<16, 8, 1>(ctx, st, by[7])));
  for (size_t i0 = 0; i0 < beyond.size(); i0 += kMaxBatch) {
    const int nb = (int)std::min<size_t>(kMaxBatch, beyond.size() - i0);
    Pack<FqArgs> pk{};
    int gx = 1;
    for (int i = 0; i < nb; ++i) {
      pk.a[i] = beyond[i0 + i];
      gx = std::max(gx, (pk.a[i].p + 7) / 8);
    }
    VP_TRY((launch_after(ctx, "formq_long", kb_formq_long, dim3(gx, nb), dim3(256), 0, st, kNoCluster, pk)));
  }
  return VP_OK;
}

}  // namespace vp
