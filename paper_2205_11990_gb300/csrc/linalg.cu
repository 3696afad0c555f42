// FP64 dense linear algebra of the compression sweeps (SI "Canonicalization and
// Compression"): Householder QR, explicit Q, GEMM, one-sided Jacobi SVD and the
// truncation rule of the truncation-error equation (main text, "MPS
// Representation"): the choice between their kernels, the small ones, and the FP64
// and grid kernels of what the others do not take (panel QR: qrpanel.cu, Q:
// formq.cu, block Jacobi: jacobi.cu, contractions: fgemm.cu, ozgemm.cu, tcgemm.cu).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>

#include <cooperative_groups.h>
#include <cuda/atomic>

#include "common.cuh"
#include "dw.cuh"

namespace cg = cooperative_groups;

namespace vp {

// ------------------------------------------------------------------ helpers
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Sum over the block; every thread receives the result.  `red` holds kWarps+1.
__device__ __forceinline__ double block_sum(double v, double* red) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  v = warp_sum(v);
  __syncthreads();
  if (lane == 0) red[warp] = v;
  __syncthreads();
  if (warp == 0) {
    double t = lane < kWarps ? red[lane] : 0.0;
    t = warp_sum(t);
    if (lane == 0) red[kWarps] = t;
  }
  __syncthreads();
  return red[kWarps];
}

__device__ __forceinline__ int ld_volatile(const int* p) { return *(const volatile int*)p; }

// Grid-wide barrier for cooperative launches: one monotonic 64-bit arrival
// counter, a release add per block and acquire polling (no reset, no
// generation word).  Every block starts from the counter value the previous
// cooperative kernel left in bar_base.  Waits have a clock limit
// (DevStatus::wait_clocks, ~1 s by default): on expiry the block records
// err = 1 and the barrier reports failure, so the kernel returns instead of
// hanging.
struct GridSync {
  DevStatus* st;
  unsigned nb;
  unsigned long long target;
  __device__ GridSync(DevStatus* s, unsigned n) : st(s), nb(n), target(0) {
    if (nb > 1) target = *(volatile unsigned long long*)&st->bar_base;
  }
  __device__ bool sync() {
    __syncthreads();
    if (nb > 1) {
      target += nb;
      if (threadIdx.x == 0) {
        cuda::atomic_ref<unsigned long long, cuda::thread_scope_device> cnt(st->bar_count);
        cnt.fetch_add(1ull, cuda::memory_order_release);
        const long long t0 = clock64(), limit = *(volatile long long*)&st->wait_clocks;
        while (cnt.load(cuda::memory_order_acquire) < target) {
          if (ld_volatile(&st->err) != 0) break;
          if (clock64() - t0 > limit) {
            atomicExch(&st->err, 1);
            break;
          }
        }
      }
      __syncthreads();
    }
    return ld_volatile(&st->err) == 0;
  }
  // Called by every block after its last sync(); block 0 publishes the base.
  __device__ void finish() {
    if (nb > 1 && blockIdx.x == 0 && threadIdx.x == 0) st->bar_base = target;
  }
};

static int coop_launch(vp_ctx* ctx, cudaStream_t stream, const void* fn, int blocks, int threads, void** args,
                       size_t smem, const char* what) {
  ctx->launches++;
  cudaError_t e = cudaLaunchCooperativeKernel(fn, dim3(blocks), dim3(threads), args, smem, stream);
  if (e != cudaSuccess) return cuda_fail(ctx, e, what);
  return VP_OK;
}

// ------------------------------------------------------- strided gathers
// A (m x n, column-major) from its source (QRSrc), through 32 x 32 tiles: the
// kernels that do not read a source themselves.
__device__ __forceinline__ void gather_tile(const QRSrc& s, int m, int n, double* __restrict__ A, int bx, int by) {
  __shared__ double tile[32][33];
  const int i0 = by * 32, k0 = bx * 32;
  if (i0 >= m || k0 >= n) return;  // the whole block is outside this problem
  const bool along_k = s.cs == 1;  // lanes along the contiguous direction
  for (int y = threadIdx.y; y < 32; y += 8) {
    const int i = along_k ? i0 + y : i0 + threadIdx.x, k = along_k ? k0 + threadIdx.x : k0 + y;
    if (i < m && k < n) {
      const int c = s.perm ? s.perm[k] : k;
      const double v = s.lower && i < c ? 0.0 : s.p[i * s.rs + c * s.cs];
      tile[i - i0][k - k0] = v;
    }
  }
  __syncthreads();
  for (int y = threadIdx.y; y < 32; y += 8) {
    const int k = k0 + y, i = i0 + threadIdx.x;
    if (i < m && k < n) A[(size_t)k * m + i] = tile[threadIdx.x][y];
  }
}
__global__ void kb_gather(const __grid_constant__ Pack<BGather> pk) {
  follow();
  const BGather& a = pk.a[blockIdx.z];
  gather_tile(a.src, a.m, a.n, a.A, blockIdx.x, blockIdx.y);
}
static int blaunch_gather(vp_ctx* ctx, cudaStream_t st, const std::vector<BGather>& v) {
  for (size_t i0 = 0; i0 < v.size(); i0 += kMaxBatch) {
    const int nb = (int)std::min<size_t>(kMaxBatch, v.size() - i0);
    Pack<BGather> pk{};
    int gx = 1, gy = 1;
    for (int i = 0; i < nb; ++i) {
      pk.a[i] = v[i0 + i];
      gx = std::max(gx, (v[i0 + i].n + 31) / 32);
      gy = std::max(gy, (v[i0 + i].m + 31) / 32);
    }
    VP_TRY((launch_after(ctx, "gather", kb_gather, dim3(gx, gy, nb), dim3(32, 8), 0, st, kNoCluster, pk)));
  }
  return VP_OK;
}
// Row-major (m x n) -> column-major copy.
int launch_to_colmajor(vp_ctx* ctx, const double* A, int m, int n, double* out) {
  QRSrc s;
  s.p = A;
  s.rs = n;
  s.cs = 1;
  return blaunch_gather(ctx, ctx->stream, {BGather{s, m, n, out}});
}

// ------------------------------------------------------------ Householder QR
// Column-cyclic ownership: column k belongs to block k % gridDim.x.  Step j:
// the owner of column j (already updated by H_0..H_{j-1}, which it applied
// itself) forms the reflector H_j = I - tau v v^T (LAPACK dlarfg convention,
// v_j = 1) and publishes v in a double buffer; after one grid barrier every
// block applies H_j to the columns it owns.  One barrier per column.
template <class Sync>
__global__ void __launch_bounds__(kThreads) k_qr_factor(double* A, int m, int n, double* tau,
                                                        double* vbuf, DevStatus* st) {
  __shared__ double red[kWarps + 1];
  const int nb = gridDim.x, bid = blockIdx.x;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int p = min(m, n);
  Sync gs(st, nb);
  for (int j = 0; j < p; ++j) {
    __syncthreads();
    double* vj = vbuf + (size_t)(j & 1) * m;
    if (bid == j % nb) {
      double* col = A + (size_t)j * m;
      double s = 0.0;
      for (int i = j + 1 + threadIdx.x; i < m; i += kThreads) {
        const double x = col[i];
        s = fma(x, x, s);
      }
      s = block_sum(s, red);
      const double x0 = col[j];
      double t = 0.0, beta = x0, scale = 0.0;
      if (s > 0.0) {
        const double nrm = sqrt(fma(x0, x0, s));
        beta = x0 >= 0.0 ? -nrm : nrm;
        t = (beta - x0) / beta;
        scale = 1.0 / (x0 - beta);
      }
      for (int i = j + 1 + threadIdx.x; i < m; i += kThreads) {
        const double v = col[i] * scale;
        col[i] = v;
        __stcg(vj + i, v);
      }
      if (threadIdx.x == 0) {
        col[j] = beta;
        __stcg(vj + j, 1.0);
        __stcg(tau + j, t);
      }
      __threadfence();
    }
    if (!gs.sync()) return;
    const double t = __ldcg(tau + j);
    if (t == 0.0) continue;
    // first owned column strictly right of j
    const int k0 = (j + 1) + ((bid - (j + 1) % nb) % nb + nb) % nb;
    for (int k = k0 + warp * nb; k < n; k += kWarps * nb) {
      double* col = A + (size_t)k * m;
      double w = 0.0;
      for (int i = j + lane; i < m; i += 32) w = fma(__ldcg(vj + i), col[i], w);
      w = warp_sum(w) * t;
      for (int i = j + lane; i < m; i += 32) col[i] = fma(-w, __ldcg(vj + i), col[i]);
    }
  }
  gs.finish();
}

// Look-ahead QR for the cooperative grid (factors too large for one cluster):
// no grid barrier.  Reflector j is published as double words in V (column j,
// V[j][j] = 1) and T[j] by a release store of a monotonic counter; at step j
// every block waits only for reflector j.  In the owner of column j+1, warp
// 0 applies H_j to that column, forms and publishes reflector j+1 while the
// other warps apply H_j to the rest of the block's columns; the counter base
// carries over between launches (the last block to finish records it).  The
// block's columns are held as double-word values (dw.cuh) in shared memory
// (in global scratch when they do not fit), the arithmetic on the FP32 pipe.
// Column k is scaled by 2^-e_k on load (A D = Q (R D): only R changes, and
// is unscaled on store); each reflector is formed on its column rescaled by
// a further power of two (v and tau do not depend on the scale), so no
// square leaves the FP32 range.  The output A, tau is the FP64 LAPACK layout
// of k_qr_factor.
// nb blocks factor the matrix, this block is number bid of them.
__device__ __forceinline__ void qr_factor_dw_body(double* A, int m, int n, double* tau, dw* V, dw* T, dw* gcols,
                                                  int* gexp, DevStatus* st, const int nb, const int bid) {
  extern __shared__ dw cols_sm[];
  __shared__ int s_ok;
  const int tid = threadIdx.x;
  const int lane = tid & 31, warp = tid >> 5;
  const int p = min(m, n);
  const int nown = bid < n ? (n - bid + nb - 1) / nb : 0;
  const int nmax = (n + nb - 1) / nb;
  // the block's columns (and their scale exponents) in shared memory, or in
  // global scratch (gcols, gexp: column k at k m) when they do not fit
  dw* cols = gcols ? gcols + (size_t)bid * m : cols_sm;
  const size_t cstride = gcols ? (size_t)nb * m : (size_t)m;
  int* cexp = gcols ? gexp + bid : reinterpret_cast<int*>(cols_sm + (size_t)nmax * m);
  const int estride = gcols ? nb : 1;
  const unsigned long long base = *(volatile unsigned long long*)&st->pub_base;
  cuda::atomic_ref<unsigned long long, cuda::thread_scope_device> pub(st->pub_count);

  // load the owned columns (k = bid + lc nb), each scaled by a power of two
  for (int lc = warp; lc < nown; lc += kWarps) {
    const double* a = A + (size_t)(bid + lc * nb) * m;
    float mx = 0.f;
    for (int i = lane; i < m; i += 32) mx = fmaxf(mx, fabsf(__double2float_rn(a[i])));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    int e = 0;
    if (mx > 0.f) frexpf(mx, &e);
    if (lane == 0) cexp[lc * estride] = e;
    const double sc = ldexp(1.0, -e);
    dw* c = cols + (size_t)lc * cstride;
    for (int i = lane; i < m; i += 32) c[i] = dw_from(a[i] * sc);
  }
  __syncthreads();

  // H_j applied to a local column by one warp: c -= (t (v . c)) v, rows >= j
  auto apply = [&](int j, dw* c) {
    const dw* v = V + (size_t)j * m;
    const float2 t2 = __ldcg(reinterpret_cast<const float2*>(T + j));
    const dw t = {t2.x, t2.y};
    dw_acc acc;
    for (int i = j + lane; i < m; i += 32) {
      const float2 vv = __ldcg(reinterpret_cast<const float2*>(v + i));
      dw_dot_step(acc, {vv.x, vv.y}, c[i]);
    }
    const dw w = dw_mul(dw_warp_sum(dw_acc_value(acc)), t);
    if (w.hi == 0.f) return;
    for (int i = j + lane; i < m; i += 32) {
      const float2 vv = __ldcg(reinterpret_cast<const float2*>(v + i));
      c[i] = dw_add(c[i], dw_neg(dw_mul(w, {vv.x, vv.y})));
    }
  };
  // the critical chain of column j (one warp of its owner): H_{j-1}, then
  // reflector j formed, stored locally and published
  auto critical = [&](int j) {
    dw* c = cols + (size_t)(j / nb) * cstride;
    if (j > 0) apply(j - 1, c);
    __syncwarp();
    float mx = 0.f;
    for (int i = j + lane; i < m; i += 32) mx = fmaxf(mx, fabsf(c[i].hi));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    int e = 0;
    if (mx > 0.f) frexpf(mx, &e);
    dw_acc acc;
    for (int i = j + 1 + lane; i < m; i += 32) {
      const dw x = dw_ldexp(c[i], -e);
      dw_dot_step(acc, x, x);
    }
    const dw s = dw_warp_sum(dw_acc_value(acc));
    const dw x0 = dw_ldexp(c[j], -e);
    dw t = {0.f, 0.f}, beta = x0, scale = {0.f, 0.f};
    if (s.hi > 0.f) {
      const dw nrm = dw_sqrt(dw_add(dw_mul(x0, x0), s));
      beta = x0.hi >= 0.f ? dw_neg(nrm) : nrm;
      t = dw_div(dw_add(beta, dw_neg(x0)), beta);
      scale = dw_div({1.0f, 0.0f}, dw_add(x0, dw_neg(beta)));
    }
    dw* v = V + (size_t)j * m;
    for (int i = j + 1 + lane; i < m; i += 32) {
      const dw vi = dw_mul(dw_ldexp(c[i], -e), scale);
      c[i] = vi;
      __stcg(reinterpret_cast<float2*>(v + i), make_float2(vi.hi, vi.lo));
    }
    __syncwarp();
    if (lane == 0) {
      c[j] = dw_ldexp(beta, e);
      __stcg(reinterpret_cast<float2*>(v + j), make_float2(1.0f, 0.0f));
      __stcg(reinterpret_cast<float2*>(T + j), make_float2(t.hi, t.lo));
      tau[j] = dw_to(t);
    }
    __threadfence();
    __syncwarp();
    if (lane == 0) pub.store(base + j + 1, cuda::memory_order_release);
  };
  auto wait = [&](int j) -> bool {
    if (tid == 0) {
      int ok = 1;
      const long long t0 = clock64(), limit = *(volatile long long*)&st->wait_clocks;
      while (pub.load(cuda::memory_order_acquire) < base + j + 1) {
        if (ld_volatile(&st->err) != 0) {
          ok = 0;
          break;
        }
        if (clock64() - t0 > limit) {
          atomicExch(&st->err, 1);
          ok = 0;
          break;
        }
      }
      s_ok = ok;
    }
    __syncthreads();
    return s_ok != 0;
  };

  if (bid == 0 && warp == 0) critical(0);
  bool ok = true;
  for (int j = 0; j < p; ++j) {
    if (!wait(j)) {
      ok = false;
      break;
    }
    const bool owner = j + 1 < p && bid == (j + 1) % nb;
    if (owner && warp == 0) {
      critical(j + 1);
      continue;
    }
    const int wk = owner ? warp - 1 : warp, nwk = owner ? kWarps - 1 : kWarps;
    // owned columns k >= j + 2: local index lc with bid + lc nb >= j + 2
    const int lc0 = (j + 2 - bid + nb - 1) / nb > 0 ? (j + 2 - bid + nb - 1) / nb : 0;
    for (int lc = lc0 + wk; lc < nown; lc += nwk) apply(j, cols + (size_t)lc * cstride);
  }
  __syncthreads();
  // store: R part unscaled by 2^e_k, reflectors (below the diagonal of the
  // first p columns) as they are
  for (int lc = warp; lc < nown; lc += kWarps) {
    const int k = bid + lc * nb;
    const double sc = ldexp(1.0, cexp[lc * estride]);
    const dw* c = cols + (size_t)lc * cstride;
    double* a = A + (size_t)k * m;
    for (int i = lane; i < m; i += 32) a[i] = (k < p && i > k) ? dw_to(c[i]) : dw_to(c[i]) * sc;
  }
  __syncthreads();
  if (tid == 0 && ok) {
    __threadfence();
    if (atomicAdd(&st->pub_done, 1u) == (unsigned)nb - 1) {
      st->pub_base = base + p;
      st->pub_done = 0u;
      __threadfence();
    }
  }
}

__global__ void __launch_bounds__(kThreads) k_qr_factor_dw(double* A, int m, int n, double* tau, dw* V, dw* T,
                                                          dw* gcols, int* gexp, DevStatus* st) {
  qr_factor_dw_body(A, m, n, tau, V, T, gcols, gexp, st, gridDim.x, blockIdx.x);
}

// Which kernel factors an m x n matrix.  Factors more than twice as wide as
// tall: the m reflectors depend on the leading m columns alone, so that square
// block (contiguous in the column-major layout) is factored in place, Q is
// formed from its reflectors, and the rest of R is one FP64 GEMM, R2 = Q^T A2
// (stored as R2^T = A2^T Q, which is A2's column-major layout), instead of
// applying every reflector to all n columns.  Not where one block or a cluster
// applies a panel to all of them in one pass, two columns a warp: those six launches
// then cost more (us, this way / the panel QR: 4 x 32 53 / 25, 16 x 128 63 / 46, 32 x
// 384 80 / 51; but 64 x 3392 198 / 355, 128 x 1696 332 / 436).  Otherwise the panel
// QR; what has more rows than its panel holds in registers goes to the grid kernel.  The
// choice depends on the shape and the device only, so that results do not depend
// on the context or on the batch.
QRPlan qr_plan(const vp_ctx* ctx, int m, int n) {
  if (std::min(m, n) <= 0) return {QR_NONE, {}};
  const PanelPlan pl = qr_panel_plan(ctx, m, n);
  const bool one_pass = pl.kind == PANEL_SOLO || (pl.kind == PANEL_CLUSTER && n <= 32 * (pl.cs - 1));
  if (n > 2 * m && m >= 2 && !one_pass) return {QR_WIDE, {}};
  if (pl.kind != PANEL_NONE) return {QR_PANEL, pl};
  return {QR_GRID, {}};
}

// The cooperative grid kernels, for factors beyond a cluster's shared memory:
// enough blocks that each owns a few columns, never more than one per SM.
// st, qrv, qrc: the status words and scratch of the caller (context or batch
// problem).
int qr_factor_grid(vp_ctx* ctx, cudaStream_t stream, DevStatus* st, DevBuf& qrv, DevBuf& qrc, double* A, int m,
                   int n, double* tau, double* vbuf) {
  const int p = std::min(m, n);
  const int cap = ctx->coop_cap > 0 ? std::min(ctx->coop_cap, ctx->num_sms) : ctx->num_sms;
  const int blocks = std::min(cap, std::max(1, n / 2));
  if (blocks > 1) {
    // the same double-word arithmetic whichever the storage, so that the
    // result does not depend on the context's block cap
    const int nmax = (n + blocks - 1) / blocks;
    const size_t smem = (size_t)nmax * m * sizeof(dw) + (size_t)nmax * sizeof(int);
    static AttrOnce qattr;
    VP_TRY(qattr.ensure(ctx, (const void*)k_qr_factor_dw, 200 * 1024, false));
    VP_TRY(reserve(ctx, qrv, (size_t)m * p + p + 8));
    dw* V = reinterpret_cast<dw*>(qrv.p);
    dw* T = V + (size_t)m * p;
    dw* gcols = nullptr;
    int* gexp = nullptr;
    size_t dyn = smem;
    if (smem > 200 * 1024) {
      VP_TRY(reserve(ctx, qrc, (size_t)m * n + n / 2 + 8));
      gcols = reinterpret_cast<dw*>(qrc.p);
      gexp = reinterpret_cast<int*>(gcols + (size_t)m * n);
      dyn = 0;
    }
    void* args[] = {&A, &m, &n, &tau, &V, &T, &gcols, &gexp, &st};
    return coop_launch(ctx, stream, (const void*)k_qr_factor_dw, blocks, kThreads, args, dyn, "qr_factor_dw");
  }
  void* args[] = {&A, &m, &n, &tau, &vbuf, &st};
  return coop_launch(ctx, stream, (const void*)k_qr_factor<GridSync>, blocks, kThreads, args, 0, "qr_factor");
}

int launch_qr_factor(vp_ctx* ctx, double* A, int m, int n, double* tau, double* vbuf, const QRSrc& src) {
  const QRPlan pl = qr_plan(ctx, m, n);
  if (src.p && (pl.kind == QR_WIDE || pl.kind == QR_GRID))
    VP_TRY(blaunch_gather(ctx, ctx->stream, {BGather{src, m, n, A}}));
  switch (pl.kind) {
    case QR_NONE:
      return VP_OK;
    case QR_WIDE: {
      VP_TRY(launch_qr_factor(ctx, A, m, m, tau, vbuf));
      VP_TRY(reserve(ctx, ctx->w_wq, (size_t)m * m));
      VP_TRY(launch_qr_formq(ctx, A, m, m, tau, ctx->w_wq.p));
      const size_t rest = (size_t)(n - m) * m;
      VP_TRY(reserve(ctx, ctx->w_wr, rest));
      const int prec = ctx->precision;  // R is part of the factorisation: FP64 in every mode
      ctx->precision = VP_PREC_FP64;
      const int st = launch_gemm(ctx, n - m, m, m, 1.0, A + (size_t)m * m, m, ctx->w_wq.p, m, ctx->w_wr.p, m, OZ_ROWS);
      ctx->precision = prec;
      VP_TRY(st);
      return launch_copy(ctx, ctx->w_wr.p, A + (size_t)m * m, rest);
    }
    case QR_PANEL:
      return blaunch_qr_panel(ctx, ctx->stream, {PanelJob{A, m, n, tau, pl.panel, src, &ctx->w_qrv, &ctx->w_qrc, ctx->status}});
    default:
      return qr_factor_grid(ctx, ctx->stream, ctx->status, ctx->w_qrv, ctx->w_qrc, A, m, n, tau, vbuf);
  }
}

int launch_qr_formq(vp_ctx* ctx, const double* A, int m, int n, const double* tau, double* Q, const int* rows) {
  return blaunch_formq(ctx, ctx->stream, {FormQJob{A, m, n, tau, Q, rows, &ctx->w_fq, &ctx->w_q}});
}

__device__ __forceinline__ void k_qr_getr_body(const double* __restrict__ A, int m, int n, int p, double* __restrict__ R) {
  const size_t total = (size_t)p * n;
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < total; e += (size_t)gridDim.x * blockDim.x) {
    const int j = (int)(e / n), k = (int)(e % n);
    R[e] = (j <= k) ? A[(size_t)k * m + j] : 0.0;
  }
}
__global__ void k_qr_getr(const double* __restrict__ A, int m, int n, int p, double* __restrict__ R) {
  follow();
  k_qr_getr_body(A, m, n, p, R); }

int launch_qr_getr(vp_ctx* ctx, const double* A, int m, int n, double* R) {
  const int p = std::min(m, n);
  const size_t total = (size_t)p * n;
  if (total == 0) return VP_OK;
  const int blocks = (int)std::min<size_t>((total + 255) / 256, (size_t)ctx->num_sms * 16);
  return launch_after(ctx, "qr_getr", k_qr_getr, dim3(blocks), dim3(256), 0, ctx->stream, kNoCluster, A, m, n, p, R);
}

// ------------------------------------------------------------------- GEMM
// The FP32 contraction mode: TILE x TILE output tile per block (64 or 32), K step
// 16, 256 threads with a (TILE / 16)^2 register tile each, inputs rounded to FP32
// and FP32 FMA (FP64 contractions: fgemm.cu, ozgemm.cu).  ALoad selects the A
// operand: row-major, or the column-major upper triangle of a QR factor.  Each
// output is the sum over its K slice in ascending k; the K slicing is gemm_plan's.
// kfirst(row0): the first k that can be nonzero in rows >= row0.
struct ARowMajor {
  const double* A;
  int lda;
  __device__ double operator()(int r, int k) const { return A[(size_t)r * lda + k]; }
  __device__ int kfirst(int) const { return 0; }
};
struct AUpperColMajor {
  const double* A;
  int lda;
  __device__ double operator()(int r, int k) const { return r <= k ? A[(size_t)k * lda + r] : 0.0; }
  __device__ int kfirst(int row0) const { return row0; }  // R[r][k] = 0 for k < r
};

// blockIdx.z selects a K slice of `kslice` columns (split-K); slice s writes
// its partial product to C + s * slice_stride.
// B operand: row-major (K x N), or given as its transpose (N x K row-major).
struct BRowMajor {
  const double* B;
  int ldb;
  __device__ double operator()(int k, int n) const { return B[(size_t)k * ldb + n]; }
};
struct BTransposed {
  const double* B;
  int ldb;
  __device__ double operator()(int k, int n) const { return B[(size_t)n * ldb + k]; }
};

template <class ALoad, class BLoad, int TILE>
__device__ __forceinline__ void gemm_body(int M, int N, int K, double alpha, ALoad a, BLoad bl, double* __restrict__ C,
                                          int ldc, int kslice, size_t slice_stride, int bx, int by, int bz) {
  constexpr int R = TILE / 16;  // outputs per thread along each dimension
  using T = float;
  __shared__ T As[16][TILE + 1];
  __shared__ T Bs[16][TILE];
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  const int row0 = bx * TILE, col0 = by * TILE;
  // the terms below the triangle of an upper-triangular A are exact zeros:
  // starting past them leaves every output's sum unchanged
  const int kbeg = max(bz * kslice, a.kfirst(row0)), kend = min(K, bz * kslice + kslice);
  C += bz * slice_stride;
  T acc[R][R] = {};
  for (int k0 = kbeg; k0 < kend; k0 += 16) {
    for (int e = threadIdx.x; e < TILE * 16; e += 256) {
      const int r = e / 16, kk = e % 16;
      const int gr = row0 + r, gk = k0 + kk;
      As[kk][r] = (T)((gr < M && gk < kend) ? a(gr, gk) : 0.0);
    }
    for (int e = threadIdx.x; e < 16 * TILE; e += 256) {
      const int kk = e / TILE, c = e % TILE;
      const int gk = k0 + kk, gc = col0 + c;
      Bs[kk][c] = (T)((gk < kend && gc < N) ? bl(gk, gc) : 0.0);
    }
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < 16; ++kk) {
      T av[R], bv[R];
#pragma unroll
      for (int i = 0; i < R; ++i) av[i] = As[kk][ty + 16 * i];
#pragma unroll
      for (int i = 0; i < R; ++i) bv[i] = Bs[kk][tx + 16 * i];
#pragma unroll
      for (int i = 0; i < R; ++i)
#pragma unroll
        for (int jj = 0; jj < R; ++jj) acc[i][jj] = fma(av[i], bv[jj], acc[i][jj]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < R; ++i) {
    const int r = row0 + ty + 16 * i;
    if (r >= M) continue;
#pragma unroll
    for (int jj = 0; jj < R; ++jj) {
      const int c = col0 + tx + 16 * jj;
      if (c < N) C[(size_t)r * ldc + c] = alpha * (double)acc[i][jj];
    }
  }
}

template <class ALoad, class BLoad, int TILE>
__global__ void __launch_bounds__(256) k_gemm(int M, int N, int K, double alpha, ALoad a, BLoad bl,
                                              double* __restrict__ C, int ldc, int kslice, size_t slice_stride) {
  gemm_body<ALoad, BLoad, TILE>(M, N, K, alpha, a, bl, C, ldc, kslice, slice_stride, blockIdx.x, blockIdx.y,
                                   blockIdx.z);
}

// How an FP32 contraction is spread over the SMs: 64 x 64 tiles when they alone
// give every SM a block, else 32 x 32 tiles, and K split into slices (multiples of
// 16, at most 32) until there are about two blocks per SM; the slices' partial
// products are summed in a fixed order.  Shape and device only, so a GEMM gives
// the same bits alone, in a batch or in a group.
GemmPlan gemm_plan(const vp_ctx* ctx, int M, int N, int K) {
  GemmPlan g{64, 1, K};
  const int t64 = ((M + 63) / 64) * ((N + 63) / 64);
  if (t64 >= ctx->num_sms || K <= 16) return g;
  int tiles = t64;
  if (2 * t64 < ctx->num_sms) {
    g.tile = 32;
    tiles = ((M + 31) / 32) * ((N + 31) / 32);
  }
  const int target = 2 * ctx->num_sms;
  if (tiles >= target) return g;
  const int sl = std::min(std::min((target + tiles - 1) / tiles, K / 16), 32);
  if (sl <= 1) return g;
  const int ks = ((K + sl - 1) / sl + 15) / 16 * 16;
  g.kslice = ks;
  g.slices = (K + ks - 1) / ks;
  if (g.slices <= 1) g.kslice = K;
  return g;
}

// Sum of `slices` partial products (fixed order: deterministic).
__device__ __forceinline__ void k_sum_slices_body(const double* __restrict__ P, int M, int N, int slices, size_t stride, double* C,
                             int ldc) {
  const size_t total = (size_t)M * N;
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < total; e += (size_t)gridDim.x * blockDim.x) {
    double acc = 0.0;
    for (int s = 0; s < slices; ++s) acc += P[s * stride + e];
    C[(e / N) * ldc + e % N] = acc;
  }
}
__global__ void k_sum_slices(const double* __restrict__ P, int M, int N, int slices, size_t stride, double* C,
                             int ldc) {
  follow();
  k_sum_slices_body(P, M, N, slices, stride, C, ldc);
}

// The same operands as (row, k) maps for the tensor-core path.
static TcOperand tc_a(const ARowMajor& a) { return {a.A, a.lda, 0}; }
static TcOperand tc_a(const AUpperColMajor& a) { return {a.A, a.lda, 2}; }
static TcOperand tc_b(const BRowMajor& b) { return {b.B, b.ldb, 1}; }
static TcOperand tc_b(const BTransposed& b) { return {b.B, b.ldb, 0}; }

static OzGemm oz_job(const TcOperand& a, const TcOperand& b, int M, int N, int K, double alpha, double* C, int ldc,
                     DevBuf* wa, DevBuf* wb, DevBuf* wsum, DevStatus* st, const OzPlan& plan, OzBound bound) {
  OzGemm g;
  g.a = a;
  g.b = b;
  g.M = M;
  g.N = N;
  g.K = K;
  g.alpha = alpha;
  g.C = C;
  g.ldc = ldc;
  g.wa = wa;
  g.wb = wb;
  g.wsum = wsum;
  g.stride = 0;
  g.st = st;
  g.plan = plan;
  g.bound = bound;
  return g;
}

// One GEMM: FP64 by oz_plan and fma_plan; FP32 split over K per gemm_plan, then the
// fixed-order slice sum.
template <class ALoad, class BLoad>
static int gemm_dispatch(vp_ctx* ctx, int M, int N, int K, double alpha, ALoad a, BLoad b, double* C, int ldc,
                         const char* what, OzBound bound) {
  if (M <= 0 || N <= 0) return VP_OK;
  if (ctx->precision >= VP_PREC_TF32 && K > 0) return launch_tc_gemm(ctx, M, N, K, alpha, tc_a(a), tc_b(b), C, ldc);
  if (ctx->precision == VP_PREC_FP64) {
    const OzPlan oz = oz_plan(ctx, M, N, K);
    const std::vector<OzGemm> job{
        oz_job(tc_a(a), tc_b(b), M, N, K, alpha, C, ldc, &ctx->w_tca, &ctx->w_tcb, &ctx->w_split, ctx->status, oz, bound)};
    return oz.use ? blaunch_oz_gemm(ctx, ctx->stream, job) : blaunch_fma_gemm(ctx, ctx->stream, job);
  }
  const GemmPlan pl = gemm_plan(ctx, M, N, K);
  dim3 grid((M + pl.tile - 1) / pl.tile, (N + pl.tile - 1) / pl.tile, 1);
  if (grid.y > 65535) return fail(ctx, VP_ECAPACITY, "gemm: N too large");
  // FP32 contraction mode: inputs rounded to FP32, FP32 FMA and accumulation
  auto kern = pl.tile == 64 ? k_gemm<ALoad, BLoad, 64> : k_gemm<ALoad, BLoad, 32>;
  int slices = pl.slices;
  const int kslice = pl.kslice;
  if (slices <= 1) {
    ctx->launches++;
    kern<<<grid, 256, 0, ctx->stream>>>(M, N, K, alpha, a, b, C, ldc, K, 0);
    return check_launch(ctx, what);
  }
  const size_t stride = (size_t)M * N;
  VP_TRY(reserve(ctx, ctx->w_split, stride * slices));
  grid.z = slices;
  ctx->launches += 2;
  kern<<<grid, 256, 0, ctx->stream>>>(M, N, K, alpha, a, b, ctx->w_split.p, N, kslice, stride);
  VP_TRY(check_launch(ctx, what));
  const int blocks = (int)std::min<size_t>((stride + 255) / 256, (size_t)ctx->num_sms * 8);
  return launch_after(ctx, what, k_sum_slices, dim3(blocks), dim3(256), 0, ctx->stream, kNoCluster, ctx->w_split.p,
                      M, N, slices, stride, C, ldc);
}

int launch_gemm(vp_ctx* ctx, int M, int N, int K, double alpha, const double* A, int lda, const double* B,
                int ldb, double* C, int ldc, OzBound bound) {
  return gemm_dispatch(ctx, M, N, K, alpha, ARowMajor{A, lda}, BRowMajor{B, ldb}, C, ldc, "gemm", bound);
}

int launch_gemm_bt(vp_ctx* ctx, int M, int N, int K, const double* A, int lda, const double* Bt, int ldbt, double* C,
                   int ldc, OzBound bound) {
  return gemm_dispatch(ctx, M, N, K, 1.0, ARowMajor{A, lda}, BTransposed{Bt, ldbt}, C, ldc, "gemm_bt", bound);
}

int launch_gemm_r(vp_ctx* ctx, int M, int N, int K, const double* Acm, int lda, const double* B, int ldb,
                  double* C, int ldc) {
  return gemm_dispatch(ctx, M, N, K, 1.0, AUpperColMajor{Acm, lda}, BRowMajor{B, ldb}, C, ldc, "gemm_r", OZ_COLS);
}

// ------------------------------------------------------------ Jacobi SVD
// One-sided (Hestenes) Jacobi on the rows of X: rotate row pairs until all
// are mutually orthogonal; then X = diag(s) V^T.  Round-robin ("circle") ordering: b' - 1
// rounds of b'/2 disjoint pairs per sweep, one warp per pair, one grid
// barrier per round.
__device__ __forceinline__ int rr_index(int pos, int round, int bp) {
  return pos == 0 ? 0 : 1 + (pos - 1 + round) % (bp - 1);
}

// Plane rotation that zeroes the Gram entry gamma of a row pair with squared
// norms alpha, beta: tan(theta) = t is the smaller root of
// t^2 + 2 t d / gamma - 1 = 0, d = (beta - alpha) / 2, written without the
// quotient d / gamma as t = sign(d) gamma / (|d| + sqrt(d^2 + gamma^2)); then
// cos = 1 / sqrt(1 + t^2), sin = t cos.  Three long-latency operations.
__device__ __forceinline__ void jacobi_rotation(double al, double be, double ga, double& t, double& cs, double& sn) {
  const double d = 0.5 * (be - al);
  t = copysign(1.0, d) * ga / (fabs(d) + sqrt(fma(d, d, ga * ga)));
  cs = rsqrt(fma(t, t, 1.0));
  sn = cs * t;
}

__global__ void __launch_bounds__(kThreads) k_jacobi_rows(double* X, int b, int c, double eps,
                                                          int max_sweeps, DevStatus* st) {
  const int nb = gridDim.x;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int gw = blockIdx.x * kWarps + warp, nw = nb * kWarps;
  const int bp = b + (b & 1), npairs = bp / 2, rounds = bp - 1;
  int sweep = 0;
  bool converged = false;
  GridSync gs(st, nb);
  for (; sweep < max_sweeps; ++sweep) {
    unsigned* cnt = &st->rot[sweep % 3];
    if (blockIdx.x == 0 && threadIdx.x == 0) atomicExch(&st->rot[(sweep + 1) % 3], 0u);
    for (int round = 0; round < rounds; ++round) {
      for (int pr = gw; pr < npairs; pr += nw) {
        int i = rr_index(pr, round, bp), j = rr_index(bp - 1 - pr, round, bp);
        if (i >= b || j >= b) continue;
        if (i > j) {
          const int t = i;
          i = j;
          j = t;
        }
        double* xi = X + (size_t)i * c;
        double* xj = X + (size_t)j * c;
        double al = 0.0, be = 0.0, ga = 0.0;
        for (int q = lane; q < c; q += 32) {
          const double u = __ldcg(xi + q), v = __ldcg(xj + q);
          al = fma(u, u, al);
          be = fma(v, v, be);
          ga = fma(u, v, ga);
        }
        al = warp_sum(al);
        be = warp_sum(be);
        ga = warp_sum(ga);
        if (!(al > 0.0 && be > 0.0)) continue;
        if (!(ga * ga > eps * eps * al * be)) continue;
        double t, cs, sn;
        jacobi_rotation(al, be, ga, t, cs, sn);
        for (int q = lane; q < c; q += 32) {
          const double u = __ldcg(xi + q), v = __ldcg(xj + q);
          __stcg(xi + q, cs * u - sn * v);
          __stcg(xj + q, sn * u + cs * v);
        }
        if (lane == 0) atomicAdd(cnt, 1u);
      }
      if (!gs.sync()) return;
    }
    if (__ldcg(cnt) == 0u) {
      converged = true;
      break;
    }
  }
  gs.finish();
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    st->pad2 = sweep + 1;
    if (!converged) atomicCAS(&st->err, 0, 3);
  }
}

// Cluster-resident variant: the b rows of X (length c) live in the distributed
// shared memory of one thread-block cluster (row x in CTA x % CS, slot x / CS),
// one CTA per SM.  A pair is processed by one warp through
// DSMEM pointers; rounds are separated by the hardware cluster barrier
// (about 0.2 us on GB300, against 2 us for a grid-wide software barrier).
__global__ void __launch_bounds__(kThreads) k_jacobi_cluster(double* X, int b, int c, double eps,
                                                             int max_sweeps, DevStatus* st) {
  cg::cluster_group cl = cg::this_cluster();
  extern __shared__ double sm[];
  const int CS = (int)cl.num_blocks(), rank = (int)cl.block_rank();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int rpc = (b + CS - 1) / CS, stride = c;
  double* nrm = sm + (size_t)rpc * stride;                   // squared row norms, one per local row
  unsigned* cnt = reinterpret_cast<unsigned*>(nrm + rpc);
  for (int sl = 0; sl < rpc; ++sl) {
    const int x = sl * CS + rank;
    if (x >= b) break;
    double* row = sm + (size_t)sl * stride;
    for (int q = tid; q < c; q += kThreads) row[q] = X[(size_t)x * c + q];
  }
  if (tid < 4) cnt[tid] = 0u;
  unsigned* c0 = cl.map_shared_rank(cnt, 0);
  const int bp = b + (b & 1), npairs = bp / 2, rounds = bp - 1;
  int sweep = 0;
  bool converged = false;
  for (; sweep < max_sweeps; ++sweep) {
    // exact squared norms of the local rows once per sweep; a rotation then
    // updates them as alpha' = alpha - t gamma, beta' = beta + t gamma
    __syncthreads();
    for (int sl = warp; sl < rpc; sl += kWarps) {
      if (sl * CS + rank >= b) break;
      const double* row = sm + (size_t)sl * stride;
      double a = 0.0;
      for (int q = lane; q < c; q += 32) a = fma(row[q], row[q], a);
      a = warp_sum(a);
      if (lane == 0) nrm[sl] = a;
    }
    if (rank == 0 && tid == 0) cnt[(sweep + 1) % 3] = 0u;
    cl.sync();
    unsigned rotated = 0;
    for (int round = 0; round < rounds; ++round) {
      for (int pr = rank + warp * CS; pr < npairs; pr += CS * kWarps) {
        int i = rr_index(pr, round, bp), j = rr_index(bp - 1 - pr, round, bp);
        if (i >= b || j >= b) continue;
        if (i > j) {
          const int t = i;
          i = j;
          j = t;
        }
        double* xi = cl.map_shared_rank(sm + (size_t)(i / CS) * stride, i % CS);
        double* xj = cl.map_shared_rank(sm + (size_t)(j / CS) * stride, j % CS);
        double* ni = cl.map_shared_rank(nrm + i / CS, i % CS);
        double* nj = cl.map_shared_rank(nrm + j / CS, j % CS);
        const double al = *ni, be = *nj;
        double ga = 0.0;
        for (int q = lane; q < c; q += 32) ga = fma(xi[q], xj[q], ga);
        ga = warp_sum(ga);
        if (!(al > 0.0 && be > 0.0)) continue;
        if (!(ga * ga > eps * eps * al * be)) continue;
        double t, cs, sn;
        jacobi_rotation(al, be, ga, t, cs, sn);
        for (int q = lane; q < stride; q += 32) {
          const double u = xi[q], v = xj[q];
          xi[q] = cs * u - sn * v;
          xj[q] = sn * u + cs * v;
        }
        if (lane == 0) {
          *ni = fma(-t, ga, al);
          *nj = fma(t, ga, be);
        }
        ++rotated;
      }
      if (round == rounds - 1 && lane == 0 && rotated) atomicAdd(&c0[sweep % 3], rotated);
      cl.sync();
    }
    if (*(volatile unsigned*)&c0[sweep % 3] == 0u) {
      converged = true;
      break;
    }
  }
  for (int sl = 0; sl < rpc; ++sl) {
    const int x = sl * CS + rank;
    if (x >= b) break;
    const double* row = sm + (size_t)sl * stride;
    for (int q = tid; q < c; q += kThreads) X[(size_t)x * c + q] = row[q];
  }
  if (rank == 0 && tid == 0) {
    st->pad2 = sweep + 1;
    if (!converged) atomicCAS(&st->err, 0, 3);
  }
  cl.sync();  // keep every CTA's shared memory alive until all remote accesses are done
}

int probe_cluster_size() {
  if (cudaFuncSetAttribute(k_jacobi_cluster, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024) != cudaSuccess)
    return 0;
  cudaFuncSetAttribute(k_jacobi_cluster, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  for (int cs : {16, 8}) {
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[1];
    cfg.gridDim = dim3(cs);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = 120 * 1024;
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = cs;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, k_jacobi_cluster, &cfg) == cudaSuccess && n >= 1) return cs;
    cudaGetLastError();
  }
  return 0;
}

static size_t cluster_jacobi_smem(int b, int c, int CS) {
  const size_t rpc = (size_t)(b + CS - 1) / CS;
  return rpc * (size_t)(c + 1) * sizeof(double) + 4 * sizeof(unsigned);
}

// Block-local variant.  The b rows are split into 2 CS blocks of nb rows (nb
// even, padding rows zero); CTA c of a CS-CTA cluster holds two blocks, "top"
// and "bottom", in its own shared memory.  One block round rotates every
// pair between the two local blocks (nb inner rounds of nb disjoint pairs,
// separated by __syncthreads only); the first block round of a sweep also
// rotates the pairs inside each block.  Then the blocks move on the circle
// schedule (block positions 0..2CS-1, top of CTA c = c, bottom = 2CS-1-c;
// position 0 stays, every other position advances by one), by DSMEM copies
// into the other half of a double buffer and one cluster barrier.  After
// 2CS-1 block rounds every pair of rows has met once (one sweep) and every
// block is back home.
//
// Rotations are applied in scaled form: a row is stored as x~ with a scale
// d (x = d x~), its squared norm alpha kept beside it.  The rotation with
// tan t and cos c becomes x~_i <- x~_i - (t d_j / d_i) x~_j,
// x~_j <- x~_j + (t d_i / d_j) x~_i, d <- c d: two FMAs per element pair
// instead of four operations, with the same rounding bound.  Each sweep
// starts by folding d back into the rows and recomputing alpha exactly.
// Row layout (stride c + 2 doubles): x~ (c), alpha, d.
struct JacBlockCfg {
  int CS, nb, stride;
};

__device__ __forceinline__ int jac_pos_cta(int pos, int CS) { return pos < CS ? pos : 2 * CS - 1 - pos; }
__device__ __forceinline__ int jac_pos_slot(int pos, int CS) { return pos < CS ? 0 : 1; }
__device__ __forceinline__ int jac_next_pos(int pos, int CS) {
  return pos == 0 ? 0 : (pos == 2 * CS - 1 ? 1 : pos + 1);
}

// The pairs of one inner round are processed in three phases, because FP64
// issues at two lanes per clock per SM on GB300 and the scalar work of a
// rotation (threshold, square root, divisions) costs as much as a whole
// 128-element update when every warp repeats it:
//   A  one warp per pair: gamma~ = <x~_i, x~_j> (FMA + warp reduction);
//   B  one lane per pair (warp 0): threshold, rotation, new alpha and d, the
//      two update coefficients;
//   C  one warp per pair: x~_i -= a x~_j, x~_j += b x~_i.
// par[4 p + 0..3]: gamma~, a, b, rotate flag of pair p.
__device__ __forceinline__ void jac_dot(const double* ri, const double* rj, int c, int lane, double* par) {
  double g = 0.0;
  for (int q = lane; q < c; q += 32) g = fma(ri[q], rj[q], g);
  g = warp_sum(g);
  if (lane == 0) par[0] = g;
}

// Returns 1 when the pair is rotated.
__device__ __forceinline__ int jac_params(double* ri, double* rj, int w, double eps2, double* par) {
  double* ei = ri + w;  // alpha, d of row i
  double* ej = rj + w;
  const double al = ei[0], be = ej[0], di = ei[1], dj = ej[1];
  par[3] = 0.0;
  if (!(al > 0.0 && be > 0.0)) return 0;
  const double ga = di * dj * par[0];
  if (!(ga * ga > eps2 * al * be)) return 0;
  double t, cs, sn;
  jacobi_rotation(al, be, ga, t, cs, sn);
  const double inv = 1.0 / (di * dj);
  par[1] = t * dj * dj * inv;
  par[2] = t * di * di * inv;
  par[3] = 1.0;
  ei[0] = fma(-t, ga, al);
  ej[0] = fma(t, ga, be);
  ei[1] = cs * di;
  ej[1] = cs * dj;
  return 1;
}

__device__ __forceinline__ void jac_update(double* ri, double* rj, int w, int lane, const double* par) {
  if (par[3] == 0.0) return;
  const double a = par[1], bb = par[2];
  for (int q = lane; q < w; q += 32) {
    const double u = ri[q], v = rj[q];
    ri[q] = fma(-a, v, u);
    rj[q] = fma(bb, u, v);
  }
}

__global__ void __launch_bounds__(kThreads) k_jacobi_block(double* X, int b, int c, double eps,
                                                           int max_sweeps, int nb, DevStatus* st) {
  cg::cluster_group cl = cg::this_cluster();
  extern __shared__ double sm[];
  const int CS = (int)cl.num_blocks(), rank = (int)cl.block_rank();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int w = c, stride = w + 2;
  const size_t slot_sz = (size_t)nb * stride;
  // buffer set s, slot (0 top, 1 bottom), row r
  auto row = [&](int s, int slot, int r) { return sm + ((size_t)(s * 2 + slot)) * slot_sz + (size_t)r * stride; };
  double* par = sm + 4 * slot_sz;  // 4 doubles per pair of an inner round
  unsigned* cnt = reinterpret_cast<unsigned*>(par + 4 * nb);
  const double eps2 = eps * eps;
  // one inner round over nb disjoint pairs (rows given by pair_rows)
  auto inner_round = [&](auto pair_rows, unsigned& rotated) {
    for (int pi = warp; pi < nb; pi += kWarps) {
      double *ri, *rj;
      pair_rows(pi, ri, rj);
      jac_dot(ri, rj, c, lane, par + 4 * pi);
    }
    __syncthreads();
    if (warp == 0) {
      for (int pi = lane; pi < nb; pi += 32) {
        double *ri, *rj;
        pair_rows(pi, ri, rj);
        rotated += jac_params(ri, rj, w, eps2, par + 4 * pi);
      }
    }
    __syncthreads();
    for (int pi = warp; pi < nb; pi += kWarps) {
      double *ri, *rj;
      pair_rows(pi, ri, rj);
      jac_update(ri, rj, w, lane, par + 4 * pi);
    }
    __syncthreads();
  };

  // home placement: top = block rank, bottom = block 2 CS - 1 - rank
  for (int slot = 0; slot < 2; ++slot) {
    const int blk = slot == 0 ? rank : 2 * CS - 1 - rank;
    for (int r = 0; r < nb; ++r) {
      const int x = blk * nb + r;
      double* d = row(0, slot, r);
      for (int q = tid; q < stride; q += kThreads) {
        double v = 0.0;
        if (x < b) {
          if (q < c) v = X[(size_t)x * c + q];
        }
        if (q == w + 1) v = 1.0;  // scale d
        d[q] = v;
      }
    }
  }
  if (tid < 4) cnt[tid] = 0u;
  unsigned* c0 = cl.map_shared_rank(cnt, 0);
  int cur = 0, sweep = 0;
  bool converged = false;
  const int brounds = 2 * CS - 1;
  for (; sweep < max_sweeps; ++sweep) {
    // fold the scales into the rows, exact squared norms
    __syncthreads();
    for (int rr = warp; rr < 2 * nb; rr += kWarps) {
      double* d = row(cur, rr / nb, rr % nb);
      const double sc = d[w + 1];
      double a = 0.0;
      for (int q = lane; q < w; q += 32) {
        const double v = d[q] * sc;
        d[q] = v;
        if (q < c) a = fma(v, v, a);
      }
      a = warp_sum(a);
      __syncwarp();
      if (lane == 0) {
        d[w] = a;
        d[w + 1] = 1.0;
      }
    }
    if (rank == 0 && tid == 0) cnt[(sweep + 1) % 3] = 0u;
    cl.sync();
    unsigned rotated = 0;
    for (int br = 0; br < brounds; ++br) {
      if (br == 0) {
        // pairs inside each local block: round robin over nb rows
        for (int ir = 0; ir < nb - 1; ++ir)
          inner_round(
              [&](int pi, double*& ri, double*& rj) {
                const int slot = pi / (nb / 2), pos = pi % (nb / 2);
                ri = row(cur, slot, rr_index(pos, ir, nb));
                rj = row(cur, slot, rr_index(nb - 1 - pos, ir, nb));
              },
              rotated);
      }
      // pairs between the two local blocks
      for (int s = 0; s < nb; ++s)
        inner_round(
            [&](int pi, double*& ri, double*& rj) {
              ri = row(cur, 0, pi);
              rj = row(cur, 1, (pi + s) % nb);
            },
            rotated);
      if (br == brounds - 1 && warp == 0) {
        const unsigned tot = __reduce_add_sync(0xffffffffu, rotated);
        if (lane == 0 && tot) atomicAdd(&c0[sweep % 3], tot);
      }
      // move both blocks to their next positions (other half of the buffer)
      if (CS > 1) {
        for (int slot = 0; slot < 2; ++slot) {
          const int pos = slot == 0 ? rank : 2 * CS - 1 - rank;
          const int np = jac_next_pos(pos, CS);
          double* dst = cl.map_shared_rank(row(cur ^ 1, jac_pos_slot(np, CS), 0), jac_pos_cta(np, CS));
          const double* src = row(cur, slot, 0);
          for (size_t e = tid; e < slot_sz; e += kThreads) dst[e] = src[e];
        }
        cur ^= 1;
      }
      cl.sync();
    }
    if (*(volatile unsigned*)&c0[sweep % 3] == 0u) {
      converged = true;
      break;
    }
  }
  // blocks are home after a whole number of sweeps: write back x = d x~
  __syncthreads();
  for (int slot = 0; slot < 2; ++slot) {
    const int blk = slot == 0 ? rank : 2 * CS - 1 - rank;
    for (int r = 0; r < nb; ++r) {
      const int x = blk * nb + r;
      if (x >= b) continue;
      const double* d = row(cur, slot, r);
      const double sc = d[w + 1];
      for (int q = tid; q < c; q += kThreads) X[(size_t)x * c + q] = sc * d[q];
    }
  }
  if (rank == 0 && tid == 0) {
    st->pad2 = sweep + 1;
    if (!converged) atomicCAS(&st->err, 0, 3);
  }
  cl.sync();  // keep every CTA's shared memory alive until all remote accesses are done
}

static JacBlockCfg jac_block_cfg(int b, int c, int cs_max) {
  JacBlockCfg g{1, 2, 0};
  int cs = 1;
  while (cs < 16 && cs < cs_max && cs * 8 < b) cs *= 2;
  int nb = (b + 2 * cs - 1) / (2 * cs);
  nb += nb & 1;
  if (nb < 2) nb = 2;
  g.CS = cs;
  g.nb = nb;
  g.stride = c + 2;
  return g;
}

static size_t jac_block_smem(const JacBlockCfg& g) {
  return (4 * (size_t)g.nb * g.stride + 4 * (size_t)g.nb) * sizeof(double) + 4 * sizeof(unsigned);
}

int jacobi_rows_on(vp_ctx* ctx, cudaStream_t stream, DevStatus* status, const double* R, double* X, int b, double* norms,
                   bool floor_ok, bool* have_norms) {
  *have_norms = false;
  if (b <= 0) return VP_OK;
  const int CS = ctx->cluster_size;
  int c = b;
  if (floor_ok && jacobi_dw_fits(ctx, b)) {
    *have_norms = true;
    return blaunch_jacobi_dw(ctx, stream, {BJacobi{R, X, b, norms, status}});
  }
  VP_TRY(blaunch_qr_getr(ctx, stream, {BGetR{R, b, b, X}}));
  const JacBlockCfg bc = jac_block_cfg(b, c, std::max(1, CS));
  if (b > 1 && jac_block_smem(bc) <= 200 * 1024) {
    static AttrOnce battr_done;
    VP_TRY(battr_done.ensure(ctx, (const void*)k_jacobi_block, 200 * 1024, true));
    // one CTA per SM: the FP64 pipe of each SM is the limit
    const size_t smem = std::max<size_t>(jac_block_smem(bc), 120 * 1024);
    double eps = 1e-15 * std::sqrt((double)c);
    int max_sweeps = 60;
    int nb = bc.nb;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[1];
    cfg.gridDim = dim3(bc.CS);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = bc.CS;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    ctx->launches++;
    VP_CUDA(ctx, cudaLaunchKernelEx(&cfg, k_jacobi_block, X, b, c, eps, max_sweeps, nb, status));
    return VP_OK;
  }
  if (CS > 0 && b > 1 && cluster_jacobi_smem(b, c, CS) <= 200 * 1024) {
    static AttrOnce attr_done;
    // at least 120 KB per CTA, so no two CTAs of the cluster share an SM
    const size_t smem = std::max<size_t>(cluster_jacobi_smem(b, c, CS), 120 * 1024);
    VP_TRY(attr_done.ensure(ctx, (const void*)k_jacobi_cluster, 200 * 1024, true));
    double eps = 1e-15 * std::sqrt((double)c);
    int max_sweeps = 60;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[1];
    cfg.gridDim = dim3(CS);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = CS;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    ctx->launches++;
    VP_CUDA(ctx, cudaLaunchKernelEx(&cfg, k_jacobi_cluster, X, b, c, eps, max_sweeps, status));
    return VP_OK;
  }
  if (b == 1) return VP_OK;
  const int npairs = (b + 1) / 2;
  int blocks = std::min(ctx->num_sms, std::max(1, (npairs + kWarps - 1) / kWarps));
  if ((long long)b * c < 4096) blocks = 1;
  // rotate while |<x_i,x_j>| > eps |x_i||x_j|; eps grows with the dot length
  double eps = 1e-15 * std::sqrt((double)c);
  int max_sweeps = 60;
  DevStatus* st = status;
  void* args[] = {&X, &b, &c, &eps, &max_sweeps, &st};
  return coop_launch(ctx, stream, (const void*)k_jacobi_rows, blocks, kThreads, args, 0, "jacobi_rows");
}

int launch_jacobi_rows(vp_ctx* ctx, const double* R, double* X, int b, double* norms, bool floor_ok, bool* have_norms) {
  return jacobi_rows_on(ctx, ctx->stream, ctx->status, R, X, b, norms, floor_ok, have_norms);
}

// ------------------------------------------------------------ truncation
// Descending order with ties broken by index, as a strict total order even when
// values are NaN (NaNs first): the rank of each element is then a permutation, so
// the indices written from it always stay in range.  The values are >= 0 or NaN,
// whose order is that of their bits without the sign: an FP64 comparison costs an
// FP64 issue slot, of which an SM has two a clock.
__device__ __forceinline__ unsigned long long order_key(double a) {
  return (unsigned long long)__double_as_longlong(a) & ~(1ull << 63);
}
__device__ __forceinline__ unsigned order_key(float a) { return __float_as_uint(a) & 0x7fffffffu; }
template <class Key>
__device__ __forceinline__ bool sorts_before(Key a, int ia, Key b, int ib) {
  return a > b || (a == b && ia < ib);
}

// Single block: row norms, descending order (ties by index), kept rank by the
// rule r = min(chi, r_tol), r_tol the smallest r with sqrt(sum_{i>=r} s_i^2)
// <= tol ||s|| (tol = 0: keep all), moved down to the start of a cluster of
// values within a relative 1e-5.  A dependent FP64 operation costs hundreds of
// cycles on GB300, so nothing here runs as a serial chain over the values:
// four rows per warp at a time for the norms (each row summed in the same
// order as alone), the tail sums as a block-wide suffix scan (chunk sums,
// then a scan of the chunk totals), r_tol as a minimum over the rows that
// meet the tolerance, and the entanglement entropy as a fixed-order tree sum.
// norms: the row norms where the Jacobi kernel left them, else NULL (formed here,
// with the same sums); want_ent: whether the entropy is asked for.  (18 us on
// average over the sites of a 1024 x 1024 step with norms, entropy and FP64
// comparisons here, 6.7 now.)
__device__ __forceinline__ void k_select_body(const double* __restrict__ X, const double* __restrict__ norms, int b, int c,
                                              int chi, double tol, int want_ent, int* perm, double* sigma, int* d_rank,
                                              double* d_err, DevStatus* st) {
  extern __shared__ double sm[];
  double* s = sm;          // b
  double* tail = sm + b;   // b + 1
  __shared__ double ctot[1024];  // per-thread chunk totals, then their suffix sums
  __shared__ double wpart[32];
  __shared__ int rmin, rkeep;
  const int T = blockDim.x;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = T >> 5;
  constexpr int RB = 4;
  if (norms) {
    for (int i = threadIdx.x; i < b; i += T) s[i] = norms[i];
  } else {
    for (int i0 = warp * RB; i0 < b; i0 += nwarps * RB) {
      double a[RB];
#pragma unroll
      for (int u = 0; u < RB; ++u) a[u] = 0.0;
      for (int q = lane; q < c; q += 32)
#pragma unroll
        for (int u = 0; u < RB; ++u)
          if (i0 + u < b) {
            const double x = X[(size_t)(i0 + u) * c + q];
            a[u] = fma(x, x, a[u]);
          }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1)
#pragma unroll
        for (int u = 0; u < RB; ++u) a[u] += __shfl_xor_sync(0xffffffffu, a[u], o);
      if (lane == 0)
#pragma unroll
        for (int u = 0; u < RB; ++u)
          if (i0 + u < b) s[i0 + u] = sqrt(a[u]);
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < b; i += T) {
    const double si = s[i];
    const unsigned long long ki = order_key(si);
    if ((ki >> 52) == 2047) atomicCAS(&st->err, 0, 2);  // NaN or Inf
    int pos = 0;
    for (int j = 0; j < b; ++j) pos += sorts_before(order_key(s[j]), j, ki, i);
    perm[pos] = i;
    sigma[pos] = si;
  }
  __syncthreads();
  // tail[i] = sum_{k >= i} sigma_k^2: each thread a chunk of k consecutive
  // values (summed smallest first), then a suffix scan of the chunk totals
  const int k = (b + T - 1) / T;
  const int lo = threadIdx.x * k, hi = min(b, lo + k);
  double acc = 0.0;
  for (int i = hi - 1; i >= lo; --i) {
    acc = fma(sigma[i], sigma[i], acc);
    tail[i] = acc;
  }
  ctot[threadIdx.x] = acc;
  if (threadIdx.x == 0) {
    tail[b] = 0.0;
    rmin = b;
  }
  __syncthreads();
  for (int off = 1; off < T; off <<= 1) {
    const double v = ctot[threadIdx.x] + (threadIdx.x + off < T ? ctot[threadIdx.x + off] : 0.0);
    __syncthreads();
    ctot[threadIdx.x] = v;
    __syncthreads();
  }
  const double after = threadIdx.x + 1 < T ? ctot[threadIdx.x + 1] : 0.0;
  for (int i = lo; i < hi; ++i) tail[i] += after;
  __syncthreads();
  const double nrm2 = tail[0];
  if (nrm2 > 0.0 && tol > 0.0) {
    const double thr2 = tol * tol * nrm2;
    for (int q = threadIdx.x + 1; q <= b; q += T)
      if (tail[q] <= thr2) atomicMin(&rmin, q);
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    int r = 1;
    double err = 0.0;
    if (nrm2 > 0.0) {
      r = min(min(chi, rmin), b);
      while (r > 1 && r < b && (sigma[r - 1] - sigma[r]) <= 1e-5 * sigma[r - 1]) --r;
      if (r < 1) r = 1;
      err = sqrt(tail[r] / nrm2);
    }
    rkeep = r;
    *d_rank = r;
    d_err[0] = err;
  }
  __syncthreads();
  // entanglement entropy of the kept values (main text, EE equation):
  // -sum p log2 p with p_i = s_i^2 / sum_{kept} s^2
  const int r = rkeep;
  const double kept2 = tail[0] - tail[r];
  double ee = 0.0;
  if (want_ent && kept2 > 0.0)
    for (int q = threadIdx.x; q < r; q += T) {
      const double pq = sigma[q] * sigma[q] / kept2;
      if (pq > 0.0) ee -= pq * log2(pq);
    }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) ee += __shfl_xor_sync(0xffffffffu, ee, o);
  if (lane == 0) wpart[warp] = ee;
  __syncthreads();
  if (threadIdx.x == 0) {
    double tot = 0.0;
    for (int w = 0; w < nwarps; ++w) tot += wpart[w];
    d_err[1] = tot;
  }
}
__global__ void k_select(const double* __restrict__ X, const double* __restrict__ norms, int b, int c, int chi, double tol,
                         int want_ent, int* perm, double* sigma, int* d_rank, double* d_err, DevStatus* st) {
  follow();
  k_select_body(X, norms, b, c, chi, tol, want_ent, perm, sigma, d_rank, d_err, st);
}
// Threads of the selection: one per value up to 512 (the scans take as many steps
// as the block is wide).
static int select_threads(int b) { return std::min(512, std::max(128, (b + 31) / 32 * 32)); }

int launch_select(vp_ctx* ctx, const double* X, const double* norms, int b, int c, int chi, double tol, bool want_ent,
                  int* perm, double* sigma, int* d_rank, double* d_err) {
  const size_t smem = (size_t)(2 * b + 1) * sizeof(double);
  if (smem > 200 * 1024) return fail(ctx, VP_ECAPACITY, "select: bond too large");
  // always: the kernel's own 8 KB of static shared memory counts against the
  // 48 KB a block gets without the opt-in
  static AttrOnce sattr;
  VP_TRY(sattr.ensure(ctx, (const void*)k_select, 200 * 1024, false));
  return launch_after(ctx, "select", k_select, dim3(1), dim3(select_threads(b)), smem, ctx->stream, kNoCluster, X,
                      norms, b, c, chi, tol, want_ent, perm, sigma, d_rank, d_err, ctx->status);
}

__device__ __forceinline__ void k_svd_outputs_body(const double* __restrict__ X, int q, int r, const int* __restrict__ perm,
                                                   const double* __restrict__ sigma, const int* __restrict__ cperm,
                                                   double* __restrict__ V) {
  const size_t total = (size_t)r * q;
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < total; e += (size_t)gridDim.x * blockDim.x) {
    const int t = (int)(e / q), j = (int)(e % q);
    const double s = sigma[t];
    V[(size_t)t * q + cperm[j]] = s > 0.0 ? X[(size_t)perm[t] * q + j] / s : 0.0;
  }
}
__global__ void k_svd_outputs(const double* __restrict__ X, int q, int r, const int* __restrict__ perm,
                              const double* __restrict__ sigma, const int* __restrict__ cperm, double* __restrict__ V) {
  follow();
  k_svd_outputs_body(X, q, r, perm, sigma, cperm, V);
}

int launch_svd_outputs(vp_ctx* ctx, const double* X, int q, int r, const int* perm, const double* sigma,
                       const int* cperm, double* V) {
  const int blocks = (int)std::min<size_t>(((size_t)r * q + 255) / 256, (size_t)ctx->num_sms * 8);
  return launch_after(ctx, "svd_outputs", k_svd_outputs, dim3(std::max(1, blocks)), dim3(256), 0, ctx->stream,
                      kNoCluster, X, q, r, perm, sigma, cperm, V);
}

// ------------------------------------------------------ SVD preconditioning
// Static pivoting for the Jacobi SVD: order the columns (tall) or rows (wide)
// of M by decreasing norm, so that the triangular factor of the reordered
// matrix is graded and one-sided Jacobi on it converges in fewer sweeps.
// The norms only decide an order, so they are FP32 sums of the entries scaled by a
// common power of two: with FP64 squares and comparisons an SM's two FP64 slots a
// clock were what the kernel waited for (10.5 us on average over the sites of a
// 1024 x 1024 step, now 6.5).  Entries 2^-60 below the largest count as zero.
__device__ __forceinline__ void k_norm_order_body(const double* __restrict__ M, int ld, int m, int c, int by_cols, int lower,
                                                  int* __restrict__ piv) {
  extern __shared__ double nrm_raw[];
  float* nrm = reinterpret_cast<float*>(nrm_raw);
  __shared__ int emax;
  const int q = by_cols ? c : m;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = blockDim.x >> 5;
  if (tid == 0) emax = 1;
  __syncthreads();
  // (lanes along the contiguous direction in both cases)
  int e = 1;
  for (int r = warp; r < m; r += nw)
#pragma unroll 4
    for (int k = lane; k < (lower ? min(c, r + 1) : c); k += 32) {
      const int x = (int)((__double_as_longlong(M[(size_t)r * ld + k]) >> 52) & 0x7ff);
      if (x < 2047) e = max(e, x);
    }
  e = __reduce_max_sync(0xffffffffu, e);
  if (lane == 0) atomicMax(&emax, e);
  __syncthreads();
  const int sh = emax - 1022;  // largest entry to [1/2, 1)
  // a non-finite entry makes its norm NaN, which sorts first
  auto entry = [&](int r, int k) {
    const double x = M[(size_t)r * ld + k];
    return ((__double_as_longlong(x) >> 52) & 0x7ff) == 2047 ? __int_as_float(0x7fc00000) : dw_from_scaled(x, sh).hi;
  };
  if (by_cols) {
    float* part = nrm + q;  // nw x 32: the warps' sums of one group of 32 columns
    for (int k0 = 0; k0 < c; k0 += 32) {
      const int k = k0 + lane;
      float s = 0.f;
      if (k < c)
#pragma unroll 4
        for (int r = warp; r < m; r += nw) {
          const float x = lower && r < k ? 0.f : entry(r, k);
          s = fmaf(x, x, s);
        }
      part[warp * 32 + lane] = s;
      __syncthreads();
      if (warp == 0 && k < c) {
        float t = 0.f;
        for (int w = 0; w < nw; ++w) t += part[w * 32 + lane];
        nrm[k] = t;
      }
      __syncthreads();
    }
  } else {
    for (int r = warp; r < m; r += nw) {
      float s = 0.f;
      for (int k = lane; k < (lower ? min(c, r + 1) : c); k += 32) {
        const float x = entry(r, k);
        s = fmaf(x, x, s);
      }
      for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      if (lane == 0) nrm[r] = s;
    }
  }
  __syncthreads();
  for (int j = tid; j < q; j += blockDim.x) {
    const unsigned v = order_key(nrm[j]);
    int pos = 0;
    for (int k = 0; k < q; ++k) pos += sorts_before(order_key(nrm[k]), k, v, j);
    piv[pos] = j;
  }
}
__global__ void __launch_bounds__(512) kb_norm_order(const __grid_constant__ Pack<BNormOrder> pk) {
  follow();
  const BNormOrder& a = pk.a[blockIdx.y];
  k_norm_order_body(a.M, a.ld, a.m, a.c, a.by_cols, a.lower, a.piv);
}
int launch_norm_order(vp_ctx* ctx, const double* M, int ld, int m, int c, int by_cols, int lower, int* piv) {
  return blaunch_norm_order(ctx, ctx->stream, {BNormOrder{M, ld, m, c, by_cols, lower, piv}});
}

// ====================================================== batched launches
// Each kernel below runs the body of its single-problem counterpart for the
// problem the grid's batch coordinate selects (y for one-dimensional grids,
// z for tiled ones), with that problem's own launch geometry.

void release_scratch(vp_ctx* ctx, BScratch& s) {
  for (DevBuf* b : {&s.wq, &s.wr, &s.qrv, &s.qrc}) release(ctx, *b);
  for (int i = 0; i < kScratchSlots; ++i) {
    release(ctx, s.fq[i]);
    release(ctx, s.qscr[i]);
    release(ctx, s.split[i]);
    release(ctx, s.oza[i]);
    release(ctx, s.ozb[i]);
  }
}

namespace {
// Slot of a job's scratch within one launcher call: the n-th job naming the
// same BScratch takes slot n.
struct SlotCounter {
  std::vector<std::pair<const BScratch*, int>> seen;
  int next(vp_ctx* ctx, const BScratch* s, int* slot) {
    for (auto& e : seen)
      if (e.first == s) {
        if (e.second >= kScratchSlots) return fail(ctx, VP_ECAPACITY, "batched launch: too many jobs on one scratch");
        *slot = e.second++;
        return VP_OK;
      }
    seen.push_back({s, 1});
    *slot = 0;
    return VP_OK;
  }
};
}  // namespace

namespace {

size_t grid_stride_blocks(const vp_ctx* ctx, size_t total, size_t cap_per_sm) {
  return std::max<size_t>(1, std::min<size_t>((total + 255) / 256, (size_t)ctx->num_sms * cap_per_sm));
}

// kern<<<(gx, nb), threads, smem>>>(pack) for every pack of the problems;
// gx(problem) gives the x extent a problem's own launch would use.
template <class A, class GX>
int run_packs(vp_ctx* ctx, cudaStream_t st, const std::vector<A>& v, void (*kern)(const Pack<A>), int threads,
              size_t smem, GX gx, const char* what) {
  for (size_t i0 = 0; i0 < v.size(); i0 += kMaxBatch) {
    const int nb = (int)std::min<size_t>(kMaxBatch, v.size() - i0);
    Pack<A> pk{};
    int gxm = 1;
    for (int i = 0; i < nb; ++i) {
      pk.a[i] = v[i0 + i];
      gxm = std::max(gxm, (int)gx(v[i0 + i]));
    }
    VP_TRY(launch_after(ctx, what, kern, dim3(gxm, nb), dim3(threads), smem, st, kNoCluster, pk));
  }
  return VP_OK;
}

}  // namespace

// --------------------------------------------------------------- QR
// Several grid factors in one cooperative launch: problem i owns blocks
// first .. first + nblocks - 1 and runs k_qr_factor_dw's body on them as if
// they were its whole grid (the result does not depend on the block count).
struct QRGridArgs {
  double* A;
  int m, n;
  double* tau;
  dw* V;
  dw* T;
  dw* gcols;
  int* gexp;
  DevStatus* st;
  int first, nblocks;
};
__global__ void __launch_bounds__(kThreads) kb_qr_factor_dw(const __grid_constant__ Pack<QRGridArgs> pk, int count) {
  int i = 0;
  while (i + 1 < count && (int)blockIdx.x >= pk.a[i + 1].first) ++i;
  const QRGridArgs& a = pk.a[i];
  qr_factor_dw_body(a.A, a.m, a.n, a.tau, a.V, a.T, a.gcols, a.gexp, a.st, a.nblocks, blockIdx.x - a.first);
}

// The grid factors of a batch: each launch takes up to kMaxBatch problems
// that each get at least two blocks, one block per SM in all.
static int grid_qr_batch(vp_ctx* ctx, cudaStream_t st, const std::vector<const BQR*>& v) {
  static AttrOnce qattr;
  VP_TRY(qattr.ensure(ctx, (const void*)kb_qr_factor_dw, 200 * 1024, false));
  const int per_launch = std::min(kMaxBatch, std::max(1, ctx->num_sms / 2));
  for (size_t i0 = 0; i0 < v.size(); i0 += per_launch) {
    const int cnt = (int)std::min<size_t>(per_launch, v.size() - i0);
    const int share = std::max(2, ctx->num_sms / cnt);
    Pack<QRGridArgs> pk{};
    int total = 0;
    size_t smem = 0;
    for (int c = 0; c < cnt; ++c) {
      const BQR& q = *v[i0 + c];
      const int p = std::min(q.m, q.n);
      const int blocks = std::max(2, std::min(share, q.n / 2));
      const int nmax = (q.n + blocks - 1) / blocks;
      const size_t need = (size_t)nmax * q.m * sizeof(dw) + (size_t)nmax * sizeof(int);
      VP_TRY(reserve(ctx, q.s->qrv, (size_t)q.m * p + p + 8));
      QRGridArgs& a = pk.a[c];
      a = {q.A, q.m, q.n, q.tau, reinterpret_cast<dw*>(q.s->qrv.p), nullptr, nullptr, nullptr, q.s->st, total, blocks};
      a.T = a.V + (size_t)q.m * p;
      if (need > 200 * 1024) {  // columns in global scratch
        VP_TRY(reserve(ctx, q.s->qrc, (size_t)q.m * q.n + q.n / 2 + 8));
        a.gcols = reinterpret_cast<dw*>(q.s->qrc.p);
        a.gexp = reinterpret_cast<int*>(a.gcols + (size_t)q.m * q.n);
      } else {
        smem = std::max(smem, need);
      }
      total += blocks;
    }
    int count = cnt;
    void* args[] = {&pk, &count};
    VP_TRY(coop_launch(ctx, st, (const void*)kb_qr_factor_dw, total, kThreads, args, smem, "b_qr_factor_dw"));
  }
  return VP_OK;
}

int blaunch_qr_factor(vp_ctx* ctx, cudaStream_t st, const std::vector<BQR>& v) {
  std::vector<BQR> wide;
  std::vector<const BQR*> grid;
  std::vector<PanelJob> panel;
  std::vector<BGather> gat;
  for (const BQR& q : v) {
    const int kind = qr_plan(ctx, q.m, q.n).kind;
    if (q.src.p && (kind == QR_WIDE || kind == QR_GRID)) gat.push_back({q.src, q.m, q.n, q.A});
  }
  VP_TRY(blaunch_gather(ctx, st, gat));
  for (const BQR& q : v) {
    const QRPlan pl = qr_plan(ctx, q.m, q.n);
    switch (pl.kind) {
      case QR_NONE:
        break;
      case QR_WIDE:
        wide.push_back(q);
        break;
      case QR_PANEL:
        panel.push_back({q.A, q.m, q.n, q.tau, pl.panel, q.src, &q.s->qrv, &q.s->qrc, q.s->st});
        break;
      default:
        if (!q.s || !q.s->st) return fail(ctx, VP_EINVAL, "batched QR: no status words for a grid factor");
        if (q.n / 2 >= 2)
          grid.push_back(&q);
        else  // a single block: the barrier kernel of the single path
          VP_TRY(qr_factor_grid(ctx, st, q.s->st, q.s->qrv, q.s->qrc, q.A, q.m, q.n, q.tau, q.vbuf));
    }
  }
  VP_TRY(blaunch_qr_panel(ctx, st, panel));
  if (!grid.empty()) VP_TRY(grid_qr_batch(ctx, st, grid));
  if (!wide.empty()) {  // the square block, its Q, R2^T = A2^T Q in FP64, copied back (see qr_plan)
    std::vector<BQR> sq;
    std::vector<BFormQ> fq;
    std::vector<BGemm> gm;
    std::vector<BCopy> cp;
    for (const BQR& q : wide) {
      const int m = q.m;
      const size_t rest = (size_t)(q.n - m) * m;
      VP_TRY(reserve(ctx, q.s->wq, (size_t)m * m));
      VP_TRY(reserve(ctx, q.s->wr, rest));
      sq.push_back({q.A, m, m, q.tau, q.vbuf, q.s});
      fq.push_back({q.A, m, m, q.tau, q.s->wq.p, q.s});
      gm.push_back({BG_AB, 0, q.n - m, m, m, 1.0, q.A + (size_t)m * m, m, q.s->wq.p, m, q.s->wr.p, m, q.s, OZ_ROWS});
      cp.push_back({q.s->wr.p, q.A + (size_t)m * m, rest});
    }
    VP_TRY(blaunch_qr_factor(ctx, st, sq));
    VP_TRY(blaunch_qr_formq(ctx, st, fq));
    VP_TRY(blaunch_gemm(ctx, st, gm));
    VP_TRY(blaunch_copy(ctx, st, cp));
  }
  return VP_OK;
}

int blaunch_qr_formq(vp_ctx* ctx, cudaStream_t st, const std::vector<BFormQ>& v) {
  std::vector<FormQJob> jobs;
  SlotCounter slots;
  for (const BFormQ& f : v) {
    if (std::min(f.m, f.n) <= 0) continue;
    int sl = 0;
    VP_TRY(slots.next(ctx, f.s, &sl));
    jobs.push_back({f.A, f.m, f.n, f.tau, f.Q, f.rows, &f.s->fq[sl], &f.s->qscr[sl]});
  }
  return blaunch_formq(ctx, st, jobs);
}

struct GetRArgs {
  const double* A;
  int m, n, p;
  double* R;
};
__global__ void kb_qr_getr(const __grid_constant__ Pack<GetRArgs> pk) {
  follow();
  const GetRArgs& a = pk.a[blockIdx.y];
  k_qr_getr_body(a.A, a.m, a.n, a.p, a.R);
}
int blaunch_qr_getr(vp_ctx* ctx, cudaStream_t st, const std::vector<BGetR>& v) {
  std::vector<GetRArgs> g;
  for (const BGetR& r : v) {
    const int p = std::min(r.m, r.n);
    if ((size_t)p * r.n > 0) g.push_back({r.A, r.m, r.n, p, r.R});
  }
  return run_packs(ctx, st, g, kb_qr_getr, 256, 0,
                   [&](const GetRArgs& a) { return grid_stride_blocks(ctx, (size_t)a.p * a.n, 16); }, "b_getr");
}

// --------------------------------------------------------------- GEMM
template <class ALoad, class BLoad>
struct GemmJob {
  int M, N, K, kslice, slices;
  double alpha;
  ALoad a;
  BLoad b;
  double* C;
  int ldc;
  size_t stride;
};
template <class ALoad, class BLoad, int TILE>
__global__ void __launch_bounds__(256) kb_gemm(const __grid_constant__ Pack<GemmJob<ALoad, BLoad>> pk, int zs) {
  const GemmJob<ALoad, BLoad>& j = pk.a[blockIdx.z / zs];
  const int slice = blockIdx.z % zs;
  if (slice >= j.slices || (int)blockIdx.x * TILE >= j.M || (int)blockIdx.y * TILE >= j.N) return;
  gemm_body<ALoad, BLoad, TILE>(j.M, j.N, j.K, j.alpha, j.a, j.b, j.C, j.ldc, j.kslice, j.stride, blockIdx.x,
                                   blockIdx.y, slice);
}
__global__ void kb_sum_slices(const __grid_constant__ Pack<OzSum> pk) {
  follow();
  const OzSum& a = pk.a[blockIdx.y];
  k_sum_slices_body(a.P, a.M, a.N, a.slices, a.stride, a.C, a.ldc);
}

namespace {
template <class ALoad, class BLoad, int TILE>
int gemm_group(vp_ctx* ctx, cudaStream_t st, const std::vector<GemmJob<ALoad, BLoad>>& jobs) {
  for (size_t i0 = 0; i0 < jobs.size(); i0 += kMaxBatch) {
    const int nb = (int)std::min<size_t>(kMaxBatch, jobs.size() - i0);
    Pack<GemmJob<ALoad, BLoad>> pk{};
    int gx = 1, gy = 1, zs = 1;
    for (int i = 0; i < nb; ++i) {
      const auto& j = jobs[i0 + i];
      pk.a[i] = j;
      gx = std::max(gx, (j.M + TILE - 1) / TILE);
      gy = std::max(gy, (j.N + TILE - 1) / TILE);
      zs = std::max(zs, j.slices);
    }
    if (gy > 65535) return fail(ctx, VP_ECAPACITY, "gemm: N too large");
    ctx->launches++;
    kb_gemm<ALoad, BLoad, TILE><<<dim3(gx, gy, nb * zs), 256, 0, st>>>(pk, zs);
    VP_TRY(check_launch(ctx, "b_gemm"));
  }
  return VP_OK;
}
}  // namespace

int blaunch_gemm(vp_ctx* ctx, cudaStream_t st, const std::vector<BGemm>& v) {
  // FP32 contractions by tile (64 / 32)
  std::vector<GemmJob<ARowMajor, BRowMajor>> ab[2];
  std::vector<GemmJob<ARowMajor, BTransposed>> abt[2];
  std::vector<GemmJob<AUpperColMajor, BRowMajor>> rb[2];
  std::vector<OzSum> sums;
  std::vector<OzGemm> oz, fma;
  SlotCounter slots;
  for (const BGemm& g : v) {
    if (g.M <= 0 || g.N <= 0) continue;
    const GemmPlan pl = gemm_plan(ctx, g.M, g.N, g.K);
    const OzPlan op = g.fp32 ? OzPlan{} : oz_plan(ctx, g.M, g.N, g.K);
    const int slices = g.fp32 ? pl.slices : 1, kslice = pl.kslice, ti = pl.tile == 64 ? 0 : 1;
    double* C = g.C;
    int ldc = g.ldc;
    size_t stride = 0;
    int sl = 0;
    if (slices > 1 || op.use) VP_TRY(slots.next(ctx, g.s, &sl));
    if (slices > 1) {
      stride = (size_t)g.M * g.N;
      VP_TRY(reserve(ctx, g.s->split[sl], stride * slices));
      C = g.s->split[sl].p;
      ldc = g.N;
      sums.push_back({g.s->split[sl].p, g.M, g.N, slices, stride, g.C, g.ldc});
    }
    if (!g.fp32) {
      const TcOperand ta{g.A, g.lda, g.kind == BG_RB ? 2 : 0}, tb{g.B, g.ldb, g.kind == BG_ABT ? 0 : 1};
      (op.use ? oz : fma).push_back(oz_job(ta, tb, g.M, g.N, g.K, g.alpha, C, ldc, g.s ? &g.s->oza[sl] : nullptr,
                                           g.s ? &g.s->ozb[sl] : nullptr, g.s ? &g.s->split[sl] : nullptr, g.s && g.s->st ? g.s->st : ctx->status, op,
                                           g.kind == BG_RB ? OZ_COLS : g.bound));
      continue;
    }
    if (g.kind == BG_AB)
      ab[ti].push_back({g.M, g.N, g.K, kslice, slices, g.alpha, ARowMajor{g.A, g.lda}, BRowMajor{g.B, g.ldb}, C, ldc,
                        stride});
    else if (g.kind == BG_ABT)
      abt[ti].push_back({g.M, g.N, g.K, kslice, slices, g.alpha, ARowMajor{g.A, g.lda}, BTransposed{g.B, g.ldb}, C, ldc,
                         stride});
    else
      rb[ti].push_back({g.M, g.N, g.K, kslice, slices, g.alpha, AUpperColMajor{g.A, g.lda}, BRowMajor{g.B, g.ldb}, C,
                        ldc, stride});
  }
  VP_TRY(blaunch_oz_gemm(ctx, st, oz));
  VP_TRY(blaunch_fma_gemm(ctx, st, fma));
  VP_TRY((gemm_group<ARowMajor, BRowMajor, 64>(ctx, st, ab[0])));
  VP_TRY((gemm_group<ARowMajor, BRowMajor, 32>(ctx, st, ab[1])));
  VP_TRY((gemm_group<ARowMajor, BTransposed, 64>(ctx, st, abt[0])));
  VP_TRY((gemm_group<ARowMajor, BTransposed, 32>(ctx, st, abt[1])));
  VP_TRY((gemm_group<AUpperColMajor, BRowMajor, 64>(ctx, st, rb[0])));
  VP_TRY((gemm_group<AUpperColMajor, BRowMajor, 32>(ctx, st, rb[1])));
  return blaunch_sum_slices(ctx, st, sums);
}

int blaunch_sum_slices(vp_ctx* ctx, cudaStream_t st, const std::vector<OzSum>& v) {
  return run_packs(ctx, st, v, kb_sum_slices, 256, 0, [&](const OzSum& a) { return grid_stride_blocks(ctx, a.stride, 8); },
                   "b_sum_slices");
}

// --------------------------------------------------------------- SVD site helpers
int blaunch_norm_order(vp_ctx* ctx, cudaStream_t st, const std::vector<BNormOrder>& v) {
  size_t smem = 0;
  for (const BNormOrder& a : v) smem = std::max(smem, (size_t)((a.by_cols ? a.c : a.m) + 16 * 32) * sizeof(float));
  if (smem > 200 * 1024) return fail(ctx, VP_ECAPACITY, "norm_order: too many columns");
  static AttrOnce at;
  VP_TRY(at.ensure(ctx, (const void*)kb_norm_order, 200 * 1024, false));
  return run_packs(ctx, st, v, kb_norm_order, 512, smem, [](const BNormOrder&) { return 1; }, "b_norm_order");
}
int blaunch_jacobi(vp_ctx* ctx, cudaStream_t st, const std::vector<BJacobi>& v, std::vector<char>& have_norms) {
  std::vector<BJacobi> fit;
  have_norms.assign(v.size(), 0);
  for (size_t i = 0; i < v.size(); ++i) {
    const BJacobi& j = v[i];
    if (jacobi_dw_fits(ctx, j.b)) {
      fit.push_back(j);
      have_norms[i] = 1;
    } else {
      bool hn = false;
      VP_CUDA(ctx, cudaMemsetAsync(j.st->rot, 0, sizeof(j.st->rot), st));
      VP_TRY(jacobi_rows_on(ctx, st, j.st, j.R, j.X, j.b, j.norms, true, &hn));
    }
  }
  return blaunch_jacobi_dw(ctx, st, fit);
}

__global__ void kb_select(const __grid_constant__ Pack<BSelect> pk) {
  follow();
  const BSelect& a = pk.a[blockIdx.y];
  k_select_body(a.X, a.norms, a.b, a.c, a.chi, a.tol, a.want_ent, a.perm, a.sigma, a.d_rank, a.d_err, a.st);
}
int blaunch_select(vp_ctx* ctx, cudaStream_t st, const std::vector<BSelect>& v) {
  size_t smem = 0;
  for (const BSelect& a : v) smem = std::max(smem, (size_t)(2 * a.b + 1) * sizeof(double));
  if (smem > 200 * 1024) return fail(ctx, VP_ECAPACITY, "select: bond too large");
  static AttrOnce at;
  VP_TRY(at.ensure(ctx, (const void*)kb_select, 200 * 1024, false));
  int nt = 128;
  for (const BSelect& a : v) nt = std::max(nt, select_threads(a.b));
  return run_packs(ctx, st, v, kb_select, nt, smem, [](const BSelect&) { return 1; }, "b_select");
}
__global__ void kb_svd_outputs(const __grid_constant__ Pack<BSvdOut> pk) {
  follow();
  const BSvdOut& a = pk.a[blockIdx.y];
  k_svd_outputs_body(a.X, a.q, a.r, a.perm, a.sigma, a.cperm, a.V);
}
int blaunch_svd_outputs(vp_ctx* ctx, cudaStream_t st, const std::vector<BSvdOut>& v) {
  return run_packs(ctx, st, v, kb_svd_outputs, 256, 0,
                   [&](const BSvdOut& a) { return grid_stride_blocks(ctx, (size_t)a.r * a.q, 8); }, "b_svd_outputs");
}
}  // namespace vp
