// One-sided Jacobi SVD of the sweeps' truncating compressions (SI
// "Canonicalization and Compression"), in double words, block by block through
// Gram matrices.
//
// The rows of X are split into 2 CS blocks of nb rows over a cluster of CS CTAs;
// each CTA holds two blocks in shared memory and the blocks move on the circle
// schedule (position 0 stays, every other advances by one), so that after 2 CS - 1
// block rounds every pair of rows has met once: one sweep.  A block round
//   1. forms the products of the two blocks' rows (in a sweep's first block round
//      all products of its 2 nb rows; later the ones inside a block come along
//      with it),
//   2. rotates on the Gram matrix alone, both sides, in one warp: nb rounds of nb
//      disjoint pairs across the two blocks (the first block round of a sweep also
//      the pairs inside each block), while the other warps apply the rotations of
//      the round before to the rows,
//   3. writes rows and products into the CTA where their block goes next.
// A row-by-row rotation pays a dot product with its warp reduction, two norms and
// a long update for each of its dependent rounds; here a dependent round is a few
// operations on a 2 nb x 2 nb matrix.  Rows and rotations are double words, so the
// rows stay the accurate images of the input; the Gram matrix, recomputed from
// them every sweep, only steers the rotations.  Its diagonal is a double word (two
// nearly equal norms decide an angle by their difference); what is off it needs only
// its own digits and is FP32 between two recomputations.
//
// Measured on GB300 (event-timed, one problem; before: row-by-row rotations of the
// same rows, whose every round was a dot product, parameters and an update):
// a block round of 2 x 4 rows of 128 is ~1300 cycles of products, 650-900 a round
// of rotations, 1500 for the move and 700 for the cluster barrier; 128 rows 142 us
// a sweep (243), 64: 51 (83), 44: 40 (82), 16: 13 (19), 212: 334 (519).  With double
// words on eight-byte boundaries and the FP32 part: 128 rows 110, 64: 47, 44: 36,
// 16: 12, 212: 270.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>

#include <cooperative_groups.h>

#include "common.cuh"
#include "dw.cuh"
#include "dwsum.cuh"

namespace cg = cooperative_groups;

namespace vp {
namespace {

constexpr int kJT = 512, kJW = kJT / 32;
constexpr int kJMaxNb = 15;       // pairs of a round fit one warp's ballot and the tables
constexpr float kTiny = 1e-30f;   // squared norm (largest entry ~1) below which a row is left alone

struct JacArgs {
  const double* R;  // upper triangle of a column-major b x b factor: the rows
  double* X;        // out, row-major
  double* norms;    // out: row norms
  int b;
  float eps;
  int max_sweeps, nb;
  DevStatus* st;
};

__device__ __forceinline__ int rr_index(int pos, int round, int bp) {
  return pos == 0 ? 0 : 1 + (pos - 1 + round) % (bp - 1);
}
__device__ __forceinline__ int pos_cta(int pos, int CS) { return pos < CS ? pos : 2 * CS - 1 - pos; }
__device__ __forceinline__ int pos_slot(int pos, int CS) { return pos < CS ? 0 : 1; }
__device__ __forceinline__ int next_pos(int pos, int CS) {
  return pos == 0 ? 0 : (pos == 2 * CS - 1 ? 1 : pos + 1);
}

// Rotation that zeroes gamma between rows of squared norms alpha, beta: an FP32
// tangent (the angle need not be exact), its cosine to a double word so that the
// rotation is orthogonal to 2^-47.  False: the pair is left alone.
__device__ __forceinline__ bool rotation(dw al, dw be, float g, float eps, dw& cs, dw& sn, float& t) {
  cs = {1.0f, 0.0f};
  sn = {0.0f, 0.0f};
  if (!(al.hi > kTiny && be.hi > kTiny && fabsf(g) * rsqrt_approx(al.hi) * rsqrt_approx(be.hi) > eps)) return false;
  const float d0 = 0.5f * ((be.hi - al.hi) + (be.lo - al.lo));
  // a power of two brings the larger of the two to [1, 2): no square leaves FP32
  const int ex = (__float_as_int(fmaxf(fabsf(d0), fabsf(g))) >> 23) & 255;
  const float sc = __int_as_float((254 - min(ex, 253)) << 23);
  const float d = d0 * sc, gs = g * sc;
  const float x = fmaf(d, d, gs * gs);
  t = copysignf(1.0f, d) * gs * rcp_approx(fabsf(d) + x * rsqrt_approx(x));
  if (t == 0.f) return false;
  // u = 1 + t^2; y = 1 / sqrt(u) refined in FP32, then with the residual
  // r = 1 - u y^2 in double words: y (1 + r / 2 + 3 r^2 / 8)
  const dw t2 = two_prod(t, t);
  const float uh = 1.0f + t2.hi;
  const dw u = {uh, (t2.hi - (uh - 1.0f)) + t2.lo};
  float y = rsqrt_approx(uh);
  y = fmaf(0.5f * y, fmaf(-uh * y, y, 1.0f), y);
  const dw m = dw_mul(u, two_prod(y, y));
  const float r = (1.0f - m.hi) - m.lo;
  cs = fast_two_sum(y, y * fmaf(0.375f * r, r, 0.5f * r));
  sn = dw_mul_f(cs, t);
  return true;
}

// a x + b y to a double word
__device__ __forceinline__ dw comb(dw a, dw x, dw b, dw y) {
  const dw p = two_prod(a.hi, x.hi);
  float e = fmaf(a.hi, x.lo, p.lo);
  e = fmaf(a.lo, x.hi, e);
  float s = p.hi;
  fnma_acc(s, e, dw_neg(b), y);
  return fast_two_sum(s, e);
}

// Products of row pairs into G (both triangles; of a row with itself into Dg): warp
// w takes the pairs w NV .. of tab, then those kJW NV further on.
template <int NV>
__device__ __forceinline__ void gram(const dw* rows, int c, int B, const unsigned short* tab, int npair, dw* Dg, float* G,
                                     int lane, int warp) {
  for (int base = warp * NV; base < npair; base += kJW * NV) {
    dw_acc acc[NV];
    int oi[NV], oj[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      const int e = tab[min(base + v, npair - 1)];
      oi[v] = (e >> 8) * c;
      oj[v] = (e & 255) * c;
    }
    const int v = lane / (32 / NV);
    const int mine = tab[min(base + v, npair - 1)];
    int q = lane;
    for (; q + 32 < c; q += 64) {
      dw x[2][NV], y[2][NV];
#pragma unroll
      for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int u = 0; u < NV; ++u) {
          x[h][u] = rows[oi[u] + q + 32 * h];
          y[h][u] = rows[oj[u] + q + 32 * h];
        }
#pragma unroll
      for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int u = 0; u < NV; ++u) dw_dot_step(acc[u], x[h][u], y[h][u]);
    }
    if (q < c) {
#pragma unroll
      for (int u = 0; u < NV; ++u) dw_dot_step(acc[u], rows[oi[u] + q], rows[oj[u] + q]);
    }
    dw val[NV];
#pragma unroll
    for (int u = 0; u < NV; ++u) val[u] = {acc[u].s, acc[u].c};
    const dw s = norm2(warp_sums<NV>(val, lane));
    if (lane % (32 / NV) == 0 && base + v < npair) {
      const int i = mine >> 8, j = mine & 255;
      if (i == j)
        Dg[i] = s;
      else
        G[i * B + j] = G[j * B + i] = s.hi;
    }
  }
}

__device__ __forceinline__ void jacobi_body(const JacArgs& a) {
  cg::cluster_group cl = cg::this_cluster();
  extern __shared__ double smd[];
  const int CS = (int)cl.num_blocks(), rank = (int)cl.block_rank();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int b = a.b, c = a.b, nb = a.nb, B = 2 * nb;
  dw* rows = reinterpret_cast<dw*>(smd);  // two sets of B rows: top block, bottom block
  dw* D2 = rows + 2 * (size_t)B * c;      // their squared norms
  float* G2 = reinterpret_cast<float*>(D2 + 2 * B);  // two Gram matrices (off the diagonal)
  dw* par = reinterpret_cast<dw*>(G2 + 2 * B * B);   // cosine, sine of pair p of round rd at 2 (16 rd + p)
  unsigned short* tab = reinterpret_cast<unsigned short*>(par + 32 * (2 * nb + 1));  // all pairs of rows
  unsigned short* xtab = tab + B * (B + 1) / 2;     // the pairs across the two blocks
  unsigned short* prow = xtab + nb * nb;            // rows (i << 8 | j) of pair p of round rd at 16 rd + p
  unsigned short* ptab = prow + 16 * (2 * nb + 1);  // pairs of pairs (P << 8 | Q), P < Q, of np = nb, then bp
  __shared__ int red[kJW + 1];
  __shared__ unsigned cnt[4];
  __shared__ unsigned rmask[2 * (kJMaxNb + 1)];  // pairs that rotate in each round
  // rounds: the pairs inside both blocks (bp - 1 rounds of bp pairs, a row of an
  // odd block meeting itself sits out), then nb rounds of nb pairs across
  const int bp = nb + (nb & 1), inside = bp - 1;
  const int npair = B * (B + 1) / 2;

  // common power-of-two scale: largest |x| over the cluster's rows
  auto home = [&](int slot) { return slot == 0 ? rank : 2 * CS - 1 - rank; };
  // (a row of the block is strided in the factor: a warp takes 8 rows by 4 columns,
  // the entries in place as they are while their largest exponent is taken)
  int mx = 0;
  for (int l0 = 0; l0 < B; l0 += 8) {
    const int l = l0 + (lane & 7);
    if (l >= B) continue;
    const int x = home(l / nb) * nb + l % nb;
    for (int q = 4 * warp + (lane >> 3); q < c; q += 4 * kJW) {
      const double v = x < b && q >= x ? a.R[(size_t)q * b + x] : 0.0;
      reinterpret_cast<double*>(rows)[l * c + q] = v;
      mx = max(mx, (int)((__double_as_longlong(v) >> 52) & 0x7ff));
    }
  }
  __syncwarp();
  mx = __reduce_max_sync(0xffffffffu, mx);
  if (lane == 0) red[warp] = mx;
  if (tid < 4) cnt[tid] = 0u;
  for (int i = tid; i < B; i += kJT) {
    int e = i * B - i * (i - 1) / 2;  // pairs (i, i .. B - 1)
    for (int j = i; j < B; ++j) tab[e++] = (unsigned short)((i << 8) | j);
  }
  for (int e = tid; e < nb * nb; e += kJT) xtab[e] = (unsigned short)(((e / nb) << 8) | (nb + e % nb));
  for (int e = tid; e < 16 * (inside + nb); e += kJT) {
    const int rd = e >> 4, pr = e & 15;
    int i = 0, j = 0;
    if (rd < inside) {
      const int slot = pr / (bp / 2), pos = pr % (bp / 2);
      i = rr_index(pos, rd, bp);
      j = rr_index(bp - 1 - pos, rd, bp);
      if (i > j) {
        const int t = i;
        i = j;
        j = t;
      }
      if (j >= nb) j = i;
      i += min(slot, 1) * nb;
      j += min(slot, 1) * nb;
    } else {
      i = min(pr, nb - 1);
      j = nb + (i + rd - inside) % nb;
    }
    prow[e] = (unsigned short)((i << 8) | j);
  }
  const int nt0 = nb * (nb - 1) / 2, nt1 = bp * (bp - 1) / 2;
  if (tid < 2) {
    const int np = tid ? bp : nb;
    unsigned short* o = ptab + (tid ? nt0 : 0);
    for (int P = 0; P < np; ++P)
      for (int Q = P + 1; Q < np; ++Q) *o++ = (unsigned short)((P << 8) | Q);
  }
  __syncthreads();
  if (tid == 0) {
    int m = 0;
    for (int i = 0; i < kJW; ++i) m = max(m, red[i]);
    red[kJW] = m;
  }
  cl.sync();
  int gmax = 0;
  for (int r = 0; r < CS; ++r) gmax = max(gmax, *cl.map_shared_rank(red + kJW, r));
  const int ex = gmax - 1022;  // largest entry to [1/2, 1)
  for (int e = tid; e < B * c; e += kJT) rows[e] = dw_from_scaled(reinterpret_cast<double*>(rows)[e], ex);
  __syncthreads();  // every row of the block in place before the first products
  unsigned* c0 = cl.map_shared_rank(cnt, 0);

  int cur = 0, sweep = 0;
  bool converged = false;
  const int brounds = 2 * CS - 1;
  for (; sweep < a.max_sweeps; ++sweep) {
    if (rank == 0 && tid == 0) cnt[(sweep + 1) % 3] = 0u;
    unsigned rotated = 0;
    for (int br = 0; br < brounds; ++br) {
      dw* R = rows + (size_t)cur * B * c;
      dw* Dg = D2 + cur * B;
      float* G = G2 + cur * B * B;
      const unsigned short* tb = br == 0 ? tab : xtab;
      const int ng = br == 0 ? npair : nb * nb, chunk = (ng + kJW - 1) / kJW;
      if (chunk <= 1)
        gram<1>(R, c, B, tb, ng, Dg, G, lane, warp);
      else if (chunk <= 2)
        gram<2>(R, c, B, tb, ng, Dg, G, lane, warp);
      else if (chunk <= 4)
        gram<4>(R, c, B, tb, ng, Dg, G, lane, warp);
      else if (chunk <= 8)
        gram<8>(R, c, B, tb, ng, Dg, G, lane, warp);
      else
        gram<16>(R, c, B, tb, ng, Dg, G, lane, warp);
      __syncthreads();
      const int rd0 = br == 0 ? 0 : inside, rd1 = inside + nb;
      // round rd's rotations applied to the rows: a task is one pair of one column
      auto apply = [&](int rd, int t, int nt) {
        const unsigned mask = rmask[rd];
        if (mask == 0) return;
        const int np = rd < inside ? bp : nb;
        for (int e = t; e < np * c; e += nt) {
          const int pr = e / c, q = e - pr * c;
          if (!(mask >> pr & 1)) continue;
          const int ij = prow[16 * rd + pr];
          const float4 w = *reinterpret_cast<const float4*>(par + 2 * (16 * rd + pr));
          const dw cs = {w.x, w.y}, sn = {w.z, w.w};
          dw* x = R + (ij >> 8) * c + q;
          dw* y = R + (ij & 255) * c + q;
          const dw u = *x, v = *y;
          *x = comb(cs, u, dw_neg(sn), v);
          *y = comb(sn, u, cs, v);
        }
      };
      for (int rd = rd0; rd < rd1; ++rd) {
        if (warp != 0) {
          if (rd > rd0) apply(rd - 1, tid - 32, kJT - 32);
        } else {
          const int np = rd < inside ? bp : nb, nt = rd < inside ? nt1 : nt0;
          const unsigned short* pt = ptab + (rd < inside ? nt0 : 0);
          dw cs = {1.0f, 0.0f}, sn = {0.0f, 0.0f};
          float t = 0.f;
          bool rot = false;
          const int ij = prow[16 * rd + (lane & 15)];
          if (lane < np) {
            const int i = ij >> 8, j = ij & 255;
            const dw al = Dg[i], be = Dg[j];
            const float g = G[i * B + j];
            if (i != j) rot = rotation(al, be, g, a.eps, cs, sn, t);
            if (rot) {
              const dw tg = two_prod(t, g);
              Dg[i] = dw_add_fast(al, dw_neg(tg));
              Dg[j] = dw_add_fast(be, tg);
              G[i * B + j] = G[j * B + i] = 0.f;
              par[2 * (16 * rd + lane)] = cs;
              par[2 * (16 * rd + lane) + 1] = sn;
              ++rotated;
            }
          }
          const unsigned any = __ballot_sync(0xffffffffu, rot);
          if (lane == 0) rmask[rd] = any;
          // both sides of the Gram matrix: the 2 x 2 block of pairs P < Q by one lane
          for (int e0 = 0; any != 0 && e0 < nt; e0 += 32) {
            const int e = e0 + lane, PQ = pt[min(e, nt - 1)], P = PQ >> 8, Q = PQ & 255;
            const float cp = __shfl_sync(0xffffffffu, cs.hi, P), sp = __shfl_sync(0xffffffffu, sn.hi, P);
            const float cq = __shfl_sync(0xffffffffu, cs.hi, Q), sq = __shfl_sync(0xffffffffu, sn.hi, Q);
            const int ip = __shfl_sync(0xffffffffu, ij, P), iq = __shfl_sync(0xffffffffu, ij, Q);
            const int i = ip >> 8, j = ip & 255, k = iq >> 8, l = iq & 255;
            if (e < nt && (sp != 0.f || sq != 0.f)) {
              // (a row that sits out: i == j or k == l, with cosine 1 and sine 0 on
              // its side, where both halves of the block are the same numbers)
              const float g00 = G[i * B + k], g01 = G[i * B + l], g10 = G[j * B + k], g11 = G[j * B + l];
              const float a0 = fmaf(cp, g00, -sp * g10), a1 = fmaf(sp, g00, cp * g10);
              const float b0 = fmaf(cp, g01, -sp * g11), b1 = fmaf(sp, g01, cp * g11);
              const float h00 = fmaf(cq, a0, -sq * b0), h01 = fmaf(sq, a0, cq * b0);
              const float h10 = fmaf(cq, a1, -sq * b1), h11 = fmaf(sq, a1, cq * b1);
              G[i * B + k] = G[k * B + i] = h00;
              G[i * B + l] = G[l * B + i] = h01;
              G[j * B + k] = G[k * B + j] = h10;
              G[j * B + l] = G[l * B + j] = h11;
            }
          }
        }
        __syncthreads();
      }
      apply(rd1 - 1, tid, kJT);
      if (br == brounds - 1 && warp == 0) {
        const unsigned tot = __reduce_add_sync(0xffffffffu, rotated);
        if (lane == 0 && tot) atomicAdd(&c0[sweep % 3], tot);
      }
      __syncthreads();
      // rows and the products inside each block to where the two blocks go next
#pragma unroll
      for (int slot = 0; slot < 2; ++slot) {
        const int np = next_pos(home(slot), CS), ds = pos_slot(np, CS);
        dw* to = cl.map_shared_rank(rows + (size_t)(cur ^ 1) * B * c + (size_t)ds * nb * c, pos_cta(np, CS));
        const dw* from = R + (size_t)slot * nb * c;
        for (int e = tid; e < nb * c; e += kJT) to[e] = from[e];
        float* tg = cl.map_shared_rank(G2 + (cur ^ 1) * B * B, pos_cta(np, CS));
        if (tid < nb) cl.map_shared_rank(D2 + (cur ^ 1) * B, pos_cta(np, CS))[ds * nb + tid] = Dg[slot * nb + tid];
        for (int e = tid; e < nb * nb; e += kJT) {
          const int i = e / nb, j = e - i * nb;
          tg[(ds * nb + i) * B + ds * nb + j] = G[(slot * nb + i) * B + slot * nb + j];
        }
      }
      cur ^= 1;
      cl.sync();
    }
    if (*(volatile unsigned*)&c0[sweep % 3] == 0u) {
      converged = true;
      ++sweep;
      break;
    }
  }
  // blocks are home after a whole number of sweeps
  for (int l = warp; l < B; l += kJW) {
    const int x = home(l / nb) * nb + l % nb;
    if (x >= b) continue;
    const dw* d = rows + ((size_t)cur * B + l) * c;
    double sum = 0.0;  // the norm as the selection would form it
    for (int q = lane; q < c; q += 32) {
      const double v = dw_to_scaled(d[q], ex);
      a.X[(size_t)x * c + q] = v;
      sum = fma(v, v, sum);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    if (lane == 0) a.norms[x] = sqrt(sum);
  }
  if (rank == 0 && tid == 0) {
    a.st->pad2 = converged ? sweep : a.max_sweeps + 1;
    if (!converged) atomicCAS(&a.st->err, 0, 3);
  }
  cl.sync();  // keep every CTA's shared memory alive until all remote accesses are done
}

__global__ void __launch_bounds__(kJT, 1) kb_jacobi_dw(const __grid_constant__ Pack<JacArgs> pk) {
  follow();
  jacobi_body(pk.a[blockIdx.y]);
}

struct JacCfg {
  int cs, nb;
};
// Four to six rows a block (more only beyond 16 CTAs): fewer would leave too
// little rotation between two meetings, more makes the products and the move grow
// with the square of the block (8 rows of 128 on 8 CTAs took as long as 4 on 16).
JacCfg jac_cfg(int b, int cs_max) {
  int cs = 1;
  while (cs < 16 && cs < cs_max && cs * 12 < b) cs *= 2;
  return {cs, std::max(1, (b + 2 * cs - 1) / (2 * cs))};
}
size_t jac_smem(const JacCfg& g, int c) {
  const size_t B = 2 * (size_t)g.nb, bp = g.nb + (g.nb & 1);
  return (2 * B * c + 2 * B + 32 * (B + 1)) * sizeof(dw) + 2 * B * B * sizeof(float) +
         (B * (B + 1) / 2 + g.nb * g.nb + 16 * (B + 1) + g.nb * (g.nb + 1) / 2 + bp * (bp + 1) / 2) * sizeof(unsigned short);
}
constexpr size_t kJacSmemMax = 216 * 1024;

}  // namespace

bool jacobi_dw_fits(const vp_ctx* ctx, int b) {
  const JacCfg g = jac_cfg(b, std::max(1, ctx->cluster_size));
  return b > 1 && g.nb <= kJMaxNb && jac_smem(g, b) <= kJacSmemMax;
}

int blaunch_jacobi_dw(vp_ctx* ctx, cudaStream_t st, const std::vector<BJacobi>& v) {
  std::vector<JacArgs> grp[17];
  size_t smem[17] = {};
  for (const BJacobi& j : v) {
    const JacCfg g = jac_cfg(j.b, std::max(1, ctx->cluster_size));
    // rotate while |gamma| > eps sqrt(alpha beta), eps above the noise of the
    // double-word products (~1e-14).  core_{k-1} takes M V, so what is left of
    // gamma enters the state twice: at 4e-13 sqrt(c) random states of 40 .. 200
    // rows kept 2.2 times the error, at 1e-13 half of it, for at most a sweep more
    grp[g.cs].push_back({j.R, j.X, j.norms, j.b, (float)(1e-13 * std::sqrt((double)j.b)), 60, g.nb, j.st});
    smem[g.cs] = std::max(smem[g.cs], jac_smem(g, j.b));
  }
  for (int cs = 1; cs <= 16; ++cs) {
    if (grp[cs].empty()) continue;
    static AttrOnce at;
    VP_TRY(at.ensure(ctx, (const void*)kb_jacobi_dw, (int)kJacSmemMax, true));
    for (size_t i0 = 0; i0 < grp[cs].size(); i0 += kMaxBatch) {
      const int nb = (int)std::min<size_t>(kMaxBatch, grp[cs].size() - i0);
      Pack<JacArgs> pk{};
      for (int i = 0; i < nb; ++i) pk.a[i] = grp[cs][i0 + i];
      VP_TRY(launch_after(ctx, "jacobi_dw", kb_jacobi_dw, dim3(cs, nb), dim3(kJT),
                          std::max<size_t>(smem[cs], 116 * 1024),  // one CTA of the cluster per SM
                          st, dim3(cs), pk));
    }
  }
  return VP_OK;
}

}  // namespace vp
