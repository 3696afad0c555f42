// FP64 contractions on the tensor cores by exact slicing (the Ozaki scheme:
// K. Ozaki, T. Ogita, S. Oishi, S. Rump, "Error-free transformations of matrix
// multiplication by using fast routines of matrix multiplication and its
// applications", Numer. Algorithms 59 (2012); on FP16 tensor cores: D. Mukunoki
// et al., ISC High Performance 2020).
//
// GB300 issues two FP64 FMAs per SM and clock (1.26 TFLOP/s in all) and 4096
// FP16 ones on the tensor cores.  Every element of A and B becomes a fixed-point
// number of 56 bits relative to a power of two above its row's (A) or column's
// (B) largest magnitude within a K slice, cut into eight signed 7-bit digits,
//   a = 2^(e - 55) sum_i d_i 2^(7 (7 - i)),  -64 <= d_i <= 64,
// which are exact FP16 integers; -a has the digits -d_i.  Products of digits are at
// most 2^12, so the FP32 accumulator holds the sum of up to eight digit products over
// K <= 512 exactly (2^24).  The digit products with i + j = l, l = 0..8 (43 of the 64)
// accumulate into nine 128 x 48 accumulators of tensor memory, and the epilogue adds the
// nine integers with their weights exactly and rounds once to FP64, to nearest.  What is
// dropped (l > 8) is below 2^-60.4 of the two scales per product; an element is held to
// 2^-56 of its scale, and exactly from an eighth of the scale on.
//
// So a product is as accurate as its row's and column's largest elements make it,
// where an FP64 sum is as accurate as the products that meet in it: a row (1e20, 1,
// ..) against a column (0, 1, ..) loses every digit.  What the caller needs decides
// (OzBound):
//   OZ_ELEMENT  the kernel proves each element of each K slice or forms it again by FP64
//     FMAs.  Of its products n are nonzero, none off by more than 2^-56 + 2^-60.4 of the
//     scales' product; where (|A| |B|)_ij is W times that product, an FP64 sum may be off
//     by n 2^-53 W, so the element passes from W = 2180 / 2^14 = 0.133 on.  W is summed
//     from 7-bit magnitudes (of the first digits) that kb_oz_pack writes beside the digits
//     (four products an instruction, by four warps that would wait while the products
//     run): the first 32 k suffice where sizes are even (standard normal entries: W = 1.1
//     there, 0.2 where one outlier each doubles both scales), else all of them are
//     summed.  An element all of whose products are zero passes as well.
//   OZ_ROWS     nothing to prove: 2^-56 of the scales' product for each of K products.
//   OZ_COLS     kb_oz_kexp moves column k of A to one by a power of two, row k of B the
//     other way (exact), so that columns of A of any size keep their digits.
// Error against 64-bit references, standard normal entries: largest 0.14-0.5 times 2^-53
// (|A| |B|)_ij for K = 64..6147, the FMA kernel's 1.0 at K = 256; entries of exponents
// -70..70, where 97 of 100 elements stay open, 4-9 times 2^-53 (|A| |B|)_ij.
//
// Passes: kb_oz_kexp (OZ_COLS only), kb_oz_pack (digits, written as the
// 128-byte-swizzled shared-memory images of whole tiles, so that the loads are
// plain bulk copies), kb_oz_mma (a CTA per 128 x 48 tile and K slice; from kOzSums bytes
// of products on the slices that one CTA takes after the other, each adding to the sum in
// memory), and with several CTAs a tile kb_sum_slices, which adds what they leave in a
// fixed order.  The digits take 16 bytes an element; what needs more than kOzBand of them
// an operand goes band by band through the same memory.  The elements of
// a row or column that holds a NaN or Inf, or that scaling takes out of the exponent
// range, are FP64 FMAs as well, so non-finite values propagate as they do there.
//
// Measured (2048^3): 578 us in kb_oz_mma, 1.28 PFLOP/s of FP16 products, 68 % of the
// measured 1.88 (the 9-accumulator epilogue is not overlapped: the tile's accumulators
// fill tensor memory); kb_oz_pack 81 us, 25 bytes per element at 2.6 TB/s; the sum of
// four slices 38 us; whole call 738 us, 23 TFLOP/s of FP64 against 1.1 for the FMA kernel.
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <algorithm>

#include "common.cuh"
#include "tc.cuh"

namespace vp {
namespace {

constexpr int kOzS = 8;             // digits of an element
constexpr int kOzL = 9;             // accumulators: digit products i + j = 0 .. 8
constexpr int kOzM = 128, kOzN = 48, kOzKc = 64;  // tile rows, tile columns, K per stage
constexpr uint32_t kOzABytes = kOzM * 128;        // one digit of an A stage (128 bytes of K per row)
constexpr uint32_t kOzBDigit = kOzN * 128;        // one digit of a B stage
constexpr uint32_t kOzBBytes = kOzS * kOzBDigit;  // all digits of a B stage
constexpr int kOzAStages = kOzS;  // one slot per digit of a stage
constexpr int kOzMaxK = 512;        // K whose digit products one accumulator holds exactly
constexpr int kOzPackRows = 32;
constexpr uint32_t kOzTmem = 512;   // columns allocated (a power of two >= 9 x 48)
constexpr size_t kOzBand = size_t(1) << 30;  // bytes of an operand's digits at a time
constexpr size_t kOzSums = size_t(256) << 20;  // bytes that the CTAs of all tiles leave to be added
constexpr size_t kOzSmem = 1024 + 2 * (size_t)kOzBBytes + (size_t)kOzAStages * kOzABytes + 256;

__device__ __forceinline__ int oz_bexp(double x) { return (int)((__double_as_longlong(x) >> 52) & 0x7ff); }

// Exponent of x after its column's shift (0 for a zero, 2047 for a non-finite
// value, clamped into 1 .. 2047 otherwise: 2047 sends the row to the FP64 path).
__device__ __forceinline__ int oz_shifted_exp(double x, int sh) {
  const int e = oz_bexp(x);
  if (e == 2047) return 2047;
  if (x == 0.0) return 0;
  return min(max(max(e, 1) + sh, 1), 2047);
}

}  // namespace

struct OzJob {
  TcOperand a, b;        // a: M rows (tile rows), b: N rows (tile columns), both along K
  int M, N, K, kslice, slices, ranks, chunks;  // chunks: 64-wide K stages
  int swapped;           // the tile is C^T: element (i, j) goes to C[j * ldc + i]
  double alpha;
  double* C;
  int ldc;
  size_t stride;         // several ranks: rank s leaves its sums at C + s * stride
  int* kexp;             // OZ_COLS: per k, shift of a (b gets the opposite), else NULL
  int kside;             // the operand whose columns become one
  int* ea;               // slices x Mp exponents, then slices x Np
  int* eb;
  uint8_t* ma;           // OZ_ELEMENT: per slice and row kslice bytes, |element| in 128ths of
  uint8_t* mb;           // the scale, at most, + 128 where it is not zero; else NULL
  uint8_t* da;           // digit tiles
  uint8_t* db;
  DevStatus* st;
};

namespace {

// Shift of column k that brings its largest element to [1/2, 1).  One block of 32
// warps takes eight k, so that every load of an operand of up to a few hundred rows
// is in flight at once.
constexpr int kOzThreads = 1024;
__device__ __forceinline__ void oz_kexp_body(const OzJob& j, int kblk) {
  __shared__ int s[8];
  const int k0 = kblk * 8;
  if (threadIdx.x < 8) s[threadIdx.x] = 0;
  __syncthreads();
  const TcOperand& o = j.kside ? j.b : j.a;
  const int R = j.kside ? j.N : j.M;
  if (o.kind == 0) {  // k contiguous: eight k per row
    const int kk = threadIdx.x & 7, k = k0 + kk;
    int e = 0;
    if (k < j.K)
#pragma unroll 4
      for (int r = threadIdx.x >> 3; r < R; r += kOzThreads / 8) e = max(e, oz_bexp(o.p[(size_t)r * o.ld + k]));
    for (int off = 8; off < 32; off <<= 1) e = max(e, __shfl_xor_sync(0xffffffffu, e, off));
    if ((threadIdx.x & 31) < 8) atomicMax(&s[kk], e);
  } else {  // rows contiguous: four warps per k
    const int kk = threadIdx.x >> 7, k = k0 + kk;
    int e = 0;
    if (k < j.K) {
      const int rend = o.kind == 2 ? min(R, k + 1) : R;
#pragma unroll 8
      for (int r = threadIdx.x & 127; r < rend; r += 128) e = max(e, oz_bexp(o.p[(size_t)k * o.ld + r]));
    }
    e = __reduce_max_sync(0xffffffffu, e);
    if ((threadIdx.x & 31) == 0) atomicMax(&s[kk], e);
  }
  __syncthreads();
  if (threadIdx.x < 8 && k0 + threadIdx.x < j.K) {
    const int e = s[threadIdx.x], sh = e == 0 || e == 2047 ? 0 : 1022 - e;  // (zero or not finite: none)
    j.kexp[k0 + threadIdx.x] = j.kside ? -sh : sh;
  }
}

// Eight consecutive k of one row: eight digits each, one 16-byte store per digit, and
// (mag not NULL) eight bytes of magnitudes: with a first digit d, |x| is at least
// (|d| - 64 / 127) / 64 of the scale, 2 |d| - 2 of its 128ths.
__device__ __forceinline__ void oz_store_digits(const double (&x)[8], const int (&sh)[8], int emax, uint8_t* tile0,
                                                size_t digit_stride, int row, int kchunk16, uint8_t* mag) {
  constexpr long long kBias = 64ll * ((1ll << 49) - 1) / 127;  // 64 * sum_{j<7} 2^(7 j)
  unsigned long long X[8];  // bit 63: negative, bit 62: not zero
#pragma unroll
  for (int u = 0; u < 8; ++u) {
    const long long bits = __double_as_longlong(x[u]);
    const int e = (int)((bits >> 52) & 0x7ff);
    long long m = (bits & ((1ll << 52) - 1)) | (e ? 1ll << 52 : 0ll);
    const int s = emax - (max(e, 1) + sh[u]) - 2;  // right shift that puts 2^(emax - 1022) at 2^55
    if (s <= 0)
      m <<= -s;  // s >= -2: no element exceeds the row's largest
    else
      m = s <= 54 ? (m + (1ll << (s - 1))) >> s : 0ll;
    // (digits of the magnitude; the signs come last)
    X[u] = (unsigned long long)(m + kBias) | ((unsigned long long)bits & (1ull << 63)) | ((bits << 1) != 0 ? 1ull << 62 : 0ull);
  }
  if (mag) {
    unsigned w[2] = {0, 0};
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const unsigned hi = (unsigned)(X[u] >> 32), d = hi >> 17 & 127u;  // 64 at most
      w[u / 4] |= ((hi >> 23 & 128u) | (d > 1 ? 2 * d - 2 : 0u)) << (8 * (u % 4));
    }
    *reinterpret_cast<uint2*>(mag) = make_uint2(w[0], w[1]);
  }
  uint8_t* dst = tile0 + row * 128 + ((kchunk16 ^ (row & 7)) << 4);
  uint32_t sign[4];  // bits 15 and 31
#pragma unroll
  for (int h = 0; h < 4; ++h) sign[h] = __byte_perm((uint32_t)(X[2 * h] >> 32), (uint32_t)(X[2 * h + 1] >> 32), 0x7030) & 0x80008000u;
#pragma unroll
  for (int i = 0; i < kOzS; ++i) {
    uint32_t w[4];
#pragma unroll
    for (int h = 0; h < 4; ++h) {
      // 0x6400 | u is the FP16 number 1024 + u (u < 1024); digit = u - 64
      uint32_t lo, hi;
      if (i == 0) {
        lo = ((uint32_t)(X[2 * h] >> 49) & 127u) + 64;
        hi = ((uint32_t)(X[2 * h + 1] >> 49) & 127u) + 64;
      } else {
        lo = (uint32_t)(X[2 * h] >> (7 * (7 - i))) & 127u;
        hi = (uint32_t)(X[2 * h + 1] >> (7 * (7 - i))) & 127u;
      }
      const uint32_t raw = 0x64006400u | lo | (hi << 16);
      const __half2 d = __hsub2(*reinterpret_cast<const __half2*>(&raw), __float2half2_rn(1088.0f));
      w[h] = *reinterpret_cast<const uint32_t*>(&d) ^ sign[h];
    }
    *reinterpret_cast<uint4*>(dst + i * digit_stride) = make_uint4(w[0], w[1], w[2], w[3]);
  }
}

// Digits of 32 rows of one operand over one K slice: a thread holds up to two
// groups of eight k of one row, the largest exponent of the row is reduced over
// its threads, then the groups are converted from registers (one read).
__device__ __forceinline__ void oz_pack_body(const OzJob& j, int side, int rblk, int slice) {
  const TcOperand& o = side ? j.b : j.a;
  const int R = side ? j.N : j.M;
  const int tile_rows = side ? kOzN : kOzM;
  const int Rp = (R + tile_rows - 1) / tile_rows * tile_rows;
  const int row0 = rblk * kOzPackRows;
  if (row0 >= Rp) return;
  int* ex = side ? j.eb : j.ea;
  uint8_t* out = side ? j.db : j.da;
  const size_t dstride = side ? kOzBDigit : kOzABytes;
  const int kbeg = slice * j.kslice, kend = min(j.K, kbeg + j.kslice);
  const int kpad = min(j.chunks * kOzKc, kbeg + j.kslice);  // zero digits up to here
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int sgn = side ? -1 : 1;
  // a warp per row, lanes along k, so that every store fills whole sectors
  const int r = row0 + warp, g = lane;
  double x[2][8];
  if (o.kind == 0) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int k = kbeg + 8 * (g + 32 * h);
#pragma unroll
      for (int u = 0; u < 8; ++u) x[h][u] = r < R && k + u < kend ? o.p[(size_t)r * o.ld + k + u] : 0.0;
    }
  } else {
    // rows contiguous: read with the lanes along the rows and turned in shared
    // memory (row stride odd, one pad per eight k: both sides free of conflicts)
    extern __shared__ double turn[];
    const int P = j.kslice / 8 * 9 + 1;
    const int rr = row0 + lane;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int kk = 8 * (warp + 32 * h), k = kbeg + kk;
      if (kk >= j.kslice) continue;
      double y[8];
#pragma unroll
      for (int u = 0; u < 8; ++u)
        y[u] = rr < R && k + u < kend && !(o.kind == 2 && rr > k + u) ? o.p[(size_t)(k + u) * o.ld + rr] : 0.0;
#pragma unroll
      for (int u = 0; u < 8; ++u) turn[lane * P + kk / 8 * 9 + u] = y[u];
    }
    __syncthreads();
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int kk = 8 * (g + 32 * h);
#pragma unroll
      for (int u = 0; u < 8; ++u) x[h][u] = kk < j.kslice ? turn[warp * P + kk / 8 * 9 + u] : 0.0;
    }
  }
  int e = 1;
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int k = kbeg + 8 * (g + 32 * h);
#pragma unroll
    for (int u = 0; u < 8; ++u)
      if (k + u < kend) e = max(e, oz_shifted_exp(x[h][u], j.kexp ? sgn * j.kexp[k + u] : 0));
  }
  e = __reduce_max_sync(0xffffffffu, e);
  if (r >= Rp) return;
  if (g == 0) ex[(size_t)slice * Rp + r] = e;
  uint8_t* mags = side ? j.mb : j.ma;
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int k = kbeg + 8 * (g + 32 * h);
    if (k >= kpad) continue;
    int sh[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      sh[u] = j.kexp && k + u < kend ? sgn * j.kexp[k + u] : 0;
      if (e >= 2047) x[h][u] = 0.0;  // the row takes the FP64 path
    }
    oz_store_digits(x[h], sh, e,
                    out + ((size_t)(r / tile_rows) * j.chunks + k / kOzKc) * kOzS * dstride, dstride, r % tile_rows,
                    (k % kOzKc) >> 3, mags ? mags + ((size_t)slice * Rp + r) * j.kslice + (k - kbeg) : nullptr);
  }
}

__device__ __forceinline__ void bulk_load(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   smem_u32(dst)),
               "l"(src), "r"(bytes), "r"(smem_u32(bar))
               : "memory");
}

__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t (&r)[8]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr));
}

// sum_l S_l 2^(7 (8 - l)), |S_l| <= 2^24 exact integers, times 2^e2 as FP64, rounded
// once, to nearest: the sum in two 64-bit integers, of which 62 or more leading
// positions and a bit for all that lies below them (a plain shift would round every sum
// of 4 and more full-scale products down: up to an ulp, half of one on average) meet in
// T.  Integer arithmetic throughout, since the FP64 pipe takes two operations per SM
// and clock.
__device__ __forceinline__ double oz_combine(const int (&S)[kOzL], int e2) {
  const long long H = ((long long)S[0] << 21) + ((long long)S[1] << 14) + ((long long)S[2] << 7) + S[3];  // times 2^35
  const long long L = ((long long)S[4] << 28) + ((long long)S[5] << 21) + ((long long)S[6] << 14) +
                      ((long long)S[7] << 7) + S[8];
  // one product of two full-scale elements is 2^68, K <= 512 of them 2^77 (|H| < 2^42.1);
  // |L| < 2^52.1: below 2^27 H leaves room for all of L
  const int sh = max(0, 64 - __clzll(H < 0 ? -H : H) - 27);
  const long long T = ((H << (35 - sh)) + (L >> sh)) | ((L & ((1ll << sh) - 1)) != 0);  // |T| < 2^63
  const unsigned long long a = T < 0 ? 0ull - (unsigned long long)T : (unsigned long long)T;
  if (a == 0) return 0.0;
  const int lz = __clzll((long long)a);
  const unsigned long long top = a << lz;
  const unsigned long long m = (top + 1023ull + ((top >> 11) & 1ull));  // to nearest, ties to even
  // a carry out of the top bit: the mantissa is 2^53
  const unsigned long long m53 = m < top ? 1ull << 53 : m >> 11;
  const int be = 63 - lz + sh + e2 + 1023;
  if (be >= 1 && be < 2046) {
    const unsigned long long bits = m53 + ((unsigned long long)(be - 1) << 52) + ((unsigned long long)T & (1ull << 63));
    return __longlong_as_double((long long)bits);
  }
  const double v = scalbn((double)m53, be - 1023 - 52);  // subnormal or overflow
  return T < 0 ? -v : v;
}

// One 128 x 48 tile over a rank's K slices.  Warp 0: bulk copies (all digits of a B
// stage, double-buffered; the A digits of a stage one by one into their
// slots); warp 1: per A digit i the products with B digits 0 .. min(7, 8 - i),
// neighbouring B digits joined into one instruction of up to 240 columns, whose
// accumulators lie next to each other in tensor memory; warps 2 to 5: which elements
// are FP64 sums instead (oz_unproven); then all eight warps read the accumulators,
// combine and add.
// Columns of a tile (a bit each) whose element in the row with magnitudes at ma and
// exponent er is to be formed again (see OZ_ELEMENT above); mb, eb: the tile's columns,
// of which nc exist; kn of a slice's kslice magnitudes are there.
__device__ __forceinline__ unsigned long long oz_unproven(const uint8_t* ma, int er, const uint8_t* mb, const int* eb,
                                                          int nc, int kslice, int kn) {
  constexpr unsigned kEnough = 2180, kMag = 0x7f7f7f7fu, kAny = 0x80808080u;
  const int lane = threadIdx.x & 31;
  unsigned long long bad = (unsigned long long)__ballot_sync(0xffffffffu, lane < kOzN - 32 && eb[32 + lane % 16] >= 2047) << 32 |
                           __ballot_sync(0xffffffffu, eb[lane] >= 2047);
  if (er >= 2047) bad = (1ull << kOzN) - 1;
  if (!ma) return bad;
  // the columns' first 32 k into L1 in one go, for the loop below
  unsigned touch = 0;
#pragma unroll
  for (int c = lane; c < kOzN; c += 32) touch |= *reinterpret_cast<const unsigned*>(mb + (size_t)c * kslice);
  asm volatile("" ::"r"(touch));  // (the loads are for their lines alone)
  // four sums, so that an instruction need not wait for the one before
  auto add = [&](const uint4& a, const uint4& b, uint4& sum, unsigned& any) {
    sum.x = __dp4a(a.x & kMag, b.x & kMag, sum.x);
    sum.y = __dp4a(a.y & kMag, b.y & kMag, sum.y);
    sum.z = __dp4a(a.z & kMag, b.z & kMag, sum.z);
    sum.w = __dp4a(a.w & kMag, b.w & kMag, sum.w);
    any |= (a.x & b.x) | (a.y & b.y) | (a.z & b.z) | (a.w & b.w);
  };
  auto little = [&](const uint4& sum) { return sum.x + sum.y + sum.z + sum.w < kEnough; };
  const int words = kn / 16;
  uint4 mine[kOzMaxK / 16];
#pragma unroll
  for (int w = 0; w < 2; ++w) mine[w] = reinterpret_cast<const uint4*>(ma)[w];
  unsigned long long open = 0;
#pragma unroll 8
  for (int c = 0; c < kOzN; ++c) {
    const uint4* m = reinterpret_cast<const uint4*>(mb + (size_t)c * kslice);
    uint4 sum = make_uint4(0, 0, 0, 0);
    unsigned any = 0;
#pragma unroll
    for (int w = 0; w < 2; ++w) add(mine[w], m[w], sum, any);
    open |= (unsigned long long)little(sum) << c;
  }
  open &= ~bad & ((1ull << nc) - 1);
  if (__all_sync(0xffffffffu, open == 0)) return bad;
  // all k of the columns that any row has open; a row of zeros has none
  unsigned some = 0;
#pragma unroll
  for (int w = 0; w < kOzMaxK / 16; ++w) {
    if (w >= 2) mine[w] = w < words ? reinterpret_cast<const uint4*>(ma)[w] : make_uint4(0, 0, 0, 0);
    some |= mine[w].x | mine[w].y | mine[w].z | mine[w].w;
  }
  if (some == 0) open = 0;
  unsigned long long cols = (unsigned long long)__reduce_or_sync(0xffffffffu, (unsigned)open) |
                            (unsigned long long)__reduce_or_sync(0xffffffffu, (unsigned)(open >> 32)) << 32;
  for (; cols; cols &= cols - 1) {
    const int c = __ffsll((long long)cols) - 1;
    const uint4* m = reinterpret_cast<const uint4*>(mb + (size_t)c * kslice);
    uint4 sum = make_uint4(0, 0, 0, 0);
    unsigned any = 0;
#pragma unroll
    for (int w = 0; w < kOzMaxK / 16; ++w)
      if (w < words) add(mine[w], m[w], sum, any);
    bad |= (unsigned long long)(little(sum) && (any & kAny) != 0 && (open >> c & 1)) << c;
  }
  return bad;
}

// Where an operand's row r lies: element k at p[k * step], zero for k < first.
struct OzRow {
  const double* p;
  size_t step;
  int first;
};
__device__ __forceinline__ OzRow oz_row(const TcOperand& o, int r) {
  if (o.kind == 0) return {o.p + (size_t)r * o.ld, 1, 0};
  return {o.p + r, (size_t)o.ld, o.kind == 2 ? r : 0};
}
// FP64 sums over k in [kb, ke) of one row with columns [col, col + 8) (rows and columns
// beyond the operands: any value).
__device__ __forceinline__ void oz_plain(const OzJob& j, int row, int col, int kb, int ke, double (&t)[8]) {
  const OzRow a = oz_row(j.a, min(row, j.M - 1));
  OzRow b[8];
#pragma unroll
  for (int u = 0; u < 8; ++u) {
    b[u] = oz_row(j.b, min(col + u, j.N - 1));
    t[u] = 0.0;
  }
#pragma unroll 4
  for (int k = kb; k < ke; ++k) {
    const double x = k < a.first ? 0.0 : a.p[k * a.step];
#pragma unroll
    for (int u = 0; u < 8; ++u) t[u] = fma(x, k < b[u].first ? 0.0 : b[u].p[k * b[u].step], t[u]);
  }
}
// One such sum by a warp.
__device__ __forceinline__ double oz_plain_warp(const OzJob& j, int row, int col, int kb, int ke, int lane) {
  const OzRow a = oz_row(j.a, row), b = oz_row(j.b, col);
  double t = 0.0;
#pragma unroll 4
  for (int k = kb + lane; k < ke; k += 32)
    t = fma(k < a.first ? 0.0 : a.p[k * a.step], k < b.first ? 0.0 : b.p[k * b.step], t);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
  return t;
}

// MORE: a rank has several slices.
template <bool MORE>
__device__ __forceinline__ void oz_mma_body(const OzJob& j, int mt, int nt, int rank, int ranks) {
  extern __shared__ uint8_t oz_raw[];
  uint8_t* base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(oz_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* sB = base;
  uint8_t* sA = base + 2 * kOzBBytes;
  uint64_t* fullA = reinterpret_cast<uint64_t*>(sA + kOzAStages * kOzABytes);
  uint64_t* emptyA = fullA + kOzAStages;
  uint64_t* fullB = emptyA + kOzAStages;
  uint64_t* emptyB = fullB + 2;
  uint64_t* done = emptyB + 2;
  uint32_t* tmem_holder = reinterpret_cast<uint32_t*>(done + 1);
  __shared__ int s_abort;
  __shared__ unsigned long long s_bad[kOzM];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int m0 = mt * kOzM, n0 = nt * kOzN;
  const int Mp = (j.M + kOzM - 1) / kOzM * kOzM, Np = (j.N + kOzN - 1) / kOzN * kOzN;
  // an upper-triangular operand is zero for k below its first row
  int kskip = 0;
  if (j.a.kind == 2) kskip = m0;
  if (j.b.kind == 2) kskip = max(kskip, n0);
  const int cper = j.kslice / kOzKc;
  const int per = MORE ? (j.slices + ranks - 1) / ranks : 1, s0 = rank * per, s1 = MORE ? min(j.slices, s0 + per) : s0 + 1;

  if (tid == 0) {
    s_abort = 0;
    for (int s = 0; s < kOzAStages; ++s) {
      mbar_init(&fullA[s], 1);
      mbar_init(&emptyA[s], 1);
    }
    for (int s = 0; s < 2; ++s) {
      mbar_init(&fullB[s], 1);
      mbar_init(&emptyB[s], 1);
    }
    mbar_init(done, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  __syncwarp();
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_holder)),
                 "r"(kOzTmem)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_holder;
  bool ok = true;
  bool first = true;  // (later slices add to what the one before left in C)
  double* C = j.C + rank * j.stride;
  auto put = [&](int i, int col, double v) {
    if (i >= j.M || col >= j.N) return;
    double* c = C + (j.swapped ? (size_t)col * j.ldc + i : (size_t)i * j.ldc + col);
    *c = !MORE || first ? v : *c + v;
  };
  int na = 0, nb = 0;  // A digits and B stages issued, or B stages taken (warp 1)
  int phase = 0;
  for (int slice = s0; slice < s1; ++slice) {
    const int c1 = min(j.chunks, (slice + 1) * cper), c0 = min(c1, max(slice * cper, kskip / kOzKc));
    if (c0 >= c1) continue;  // a K range of exact zeros
    const int* ea = j.ea + (size_t)slice * Mp + m0;
    const int* eb = j.eb + (size_t)slice * Np + n0;
    if (warp == 0 && lane == 0) {
      const uint8_t* ga = j.da + (size_t)mt * j.chunks * kOzS * kOzABytes;
      const uint8_t* gb = j.db + (size_t)nt * j.chunks * kOzBBytes;
      for (int c = c0; c < c1 && ok; ++c) {
        const int sb = nb & 1;
        if (nb >= 2 && !mbar_wait(&emptyB[sb], ((nb >> 1) - 1) & 1)) {
          ok = false;
          break;
        }
        mbar_expect_tx(&fullB[sb], kOzBBytes);
        bulk_load(sB + sb * kOzBBytes, gb + (size_t)c * kOzBBytes, kOzBBytes, &fullB[sb]);
        ++nb;
        for (int i = 0; i < kOzS; ++i) {
          const int sa = na % kOzAStages;
          if (na >= kOzAStages && !mbar_wait(&emptyA[sa], ((na / kOzAStages) - 1) & 1)) {
            ok = false;
            break;
          }
          mbar_expect_tx(&fullA[sa], kOzABytes);
          bulk_load(sA + sa * kOzABytes, ga + ((size_t)c * kOzS + i) * kOzABytes, kOzABytes, &fullA[sa]);
          ++na;
        }
      }
      // every issued copy lands before the CTA can exit
      for (int q = max(0, nb - 2); q < nb; ++q)
        if (!mbar_wait(&fullB[q & 1], (q >> 1) & 1)) ok = false;
      for (int q = max(0, na - kOzAStages); q < na; ++q)
        if (!mbar_wait(&fullA[q % kOzAStages], (q / kOzAStages) & 1)) ok = false;
    } else if (warp == 1 && lane == 0) {
      // everything but the stage is a constant of the unrolled loops: a descriptor
      // built at run time costs more issue slots than the smaller products take
      const uint64_t a_desc = sw128_desc(smem_u32(sA)), b_desc = sw128_desc(smem_u32(sB));
      for (int c = c0; c < c1 && ok; ++c, ++nb) {
        const int sb = nb & 1;
        if (!mbar_wait(&fullB[sb], (nb >> 1) & 1)) {
          ok = false;
          break;
        }
        const uint64_t bd = b_desc + (uint32_t)sb * (kOzBBytes >> 4);
        const uint32_t later = c > c0 ? 1u : 0u;
#pragma unroll
        for (int i = 0; i < kOzS; ++i) {
          if (ok && !mbar_wait(&fullA[i], nb & 1)) ok = false;
          if (!ok) continue;
          tc_fence_after();
          constexpr int kW[kOzS][3] = {{5, 3, 0}, {5, 2, 1}, {5, 2, 0}, {5, 1, 0}, {5, 0, 0}, {4, 0, 0}, {3, 0, 0}, {2, 0, 0}};
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            // accumulators are first written by digit 0 (0 .. 7) and by the pair (1, 7) (8)
            int q = 0;
#pragma unroll
            for (int part = 0; part < 3; ++part) {
              const int w = kW[i][part];
              if (w == 0) continue;
              const bool opens = k == 0 && (i == 0 || (i == 1 && part == 2));
              tc_mma<true>(tmem + (i + q) * kOzN, a_desc + i * (kOzABytes >> 4) + 2 * k, bd + q * (kOzBDigit >> 4) + 2 * k,
                           tc_idesc(0, w * kOzN), opens ? later : 1u);
              q += w;
            }
          }
          tc_commit(&emptyA[i]);
        }
        if (ok) tc_commit(&emptyB[sb]);
      }
      tc_commit(done);
    } else if (warp >= 2 && warp < 6) {
      const int r = tid - 64;
      const size_t rec = (size_t)j.kslice, ra = (size_t)slice * Mp + m0 + r, rb = (size_t)slice * Np + n0;
      s_bad[r] = j.ma ? oz_unproven(j.ma + ra * rec, ea[r], j.mb + rb * rec, eb, min(kOzN, j.N - n0), j.kslice,
                                      min(j.kslice, j.chunks * kOzKc - slice * j.kslice))
                        : oz_unproven(nullptr, ea[r], nullptr, eb, 0, 0, 0);
    }
    if (!ok) atomicExch(&s_abort, 1);
    __syncwarp();
    __syncthreads();

    const bool got = mbar_wait(done, phase);
    phase ^= 1;
    const int good = __syncthreads_and(got && s_abort == 0);
    tc_fence_after();
    if (!good) {
      if (tid == 0) atomicCAS(&j.st->err, 0, 1);
      break;
    }
    // warp w reads lanes 32 (w mod 4) .., the column groups of 8 with (w / 4)
    const int row = (warp & 3) * 32 + lane;
    const int er = ea[row], kb = c0 * kOzKc, ke = min(j.K, c1 * kOzKc);
    const unsigned long long bad = s_bad[row];
#pragma unroll 1
    for (int g = warp >> 2; g < kOzN / 8; g += 2) {
      uint32_t r[kOzL][8];
#pragma unroll
      for (int l = 0; l < kOzL; ++l)
        tmem_ld8(tmem + (static_cast<uint32_t>((warp & 3) * 32) << 16) + l * kOzN + 8 * g, r[l]);
      asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        int S[kOzL];
#pragma unroll
        for (int l = 0; l < kOzL; ++l) S[l] = __float2int_rn(__uint_as_float(r[l][u]));
        const int col = 8 * g + u;
        // digit products carry 2^(7 (14 - l)); scales 2^(er - 1022 - 55), 2^(ec - 1022 - 55)
        double v = oz_combine(S, er + eb[col] - 2 * 1077 + 42);
        if (j.alpha != 1.0) v *= j.alpha;
        if (!(bad >> col & 1)) put(m0 + row, n0 + col, v);
      }
      // the elements that were not proven: few one by one, more as the whole group of
      // 32 x 8 (the FP64 pipe takes 16 clocks a warp's FMA: at K = 512 the group's 8 per k
      // cost as much as some 16 elements one by one)
      const int i0 = m0 + (warp & 3) * 32;
      const unsigned mine =
          m0 + row < j.M ? (unsigned)(bad >> (8 * g)) & 255u & ((1u << min(8, max(0, j.N - n0 - 8 * g))) - 1) : 0u;
      unsigned rows = __ballot_sync(0xffffffffu, mine != 0);
      if (__reduce_add_sync(0xffffffffu, __popc(mine)) > 16) {
        double t[8];
        oz_plain(j, m0 + row, n0 + 8 * g, kb, ke, t);
#pragma unroll
        for (int u = 0; u < 8; ++u)
          if (mine >> u & 1) put(m0 + row, n0 + 8 * g + u, j.alpha * t[u]);
        rows = 0;
      }
      for (; rows; rows &= rows - 1) {
        const int l = __ffs(rows) - 1;
        for (unsigned us = __shfl_sync(0xffffffffu, mine, l); us; us &= us - 1) {
          const int u = __ffs(us) - 1;
          const double t = oz_plain_warp(j, i0 + l, n0 + 8 * g + u, kb, ke, lane);
          if (lane == 0) put(i0 + l, n0 + 8 * g + u, j.alpha * t);
        }
      }
    }
    first = false;
    tc_fence_before();
    __syncthreads();  // the accumulators are read
    tc_fence_after();
  }

  if (first)  // nothing but slices of exact zeros
    for (int e = tid; e < kOzM * kOzN; e += 256) put(m0 + e / kOzN, n0 + e % kOzN, 0.0);
  tc_fence_before();
  __syncthreads();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kOzTmem) : "memory");
}

__global__ void __launch_bounds__(kOzThreads) kb_oz_kexp(const __grid_constant__ Pack<OzJob> pk) {
  follow();
  const OzJob& j = pk.a[blockIdx.y];
  if (!j.kexp || (int)blockIdx.x * 8 >= j.K) return;
  oz_kexp_body(j, blockIdx.x);
}
// x: 32-row blocks of A, then of B (ablk of A at most); y: K slice; z: job
__global__ void __launch_bounds__(kOzThreads) kb_oz_pack(const __grid_constant__ Pack<OzJob> pk, int ablk) {
  follow();
  const OzJob& j = pk.a[blockIdx.z];
  if ((int)blockIdx.y >= j.slices) return;
  const int side = (int)blockIdx.x >= ablk;
  oz_pack_body(j, side, (int)blockIdx.x - (side ? ablk : 0), blockIdx.y);
}
// z: job x rank (of at most zs)
template <bool MORE>
__global__ void __launch_bounds__(256, 1) kb_oz_mma(const __grid_constant__ Pack<OzJob> pk, int zs) {
  follow();
  const OzJob& j = pk.a[blockIdx.z / zs];
  const int rank = blockIdx.z % zs;
  if (rank >= j.ranks || (int)blockIdx.x * kOzM >= j.M || (int)blockIdx.y * kOzN >= j.N) return;
  oz_mma_body<MORE>(j, blockIdx.x, blockIdx.y, rank, j.ranks);
}

size_t oz_pack_smem(int kslice) { return (size_t)kOzPackRows * (kslice / 8 * 9 + 1) * sizeof(double); }
long long tiles_of(int M, int N) { return (long long)((M + kOzM - 1) / kOzM) * ((N + kOzN - 1) / kOzN); }

}  // namespace

// Which FP64 contractions are sliced.  Two launches of ~14 + 26 us at the smallest
// sizes stand against the FMA kernel's 2 M N K / 1.1 TFLOP/s: whole vp_gemm calls on
// GB300, sliced / FMA, us: 320 x 256 x 256 (M N K = 2.1e7) 56 / 86, 300^3 59 / 99, 512 x
// 324 x 256 (4.3e7) 62 / 135, 341 x 1008 x 503 (1.7e8) 65 / 430, 128 x 6784 x 6147 (5.3e9)
// 870 / 12300 (operands whose elements the proof leaves open: 300^3 320, 341 x 1008 x 503
// 560, 128 x 6784 x 6147 15300), and 256^3 (1.7e7) 61 on the FMA kernel; the line is drawn
// at 2e7.  Below K = 64 (one stage) or 16 rows or columns most of a tile would be padding;
// so would a shape that fills less than a quarter of its tiles in the better of the two
// orientations; and from K = 524288 on a band of one tile's rows would take more than
// kOzBand.  K is cut into slices of at most 512, where the accumulators stop being exact,
// and into at least as many as fill the SMs with tiles once (128 of K each, two stages); a
// CTA takes one, while what they leave to be added stays below kOzSums.  (Slices added in
// registers, or over the CTAs of a cluster, took 5 to 15 us longer a product than a CTA
// each and the launch that adds.)
OzPlan oz_plan(const vp_ctx* ctx, int M, int N, int K) {
  OzPlan p{0, 0, 1, 0, 1};
  if (K < 64 || K >= 1 << 19 || std::min(M, N) < 16 || (double)M * N * K < 2e7) return p;
  const long long t = tiles_of(M, N), ts = tiles_of(N, M);
  p.swapped = ts < t;
  const long long tiles = std::min(t, ts);
  // partial tiles compute their padding: not worth it where most of it is
  if ((double)tiles * kOzM * kOzN > 4.0 * M * N) return p;
  const int chunks = (K + kOzKc - 1) / kOzKc, most = kOzMaxK / kOzKc;
  int sl = (K + kOzMaxK - 1) / kOzMaxK;
  sl = std::max<long long>(sl, std::min<long long>(ctx->num_sms / tiles, (chunks + 1) / 2));
  const int per = std::min(most, (chunks + sl - 1) / sl);
  p.use = 1;
  p.kslice = per * kOzKc;
  p.slices = (chunks + per - 1) / per;
  const long long held = std::max(1ll, (long long)kOzSums / (8ll * M * N));
  const int rounds = (int)((p.slices + held - 1) / held);  // slices a CTA
  p.ranks = (p.slices + rounds - 1) / rounds;
  return p;
}

namespace {

// Scratch of a product in doubles: A's digits, the magnitudes, exponents and shifts;
// B's digits.
void oz_scratch(const OzGemm& g, size_t& wa, size_t& wb) {
  const size_t M = g.plan.swapped ? g.N : g.M, N = g.plan.swapped ? g.M : g.N;
  const size_t Mp = (M + kOzM - 1) / kOzM * kOzM, Np = (N + kOzN - 1) / kOzN * kOzN;
  const size_t chunks = (g.K + kOzKc - 1) / kOzKc, rec = g.bound == OZ_ELEMENT ? g.plan.kslice : 0;
  const size_t ints = (size_t)g.K + g.plan.slices * (Mp + Np);
  wa = (Mp / kOzM * chunks * kOzS * kOzABytes + g.plan.slices * (Mp + Np) * rec) / 8 + ints / 2 + 64;
  wb = Np / kOzN * chunks * kOzBBytes / 8 + 64;
}

template <bool MORE>
int launch_oz(vp_ctx* ctx, cudaStream_t st, const std::vector<OzGemm>& v) {
  static AttrOnce attr, pattr;
  VP_TRY(attr.ensure(ctx, (const void*)kb_oz_mma<MORE>, (int)kOzSmem, false));
  VP_TRY(pattr.ensure(ctx, (const void*)kb_oz_pack, (int)oz_pack_smem(kOzMaxK), false));
  for (size_t i0 = 0; i0 < v.size(); i0 += kMaxBatch) {
    const int nb = (int)std::min<size_t>(kMaxBatch, v.size() - i0);
    Pack<OzJob> pk{};
    int ks = 1, ablk = 1, bblk = 1, slices = 1, zs = 1, gx = 1, gy = 1, ksl = kOzKc;
    bool shifts = false;
    for (int i = 0; i < nb; ++i) {
      const OzGemm& g = v[i0 + i];
      OzJob& j = pk.a[i];
      j.a = g.plan.swapped ? g.b : g.a;
      j.b = g.plan.swapped ? g.a : g.b;
      j.M = g.plan.swapped ? g.N : g.M;
      j.N = g.plan.swapped ? g.M : g.N;
      j.K = g.K;
      j.kslice = g.plan.kslice;
      j.slices = g.plan.slices;
      j.ranks = g.plan.ranks;
      j.chunks = (g.K + kOzKc - 1) / kOzKc;
      j.swapped = g.plan.swapped;
      j.alpha = g.alpha;
      j.C = g.C;
      j.ldc = g.ldc;
      j.stride = g.stride;
      j.st = g.st;
      const size_t Mp = (size_t)(j.M + kOzM - 1) / kOzM * kOzM, Np = (size_t)(j.N + kOzN - 1) / kOzN * kOzN;
      const size_t abytes = Mp / kOzM * j.chunks * kOzS * kOzABytes;
      // magnitudes of OZ_ELEMENT, on 16-byte boundaries behind the digits
      const size_t rec = g.bound == OZ_ELEMENT ? (size_t)j.kslice : 0, mbytes = j.slices * (Mp + Np) * rec;
      // bulk copies start on 16-byte boundaries, whatever the allocator's alignment
      auto aligned = [](double* p) { return reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(p) + 127) & ~uintptr_t(127)); };
      j.da = aligned(g.wa->p);
      j.db = aligned(g.wb->p);
      j.ma = rec ? j.da + abytes : nullptr;
      j.mb = rec ? j.ma + j.slices * Mp * rec : nullptr;
      j.ea = reinterpret_cast<int*>(j.da + abytes + mbytes);
      j.eb = j.ea + (size_t)j.slices * Mp;
      if (g.bound == OZ_COLS || g.bound == OZ_COLS_B) {
        j.kexp = j.eb + (size_t)j.slices * Np;
        j.kside = (g.bound == OZ_COLS_B) != (j.swapped != 0);
        ks = std::max(ks, (j.K + 7) / 8);
        shifts = true;
      }
      ablk = std::max(ablk, (int)((Mp + kOzPackRows - 1) / kOzPackRows));
      bblk = std::max(bblk, (int)((Np + kOzPackRows - 1) / kOzPackRows));
      slices = std::max(slices, j.slices);
      zs = std::max(zs, j.ranks);
      ksl = std::max(ksl, j.kslice);
      gx = std::max(gx, (int)(Mp / kOzM));
      gy = std::max(gy, (int)(Np / kOzN));
    }
    if (shifts)
      VP_TRY(launch_after(ctx, "oz_kexp", kb_oz_kexp, dim3(ks, nb), dim3(kOzThreads), 0, st, kNoCluster, pk));
    VP_TRY(launch_after(ctx, "oz_pack", kb_oz_pack, dim3(ablk + bblk, slices, nb), dim3(kOzThreads), oz_pack_smem(ksl),
                        st, kNoCluster,
                        pk, ablk));
    VP_TRY(launch_after(ctx, "oz_mma", kb_oz_mma<MORE>, dim3(gx, gy, nb * zs), dim3(256), kOzSmem, st, kNoCluster, pk, zs));
  }
  return VP_OK;
}

}  // namespace

int blaunch_oz_gemm(vp_ctx* ctx, cudaStream_t st, const std::vector<OzGemm>& v) {
  std::vector<OzGemm> sliced, one, more, fma;  // a slice a CTA, or several
  for (const OzGemm& g : v) {
    if (!g.plan.use) {
      fma.push_back(g);
      continue;
    }
    if (g.N > kGemmMaxN) return fail(ctx, VP_ECAPACITY, "gemm: N too large");
    // rows of A and of B in bands whose digits fit (a million of them at K = 64: 22000 tiles)
    const long long fit = (long long)(kOzBand / 16) / ((g.K + kOzKc - 1) / kOzKc * kOzKc) / kOzM * kOzM;
    if (g.M > fit || g.N > fit) {
      const int mb = (int)((g.M + fit - 1) / fit), nb = (int)((g.N + fit - 1) / fit);
      const int mr = ((g.M + mb - 1) / mb + kOzM - 1) / kOzM * kOzM, nr = ((g.N + nb - 1) / nb + kOzM - 1) / kOzM * kOzM;
      for (int m0 = 0; m0 < g.M; m0 += mr)
        for (int n0 = 0; n0 < g.N; n0 += nr) {
          OzGemm s = g;
          s.M = std::min(mr, g.M - m0);
          s.N = std::min(nr, g.N - n0);
          s.C = g.C + (size_t)m0 * g.ldc + n0;
          const int k0 = g.a.kind == 2 ? m0 : 0;  // a triangle below row m0: from its column m0 on
          s.K = g.K - k0;
          s.a.p += g.a.kind == 0 ? (size_t)m0 * g.a.ld : (size_t)k0 * g.a.ld + m0;
          s.b.p += g.b.kind == 0 ? (size_t)n0 * g.b.ld + k0 : (size_t)k0 * g.b.ld + n0;
          s.plan = oz_plan(ctx, s.M, s.N, s.K);
          VP_TRY(blaunch_oz_gemm(ctx, st, {s}));  // in turn: the bands share the scratch
        }
      continue;
    }
    sliced.push_back(g);
  }
  // scratch of every product before the first launch; without it: FMAs
  const std::string err = ctx->err;
  std::vector<OzSum> sums;
  for (OzGemm g : sliced) {
    size_t wa, wb;
    oz_scratch(g, wa, wb);
    const size_t stride = (size_t)g.M * g.N;
    if (reserve(ctx, *g.wa, wa) != VP_OK || reserve(ctx, *g.wb, wb) != VP_OK ||
        (g.plan.ranks > 1 && reserve(ctx, *g.wsum, stride * g.plan.ranks) != VP_OK)) {
      ctx->err = err;
      fma.push_back(g);
      continue;
    }
    if (g.plan.ranks > 1) {
      sums.push_back({g.wsum->p, g.M, g.N, g.plan.ranks, stride, g.C, g.ldc});
      g.C = g.wsum->p;
      g.ldc = g.N;
      g.stride = stride;
    }
    (g.plan.slices > g.plan.ranks ? more : one).push_back(g);
  }
  VP_TRY(launch_oz<false>(ctx, st, one));
  VP_TRY(launch_oz<true>(ctx, st, more));
  VP_TRY(blaunch_sum_slices(ctx, st, sums));
  return blaunch_fma_gemm(ctx, st, fma);
}

}  // namespace vp
