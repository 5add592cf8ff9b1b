// Block Gram matrices of the mixed policy on the tensor cores (tcgen05, accumulators in TMEM).
//
// The sums of k_gram_df (dense.cu) - GM = S^* M S through the bidiagonal factor of the mass matrix
// and GA = (C S)^* W (C S) - are products P = V V^T of real operands V, rows (trial column,
// component), columns mesh nodes:
//   GM: v = z_x and z_y, z_x = sqrt(mx)(alpha x(i,j) + beta x(i,j+1)), z_y likewise along i;
//   GA: v = sqrt(w) curl.
// Each operand value is brought to a fixed-point integer relative to a power of two that bounds its
// trial column's operands (k_gram_exponents: sqrt(mx) |x| and sqrt(my) |y| for GM, sqrt(w) |curl| for
// GA), of 48 bits (GM) or 49 (GA), and cut into six signed digits of 8 bits (GA's first: nine), held as
// binary16 integers.  A digit product is exact in the tensor core's FP32 sums: P = sum over digit pairs
// i + j <= 6, and those with i odd and i + j = 7, of P_ij 2^{-8(i+j)} (the error-free splitting of
// Ozaki, Ogita, Oishi and Rump, 2012).  256 nodes add at most 2 x 512 x 2^14 = 2^24 to a sum of equal
// i + j <= 3 (GA, one product per node: 256 x 2^16 for two ninth bits, and 2 x 256 x 2^15), so FP32
// sums of 256 nodes are exact; they are then taken out of TMEM and added up as 64-bit integers, in
// units that leave the CTA's chunks their room (2^-46 to 2^-53 of the scales).  What is left is the
// rounding of the operands, 2^-48 (GM) and 2^-49 (GA) of a power of two up to four times the column's
// largest operand; the double-float kernel rounds each value to 2^-47 of itself, and its curls to 2^-47
// of the edge values they are differences of, always towards zero.  Largest errors relative to
// sqrt(G_aa G_bb), 32 x 48 / 128 x 96, 12 columns, h2/h1 from 1/64 to 64: noise 1.2e-15 / 5e-16, smooth
// fields 8e-16 / 4e-16 in GM and 1.6e-15 / 1.9e-15 (curls of 1/20 of their edges' size) in GA;
// double-float 1.9e-15 / 3.4e-15, 2.6e-15 / 4.6e-15 and 2.9e-15 / 3.5e-15.  What matters for that:
//  * the pairs (2, 4) and (4, 2), 2^-48 of the scales each (without them 6e-15 to 1e-14 for noise and
//    6e-14 for smooth curls);
//  * both fields' operands at full scale: edge values are line integrals, |y| / |x| of a smooth field
//    is about h2/h1, and relative to a bound of the unweighted values the dropped pairs weigh
//    (h2/h1)^2 times as much (2.4e-13 for smooth fields at h2/h1 = 16, 3.8e-12 at 64);
//  * inputs rounded down, what that takes given back by a constant (cut off towards zero they left a
//    bias of 1e-15 to 2e-15 on the diagonal; eight bits more for them cost 2 % of the kernel);
//  * GA's ninth bit: its operands are rounded, not its values, and the weights spread them (without it
//    1.3e-15 to 2e-15 for noise on 32 x 48, now 6e-16 to 7e-16).
// None of the four shows in the time: 1024 x 1024, q = 30: 1.26 ms, q = 42: 4.1.
//
// Digits come from integers, not from double-float: FP64 input is shifted into 64-bit fixed point
// (the curl's differences are then exact), multiplied by 63-bit constants, and a byte permutation
// with the exponent byte of 1024 turns a digit into a binary16 number.  About 200 integer
// instructions per node, column and matrix against 79 floating-point ones per node and entry of
// the matrix (q (q + 1) / 2 of them) in k_gram_df.
//
// One CTA per SM (shared memory) owns a pair (I <= J) of 32-column blocks of GM or of GA (blockIdx.z)
// and every npart-th chunk of 32 nodes x 8 mesh rows.  16 producer warps fill a ring of 32-node stages; one
// thread of a 17th warp issues the MMAs (A = two digits of block I, 128 rows; B = up to four
// digits of block J, 64 rows each; K-major, no swizzle); after each chunk the producers read
// TMEM.  Accumulator D_t (t = 0 .. 6, 128 rows x 64 columns) holds the pairs i + j = t of even i in
// rows 0-63 and i + j = t + 1 of odd i in rows 64-127: A = digits (2 u, 2 u + 1), B = digit t - 2 u.
// For I = J the product is symmetric, even-odd pairs are the transposes of odd-even ones, and the
// rows 0-63 of odd t are not used.
#include <algorithm>
#include <cmath>
#include <cstdlib>
#include <cstring>

#include "internal.h"
#include "tc.cuh"

namespace pbs {

namespace {

constexpr int kProducers = 512;            // producer and epilogue threads (16 warps)
constexpr int kThreads = kProducers + 32;  // and the warp whose first lane issues the MMAs
constexpr int kCols = 32;                  // trial columns per block: 64 operand rows
constexpr int kSlices = 6;
constexpr int kRows = 64 * kSlices;        // operand rows of a block in shared memory, digit-major
constexpr int kChunk = 256, kStage = 32;   // nodes per TMEM sum (gram_tc_chunks), per ring stage
static_assert(kStage == 32 && kChunk == 8 * kStage, "gram_tc_chunks counts tiles of 32 x 8 nodes");
constexpr int kOctet = kRows * 16;         // bytes of 8 nodes of a block's rows
constexpr int kArray = kStage / 8 * kOctet;
constexpr int kSmem = 196608 + 1024;       // ring and barriers
constexpr unsigned kTmemCols = 512;

// ---- fixed point ----------------------------------------------------------------
// A factor 0 <= f < 1 as (hi + lo 2^-31) 2^-31.
struct Fix {
  int hi, lo;
};
inline Fix make_fix(double f) {
  Fix r;
  const double s = f * 2147483648.0;
  r.hi = (int)s;
  r.lo = (int)((s - (double)r.hi) * 2147483648.0);
  return r;
}
// v 2^{52 - E}, |v| < 2^{E+1}, E > kMinExp, rounded down to an integer (one unit off where v is zero or
// subnormal, exponent field 0, and its sign is set).  Down, not towards zero: that pulls in every value,
// which adds up on the diagonal of a Gram (1e-15 to 2e-15 for noise), where half a unit of all alike is
// taken back by the constants of digits1 and digits2.
__device__ __forceinline__ long long to_fixed(double v, int E) {
  const int hi = __double2hiint(v), sh = min(E + 1023 - ((hi >> 20) & 0x7FF), 63);  // at least 0
  const long long m = ((long long)((hi & 0xFFFFF) | 0x100000) << 32) | (unsigned)__double2loint(v);
  const long long s = (long long)(hi >> 31);
  return ((m ^ s) - s) >> sh;
}
// Operand digits of z rounded to the nearest integer: six bytes that carry 0x80 too much each, and in
// digits1 a ninth bit of the first digit, which carries 0x100 too much.  digits1: z = X f / 16,
// |z| < 0.99 2^48; digits2: z = (X f + Y g) / 32, |z| < 0.99 2^47.  h f.hi is exact; the high products
// (and X, Y) are rounded down, by 1.7 units of 2^-3 on average in digits1 and 3.2 of 2^-4 in digits2, which
// comes on top of the half that rounds to nearest (4 + 2, 8 + 3).
constexpr long long kDigitBias = 0x808080808080ll * 16 + 8 + 3, kDigitBias9 = 0x1008080808080ll * 8 + 4 + 2;
__device__ __forceinline__ unsigned long long digits1(long long X, Fix f) {
  const int h = (int)(X >> 32);
  const long long t = (long long)h * f.hi + kDigitBias9 + (long long)__umulhi((unsigned)X, (unsigned)f.hi);
  return (unsigned long long)(t + 2 * (long long)__mulhi(h, f.lo)) >> 3;
}
__device__ __forceinline__ unsigned long long digits2(long long X, Fix f, long long Y, Fix g) {
  const int h = (int)(X >> 32), k = (int)(Y >> 32);
  const long long t = (long long)h * f.hi + ((long long)k * g.hi + kDigitBias);
  const unsigned l = __umulhi((unsigned)X, (unsigned)f.hi) + __umulhi((unsigned)Y, (unsigned)g.hi);  // below 2^32
  return (unsigned long long)(t + (long long)l + 2 * (long long)(__mulhi(h, f.lo) + __mulhi(k, g.lo))) >> 4;
}

// Operand values of two neighbouring nodes and one component (biased digits b0, b1): stores digit s
// of both at base + 1024 s (64 rows of 16 bytes) as two binary16 integers -128 .. 127 (the first digit
// of nine bits: -256 .. 255).  A byte next to the byte 0x64 is the binary16 number 1024 + byte.
template <bool NINE> __device__ __forceinline__ void store_digits(unsigned base, unsigned long long b0, unsigned long long b1) {
  const unsigned l0 = (unsigned)b0, h0 = (unsigned)(b0 >> 32), l1 = (unsigned)b1, h1 = (unsigned)(b1 >> 32);
  const __half2 bias = __halves2half2(__ushort_as_half(0x6480), __ushort_as_half(0x6480));  // 1024 + 128
  auto put = [&](int s, unsigned two) {
    const __half2 d = __hsub2(*reinterpret_cast<const __half2*>(&two), bias);
    asm volatile("st.shared.b32 [%0], %1;" ::"r"(base + 1024u * s), "r"(*reinterpret_cast<const unsigned*>(&d)) : "memory");
  };
  // (byte i, byte i + 1 of both words), then each pair with the exponent byte
  const unsigned t45 = __byte_perm(h0, h1, 0x5140), t23 = __byte_perm(l0, l1, 0x7362), t01 = __byte_perm(l0, l1, 0x5140);
  if (NINE) {
    const unsigned two = __byte_perm(h0, h1, 0x6521) | 0x64006400u;
    const __half2 bias9 = __halves2half2(__ushort_as_half(0x6500), __ushort_as_half(0x6500));  // 1024 + 256
    const __half2 d = __hsub2(*reinterpret_cast<const __half2*>(&two), bias9);
    asm volatile("st.shared.b32 [%0], %1;" ::"r"(base), "r"(*reinterpret_cast<const unsigned*>(&d)) : "memory");
  } else {
    put(0, __byte_perm(t45, 0x64646464u, 0x4342));
  }
  put(1, __byte_perm(t45, 0x64646464u, 0x4140));
  put(2, __byte_perm(t23, 0x64646464u, 0x4342));
  put(3, __byte_perm(t23, 0x64646464u, 0x4140));
  put(4, __byte_perm(t01, 0x64646464u, 0x4342));
  put(5, __byte_perm(t01, 0x64646464u, 0x4140));
}

// Bloch continuation of a value across the level's boundary, out of line: its FP64 products are
// otherwise evaluated (predicated) for every value, and the FP64 pipe is narrow.
__device__ __noinline__ double2 rotate(double2 v, double2 phase) { return cmul(v, phase); }

__device__ __forceinline__ const double2* trial_col(const Roles& R, int g, int a) {
  const int r = a / R.pr;
  const double2* base = r == 0 ? R.b[0] : (r == 1 ? R.b[1] : R.b[2]);
  return base + ((long)g * R.pr + a % R.pr) * R.ld;
}

// x-edges of two neighbouring nodes (i even; i + 1 on the same mesh row) on mesh row j <= m, y-edges of
// the two and the next node on row j < m; Bloch-continued.
struct PairX {
  double2 v[2];
};
struct PairY {
  double2 v[3];
};
__device__ __forceinline__ PairX load_x(const double2* __restrict__ X, int i, int j, int n, int m, const double2& be,
                                        bool in) {
  PairX p;
  p.v[0] = p.v[1] = make_double2(0.0, 0.0);
  if (in) {
    const double2* a = X + (long)(j == m ? 0 : j) * n + i;
    p.v[0] = a[0];
    p.v[1] = a[1];
    if (j == m) {
      p.v[0] = rotate(p.v[0], be);
      p.v[1] = rotate(p.v[1], be);
    }
  }
  return p;
}
__device__ __forceinline__ PairY load_y(const double2* __restrict__ Y, int i, int j, int n, const double2& al, bool in) {
  PairY p;
  p.v[0] = p.v[1] = p.v[2] = make_double2(0.0, 0.0);
  if (in) {
    const double2* a = Y + (long)j * n;
    p.v[0] = a[i];
    p.v[1] = a[i + 1];
    p.v[2] = a[i + 2 == n ? 0 : i + 2];
    if (i + 2 == n) p.v[2] = rotate(p.v[2], al);
  }
  return p;
}

// Exponents of every trial column c = g q + column: E[2 c] with |x|, |y| < 2^E, E[2 c + 1] with
// sqrt(w) |curl| < 0.99 2^E, Em[2 c] with sx |x|, sy |y| < 2^E (sx, sy: sqrt(mx), sqrt(my) over 0.99;
// kExpInf where a value is not finite; very negative for a column of zeros).  A bound needs few bits: the curl is formed in binary32 from the leading
// 21 bits of its edge values, 2^-18 of which is added to it (the digits then still reach 2^-60 of
// the edge values, below their FP64 rounding).  One pass over the block, bound by memory: 8 rows per
// thread, two nodes wide, the upper row's x-edges carried to the next; a block whose largest value is
// outside the middle of the binary32 range walks its tile again relative to that value.
constexpr int kExpThreads = 256, kExpTile = 64;  // a block's tile: 64 nodes x 64 mesh rows
__global__ void __launch_bounds__(kExpThreads) k_gram_exponents(int n, int m, const double* __restrict__ ph, Roles roles, int q,
                                                                const uint2* __restrict__ sw, int sw_exp, double sx, double sy,
                                                                int* __restrict__ E, int* __restrict__ Em) {
  __shared__ int red[3][kExpThreads / 32];
  const int col = blockIdx.y, g = blockIdx.z, tid = threadIdx.x, lane = tid & 31;
  const int tx = (n + kExpTile - 1) / kExpTile, by = blockIdx.x / tx, bx = blockIdx.x - by * tx;
  const double2* X = trial_col(roles, g, col);
  const double2* Y = X + (long)n * m;
  const Ph<double> p = load_ph<double>(ph, g);
  const int i = bx * kExpTile + 2 * lane, j0 = by * kExpTile + 8 * (tid >> 5);
  const bool in = i < n;
  int base = 896, hx = 0, hy = 0, cb = 0;  // base: binary64 exponent field that becomes binary32's 0
  for (int pass = 0; pass < 2; ++pass) {
    int topx = 0, topy = 0;  // largest high words (sign off): the exponents of the fields' largest values
    float cmax = 0.0f;  // largest 2^-sw_exp sqrt(w) (|c| + 2^-18 of the values), relative to 2^(base - 896)
    auto lead = [&](double d, int& top) {
      const int h = __double2hiint(d), a = h & 0x7FFFFFFF;
      top = max(top, a);
      const int f = a < ((base + 4) << 20) ? 0 : (a - (base << 20)) << 3;
      return __int_as_float((h & 0x80000000) | f);
    };
    float x0[2][2];
    {
      const PairX v = load_x(X, i, j0, n, m, p.be, in && j0 < m);
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        x0[k][0] = lead(v.v[k].x, topx);
        x0[k][1] = lead(v.v[k].y, topx);
      }
    }
    for (int j = j0; j < min(j0 + 8, m); ++j) {
      const PairX v = load_x(X, i, j + 1, n, m, p.be, in);
      const PairY u = load_y(Y, i, j, n, p.al, in);
      float y[3][2];
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        y[k][0] = lead(u.v[k].x, topy);
        y[k][1] = lead(u.v[k].y, topy);
      }
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        const float s = in ? (float)sw[(long)j * n + i + k].x : 0.0f;
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          const float x1 = lead(c ? v.v[k].y : v.v[k].x, topx);
          const float d = fabsf((x1 - x0[k][c]) - (y[k + 1][c] - y[k][c]));
          const float e = fmaxf(fmaxf(fabsf(x1), fabsf(x0[k][c])), fmaxf(fabsf(y[k + 1][c]), fabsf(y[k][c])));
          cmax = fmaxf(cmax, s * fmaf(e, 0x1p-18f, d));
          x0[k][c] = x1;
        }
      }
    }
    // high words order like the values, bits of non-negative floats too
    const int t = __reduce_max_sync(0xffffffffu, topx);
    const int u = __reduce_max_sync(0xffffffffu, topy);
    const int c = __reduce_max_sync(0xffffffffu, __float_as_int(cmax));
    if (lane == 0) {
      red[0][tid >> 5] = t;
      red[1][tid >> 5] = u;
      red[2][tid >> 5] = c;
    }
    __syncthreads();
    hx = hy = cb = 0;
    for (int w = 0; w < kExpThreads / 32; ++w) {
      hx = max(hx, red[0][w]);
      hy = max(hy, red[1][w]);
      cb = max(cb, red[2][w]);
    }
    const int e = max(hx, hy) >> 20;
    if (e == 0 || e == 0x7FF || (e >= 960 && e <= 1080)) break;
    base = e - 127;
    __syncthreads();
  }
  if (tid != 0) return;
  const int e = max(hx, hy) >> 20;
  if (e == 0) return;
  int ex = e - 1022, ez, em;
  if (e == 0x7FF) {
    ex = ez = em = kExpInf;
  } else {
    // s v < 2^(result) for the largest v with high word h
    auto weighted = [](int h, double s) {
      if ((h >> 20) == 0) return -kExpInf;
      return (h >> 20) - 1023 + ilogb(s * __hiloint2double((h & 0xFFFFF) | 0x3FF00000, -1)) + 1;
    };
    em = max(weighted(hx, sx), weighted(hy, sy));
    // sw holds 31 bits; 2 % for the roundings and the margin; a block without curl counts as tiny
    const float v = __int_as_float(cb) * (1.02f * 0x1p-31f);
    ez = v > 0.0f ? ilogbf(v) + 1 + sw_exp + base - 896 : ex + sw_exp - 18;
  }
  int* Ec = E + 2 * ((long)g * q + col);
  atomicMax(Ec, ex);
  atomicMax(Ec + 1, ez);
  atomicMax(Em + 2 * ((long)g * q + col), em);
}

struct GramArgs {
  int n, m;
  long N;
  Fix ax, bx, ay, by;  // mass factor times 2^ox (x-edges) and 2^oy (y-edges)
  int ox, oy;          // x 2^{52 - Em - ox} < 2^53 likewise
  const uint2* sw;
  int sw_exp;
  const double* ph;
  Roles roles;
  int q;
  const int *E, *Em;  // exponents, entry 2 (g q + column)
  double2* part;
  int npart;
};

// One producer warp's part of a chunk (tile of 32 nodes x 8 mesh rows from (i0, j0)): per stage one
// mesh row, 8 nodes of it (this lane's two from i), the colgroup of `blocks` 32-column blocks.  The
// fixed-point x-edges of a row are those one row up of the row before: read and converted once.
// `wait` blocks until the stage's place in the ring is free and returns it, `ready` hands it on.
template <bool MASS, int BLOCKS, class Wait, class Ready>
__device__ __forceinline__ void produce_chunk(const GramArgs& A, const double2* const (&Xc)[2], const int (&Ex)[2],
                                              const int (&Ez)[2], const bool (&on)[2], const Ph<double>& p, int i, int j0,
                                              unsigned place, Wait&& wait, Ready&& ready) {
  const bool col_in = i < A.n;
  const int dy = MASS ? A.oy - A.ox : 0;  // the fields' own fixed point
  long long xf[BLOCKS][2][2];  // x-edges of the current row: block, node, component
  PairX nx;                    // loads of the next step (a single block's; two blocks load as they go)
  PairY ny;
#pragma unroll
  for (int b = 0; b < BLOCKS; ++b) {
    const PairX v = load_x(Xc[b], i, j0, A.n, A.m, p.be, on[b] && col_in && j0 < A.m);
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      xf[b][k][0] = to_fixed(v.v[k].x, Ex[b]);
      xf[b][k][1] = to_fixed(v.v[k].y, Ex[b]);
    }
  }
  if (BLOCKS == 1) {
    const bool in = on[0] && col_in && j0 < A.m;
    nx = load_x(Xc[0], i, j0 + 1, A.n, A.m, p.be, in);
    ny = load_y(Xc[0] + A.N, i, j0, A.n, p.al, in);
  }
  for (int s = 0; s < kChunk / kStage; ++s) {
    const int j = j0 + s;
    const bool row_in = col_in && j < A.m;
    uint2 w[2];
    if (!MASS) {
#pragma unroll
      for (int k = 0; k < 2; ++k) w[k] = row_in ? A.sw[(long)j * A.n + i + k] : make_uint2(0, 0);
    }
    const unsigned dst = wait() + place;
#pragma unroll
    for (int b = 0; b < BLOCKS; ++b) {
      if (BLOCKS == 2) {
        nx = load_x(Xc[b], i, j + 1, A.n, A.m, p.be, on[b] && row_in);
        ny = load_y(Xc[b] + A.N, i, j, A.n, p.al, on[b] && row_in);
      }
      long long x1[2][2], y[3][2];
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        x1[k][0] = to_fixed(nx.v[k].x, Ex[b]);
        x1[k][1] = to_fixed(nx.v[k].y, Ex[b]);
      }
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        y[k][0] = to_fixed(ny.v[k].x, Ex[b] + dy);
        y[k][1] = to_fixed(ny.v[k].y, Ex[b] + dy);
      }
      if (BLOCKS == 1) {
        const bool in = on[0] && col_in && j + 1 < A.m && s + 1 < kChunk / kStage;
        nx = load_x(Xc[0], i, j + 2, A.n, A.m, p.be, in);
        ny = load_y(Xc[0] + A.N, i, j + 1, A.n, p.al, in);
      }
      const unsigned at = dst + b * kArray;
      const int sh = Ex[b] + A.sw_exp - Ez[b];
#pragma unroll
      for (int im = 0; im < 2; ++im) {
        // (a row or column outside the level leaves zeros: its loads were zero, and the last row's
        // carried x-edges are not used)
        if (MASS) {
          const long long u0 = row_in ? xf[b][0][im] : 0, u1 = row_in ? xf[b][1][im] : 0;
          store_digits<false>(at + im * 512, digits2(u0, A.ax, x1[0][im], A.bx), digits2(u1, A.ax, x1[1][im], A.bx));
          store_digits<false>(at + BLOCKS * kArray + im * 512, digits2(y[0][im], A.ay, y[1][im], A.by),
                       digits2(y[1][im], A.ay, y[2][im], A.by));
        } else {
          unsigned long long z[2];
#pragma unroll
          for (int k = 0; k < 2; ++k) {
            const long long d = (x1[k][im] - xf[b][k][im]) - (y[k + 1][im] - y[k][im]);
            const long long e = sh >= 0 ? (long long)((unsigned long long)d << min(sh, 62)) : d >> min(-sh, 62);
            z[k] = digits1(e, Fix{(int)w[k].x, (int)w[k].y});
          }
          store_digits<true>(at + im * 512, z[0], z[1]);
        }
      }
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        xf[b][k][0] = x1[k][0];
        xf[b][k][1] = x1[k][1];
      }
    }
    ready();
  }
}

__global__ void __launch_bounds__(kThreads, 1) k_gram_tc(GramArgs A) {
  extern __shared__ unsigned char ring[];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int g = blockIdx.y, nb = (A.q + kCols - 1) / kCols, npair = nb * (nb + 1) / 2;
  const bool mass = (int)blockIdx.z < npair;  // GM first: its CTAs take twice as long
  int I = 0, J = (int)blockIdx.z % npair;     // pair index -> (I <= J), J-major
  {
    int j = 0;
    while ((j + 1) * (j + 2) / 2 <= J) ++j;
    I = J - j * (j + 1) / 2;
    J = j;
  }
  const bool diag = I == J;
  const int arrays = mass ? 2 : 1, blocks = diag ? 1 : 2;
  const int stage_bytes = arrays * blocks * kArray;  // array-major, block I then block J
  const int nstage = min(8, 196608 / stage_bytes);
  const unsigned ring0 = smem_u32(ring), bars = ring0 + 196608;
  const unsigned full = bars, empty = bars + 64, done = bars + 128, tfree = bars + 136;
  volatile int* abort = reinterpret_cast<volatile int*>(ring + 196608 + 144);
  unsigned* tmem_slot = reinterpret_cast<unsigned*>(ring + 196608 + 148);
  if (tid == 0) {
    for (int s = 0; s < nstage; ++s) {
      mbar_init(full + 8 * s, kProducers / 32);
      mbar_init(empty + 8 * s, 1);
    }
    mbar_init(done, 1);
    mbar_init(tfree, kProducers / 32);
    *abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  // rows of absent columns stay zero
  for (int t = tid; t < 196608 / 16; t += kThreads) reinterpret_cast<int4*>(ring)[t] = make_int4(0, 0, 0, 0);
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  if (warp == kProducers / 32) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const unsigned tmem = *tmem_slot;
  const int tx = (A.n + kStage - 1) / kStage, nchunk = tx * ((A.m + 7) / 8), first = blockIdx.x;
  const int mine = first < nchunk ? (nchunk - first + A.npart - 1) / A.npart : 0;
  constexpr int kStages = kChunk / kStage;

  long long acc[16];  // this thread's sums: row lane + 32 (warp & 3) of the pair, 16 columns from 16 (warp >> 2)
#pragma unroll
  for (int k = 0; k < 16; ++k) acc[k] = 0;
  // a chunk adds less than 2^55 (GA: 2^56) at weight 2^32: 2^up times that for up to 2^(7 - up) chunks
  // (2^(6 - up))
  int up = mass ? 7 : 6;
  for (int c = (nchunk + A.npart - 1) / A.npart; c > 1; c = (c + 1) / 2) --up;

  if (warp == kProducers / 32) {
    if (lane == 0) {
      int st = 0;
      unsigned par = 0;
      for (int c = 0; c < mine; ++c) {
        if (c > 0) {
          mbar_wait(tfree, (c - 1) & 1, abort);
          tc_fence_after();
        }
        for (int s = 0; s < kStages; ++s) {
          mbar_wait(full + 8 * st, par, abort);
          tc_fence_after();
          for (int ar = 0; ar < arrays; ++ar) {
            const unsigned a0 = ring0 + st * stage_bytes + ar * blocks * kArray, b0 = diag ? a0 : a0 + kArray;
#pragma unroll
            for (int ks = 0; ks < kStage / 16; ++ks) {
              const unsigned a = a0 + 2 * ks * kOctet, b = b0 + 2 * ks * kOctet;
              const unsigned acm = !(s == 0 && ar == 0 && ks == 0);
              // D_t (64 columns each) += (digits 2 u, 2 u + 1 of I) x (digit t - 2 u of J)
              tc_mma(tmem, tc_desc(a, kOctet), tc_desc(b, kOctet), tc_idesc(256), acm);
              tc_mma(tmem + 256, tc_desc(a, kOctet), tc_desc(b + 4 * 1024, kOctet), tc_idesc(128), acm);
              tc_mma(tmem + 128, tc_desc(a + 2048, kOctet), tc_desc(b, kOctet), tc_idesc(256), 1);
              tc_mma(tmem + 384, tc_desc(a + 2048, kOctet), tc_desc(b + 4 * 1024, kOctet), tc_idesc(64), acm);
              tc_mma(tmem + 256, tc_desc(a + 4096, kOctet), tc_desc(b, kOctet), tc_idesc(192), 1);
            }
          }
          tc_commit(empty + 8 * st);
          if (++st == nstage) {
            st = 0;
            par ^= 1;
          }
        }
        tc_commit(done);
      }
      // the last commits have to land before the barriers' memory goes away
      if (mine > 0) mbar_wait(done, (mine - 1) & 1, abort);
    }
    __syncwarp();
  } else {
    const Ph<double> p = load_ph<double>(A.ph, g);
    const int octet = warp & 3, sub = lane & 3;  // 8 nodes of the stage, 2 of them this lane's
    // trial columns of this lane: colgroup (warp >> 2) of block I, and of block J
    const double2* Xc[2];
    int Ex[2], Ez[2];
    bool on[2];
#pragma unroll
    for (int b = 0; b < 2; ++b) {
      const int cl = (warp >> 2) * 8 + (lane >> 2), col = (b ? J : I) * kCols + cl;
      on[b] = b < blocks && col < A.q;
      Xc[b] = trial_col(A.roles, g, on[b] ? col : 0);
      Ex[b] = Ez[b] = 0;
      if (on[b]) {
        const int e0 = (mass ? A.Em : A.E)[2 * ((long)g * A.q + col)], e1 = A.E[2 * ((long)g * A.q + col) + 1];
        on[b] = e0 > kMinExp && e0 < kExpInf;  // zero columns stay zero, non-finite ones are marked at the end
        Ex[b] = on[b] ? e0 + (mass ? A.ox : 0) : 0;
        Ez[b] = on[b] ? e1 : 0;
      }
    }
    const bool any = __any_sync(0xffffffffu, on[0] || on[1]);
    int st = 0;
    unsigned par = 1;  // the ring starts empty
    auto wait = [&] {
      mbar_wait(empty + 8 * st, par, abort);
      return ring0 + st * stage_bytes;
    };
    auto ready = [&] {
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive(full + 8 * st);
      if (++st == nstage) {
        st = 0;
        par ^= 1;
      }
    };
    const unsigned place = octet * kOctet + (warp >> 2) * 128 + lane * 4;
    for (int c = 0; c < mine; ++c) {
      const int t = first + c * A.npart, j0 = t / tx * 8, i = (t - t / tx * tx) * kStage + octet * 8 + sub * 2;
      if (!any) {
        for (int s = 0; s < kStages; ++s) {
          wait();
          ready();
        }
      } else if (mass) {
        if (diag) produce_chunk<true, 1>(A, Xc, Ex, Ez, on, p, i, j0, place, wait, ready);
        else produce_chunk<true, 2>(A, Xc, Ex, Ez, on, p, i, j0, place, wait, ready);
      } else {
        if (diag) produce_chunk<false, 1>(A, Xc, Ex, Ez, on, p, i, j0, place, wait, ready);
        else produce_chunk<false, 2>(A, Xc, Ex, Ez, on, p, i, j0, place, wait, ready);
      }
      // the chunk's sums: rows 0-63 belong to even digits of I, rows 64-127 to odd ones
      mbar_wait(done, c & 1, abort);
      __syncwarp();
      tc_fence_after();
      const unsigned ta = tmem + ((unsigned)(warp & 3) << 21) + 16 * (warp >> 2);
      const bool odd = (warp & 2) != 0;
      // weights of D_t in the 64-bit sum: 2^(32 + up - 8 t); on the diagonal odd t count on odd rows
      // only, halved (their product is symmetric there)
#pragma unroll
      for (int t = 0; t < 7; ++t) {
        float d[16];
        tc_ld16(ta + 64 * t, d);
        if (diag && (t & 1) && !odd) continue;
        const int sh = 32 + up - 8 * t - (diag && (t & 1) ? 1 : 0);  // t = 6: -17 to -9
#pragma unroll
        for (int k = 0; k < 16; ++k) {
          const long long v = (long long)__float2int_rn(d[k]);
          acc[k] += sh >= 0 ? (long long)((unsigned long long)v << sh) : (v + (1 << (-sh - 1))) >> -sh;
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(tfree);
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == kProducers / 32)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
  // the sums of the pair as doubles, in the ring's memory: S[half][row 0-63][column 0-63]
  double* S = reinterpret_cast<double*>(ring);
  if (warp < kProducers / 32) {
    const int rr = 32 * (warp & 3) + lane;
#pragma unroll
    for (int k = 0; k < 16; ++k) S[rr * 65 + 16 * (warp >> 2) + k] = (double)acc[k];
  }
  __syncthreads();
  const int ne = A.q * (A.q + 1) / 2;
  double2* out = A.part + ((long)g * A.npart + blockIdx.x) * 2 * ne + (mass ? 0 : ne);
  const bool bad = *abort != 0;
  for (int t = tid; t < kCols * kCols; t += kThreads) {
    const int a = t % kCols, b = t / kCols, ca = I * kCols + a, cb = J * kCols + b;
    if (ca > cb || cb >= A.q) continue;
    const int* exps = mass ? A.Em : A.E + 1;
    const int ea = exps[2 * ((long)g * A.q + ca)], eb = exps[2 * ((long)g * A.q + cb)];
    auto sum = [&](int r, int c) {
      const double even = S[r * 65 + c], odd = S[(64 + r) * 65 + c];
      return even + 0x1p-8 * (diag ? odd + S[(64 + c) * 65 + r] : odd);
    };
    double2 v = make_double2(sum(a, b) + sum(32 + a, 32 + b), sum(a, 32 + b) - sum(32 + a, b));
    if (ea <= kMinExp || eb <= kMinExp) {
      v = make_double2(0.0, 0.0);
    } else {
      const int ex = ea + eb - (mass ? 46 : 48) - up;
      v = make_double2(scalbn(v.x, ex), scalbn(v.y, ex));
    }
    if (bad || ea == kExpInf || eb == kExpInf) v = make_double2(nan(""), nan(""));
    out[cb * (cb + 1) / 2 + ca] = v;
  }
}

}  // namespace

// Partial sums per group: enough CTAs for a few waves of one per SM, at most kGramTcRoom chunks each.
int gram_tc_partials(int n, int m, int q, int ngroups) {
  const int nb = (q + kCols - 1) / kCols, per = nb * (nb + 1);  // CTAs per group and partial block
  const long chunks = gram_tc_chunks(n, m);
  long np = (4L * 152 + (long)per * ngroups - 1) / ((long)per * ngroups);
  np = std::max(np, (chunks + kGramTcRoom - 1) / kGramTcRoom);
  return (int)std::max<long>(1, std::min(np, chunks));
}

// E and Em
size_t gram_tc_scratch(int q, int ngroups) { return 4 * sizeof(int) * (size_t)q * ngroups; }

ColumnExps gram_tc(const Level& L, const double* d_ph, Roles roles, int q, int ngroups, int npart, double2* d_partials,
                   int* d_exps, cudaStream_t s) {
  static PerDeviceOnce once;
  once([] { PBS_CUDA(cudaFuncSetAttribute(k_gram_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem)); });
  // every byte 0x80: below -kExpInf
  PBS_CUDA(cudaMemsetAsync(d_exps, 0x80, gram_tc_scratch(q, ngroups), s));
  int* d_em = d_exps + 2 * (long)q * ngroups;
  // sqrt(mx) over 0.99, so that |z| < 0.99 times the bound 2^Em, and the power of two that brings
  // sqrt(mx) to 0.495 .. 0.99: |x| < 2^(Em + ox + 1) then
  const double sx = std::sqrt(L.h2 / L.h1), sy = std::sqrt(L.h1 / L.h2);
  int ox = 0, oy = 0;
  std::frexp(0.99 / sx, &ox);
  std::frexp(0.99 / sy, &oy);
  --ox, --oy;
  const unsigned tiles = ((L.n + kExpTile - 1) / kExpTile) * ((L.m + kExpTile - 1) / kExpTile);
  k_gram_exponents<<<dim3(tiles, q, ngroups), kExpThreads, 0, s>>>(L.n, L.m, d_ph, roles, q, L.sw, L.sw_exp, sx / 0.99, sy / 0.99,
                                                                   d_exps, d_em);
  PBS_LAUNCHED();
  const double r3 = 1.0 / std::sqrt(3.0), al = 0.5 * (1.0 + r3), be = 0.5 * (1.0 - r3);
  const double fx = std::ldexp(sx, ox), fy = std::ldexp(sy, oy);
  GramArgs a{};
  a.n = L.n;
  a.m = L.m;
  a.N = L.N();
  a.ax = make_fix(fx * al);
  a.bx = make_fix(fx * be);
  a.ay = make_fix(fy * al);
  a.by = make_fix(fy * be);
  a.ox = ox;
  a.oy = oy;
  a.sw = L.sw;
  a.sw_exp = L.sw_exp;
  a.ph = d_ph;
  a.roles = roles;
  a.q = q;
  a.E = d_exps;
  a.Em = d_em;
  a.part = d_partials;
  a.npart = npart;
  const int nb = (q + kCols - 1) / kCols;
  k_gram_tc<<<dim3(npart, ngroups, nb * (nb + 1)), kThreads, kSmem, s>>>(a);
  PBS_LAUNCHED();
  return ColumnExps{d_em, 2 * q, ox + 1, oy + 1};
}

}  // namespace pbs
