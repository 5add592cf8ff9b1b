// Stencil passes of the mixed policy over FP64 edge blocks: Rayleigh quotients, residual and the
// projection's right-hand side (included by dense.cu).
//
// A warp walks up a strip of 32 neighbouring mesh columns, `rows` rows of it: lane l has node column
// i0 - 1 + l, every edge value is loaded and converted once (one new x-edge and one y-edge per node),
// what the row above needs again stays in registers, and neighbours to the left and right come by
// shuffles.  No shared memory, no barrier; sums are kept per lane and reduced once per strip.  (One
// node per thread, the form before, converted each value two or three times, spent as many
// instructions on the block sums as on the node, and its FP64 curls waited for the FP64 pipe.)  The
// outer lanes are halo: 30 nodes of 32 lanes (31 where only the right neighbour is read).  40 columns
// at 1024 x 1024, before and now: residual 2.07 -> 0.94 ms, right-hand side 0.87 -> 0.53, Rayleigh
// quotients 1.4 -> 0.55; bound by issue (the memory floors are 0.30, 0.25 and 0.20 ms).
#pragma once
#include "common.cuh"
#include "df32.cuh"

namespace pbs {

constexpr int kStripWarps = 8;

// Bloch extension along j, out of line: its FP64 products would otherwise be predicated into every load.
__device__ __noinline__ double2 strip_extend(double2 v, double2 be, int below) {
  return cmul(v, below ? conj(be) : be);
}

// A column's x- or y-edges as seen by one lane: node column i of -1 .. n, rows -1 .. m by Bloch extension.
// The phase of a column outside the level (wrap) is left to the kernel, after its conversion: FP64
// products would hold up the strips at the level's sides in every row.  Lanes beyond column n read
// column 0 (nothing uses them).
struct StripCol {
  const double2* X;  // x-edges, y-edges N further
  long N;
  int n, m, ii;
  bool wrap;
  double2 pi, be;  // phases of the wrap and of one period along j
  __device__ __forceinline__ StripCol(const double2* x, int n_, int m_, int i, const Ph<double>& p)
      : X(x), N((long)n_ * m_), n(n_), m(m_), ii(i < 0 ? n_ - 1 : (i < n_ ? i : 0)), wrap(i < 0 || i == n_),
        pi(i < 0 ? conj(p.al) : p.al), be(p.be) {}
  __device__ __forceinline__ double2 at(const double2* F, int j) const {
    const int jj = j < 0 ? j + m : (j >= m ? j - m : j);
    double2 v = F[(long)jj * n + ii];
    if (jj != j) v = strip_extend(v, be, j < 0);
    return v;
  }
  __device__ __forceinline__ double2 x(int j) const { return at(X, j); }
  __device__ __forceinline__ double2 y(int j) const { return at(X + N, j); }
  __device__ __forceinline__ dcx split(double2 v) const {
    const dcx d = dcx_split(v);
    return wrap ? cmul(d, dcx_split(pi)) : d;
  }
};

// The warp's strip: first node column i0 and row range [j0, j1); false: no strip.
struct Strip {
  int i0, j0, j1;
};
template <int WIDTH> __device__ __forceinline__ bool strip_of(int n, int m, int rows, Strip& s) {
  const int nx = (n + WIDTH - 1) / WIDTH, w = blockIdx.x * kStripWarps + (threadIdx.x >> 5);
  s.i0 = (w % nx) * WIDTH;
  s.j0 = (w / nx) * rows;
  s.j1 = min(s.j0 + rows, m);
  return s.j0 < m;
}

__device__ __forceinline__ df shfl_df_up(df v) {
  return df_make(__shfl_up_sync(0xffffffffu, v.hi, 1), __shfl_up_sync(0xffffffffu, v.lo, 1));
}
__device__ __forceinline__ df shfl_df_down(df v) {
  return df_make(__shfl_down_sync(0xffffffffu, v.hi, 1), __shfl_down_sync(0xffffffffu, v.lo, 1));
}
__device__ __forceinline__ dcx left(dcx v) { return dcx_make(shfl_df_up(v.x), shfl_df_up(v.y)); }
__device__ __forceinline__ dcx right(dcx v) { return dcx_make(shfl_df_down(v.x), shfl_df_down(v.y)); }
__device__ __forceinline__ dcx twice(dcx v, float f) {  // f a power of two
  return dcx_make(df_make(f * v.x.hi, f * v.x.lo), df_make(f * v.y.hi, f * v.y.lo));
}

// Sums of a block's warps (a, b valid on every lane as the lane's own parts); result on thread 0.
__device__ __forceinline__ void strip_sums(double a, double b, double* __restrict__ part) {
  __shared__ double s[2][kStripWarps];
  for (int o = 16; o > 0; o >>= 1) {
    a += __shfl_xor_sync(0xffffffffu, a, o);
    b += __shfl_xor_sync(0xffffffffu, b, o);
  }
  const int warp = threadIdx.x >> 5;
  if ((threadIdx.x & 31) == 0) {
    s[0][warp] = a;
    s[1][warp] = b;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    a = b = 0.0;
    for (int w = 0; w < kStripWarps; ++w) {
      a += s[0][w];
      b += s[1][w];
    }
    double* p = part + ((long)blockIdx.y * gridDim.x + blockIdx.x) * 2;
    p[0] = a;
    p[1] = b;
  }
}

// e^* M e and (C e)^* W (C e) per column, double-float with compensated sums.  The x part of e^* M e is
// (mx / 3) sum Re conj(x(i,j)) (2 x(i,j) + x(i,j+1)), half of the symmetric stencil, likewise y along i.
__global__ void __launch_bounds__(32 * kStripWarps)
    k_rayleigh_strips(Lvl<df> L, WtsDF w, const double* ph, int cpg, const double2* __restrict__ X, long ld, int rows,
                      double* __restrict__ part) {
  const int lane = threadIdx.x & 31, c = blockIdx.y;
  Strip s;
  acc2 dx = acc2_zero(), dy = acc2_zero(), num = acc2_zero();
  if (strip_of<31>(L.n, L.m, rows, s)) {
    const int i = s.i0 + lane;
    const bool on = lane < 31 && i < L.n;
    const StripCol col(X + c * ld, L.n, L.m, i, load_ph<double>(ph, c / cpg));
    dcx x0 = col.split(col.x(s.j0));
    double2 nx = col.x(s.j0 + 1), ny = col.y(s.j0);
    for (int j = s.j0; j < s.j1; ++j) {
      const dcx x1 = col.split(nx), y0 = col.split(ny);
      if (j + 1 < s.j1) {
        nx = col.x(j + 2);
        ny = col.y(j + 1);
      }
      const dcx y1 = right(y0);
      if (on) {
        const dcx tx = twice(x0, 2.0f) + x1, ty = twice(y0, 2.0f) + y1;
        dot2(dx, x0.x, tx.x);
        dot2(dx, x0.y, tx.y);
        dot2(dy, y0.x, ty.x);
        dot2(dy, y0.y, ty.y);
        const dcx h = x1 - x0 - y1 + y0;
        const float2 v = w.w[(long)j * L.n + i];
        const dcx wh = df_make(v.x, v.y) * h;
        dot2(num, h.x, wh.x);
        dot2(num, h.y, wh.y);
      }
      if ((j & 7) == 7) {
        dot2_fold(dx);
        dot2_fold(dy);
        dot2_fold(num);
      }
      x0 = x1;
    }
  }
  const df third = df(1.0 / 3.0);
  strip_sums(df_to(L.mx * third * acc2_df(dx) + L.my * third * acc2_df(dy)), df_to(acc2_df(num)), part);
}

// v 2^{60 - E} truncated to an integer, |v| < 2^E (subnormals and zero are shifted out for E > -900)
__device__ __forceinline__ long long fixed60(double v, int E) {
  const int hi = __double2hiint(v), sh = min(E + 1023 - ((hi >> 20) & 0x7FF), 63);
  const unsigned long long m = (((unsigned long long)((hi & 0xFFFFF) | 0x100000) << 32) | (unsigned)__double2loint(v)) << 8 >> sh;
  const long long s = (long long)(hi >> 31);
  return ((long long)m ^ s) - s;
}
struct Fixed2 {
  long long x, y;
};
__device__ __forceinline__ Fixed2 fixed60(double2 v, int E) { return Fixed2{fixed60(v.x, E), fixed60(v.y, E)}; }
__device__ __forceinline__ Fixed2 rescale(Fixed2 v, int sh) {  // v 2^sh, uniform over the warp
  if (sh >= 0) return Fixed2{v.x << min(sh, 63), v.y << min(sh, 63)};
  return Fixed2{v.x >> min(-sh, 63), v.y >> min(-sh, 63)};
}
// v p for |p| <= 1 given as p 2^62
__device__ __forceinline__ Fixed2 turn(Fixed2 v, Fixed2 p) {
  const long long x = v.x << 2, y = v.y << 2;
  return Fixed2{__mul64hi(x, p.x) - __mul64hi(y, p.y), __mul64hi(x, p.y) + __mul64hi(y, p.x)};
}
__device__ __forceinline__ long long shfl_up_ll(long long v) { return (long long)__shfl_up_sync(0xffffffffu, v, 1); }
__device__ __forceinline__ long long shfl_down_ll(long long v) { return (long long)__shfl_down_sync(0xffffffffu, v, 1); }
// a 64-bit integer as double-float (rounded to 2^-47 or better): 22, 21 and 21 bits, each exact in
// binary32 by way of the low bits of 1.5 2^23 and 2^23
__device__ __forceinline__ df df_of(long long d) {
  const int hi = (int)(d >> 32);
  const unsigned c1 = (unsigned)(d >> 21) & 0x1FFFFFu, c2 = (unsigned)d & 0x1FFFFFu;
  const float f0 = __fmaf_rn(__int_as_float(0x4B400000 + (hi >> 10)), 0x1p42f, -12582912.0f * 0x1p42f);
  const float f1 = __fmaf_rn(__uint_as_float(0x4B000000u | c1), 0x1p21f, -8388608.0f * 0x1p21f);
  const float f2 = __fsub_rn(__uint_as_float(0x4B000000u | c2), 8388608.0f);
  const df s = quick_two_sum(f0, f1);
  return quick_two_sum(s.hi, __fadd_rn(s.lo, f2));
}
__device__ __forceinline__ dcx df_of(Fixed2 v) { return dcx_make(df_of(v.x), df_of(v.y)); }
__device__ __forceinline__ int top_of(double2 v) {  // high word of the larger part, sign off
  return max(__double2hiint(v.x) & 0x7FFFFFFF, __double2hiint(v.y) & 0x7FFFFFFF);
}

// R = A e - lambda M e for the mixed policy, whose preconditioner reads it in FP32, and per column
// |R|^2 and |M e|^2.  The curls c = x(i,j+1) - x(i,j) - y(i+1,j) + y(i,j) are where the stencil cancels
// (neighbouring values of a smooth iterate nearly agree); they are formed exactly, on integers of 60
// bits relative to the largest value of the warp's rows (2^-60 of it, against the 2^-53 of each value
// that FP64 differences lose), as are the mass sums 4 x + x+ + x-.  Everything after them - H = w c,
// the differences of H, R = A e - lambda M e - is double-float: those steps see the curls and the
// iterate's values themselves, so a relative rounding of 2^-47 there moves the relative residual by
// about 2^-47 (H differences: 2^-47 sqrt(lambda_max / lambda), 1e-10 next to Gamma at 1024^2), far below
// any tolerance.  R is stored rounded to FP32; its norm and that of M e are summed in compensated FP32
// per lane and in FP64 across the block.
__global__ void __launch_bounds__(32 * kStripWarps)
    k_residual_strips(Lvl<df> L, WtsDF w, const double* ph, int cpg, const double2* __restrict__ E, float2* __restrict__ R,
                      long ld, const double* __restrict__ lam, int rows, double* __restrict__ part) {
  const int lane = threadIdx.x & 31, c = blockIdx.y;
  Strip s;
  df rr = df_zero(), mm = df_zero();
  if (strip_of<30>(L.n, L.m, rows, s)) {
    const int i = s.i0 - 1 + lane;
    const bool on = lane >= 1 && lane <= 30 && i < L.n;
    const StripCol col(E + c * ld, L.n, L.m, i, load_ph<double>(ph, c / cpg));
    const df l = df_split(lam[c]), sx = L.mx * df(1.0 / 6.0), sy = L.my * df(1.0 / 6.0), lx = l * sx, ly = l * sy;
    const long N = (long)L.n * L.m;
    float2* Rc = R + c * ld;
    double2 v = col.x(s.j0 - 1), nx = col.x(s.j0), ny = col.y(s.j0 - 1);
    int top1 = __reduce_max_sync(0xffffffffu, top_of(v)), top0 = 0;  // of the last row and the one before
    int e = max((top1 >> 20) - 1022, -60);
    const Fixed2 pf{fixed60(col.pi.x, 1) << 3, fixed60(col.pi.y, 1) << 3};
    Fixed2 xc = fixed60(v, e), xm{0, 0};
    if (col.wrap) xc = turn(xc, pf);
    dcx hb = dcx_make(df_zero(), df_zero());
    for (int j = s.j0 - 1; j < s.j1; ++j) {
      const int top2 = __reduce_max_sync(0xffffffffu, max(top_of(nx), top_of(ny)));
      const int en = max((max(max(top0, top1), top2) >> 20) - 1022, -60);
      xc = rescale(xc, e - en);
      xm = rescale(xm, e - en);
      e = en;
      top0 = top1;
      top1 = top2;
      Fixed2 xn = fixed60(nx, e), y = fixed60(ny, e);
      if (col.wrap) {  // (components up to 2^60.5 then: the sums below stay under 2^63)
        xn = turn(xn, pf);
        y = turn(y, pf);
      }
      if (j + 1 < s.j1) {
        nx = col.x(j + 2);
        ny = col.y(j + 1);
      }
      const Fixed2 yr{shfl_down_ll(y.x), shfl_down_ll(y.y)}, yl{shfl_up_ll(y.x), shfl_up_ll(y.y)};
      // 2^{e - 60}; beyond the binary32 range (and for NaN) everything becomes NaN
      const float sc = e > 126 ? __int_as_float(0x7FFFFFFF) : __int_as_float((e - 60 + 127) << 23);
      const float2 wv = w.w[(long)(j < 0 ? L.m - 1 : j) * L.n + col.ii];
      const dcx h = df_make(sc * wv.x, sc * wv.y) * df_of(Fixed2{(xn.x - xc.x) - (yr.x - y.x), (xn.y - xc.y) - (yr.y - y.y)});
      const dcx hl = left(h);
      if (j >= s.j0 && on) {
        const dcx mx = df_of(Fixed2{4 * xc.x + (xn.x + xm.x), 4 * xc.y + (xn.y + xm.y)});
        const dcx my = df_of(Fixed2{4 * y.x + (yr.x + yl.x), 4 * y.y + (yr.y + yl.y)});
        const dcx rx = (hb - h) - df_make(sc * lx.hi, sc * lx.lo) * mx;
        const dcx ry = (h - hl) - df_make(sc * ly.hi, sc * ly.lo) * my;
        const float2 fx = make_float2(df_to_float(rx.x), df_to_float(rx.y));
        const float2 fy = make_float2(df_to_float(ry.x), df_to_float(ry.y));
        const long at = (long)j * L.n + i;
        Rc[at] = fx;
        Rc[N + at] = fy;
        const float ax = sc * sx.hi, ay = sc * sy.hi;
        const float m0 = ax * mx.x.hi, m1 = ax * mx.y.hi, m2 = ay * my.x.hi, m3 = ay * my.y.hi;
        const df r = two_sum(rr.hi, fmaf(fx.x, fx.x, fmaf(fx.y, fx.y, fmaf(fy.x, fy.x, fy.y * fy.y))));
        rr = df_make(r.hi, rr.lo + r.lo);
        const df q = two_sum(mm.hi, fmaf(m0, m0, fmaf(m1, m1, fmaf(m2, m2, m3 * m3))));
        mm = df_make(q.hi, mm.lo + q.lo);
      }
      hb = h;
      xm = xc;
      xc = xn;
    }
  }
  strip_sums(df_to(rr), df_to(mm), part);
}

// rhs(i,j) = (L^* M x)(i,j) = (Mx)_x(i-1,j) - (Mx)_x(i,j) + (Mx)_y(i,j-1) - (Mx)_y(i,j) in double-float,
// stored in T; the mass scalings are applied to the differences.
template <class T>
__global__ void __launch_bounds__(32 * kStripWarps)
    k_lift_adj_mass_strips(Lvl<df> L, const double* ph, int cpg, const double2* __restrict__ X, long ldx, cx<T>* __restrict__ Y,
                           long ldy, int rows) {
  const int lane = threadIdx.x & 31, c = blockIdx.y;
  Strip s;
  if (!strip_of<30>(L.n, L.m, rows, s)) return;
  const int i = s.i0 - 1 + lane;
  const bool on = lane >= 1 && lane <= 30 && i < L.n;
  const StripCol col(X + c * ldx, L.n, L.m, i, load_ph<double>(ph, c / cpg));
  const df sx = L.mx * df(1.0 / 6.0), sy = L.my * df(1.0 / 6.0);
  cx<T>* Yc = Y + c * ldy;
  dcx xm = col.split(col.x(s.j0 - 1)), xc = col.split(col.x(s.j0)), myb;
  double2 nx = col.x(s.j0 + 1), ny = col.y(s.j0);
  {
    const dcx y = col.split(col.y(s.j0 - 1));
    myb = twice(y, 4.0f) + (right(y) + left(y));
  }
  for (int j = s.j0; j < s.j1; ++j) {
    const dcx xn = col.split(nx), y = col.split(ny);
    if (j + 1 < s.j1) {
      nx = col.x(j + 2);
      ny = col.y(j + 1);
    }
    const dcx mx = twice(xc, 4.0f) + (xn + xm), my = twice(y, 4.0f) + (right(y) + left(y));
    const dcx v = sx * (left(mx) - mx) + sy * (myb - my);
    if (on) Yc[(long)j * L.n + i] = mk<T>(narrow<T>(v.x), narrow<T>(v.y));
    myb = my;
    xm = xc;
    xc = xn;
  }
}

// Rows of a strip: more of them share the halo rows, fewer are more strips in flight and, where the
// chip is not full, a shorter chain of rows.  Doubled from two while the launch has more warps than a
// limit per choice.  Rayleigh quotient, residual and right-hand side in us for 2 / 4 / 8 / 16 / 32 rows:
//   16 x 16, 10 columns     8, 8, 6 / 8, 10, 8 / 12, 13, 10
//   96 x 96, 4 columns      8, 8, 6 / 8, 10, 8 / 12, 16, 12
//   128 x 128, 10 columns   10, 16, 10 / 10, 15, 10 / 12, 17, 12 / 21, 25, 19
//   128 x 128, 40 columns   23, 40, 23 / 21, 34, 21 / 21, 32, 21 / 25, 37, 25 / 35, 43, 33
//   256 x 256, 40 columns   66, 136, 66 / 51, 103, 53 / 49, 89, 49 / 49, 86, 50 / 60, 102, 60
//   512 x 512, 10 columns   63, 131, 66 / 49, 99, 52 / 45, 86, 48 / 47, 88, 54 / 58, 95, 60
//   512 x 512, 40 columns   240, 501, 242 / 180, 368, 190 / 155, 309, 166 / 146, 282, 156 / 147, 279, 163
//   1024 x 1024, 40 columns 928, 1888, 901 / 692, 1373, 703 / 588, 1133, 606 / 541, 1010, 561 / 523, 962, 544
// (a rule on the mesh alone, eight rows from 96 x 96 on, took 15 us for the right-hand side of two
// columns there, the 32 x 8 tiles before it 10).  From two rows on no launch has more blocks than the
// mesh has 32 x 8 tiles, for which the partial sums have room.
inline int strip_rows(int n, int m, int ncols) {
  const auto warps = [&](int rows) { return (long)((n + 29) / 30) * ((m + rows - 1) / rows) * ncols; };
  return warps(2) <= 3000 ? 2 : warps(4) <= 3700 ? 4 : warps(8) <= 12000 ? 8 : warps(16) <= 24000 ? 16 : 32;
}
template <int WIDTH> inline unsigned strip_blocks(int n, int m, int rows) {
  const long warps = (long)((n + WIDTH - 1) / WIDTH) * ((m + rows - 1) / rows);
  return (unsigned)((warps + kStripWarps - 1) / kStripWarps);
}

}  // namespace pbs
