// Fine-level steps of the nodal multigrid cycle with one sweep per side, as row pipelines (included by
// mg.cu): the same two steps as nodal_tiles.cuh, on the same operands in the same order.
//
// The colour order even/odd i on even rows, then even/odd i on odd rows ("down"; "up" runs it
// backwards) only reaches one row further per colour, so a sweep, the residual and the restriction
// can follow each other up the mesh a row or two apart: a warp walks up a strip of 64 columns, lane l
// with the node columns 2 l and 2 l + 1 of it, five rows in registers.  Neighbours within a lane's
// pair are its own registers, the others come by shuffles; every value is read from memory once, and
// there is no shared memory and no barrier.  Four colours, residual and restriction reach five columns
// to the left and right, so 27 (down) and 28 (up) of the 32 lanes have results; below and above a
// strip of `rows` rows five more are walked through.  A 32 x 32 tile with its halo in shared memory
// instead works on 1.9 times its nodes and reads nine values per node back from shared memory (five
// with 2 x 2 blocks in registers).  Down + up step of 40 FP32 columns at 1024 x 1024: 0.85 -> 0.44 ms,
// of which memory takes 0.29; 20 FP64 columns at 512 x 512, bound by the FP64 pipe: 1.55 -> 1.11 ms.
// Results do not depend on `rows`.
#pragma once
#include "mgpoint.cuh"

namespace pbs {

constexpr int kNodeStripWarps = 4;
constexpr int kDownLanes = 27, kUpLanes = 28;  // lanes with results

template <class T> struct NodePair {
  cx<T> e, o;  // even and odd node column
};
// one row of a strip: the lane's pair, the odd column to the left of it, the even one to the right
template <class T> struct NodeRow {
  cx<T> e, o, lo, re;
};

__device__ __forceinline__ float2 lane_up(float2 v) {
  return make_float2(__shfl_up_sync(0xffffffffu, v.x, 1), __shfl_up_sync(0xffffffffu, v.y, 1));
}
__device__ __forceinline__ float2 lane_down(float2 v) {
  return make_float2(__shfl_down_sync(0xffffffffu, v.x, 1), __shfl_down_sync(0xffffffffu, v.y, 1));
}
__device__ __forceinline__ double2 lane_up(double2 v) {
  return make_double2(__shfl_up_sync(0xffffffffu, v.x, 1), __shfl_up_sync(0xffffffffu, v.y, 1));
}
__device__ __forceinline__ double2 lane_down(double2 v) {
  return make_double2(__shfl_down_sync(0xffffffffu, v.x, 1), __shfl_down_sync(0xffffffffu, v.y, 1));
}
__device__ __forceinline__ NodePair<float> pair_at(const float2* f) {  // f 16-byte aligned
  const float4 v = *reinterpret_cast<const float4*>(f);
  return NodePair<float>{make_float2(v.x, v.y), make_float2(v.z, v.w)};
}
__device__ __forceinline__ NodePair<double> pair_at(const double2* f) { return NodePair<double>{f[0], f[1]}; }
__device__ __forceinline__ void put_pair(float2* f, float2 e, float2 o) {
  *reinterpret_cast<float4*>(f) = make_float4(e.x, e.y, o.x, o.y);
}
__device__ __forceinline__ void put_pair(double2* f, double2 e, double2 o) {
  f[0] = e;
  f[1] = o;
}
// Products and fused products spelled out: the compiler is free to fuse differently in every copy of an
// expression, and a node's value must not depend on where its strip begins.
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float fma_rn(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double fma_rn(double a, double b, double c) { return __fma_rn(a, b, c); }
template <class T> __device__ __forceinline__ cx<T> scaled_rn(T s, cx<T> v) { return mk<T>(mul_rn(s, v.x), mul_rn(s, v.y)); }
template <class T> __device__ __forceinline__ cx<T> fma_rn(T s, cx<T> v, cx<T> a) { return mk<T>(fma_rn(s, v.x, a.x), fma_rn(s, v.y, a.y)); }
template <class T> __device__ __forceinline__ cx<T> cmul_rn(cx<T> a, cx<T> b) {
  return mk<T>(fma_rn(a.x, b.x, -mul_rn(a.y, b.y)), fma_rn(a.x, b.y, mul_rn(a.y, b.x)));
}

// A lane's node columns i, i + 1 (i even) of an n x m level, read with the Bloch extension of one period.
template <class T> struct NodeCols {
  int n, m, ii;
  bool wrap;
  cx<T> pi;  // phase of the wrap along i
  Ph<T> p;
  __device__ __forceinline__ NodeCols(int n_, int m_, int i, const Ph<T>& ph)
      : n(n_), m(m_), ii(i < 0 ? i + n_ : (i >= n_ ? i - n_ : i)), wrap(i < 0 || i >= n_),
        pi(i < 0 ? conj(ph.al) : (i >= n_ ? ph.al : mk<T>(T(1), T(0)))), p(ph) {}
  __device__ __forceinline__ NodePair<T> row(const cx<T>* __restrict__ f, int j) const {
    const int jj = j < 0 ? j + m : (j >= m ? j - m : j);
    NodePair<T> v = pair_at(f + (long)jj * n + ii);
    if (wrap || jj != j) {
      const cx<T> ph = phase(j);
      v.e = cmul_rn<T>(v.e, ph);
      v.o = cmul_rn<T>(v.o, ph);
    }
    return v;
  }
  // coarse node column i / 2 of the n / 2 x m / 2 level
  __device__ __forceinline__ cx<T> coarse(const cx<T>* __restrict__ f, int J) const {
    const int mc = m / 2, JJ = J < 0 ? J + mc : (J >= mc ? J - mc : J);
    const cx<T> v = f[(long)JJ * (n / 2) + ii / 2];
    return wrap || JJ != J ? cmul_rn<T>(v, phase(2 * J)) : v;
  }
  __device__ __forceinline__ cx<T> phase(int j) const {
    return j < 0 ? cmul_rn<T>(pi, conj(p.be)) : (j >= m ? cmul_rn<T>(pi, p.be) : pi);
  }
};

// P x at a node from its nine values, in the order of P_at
template <class T>
__device__ __forceinline__ cx<T> P_of(const Lvl<T>& L, cx<T> c, cx<T> w, cx<T> e, cx<T> s, cx<T> n, cx<T> sw, cx<T> se,
                                      cx<T> nw, cx<T> ne) {
  const cx<T> h = (w + e) - T(2) * c;
  const cx<T> v = (s + n) - T(2) * c;
  const cx<T> d = ((sw + se) + (nw + ne)) - T(4) * c;
  return fma_rn<T>(L.pd, d, fma_rn<T>(L.pn, v, scaled_rn<T>(L.pe, h)));
}
// of the even node of row r between the rows s (below) and n, and of the odd node
template <class T> __device__ __forceinline__ cx<T> P_even(const Lvl<T>& L, const NodeRow<T>& s, const NodeRow<T>& r, const NodeRow<T>& n) {
  return P_of<T>(L, r.e, r.lo, r.o, s.e, n.e, s.lo, s.o, n.lo, n.o);
}
template <class T> __device__ __forceinline__ cx<T> P_odd(const Lvl<T>& L, const NodeRow<T>& s, const NodeRow<T>& r, const NodeRow<T>& n) {
  return P_of<T>(L, r.o, r.e, r.re, s.o, n.o, s.e, s.re, n.e, n.re);
}

// Pre-smoothing from X0 (GUESS) or zero, residual, restriction: x to Xs, the restricted residual to Bc.
template <class T, bool GUESS>
__global__ void __launch_bounds__(32 * kNodeStripWarps)
    k_node_down_strips(Lvl<T> L, const double* ph, int cpg, const cx<T>* __restrict__ B, long ldb, const cx<T>* __restrict__ X0,
                       long ld0, cx<T>* __restrict__ Xs, long lds, cx<T>* __restrict__ Bc, long ldc, int rows) {
  const int lane = threadIdx.x & 31, c = blockIdx.y, width = 2 * kDownLanes, nx = (L.n + width - 1) / width;
  const int w = blockIdx.x * kNodeStripWarps + (threadIdx.x >> 5), j0 = w / nx * rows, j1 = min(j0 + rows, L.m);
  if (j0 >= L.m) return;
  const int i = w % nx * width - 6 + 2 * lane;
  const bool on = lane >= 3 && lane < 3 + kDownLanes && i < L.n;
  const NodeCols<T> col(L.n, L.m, i, load_ph<T>(ph, c / cpg));
  const cx<T>* b = B + c * ldb;
  const cx<T>* x0 = GUESS ? X0 + c * ld0 : nullptr;
  const T inv = L.pinv;
  const cx<T> zero = czero<T>();
  const NodeRow<T> none{zero, zero, zero, zero};
  auto start = [&](NodePair<T> v) { return NodeRow<T>{v.e, v.o, lane_up(v.o), lane_down(v.e)}; };
  // finished rows j - 3 and j - 2 and their right-hand sides; rows j - 1, j, j + 1 of the starting iterate
  NodeRow<T> f1 = none, f0 = none, a = none, d = none, u = none;
  NodePair<T> b0{zero, zero}, ba{zero, zero}, bd = col.row(b, j0 - 2), bu = col.row(b, j0 - 1), xd{zero, zero}, xu{zero, zero};
  if (GUESS) {
    a = start(col.row(x0, j0 - 3));
    xd = col.row(x0, j0 - 2);
    xu = col.row(x0, j0 - 1);
  }
  cx<T> acc = zero;  // restricted residual so far
  for (int j = j0 - 2; j <= j1; j += 2) {
    const NodePair<T> cb = bd, cu = bu;
    if (GUESS) {
      d = NodeRow<T>{xd.e, xd.o, lane_up(xd.o), zero};
      u = start(xu);
    } else {
      d = u = none;
    }
    if (j < j1) {
      bd = col.row(b, j + 2);
      if (j + 2 < j1) bu = col.row(b, j + 3);
      if (GUESS) {
        xd = col.row(x0, j + 2);
        xu = col.row(x0, j + 3);
      }
    }
    // row j: even, then odd nodes
    if (GUESS) d.e = fma_rn<T>(inv, cb.e - P_even<T>(L, a, d, u), d.e);
    else d.e = scaled_rn<T>(inv, cb.e);
    d.re = lane_down(d.e);
    if (GUESS) d.o = fma_rn<T>(inv, cb.o - P_odd<T>(L, a, d, u), d.o);
    else d.o = scaled_rn<T>(inv, cb.o - scaled_rn<T>(L.pe, d.e + d.re));
    d.lo = lane_up(d.o);
    if (j >= j0) {
      // row j - 1
      if (GUESS) a.e = fma_rn<T>(inv, ba.e - P_even<T>(L, f0, a, d), a.e);
      else a.e = scaled_rn<T>(inv, ba.e - fma_rn<T>(L.pd, (f0.lo + f0.o) + (d.lo + d.o), scaled_rn<T>(L.pn, f0.e + d.e)));
      a.re = lane_down(a.e);
      a.o = fma_rn<T>(inv, ba.o - P_odd<T>(L, f0, a, d), a.o);
      a.lo = lane_up(a.o);
      if (j > j0) {
        // row j - 2: residual, middle row of the restriction
        const cx<T> re = b0.e - P_even<T>(L, f1, f0, a), ro = b0.o - P_odd<T>(L, f1, f0, a);
        acc = acc + T(0.5) * lane_up(ro);
        acc = acc + T(1) * re;
        acc = acc + T(0.5) * ro;
        if (on) {
          put_pair(Xs + c * lds + (long)(j - 2) * L.n + i, f0.e, f0.o);
          put_pair(Xs + c * lds + (long)(j - 1) * L.n + i, a.e, a.o);
        }
      }
      // row j - 1: above one coarse row, below the next
      const cx<T> re = ba.e - P_even<T>(L, f0, a, d), ro = ba.o - P_odd<T>(L, f0, a, d), rl = lane_up(ro);
      if (j > j0 && on) {
        acc = acc + T(0.25) * rl;
        acc = acc + T(0.5) * re;
        acc = acc + T(0.25) * ro;
        Bc[c * ldc + (long)((j - 2) / 2) * (L.n / 2) + i / 2] = acc;
      }
      acc = T(0.25) * rl;
      acc = acc + T(0.5) * re;
      acc = acc + T(0.25) * ro;
    }
    f1 = a;
    f0 = d;
    a = u;
    b0 = cb;
    ba = cu;
  }
}

// Prolongation of Xc onto Xs and post-smoothing (colours backwards), to X.
template <class T>
__global__ void __launch_bounds__(32 * kNodeStripWarps)
    k_node_up_strips(Lvl<T> L, const double* ph, int cpg, const cx<T>* __restrict__ B, long ldb, const cx<T>* __restrict__ Xs,
                     long lds, const cx<T>* __restrict__ Xc, long ldc, cx<T>* __restrict__ X, long ldx, int rows) {
  const int lane = threadIdx.x & 31, c = blockIdx.y, width = 2 * kUpLanes, nx = (L.n + width - 1) / width;
  const int w = blockIdx.x * kNodeStripWarps + (threadIdx.x >> 5), j0 = w / nx * rows, j1 = min(j0 + rows, L.m);
  if (j0 >= L.m) return;
  const int i = w % nx * width - 4 + 2 * lane;
  const bool on = lane >= 2 && lane < 2 + kUpLanes && i < L.n;
  const NodeCols<T> col(L.n, L.m, i, load_ph<T>(ph, c / cpg));
  const cx<T>* b = B + c * ldb;
  const cx<T>* xs = Xs + c * lds;
  const cx<T>* xc = Xc + c * ldc;
  const T inv = L.pinv;
  const cx<T> zero = czero<T>();
  // the starting iterate: row 2 J and row 2 J + 1 from the coarse rows J and J + 1 (own column, next one)
  auto even_row = [&](NodePair<T> v, cx<T> c0, cx<T> c1) {
    const cx<T> e = v.e + c0, o = v.o + T(0.5) * (c0 + c1);
    return NodeRow<T>{e, o, lane_up(o), lane_down(e)};
  };
  auto odd_row = [&](NodePair<T> v, cx<T> c0, cx<T> c1, cx<T> n0, cx<T> n1) {
    const cx<T> e = v.e + T(0.5) * (c0 + n0), o = v.o + T(0.25) * (((c0 + c1) + n0) + n1);
    return NodeRow<T>{e, o, zero, lane_down(e)};
  };
  // rows j - 2 (finished), j - 1, j, j + 1
  cx<T> c0 = col.coarse(xc, j0 / 2 - 1), c1 = lane_down(c0);
  NodeRow<T> f{zero, zero, zero, zero}, a = even_row(col.row(xs, j0 - 2), c0, c1);
  NodePair<T> ba{zero, zero}, bd = col.row(b, j0 - 1), bu = col.row(b, j0), xd = col.row(xs, j0 - 1), xu = col.row(xs, j0);
  cx<T> cn = col.coarse(xc, j0 / 2);
  for (int j = j0 - 1; j < j1; j += 2) {
    const NodePair<T> cb = bd, cu = bu;
    const cx<T> n0 = cn, n1 = lane_down(n0);
    NodeRow<T> d = odd_row(xd, c0, c1, n0, n1);
    const NodeRow<T> u = even_row(xu, n0, n1);
    if (j + 2 < j1) {
      bd = col.row(b, j + 2);
      xd = col.row(xs, j + 2);
      bu = col.row(b, j + 3);
      xu = col.row(xs, j + 3);
      cn = col.coarse(xc, (j + 3) / 2);
    }
    // row j: odd, then even nodes
    d.o = fma_rn<T>(inv, cb.o - P_odd<T>(L, a, d, u), d.o);
    d.lo = lane_up(d.o);
    d.e = fma_rn<T>(inv, cb.e - P_even<T>(L, a, d, u), d.e);
    d.re = lane_down(d.e);
    if (j > j0) {
      // row j - 1
      a.o = fma_rn<T>(inv, ba.o - P_odd<T>(L, f, a, d), a.o);
      a.lo = lane_up(a.o);
      a.e = fma_rn<T>(inv, ba.e - P_even<T>(L, f, a, d), a.e);
      if (on) {
        put_pair(X + c * ldx + (long)(j - 1) * L.n + i, a.e, a.o);
        put_pair(X + c * ldx + (long)j * L.n + i, d.e, d.o);
      }
    }
    f = d;
    a = u;
    ba = cu;
    c0 = n0;
    c1 = n1;
  }
}

template <int LANES> inline unsigned node_strip_blocks(int n, int m, int rows) {
  const long warps = (long)((n + 2 * LANES - 1) / (2 * LANES)) * ((m + rows - 1) / rows);
  return (unsigned)((warps + kNodeStripWarps - 1) / kNodeStripWarps);
}

}  // namespace pbs
