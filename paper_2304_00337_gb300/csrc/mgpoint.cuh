// Per-point bodies of the multigrid steps (Section 5): point and patch
// Gauss-Seidel updates, level residuals and grid transfers.  The one-launch-per-step kernels (ops.cu, mg.cu) and the
// fused coarse-level V-cycle kernels (mg.cu) call the same functions, so both
// schedules perform the same arithmetic on every point.
//
// Readers come in two kinds: the __restrict__ ones of common.cuh for kernels
// that never write what they read, and the plain ones below for fused kernels
// that rewrite their buffers between block-wide barriers (a read-only cache path
// would not see those writes).
#pragma once
#include "common.cuh"

namespace pbs {

template <class T>
__device__ __forceinline__ cx<T> gread_plain(const cx<T>* f, int i, int j, int n, int m, const Ph<T>& p) {
  bool w = false;
  cx<T> ph = mk<T>(T(1), T(0));
  if (i < 0) {
    i += n;
    ph = conj(p.al);
    w = true;
  } else if (i >= n) {
    i -= n;
    ph = p.al;
    w = true;
  }
  if (j < 0) {
    j += m;
    ph = cmul(ph, conj(p.be));
    w = true;
  } else if (j >= m) {
    j -= m;
    ph = cmul(ph, p.be);
    w = true;
  }
  cx<T> v = f[(long)j * n + i];
  return w ? cmul(v, ph) : v;
}

template <class T> struct NRdPlain {
  const cx<T>* X;
  int n, m;
  Ph<T> p;
  __device__ __forceinline__ cx<T> v(int i, int j) const { return gread_plain<T>(X, i, j, n, m, p); }
};
template <class T> struct ERdPlain {
  const cx<T>* X;
  int n, m;
  Ph<T> p;
  __device__ __forceinline__ cx<T> x(int i, int j) const { return gread_plain<T>(X, i, j, n, m, p); }
  __device__ __forceinline__ cx<T> y(int i, int j) const { return gread_plain<T>(X + (long)n * m, i, j, n, m, p); }
};

// Readers without the Bloch extension, for stencils that stay inside the level:
// there the extended readers return the stored value unchanged, so a point
// computed through these gives the same result without the wrap tests.
template <class T> struct NRdIn {
  const cx<T>* X;
  int n;
  __device__ __forceinline__ cx<T> v(int i, int j) const { return X[(long)j * n + i]; }
};
template <class T> struct ERdIn {
  const cx<T>* X;
  int n;
  long N;
  __device__ __forceinline__ cx<T> x(int i, int j) const { return X[(long)j * n + i]; }
  __device__ __forceinline__ cx<T> y(int i, int j) const { return X[N + (long)j * n + i]; }
};
template <class T> struct WtsIn {
  const T* winv;
  int n;
  T scale;
  __device__ __forceinline__ T operator()(int i, int j) const { return scale * winv[(long)j * n + i]; }
};
template <class T> __device__ __forceinline__ WtsIn<T> inner(const Wts<T>& w) { return WtsIn<T>{w.winv, w.n, w.scale}; }
template <class T> __device__ __forceinline__ NRdIn<T> inner_n(const cx<T>* X, int n) { return NRdIn<T>{X, n}; }
template <class T> __device__ __forceinline__ ERdIn<T> inner_e(const cx<T>* X, int n, int m) {
  return ERdIn<T>{X, n, (long)n * m};
}
// the neighbourhood [i - lo, i + hi] x [j - lo, j + hi] lies inside an n x m level
__device__ __forceinline__ bool inside(int i, int j, int n, int m, int lo, int hi) {
  return i >= lo && j >= lo && i + hi < n && j + hi < m;
}

// ---- nodal (P = L^* M L) ----------------------------------------------------

// point Gauss-Seidel update of node (i,j); r reads x
template <class T, class R>
__device__ __forceinline__ void node_smooth_at(const Lvl<T>& L, const R& r, cx<T>* x, const cx<T>* b, int i, int j) {
  const long e = (long)j * L.n + i;
  const cx<T> res = b[e] - P_at<T>(r, L, i, j);
  x[e] = x[e] + L.pinv * res;
}

// sP (P x)(i,j) + sB b(i,j)
template <class T, class R>
__device__ __forceinline__ cx<T> apply_nodal_at(const Lvl<T>& L, const R& r, const cx<T>* b, T sP, T sB, int i,
                                                int j) {
  cx<T> y = sP * P_at<T>(r, L, i, j);
  if (b) y = y + sB * b[(long)j * L.n + i];
  return y;
}

// bilinear embedding: fine node (i,j) from coarse reader rc (nc x mc)
template <class T, class R> __device__ __forceinline__ cx<T> prolong_node_at(const R& rc, int i, int j) {
  const int I = i >> 1, J = j >> 1;
  if (!(i & 1) && !(j & 1)) return rc.v(I, J);
  if ((i & 1) && !(j & 1)) return T(0.5) * (rc.v(I, J) + rc.v(I + 1, J));
  if (!(i & 1) && (j & 1)) return T(0.5) * (rc.v(I, J) + rc.v(I, J + 1));
  return T(0.25) * (rc.v(I, J) + rc.v(I + 1, J) + rc.v(I, J + 1) + rc.v(I + 1, J + 1));
}

// adjoint of the bilinear embedding: coarse node (I,J) from fine reader rf
template <class T, class R> __device__ __forceinline__ cx<T> restrict_node_at(const R& rf, int I, int J) {
  cx<T> acc = czero<T>();
#pragma unroll
  for (int dj = -1; dj <= 1; ++dj) {
#pragma unroll
    for (int di = -1; di <= 1; ++di) {
      const T wgt = (di == 0 ? T(1) : T(0.5)) * (dj == 0 ? T(1) : T(0.5));
      acc = acc + wgt * rf.v(2 * I + di, 2 * J + dj);
    }
  }
  return acc;
}

// ---- edges (A + mu M) -------------------------------------------------------

// (sA A + s M) x + sB b at x-edge and y-edge (i,j)
template <class T, class R, class W>
__device__ __forceinline__ void apply_edge_at(const Lvl<T>& L, const W& w, const R& r, const cx<T>* B, T sA, T s,
                                              T sB, int i, int j, cx<T>& yx, cx<T>& yy) {
  const long N = (long)L.n * L.m, e = (long)j * L.n + i;
  yx = czero<T>();
  yy = czero<T>();
  if (sA != T(0)) {
    yx = sA * A_x<T>(r, w, i, j);
    yy = sA * A_y<T>(r, w, i, j);
  }
  if (s != T(0)) {
    yx = yx + s * M_x<T>(r, L, i, j);
    yy = yy + s * M_y<T>(r, L, i, j);
  }
  if (B) {
    yx = yx + sB * B[e];
    yy = yy + sB * B[N + e];
  }
}

// Constants of the patch smoother on one level, formed on the host.
template <class T> struct PatchCoef {
  T m1, m2;  // 2/3 mx, 2/3 my: the mass matrix's diagonal
  T ux, uy;  // mu mx / 6, mu my / 6
  T cs;      // 1 / (mu g^T M_loc g), g the gradient of the node's hat function
};
template <class T> inline PatchCoef<T> patch_coef(const Lvl<T>& L, double mu) {
  const double m1 = 2.0 / 3.0 * (double)L.mx, m2 = 2.0 / 3.0 * (double)L.my;
  return PatchCoef<T>{T(m1), T(m2), T(mu * (double)L.mx / 6.0), T(mu * (double)L.my / 6.0), T(1.0 / (2.0 * mu * (m1 + m2)))};
}

// Changes of the edges L, R, B, T of a node's patch from the patch residual r* and the stored
// K3^{-1} = (k00, k01, k02, k11, k12, k22); V is a real component or a complex value.
template <class T, class V>
__device__ __forceinline__ void patch_solve(const PatchCoef<T>& c, const T k00, const T k01, const T k02, const T k11,
                                            const T k12, const T k22, V rL, V rR, V rB, V rT, V& dL, V& dR, V& dB,
                                            V& dT) {
  const V du = rL - rR, dv = rT - rB, s0 = c.cs * (du - dv);
  const V ya = rL + rR, yb = rB + rT, yc = c.m2 * du + c.m1 * dv;
  const V za = k00 * ya + k01 * yb + k02 * yc, zb = k01 * ya + k11 * yb + k12 * yc, zc = k02 * ya + k12 * yb + k22 * yc;
  const V tx = s0 + c.m2 * zc, ty = s0 - c.m1 * zc;
  dL = za + tx;
  dR = za - tx;
  dB = zb + ty;
  dT = zb - ty;
}

// Block Gauss-Seidel update of the patch of node (i,j) (its edges L, R, B, T);
// r reads x, rb reads b; K3^{-1} of the node in k3 (SoA [6][N]).  The residual
// b - (A + mu M) x on the four edges shares the curls of the four cells around the node.
template <class T, class R, class RB, class W>
__device__ __forceinline__ void edge_smooth_at(const Lvl<T>& L, const W& w, const T* k3, const PatchCoef<T>& pc,
                                               const Ph<T>& p, const R& r, const RB& rb, cx<T>* X, int i, int j) {
  // ghost coordinates
  const cx<T> xL = r.x(i - 1, j), xR = r.x(i, j), xLu = r.x(i - 1, j + 1), xRu = r.x(i, j + 1),
              xLd = r.x(i - 1, j - 1), xRd = r.x(i, j - 1);
  const cx<T> yB = r.y(i, j - 1), yT = r.y(i, j), yBl = r.y(i - 1, j - 1), yTl = r.y(i - 1, j),
              yBr = r.y(i + 1, j - 1), yTr = r.y(i + 1, j);
  const cx<T> hNE = w(i, j) * ((xRu - xR) - (yTr - yT)), hNW = w(i - 1, j) * ((xLu - xL) - (yT - yTl));
  const cx<T> hSE = w(i, j - 1) * ((xR - xRd) - (yBr - yB)), hSW = w(i - 1, j - 1) * ((xL - xLd) - (yB - yBl));
  const cx<T> rL = rb.x(i - 1, j) - ((hSW - hNW) + pc.ux * (T(4) * xL + (xLu + xLd)));
  const cx<T> rR = rb.x(i, j) - ((hSE - hNE) + pc.ux * (T(4) * xR + (xRu + xRd)));
  const cx<T> rB = rb.y(i, j - 1) - ((hSE - hSW) + pc.uy * (T(4) * yB + (yBr + yBl)));
  const cx<T> rT = rb.y(i, j) - ((hNE - hNW) + pc.uy * (T(4) * yT + (yTr + yTl)));
  const long N = (long)L.n * L.m, e = (long)j * L.n + i;
  cx<T> dL, dR, dB, dT;
  patch_solve<T>(pc, k3[e], k3[N + e], k3[2 * N + e], k3[3 * N + e], k3[4 * N + e], k3[5 * N + e], rL, rR, rB, rT, dL,
                 dR, dB, dT);
  cx<T>* Xx = X;
  cx<T>* Xy = X + N;
  Xx[e] = xR + dR;
  Xy[e] = yT + dT;
  // a ghost-coordinate change d of an edge read as conj(alpha) x is alpha d in storage
  if (i > 0) Xx[e - 1] = xL + dL;
  else Xx[(long)j * L.n + L.n - 1] = Xx[(long)j * L.n + L.n - 1] + cmul(p.al, dL);
  if (j > 0) Xy[e - L.n] = yB + dB;
  else Xy[(long)(L.m - 1) * L.n + i] = Xy[(long)(L.m - 1) * L.n + i] + cmul(p.be, dB);
}

// Natural embedding (Section 5) at fine edge index (i,j): a fine edge on a coarse
// edge takes 1/2 of it, one on a coarse cell's midline 1/4 of each of the two
// parallel coarse edges bounding that cell.  rc reads the coarse vector.
template <class T, class R>
__device__ __forceinline__ void prolong_edge_at(const R& rc, int i, int j, cx<T>& vx, cx<T>& vy) {
  {
    const int I = i >> 1;
    if ((j & 1) == 0) vx = T(0.5) * rc.x(I, j >> 1);
    else vx = T(0.25) * (rc.x(I, j >> 1) + rc.x(I, (j >> 1) + 1));
  }
  {
    const int J = j >> 1;
    if ((i & 1) == 0) vy = T(0.5) * rc.y(i >> 1, J);
    else vy = T(0.25) * (rc.y(i >> 1, J) + rc.y((i >> 1) + 1, J));
  }
}

// adjoint of the embedding at coarse index (I,J); rf reads the fine vector
template <class T, class R>
__device__ __forceinline__ void restrict_edge_at(const R& rf, int I, int J, cx<T>& vx, cx<T>& vy) {
  const int i = 2 * I, j = 2 * J;
  vx = T(0.5) * (rf.x(i, j) + rf.x(i + 1, j)) +
       T(0.25) * (rf.x(i, j + 1) + rf.x(i + 1, j + 1) + rf.x(i, j - 1) + rf.x(i + 1, j - 1));
  vy = T(0.5) * (rf.y(i, j) + rf.y(i, j + 1)) +
       T(0.25) * (rf.y(i + 1, j) + rf.y(i + 1, j + 1) + rf.y(i - 1, j) + rf.y(i - 1, j + 1));
}

}  // namespace pbs
