// Coarse levels of the V-cycles as one kernel: a cluster of CTAs per column walks the levels
// from the tail's top one to the coarsest and back (pre-smoothing by colour, residual and
// restriction; the coarsest solve; prolongation and post-smoothing), the level vectors in shared
// memory throughout.  Included by mg.cu.
//
// What bounds it.  A colour step of a level this small is latency: shared-memory reads, a short
// chain of arithmetic, a barrier, and the instruction fetch of code that runs once per step (a
// first form with a copy of the step for each colour and direction stalled on that most).  In FP64
// it is the FP64 pipe: a warp instruction holds its quarter of the SM's pipe for 64 cycles however
// many lanes are active.  Hence
//  * the work is split by 2 x 2 node blocks and by component: a thread (a "unit") owns the real or
//    the imaginary part of one block, so a colour step is one node (or patch) per unit with no
//    index arithmetic, and twice the lanes share the FP64 instructions;
//  * a level's vector lies in four colour planes, and each plane carries one ghost column and one
//    ghost row with the Bloch-continued values, which the owner of a boundary value writes beside
//    it: every read is a plain local one, the steps themselves are real arithmetic, and one body
//    per colour serves smoothing and residual, down and up;
//  * the rows of the larger levels are spread over K CTAs of a cluster (the ghost rows then hold
//    copies of the neighbouring band's edge rows, stored through distributed shared memory), the
//    smaller levels run on the first CTA alone.  K changes where a value is computed, not how.
#pragma once
#include <cooperative_groups.h>

#include <type_traits>

#include "coarse.cuh"
#include "mgpoint.cuh"

namespace pbs {

template <class T> struct TailLevel {
  Lvl<T> L;
  const T* winv;  // edge cycles only
  T wscale;
  const T* k3;
  PatchCoef<T> pc;
  int H, V, Vb;   // 2 x 2 blocks per row, block rows of the level and of one CTA's band
  int sx, sb;     // shared-memory offsets (complex elements) of x and b
};
constexpr int kTailMaxLevels = 12;
template <class T> struct TailArgs {
  int nl;  // levels in the tail, the last one the coarsest (plain vectors on the first CTA)
  int lc;  // levels 0 .. lc - 1 are spread over the cluster, the others run on its first CTA
  int K;   // CTAs per cluster
  TailLevel<T> lev[kTailMaxLevels];
  int sr, sr1;      // offsets of the residuals: of the top level, and of the levels below it
  int sf;           // offset of the column's coarsest factor (leading dimension nfac + 1), or -1
  int sw;           // offset of the coarsest solve's second vector
  const cx<T>* b0;  // top level right-hand sides and solutions, columns at stride ld0
  cx<T>* x0;
  long ld0;
  const double* ph;
  int cpg;
  const cx<T>* factor;  // per-group coarsest factors (nfac x nfac)
  int nfac, ngroups, goff;
  int nu_pre, nu_post;
};
constexpr int kTailMaxThreads = 512;
constexpr long kTailMaxNodes = 4096;        // a level joins the tail when it has at most this many nodes
constexpr int kTailSmemBytes = 220 * 1024;  // and the tail's shared-memory vectors fit in this

// complex elements of one field of a level: four planes with a ghost column and a ghost row each
__host__ __device__ inline int tail_plane(int H, int Vb) { return (H + 1) * (Vb + 1); }

// the other component of a pair (both lanes of a pair always take the same path)
template <class T> __device__ __forceinline__ T pair_other(T v) {
  return __shfl_xor_sync(3u << (threadIdx.x & 30), v, 1);
}
// component `im` of (re + i im) * z, v this lane's component and o the other's
template <class T> __device__ __forceinline__ T cmul_part(T v, T o, cx<T> z, int im) {
  return im ? v * z.x + o * z.y : v * z.x - o * z.y;
}

template <class T, bool CL> __device__ __forceinline__ T* tail_rank(T* sm, int rank) {
  if constexpr (CL) return cooperative_groups::this_cluster().map_shared_rank(sm, rank);
  return sm;
}

// What a thread knows of the level at work, and its unit: block (bu, row lv of this CTA's band, bv
// of the level), component im.
template <class T, bool CL> struct TailAt {
  T* sm;  // this CTA's shared memory, as reals
  Ph<T> p;
  int rank, K;  // this CTA's band and the number of bands of the level
  int H, Vb, RW, PS;
  float inv_h;
  int bu, lv, bv, im, place;
  bool x0, x1, y0, y1;  // the block lies on the first / last column of the level, row of the band
  __device__ __forceinline__ void unit(int u) {  // blocks row by row, a block's components in neighbouring lanes
    im = u & 1;
    lv = (int)(((float)(u >> 1) + 0.5f) * inv_h);  // exact: see split_index
    bu = (u >> 1) - lv * H;
    bv = rank * Vb + lv;
    place = 2 * (lv * RW + bu) + im;
    x0 = bu == 0;
    x1 = bu == H - 1;
    y0 = lv == 0;
    y1 = lv == Vb - 1;
  }
  // Offset of field f at node offset (a, b), -1 .. 2, from the block's even node.  Odd coordinates
  // lie one storage place further than their block, so that place 0 (odd planes) and place H or Vb
  // (even planes) are the ghosts.
  __device__ __forceinline__ int off(int f, int a, int b) const {
    return 2 * (f + ((a & 1) + 2 * (b & 1)) * PS + ((b + 1) >> 1) * RW + ((a + 1) >> 1));
  }
  __device__ __forceinline__ T at(int f, int a, int b) const { return sm[place + off(f, a, b)]; }
  // Stores the copies of value x at `e` (storage index; memory of band r at `base`; parities ca, cb):
  // the ghost column where gx, the ghost row of the band below or above where gy.
  __device__ __forceinline__ void ghosts(T* base, int r, int e, int ca, int cb, bool gx, bool gy, T x) const {
    const T o = pair_other(x);
    const cx<T> px = mk<T>(p.al.x, ca ? -p.al.y : p.al.y), py = mk<T>(p.be.x, cb ? -p.be.y : p.be.y);
    const int dx = ca ? -2 * H : 2 * H, dy = cb ? -2 * Vb * RW : 2 * Vb * RW;
    const T xx = cmul_part(x, o, px, im);
    if (gx) base[e + dx] = xx;
    T* far = base;
    T xy = x, xxy = xx;
    if (!CL || (cb ? r == K - 1 : r == 0)) {  // the level's boundary
      xy = cmul_part(x, o, py, im);
      xxy = cmul_part(xy, pair_other(xy), px, im);
      if (CL) far = tail_rank<T, CL>(sm, K - 1 - r);
    } else if (gy) {
      far = tail_rank<T, CL>(sm, cb ? r + 1 : r - 1);
    }
    if (gy) far[e + dy] = xy;
    if (gx && gy) far[e + dx + dy] = xxy;
  }
  // stores x at the unit's node (ca, cb) of field f
  __device__ __forceinline__ void put_own(int f, int ca, int cb, T x) const {
    const int e = place + off(f, ca, cb);
    sm[e] = x;
    const bool gx = ca ? x1 : x0, gy = cb ? y1 : y0;
    if (gx || gy) ghosts(sm, rank, e, ca, cb, gx, gy, x);
  }
  // Adds d to the value at node offset (a, b), -1 .. 1, at most one of them -1, whose stored copy
  // here is `old`.  Across the level's boundary that copy is the Bloch-continued one, and d changes
  // the value itself by d times the phase; across a band's edge it is a plain copy.
  __device__ __forceinline__ void add(int f, int a, int b, T d, T old) const {
    const int ca = a & 1, cb = b & 1;
    int e = place + off(f, a, b), r = rank;
    T* base = sm;
    T x = old + d;
    if (a < 0 && x0) {  // the last column's value
      e += 2 * H;
      x = sm[e] + cmul_part(d, pair_other(d), p.al, im);
    }
    if (b < 0 && y0) {  // the last row's value, or the band below's
      e += 2 * Vb * RW;
      const bool wrap = !CL || rank == 0;
      if (CL) {
        r = wrap ? K - 1 : rank - 1;
        base = tail_rank<T, CL>(sm, r);
      }
      if (wrap) x = base[e] + cmul_part(d, pair_other(d), p.be, im);
    }
    base[e] = x;
    const bool gx = a < 0 || !ca ? x0 : x1, gy = b < 0 || !cb ? y0 : y1;
    if (gx || gy) ghosts(base, r, e, ca, cb, gx, gy, x);
  }
};

// Places on the next coarser level: planes spread like this one's or on the first CTA, or the
// coarsest level's plain vector there.
template <class T, bool CL>
__device__ __forceinline__ T tail_coarse(const TailLevel<T>& tc, const TailAt<T, CL>& v, bool last, bool spread, int f,
                                         int I, int J) {
  if (last) {
    const int nc = tc.L.n, mc = tc.L.m;
    const bool wx = I >= nc, wy = J >= mc;
    const T* b = tail_rank<T, CL>(v.sm, 0) + 2 * (f + (J - (wy ? mc : 0)) * nc + I - (wx ? nc : 0));
    T x = b[v.im];
    if (wx || wy) x = cmul_part(x, b[v.im ^ 1], wx && wy ? cmul(v.p.al, v.p.be) : wx ? v.p.al : v.p.be, v.im);
    return x;
  }
  // (n and m here are even: an index one past the end is an even one, its ghost's)
  const int row = (J >> 1) - (spread ? v.rank * tc.Vb : 0);
  return tail_rank<T, CL>(v.sm, spread ? v.rank : 0)[2 * (f + ((I & 1) + 2 * (J & 1)) * tail_plane(tc.H, tc.Vb) +
                                                          (row + (J & 1)) * (tc.H + 1) + (I >> 1) + (I & 1)) + v.im];
}

// One V-cycle of the tail's levels; E: the edge cycle (fields of a level: x-edges, and y-edges four
// planes further), else the nodal one.  The top level's b lies in its residual's place (and is read
// again from global memory on the way up).
template <class T, bool CL, bool E> __device__ __forceinline__ void tail_cycle(const TailArgs<T>& a, T* sm) {
  const int tid = threadIdx.x, NT = blockDim.x;
  const int c = CL ? blockIdx.x / a.K : blockIdx.x, rank = CL ? blockIdx.x - c * a.K : 0;
  TailAt<T, CL> v;
  v.sm = sm;
  v.p = load_ph<T>(a.ph, c / a.cpg);
  v.rank = rank;
  const cx<T>* F = a.factor + (long)((c / a.cpg + a.goff) % a.ngroups) * a.nfac * a.nfac;
  const T* b0 = reinterpret_cast<const T*>(a.b0 + c * a.ld0);
  T* x0 = reinterpret_cast<T*>(a.x0 + c * a.ld0);
  if (rank == 0 && a.sf >= 0) {
    cx<T>* S = reinterpret_cast<cx<T>*>(sm) + a.sf;
    for (int t = tid; t < a.nfac * a.nfac; t += NT) S[(t / a.nfac) * (a.nfac + 1) + t % a.nfac] = F[t];
  }
  if (CL) cooperative_groups::this_cluster().sync();  // every CTA has started before any remote access
  const int nv = a.nl - 1;  // levels but the coarsest; visits 0 .. nv - 1 go down, nv .. 2 nv - 1 up
#pragma unroll 1
  for (int visit = 0; visit < 2 * nv; ++visit) {
    const bool up = visit >= nv;
    const int l = up ? 2 * nv - 1 - visit : visit;
    const bool shared = CL && l < a.lc;
    auto sync = [&] {
      if (shared) cooperative_groups::this_cluster().sync();
      else __syncthreads();
    };
    if (visit == nv && rank == 0) {
      cx<T>* s = reinterpret_cast<cx<T>*>(sm);
      coarse_solve<T>(a.sf >= 0 ? s + a.sf : F, a.sf >= 0 ? a.nfac + 1 : a.nfac, a.nfac, s + a.lev[nv].sb,
                      s + a.lev[nv].sx, s + a.sw);
    }
    if (CL && rank > 0 && !shared) continue;         // the smaller levels run on the first CTA
    if (CL && up && l == a.lc - 1) cooperative_groups::this_cluster().sync();  // ... which has finished them
    const TailLevel<T> t = a.lev[l];
    v.K = shared ? a.K : 1;
    v.H = t.H;
    v.Vb = t.Vb;
    v.RW = t.H + 1;
    v.PS = tail_plane(t.H, t.Vb);
    v.inv_h = 1.0f / (float)t.H;
    v.unit(tid);
    const int units = 2 * t.H * t.Vb, n = t.L.n, m = t.L.m, N = n * m, P4 = 4 * v.PS;
    const int sx = t.sx, sr = l == 0 ? a.sr : a.sr1, sb = l == 0 ? a.sr : t.sb;
    const bool last = l + 1 == nv, spread = CL && l + 1 < a.lc;
    const int sxc = a.lev[l + 1].sx, cy = last ? a.lev[l + 1].L.n * a.lev[l + 1].L.m
                                               : 4 * tail_plane(a.lev[l + 1].H, a.lev[l + 1].Vb);
    // x <- 0 (down) or x + prolongated coarse x (up); the top level's b
    if (!up)
      for (int e = tid; e < (E ? 4 : 2) * P4; e += NT) sm[2 * sx + e] = T(0);
#pragma unroll 1
    for (int u = tid; u < units; u += NT) {
      v.unit(u);
      if (l == 0) {
#pragma unroll 1
        for (int q = 0; q < 4; ++q) {
          const int e = 2 * ((2 * v.bv + (q >> 1)) * n + 2 * v.bu + (q & 1)) + v.im;
          v.put_own(sb, q & 1, q >> 1, b0[e]);
          if (E) v.put_own(sb + P4, q & 1, q >> 1, b0[2 * N + e]);
        }
      }
      if (up) {
        auto xc = [&](int f, int I, int J) {
          return tail_coarse<T, CL>(a.lev[l + 1], v, last, spread, sxc + f, v.bu + I, v.bv + J);
        };
        if (E) {
          const T c0 = xc(0, 0, 0), c1 = xc(0, 0, 1), d0 = xc(cy, 0, 0), d1 = xc(cy, 1, 0);
#pragma unroll 1
          for (int q = 0; q < 4; ++q) {
            const int x = q & 1, y = q >> 1;
            v.put_own(sx, x, y, v.at(sx, x, y) + (y ? T(0.25) * (c0 + c1) : T(0.5) * c0));
            v.put_own(sx + P4, x, y, v.at(sx + P4, x, y) + (x ? T(0.25) * (d0 + d1) : T(0.5) * d0));
          }
        } else {
          const T c00 = xc(0, 0, 0), c10 = xc(0, 1, 0), c01 = xc(0, 0, 1), c11 = xc(0, 1, 1);
#pragma unroll 1
          for (int q = 0; q < 4; ++q) {
            const T h = q == 0 ? c00 : q == 1 ? T(0.5) * (c00 + c10) : q == 2 ? T(0.5) * (c00 + c01)
                                                                          : T(0.25) * ((c00 + c10) + (c01 + c11));
            v.put_own(sx, q & 1, q >> 1, v.at(sx, q & 1, q >> 1) + h);
          }
        }
      }
    }
    sync();
    // the colour steps, and (down) the residual on all four colours of nodes
    const int smooth = 4 * (up ? a.nu_post : a.nu_pre), steps = smooth + (up ? 0 : 4);
    const int RW2 = 2 * v.RW;
    // one colour (X, Y) of the unit, or its residual: `x` and `b` point at the unit's place in plane 0
    // of the fields; element (col, row) of plane q, col and row in {0, 1}, is at q P2 + row RW2 + 2 col
    const int P2 = 2 * v.PS;
    auto step = [&](auto XC, auto YC, bool res, bool zero) {
      constexpr int X = XC, Y = YC, Q = X + 2 * Y, QX = 1 - X + 2 * Y, QY = X + 2 * (1 - Y), QD = 3 - Q;
      const T* px = sm + 2 * sx + v.place;
      const T* pb = sm + 2 * sb + v.place;
      auto at = [&](const T* f, int q, int col, int row) { return f[q * P2 + row * RW2 + 2 * col]; };
      if constexpr (E) {
        const T* py = px + 4 * P2;
        const T* pc = pb + 4 * P2;
        const int i = 2 * v.bu + X, j = 2 * v.bv + Y, e = j * n + i;
        const int il = X || !v.x0 ? -1 : n - 1, jl = Y || v.bv > 0 ? -n : N - n;
        T k00 = T(0), k01 = T(0), k02 = T(0), k11 = T(0), k12 = T(0), k22 = T(0);
        if (!res) {
          const T* k = t.k3 + e;
          k00 = k[0], k01 = k[N], k02 = k[2 * N], k11 = k[3 * N], k12 = k[4 * N], k22 = k[5 * N];
        }
        T xL = T(0), xR = T(0), yB = T(0), yT = T(0);
        T rL = at(pb, QX, 0, Y), rR = at(pb, Q, X, Y), rB = at(pc, QY, X, 0), rT = at(pc, Q, X, Y);
        if (!zero) {
          const T* wp = t.winv + e;
          const T wNE = t.wscale * wp[0], wNW = t.wscale * wp[il], wSE = t.wscale * wp[jl], wSW = t.wscale * wp[il + jl];
          xL = at(px, QX, 0, Y), xR = at(px, Q, X, Y), yB = at(py, QY, X, 0), yT = at(py, Q, X, Y);
          const T xLu = at(px, QD, 0, 1), xRu = at(px, QY, X, 1), xLd = at(px, QD, 0, 0), xRd = at(px, QY, X, 0);
          const T yBl = at(py, QD, 0, 0), yTl = at(py, QX, 0, Y), yBr = at(py, QD, 1, 0), yTr = at(py, QX, 1, Y);
          const T hNE = wNE * ((xRu - xR) - (yTr - yT)), hNW = wNW * ((xLu - xL) - (yT - yTl));
          const T hSE = wSE * ((xR - xRd) - (yBr - yB)), hSW = wSW * ((xL - xLd) - (yB - yBl));
          rR = rR - ((hSE - hNE) + t.pc.ux * (T(4) * xR + (xRu + xRd)));
          rT = rT - ((hNE - hNW) + t.pc.uy * (T(4) * yT + (yTr + yTl)));
          if (!res) {
            rL = rL - ((hSW - hNW) + t.pc.ux * (T(4) * xL + (xLu + xLd)));
            rB = rB - ((hSE - hSW) + t.pc.uy * (T(4) * yB + (yBr + yBl)));
          }
        }
        if (res) {  // (the top level's over b: an edge's b is used by its own unit only)
          v.put_own(sr, X, Y, rR);
          v.put_own(sr + P4, X, Y, rT);
        } else {
          T dL, dR, dB, dT;
          patch_solve<T>(t.pc, k00, k01, k02, k11, k12, k22, rL, rR, rB, rT, dL, dR, dB, dT);
          v.add(sx, X, Y, dR, xR);
          v.add(sx, X - 1, Y, dL, xL);
          v.add(sx + P4, X, Y, dT, yT);
          v.add(sx + P4, X, Y - 1, dB, yB);
        }
      } else {
        const T b = at(pb, Q, X, Y);
        T w = t.L.pinv * b;
        if (!zero) {
          const T v0 = at(px, Q, X, Y);
          const T ew = (at(px, QX, 0, Y) + at(px, QX, 1, Y)) - T(2) * v0;
          const T ns = (at(px, QY, X, 0) + at(px, QY, X, 1)) - T(2) * v0;
          const T dd = ((at(px, QD, 0, 0) + at(px, QD, 1, 0)) + (at(px, QD, 0, 1) + at(px, QD, 1, 1))) - T(4) * v0;
          const T r = b - (t.L.pe * ew + t.L.pn * ns + t.L.pd * dd);
          w = res ? r : v0 + t.L.pinv * r;
        } else if (res) {
          w = b;
        }
        v.put_own(res ? sr : sx, X, Y, w);
      }
    };
    using I0 = std::integral_constant<int, 0>;
    using I1 = std::integral_constant<int, 1>;
#pragma unroll 1
    for (int s = 0; s < steps; ++s) {
      const int q = up ? 3 - (s & 3) : s & 3;
      const bool res = s >= smooth, zero = !up && s == 0 && !res;  // zero: x is still zero everywhere
#pragma unroll 1
      for (int u = tid; u < units; u += NT) {
        if (units > NT) v.unit(u);  // else the thread's only unit, set above
        switch (q) {
          case 0: step(I0{}, I0{}, res, zero); break;
          case 1: step(I1{}, I0{}, res, zero); break;
          case 2: step(I0{}, I1{}, res, zero); break;
          default: step(I1{}, I1{}, res, zero);
        }
      }
      if (!res || s + 1 == steps) sync();
    }
    if (!up) {
      // restriction to coarse node (or edges) (I, J) = (bu, bv) on the block's even node
      const TailLevel<T> tc = a.lev[l + 1];
#pragma unroll 1
      for (int u = tid; u < units; u += NT) {
        v.unit(u);
        T c0, c1 = T(0);
        if (E) {
          const int ry = sr + P4;
          c0 = T(0.5) * (v.at(sr, 0, 0) + v.at(sr, 1, 0)) +
               T(0.25) * ((v.at(sr, 0, 1) + v.at(sr, 1, 1)) + (v.at(sr, 0, -1) + v.at(sr, 1, -1)));
          c1 = T(0.5) * (v.at(ry, 0, 0) + v.at(ry, 0, 1)) +
               T(0.25) * ((v.at(ry, 1, 0) + v.at(ry, 1, 1)) + (v.at(ry, -1, 0) + v.at(ry, -1, 1)));
        } else {
          const T s1 = (v.at(sr, 1, 0) + v.at(sr, -1, 0)) + (v.at(sr, 0, 1) + v.at(sr, 0, -1));
          const T s2 = (v.at(sr, 1, 1) + v.at(sr, -1, 1)) + (v.at(sr, 1, -1) + v.at(sr, -1, -1));
          c0 = v.at(sr, 0, 0) + T(0.5) * s1 + T(0.25) * s2;
        }
        T* base = tail_rank<T, CL>(sm, spread ? rank : 0);
        if (last) {
          T* d = base + 2 * (tc.sb + v.bv * tc.L.n + v.bu) + v.im;
          d[0] = c0;
          if (E) d[2 * cy] = c1;
        } else {
          // the coarse level's planes, with ghosts (its patches read b across the boundary)
          TailAt<T, CL> w = v;
          w.rank = spread ? rank : 0;
          w.K = spread ? a.K : 1;
          w.H = tc.H;
          w.Vb = tc.Vb;
          w.RW = tc.H + 1;
          w.PS = tail_plane(tc.H, tc.Vb);
          const int ca = v.bu & 1, cb = v.bv & 1, I = v.bu >> 1, J = (v.bv >> 1) - w.rank * tc.Vb;
          const bool gx = ca ? I == tc.H - 1 : I == 0, gy = cb ? J == tc.Vb - 1 : J == 0;
          const int e = 2 * (J * w.RW + I) + v.im + w.off(tc.sb, ca, cb);
          base[e] = c0;
          if (E) base[e + 2 * cy] = c1;
          if (gx || gy) {
            w.ghosts(base, w.rank, e, ca, cb, gx, gy, c0);
            if (E) w.ghosts(base, w.rank, e + 2 * cy, ca, cb, gx, gy, c1);
          }
        }
      }
      sync();
    } else if (l == 0) {
#pragma unroll 1
      for (int u = tid; u < units; u += NT) {
        v.unit(u);
#pragma unroll 1
        for (int q = 0; q < 4; ++q) {
          const int e = 2 * ((2 * v.bv + (q >> 1)) * n + 2 * v.bu + (q & 1)) + v.im;
          x0[e] = v.at(sx, q & 1, q >> 1);
          if (E) x0[2 * N + e] = v.at(sx + P4, q & 1, q >> 1);
        }
      }
    }
  }
  if (CL) cooperative_groups::this_cluster().sync();  // no CTA ends while another may still reach its memory
}

template <class T, bool CL> __global__ void __launch_bounds__(kTailMaxThreads) k_node_tail(TailArgs<T> a) {
  extern __shared__ float4 fine_sm[];
  tail_cycle<T, CL, false>(a, reinterpret_cast<T*>(fine_sm));
}
template <class T, bool CL> __global__ void __launch_bounds__(kTailMaxThreads) k_edge_tail(TailArgs<T> a) {
  extern __shared__ float4 fine_sm[];
  tail_cycle<T, CL, true>(a, reinterpret_cast<T*>(fine_sm));
}

}  // namespace pbs
