// Geometric multigrid of Section 5: bisection hierarchy with Galerkin coarse
// operators, node-patch block Gauss-Seidel for A + mu M (edges), point
// Gauss-Seidel for P = L^* M L (nodes), dense Cholesky on the coarsest level.
//
// Coarse operators.  With the natural embedding as prolongation the Galerkin
// product P^* A_f P is the curl-curl matrix of the coarse mesh whose 1/eps is
// the mean of the four children's 1/eps, and P^* M_f P is the coarse mass
// matrix (the curl is constant per cell, so a coarse cell's energy is the sum
// of its children's).  Hence every level uses the same stencil code with its
// own 1/eps and mesh widths, and the Bloch phases are unchanged (the periods
// a, b are the same on every level).
//
// Patch solve.  The patch of node (i,j) holds its left, right, bottom and top
// edges (L, R, B, T).  In "ghost" coordinates (values read through the Bloch
// extension) the 4x4 block of A + mu M is real and independent of k:
//   K = sum_cells w_c v_c v_c^T + mu diag(m1, m1, m2, m2),  m1 = 2/3 h2/h1, m2 = 2/3 h1/h2,
//   v_SW = (1,0,-1,0), v_NW = (-1,0,0,-1), v_SE = (0,1,1,0), v_NE = (0,-1,0,1).
// The gradient g = (1,-1,1,-1) of the node's hat function satisfies K g =
// mu M_loc g, which makes K ill-conditioned for small mu (Section 5).  Following
// the paper's stable variant, T = [g, t_a, t_b, t_c] with the M_loc-orthogonal
// complement t_a = (1,1,0,0), t_b = (0,0,1,1), t_c = (m2,-m2,-m1,m1) gives
// T^T K T = diag(mu g^T M_loc g, K3), so K^{-1} r = g (g^T r)/(mu g^T M_loc g)
// + T3 K3^{-1} T3^T r.  K3^{-1} (3x3, symmetric) is stored per node and level.
//
// Colouring.  Nodes are processed by colour (i mod 2, j mod 2) in the order
// (0,0), (1,0), (0,1), (1,1) (pre-smoothing) and reversed (post-smoothing).
// Same-colour patches share no edge and are not coupled by A or M, so each
// colour is one parallel launch and equals the sequential block Gauss-Seidel
// sweep; the resulting V-cycle is Hermitian.
#include <algorithm>
#include <cmath>
#include <cstdlib>
#include <cstring>
#include <string>
#include <type_traits>

#include "internal.h"
#include "mgpoint.cuh"
#include "node_strips.cuh"
#include "nodal_tiles.cuh"
#include "tail.cuh"

namespace pbs {

namespace {

constexpr int kBX = 32, kBY = 8;
constexpr int kColours[4][2] = {{0, 0}, {1, 0}, {0, 1}, {1, 1}};

// w = (1/eps) / (h1 h2) as a double-float pair per cell
__global__ void k_weights_df(const double* __restrict__ winv, double scale, float2* __restrict__ w, long N) {
  const long t = blockIdx.x * (long)blockDim.x + threadIdx.x;
  if (t >= N) return;
  const df v = df_from(scale * winv[t]);
  w[t] = make_float2(v.hi, v.lo);
}

// sqrt(w) 2^-ex in 62-bit fixed point (two 31-bit words), w = scale / eps
__global__ void k_weights_sqrt(const double* __restrict__ winv, double scale, double down, uint2* __restrict__ sw, long N) {
  const long t = blockIdx.x * (long)blockDim.x + threadIdx.x;
  if (t >= N) return;
  const double s = sqrt(scale * winv[t]) * down * 2147483648.0, hi = floor(s);
  sw[t] = make_uint2((unsigned)hi, (unsigned)((s - hi) * 2147483648.0));
}

__global__ void k_inv_eps(const double* __restrict__ eps, double* __restrict__ w64, float* __restrict__ w32, long N,
                          int* __restrict__ bad, unsigned long long* __restrict__ wmax,
                          unsigned long long* __restrict__ wmin) {
  const long t = blockIdx.x * (long)blockDim.x + threadIdx.x;
  if (t >= N) return;
  const double e = eps[t];
  if (!(e > 0.0) || !isfinite(e)) {
    atomicExch(bad, 1);
    w64[t] = 1.0;
    w32[t] = 1.0f;
    return;
  }
  w64[t] = 1.0 / e;
  w32[t] = float(1.0 / e);
  // positive doubles order like their bit patterns
  atomicMax(wmax, (unsigned long long)__double_as_longlong(1.0 / e));
  atomicMin(wmin, (unsigned long long)__double_as_longlong(1.0 / e));
}

__global__ void k_coarsen_w(const double* __restrict__ wf, int nf, double* __restrict__ wc, float* __restrict__ wc32,
                            int nc, int mc) {
  const int I = blockIdx.x * kBX + threadIdx.x, J = blockIdx.y * kBY + threadIdx.y;
  if (I >= nc || J >= mc) return;
  const long a = (long)(2 * J) * nf + 2 * I, b = a + nf;
  const double v = 0.25 * (wf[a] + wf[a + 1] + wf[b] + wf[b + 1]);
  wc[(long)J * nc + I] = v;
  wc32[(long)J * nc + I] = float(v);
}

// K3 = sum_c w_c u_c u_c^T + mu diag(2 m1, 2 m2, 2 m1 m2 s), u_c = T3^T v_c, s = m1 + m2
__global__ void k_patch_factors(const double* __restrict__ winv, int n, int m, double scale, double m1, double m2,
                                double mu, double* __restrict__ k64, float* __restrict__ k32) {
  const int i = blockIdx.x * kBX + threadIdx.x, j = blockIdx.y * kBY + threadIdx.y;
  if (i >= n || j >= m) return;
  const int im = (i + n - 1) % n, jm = (j + m - 1) % m;
  const double wSW = scale * winv[(long)jm * n + im], wNW = scale * winv[(long)j * n + im];
  const double wSE = scale * winv[(long)jm * n + i], wNE = scale * winv[(long)j * n + i];
  const double s = m1 + m2;
  const double u[4][3] = {{1, -1, s}, {-1, -1, -s}, {1, 1, -s}, {-1, 1, s}};
  const double w[4] = {wSW, wNW, wSE, wNE};
  double K[3][3] = {{mu * 2 * m1, 0, 0}, {0, mu * 2 * m2, 0}, {0, 0, mu * 2 * m1 * m2 * s}};
  for (int c = 0; c < 4; ++c)
    for (int a = 0; a < 3; ++a)
      for (int b = 0; b < 3; ++b) K[a][b] += w[c] * u[c][a] * u[c][b];
  // inverse via the adjugate (K3 is symmetric positive definite and well conditioned)
  const double c00 = K[1][1] * K[2][2] - K[1][2] * K[2][1];
  const double c01 = K[0][2] * K[2][1] - K[0][1] * K[2][2];
  const double c02 = K[0][1] * K[1][2] - K[0][2] * K[1][1];
  const double c11 = K[0][0] * K[2][2] - K[0][2] * K[2][0];
  const double c12 = K[0][2] * K[1][0] - K[0][0] * K[1][2];
  const double c22 = K[0][0] * K[1][1] - K[0][1] * K[1][0];
  const double det = K[0][0] * c00 + K[0][1] * (K[1][2] * K[2][0] - K[1][0] * K[2][2]) + K[0][2] * (K[1][0] * K[2][1] - K[1][1] * K[2][0]);
  const double id = 1.0 / det;
  const double inv[6] = {c00 * id, c01 * id, c02 * id, c11 * id, c12 * id, c22 * id};
  const long N = (long)n * m, e = (long)j * n + i;
  for (int q = 0; q < 6; ++q) {
    k64[q * N + e] = inv[q];
    k32[q * N + e] = float(inv[q]);
  }
}

// Dense coarsest-level matrices, column-major: entry (row, col) = operator applied to unit
// vector `col`, read at `row`.
__device__ __forceinline__ double2 coarse_edge_entry(const Lvl<double>& L, const Wts<double>& w, double mu,
                                                     const Ph<double>& p, int row, int col) {
  const int Nc = L.n * L.m;
  const UnitERd<double> r{L.n, L.m, col / Nc, col % Nc, p};
  const int kind = row / Nc, e = row % Nc, i = e % L.n, j = e / L.n;
  return kind == 0 ? A_x<double>(r, w, i, j) + mu * M_x<double>(r, L, i, j)
                   : A_y<double>(r, w, i, j) + mu * M_y<double>(r, L, i, j);
}
__device__ __forceinline__ double2 coarse_node_entry(const Lvl<double>& L, const Ph<double>& p, double shift, int row,
                                                     int col) {
  const int Nc = L.n * L.m;
  const UnitNRd<double> r{L.n, L.m, col, p};
  double2 v = P_at<double>(r, L, row % L.n, row / L.n);
  v.x += shift / Nc;  // k = 0: the constant mode gets eigenvalue `shift` (zero-mean solutions)
  return v;
}

// The lower triangles of every group of the launch (blockIdx.z).
__global__ void k_assemble(Lvl<double> L, Wts<double> w, double mu, const double* ph, const int* gamma, int node,
                           double2* K) {
  const int n = (node ? 1 : 2) * L.n * L.m, g = blockIdx.z;
  const int row = blockIdx.x * blockDim.x + threadIdx.x, col = blockIdx.y;
  if (row >= n || col > row) return;
  const Ph<double> p = load_ph<double>(ph, g);
  const double shift = gamma[g] ? P_diag<double>(L) : 0.0;
  K[((long)g * n + col) * n + row] =
      node ? coarse_node_entry(L, p, shift, row, col) : coarse_edge_entry(L, w, mu, p, row, col);
}

// The phase and k = 0 tables of one group (three copies each), from kernel arguments: one
// launch where six small host copies took longer than the operators that follow them.
__global__ void k_set_phases(double* d_ph, int* d_gamma, int ngroups, int g, double ar, double ai, double br, double bi,
                             int gamma) {
  const int rep = threadIdx.x;
  if (rep >= 3) return;
  double* p = d_ph + 4 * ((long)rep * ngroups + g);
  p[0] = ar; p[1] = ai; p[2] = br; p[3] = bi;
  d_gamma[(long)rep * ngroups + g] = gamma;
}

// Cholesky factor (lower) of the bs x bs matrix at Am (shared memory, entry (i, j), i >= j, at
// j ld + i), in place, by the whole thread block.  Returns false from every thread when a pivot
// is not positive.  A step is one reciprocal square root and two barriers.
__device__ __forceinline__ bool chol_shared(double2* Am, int ld, int n) {
  __shared__ double piv[2];  // pivot and its reciprocal
  __shared__ int good;
  const int tid = threadIdx.x, nt = blockDim.x;
  if (tid == 0) good = 1;
  for (int k = 0; k < n; ++k) {
    if (tid == 0) {
      const double d = Am[k * ld + k].x;
      const bool ok = d > 0.0 && isfinite(d);
      if (!ok) good = 0;
      const double r = ok ? sqrt(d) : 1.0;
      piv[0] = r;
      piv[1] = 1.0 / r;
    }
    __syncthreads();
    const double inv = piv[1];
    const int rem = n - k - 1;
    // the pivot column is scaled by the threads of its own entries after the update, which
    // forms the two scaled entries it needs from the unscaled ones
    for (int t = tid; t < rem * rem; t += nt) {
      const int jj = k + 1 + t / rem, ii = k + 1 + t % rem;
      if (ii < jj) continue;
      const double2 lik = inv * Am[k * ld + ii], ljk = inv * Am[k * ld + jj];
      double2 v = Am[jj * ld + ii];
      v.x -= lik.x * ljk.x + lik.y * ljk.y;
      v.y -= lik.y * ljk.x - lik.x * ljk.y;
      Am[jj * ld + ii] = v;
    }
    __syncthreads();
    for (int i = k + 1 + tid; i < n; i += nt) Am[k * ld + i] = inv * Am[k * ld + i];
    if (tid == 0) Am[k * ld + k] = make_double2(piv[0], 0.0);
  }
  __syncthreads();
  return good != 0;
}

// Inverse of the lower triangular bs x bs block of Am that starts at (k0, k0), in place (shared
// memory; bs <= kCoarseBlock): column c of the inverse by forward substitution, all columns at
// once, a barrier per row.  The block's columns are rewritten behind the row front in X.
__device__ __forceinline__ void invert_block(double2* Am, int ld, int k0, int bs) {
  __shared__ double2 X[kCoarseBlock][kCoarseBlock + 1];  // X[row][col]
  __shared__ double dinv[kCoarseBlock];
  const int tid = threadIdx.x, nt = blockDim.x;
  if (tid < bs) dinv[tid] = 1.0 / Am[(k0 + tid) * ld + k0 + tid].x;
  for (int t = tid; t < bs * bs; t += nt) X[t / bs][t % bs] = make_double2(t / bs == t % bs ? 1.0 : 0.0, 0.0);
  __syncthreads();
  for (int r = 0; r < bs; ++r) {
    // row r is complete but for its pivot: X[r] *= 1 / L_rr, then X[i] -= L_ir X[r] for i > r
    for (int c = tid; c <= r; c += nt) X[r][c] = dinv[r] * X[r][c];
    __syncthreads();
    for (int t = tid; t < (bs - r - 1) * (r + 1); t += nt) {
      const int i = r + 1 + t / (r + 1), c = t % (r + 1);
      X[i][c] = X[i][c] - cmul(Am[(k0 + r) * ld + k0 + i], X[r][c]);
    }
    __syncthreads();
  }
  for (int t = tid; t < bs * bs; t += nt) {
    const int i = t % bs, c = t / bs;
    if (i >= c) Am[(k0 + c) * ld + k0 + i] = X[i][c];
  }
  __syncthreads();
}

// Small coarsest systems (n <= kSmallFactor, the usual 4 x 4 mesh has 32 edges and 16 nodes):
// assembly and factorisation of both matrices of blockIdx.y's group in one launch (blockIdx.x:
// 0 edge, 1 node), the lower triangle in shared memory: the chain of pivots is what takes the
// time, and it makes no trip to global memory.
constexpr int kSmallFactor = 64;
__global__ void __launch_bounds__(256) k_coarse_factors(Lvl<double> L, Wts<double> w, double mu, const double* ph,
                                                        const int* gamma, double2* e64, float2* e32, double2* n64,
                                                        float2* n32, int* info) {
  extern __shared__ double2 Am[];  // entry (i, j), i >= j, at j (n + 1) + i
  const int g = blockIdx.y, node = blockIdx.x, Nc = L.n * L.m, n = node ? Nc : 2 * Nc, ld = n + 1;
  const int tid = threadIdx.x, nt = blockDim.x;
  const Ph<double> p = load_ph<double>(ph, g);
  const double shift = gamma[g] ? P_diag<double>(L) : 0.0;
  for (int t = tid; t < n * n; t += nt) {
    const int row = t % n, col = t / n;
    if (row >= col)
      Am[col * ld + row] = node ? coarse_node_entry(L, p, shift, row, col) : coarse_edge_entry(L, w, mu, p, row, col);
  }
  __syncthreads();
  if (!chol_shared(Am, ld, n) && tid == 0) info[node] = 1;
  for (int k0 = 0; k0 < n; k0 += kCoarseBlock) invert_block(Am, ld, k0, min(kCoarseBlock, n - k0));
  double2* F = (node ? n64 : e64) + (long)g * n * n;
  float2* F32 = (node ? n32 : e32) + (long)g * n * n;
  for (int t = tid; t < n * n; t += nt) {
    const int row = t % n, col = t / n;
    const double2 v = row >= col ? Am[col * ld + row] : make_double2(0.0, 0.0);
    F[t] = v;
    F32[t] = make_float2(float(v.x), float(v.y));
  }
}

// Larger ones (odd factors left on the coarsest mesh: 13 x 9 cells have 234 edges): a right-looking
// factorisation in blocks of 32 columns over many thread blocks and all groups (blockIdx.z or .y),
// three launches per block: the diagonal block and its inverse, the panel below it, the trailing
// matrix.  One thread block on the whole matrix took 3.6 ms at n = 234 (the FP64 rate of one SM).
__global__ void __launch_bounds__(256) k_chol_diag(double2* A, float2* A32, int n, int k0, int* info) {
  __shared__ double2 Am[kCoarseBlock * (kCoarseBlock + 1)];
  constexpr int ld = kCoarseBlock + 1;
  const int bs = min(kCoarseBlock, n - k0), tid = threadIdx.x, nt = blockDim.x;
  A += (long)blockIdx.x * n * n;
  A32 += (long)blockIdx.x * n * n;
  for (int t = tid; t < bs * bs; t += nt) {
    const int i = t % bs, j = t / bs;
    if (i >= j) Am[j * ld + i] = A[(long)(k0 + j) * n + k0 + i];
  }
  __syncthreads();
  if (!chol_shared(Am, ld, bs) && tid == 0) *info = 1;
  invert_block(Am, ld, 0, bs);
  for (int t = tid; t < bs * bs; t += nt) {
    const int i = t % bs, j = t / bs;
    const double2 v = i >= j ? Am[j * ld + i] : make_double2(0.0, 0.0);
    A[(long)(k0 + j) * n + k0 + i] = v;
    A32[(long)(k0 + j) * n + k0 + i] = make_float2(float(v.x), float(v.y));
  }
}
// rows i0 .. i0 + 31 below a full diagonal block: L(i, k) = sum_{c <= k} A(i, c) conj(Dinv(k, c))
__global__ void __launch_bounds__(256) k_chol_panel(double2* A, float2* A32, int n, int k0) {
  __shared__ double2 D[kCoarseBlock][kCoarseBlock + 1], P[kCoarseBlock][kCoarseBlock + 1];  // D[col][row], P[col][row]
  const int i0 = k0 + kCoarseBlock * (1 + blockIdx.x), rows = min(kCoarseBlock, n - i0), tid = threadIdx.x;
  A += (long)blockIdx.y * n * n;
  A32 += (long)blockIdx.y * n * n;
  for (int t = tid; t < kCoarseBlock * kCoarseBlock; t += blockDim.x) {
    const int i = t % kCoarseBlock, c = t / kCoarseBlock;
    D[c][i] = A[(long)(k0 + c) * n + k0 + i];
    P[c][i] = i < rows ? A[(long)(k0 + c) * n + i0 + i] : make_double2(0.0, 0.0);
  }
  __syncthreads();
  for (int t = tid; t < kCoarseBlock * kCoarseBlock; t += blockDim.x) {
    const int i = t % kCoarseBlock, k = t / kCoarseBlock;
    double2 v = make_double2(0.0, 0.0);
    for (int c = 0; c <= k; ++c) v = v + cmulc(D[c][k], P[c][i]);
    if (i < rows) {
      A[(long)(k0 + k) * n + i0 + i] = v;
      A32[(long)(k0 + k) * n + i0 + i] = make_float2(float(v.x), float(v.y));
    }
  }
}
// tile (blockIdx.x, blockIdx.y) of the trailing matrix, lower ones: A(i, j) -= sum_c L(i, c) conj(L(j, c))
__global__ void __launch_bounds__(256) k_chol_trail(double2* A, int n, int k0) {
  if (blockIdx.x < blockIdx.y) return;
  __shared__ double2 I[kCoarseBlock][kCoarseBlock + 1], J[kCoarseBlock][kCoarseBlock + 1];  // [col][row]
  const int i0 = k0 + kCoarseBlock * (1 + blockIdx.x), j0 = k0 + kCoarseBlock * (1 + blockIdx.y), tid = threadIdx.x;
  A += (long)blockIdx.z * n * n;
  for (int t = tid; t < kCoarseBlock * kCoarseBlock; t += blockDim.x) {
    const int i = t % kCoarseBlock, c = t / kCoarseBlock;
    I[c][i] = i0 + i < n ? A[(long)(k0 + c) * n + i0 + i] : make_double2(0.0, 0.0);
    J[c][i] = j0 + i < n ? A[(long)(k0 + c) * n + j0 + i] : make_double2(0.0, 0.0);
  }
  __syncthreads();
  for (int t = tid; t < kCoarseBlock * kCoarseBlock; t += blockDim.x) {
    const int i = t % kCoarseBlock, j = t / kCoarseBlock;
    if (i0 + i >= n || j0 + j > i0 + i) continue;
    double2 v = A[(long)(j0 + j) * n + i0 + i];
    for (int c = 0; c < kCoarseBlock; ++c) {
      const double2 a = I[c][i], b = J[c][j];
      v.x -= a.x * b.x + a.y * b.y;
      v.y -= a.y * b.x - a.x * b.y;
    }
    A[(long)(j0 + j) * n + i0 + i] = v;
  }
}

// Solve L L^* x = b for each column (one block per column; a hierarchy of one level).
constexpr int kSolveThreads = 512;
template <class T>
__global__ void __launch_bounds__(kSolveThreads) k_chol_solve(const cx<T>* __restrict__ Lbase, int n,
                                                              const cx<T>* __restrict__ B, long ldb,
                                                              cx<T>* __restrict__ X, long ldx, int cpg, int ngroups,
                                                              int goff) {
  extern __shared__ float4 fine_sm[];
  cx<T>* x = reinterpret_cast<cx<T>*>(fine_sm);
  const int c = blockIdx.x;
  for (int t = threadIdx.x; t < n; t += blockDim.x) x[t] = B[c * ldb + t];
  __syncthreads();
  coarse_solve<T>(Lbase + (long)((c / cpg + goff) % ngroups) * n * n, n, n, x, x, x + n);
  for (int t = threadIdx.x; t < n; t += blockDim.x) X[c * ldx + t] = x[t];
}

// One colour of the node-patch block Gauss-Seidel sweep for A + mu M.
template <class T>
__global__ void k_edge_smooth(Lvl<T> L, Wts<T> w, const T* __restrict__ k3, PatchCoef<T> pc, const double* ph, int cpg,
                              cx<T>* X, const cx<T>* __restrict__ B, long ld, int ci, int cj) {
  const int i = 2 * (blockIdx.x * kBX + threadIdx.x) + ci, j = 2 * (blockIdx.y * kBY + threadIdx.y) + cj;
  const int c = blockIdx.z;
  if (i >= L.n || j >= L.m) return;
  const Ph<T> p = load_ph<T>(ph, c / cpg);
  const ERd<T> r{X + c * ld, L.n, L.m, p};
  const ERd<T> rb{B + c * ld, L.n, L.m, p};
  if (inside(i, j, L.n, L.m, 1, 1))
    edge_smooth_at<T>(L, inner<T>(w), k3, pc, p, inner_e<T>(X + c * ld, L.n, L.m), inner_e<T>(B + c * ld, L.n, L.m),
                      X + c * ld, i, j);
  else
    edge_smooth_at<T>(L, w, k3, pc, p, r, rb, X + c * ld, i, j);
}

// One colour of point Gauss-Seidel for P = L^* M L.
template <class T>
__global__ void k_node_smooth(Lvl<T> L, const double* ph, int cpg, cx<T>* X, const cx<T>* __restrict__ B, long ld,
                              int ci, int cj) {
  const int i = 2 * (blockIdx.x * kBX + threadIdx.x) + ci, j = 2 * (blockIdx.y * kBY + threadIdx.y) + cj;
  const int c = blockIdx.z;
  if (i >= L.n || j >= L.m) return;
  const NRd<T> r{X + c * ld, L.n, L.m, load_ph<T>(ph, c / cpg)};
  if (inside(i, j, L.n, L.m, 1, 1))
    node_smooth_at<T>(L, inner_n<T>(X + c * ld, L.n), X + c * ld, B + c * ld, i, j);
  else
    node_smooth_at<T>(L, r, X + c * ld, B + c * ld, i, j);
}

template <class T> const cx<T>* edge_factor(const KData& K);
template <> const double2* edge_factor<double>(const KData& K) { return K.edge64; }
template <> const float2* edge_factor<float>(const KData& K) { return K.edge32; }
template <class T> const cx<T>* node_factor(const KData& K);
template <> const double2* node_factor<double>(const KData& K) { return K.node64; }
template <> const float2* node_factor<float>(const KData& K) { return K.node32; }
template <class T> const T* k3_of(const Level& L);
template <> const double* k3_of<double>(const Level& L) { return L.k3_64; }
template <> const float* k3_of<float>(const Level& L) { return L.k3_32; }

// Algorithmic bytes of one colour launch: every x value is read once (the
// patch residuals need the neighbours), the colour's edges (half of them) read b
// and write x, plus the colour's patch factors (6 reals per node) and 1/eps.
template <class T> double smooth_bytes(const Level& L, int ncols) {
  const double c = 2.0 * sizeof(T), D = (double)L.D(), N = (double)L.N();
  return ncols * (c * D + 2 * c * D / 2) + 6.0 * sizeof(T) * N / 4 + sizeof(T) * N;
}
// point smoother: read x once, read b and write x on a quarter of the nodes
template <class T> double node_smooth_bytes(const Level& L, int ncols) {
  const double c = 2.0 * sizeof(T), N = (double)L.N();
  return ncols * (c * N + 2 * c * N / 4);
}

inline dim3 half_grid(int n, int m, int ncols) {
  return dim3(((n + 1) / 2 + kBX - 1) / kBX, ((m + 1) / 2 + kBY - 1) / kBY, ncols);
}

}  // namespace

int num_levels(int n, int m, int coarsest) {
  if (n < 2 || m < 2 || coarsest < 2) return PBS_EINVAL;
  int L = 1;
  while (n % 2 == 0 && m % 2 == 0 && n / 2 >= coarsest && m / 2 >= coarsest && L < kMaxLevels) {
    n /= 2;
    m /= 2;
    ++L;
  }
  return L;
}

void build_hierarchy(DevMem& mem, Hierarchy& H, const double* d_eps, int coarsest, cudaStream_t s) {
  H.nlev = num_levels(H.n, H.m, coarsest);
  if (H.nlev < 1) fail(-1, "invalid mesh for the hierarchy");
  int* d_bad = (int*)mem.alloc(3 * sizeof(unsigned long long));
  unsigned long long* d_wmax = (unsigned long long*)d_bad + 1;
  H.allocs.push_back(d_bad);
  PBS_CUDA(cudaMemsetAsync(d_bad, 0, 2 * sizeof(unsigned long long), s));
  PBS_CUDA(cudaMemsetAsync(d_wmax + 1, 0xff, sizeof(unsigned long long), s));
  int n = H.n, m = H.m;
  for (int l = 0; l < H.nlev; ++l) {
    Level& L = H.lev[l];
    L.n = n;
    L.m = m;
    L.h1 = H.a / n;
    L.h2 = H.b / m;
    const long N = (long)n * m;
    L.winv64 = (double*)mem.alloc(N * sizeof(double));
    L.winv32 = (float*)mem.alloc(N * sizeof(float));
    L.k3_64 = (double*)mem.alloc(6 * N * sizeof(double));
    L.k3_32 = (float*)mem.alloc(6 * N * sizeof(float));
    H.allocs.insert(H.allocs.end(), {L.winv64, L.winv32, L.k3_64, L.k3_32});
    if (l == 0) {
      k_inv_eps<<<(unsigned)((N + 255) / 256), 256, 0, s>>>(d_eps, L.winv64, L.winv32, N, d_bad, d_wmax, d_wmax + 1);
    } else {
      const Level& F = H.lev[l - 1];
      k_coarsen_w<<<dim3((n + kBX - 1) / kBX, (m + kBY - 1) / kBY), dim3(kBX, kBY), 0, s>>>(F.winv64, F.n, L.winv64,
                                                                                           L.winv32, n, m);
    }
    PBS_LAUNCHED();
    if (l == 0) {
      L.wdf = (float2*)mem.alloc(N * sizeof(float2));
      H.allocs.push_back(L.wdf);
      L.sw = (uint2*)mem.alloc(N * sizeof(uint2));
      H.allocs.push_back(L.sw);
      k_weights_df<<<(unsigned)((N + 255) / 256), 256, 0, s>>>(L.winv64, 1.0 / (L.h1 * L.h2), L.wdf, N);
      PBS_LAUNCHED();
    }
    const double m1 = 2.0 / 3.0 * L.h2 / L.h1, m2 = 2.0 / 3.0 * L.h1 / L.h2;
    k_patch_factors<<<dim3((n + kBX - 1) / kBX, (m + kBY - 1) / kBY), dim3(kBX, kBY), 0, s>>>(
        L.winv64, n, m, 1.0 / (L.h1 * L.h2), m1, m2, H.mu, L.k3_64, L.k3_32);
    PBS_LAUNCHED();
    n /= 2;
    m /= 2;
  }
  int bad = 0;
  unsigned long long wlim[2] = {0, 0};
  PBS_CUDA(cudaMemcpyAsync(&bad, d_bad, sizeof(int), cudaMemcpyDeviceToHost, s));
  PBS_CUDA(cudaMemcpyAsync(wlim, d_wmax, sizeof(wlim), cudaMemcpyDeviceToHost, s));
  PBS_CUDA(cudaStreamSynchronize(s));
  if (bad) fail(-1, "eps must be finite and positive");
  std::memcpy(&H.winv_max, &wlim[0], sizeof(double));
  double winv_min = 0.0;
  std::memcpy(&winv_min, &wlim[1], sizeof(double));
  {
    Level& L = H.lev[0];
    const double scale = 1.0 / (L.h1 * L.h2);
    L.wmax = H.winv_max * scale;
    L.wmin = winv_min * scale;
    std::frexp(std::sqrt(L.wmax) * (1.0 + 1e-9), &L.sw_exp);  // sqrt(wmax) < 2^sw_exp
    k_weights_sqrt<<<(unsigned)((L.N() + 255) / 256), 256, 0, s>>>(L.winv64, scale, std::ldexp(1.0, -L.sw_exp), L.sw, L.N());
    PBS_LAUNCHED();
  }
  const Level& C = H.lev[H.nlev - 1];
  if (C.D() > kMaxCoarseEdges) fail(-1, "coarsest level too large for the dense solve (raise coarsest or use sides with more factors of 2)");
}

void free_hierarchy(DevMem& mem, Hierarchy& H) {
  for (void* p : H.allocs) mem.free(p);
  H.allocs.clear();
  H.nlev = 0;
}

void alloc_kdata(DevMem& mem, const Hierarchy& H, KData& K, int ngroups) {
  const Level& C = H.lev[H.nlev - 1];
  const int Dc = (int)C.D(), Nc = (int)C.N();
  if (K.ngroups == ngroups && K.Dc == Dc && K.d_info) return;
  free_kdata(mem, K);
  KData k;  // filled completely before it replaces K: a failed allocation leaves K empty
  k.owner = true;
  try {
    k.d_ph = (double*)mem.alloc(12ull * ngroups * sizeof(double));
    k.d_gamma = (int*)mem.alloc(3ull * ngroups * sizeof(int));
    k.edge64 = (double2*)mem.alloc((size_t)ngroups * Dc * Dc * sizeof(double2));
    k.edge32 = (float2*)mem.alloc((size_t)ngroups * Dc * Dc * sizeof(float2));
    k.node64 = (double2*)mem.alloc((size_t)ngroups * Nc * Nc * sizeof(double2));
    k.node32 = (float2*)mem.alloc((size_t)ngroups * Nc * Nc * sizeof(float2));
    k.d_info = (int*)mem.alloc(2 * sizeof(int));
  } catch (...) {
    free_kdata(mem, k);
    throw;
  }
  k.ngroups = ngroups;
  k.Dc = Dc;
  k.Nc = Nc;
  k.k1.assign(ngroups, 0.0);
  k.k2.assign(ngroups, 0.0);
  k.gamma.assign(ngroups, 0);
  K = k;
}

namespace {

// Bloch phases (alpha, beta) of a Bloch vector; exact ones at the lattice points.  Returns
// whether k = 0.
bool bloch_phases(const Hierarchy& H, double k1, double k2, double ph[4]) {
  ph[0] = std::cos(k1 * H.a);
  ph[1] = std::sin(k1 * H.a);
  ph[2] = std::cos(k2 * H.b);
  ph[3] = std::sin(k2 * H.b);
  const bool gamma = std::hypot(ph[0] - 1.0, ph[1]) < 1e-14 && std::hypot(ph[2] - 1.0, ph[3]) < 1e-14;
  if (gamma) {
    ph[0] = 1.0; ph[1] = 0.0; ph[2] = 1.0; ph[3] = 0.0;
  }
  return gamma;
}

void check_factors(const KData& K, cudaStream_t s) {
  int info[2] = {0, 0};
  PBS_CUDA(cudaMemcpyAsync(info, K.d_info, 2 * sizeof(int), cudaMemcpyDeviceToHost, s));
  PBS_CUDA(cudaStreamSynchronize(s));
  if (info[0] || info[1]) fail(PBS_ENUMERIC, "coarsest-level Cholesky factorisation failed");
}

// Coarsest factors of groups g0 .. g0 + ng - 1 from their phase tables.
void factor_groups(const Hierarchy& H, KData& K, int g0, int ng, cudaStream_t s) {
  const Level& C = H.lev[H.nlev - 1];
  const size_t Dc = K.Dc, Nc = K.Nc;
  PBS_CUDA(cudaMemsetAsync(K.d_info, 0, 2 * sizeof(int), s));
  if (K.Dc <= kSmallFactor) {
    const size_t smem = Dc * (Dc + 1) * sizeof(double2);
    static PerDeviceOnce once;
    once([] {
      PBS_CUDA(cudaFuncSetAttribute(k_coarse_factors, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    kSmallFactor * (kSmallFactor + 1) * (int)sizeof(double2)));
    });
    k_coarse_factors<<<dim3(2, ng), 256, smem, s>>>(C.lvl<double>(), C.wts<double>(), H.mu, K.d_ph + 4L * g0,
                                                    K.d_gamma + g0, K.edge64 + g0 * Dc * Dc, K.edge32 + g0 * Dc * Dc,
                                                    K.node64 + g0 * Nc * Nc, K.node32 + g0 * Nc * Nc, K.d_info);
    PBS_LAUNCHED();
    return;
  }
  for (int node = 0; node < 2; ++node) {
    const int n = node ? K.Nc : K.Dc;
    double2* F = (node ? K.node64 : K.edge64) + (size_t)g0 * n * n;
    float2* F32 = (node ? K.node32 : K.edge32) + (size_t)g0 * n * n;
    k_assemble<<<dim3((n + 127) / 128, n, ng), 128, 0, s>>>(C.lvl<double>(), C.wts<double>(), H.mu, K.d_ph + 4L * g0,
                                                            K.d_gamma + g0, node, F);
    PBS_LAUNCHED();
    for (int k0 = 0; k0 < n; k0 += kCoarseBlock) {
      k_chol_diag<<<ng, 256, 0, s>>>(F, F32, n, k0, K.d_info + node);
      PBS_LAUNCHED();
      const int tiles = (n - k0 - 1) / kCoarseBlock;  // row tiles below the block
      if (tiles == 0) break;
      k_chol_panel<<<dim3(tiles, ng), 256, 0, s>>>(F, F32, n, k0);
      PBS_LAUNCHED();
      k_chol_trail<<<dim3(tiles, tiles, ng), 256, 0, s>>>(F, n, k0);
      PBS_LAUNCHED();
    }
  }
}

// The tables of one group without its coarsest factors.
bool put_phases(const Hierarchy& H, KData& K, int g, double k1, double k2, double ph[4], cudaStream_t s) {
  if (g < 0 || g >= K.ngroups) fail(PBS_EINVAL, "group out of range");
  const bool gamma = bloch_phases(H, k1, k2, ph);
  K.k1[g] = k1;
  K.k2[g] = k2;
  K.gamma[g] = gamma;
  k_set_phases<<<1, 32, 0, s>>>(K.d_ph, K.d_gamma, K.ngroups, g, ph[0], ph[1], ph[2], ph[3], gamma ? 1 : 0);
  PBS_LAUNCHED();
  return gamma;
}

// Whether both coarsest matrices are so far from singular that their factorisation cannot
// fail: A_c + mu M_c >= (mu / 3) min(mx, my), against rounding errors of about n 2^-53 times
// the largest symbol value, and P_c >= |k|^2 a b / N_c (its lowest Bloch mode).
bool factors_certain(const Hierarchy& H, const double ph[4], bool gamma) {
  const Level& C = H.lev[H.nlev - 1];
  const double mx = C.h2 / C.h1, my = C.h1 / C.h2, mn = std::min(mx, my), mxy = std::max(mx, my);
  const double amax = 16.0 * H.winv_max / (C.h1 * C.h2) + H.mu * mxy;
  if (!(H.mu * mn / 3.0 > 1e-10 * amax) || !std::isfinite(amax)) return false;
  if (gamma) return true;
  const double t1 = std::hypot(ph[0] - 1.0, ph[1]), t2 = std::hypot(ph[2] - 1.0, ph[3]);
  const double low = 0.25 * mn * (t1 * t1 + t2 * t2) / (double)C.N();
  return std::isfinite(low) && low > 1e-10 * mxy;
}

}  // namespace

void set_group_k(DevMem& mem, const Hierarchy& H, KData& K, int g, double k1, double k2, cudaStream_t s) {
  double ph[4];
  put_phases(H, K, g, k1, k2, ph, s);
  factor_groups(H, K, g, 1, s);
  check_factors(K, s);
}

void set_group_phases(const Hierarchy& H, KData& K, int g, double k1, double k2, cudaStream_t s) {
  double ph[4];
  const bool gamma = put_phases(H, K, g, k1, k2, ph, s);
  if (factors_certain(H, ph, gamma)) return;
  factor_groups(H, K, g, 1, s);
  check_factors(K, s);
}

void set_all_k(const Hierarchy& H, KData& K, const double* ks, cudaStream_t s) {
  const int G = K.ngroups;
  std::vector<double> ph(12 * (size_t)G);
  std::vector<int> gi(3 * (size_t)G);
  for (int g = 0; g < G; ++g) {
    K.k1[g] = ks[2 * g];
    K.k2[g] = ks[2 * g + 1];
    K.gamma[g] = bloch_phases(H, ks[2 * g], ks[2 * g + 1], &ph[4 * g]);
    gi[g] = K.gamma[g];
  }
  for (int rep = 1; rep < 3; ++rep) {
    std::copy(ph.begin(), ph.begin() + 4 * G, ph.begin() + 4 * (size_t)G * rep);
    std::copy(gi.begin(), gi.begin() + G, gi.begin() + (size_t)G * rep);
  }
  PBS_CUDA(cudaMemcpyAsync(K.d_ph, ph.data(), ph.size() * sizeof(double), cudaMemcpyHostToDevice, s));
  PBS_CUDA(cudaMemcpyAsync(K.d_gamma, gi.data(), gi.size() * sizeof(int), cudaMemcpyHostToDevice, s));
  factor_groups(H, K, 0, G, s);
  check_factors(K, s);
}

void copy_group_k(KData& K, int src, int dst, cudaStream_t s) {
  if (src < 0 || dst < 0 || src >= K.ngroups || dst >= K.ngroups) fail(PBS_EINVAL, "group out of range");
  if (src == dst) return;
  K.k1[dst] = K.k1[src];
  K.k2[dst] = K.k2[src];
  K.gamma[dst] = K.gamma[src];
  for (int rep = 0; rep < 3; ++rep) {
    const long es = (long)rep * K.ngroups + src, ed = (long)rep * K.ngroups + dst;
    PBS_CUDA(cudaMemcpyAsync(K.d_ph + 4 * ed, K.d_ph + 4 * es, 4 * sizeof(double), cudaMemcpyDeviceToDevice, s));
    PBS_CUDA(cudaMemcpyAsync(K.d_gamma + ed, K.d_gamma + es, sizeof(int), cudaMemcpyDeviceToDevice, s));
  }
  const size_t de = (size_t)K.Dc * K.Dc, dn = (size_t)K.Nc * K.Nc;
  PBS_CUDA(cudaMemcpyAsync(K.edge64 + dst * de, K.edge64 + src * de, de * sizeof(double2), cudaMemcpyDeviceToDevice, s));
  PBS_CUDA(cudaMemcpyAsync(K.edge32 + dst * de, K.edge32 + src * de, de * sizeof(float2), cudaMemcpyDeviceToDevice, s));
  PBS_CUDA(cudaMemcpyAsync(K.node64 + dst * dn, K.node64 + src * dn, dn * sizeof(double2), cudaMemcpyDeviceToDevice, s));
  PBS_CUDA(cudaMemcpyAsync(K.node32 + dst * dn, K.node32 + src * dn, dn * sizeof(float2), cudaMemcpyDeviceToDevice, s));
}

KData kdata_view(const KData& K, int g) {
  KData v;
  v.ngroups = 1;
  v.Dc = K.Dc;
  v.Nc = K.Nc;
  v.d_ph = K.d_ph + 4 * g;
  v.d_gamma = K.d_gamma + g;
  v.edge64 = K.edge64 + (size_t)g * K.Dc * K.Dc;
  v.edge32 = K.edge32 + (size_t)g * K.Dc * K.Dc;
  v.node64 = K.node64 + (size_t)g * K.Nc * K.Nc;
  v.node32 = K.node32 + (size_t)g * K.Nc * K.Nc;
  v.d_info = K.d_info;
  v.k1 = {K.k1[g]};
  v.k2 = {K.k2[g]};
  v.gamma = {K.gamma[g]};
  v.owner = false;
  return v;
}

KData kdata_chunk(const KData& K, int v0) {
  KData v;
  v.ngroups = K.ngroups;
  v.Dc = K.Dc;
  v.Nc = K.Nc;
  v.d_ph = K.d_ph + 4L * v0;
  v.d_gamma = K.d_gamma + v0;
  v.edge64 = K.edge64;
  v.edge32 = K.edge32;
  v.node64 = K.node64;
  v.node32 = K.node32;
  v.d_info = K.d_info;
  v.k1 = K.k1;
  v.k2 = K.k2;
  v.gamma = K.gamma;
  v.goff = (K.goff + v0) % K.ngroups;
  v.owner = false;
  return v;
}

void free_kdata(DevMem& mem, KData& K) {
  if (K.owner)
    for (void* p : {(void*)K.d_ph, (void*)K.d_gamma, (void*)K.edge64, (void*)K.edge32, (void*)K.node64,
                    (void*)K.node32, (void*)K.d_info})
      if (p) mem.free(p);
  K = KData();
}

template <class T> void alloc_mg_work(DevMem& mem, const Hierarchy& H, int ncols, bool nodal, MgWork<T>& w) {
  free_mg_work<T>(mem, w);
  w.ncols = ncols;
  for (int l = 0; l < H.nlev; ++l) {
    const long len = nodal ? H.lev[l].N() : H.lev[l].D();
    const size_t bytes = (size_t)len * ncols * sizeof(cx<T>);
    w.r[l] = (cx<T>*)mem.alloc(bytes);
    if (l > 0) {
      w.x[l] = (cx<T>*)mem.alloc(bytes);
      w.b[l] = (cx<T>*)mem.alloc(bytes);
    }
  }
}

template <class T> void free_mg_work(DevMem& mem, MgWork<T>& w) {
  for (int l = 0; l < kMaxLevels; ++l) {
    for (cx<T>** p : {&w.x[l], &w.b[l], &w.r[l]}) {
      if (*p) mem.free(*p);
      *p = nullptr;
    }
  }
  w.ncols = 0;
}

namespace {

// Columns of `len` values at stride ld set to zero (one call when they are contiguous).
template <class T> void zero_columns(cx<T>* x, long ld, long len, int ncols, cudaStream_t s) {
  if (ld == len) {
    PBS_CUDA(cudaMemsetAsync(x, 0, (size_t)len * ncols * sizeof(cx<T>), s));
  } else {
    for (int c = 0; c < ncols; ++c) PBS_CUDA(cudaMemsetAsync(x + c * ld, 0, len * sizeof(cx<T>), s));
  }
}

// ---- fused coarse levels (tail.cuh) ----
// The tail covers level l and everything below when l is not the coarsest, has at most
// kTailMaxNodes nodes and its vectors fit in one CTA's shared memory.
//
// Layout of a tail from level l with K CTAs (the same offsets in every CTA): level vectors, the
// residuals, the coarsest factor where it fits.  Level l + t is spread over the cluster while its
// block rows divide by K and every CTA keeps kTailMinUnits units; the levels below run on the
// first CTA.  Returns the shared-memory bytes, or 0 where K does not fit the mesh.
constexpr int kTailMinUnits = 128;  // four warps: one per quarter of the SM
template <class T> size_t tail_layout(const Hierarchy& H, int l, bool nodal, int K, TailArgs<T>& a) {
  a.nl = H.nlev - l;
  a.lc = 0;
  a.K = K;
  if (a.nl > kTailMaxLevels) return 0;
  const int fields = nodal ? 1 : 2;
  int off = 0;
  bool spread = K > 1;
  for (int t = 0; t < a.nl; ++t) {
    const Level& L = H.lev[l + t];
    TailLevel<T>& v = a.lev[t];
    v.L = L.lvl<T>();
    if (t == a.nl - 1) {  // plain vectors
      v.H = v.V = v.Vb = 0;
      const int len = (int)(nodal ? L.N() : L.D());
      v.sx = off;
      v.sb = off + len;
      off += 2 * len;
      break;
    }
    v.H = L.n / 2;
    v.V = v.Vb = L.m / 2;
    spread = spread && v.V % K == 0 && 2 * v.H * v.V / K >= kTailMinUnits;
    if (spread) {
      v.Vb = v.V / K;
      a.lc = t + 1;
    }
    const int len = fields * 4 * tail_plane(v.H, v.Vb);
    v.sx = off;
    off += len;
    if (t > 0) {
      v.sb = off;
      off += len;
    }
    if (t == 0) a.sr = off;  // the top residual's own place
    if (t == 1) a.sr1 = off;
    if (t <= 1) off += len;
  }
  if (K > 1 && a.lc == 0) return 0;
  const Level& C = H.lev[H.nlev - 1];
  a.nfac = (int)(nodal ? C.N() : C.D());
  a.sw = off;
  off += a.nfac;
  a.sf = -1;
  if ((off + (long)a.nfac * (a.nfac + 1)) * (long)sizeof(cx<T>) <= kTailSmemBytes) {
    a.sf = off;
    off += a.nfac * (a.nfac + 1);
  }
  return (size_t)off * sizeof(cx<T>);
}

template <class T> bool tail_fits(const Hierarchy& H, int l, bool nodal, int K, TailArgs<T>& a, size_t* smem) {
  *smem = tail_layout<T>(H, l, nodal, K, a);
  return *smem > 0 && *smem <= (size_t)kTailSmemBytes;
}
template <class T> bool tail_from(const Hierarchy& H, int l, bool nodal) {
  if (l >= H.nlev - 1 || H.lev[l].N() > kTailMaxNodes) return false;
  TailArgs<T> a{};
  size_t smem = 0;
  return tail_fits<T>(H, l, nodal, 1, a, &smem);
}
// CTAs per column.  Binary64 levels are bound by the FP64 rate of the SMs they run on: up to four
// while every CTA still has an SM of its own (32 x 32, 20 columns: nodal 118 -> 77 us with four,
// edges 297 -> 191 us; 80 columns: 119 -> 232 us).  Binary32 levels are bound by latency, and a
// cluster barrier costs more than the split saves (64 x 64: nodal 63 -> 60 us with four CTAs,
// 32 x 32: 32 -> 46 us).
template <class T> int tail_want(int ncols) {
  if (sizeof(T) == 8) return ncols <= 38 ? 4 : ncols <= 76 ? 2 : 1;
  return 1;
}

// Threads per CTA: every warp takes part in every barrier, and on the smaller levels most of them
// have nothing else to do (64 x 64, binary32 nodal: 88 us with 256 threads, 63 with 512; 32 x 32:
// 38 and 32 us; binary64 on four CTAs, 128 units each: 77 us with 128 threads, 81 with 512).
template <class T> int tail_threads(const TailArgs<T>& a) {
  const int units = 2 * a.lev[0].H * a.lev[0].Vb;
  return units >= 512 ? 512 : units > 128 ? 256 : 128;
}

template <class T, bool CL> void launch_tail(const TailArgs<T>& a, bool nodal, int ncols, size_t smem,
                                                     cudaStream_t s) {
  static PerDeviceOnce once;
  once([] {
    PBS_CUDA(cudaFuncSetAttribute(k_node_tail<T, CL>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  kTailSmemBytes));
    PBS_CUDA(cudaFuncSetAttribute(k_edge_tail<T, CL>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  kTailSmemBytes));
  });
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(ncols * a.K);
  cfg.blockDim = dim3(tail_threads<T>(a));
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = a.K;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = CL ? 1 : 0;
  PBS_CUDA(cudaLaunchKernelEx(&cfg, nodal ? k_node_tail<T, CL> : k_edge_tail<T, CL>, a));
}

// Algorithmic bytes of a fused tail: the top right-hand sides in and solutions
// out, the patch factors of its edge levels and the coarsest factors of the
// groups its columns belong to (the level vectors stay on chip).
template <class T> double tail_bytes(const Hierarchy& H, int l, int ncols, int cpg, bool nodal) {
  const Level& L = H.lev[l];
  const Level& C = H.lev[H.nlev - 1];
  const double len = nodal ? (double)L.N() : (double)L.D(), nfac = nodal ? (double)C.N() : (double)C.D();
  double b = 2.0 * len * ncols * sizeof(cx<T>) + nfac * nfac * sizeof(cx<T>) * ((ncols + cpg - 1) / cpg);
  if (!nodal)
    for (int k = l; k < H.nlev - 1; ++k) b += 6.0 * sizeof(T) * H.lev[k].N();
  return b;
}

// The tiled fine-level nodal kernels need the halo to wrap at most once (sides of at
// least one tile plus both halos) and at most three sweeps per side.
constexpr int kFineMaxNu = 3;
constexpr size_t kSmemOptIn = 232448;  // largest dynamic shared memory a CTA may opt into (227 KB)
inline bool fine_fits(const Level& L, int ft) {
  const int need = ft + 8 * kFineMaxNu + 3;
  return L.n >= need && L.m >= need;
}
inline bool fine_tiled(const Level& L, int nu_pre, int nu_post) {
  return nu_pre >= 1 && nu_post >= 1 && nu_pre <= kFineMaxNu && nu_post <= kFineMaxNu && fine_fits(L, 32);
}
// shared memory of the tiled kernels for tile side ft and nu sweeps
template <class T> size_t fine_down_smem(int ft, int nu) {
  const size_t W = ft + 8 * nu + 3;
  return 2 * W * W * sizeof(cx<T>);
}
template <class T> size_t fine_up_smem(int ft, int nu) {
  const size_t W = ft + 8 * nu, Wc = W / 2 + 1;
  return (2 * W * W + Wc * Wc) * sizeof(cx<T>);
}
// the largest of fn(nu) over the sweep counts whose shared memory fits a CTA
template <class F> size_t fine_smem_cap(F&& fn) {
  size_t m = 0;
  for (int nu = 1; nu <= kFineMaxNu; ++nu)
    if (fn(nu) <= kSmemOptIn) m = std::max(m, fn(nu));
  return m;
}
template <class T, int FT> void set_fine_smem() {
  static PerDeviceOnce once;
  once([] {
    PBS_CUDA(cudaFuncSetAttribute(k_node_down<T, FT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)fine_smem_cap([](int nu) { return fine_down_smem<T>(FT, nu); })));
    PBS_CUDA(cudaFuncSetAttribute(k_node_up<T, FT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)fine_smem_cap([](int nu) { return fine_up_smem<T>(FT, nu); })));
  });
}
// launch shapes of the fine-level steps offered to the autotuner.  Cycles with one sweep per side run as
// row strips (ft rows, nt = 0), the others as tiles (side ft, nt threads).  One GB300, down + up step
// in us, strips of 16 / 32 / 64 rows against the best tile: FP32, 40 columns: 1024 x 1024 449 / 438 /
// 437, 846; 512 x 512 139 / 146 / 174, 234; 256 x 256 42 / 40 / 57, 65; 128 x 128 24 / 31 / 51, 29;
// FP64, 20 columns: 512 x 512 1107 / 1160 / 1147, 1549; 128 x 128 121 / 219 / 413, 189.  With few
// columns a strip is a chain of rows and little else, and short strips pay for their five halo rows:
// 4 / 8 / 16 rows against the best tile, 10 columns, FP32: 72 x 72 13 / 16 / 21, 22; 128 x 128 13 / 16 /
// 21, 22; 208 x 144 13 / 17 / 21, 25; 256 x 256 21 / 17 / 22; FP64: 72 x 72 43 / 70 / 119, 111; 128 x 128
// 76 / 68 / 119, 197; 256 x 256 201 / 176 / 210.  The first shape fits every level this path takes and is
// what runs without tuning: strips of 8 rows are faster than the tiles on every level and number of
// columns (one column, FP64, a cycle's fine steps: 72 x 72 76 against 110, 208 x 144 152 against 218,
// with 16 rows 125 and 251; 40 columns, FP32, 1024 x 1024 787 against 1875, with 16 rows 737).
struct FineShape {
  int ft, nt;
};
constexpr FineShape kStripShapes[] = {{8, 0}, {16, 0}, {32, 0}, {64, 0}, {4, 0}};
constexpr FineShape kTileShapes[] = {{32, 256}, {64, 512}, {64, 256}};
constexpr int kNumFineShapes = 5;
template <class T>
int fine_shapes(const Level& L, int nu, bool down, FineShape* out) {
  int n = 0;
  if (nu == 1) {
    for (const FineShape& f : kStripShapes) out[n++] = f;
    return n;
  }
  for (const FineShape& f : kTileShapes) {
    const size_t sm = down ? fine_down_smem<T>(f.ft, nu) : fine_up_smem<T>(f.ft, nu);
    if (fine_fits(L, f.ft) && sm <= kSmemOptIn) out[n++] = f;
  }
  return n;
}
// algorithmic bytes of a tiled step: each level vector read or written once
// (down: b in, x and the coarse right-hand side out; up: b, x, the coarse
// correction in, x out)
template <class T> double fine_bytes(const Level& L, int ncols, int, bool down) {
  const double v = (double)L.N() * ncols * sizeof(cx<T>);
  return down ? 2.25 * v : 3.25 * v;
}

template <class T> std::string fine_key(const Level& L, int ncols, int cpg) {
  return std::to_string(L.n) + "x" + std::to_string(L.m) + "|c" + std::to_string(ncols) + "|g" +
         std::to_string(cpg) + "|" + (sizeof(T) == 4 ? "f32" : "f64") + "|" + device_tag();
}

template <class T, int FT>
void launch_node_down(const Level& L, const Level& C, const KData& K, MgWork<T>& w, int l, const cx<T>* b,
                      const cx<T>* x0, long ld, int ncols, int cpg, int nu, int nt, cudaStream_t s) {
  set_fine_smem<T, FT>();
  const dim3 grid((L.n + FT - 1) / FT, (L.m + FT - 1) / FT, ncols);
  k_node_down<T, FT><<<grid, nt, fine_down_smem<T>(FT, nu), s>>>(L.lvl<T>(), C.n, C.m, K.d_ph, cpg, b, ld, x0, ld,
                                                                  w.r[l], L.N(), w.b[l + 1], C.N(), nu);
  PBS_LAUNCHED();
}

template <class T, int FT>
void launch_node_up(const Level& L, const Level& C, const KData& K, MgWork<T>& w, int l, const cx<T>* b, cx<T>* x,
                    long ld, int ncols, int cpg, int nu, int nt, cudaStream_t s) {
  set_fine_smem<T, FT>();
  const dim3 grid((L.n + FT - 1) / FT, (L.m + FT - 1) / FT, ncols);
  k_node_up<T, FT><<<grid, nt, fine_up_smem<T>(FT, nu), s>>>(L.lvl<T>(), C.n, C.m, K.d_ph, cpg, b, ld, w.r[l], L.N(),
                                                              w.x[l + 1], C.N(), x, ld, nu);
  PBS_LAUNCHED();
}

template <class T>
void launch_node_down_strips(const Level& L, const Level& C, const KData& K, MgWork<T>& w, int l, const cx<T>* b, const cx<T>* x0,
                             long ld, int ncols, int cpg, int rows, cudaStream_t s) {
  const dim3 grid(node_strip_blocks<kDownLanes>(L.n, L.m, rows), ncols);
  if (x0)
    k_node_down_strips<T, true><<<grid, 32 * kNodeStripWarps, 0, s>>>(L.lvl<T>(), K.d_ph, cpg, b, ld, x0, ld, w.r[l], L.N(),
                                                                      w.b[l + 1], C.N(), rows);
  else
    k_node_down_strips<T, false><<<grid, 32 * kNodeStripWarps, 0, s>>>(L.lvl<T>(), K.d_ph, cpg, b, ld, x0, ld, w.r[l], L.N(),
                                                                       w.b[l + 1], C.N(), rows);
  PBS_LAUNCHED();
}

template <class T>
void launch_node_up_strips(const Level& L, const Level& C, const KData& K, MgWork<T>& w, int l, const cx<T>* b, cx<T>* x, long ld,
                           int ncols, int cpg, int rows, cudaStream_t s) {
  k_node_up_strips<T><<<dim3(node_strip_blocks<kUpLanes>(L.n, L.m, rows), ncols), 32 * kNodeStripWarps, 0, s>>>(
      L.lvl<T>(), K.d_ph, cpg, b, ld, w.r[l], L.N(), w.x[l + 1], C.N(), x, ld, rows);
  PBS_LAUNCHED();
}

// The coarse levels from l down in one launch.
template <class T>
void run_tail(const Hierarchy& H, const KData& K, int l, const cx<T>* b, cx<T>* x, long ld, int ncols, int cpg,
              int nu_pre, int nu_post, bool nodal, cudaStream_t s) {
  TailArgs<T> a{};
  size_t smem = 0;
  int k = tail_want<T>(ncols);
  while (k > 1 && !tail_fits<T>(H, l, nodal, k, a, &smem)) k /= 2;
  if (!tail_fits<T>(H, l, nodal, k, a, &smem)) fail(-1, "coarse levels: no layout fits");
  for (int t = 0; t < a.nl; ++t) {
    const Level& L = H.lev[l + t];
    const Wts<T> w = L.wts<T>();
    a.lev[t].winv = w.winv;
    a.lev[t].wscale = w.scale;
    a.lev[t].k3 = k3_of<T>(L);
    a.lev[t].pc = patch_coef<T>(a.lev[t].L, H.mu);
  }
  a.b0 = b;
  a.x0 = x;
  a.ld0 = ld;
  a.ph = K.d_ph;
  a.cpg = cpg;
  a.factor = nodal ? node_factor<T>(K) : edge_factor<T>(K);
  a.ngroups = K.ngroups;
  a.goff = K.goff;
  a.nu_pre = nu_pre;
  a.nu_post = nu_post;
  const int cls = nodal ? KC_NODE_TAIL : KC_EDGE_TAIL;
  timer_begin(cls, s, tail_bytes<T>(H, l, ncols, cpg, nodal));
  if (k > 1) launch_tail<T, true>(a, nodal, ncols, smem, s);
  else launch_tail<T, false>(a, nodal, ncols, smem, s);
  timer_end(cls, s);
  PBS_LAUNCHED();
}

template <class T>
void edge_cycle(const Hierarchy& H, const KData& K, MgWork<T>& w, int l, const cx<T>* b, cx<T>* x, long ld, int ncols,
                int cpg, int nu_pre, int nu_post, cudaStream_t s) {
  const Level& L = H.lev[l];
  if (l == H.nlev - 1) {
    k_chol_solve<T><<<ncols, kSolveThreads, 2 * (size_t)L.D() * sizeof(cx<T>), s>>>(edge_factor<T>(K), (int)L.D(), b, ld, x, ld,
                                                                                cpg, K.ngroups, K.goff);
    PBS_LAUNCHED();
    return;
  }
  if (tail_from<T>(H, l, false)) {
    run_tail<T>(H, K, l, b, x, ld, ncols, cpg, nu_pre, nu_post, false, s);
    return;
  }
  zero_columns<T>(x, ld, L.D(), ncols, s);
  const Lvl<T> lv = L.lvl<T>();
  const Wts<T> wt = L.wts<T>();
  const T mu = T(H.mu);
  const PatchCoef<T> pc = patch_coef<T>(lv, H.mu);
  for (int it = 0; it < nu_pre; ++it)
    for (int q = 0; q < 4; ++q) {
      timer_begin(KC_EDGE_SMOOTH, s, smooth_bytes<T>(L, ncols));
      k_edge_smooth<T><<<half_grid(L.n, L.m, ncols), dim3(kBX, kBY), 0, s>>>(lv, wt, k3_of<T>(L), pc, K.d_ph, cpg, x,
                                                                             b, ld, kColours[q][0], kColours[q][1]);
      timer_end(KC_EDGE_SMOOTH, s);
      PBS_LAUNCHED();
    }
  const Level& C = H.lev[l + 1];
  const long ldc = C.D();
  apply_edge<T>(L, K.d_ph, cpg, x, w.r[l], b, ld, ncols, T(-1), -mu, T(0), nullptr, T(1), s);
  restrict_edge<T>(L, C, K.d_ph, cpg, w.r[l], ld, w.b[l + 1], ldc, ncols, s);
  edge_cycle<T>(H, K, w, l + 1, w.b[l + 1], w.x[l + 1], ldc, ncols, cpg, nu_pre, nu_post, s);
  prolong_edge<T>(L, C, K.d_ph, cpg, w.x[l + 1], ldc, x, ld, ncols, true, s);
  for (int it = 0; it < nu_post; ++it)
    for (int q = 3; q >= 0; --q) {
      timer_begin(KC_EDGE_SMOOTH, s, smooth_bytes<T>(L, ncols));
      k_edge_smooth<T><<<half_grid(L.n, L.m, ncols), dim3(kBX, kBY), 0, s>>>(lv, wt, k3_of<T>(L), pc, K.d_ph, cpg, x,
                                                                             b, ld, kColours[q][0], kColours[q][1]);
      timer_end(KC_EDGE_SMOOTH, s);
      PBS_LAUNCHED();
    }
}

// A nodal cycle can continue from a given iterate when its top level runs the tiled steps
// (whose first kernel stages the iterate as it stages the right-hand side).
template <class T> bool takes_guess(const Hierarchy& H, int l, int nu_pre, int nu_post) {
  return l < H.nlev - 1 && !tail_from<T>(H, l, true) && fine_tiled(H.lev[l], nu_pre, nu_post);
}

template <class T>
void node_cycle(const Hierarchy& H, const KData& K, MgWork<T>& w, int l, const cx<T>* b, cx<T>* x, long ld, int ncols,
                int cpg, int nu_pre, int nu_post, cudaStream_t s, const cx<T>* x0 = nullptr) {
  const Level& L = H.lev[l];
  if (x0 && !takes_guess<T>(H, l, nu_pre, nu_post)) fail(-1, "nodal cycle: initial iterate on an untiled level");
  if (l == H.nlev - 1) {
    k_chol_solve<T><<<ncols, kSolveThreads, 2 * (size_t)L.N() * sizeof(cx<T>), s>>>(node_factor<T>(K), (int)L.N(), b, ld, x, ld,
                                                                                cpg, K.ngroups, K.goff);
    PBS_LAUNCHED();
    return;
  }
  if (tail_from<T>(H, l, true)) {
    run_tail<T>(H, K, l, b, x, ld, ncols, cpg, nu_pre, nu_post, true, s);
    return;
  }
  if (fine_tiled(L, nu_pre, nu_post)) {
    const Level& C = H.lev[l + 1];
    const auto down = [&](const FineShape& f) {
      if (f.nt == 0) launch_node_down_strips<T>(L, C, K, w, l, b, x0, ld, ncols, cpg, f.ft, s);
      else if (f.ft == 64) launch_node_down<T, 64>(L, C, K, w, l, b, x0, ld, ncols, cpg, nu_pre, f.nt, s);
      else launch_node_down<T, 32>(L, C, K, w, l, b, x0, ld, ncols, cpg, nu_pre, f.nt, s);
    };
    const auto up = [&](const FineShape& f) {
      if (f.nt == 0) launch_node_up_strips<T>(L, C, K, w, l, b, x, ld, ncols, cpg, f.ft, s);
      else if (f.ft == 64) launch_node_up<T, 64>(L, C, K, w, l, b, x, ld, ncols, cpg, nu_post, f.nt, s);
      else launch_node_up<T, 32>(L, C, K, w, l, b, x, ld, ncols, cpg, nu_post, f.nt, s);
    };
    FineShape fd[kNumFineShapes], fu[kNumFineShapes];
    const int nd = fine_shapes<T>(L, nu_pre, true, fd), nup = fine_shapes<T>(L, nu_post, false, fu);
    // both steps are idempotent (the down step reads b, the up step b, its saved
    // pre-smoothed x and the coarse correction, and neither writes what it reads)
    // (strips name their candidates in the key: plain keys with one sweep per side hold an earlier
    // build's choices among tiles, other shapes under the same index)
    const auto key = [&](const char* step, int nu, const FineShape* f, int count) {
      std::string k = step;
      if (nu == 1) {
        k += "strips";
        for (int c = 0; c < count; ++c) k += (c ? "." : "") + std::to_string(f[c].ft);
        k += "|";
      }
      return k + fine_key<T>(L, ncols, cpg) + "|nu" + std::to_string(nu);
    };
    const int pd = tune_pick(key("node_down|", nu_pre, fd, nd), nd, [&](int c) { down(fd[c]); }, s);
    timer_begin(KC_NODE_SMOOTH, s, fine_bytes<T>(L, ncols, nu_pre, true));
    down(fd[pd]);
    timer_end(KC_NODE_SMOOTH, s);
    node_cycle<T>(H, K, w, l + 1, w.b[l + 1], w.x[l + 1], C.N(), ncols, cpg, nu_pre, nu_post, s);
    const int pu = tune_pick(key("node_up|", nu_post, fu, nup), nup, [&](int c) { up(fu[c]); }, s);
    timer_begin(KC_NODE_SMOOTH, s, fine_bytes<T>(L, ncols, nu_post, false));
    up(fu[pu]);
    timer_end(KC_NODE_SMOOTH, s);
    return;
  }
  zero_columns<T>(x, ld, L.N(), ncols, s);
  const Lvl<T> lv = L.lvl<T>();
  for (int it = 0; it < nu_pre; ++it)
    for (int q = 0; q < 4; ++q) {
      timer_begin(KC_NODE_SMOOTH, s, node_smooth_bytes<T>(L, ncols));
      k_node_smooth<T><<<half_grid(L.n, L.m, ncols), dim3(kBX, kBY), 0, s>>>(lv, K.d_ph, cpg, x, b, ld,
                                                                             kColours[q][0], kColours[q][1]);
      timer_end(KC_NODE_SMOOTH, s);
      PBS_LAUNCHED();
    }
  const Level& C = H.lev[l + 1];
  const long ldc = C.N();
  apply_nodal<T>(L, K.d_ph, cpg, x, w.r[l], b, ld, ncols, T(-1), T(1), s);
  restrict_node<T>(L, C, K.d_ph, cpg, w.r[l], ld, w.b[l + 1], ldc, ncols, s);
  node_cycle<T>(H, K, w, l + 1, w.b[l + 1], w.x[l + 1], ldc, ncols, cpg, nu_pre, nu_post, s);
  prolong_node<T>(L, C, K.d_ph, cpg, w.x[l + 1], ldc, x, ld, ncols, true, s);
  for (int it = 0; it < nu_post; ++it)
    for (int q = 3; q >= 0; --q) {
      timer_begin(KC_NODE_SMOOTH, s, node_smooth_bytes<T>(L, ncols));
      k_node_smooth<T><<<half_grid(L.n, L.m, ncols), dim3(kBX, kBY), 0, s>>>(lv, K.d_ph, cpg, x, b, ld,
                                                                             kColours[q][0], kColours[q][1]);
      timer_end(KC_NODE_SMOOTH, s);
      PBS_LAUNCHED();
    }
}

}  // namespace

template <class T>
void edge_vcycle(const Hierarchy& H, const KData& K, MgWork<T>& w, int l0, const cx<T>* X, cx<T>* Y, long ld,
                 int ncols, int cpg, int nu_pre, int nu_post, cudaStream_t s) {
  if (ncols <= 0) return;
  if (ncols > w.ncols) fail(-1, "multigrid workspace too small");
  edge_cycle<T>(H, K, w, l0, X, Y, ld, ncols, cpg, nu_pre, nu_post, s);
}

template <class T>
void nodal_vcycle(const Hierarchy& H, const KData& K, MgWork<T>& w, int l0, const cx<T>* X, cx<T>* Y, long ld,
                  int ncols, int cpg, int nu_pre, int nu_post, cudaStream_t s) {
  if (ncols <= 0) return;
  if (ncols > w.ncols) fail(-1, "multigrid workspace too small");
  node_cycle<T>(H, K, w, l0, X, Y, ld, ncols, cpg, nu_pre, nu_post, s);
}

template <class T> bool nodal_takes_guess(const Hierarchy& H, int l0, int nu_pre, int nu_post) {
  return takes_guess<T>(H, l0, nu_pre, nu_post);
}

template <class T>
void nodal_vcycle_from(const Hierarchy& H, const KData& K, MgWork<T>& w, int l0, const cx<T>* X, const cx<T>* X0,
                       cx<T>* Y, long ld, int ncols, int cpg, int nu_pre, int nu_post, cudaStream_t s) {
  if (ncols <= 0) return;
  if (ncols > w.ncols) fail(-1, "multigrid workspace too small");
  node_cycle<T>(H, K, w, l0, X, Y, ld, ncols, cpg, nu_pre, nu_post, s, X0);
}

#define PBS_INST_MG(T)                                                                                            \
  template bool nodal_takes_guess<T>(const Hierarchy&, int, int, int);                                            \
  template void nodal_vcycle_from<T>(const Hierarchy&, const KData&, MgWork<T>&, int, const cx<T>*, const cx<T>*, \
                                     cx<T>*, long, int, int, int, int, cudaStream_t);                             \
  template void alloc_mg_work<T>(DevMem&, const Hierarchy&, int, bool, MgWork<T>&);                               \
  template void free_mg_work<T>(DevMem&, MgWork<T>&);                                                             \
  template void edge_vcycle<T>(const Hierarchy&, const KData&, MgWork<T>&, int, const cx<T>*, cx<T>*, long, int, \
                               int, int, int, cudaStream_t);                                                      \
  template void nodal_vcycle<T>(const Hierarchy&, const KData&, MgWork<T>&, int, const cx<T>*, cx<T>*, long, int, \
                                int, int, int, cudaStream_t);
PBS_INST_MG(double)
PBS_INST_MG(float)

}  // namespace pbs
