// Solve with the coarsest level's factor by a whole thread block (the fused coarse levels of
// tail.cuh, and hierarchies of one level).
#pragma once
#include "common.cuh"

namespace pbs {

// ---- coarsest level ----------------------------------------------------------
// The coarsest factor of A = L L^* is stored with its 32 x 32 diagonal blocks inverted: lower,
// column-major, F(i, k) = L(i, k) below the diagonal blocks, L_bb^{-1} inside them.  A triangular
// solve is then a matrix-vector product per block instead of a chain of 32 divisions, and the
// whole thread block works on it.  (Inverting the triangular blocks of 32 keeps the accuracy of
// substitution, whose error has the same bound, cond(L_bb) times the rounding.)
constexpr int kCoarseBlock = 32;

// x <- (L L^*)^{-1} b by the whole thread block (blockDim.x a multiple of 32; every thread calls
// it; 512 threads take a block's 32 rows at once, 16 lanes each): F at leading dimension ld (n + 1
// in shared memory keeps rows and columns free of bank conflicts); b, x and w are vectors in shared
// memory, b may be x.  Ends with a barrier.
template <class T>
__device__ __forceinline__ void coarse_solve(const cx<T>* F, int ld, int n, const cx<T>* b, cx<T>* x, cx<T>* w) {
  const int tid = threadIdx.x, nt = blockDim.x, seg = tid & 15;
  // f(row) summed over the 16 lanes of a row, handed to g(row, sum) on the first of them
  auto rows = [&](int bs, auto&& f, auto&& g) {
    for (int r0 = 0; r0 < bs; r0 += nt >> 4) {
      const int row = r0 + (tid >> 4);
      cx<T> v = row < bs ? f(row) : czero<T>();
      for (int o = 8; o > 0; o >>= 1) {
        v.x += __shfl_xor_sync(0xffffffffu, v.x, o);
        v.y += __shfl_xor_sync(0xffffffffu, v.y, o);
      }
      if (row < bs && seg == 0) g(row, v);
    }
    __syncthreads();
  };
  for (int j = tid; j < n; j += nt) w[j] = b[j];
  __syncthreads();
  // L y = b, y in x
  for (int k0 = 0; k0 < n; k0 += kCoarseBlock) {
    const int bs = min(kCoarseBlock, n - k0);
    rows(
        bs,
        [&](int row) {
          cx<T> acc = czero<T>();
          for (int k = seg; k <= row; k += 16) acc = acc + cmul(F[(long)(k0 + k) * ld + k0 + row], w[k0 + k]);
          return acc;
        },
        [&](int row, cx<T> v) { x[k0 + row] = v; });
    for (int i = k0 + bs + tid; i < n; i += nt) {
      cx<T> r = w[i];
#pragma unroll 8
      for (int k = 0; k < bs; ++k) r = r - cmul(F[(long)(k0 + k) * ld + i], x[k0 + k]);
      w[i] = r;
    }
    __syncthreads();
  }
  // L^* x = y, (L^*)(k, i) = conj(L(i, k))
  for (int k0 = (n - 1) / kCoarseBlock * kCoarseBlock; k0 >= 0; k0 -= kCoarseBlock) {
    const int bs = min(kCoarseBlock, n - k0);
    rows(
        bs,
        [&](int row) {
          cx<T> acc = czero<T>();
          for (int i = k0 + bs + seg; i < n; i += 16) acc = acc + cmulc(F[(long)(k0 + row) * ld + i], x[i]);
          return acc;
        },
        [&](int row, cx<T> v) { w[k0 + row] = x[k0 + row] - v; });
    rows(
        bs,
        [&](int row) {
          cx<T> acc = czero<T>();
          for (int i = row + seg; i < bs; i += 16) acc = acc + cmulc(F[(long)(k0 + row) * ld + k0 + i], w[k0 + i]);
          return acc;
        },
        [&](int row, cx<T> v) { x[k0 + row] = v; });
  }
}

}  // namespace pbs
