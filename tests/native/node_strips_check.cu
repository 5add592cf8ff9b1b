// GPU check of the row-pipelined nodal steps (csrc/node_strips.cuh) against the tiled ones
// (csrc/nodal_tiles.cuh), from zero and from a given iterate, in both precisions, on levels whose width
// leaves part of a strip and whose height leaves part of a row block; the rows per strip must not
// change a bit.  Prints "ok".
//
// Both evaluate the same sums; the compiler may fuse them differently.  A node update has at most 12
// roundings of terms of up to 5.5 max |x| (the coefficients of this level), times 1 / diagonal = 0.36:
// 24 u max |x|, and a colour passes its neighbours' differences on at a factor of at most 1: 96 u over
// four colours.  The residual adds 12 u 5.5 and takes x with 2 x 5.5, its restriction sums weights 4.
#include "node_strips.cuh"
#include "nodal_tiles.cuh"

#include <cmath>
#include <cstdio>
#include <cstring>
#include <random>
#include <vector>

using namespace pbs;

static std::mt19937_64 rng(5);
template <class V> static V* upload(const std::vector<V>& v) {
  V* d = nullptr;
  cudaMalloc(&d, sizeof(V) * v.size());
  cudaMemcpy(d, v.data(), sizeof(V) * v.size(), cudaMemcpyHostToDevice);
  return d;
}
template <class V> static std::vector<V> download(const V* d, size_t n) {
  std::vector<V> v(n);
  cudaMemcpy(v.data(), d, sizeof(V) * n, cudaMemcpyDeviceToHost);
  return v;
}
template <class T> static std::vector<cx<T>> noise(size_t n) {
  std::uniform_real_distribution<double> u(-1.0, 1.0);
  std::vector<cx<T>> v(n);
  for (auto& z : v) z = mk<T>(T(u(rng)), T(u(rng)));
  return v;
}

template <class T> static bool run(int n, int m) {
  bool ok = true;
  std::vector<cx<T>> reference[2][3];
  const int cols = 3, cpg = 2, nc = n / 2, mc = m / 2;
  const long N = (long)n * m, Nc = N / 4, ld = N + 4;
  const Lvl<T> L{n, m, T(1.3), T(1.0 / 1.3)};
  std::vector<double> ph;
  for (double a : {0.7, -1.9, 2.2, 0.4}) ph.insert(ph.end(), {std::cos(a), std::sin(a)});
  double* dph = upload(ph);
  cx<T>*b = upload(noise<T>(cols * ld)), *x0 = upload(noise<T>(cols * ld)), *xc = upload(noise<T>(cols * Nc));
  const std::vector<cx<T>> mark(cols * ld, mk<T>(T(9), T(9)));
  for (int rows : {16, 32, 64})
  for (int guess = 0; guess < 2; ++guess) {
    cx<T>* out[2][3];
    for (int k = 0; k < 2; ++k)
      for (int t = 0; t < 3; ++t) out[k][t] = upload(mark);
    const size_t sd = 2ull * 43 * 43 * sizeof(cx<T>), su = (2ull * 40 * 40 + 21 * 21) * sizeof(cx<T>);
    cudaFuncSetAttribute(k_node_down<T, 32>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sd);
    cudaFuncSetAttribute(k_node_up<T, 32>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)su);
    const dim3 tiles((n + 31) / 32, (m + 31) / 32, cols);
    k_node_down<T, 32><<<tiles, 256, sd>>>(L, nc, mc, dph, cpg, b, ld, guess ? x0 : nullptr, ld, out[0][0], ld, out[0][1], Nc, 1);
    k_node_up<T, 32><<<tiles, 256, su>>>(L, nc, mc, dph, cpg, b, ld, x0, ld, xc, Nc, out[0][2], ld, 1);
    const dim3 down(node_strip_blocks<kDownLanes>(n, m, rows), cols), up(node_strip_blocks<kUpLanes>(n, m, rows), cols);
    if (guess) k_node_down_strips<T, true><<<down, 32 * kNodeStripWarps>>>(L, dph, cpg, b, ld, x0, ld, out[1][0], ld, out[1][1], Nc, rows);
    else k_node_down_strips<T, false><<<down, 32 * kNodeStripWarps>>>(L, dph, cpg, b, ld, x0, ld, out[1][0], ld, out[1][1], Nc, rows);
    k_node_up_strips<T><<<up, 32 * kNodeStripWarps>>>(L, dph, cpg, b, ld, x0, ld, xc, Nc, out[1][2], ld, rows);
    const cudaError_t err = cudaDeviceSynchronize();
    const char* what[3] = {"x", "restricted residual", "x up"};
    for (int t = 0; t < 3; ++t) {
      const auto p = download(out[0][t], mark.size()), q = download(out[1][t], mark.size());
      const double u = sizeof(T) == 4 ? 0x1p-24 : 0x1p-53, big = 4.0;  // max |x| of these fields
      const double tol = t == 1 ? 4 * (2 * 5.5 * 96 + 66) * u * big : 96 * u * big;
      long bad = 0, first = -1;
      double worst = 0.0;
      for (size_t k = 0; k < p.size(); ++k) {
        const double e = std::max(std::fabs((double)p[k].x - q[k].x), std::fabs((double)p[k].y - q[k].y));
        worst = std::max(worst, e);
        if (!(e <= tol)) {
          if (first < 0) first = (long)k;
          ++bad;
        }
      }
      auto& same = reference[guess][t];
      if (same.empty()) same = q;
      if (std::memcmp(same.data(), q.data(), sizeof(cx<T>) * q.size()) != 0) {
        std::printf("%d x %d rows %d f%d guess %d %s: depends on the rows of a strip\n", n, m, rows, (int)sizeof(T) * 8, guess,
                    what[t]);
        ok = false;
      }
      if (bad || err != cudaSuccess) {
        std::printf("%d x %d rows %d f%d guess %d %s: %ld values differ, first %ld, by up to %.2e (%s)\n", n, m, rows,
                    (int)sizeof(T) * 8, guess, what[t], bad, first, worst, cudaGetErrorString(err));
        ok = false;
      }
    }
    for (int k = 0; k < 2; ++k)
      for (int t = 0; t < 3; ++t) cudaFree(out[k][t]);
  }
  for (void* q : {(void*)dph, (void*)b, (void*)x0, (void*)xc}) cudaFree(q);
  return ok;
}

int main() {
  bool ok = true;
  const int sizes[][2] = {{60, 60}, {64, 96}, {108, 64}, {112, 72}, {128, 128}, {62, 134}};
  for (auto& s : sizes) {
    ok = run<float>(s[0], s[1]) && ok;
    ok = run<double>(s[0], s[1]) && ok;
  }
  std::puts(ok ? "ok" : "not ok");
  return ok ? 0 : 1;
}
