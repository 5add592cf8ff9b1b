// GPU check of the tensor-core Gram (csrc/gram_tc.cu) with several groups in a launch: each group's
// partial sums are those of a launch with that group alone, bit for bit.  Prints "ok".
// (The library's launch and error helpers are stood in for below.)
#include "gram_tc.cu"

#include <cmath>
#include <cstdio>
#include <cstring>
#include <random>

namespace pbs {
void check_cuda(cudaError_t e, const char* what) {
  if (e != cudaSuccess) fail(PBS_ECUDA, std::string(what) + ": " + cudaGetErrorString(e));
}
void fail(int, const std::string& what) {
  std::printf("failed: %s\n", what.c_str());
  std::exit(2);
}
void count_launch() {}
}  // namespace pbs

using namespace pbs;

static std::mt19937_64 rng(5);
template <class T> T* upload(const std::vector<T>& v) {
  T* d = nullptr;
  PBS_CUDA(cudaMalloc(&d, sizeof(T) * v.size()));
  PBS_CUDA(cudaMemcpy(d, v.data(), sizeof(T) * v.size(), cudaMemcpyHostToDevice));
  return d;
}

// three arrays of p columns per group (a trial block [E, P, W]), phases of the group's own
static bool run(int n, int m, int p, int groups) {
  const int q = 3 * p, ne = q * (q + 1) / 2;
  Level L;
  L.n = n;
  L.m = m;
  L.h1 = 1.0 / n;
  L.h2 = 0.75 / m;
  std::normal_distribution<double> normal;
  std::vector<double2> X[3];
  for (int r = 0; r < 3; ++r) {
    X[r].resize((size_t)groups * p * L.D());
    for (size_t t = 0; t < X[r].size(); ++t) {
      const double s = std::ldexp(1.0, (int)(t / L.D()) * 3);  // every column at a scale of its own
      X[r][t] = make_double2(s * normal(rng), s * normal(rng));
    }
  }
  std::vector<uint2> sw(L.N());
  for (auto& w : sw) w = make_uint2((unsigned)(rng() >> 33) | 0x40000000u, (unsigned)(rng() >> 33));
  std::vector<double> ph(4 * groups);
  for (int g = 0; g < groups; ++g) {
    const double t = 0.3 + g, u = -1.1 * g;
    ph[4 * g] = std::cos(t), ph[4 * g + 1] = std::sin(t), ph[4 * g + 2] = std::cos(u), ph[4 * g + 3] = std::sin(u);
  }
  double2* dX[3] = {upload(X[0]), upload(X[1]), upload(X[2])};
  L.sw = upload(sw);
  double* dph = upload(ph);
  const int np = std::min<long>(7, gram_tc_chunks(n, m));
  int *de = upload(std::vector<int>(gram_tc_scratch(q, groups) / sizeof(int)));
  const size_t len = (size_t)np * 2 * ne;
  double2 *all = upload(std::vector<double2>(len * groups)), *one = upload(std::vector<double2>(len));
  gram_tc(L, dph, Roles{{dX[0], dX[1], dX[2]}, p, L.D()}, q, groups, np, all, de, 0);
  PBS_CUDA(cudaDeviceSynchronize());
  std::vector<double2> a(len * groups), b(len);
  PBS_CUDA(cudaMemcpy(a.data(), all, sizeof(double2) * a.size(), cudaMemcpyDeviceToHost));
  bool ok = true;
  for (int g = 0; g < groups; ++g) {
    const long at = (long)g * p * L.D();
    gram_tc(L, dph + 4 * g, Roles{{dX[0] + at, dX[1] + at, dX[2] + at}, p, L.D()}, q, 1, np, one, de, 0);
    PBS_CUDA(cudaDeviceSynchronize());
    PBS_CUDA(cudaMemcpy(b.data(), one, sizeof(double2) * len, cudaMemcpyDeviceToHost));
    double big = 0.0;
    for (const double2& v : b) big = std::max(big, v.x);
    ok = ok && big > 0.0 && std::memcmp(b.data(), a.data() + g * len, sizeof(double2) * len) == 0;
  }
  std::printf("%d x %d, %d groups of %d columns: %s\n", n, m, groups, q, ok ? "equal" : "different");
  for (void* f : {(void*)dX[0], (void*)dX[1], (void*)dX[2], (void*)L.sw, (void*)dph, (void*)de, (void*)all, (void*)one}) cudaFree(f);
  return ok;
}

int main() {
  bool ok = true;
  ok = run(34, 18, 3, 2) && ok;
  ok = run(64, 40, 10, 3) && ok;
  ok = run(32, 48, 24, 5) && ok;
  std::puts(ok ? "ok" : "not ok");
  return ok ? 0 : 1;
}
