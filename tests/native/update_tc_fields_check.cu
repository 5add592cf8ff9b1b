// GPU check of the tensor-core block update (csrc/update_tc.cu) on columns whose two halves (x- and
// y-edges) differ by a power of two far from one, with the exponents' offsets that go with it:
// against long double on the host, each value within the bound of its own half.  Prints "ok".
// (The library's launch and error helpers are stood in for below.)
#include "update_tc.cu"

#include <cmath>
#include <cstdio>
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
using C2 = double2;

static std::mt19937_64 rng(3);
static double normal() { return std::normal_distribution<double>()(rng); }
template <class T> T* upload(const std::vector<T>& v) {
  T* d = nullptr;
  PBS_CUDA(cudaMalloc(&d, sizeof(T) * v.size()));
  PBS_CUDA(cudaMemcpy(d, v.data(), sizeof(T) * v.size(), cudaMemcpyHostToDevice));
  return d;
}

// the first half of the rows at 2^ox, the second at 2^oy
static bool run(int q, int p, long rows, int ox, int oy) {
  std::vector<C2> X((size_t)q * rows), C((size_t)q * p);
  std::vector<int> E(2 * q);
  for (int i = 0; i < q; ++i) {
    double big = 0.0;
    for (long r = 0; r < rows; ++r) {
      const double x = normal(), y = normal();
      big = std::max({big, std::fabs(x), std::fabs(y)});
      const int o = 2 * r < rows ? ox : oy;
      X[i * rows + r] = C2{std::ldexp(x, o), std::ldexp(y, o)};
    }
    std::frexp(big, &E[2 * i]);
    for (int j = 0; j < p; ++j) C[j * q + i] = C2{normal(), normal()};
  }
  C2 *dX = upload(X), *dC = upload(C), *dY = upload(std::vector<C2>((size_t)p * rows));
  int* dE = upload(E);
  update_tc(Roles{{dX, dX, dX}, q, rows}, q, dC, q, (long)q * p, dE, 2 * q, dY, rows, p, nullptr, 0, rows, 1, 2, 0, ox, oy);
  PBS_CUDA(cudaDeviceSynchronize());
  std::vector<C2> Y((size_t)p * rows);
  PBS_CUDA(cudaMemcpy(Y.data(), dY, sizeof(C2) * Y.size(), cudaMemcpyDeviceToHost));
  double worst = 0.0;
  for (int j = 0; j < p; ++j) {
    // operands keep 2^-62 of their bounds, the pairs left out are below 7.1 2^-62 of the largest
    // product (16 2^-62 in all per real product); what the eight sums lose when put together
    long double F = 0.0L;
    for (int i = 0; i < q; ++i)
      F = std::max(F, 2 * std::max(std::fabs((long double)C[j * q + i].x), std::fabs((long double)C[j * q + i].y)) * std::exp2((long double)E[2 * i]));
    for (long r = 0; r < rows; ++r) {
      long double sx = 0, sy = 0;
      for (int i = 0; i < q; ++i) {
        const C2 x = X[i * rows + r], c = C[j * q + i];
        sx += (long double)x.x * c.x - (long double)x.y * c.y;
        sy += (long double)x.x * c.y + (long double)x.y * c.x;
      }
      const long double tol = std::ldexp(F * (2 * q * 16 * 0x1p-62L + 0x1p-57L), 2 * r < rows ? ox : oy);
      const C2 y = Y[j * rows + r];
      const long double dx = std::fabs(y.x - sx) / (tol + 0x1.02p-53L * std::fabs(sx)),
                        dy = std::fabs(y.y - sy) / (tol + 0x1.02p-53L * std::fabs(sy));
      worst = std::max({worst, (double)dx, (double)dy});
    }
  }
  std::printf("q=%d p=%d rows=%ld offsets %d, %d: %.3f of the bound\n", q, p, rows, ox, oy, worst);
  cudaFree(dX);
  cudaFree(dC);
  cudaFree(dY);
  cudaFree(dE);
  return worst <= 1.0;
}

int main() {
  bool ok = true;
  for (int o : {-40, -7, 0, 12, 40}) {
    ok = run(10, 10, 1000, 0, o) && ok;  // the halves meet inside a tile
    ok = run(20, 10, 768, o, -o) && ok;  // and between tiles
    ok = run(48, 24, 300, -o, 3) && ok;  // in parts
  }
  std::puts(ok ? "ok" : "not ok");
  return ok ? 0 : 1;
}
