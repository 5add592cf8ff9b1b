// GPU check of the tensor-core block update (csrc/update_tc.cu) against long double on the host:
// prints "ok" or the first case beyond the bound that follows from its operand digits and dropped
// digit pairs.  (The library's launch and error helpers are stood in for below.)
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

static std::mt19937_64 rng(7);
static double normal() { return std::normal_distribution<double>()(rng); }
template <class T> T* upload(const std::vector<T>& v) {
  T* d = nullptr;
  PBS_CUDA(cudaMalloc(&d, sizeof(T) * std::max<size_t>(v.size(), 1)));
  PBS_CUDA(cudaMemcpy(d, v.data(), sizeof(T) * v.size(), cudaMemcpyHostToDevice));
  return d;
}

// roles of pr columns each (q = a multiple, at most 3 roles), G groups; returns false beyond the bound
static bool run(int pr, int q, int p, long rows, int G, bool with_z, int slices, double spread) {
  const long ld = rows + 5, ncol = (long)G * pr;
  std::vector<C2> X[3], C((size_t)G * q * p), Z((size_t)G * p * ld);
  std::vector<int> E((size_t)G * q * 2, -1000000);
  const int nr = q / pr;
  for (int r = 0; r < nr; ++r) {
    X[r].resize(ncol * ld);
    for (auto& x : X[r]) x = C2{normal(), normal()};
  }
  for (int g = 0; g < G; ++g)
    for (int i = 0; i < q; ++i) {
      C2* x = X[i / pr].data() + ((long)g * pr + i % pr) * ld;
      const double sc = i == 1 ? 0.0 : std::pow(10.0, -spread * i);  // column 1 is zero
      double big = 0.0;
      for (long r = 0; r < rows; ++r) {
        x[r].x *= sc * (r % 7 == 3 ? 1e-9 : 1.0);
        x[r].y *= sc;
        big = std::max({big, std::fabs(x[r].x), std::fabs(x[r].y)});
      }
      int e = -1000000;
      if (big > 0.0) std::frexp(big, &e);
      E[2 * ((long)g * q + i)] = e;
      for (int j = 0; j < p; ++j) {
        C2 c{normal() * std::pow(10.0, spread * i - j), normal() * std::pow(10.0, spread * i - j)};
        if (j == 2) c = C2{0.0, i == 3 ? 1.0 : 0.0};
        C[((long)g * p + j) * q + i] = c;
      }
    }
  for (auto& z : Z) z = C2{normal(), normal()};
  C2* dX[3] = {};
  for (int r = 0; r < nr; ++r) dX[r] = upload(X[r]);
  C2 *dC = upload(C), *dZ = upload(Z), *dY = upload(std::vector<C2>((size_t)G * p * ld, C2{1e300, 1e300}));
  int* dE = upload(E);
  const Roles R{{dX[0], dX[nr > 1 ? 1 : 0], dX[nr > 2 ? 2 : 0]}, pr, ld};
  update_tc(R, q, dC, q, (long)q * p, dE, 2 * q, dY, ld, p, with_z ? dZ : nullptr, ld, rows, G, slices, 0);
  PBS_CUDA(cudaDeviceSynchronize());
  std::vector<C2> Y((size_t)G * p * ld);
  PBS_CUDA(cudaMemcpy(Y.data(), dY, sizeof(C2) * Y.size(), cudaMemcpyDeviceToHost));
  // largest product of a column pair times: operand digits and dropped pairs, per real product
  const long double per = 16 * 0x1p-62L;
  double worst = 0.0, e_tc = 0.0, e_64 = 0.0;
  bool ok = true;
  for (int g = 0; g < G; ++g)
    for (int j = 0; j < p; ++j) {
      long double F = 0.0L;
      for (int i = 0; i < q; ++i) {
        const C2 c = C[((long)g * p + j) * q + i];
        const int e = E[2 * ((long)g * q + i)];
        if (e > -100000) F = std::max(F, 2 * std::max(std::fabs((long double)c.x), std::fabs((long double)c.y)) * std::exp2((long double)e));
      }
      double big = 0.0, et = 0.0, e64 = 0.0;
      for (long r = 0; r < ld; ++r) {
        const C2 y = Y[((long)g * p + j) * ld + r];
        if (r >= rows) {
          ok = ok && y.x == 1e300 && y.y == 1e300;
          continue;
        }
        long double sx = 0, sy = 0, mag = 0;
        double fx = 0, fy = 0;
        for (int i = 0; i < q; ++i) {
          const C2 x = X[i / pr][((long)g * pr + i % pr) * ld + r], c = C[((long)g * p + j) * q + i];
          sx += (long double)x.x * c.x - (long double)x.y * c.y;
          sy += (long double)x.x * c.y + (long double)x.y * c.x;
          mag += (std::fabs((long double)x.x) + std::fabs((long double)x.y)) * (std::fabs((long double)c.x) + std::fabs((long double)c.y));
          fx = std::fma(x.x, c.x, std::fma(-x.y, c.y, fx));
          fy = std::fma(x.x, c.y, std::fma(x.y, c.x, fy));
        }
        const C2 z = with_z ? Z[((long)g * p + j) * ld + r] : C2{0.0, 0.0};
        const long double tol = F * (2 * q * per + 0x1p-57L);
        const long double dx = std::fabs(y.x - (sx + z.x)), dy = std::fabs(y.y - (sy + z.y));
        const int parts = (q + 31) / 32;  // of the trial columns: each is rounded, and added in FP64
        const long double bx = parts * tol + 0x1p-53L * (std::fabs(sx) + std::fabs(sx + z.x) + (parts > 1 ? 3 * mag : 0)) * 1.01L,
                          by = parts * tol + 0x1p-53L * (std::fabs(sy) + std::fabs(sy + z.y) + (parts > 1 ? 3 * mag : 0)) * 1.01L;
        ok = ok && dx <= bx && dy <= by;
        worst = std::max({worst, (double)(dx / (bx + 1e-300L)), (double)(dy / (by + 1e-300L))});
        big = std::max({big, (double)std::fabs(sx), (double)std::fabs(sy)});
        et = std::max({et, (double)std::fabs(dx), (double)std::fabs(dy)});
        e64 = std::max({e64, (double)std::fabs(fx + z.x - (sx + z.x)), (double)std::fabs(fy + z.y - (sy + z.y))});
      }
      if (big > 0.0) {
        e_tc = std::max(e_tc, et / big);
        e_64 = std::max(e_64, e64 / big);
      }
    }
  std::printf("%s p=%d q=%d rows=%ld groups=%d z=%d: %.3f of the bound; largest error / largest value %.2e (FP64 sums %.2e)\n",
              ok ? "fine" : "BEYOND", p, q, rows, G, (int)with_z, worst, e_tc, e_64);
  for (int r = 0; r < nr; ++r) cudaFree(dX[r]);
  cudaFree(dC);
  cudaFree(dZ);
  cudaFree(dY);
  cudaFree(dE);
  return ok;
}

int main() {
  bool ok = true;
  const int ps[] = {1, 3, 4, 5, 8, 9, 10, 12, 13, 16};
  for (int p : ps) {
    ok = run(p, 2 * p, p, 1000, 2, false, 3, 0.0) && ok;
    ok = run(p, p, p, 1000, 2, true, 3, 0.0) && ok;
  }
  for (long rows : {1L, 31L, 127L, 128L, 129L, 4096L}) {  // less than a tile, one, one and a row, more CTAs than tiles
    ok = run(8, 16, 8, rows, 1, true, 100, 0.0) && ok;
    ok = run(10, 10, 10, rows, 3, false, 2, 0.0) && ok;
  }
  ok = run(24, 48, 24, 700, 2, true, 2, 0.0) && ok;           // two parts of each
  ok = run(32, 64, 32, 300, 1, false, 2, 0.0) && ok;
  ok = run(17, 17, 17, 300, 2, true, 2, 0.0) && ok;           // uneven parts
  ok = run(11, 33, 31, 300, 1, false, 2, 0.0) && ok;
  ok = run(10, 20, 10, 3000, 1, false, 1, 3.0) && ok;   // column sizes over 60 decades
  ok = run(16, 16, 16, 3000, 1, false, 1, 4.0) && ok;
  ok = run(4, 12, 7, 500, 2, false, 2, 0.5) && ok;      // three roles, fewer outputs than columns
  std::puts(ok ? "ok" : "not ok");
  return ok ? 0 : 1;
}
