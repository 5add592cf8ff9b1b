// GPU check of the strip kernels (csrc/strips.cuh) against long double on the host, entry by entry:
// prints "ok" or the cases beyond the bounds that follow from double-float steps (2^-44 of the sums of
// magnitudes that enter), exact curls (2^-58 of the largest value) and the FP32 storage of the result.
#include "strips.cuh"

#include <algorithm>
#include <cmath>
#include <complex>
#include <cstdio>
#include <random>
#include <vector>

using namespace pbs;
using Z = std::complex<long double>;

static std::mt19937_64 rng(11);
static double uniform(double a, double b) { return std::uniform_real_distribution<double>(a, b)(rng); }
template <class T> T* upload(const std::vector<T>& v) {
  T* d = nullptr;
  cudaMalloc(&d, sizeof(T) * v.size());
  cudaMemcpy(d, v.data(), sizeof(T) * v.size(), cudaMemcpyHostToDevice);
  return d;
}
template <class T> std::vector<T> download(const T* d, size_t n) {
  std::vector<T> v(n);
  cudaMemcpy(v.data(), d, sizeof(T) * n, cudaMemcpyDeviceToHost);
  return v;
}

struct Field {  // one column with its Bloch extension
  const double2* X;
  int n, m;
  Z al, be;
  Z at(int comp, int i, int j) const {
    Z ph = 1;
    if (i < 0) ph *= std::conj(al);
    if (i >= n) ph *= al;
    if (j < 0) ph *= std::conj(be);
    if (j >= m) ph *= be;
    const double2 v = X[(long)comp * n * m + (long)((j + m) % m) * n + (i + n) % n];
    return ph * Z(v.x, v.y);
  }
  Z x(int i, int j) const { return at(0, i, j); }
  Z y(int i, int j) const { return at(1, i, j); }
  Z curl(int i, int j) const { return x(i, j + 1) - x(i, j) - y(i + 1, j) + y(i, j); }
  long double curl_mag(int i, int j) const {
    return std::abs(x(i, j + 1)) + std::abs(x(i, j)) + std::abs(y(i + 1, j)) + std::abs(y(i, j));
  }
  Z mx(int i, int j) const { return 4.0L * x(i, j) + x(i, j + 1) + x(i, j - 1); }
  Z my(int i, int j) const { return 4.0L * y(i, j) + y(i + 1, j) + y(i - 1, j); }
  long double mx_mag(int i, int j) const { return 4 * std::abs(x(i, j)) + std::abs(x(i, j + 1)) + std::abs(x(i, j - 1)); }
  long double my_mag(int i, int j) const { return 4 * std::abs(y(i, j)) + std::abs(y(i + 1, j)) + std::abs(y(i - 1, j)); }
};

static bool run(int n, int m, int rows, bool smooth) {
  const int cols = 3, cpg = 2;
  const long N = (long)n * m, D = 2 * N, ld = D + 3;
  const double hx = 1.0 / n, hy = 1.3 / m;
  Lvl<df> L{n, m, df(hy / hx), df(hx / hy)};
  const long double Lx = (long double)(hy / hx), Ly = (long double)(hx / hy);
  std::vector<float2> w(N);
  std::vector<long double> wl(N);
  for (long t = 0; t < N; ++t) {
    const double v = 1.0 / uniform(1.0, 12.0) / (hx * hy);
    const float h = (float)v, l = (float)(v - (double)h);
    w[t] = make_float2(h, l);
    wl[t] = (long double)h + l;
  }
  std::vector<double> ph;  // groups of cpg columns
  for (int g = 0; g < 2; ++g) {
    const double a = 0.3 + g, b = -1.1 + 2 * g;
    for (double v : {std::cos(a), std::sin(a), std::cos(b), std::sin(b)}) ph.push_back(v);
  }
  std::vector<double2> X(cols * ld);
  for (int c = 0; c < cols; ++c)
    for (long t = 0; t < D; ++t) {
      const int i = t % n, j = t / n % m;
      const double a = (0.3 + c / cpg) * i / n + (-1.1 + 2 * (c / cpg)) * j / m;
      // a smooth Bloch field whose rows span decades, or noise
      X[c * ld + t] = smooth ? make_double2(std::cos(a) * (1 + 1e-6 * uniform(-1, 1)) * std::pow(10.0, -2 * c * (j % 3)),
                                            std::sin(a) * std::pow(10.0, -2 * c * (j % 3)))
                             : make_double2(uniform(-1, 1), uniform(-1, 1) * 1e-3);
    }
  std::vector<double> lam = {3.7, 41.0, 1234.5};
  double2* dX = upload(X);
  float2* dw = upload(w);
  double *dph = upload(ph), *dlam = upload(lam);
  const unsigned n31 = strip_blocks<31>(n, m, rows), n30 = strip_blocks<30>(n, m, rows);
  double* part = upload(std::vector<double>(2 * cols * std::max(n30, n31), -1.0));
  float2* dR = upload(std::vector<float2>(cols * ld, make_float2(7, 7)));
  float2* dY = upload(std::vector<float2>(cols * (N + 1), make_float2(7, 7)));
  double2* dY2 = upload(std::vector<double2>(cols * (N + 1), make_double2(7, 7)));
  const WtsDF W{dw, n, m};
  k_rayleigh_strips<<<dim3(n31, cols), 32 * kStripWarps>>>(L, W, dph, cpg, dX, ld, rows, part);
  const std::vector<double> rq = download(part, 2 * cols * n31);
  k_residual_strips<<<dim3(n30, cols), 32 * kStripWarps>>>(L, W, dph, cpg, dX, dR, ld, dlam, rows, part);
  const std::vector<double> norms = download(part, 2 * cols * n30);
  k_lift_adj_mass_strips<float><<<dim3(n30, cols), 32 * kStripWarps>>>(L, dph, cpg, dX, ld, dY, N + 1, rows);
  k_lift_adj_mass_strips<double><<<dim3(n30, cols), 32 * kStripWarps>>>(L, dph, cpg, dX, ld, dY2, N + 1, rows);
  const cudaError_t err = cudaDeviceSynchronize();
  const std::vector<float2> R = download(dR, cols * ld), Y = download(dY, cols * (N + 1));
  const std::vector<double2> Y2 = download(dY2, cols * (N + 1));
  bool ok = err == cudaSuccess;
  long double worst[6] = {};
  auto check = [&](int k, long double e, long double bound) {
    ok = ok && e <= bound;
    worst[k] = std::max(worst[k], e / (bound + 1e-4000L));
  };
  const long double u = 0x1p-44L, f = 0x1p-23L;
  for (int c = 0; c < cols; ++c) {
    const double* p = ph.data() + 4 * (c / cpg);
    const Field F{X.data() + c * ld, n, m, Z(p[0], p[1]), Z(p[2], p[3])};
    long double den = 0, num = 0, dnum = 0, rr = 0, mm = 0, big = 0, rt = 0;
    for (long t = 0; t < D; ++t) big = std::max(big, std::max<long double>(std::fabs(X[c * ld + t].x), std::fabs(X[c * ld + t].y)));
    auto H = [&](int i, int j) { return wl[(long)((j + m) % m) * n + (i + n) % n] * F.curl(i, j); };
    auto Hm = [&](int i, int j) {  // what rounding enters H: its own size, and the exact curl's grid
      return wl[(long)((j + m) % m) * n + (i + n) % n] * (u * std::abs(F.curl(i, j)) + 0x1p-57L * big + 0x1p-51L * F.curl_mag(i, j) * (i < 0 || j < 0 || i + 1 >= n || j + 1 >= m));
    };
    for (int j = 0; j < m; ++j)
      for (int i = 0; i < n; ++i) {
        const long at = (long)j * n + i;
        const Z x = F.x(i, j), y = F.y(i, j), mx = Lx / 6 * F.mx(i, j), my = Ly / 6 * F.my(i, j);
        den += std::real(std::conj(x) * mx + std::conj(y) * my);
        num += wl[at] * std::norm(F.curl(i, j));
        dnum += wl[at] * (2 * std::abs(F.curl(i, j)) * 2 * u * F.curl_mag(i, j) + 4 * u * u * F.curl_mag(i, j) * F.curl_mag(i, j));
        const Z rx = H(i, j - 1) - H(i, j) - (long double)lam[c] * mx, ry = H(i, j) - H(i - 1, j) - (long double)lam[c] * my;
        rr += std::norm(rx) + std::norm(ry);
        mm += std::norm(mx) + std::norm(my);
        const long double ex = Hm(i, j - 1) + Hm(i, j) + u * (std::abs(H(i, j)) + std::abs(H(i, j - 1)) + lam[c] * Lx * F.mx_mag(i, j)),
                          ey = Hm(i, j) + Hm(i - 1, j) + u * (std::abs(H(i, j)) + std::abs(H(i - 1, j)) + lam[c] * Ly * F.my_mag(i, j));
        const float2 gx = R[c * ld + at], gy = R[c * ld + N + at];
        check(0, std::abs(Z(gx.x, gx.y) - rx), ex + f * std::abs(rx));
        check(0, std::abs(Z(gy.x, gy.y) - ry), ey + f * std::abs(ry));
        rt += 2 * std::abs(rx) * (ex + f * std::abs(rx)) + 2 * std::abs(ry) * (ey + f * std::abs(ry));
        const Z v = Lx / 6 * (F.mx(i - 1, j) - F.mx(i, j)) + Ly / 6 * (F.my(i, j - 1) - F.my(i, j));
        const long double vm = u * (Lx * (F.mx_mag(i - 1, j) + F.mx_mag(i, j)) + Ly * (F.my_mag(i, j - 1) + F.my_mag(i, j)));
        check(1, std::abs(Z(Y[c * (N + 1) + at].x, Y[c * (N + 1) + at].y) - v), vm + f * std::abs(v));
        check(2, std::abs(Z(Y2[c * (N + 1) + at].x, Y2[c * (N + 1) + at].y) - v), vm);
      }
    ok = ok && R[c * ld + D].x == 7 && Y[c * (N + 1) + N].x == 7 && Y2[c * (N + 1) + N].x == 7;
    long double gd = 0, gn = 0, gr = 0, gm = 0;
    for (unsigned b = 0; b < n31; ++b) gd += rq[2 * (c * n31 + b)], gn += rq[2 * (c * n31 + b) + 1];
    for (unsigned b = 0; b < n30; ++b) gr += norms[2 * (c * n30 + b)], gm += norms[2 * (c * n30 + b) + 1];
    check(3, std::fabs(gd - den), 3 * u * den);  // |x (2 x + x+)| sums to at most three times e^* M e
    check(4, std::fabs(gn - num), dnum + u * num);
    check(5, std::fabs(gr - rr), rt + 8 * f * rr);
    check(5, std::fabs(gm - mm), 8 * f * mm);
  }
  std::printf("%s %d x %d rows %d %s: of the bounds: residual %.3Lf, rhs %.3Lf / %.3Lf (FP64), e^*Me %.3Lf, curl form %.3Lf, norms %.3Lf %s\n",
              ok ? "fine" : "BEYOND", n, m, rows, smooth ? "smooth" : "noise", worst[0], worst[1], worst[2], worst[3], worst[4],
              worst[5], cudaGetErrorString(err));
  for (void* q : {(void*)dX, (void*)dw, (void*)dph, (void*)dlam, (void*)part, (void*)dR, (void*)dY, (void*)dY2}) cudaFree(q);
  return ok;
}

int main() {
  bool ok = true;
  const int sizes[][2] = {{4, 4}, {2, 6}, {30, 8}, {31, 9}, {32, 16}, {60, 33}, {62, 7}, {64, 48}, {91, 20}, {128, 70}};
  for (auto& s : sizes)
    for (int rows : {8, 16, 32})
      for (bool smooth : {false, true}) ok = run(s[0], s[1], rows, smooth) && ok;
  std::puts(ok ? "ok" : "not ok");
  return ok ? 0 : 1;
}
