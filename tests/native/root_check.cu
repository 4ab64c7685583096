// Device check of the FP64 square root of the sound speeds and wave curves (sqrt_nr) and of
// the two-step forms of a mixed grid's interface (rcp_kept, div_kept, rsqrt_kept) against the
// IEEE operations: random operands over the seeds' range and beyond it, perfect squares, the
// range's edges, zeros, subnormals, infinity and NaN. Prints the worst errors in ulps, the
// number of quotients that differ and of special operands whose root differs.
#include <cmath>
#include <cstdio>
#include <cstring>
#include <random>
#include <vector>

#include "m2c_physics.cuh"

__global__ void k_roots(const double* x, const double* a, double* o, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  o[i] = m2c::sqrt_nr(x[i]);
  o[n + i] = sqrt(x[i]);
  o[2 * n + i] = m2c::rcp_kept(x[i]);
  o[3 * n + i] = 1.0 / x[i];
  o[4 * n + i] = m2c::rsqrt_kept(x[i]);
  o[5 * n + i] = 1.0 / sqrt(x[i]);
  o[6 * n + i] = m2c::div_kept(a[i], x[i]);
  o[7 * n + i] = a[i] / x[i];
}

static bool same(double a, double b) { return std::memcmp(&a, &b, 8) == 0 || (std::isnan(a) && std::isnan(b)); }
static double ulps(double v, double r) {
  if (same(v, r)) return 0.0;
  return std::fabs(v - r) / (std::nextafter(std::fabs(r), INFINITY) - std::fabs(r));
}

int main() {
  const int n = 1 << 20;
  std::mt19937_64 g(7);
  std::vector<double> x(n), a(n), o(8 * (size_t)n);
  for (int i = 0; i < n; ++i) {
    x[i] = std::ldexp(1.0 + (double)(g() >> 11) * 0x1p-53, (int)(g() % 280) - 140);
    a[i] = std::ldexp(1.0 + (double)(g() >> 11) * 0x1p-53, (int)(g() % 200) - 100) * ((g() & 1) ? -1.0 : 1.0);
    if (i % 4 == 1) x[i] = (double)(g() % 3000000) * (double)(x[i] > 1.0 ? 1 : 4) + 1.0;
    if (i % 4 == 2) { const double r = (double)(1 + g() % 90000000); x[i] = r * r; }
    if (i % 8 == 3) x[i] = std::nextafter(std::ldexp(1.0, (int)(g() % 60) - 30), (g() & 1) ? 0.0 : 1e300);
  }
  const double sp[] = {0.0, -0.0, 4.9e-324, 1e-310, 2.2250738585072014e-308, 1e-300, std::nextafter(0x1p-125, 0.0), 0x1p-125,
                       std::nextafter(0x1p-125, 1.0), std::nextafter(0x1p125, 0.0), 0x1p125, 1e300, 1.7976931348623157e308,
                       INFINITY, NAN, 1.0, std::nextafter(1.0, 0.0), std::nextafter(1.0, 2.0), 4.0, 0.25};
  const int ns = sizeof(sp) / sizeof(sp[0]);
  for (int i = 0; i < ns; ++i) x[i] = sp[i];
  double *dx, *da, *dout;
  if (cudaMalloc(&dx, 8 * n) || cudaMalloc(&da, 8 * n) || cudaMalloc(&dout, 64 * (size_t)n)) return 1;
  cudaMemcpy(dx, x.data(), 8 * n, cudaMemcpyHostToDevice);
  cudaMemcpy(da, a.data(), 8 * n, cudaMemcpyHostToDevice);
  k_roots<<<(n + 255) / 256, 256>>>(dx, da, dout, n);
  if (cudaDeviceSynchronize() != cudaSuccess) return 1;
  cudaMemcpy(o.data(), dout, 64 * (size_t)n, cudaMemcpyDeviceToHost);
  double worst[3] = {0, 0, 0};
  int special = 0, quotients = 0;
  for (int i = 0; i < n; ++i) {
    for (int k = 0; k < 3; ++k) {
      const double u = ulps(o[2 * k * (size_t)n + i], o[(2 * k + 1) * (size_t)n + i]);
      if (!(u <= worst[k])) worst[k] = u;
    }
    const bool seeded = x[i] >= 0x1p-125 && x[i] < 0x1p125;
    if (!seeded) special += !same(o[i], o[n + i]);
    quotients += !same(o[6 * (size_t)n + i], o[7 * (size_t)n + i]);
  }
  std::printf("sqrt worst ulp %g\nrcp worst ulp %g\nrsqrt worst ulp %g\nspecial roots differing %d\nquotients differing %d\n",
              worst[0], worst[1], worst[2], special, quotients);
  return 0;
}
