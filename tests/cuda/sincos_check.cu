// Checks sincos_accurate (sincos.cuh) on rotary angles against the host's long double functions (113 bits on
// AArch64, 64 on x86-64): positions up to 2^20 and beyond, the frequencies of the bases in use, head dimensions
// 64 and 128, and angles next to multiples of pi / 2.  Within 0.505 ulp everywhere, and an fp32 rounding never
// differs from that of the exact value.  Test code only.
#include <cmath>
#include <cstdio>
#include <vector>

#include "sincos.cuh"

namespace {
__global__ void kernel(const double* a, double* s, double* c, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) bkv::sincos_accurate(a[i], s[i], c[i]);
}
}  // namespace

int main() {
  std::vector<double> a{0.0, -0.0, 1e-300, 1e-8, 0x1.921fb54442d18p-1, 0x1p-32, 0x1.fffffffffffffp-33};
  for (double theta : {1e4, 5e5, 1e6})
    for (int d : {64, 128})
      for (long long p = 0; p < 70000; p += 11)
        for (int i = 0; i < d / 2; ++i) a.push_back(static_cast<double>(p) * std::pow(theta, -2.0 * i / d));
  for (long long p = 1; p < (1ll << 59); p += p / 4 + 1)
    for (int i = 0; i < 64; ++i) a.push_back((i % 3 ? 1.0 : -1.0) * static_cast<double>(p) * std::pow(1e6, -2.0 * i / 128));
  for (int k = 1; k < 200000; k += 7) {
    const double m = k * 0x1.921fb54442d18p+0;
    a.push_back(m);
    a.push_back(std::nextafter(m, 0.0));
    a.push_back(-std::nextafter(m, 1e300));
  }
  const int n = static_cast<int>(a.size());
  double *da, *ds, *dc;
  cudaMalloc(&da, sizeof(double) * n);
  cudaMalloc(&ds, sizeof(double) * n);
  cudaMalloc(&dc, sizeof(double) * n);
  cudaMemcpy(da, a.data(), sizeof(double) * n, cudaMemcpyHostToDevice);
  kernel<<<(n + 127) / 128, 128>>>(da, ds, dc, n);
  std::vector<double> s(n), c(n);
  cudaMemcpy(s.data(), ds, sizeof(double) * n, cudaMemcpyDeviceToHost);
  if (cudaMemcpy(c.data(), dc, sizeof(double) * n, cudaMemcpyDeviceToHost) != cudaSuccess) return 2;
  double worst = 0.0, host = 0.0;
  long long off32 = 0, wrong = 0;
  for (int i = 0; i < n; ++i)
    for (int q = 0; q < 2; ++q) {
      const long double want = q ? cosl(static_cast<long double>(a[i])) : sinl(static_cast<long double>(a[i]));
      const double got = q ? c[i] : s[i], lib = q ? std::cos(a[i]) : std::sin(a[i]);
      if (want == 0.0L) {
        wrong += got != 0.0;
        continue;
      }
      const double ulp = std::ldexp(1.0, std::ilogb(static_cast<double>(want)) - 52);
      worst = std::fmax(worst, static_cast<double>(fabsl(got - want) / ulp));
      host = std::fmax(host, static_cast<double>(fabsl(lib - want) / ulp));
      off32 += static_cast<float>(got) != static_cast<float>(want);
    }
  std::printf("%d angles: at most %.4f ulp off (the host library %.4f), %lld fp32 roundings differ\n", n, worst, host, off32);
  return worst > 0.505 || off32 != 0 || wrong != 0;
}
