// Checks the squared norms that bound the batched update's screening error
// (add_squares and packed_total in k_update_math.cuh) against fp64: rows of 64 and 128 bf16 values in the
// kernel's order (four packed sums, words in turn), of one scale, of mixed scales, and one large element
// before many whose squares lie just below a bf16 rounding of it.  A sum may be off by its additions'
// roundings, (d / 8 + 3) 2^-24 relative, and never below its largest square.  Test code only.
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <vector>

#include "k_update_math.cuh"

namespace {

__global__ void norm_kernel(const uint32_t* w, int words, int n, float* out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  unsigned long long acc[4] = {0ull, 0ull, 0ull, 0ull};
  for (int k = 0; k < words; ++k) acc[k & 3] = bkv::add_squares(acc[k & 3], w[static_cast<size_t>(i) * words + k]);
  out[i] = (bkv::packed_total(acc[0]) + bkv::packed_total(acc[1])) +
           (bkv::packed_total(acc[2]) + bkv::packed_total(acc[3]));
}

uint64_t state = 0x9e3779b97f4a7c15ull;
uint64_t next() {  // xorshift64*
  state ^= state >> 12;
  state ^= state << 25;
  state ^= state >> 27;
  return state * 2685821657736338717ull;
}

uint16_t bf16(double m, int e) {  // sign random, 8 significant bits
  const float v = std::ldexp(static_cast<float>(m), e);
  uint32_t b;
  std::memcpy(&b, &v, 4);
  return static_cast<uint16_t>((b >> 16) | ((next() & 1) << 15));
}

double value(uint16_t h) {
  const uint32_t b = static_cast<uint32_t>(h) << 16;
  float v;
  std::memcpy(&v, &b, 4);
  return v;
}

}  // namespace

int main() {
  int fail = 0;
  const int n = 30000;
  for (int d : {64, 128}) {
    std::vector<uint16_t> x(static_cast<size_t>(n) * d);
    for (int i = 0; i < n; ++i)
      for (int k = 0; k < d; ++k) {
        const double m = (128 + static_cast<int>(next() % 128)) / 128.0;
        int e = -3 + static_cast<int>(next() % 4);                          // one scale
        if (i % 3 == 1) e = -30 + static_cast<int>(next() % 44);            // mixed scales
        if (i % 3 == 2) e = k < 8 ? 4 : -1;                                 // 8 large elements, then 2^-10 of their squares
        x[static_cast<size_t>(i) * d + k] = (i % 7 == 0 && k % 5 == 0) ? 0 : bf16(m, e);
      }
    uint32_t* dx;
    float* dout;
    cudaMalloc(&dx, x.size() * 2);
    cudaMalloc(&dout, sizeof(float) * n);
    cudaMemcpy(dx, x.data(), x.size() * 2, cudaMemcpyHostToDevice);
    norm_kernel<<<(n + 255) / 256, 256>>>(dx, d / 2, n, dout);
    std::vector<float> got(n);
    if (cudaMemcpy(got.data(), dout, sizeof(float) * n, cudaMemcpyDeviceToHost) != cudaSuccess) return 2;
    double worst = 0.0;
    int below = 0;
    for (int i = 0; i < n; ++i) {
      double want = 0.0, largest = 0.0;
      for (int k = 0; k < d; ++k) {
        const double v = value(x[static_cast<size_t>(i) * d + k]);
        want += v * v;
        largest = std::fmax(largest, v * v);
      }
      worst = std::fmax(worst, std::fabs(got[i] - want) / want);
      below += got[i] < largest;
    }
    const double bound = (d / 8 + 3) * std::ldexp(1.0, -24);
    std::printf("d %d: largest relative error %.3g (bound %.3g), %d below their largest square\n", d, worst, bound, below);
    fail |= worst > bound || below != 0;
    cudaFree(dx);
    cudaFree(dout);
  }
  return fail;
}
