// Checks fold_and_centroid (k_update_math.cuh), what the batched beacon update runs on every cell, against
// fold_sum and centroid_value on deterministic adversarial inputs:
//   grid    s a multiple of 2^-40 of every exponent below 2^22, |acc| up to 2^61;
//   halves  sums halfway between two doubles, and one unit to either side (ties to even);
//   carry   sums whose 53 bits are all ones, or nearly, before rounding (up to a power of two);
//   cancel  acc close to -s, down to a total of one unit, and of zero;
//   split   totals whose 24 + 29-bit halves round to even or carry (the centroid's two floats);
//   out     s off the grid, of 2^22 and more, subnormal, infinite or NaN, and |acc| of 2^61 and more.
// Where its conditions hold it returns true, with the bits of fold_sum(s, acc) and of centroid_value of that;
// where they do not (and for a total of zero) false.  Counts from 1 to 2^40.  Test code only.
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <vector>

#include "k_update_math.cuh"

namespace {

__global__ void check_kernel(const double* s, const long long* acc, const long long* cnt, int n, int* ok, double* got_s,
                             float* got_c, double* want_s, float* want_c) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const bkv::DF rcp = bkv::count_reciprocal(cnt[i]);
  ok[i] = bkv::fold_and_centroid(s[i], acc[i], rcp, got_s[i], got_c[i]);
  want_s[i] = bkv::fold_sum(s[i], acc[i]);
  want_c[i] = bkv::centroid_value(want_s[i], rcp);
}

uint64_t state = 0x2545f4914f6cdd1dull;
uint64_t next() {  // xorshift64*
  state ^= state >> 12;
  state ^= state << 25;
  state ^= state >> 27;
  return state * 2685821657736338717ull;
}
bool coin() { return next() & 1; }
double from_bits(uint64_t b) {
  double d;
  std::memcpy(&d, &b, sizeof d);
  return d;
}

// a multiple of 2^-40 with its leading bit at 2^k (k in [-40, 21]) and at most 53 bits, random sign
double grid_value(int k) {
  const int bits = k + 41 < 53 ? k + 41 : 53;
  const uint64_t m = (next() >> (64 - bits)) | (1ull << (bits - 1));
  const double v = std::ldexp(static_cast<double>(m), k - (bits - 1));
  return coin() ? -v : v;
}
long long units(double s) { return static_cast<long long>(std::ldexp(s, 40)); }
long long random_acc(int bits) {  // below 2^bits in magnitude
  const long long a = bits ? static_cast<long long>(next() >> (64 - bits)) : 0;
  return coin() ? -a : a;
}

}  // namespace

int main() {
  std::vector<double> s;
  std::vector<long long> acc, cnt;
  std::vector<int> cls;
  auto add = [&](int c, double sv, long long av) {
    s.push_back(sv);
    acc.push_back(av);
    cnt.push_back(1 + static_cast<long long>(next() >> (64 - 1 - static_cast<int>(next() % 40))));
    cls.push_back(c);
  };
  for (int i = 0; i < 200000; ++i)
    add(0, i % 50 == 0 ? (coin() ? 0.0 : -0.0) : grid_value(-40 + static_cast<int>(next() % 62)),
        random_acc(static_cast<int>(next() % 62)));
  auto total = [&](int c, long long t) {  // s and acc with s * 2^40 + acc = t
    double part = 0.0;
    do part = grid_value(-40 + static_cast<int>(next() % 60));
    while (std::llabs(t - units(part)) >= (1ll << 61));
    add(c, part, t - units(part));
  };
  for (int i = 0; i < 60000; ++i) {  // halfway cases: 54 to 60 significant bits, the dropped ones 100..0 +- 1
    const int extra = 1 + static_cast<int>(next() % 7);
    const long long top = static_cast<long long>((next() >> 12) | (1ull << 52));
    long long t = (top << extra) + (1ll << (extra - 1)) + static_cast<long long>(next() % 3) - 1;
    total(1, coin() ? -t : t);
  }
  for (int i = 0; i < 20000; ++i) {  // all ones before rounding
    const int bits = 54 + static_cast<int>(next() % 7);
    long long t = (1ll << bits) - 1 - static_cast<long long>(next() % 4);
    total(2, coin() ? -t : t);
  }
  for (int i = 0; i < 60000; ++i) {
    const double v = grid_value(-40 + static_cast<int>(next() % 61));
    add(3, v, -units(v) + (i % 4 ? random_acc(1 + static_cast<int>(next() % 12)) : 0));
  }
  for (int i = 0; i < 60000; ++i) {  // 53 bits: 24, then 1000.. +- 1 or 0111.., or all ones above
    const long long hi = i % 3 ? static_cast<long long>((next() >> 41) | (1ull << 23)) & 0xffffff : 0xffffffll;
    const long long lo = (1ll << 28) + static_cast<long long>(next() % 3) - 1;
    long long t = ((hi | (1ll << 23)) << 29) + lo;
    t >>= next() % 40;
    if (t == 0) t = 1;
    total(4, coin() ? -t : t);
  }
  for (int i = 0; i < 40000; ++i) {
    const long long a = random_acc(52);
    switch (i % 6) {
      case 0: add(5, std::ldexp(static_cast<double>((next() >> 11) | 1ull), -60), a); break;  // off the grid
      case 1: add(5, std::ldexp(grid_value(21), 1 + static_cast<int>(next() % 30)), a); break;
      case 2: add(5, from_bits((next() >> 12) | 1ull), a); break;                               // subnormal
      case 3: add(5, from_bits((0x7ffull << 52) | (coin() ? 0 : next() >> 12)), a); break;      // inf, NaN
      case 4: add(5, from_bits((next() & ~(0x7ffull << 52)) | ((900 + next() % 300) << 52)), a); break;
      default: add(5, grid_value(0), (coin() ? 1 : -1) * (1ll << (61 + next() % 2))); break;
    }
  }
  const int n = static_cast<int>(s.size());
  double *ds, *dgs, *dws;
  long long *da, *dn;
  float *dgc, *dwc;
  int* dok;
  cudaMalloc(&ds, sizeof(double) * n);
  cudaMalloc(&dgs, sizeof(double) * n);
  cudaMalloc(&dws, sizeof(double) * n);
  cudaMalloc(&da, sizeof(long long) * n);
  cudaMalloc(&dn, sizeof(long long) * n);
  cudaMalloc(&dgc, sizeof(float) * n);
  cudaMalloc(&dwc, sizeof(float) * n);
  cudaMalloc(&dok, sizeof(int) * n);
  cudaMemcpy(ds, s.data(), sizeof(double) * n, cudaMemcpyHostToDevice);
  cudaMemcpy(da, acc.data(), sizeof(long long) * n, cudaMemcpyHostToDevice);
  cudaMemcpy(dn, cnt.data(), sizeof(long long) * n, cudaMemcpyHostToDevice);
  check_kernel<<<(n + 255) / 256, 256>>>(ds, da, dn, n, dok, dgs, dgc, dws, dwc);
  std::vector<double> gs(n), ws(n);
  std::vector<float> gc(n), wc(n);
  std::vector<int> ok(n);
  cudaMemcpy(gs.data(), dgs, sizeof(double) * n, cudaMemcpyDeviceToHost);
  cudaMemcpy(ws.data(), dws, sizeof(double) * n, cudaMemcpyDeviceToHost);
  cudaMemcpy(gc.data(), dgc, sizeof(float) * n, cudaMemcpyDeviceToHost);
  cudaMemcpy(wc.data(), dwc, sizeof(float) * n, cudaMemcpyDeviceToHost);
  if (cudaMemcpy(ok.data(), dok, sizeof(int) * n, cudaMemcpyDeviceToHost) != cudaSuccess) return 2;
  const char* names[6] = {"grid", "halves", "carry", "cancel", "split", "out"};
  long long count[6] = {}, taken[6] = {}, bad[6] = {};
  for (int i = 0; i < n; ++i) {
    const double u = std::ldexp(s[i], 40);
    bool holds = std::isfinite(s[i]) && std::fabs(s[i]) < 4194304.0 && u == std::floor(u) && acc[i] > -(1ll << 61) &&
                 acc[i] < (1ll << 61);
    holds = holds && static_cast<long long>(u) + acc[i] != 0;
    const bool same = std::memcmp(&gs[i], &ws[i], 8) == 0 && std::memcmp(&gc[i], &wc[i], 4) == 0;
    ++count[cls[i]];
    taken[cls[i]] += ok[i] != 0;
    if ((ok[i] != 0) == holds && (!holds || same)) continue;
    if (bad[cls[i]]++ < 3)
      std::printf("  %s: s %a acc %lld n %lld: returned %d (%d), sum %a (%a), centroid %a (%a)\n", names[cls[i]], s[i], acc[i],
                  cnt[i], ok[i], holds, gs[i], ws[i], gc[i], wc[i]);
  }
  int fail = 0;
  for (int c = 0; c < 6; ++c) {
    std::printf("%s: %lld cases, %lld taken, %lld wrong\n", names[c], count[c], taken[c], bad[c]);
    fail |= bad[c] != 0;
  }
  return fail;
}
