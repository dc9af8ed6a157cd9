// Observation queries of every GQA group (Section 4.3; Appendix D.2):
// recent queries rotated to their own positions, beacons rotated to the
// current step, each rounded to bf16 for the tensor-core scoring.
//
// Layout written: qobs bf16 [n_inst][n_obs_pad][d]; rows h*W + w are recent
// slot w of query head h, rows G*W + b are beacon b, rows >= n_obs are zero.
// valid [n_inst][4] is a 128-bit mask of rows that take part in the maximum
// (all recent rows, beacons with count > 0).
//
// Definition of each output element: y_i = x_i c - x_{i+d/2} s and
// y_{i+d/2} = x_{i+d/2} c + x_i s evaluated in fp64 (separately rounded
// products, fp64 cos / sin), then rounded fp64 -> fp32 -> bf16.
// The kernel first evaluates y in fp32 (one FMA, fp32 copies of cos / sin).
// The fp32 value v differs from the fp64 one by at most
//   delta = 2^-22 (|x_a| + |x_b| + |v|)
// (rounding of cos and sin to fp32, of the product and of the FMA, with a
// factor 2 of margin).  The composite rounding can only change where the fp32
// value crosses a bf16 rounding midpoint (low 16 bits 0x8000) or lands within
// one fp32 ulp of it; if v is farther than delta + 1 ulp from the nearest
// midpoint, bf16(v) is the defined value.  Otherwise (about 2e-4 of the
// elements) the element is recomputed in fp64 exactly as defined.
#include <cmath>

#include "bkv_device.cuh"
#include "bkv_internal.h"
#include "sincos.cuh"

namespace bkv {
namespace {

constexpr int kQobsThreads = 256;

// Exact definition: fp64 products, fp64 sum, then fp32, then bf16.
__device__ __forceinline__ __nv_bfloat16 rot_exact(double xa, double xb, double c, double s, bool plus) {
  const double y = plus ? __dadd_rn(__dmul_rn(xa, c), __dmul_rn(xb, s)) : __dsub_rn(__dmul_rn(xa, c), __dmul_rn(xb, s));
  return __float2bfloat16_rn(__double2float_rn(y));
}

// bf16 of (xa*c +- xb*s) through the fp32 fast path when provably equal to the definition; the
// fp64 (cos, sin) pair `cs` is read only on the exact path.
__device__ __forceinline__ __nv_bfloat16 rot_fast(float xa, float xb, float c32, float s32, const double2* cs,
                                                   bool plus) {
  const float p = xb * s32;
  const float v = fmaf(xa, c32, plus ? p : -p);
  const uint32_t t = __float_as_uint(v);
  const uint32_t ex = t & 0x7f800000u;
  if (ex >= (25u << 23) && ex != 0x7f800000u) {
    const float ulp = __uint_as_float(ex - (23u << 23));
    const float delta = 0x1p-22f * (fabsf(xa) + fabsf(xb) + fabsf(v));
    const int dist = abs(static_cast<int>(t & 0xffffu) - 0x8000);
    if (static_cast<float>(dist - 1) * ulp > delta) return __float2bfloat16_rn(v);
  }
  const double2 c = *cs;
  return rot_exact(xa, xb, c.x, c.y, plus);
}

// work / n_work (per-instance lengths): block w builds instance work[w] when w < *n_work; rope_row: the
// distance between two batch rows' rotary tables (0: one table for every instance).
__global__ void __launch_bounds__(kQobsThreads) qobs_kernel(Shape s, const __nv_bfloat16* q_recent, const float* cent,
                                                             const long long* counts, const double2* rope_all,
                                                             size_t rope_row, int rotate, const int* work,
                                                             const int* n_work, __nv_bfloat16* qobs, uint32_t* valid,
                                                             int* err) {
  int e = blockIdx.x;
  grid_dependency_wait();
  if (work) {
    if (e >= *n_work) return;  // whole block
    e = work[e];
    if (!in_bounds(e, s.n_inst, err)) return;  // whole block: every thread read the same entry
  }
  const int d = s.d, h = d / 2, h4 = h / 4;
  const int GW = s.G * s.W;
  const double2* rope = rope_all + (rope_row ? static_cast<size_t>((e / s.n_kv) % s.batch) * rope_row : 0);
  const float2* rope32 = reinterpret_cast<const float2*>(rope + static_cast<size_t>(s.W + 1) * h);
  __nv_bfloat16* out = qobs + static_cast<size_t>(e) * s.n_obs_pad * d;
  for (int idx = threadIdx.x; idx < s.n_obs_pad * h4; idx += blockDim.x) {
    const int row = idx / h4, i = (idx % h4) * 4;
    float xa[4] = {0.f, 0.f, 0.f, 0.f}, xb[4] = {0.f, 0.f, 0.f, 0.f};
    int slot = 0;
    if (row < GW) {
      const __nv_bfloat16* src = q_recent + (static_cast<size_t>(e) * GW + row) * d;
      const uint2 a = *reinterpret_cast<const uint2*>(src + i);
      const uint2 b = *reinterpret_cast<const uint2*>(src + i + h);
      const float2 a0 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&a.x));
      const float2 a1 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&a.y));
      const float2 b0 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&b.x));
      const float2 b1 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&b.y));
      xa[0] = a0.x; xa[1] = a0.y; xa[2] = a1.x; xa[3] = a1.y;
      xb[0] = b0.x; xb[1] = b0.y; xb[2] = b1.x; xb[3] = b1.y;
      slot = row % s.W;
    } else if (row < s.n_obs) {
      const float* src = cent + (static_cast<size_t>(e) * s.nb + (row - GW)) * d;
      const float4 a = *reinterpret_cast<const float4*>(src + i);
      const float4 b = *reinterpret_cast<const float4*>(src + i + h);
      xa[0] = a.x; xa[1] = a.y; xa[2] = a.z; xa[3] = a.w;
      xb[0] = b.x; xb[1] = b.y; xb[2] = b.z; xb[3] = b.w;
      slot = s.W;
    }
    __nv_bfloat16 y1[4], y2[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      if (row < s.n_obs && rotate) {
        const float2 cs32 = rope32[slot * h + i + k];
        const double2* cs64 = rope + slot * h + i + k;
        y1[k] = rot_fast(xa[k], xb[k], cs32.x, cs32.y, cs64, false);
        y2[k] = rot_fast(xb[k], xa[k], cs32.x, cs32.y, cs64, true);
      } else {
        y1[k] = __float2bfloat16_rn(xa[k]);
        y2[k] = __float2bfloat16_rn(xb[k]);
      }
    }
    *reinterpret_cast<uint2*>(out + row * d + i) = *reinterpret_cast<const uint2*>(y1);
    *reinterpret_cast<uint2*>(out + row * d + i + h) = *reinterpret_cast<const uint2*>(y2);
  }
  if (threadIdx.x < 128) {  // warp w builds mask word w: one row per lane, loads in parallel
    const int row = threadIdx.x;
    bool v = row < GW;
    if (!v && row < s.n_obs) v = counts[static_cast<size_t>(e) * s.nb + (row - GW)] > 0;
    const uint32_t m = __ballot_sync(0xffffffffu, v);
    if ((threadIdx.x & 31) == 0) valid[e * 4 + (threadIdx.x >> 5)] = m;
  }
}

// One chunk of positions, by value: rows of W + 1 positions (the recent slots, then t_pos).
constexpr int kRopePositions = 1024;
template <int N>
struct RopeChunk {
  double inv_freq[64];
  long long pos[N];
};

// Rotary tables (and causal gaps) of a chunk of batch rows: block = one position and 32 frequency pairs, one
// thread each.  The angle is the fp64 product of position and frequency; its cosine and sine are within 0.501 ulp,
// in integer arithmetic (in fp64 as accurate they took 4 us more).  Formed on the host (576 pow, cos and sin for 8 recent slots and d =
// 128) the table cost a compress about 50 us of host time before its first launch, and a copy kernel reading
// pinned memory; this kernel takes 6 us.
template <int N>
__global__ void __launch_bounds__(32) rope_table_kernel(const __grid_constant__ RopeChunk<N> c, int first_row, int W,
                                                        int h, int rotate, double2* table, size_t row_stride, int* gaps,
                                                        int gap_max) {
  const int at = blockIdx.x / (h / 32), i = (blockIdx.x % (h / 32)) * 32 + threadIdx.x;
  const int row = at / (W + 1), slot = at % (W + 1);
  const long long pos = c.pos[at];
  double sn = 0.0, cs = 0.0;
  if (rotate) sincos_accurate(__dmul_rn(static_cast<double>(pos), c.inv_freq[i]), sn, cs);
  grid_dependency_wait();  // an earlier compress may still read the table
  if (rotate) {
    double2* tab = table + static_cast<size_t>(first_row + row) * row_stride;
    float2* tab32 = reinterpret_cast<float2*>(tab + static_cast<size_t>(W + 1) * h);
    tab[slot * h + i] = make_double2(cs, sn);
    tab32[slot * h + i] = make_float2(static_cast<float>(cs), static_cast<float>(sn));
  }
  if (gaps && i == 0 && slot < W) {
    const long long t = c.pos[row * (W + 1) + W];
    const long long g = pos >= t ? 0 : static_cast<long long>(static_cast<unsigned long long>(t) - static_cast<unsigned long long>(pos));
    gaps[(first_row + row) * W + slot] = static_cast<int>(g > gap_max || g < 0 ? gap_max : g);
  }
}

template <int N>
cudaError_t launch_rope_chunks(int W, int h, int rows, const double* inv_freq, const int64_t* t_pos,
                               const int64_t* recent_pos, int rotate, double2* table, size_t row_stride, int* gaps,
                               int gap_max, cudaStream_t st) {
  RopeChunk<N> c;
  for (int i = 0; i < h; ++i) c.inv_freq[i] = inv_freq[i];
  const int per = N / (W + 1);  // rows per launch (at least one: W <= 64)
  for (int r0 = 0; r0 < rows; r0 += per) {
    const int n = rows - r0 < per ? rows - r0 : per;
    for (int r = 0; r < n; ++r) {
      long long* pos = c.pos + r * (W + 1);
      for (int w = 0; w < W; ++w) pos[w] = recent_pos[static_cast<size_t>(r0 + r) * W + w];
      pos[W] = t_pos[r0 + r];
    }
    const cudaError_t e = launch_dependent(rope_table_kernel<N>, static_cast<unsigned>(n * (W + 1) * (h / 32)), 32, 0, st, c,
                                           r0, W, h, rotate, table, row_stride, gaps, gap_max);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace

void rope_frequencies(double theta, int d, double* inv_freq) {
  for (int i = 0; i < d / 2; ++i)
    inv_freq[i] = theta != 0.0 ? std::pow(theta, -static_cast<double>(2 * i) / static_cast<double>(d)) : 0.0;
}

cudaError_t launch_rope_table(int W, int h, int rows, const double* inv_freq, const int64_t* t_pos,
                              const int64_t* recent_pos, int rotate, double2* table, size_t row_stride, int* gaps,
                              int gap_max, cudaStream_t st) {
  // a single row's parameters stay small (at most 65 positions)
  return rows == 1 ? launch_rope_chunks<kMaxWindow + 1>(W, h, rows, inv_freq, t_pos, recent_pos, rotate, table,
                                                        row_stride, gaps, gap_max, st)
                   : launch_rope_chunks<kRopePositions>(W, h, rows, inv_freq, t_pos, recent_pos, rotate, table,
                                                        row_stride, gaps, gap_max, st);
}

cudaError_t launch_qobs(const Shape& s, const __nv_bfloat16* q_recent, const float* cent, const long long* counts,
                        const double2* rope, int rotate, __nv_bfloat16* qobs, uint32_t* valid, int* err,
                        cudaStream_t st) {
  return launch_dependent(qobs_kernel, static_cast<unsigned>(s.n_inst), kQobsThreads, 0, st, s, q_recent, cent, counts,
                          rope, static_cast<size_t>(0), rotate, nullptr, nullptr, qobs, valid, err);
}

cudaError_t launch_qobs_ragged(const Shape& s, const __nv_bfloat16* q_recent, const float* cent,
                               const long long* counts, const double2* rope, size_t rope_row, int rotate,
                               const int* work, const int* n_work, __nv_bfloat16* qobs, uint32_t* valid, int* err,
                               cudaStream_t st) {
  return launch_dependent(qobs_kernel, static_cast<unsigned>(s.n_inst), kQobsThreads, 0, st, s, q_recent, cent, counts,
                          rope, rope_row, rotate, work, n_work, qobs, valid, err);
}

}  // namespace bkv
