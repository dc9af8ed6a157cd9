// Beacon seeding by Farthest Point Sampling (Appendix D.1, Algorithm 1) over
// the prompt queries of every GQA group (Appendix D.2, prefill branch).
//
// One CTA per instance (or query head).  Every argmin of the algorithm is
// first screened with fp32 similarities from the tensor cores and decided
// there unless other rows lie within twice the screening error of the
// minimum; those rows alone are then compared exactly.
//
//   Screening: the rows are staged in shared memory once (swizzled 16-byte
//     chunks); a pick's dot products with all rows are mma.sync products of the
//     16-row tiles with the pick as one of the eight columns (a tcgen05 tile
//     wants 128 rows by 16 columns of which one would be used, and its result
//     would come back through tensor memory between two dependent picks).
//     S_j = max over the picks of cos(q_j, q_r) follows pick by pick.  The first
//     pick uses the identity mean_j cos(q_i, q_j) = (q_i . sum_j q_j / |q_j|) /
//     (N |q_i|), which needs O(N d) instead of O(N^2 d) work; the sum is taken in
//     fp32 and enters the product as three bf16 columns.
//   Error: bf16 products are exact; a K = 16 step rounds at most 17 additions of
//     terms bounded by |q_j||q_r|, so a cosine is within 17 (d / 16) 2^-23 +
//     2^-20 < 2^-15 of the exact one (kCosEps).  For the first pick see first_eps.
//   Exact: similarities with about 44 significant bits without fp64 arithmetic
//     (which is slow on this part): dot products in double-float arithmetic
//     (TwoSum), 1 / |q| from a Newton step, and cos(q_j, q_r) = (q_j . q_r)
//     (1 / |q_j|) (1 / |q_r|).  Rows are compared as the doubles those
//     double-floats equal, so every pick equals that of the fp64 definition
//     except at ties below ~1e-13 relative (lowest index on exact ties).  A
//     row's exact S is kept with the number of picks it covers.  Of rows with
//     the same bits (repeated tokens, zero rows) only the first is compared.
//     Where more than half of the rows left are compared exactly, as with rows
//     all closer than the screening can tell apart, nothing is screened any
//     more; nor is it in an instance with a row whose squared norm is far from 1
//     (or not finite).
//
// What bounds it: issue slots and the two barriers per pick; the rows cross HBM
// once.  Kernel and state read, 4608 instances of 256 rows of 128, 8 picks, with
// all decisions in double-float arithmetic in brackets: 214 us (1217; the rows
// cross HBM in 45); all rows equal 416 (1216), each four times 311 (1218), three in
// four zero 502 (483), all within 0.01 of one direction 1103 (1215), one row of
// extreme norm 1017 (1217).
#include "bkv_device.cuh"
#include "bkv_internal.h"
#include "k_update_math.cuh"

namespace bkv {
namespace {

constexpr size_t kFpsResident = 200 * 1024;  // rows stay in shared memory up to this many bytes
constexpr float kCosEps = 3.0517578125e-05f;  // 2^-15: bound on the error of a screened cosine
constexpr uint32_t kFpsFull = 0xffffffffu;
constexpr int kCovers = 0x3f, kPicked = 0x40, kHasInv = 0x80;  // per-row bits (at most 31 picks are covered)

__device__ __forceinline__ double bf(const __nv_bfloat16 v) { return static_cast<double>(__bfloat162float(v)); }

// Block-wide argmin of (value, index); ties go to the lower index.
__device__ void block_argmin(double v, int i, double* red_v, int* red_i, double& out_v, int& out_i) {
  const unsigned full = 0xffffffffu;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    double ov = __shfl_down_sync(full, v, o);
    int oi = __shfl_down_sync(full, i, o);
    if (ov < v || (ov == v && oi < i)) {
      v = ov;
      i = oi;
    }
  }
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (lane == 0) {
    red_v[w] = v;
    red_i[w] = i;
  }
  __syncthreads();
  if (w == 0) {
    const int nw = blockDim.x >> 5;
    v = lane < nw ? red_v[lane] : INFINITY;
    i = lane < nw ? red_i[lane] : 0x7fffffff;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      double ov = __shfl_down_sync(full, v, o);
      int oi = __shfl_down_sync(full, i, o);
      if (ov < v || (ov == v && oi < i)) {
        v = ov;
        i = oi;
      }
    }
    if (lane == 0) {
      red_v[0] = v;
      red_i[0] = i;
    }
  }
  __syncthreads();
  out_v = red_v[0];
  out_i = red_i[0];
  __syncthreads();
}

// A double-float as the double it equals (hi + lo needs at most 48 significant bits).
__device__ __forceinline__ double df_to_double(DF v) {
  return __dadd_rn(static_cast<double>(v.hi), static_cast<double>(v.lo));
}

// Shared memory of one CTA (byte offsets): the rows themselves when they fit (`resident`), padded to a
// multiple of 16, then per-row values.
struct FpsLayout {
  size_t x, sx, inv, inv32, list, kx, total;
};

__host__ __device__ inline FpsLayout fps_layout(int N, int D, int threads, bool resident) {
  const size_t np = static_cast<size_t>((N + 15) / 16 * 16);
  const size_t upart = static_cast<size_t>(threads / 32) * D * 4;
  FpsLayout l;
  size_t o = 0;
  l.x = o;  // bf16 [np][D], 16-byte chunks swizzled by row
  o += resident ? np * D * 2 : 0;
  l.sx = o;            // double [np]: exact S; before the first exact value, with inv: each warp's part of the sum
  l.inv = o + 8 * np;  // DF [np]: exact 1 / |q|
  o += 16 * np > upart ? 16 * np : upart;
  l.inv32 = o;  // float [np]: screening 1 / |q| (0 for a zero query)
  o += 4 * np;
  l.list = o;  // uint16 [np]: rows to compare exactly
  o += 2 * np;
  l.kx = o;  // uint8 [np]: picks that sx covers (kCovers); kPicked; kHasInv: inv is set
  o += np;
  l.total = o;
  return l;
}

// The 32-bit word (a bf16 pair) w of row j.
template <int D, bool RES>
__device__ __forceinline__ uint32_t row_word(const uint32_t* xs, const __nv_bfloat16* x, int j, int w) {
  if constexpr (RES) {
    return xs[j * (D / 2) + ((((w >> 2) ^ (j & 7)) << 2) | (w & 3))];
  } else {
    return reinterpret_cast<const uint32_t*>(x)[static_cast<size_t>(j) * (D / 2) + w];
  }
}

// The two bf16 values of a word as packed fp32 (low word first), and packed arithmetic on them.
__device__ __forceinline__ unsigned long long widen2(uint32_t w) {
  return static_cast<unsigned long long>(w << 16) | (static_cast<unsigned long long>(w & 0xffff0000u) << 32);
}
__device__ __forceinline__ unsigned long long fma2(unsigned long long a, unsigned long long b, unsigned long long c) {
  unsigned long long d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ float sum2(unsigned long long v) {
  return __uint_as_float(static_cast<uint32_t>(v)) + __uint_as_float(static_cast<uint32_t>(v >> 32));
}

// Element k of row j.
template <int D, bool RES>
__device__ __forceinline__ float element(const uint32_t* xs, const __nv_bfloat16* x, int j, int k) {
  const uint32_t w = row_word<D, RES>(xs, x, j, k >> 1);
  return __uint_as_float((k & 1) ? w & 0xffff0000u : w << 16);
}

// The first row that is not picked.
__device__ __forceinline__ int first_left(const unsigned char* kx, int N) {
  for (int j = 0; j < N; ++j)
    if (!(kx[j] & kPicked)) return j;
  return 0;
}

// 16-byte chunk c of row j.
template <int D, bool RES>
__device__ __forceinline__ uint4 row_chunk(const uint32_t* xs, const __nv_bfloat16* x, int j, int c) {
  if constexpr (RES) {
    const uint32_t off = static_cast<uint32_t>(j * (D * 2) + ((j & 7) << 4));  // a row is a multiple of 128 bytes
    return *reinterpret_cast<const uint4*>(reinterpret_cast<const unsigned char*>(xs) + (off ^ (c << 4)));
  } else {
    return reinterpret_cast<const uint4*>(x)[static_cast<size_t>(j) * (D / 8) + c];
  }
}

// Sum of x_k * y_k over the elements of rows i and j: each product of two bf16 values is exact in fp32, and the
// products are summed in double-float arithmetic in two interleaved chains (even and odd chunks of 8).
template <int D, bool RES>
__device__ __forceinline__ DF row_dot(const uint32_t* xs, const __nv_bfloat16* x, int i, int j) {
  DF a0{0.f, 0.f}, a1{0.f, 0.f};
#pragma unroll 2
  for (int c = 0; c < D / 8; c += 2) {
    const uint4 xa = row_chunk<D, RES>(xs, x, i, c), xb = row_chunk<D, RES>(xs, x, i, c + 1);
    const uint4 ya = row_chunk<D, RES>(xs, x, j, c), yb = row_chunk<D, RES>(xs, x, j, c + 1);
    const uint32_t wx[8] = {xa.x, xa.y, xa.z, xa.w, xb.x, xb.y, xb.z, xb.w};
    const uint32_t wy[8] = {ya.x, ya.y, ya.z, ya.w, yb.x, yb.y, yb.z, yb.w};
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      DF& acc = k < 4 ? a0 : a1;
      acc = df_add(acc, DF{__fmul_rn(__uint_as_float(wx[k] << 16), __uint_as_float(wy[k] << 16)), 0.f});
      acc = df_add(acc, DF{__fmul_rn(__uint_as_float(wx[k] & 0xffff0000u), __uint_as_float(wy[k] & 0xffff0000u)), 0.f});
    }
  }
  return df_add(a0, a1);
}

// Whether rows i and j hold the same bits.
template <int D, bool RES>
__device__ __forceinline__ bool same_row(const uint32_t* xs, const __nv_bfloat16* x, int i, int j) {
#pragma unroll 1
  for (int c = 0; c < D / 8; ++c) {
    const uint4 a = row_chunk<D, RES>(xs, x, i, c), b = row_chunk<D, RES>(xs, x, j, c);
    if (((a.x ^ b.x) | (a.y ^ b.y) | (a.z ^ b.z) | (a.w ^ b.w)) != 0u) return false;
  }
  return true;
}

// Products of the 16 rows r0 .. r0 + 15 (rows of N and more are zero) with the 8 columns whose
// fragments are bf[kk]: lane 4 g + t gets (row r0 + g, columns 2t, 2t + 1) in d[0], d[1] and
// (row r0 + g + 8, ...) in d[2], d[3].
// addr[kk]: this lane's ldmatrix address in tile r0 = 0 of its warp's (resident rows), `off` bytes before the tile.
template <int D, bool RES>
__device__ __forceinline__ void tile_products(const uint32_t* xs, const __nv_bfloat16* x, int N, int r0,
                                              const uint32_t (&addr)[D / 16], uint32_t off,
                                              const uint32_t (&bfrag)[D / 16][2], float (&d)[4]) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int i = 0; i < 4; ++i) d[i] = 0.f;
#pragma unroll
  for (int kk = 0; kk < D / 16; ++kk) {
    uint32_t a0, a1, a2, a3;
    if constexpr (RES) {
      asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                   : "=r"(a0), "=r"(a1), "=r"(a2), "=r"(a3)
                   : "r"(addr[kk] + off));
    } else {
      const int g = r0 + (lane >> 2), w = 8 * kk + (lane & 3);
      a0 = g < N ? row_word<D, RES>(xs, x, g, w) : 0u;
      a1 = g + 8 < N ? row_word<D, RES>(xs, x, g + 8, w) : 0u;
      a2 = g < N ? row_word<D, RES>(xs, x, g, w + 4) : 0u;
      a3 = g + 8 < N ? row_word<D, RES>(xs, x, g + 8, w + 4) : 0u;
    }
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(bfrag[kk][0]), "r"(bfrag[kk][1]));
  }
}

// Column fragments with row r as column 0 and zeros elsewhere.  Resident rows: ldmatrix of four 16-byte
// chunks at a time, whose matrix row 0 is the chunk and whose other rows are a zero chunk.
template <int D, bool RES>
__device__ __forceinline__ void pick_fragments(const uint32_t* xs, const __nv_bfloat16* x, int r, uint32_t zero_chunk,
                                               uint32_t (&bfrag)[D / 16][2]) {
  const int lane = threadIdx.x & 31;
  if constexpr (RES) {
    const uint32_t rbase = smem_u32(xs) + r * (D * 2);
    const uint32_t rswz = static_cast<uint32_t>((lane >> 3) ^ (r & 7)) << 4;
#pragma unroll
    for (int k2 = 0; k2 < D / 32; ++k2) {
      const uint32_t addr = (lane & 7) == 0 ? rbase + (rswz ^ (k2 << 6)) : zero_chunk;
      asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                   : "=r"(bfrag[2 * k2][0]), "=r"(bfrag[2 * k2][1]), "=r"(bfrag[2 * k2 + 1][0]),
                     "=r"(bfrag[2 * k2 + 1][1])
                   : "r"(addr));
    }
  } else {
#pragma unroll
    for (int kk = 0; kk < D / 16; ++kk) {
      bfrag[kk][0] = lane < 4 ? row_word<D, RES>(xs, x, r, 8 * kk + lane) : 0u;
      bfrag[kk][1] = lane < 4 ? row_word<D, RES>(xs, x, r, 8 * kk + 4 + lane) : 0u;
    }
  }
}

// Bound on the error of N times a screened mean cosine: the fp32 sum u over the rows in chains of
// `chain` additions and its 1 / |q| of 2^-21 (the errors' sum is bounded by N, Cauchy-Schwarz), and the
// matrix product of its three bf16 columns (17 additions per K = 16 step, terms bounded by |u|).
template <int D>
__device__ __forceinline__ float first_eps(int N, int chain, float u_norm) {
  return static_cast<float>(N) * static_cast<float>(chain + 16) * 1.1920929e-07f +
         u_norm * (17 * (D / 16) + 32) * 1.1920929e-07f;
}

// NW warps, MT 16-row tiles per warp (warp w takes tiles w, w + NW, ...).  Lane 4 g of a warp owns the
// rows g and g + 8 of each of its tiles: their screening values stay in its registers.
template <int D, int NW, int MT, bool RES>
__global__ void __launch_bounds__(32 * NW, MT == 2 ? 24 / NW : MT == 4 ? (NW == 4 ? 3 : 2) : 1)
    fps_init_kernel(const __nv_bfloat16* __restrict__ q, int N, int nb, float* __restrict__ cent,
                    double* __restrict__ sums, long long* __restrict__ counts) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ double red_v[32];
  __shared__ int red_i[32];
  __shared__ __align__(16) uint32_t zero_sh[4];
  __shared__ uint32_t ucol[3][D / 2];  // the sum of q / |q| as three bf16 columns
  __shared__ DF u[D];                  // the sum, exact path
  __shared__ DF pinv[kMaxBeacons];
  __shared__ int picks[kMaxBeacons];
  __shared__ float u2_sh[NW];          // squared norm of the sum, per warp
  __shared__ uint32_t min_sh[2];       // order key of the smallest screening value, by pick parity
  __shared__ int cnt_sh[2], wild_sh, n_pinv_sh, low_sh, left_sh;

  constexpr int T = 32 * NW;
  const int e = blockIdx.x, tid = threadIdx.x;
  const int warp = tid >> 5, lane = tid & 31;
  const FpsLayout lay = fps_layout(N, D, T, RES);
  uint32_t* xs = reinterpret_cast<uint32_t*>(smem_raw + lay.x);
  double* Sx = reinterpret_cast<double*>(smem_raw + lay.sx);
  DF* inv = reinterpret_cast<DF*>(smem_raw + lay.inv);
  float* upart = reinterpret_cast<float*>(smem_raw + lay.sx);  // [warps][D]
  float* inv32 = reinterpret_cast<float*>(smem_raw + lay.inv32);
  uint16_t* list = reinterpret_cast<uint16_t*>(smem_raw + lay.list);
  unsigned char* kx = smem_raw + lay.kx;

  constexpr int kCh = D / 8;  // 16-byte chunks per row
  const int np = (N + 15) / 16 * 16;
  const __nv_bfloat16* x = q + static_cast<size_t>(e) * N * D;
  // this thread's chunk column and first row in the passes that walk all rows, jstep rows at a time
  constexpr int jstep = T / kCh;
  static_assert(jstep % 8 == 0, "the swizzle of a thread's chunk is the same in all its rows");
  const int c0 = tid % kCh, j0 = tid / kCh;

  if (tid == 0) {
    cnt_sh[0] = cnt_sh[1] = wild_sh = n_pinv_sh = 0;
    min_sh[0] = min_sh[1] = 0xffffffffu;
  }
  if (tid < 4) zero_sh[tid] = 0u;
  if constexpr (RES) {
    for (int j = j0; j < np; j += jstep) {
      uint32_t* dst = xs + j * (D / 2) + ((c0 ^ (j & 7)) << 2);
      if (j < N)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)),
                     "l"(x + static_cast<size_t>(j) * D + c0 * 8)
                     : "memory");
      else
        *reinterpret_cast<uint4*>(dst) = make_uint4(0u, 0u, 0u, 0u);
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
  }
  __syncthreads();

  // ---- screening norms, one row per thread
  for (int j = tid; j < np; j += T) {
    float n2 = 0.f;
    uint32_t any = 0;
    if (j < N) {
      unsigned long long n2a = 0ull, n2b = 0ull;  // packed: even columns low, odd ones high
#pragma unroll 4
      for (int c = 0; c < kCh; ++c) {
        const uint4 v = row_chunk<D, RES>(xs, x, j, c);
        any |= (v.x | v.y) | (v.z | v.w);
        const unsigned long long p0 = widen2(v.x), p1 = widen2(v.y), p2 = widen2(v.z), p3 = widen2(v.w);
        n2a = fma2(p0, p0, n2a);
        n2b = fma2(p1, p1, n2b);
        n2a = fma2(p2, p2, n2a);
        n2b = fma2(p3, p3, n2b);
      }
      n2 = sum2(n2a) + sum2(n2b);
    }
    const bool zero = (any & 0x7fff7fffu) == 0u;
    if (!zero && !(n2 > 1e-25f && n2 < 1e25f)) wild_sh = 1;
    inv32[j] = zero ? 0.f : rsqrtf(n2);
    kx[j] = 0;
  }
  __syncthreads();
  const bool wild = wild_sh != 0;

  // ---- sum of q_j / |q_j|: thread (rows j0, j0 + jstep, ..; chunk c0), then the row groups of the warp and
  // the warps
  const int chain = (N + jstep - 1) / jstep + NW;
  {
    unsigned long long a2[4] = {0ull, 0ull, 0ull, 0ull};
    const uint32_t* xc = xs + j0 * (D / 2) + ((c0 ^ (j0 & 7)) << 2);
#pragma unroll 4
    for (int j = j0; j < N; j += jstep) {
      const uint4 v = RES ? *reinterpret_cast<const uint4*>(xc) : row_chunk<D, RES>(xs, x, j, c0);
      xc += jstep * (D / 2);
      const uint32_t s1 = __float_as_uint(inv32[j]);
      const unsigned long long s = s1 | (static_cast<unsigned long long>(s1) << 32);
      a2[0] = fma2(widen2(v.x), s, a2[0]);
      a2[1] = fma2(widen2(v.y), s, a2[1]);
      a2[2] = fma2(widen2(v.z), s, a2[2]);
      a2[3] = fma2(widen2(v.w), s, a2[3]);
    }
    float a[8];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      a[2 * i] = __uint_as_float(static_cast<uint32_t>(a2[i]));
      a[2 * i + 1] = __uint_as_float(static_cast<uint32_t>(a2[i] >> 32));
    }
#pragma unroll
    for (int o = kCh; o < 32; o <<= 1)
#pragma unroll
      for (int i = 0; i < 8; ++i) a[i] += __shfl_xor_sync(kFpsFull, a[i], o);
    if (lane < kCh) {
      float4* dst = reinterpret_cast<float4*>(upart + warp * D + 8 * lane);
      dst[0] = make_float4(a[0], a[1], a[2], a[3]);
      dst[1] = make_float4(a[4], a[5], a[6], a[7]);
    }
  }
  __syncthreads();
  static_assert(D / 2 <= T, "one bf16 pair of the sum per thread");
  {
    float2 a = make_float2(0.f, 0.f);
    if (tid < D / 2)
#pragma unroll
      for (int g = 0; g < NW; ++g) {
        const float2 p = *reinterpret_cast<const float2*>(&upart[g * D + 2 * tid]);
        a.x += p.x;
        a.y += p.y;
      }
    float u2 = a.x * a.x + a.y * a.y;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) u2 += __shfl_xor_sync(kFpsFull, u2, o);
    if (lane == 0) u2_sh[warp] = u2;
    if (tid < D / 2)
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const __nv_bfloat16 l = __float2bfloat16_rn(a.x), h = __float2bfloat16_rn(a.y);
        ucol[k][tid] =
            static_cast<uint32_t>(__bfloat16_as_ushort(l)) | (static_cast<uint32_t>(__bfloat16_as_ushort(h)) << 16);
        a.x -= __bfloat162float(l);
        a.y -= __bfloat162float(h);
      }
  }
  __syncthreads();

  // ---- screening values of this lane's rows (lanes 4 g): N times the mean cosine for the first pick, then
  // the largest cosine with a pick.  +inf (with a zero 1 / |q|, so that it stays) for a row that is picked
  // and where there is no row.
  uint32_t bfrag[D / 16][2];
  float S[MT][2], iv[MT][2];
  {
    const int col = lane >> 2;
#pragma unroll
    for (int kk = 0; kk < D / 16; ++kk) {
      bfrag[kk][0] = col < 3 ? ucol[col][8 * kk + (lane & 3)] : 0u;
      bfrag[kk][1] = col < 3 ? ucol[col][8 * kk + 4 + (lane & 3)] : 0u;
    }
  }
  const int row0 = 16 * warp + (lane >> 2);  // this lane's first row; row (m, h) is row0 + 16 m NW + 8 h
  uint32_t taddr[D / 16];
#pragma unroll
  for (int kk = 0; kk < D / 16; ++kk) {
    const int lrow = 16 * warp + (lane & 15);
    taddr[kk] = RES ? smem_u32(xs) + lrow * (D * 2) + (((2 * kk + (lane >> 4)) ^ (lrow & 7)) << 4) : 0u;
  }
  constexpr uint32_t kTileStep = 16 * NW * D * 2;  // bytes between a warp's tiles
  float wmin = INFINITY;
#pragma unroll
  for (int m = 0; m < MT; ++m) {
    const int r0 = 16 * (warp + m * NW);
    float d[4] = {0.f, 0.f, 0.f, 0.f};
    if (r0 < np) tile_products<D, RES>(xs, x, N, r0, taddr, m * kTileStep, bfrag, d);  // warp-uniform
    const float c2[2] = {__shfl_down_sync(kFpsFull, d[0], 1), __shfl_down_sync(kFpsFull, d[2], 1)};
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int j = row0 + 16 * m * NW + 8 * h;
      const bool has = (lane & 3) == 0 && j < N;
      iv[m][h] = has && !wild ? inv32[j] : 0.f;  // in a wild instance the products may overflow and say nothing
      S[m][h] = !has ? INFINITY : wild ? 0.f : (d[2 * h] + d[2 * h + 1] + c2[h]) * iv[m][h];
      wmin = fminf(wmin, S[m][h]);
    }
  }
  // Lists the rows whose screening value is within `margin` of the smallest (in a wild instance every row
  // not picked yet) and returns their number; k: the pick being decided.
  auto collect = [&](float margin, int k) -> int {
    const uint32_t key = __reduce_min_sync(kFpsFull, float_order_key(wmin));
    if (lane == 0) atomicMin(&min_sh[k & 1], key);
    __syncthreads();
    if (tid == 0) {  // the next pick's words: last read before this barrier
      cnt_sh[(k + 1) & 1] = 0;
      min_sh[(k + 1) & 1] = 0xffffffffu;
    }
    const uint32_t mk = min_sh[k & 1];
    const float lowest = __uint_as_float((mk & 0x80000000u) ? (mk & 0x7fffffffu) : ~mk);
    const float thr = wild ? 3.4e38f : lowest + margin;
    bool any = false;
#pragma unroll
    for (int m = 0; m < MT; ++m) any |= (S[m][0] <= thr) | (S[m][1] <= thr);
    if (wild || any) {
#pragma unroll
      for (int m = 0; m < MT; ++m)
#pragma unroll
        for (int h = 0; h < 2; ++h)
          if (wild ? S[m][h] != INFINITY : S[m][h] <= thr)
            list[atomicAdd(&cnt_sh[k & 1], 1)] = static_cast<uint16_t>(row0 + 16 * m * NW + 8 * h);
    }
    __syncthreads();
    return cnt_sh[k & 1];
  };
  // Drops from the n listed rows those with the same bits as a listed row of a lower index: they tie with it
  // exactly and lose.  Two such rows are looked for (repeated tokens, zero rows); returns what is left.
  auto drop_repeats = [&](int n) -> int {
    int above = -1;
#pragma unroll 1
    for (int round = 0; round < 2 && n > 1; ++round) {
      if (tid == 0) {
        low_sh = 0x7fffffff;
        left_sh = 0;
      }
      __syncthreads();
      int low = 0x7fffffff;
      for (int c = tid; c < n; c += T) low = list[c] > above ? min(low, static_cast<int>(list[c])) : low;
      low = __reduce_min_sync(kFpsFull, low);
      if (lane == 0) atomicMin(&low_sh, low);
      __syncthreads();
      low = low_sh;
      if (low == 0x7fffffff) break;  // block-uniform
      for (int c0 = 0; c0 < n; c0 += T) {
        const int j = c0 + tid < n ? list[c0 + tid] : -1;
        const bool stays = j >= 0 && (j <= low || !same_row<D, RES>(xs, x, j, low));
        __syncthreads();  // this part of the list is read: what stays of it moves to the front
        if (stays) list[atomicAdd(&left_sh, 1)] = static_cast<uint16_t>(j);
      }
      __syncthreads();
      n = left_sh;
      above = low;
      __syncthreads();
    }
    return n;
  };
  float u2 = u2_sh[0];
#pragma unroll
  for (int w = 1; w < (D / 2 + 31) / 32; ++w) u2 += u2_sh[w];
  int n_cand = drop_repeats(collect(2.f * first_eps<D>(N, chain, sqrtf(u2)), 0));
  bool dense = wild;  // every row not picked yet is compared exactly, nothing is screened
  int r;
  if (n_cand == 1) {
    r = list[0];
  } else {
    // exact: 1 / |q_j| of every row, u = sum_j q_j / |q_j|, then the candidates
    for (int j = tid; j < N; j += T) {
      const DF n2 = row_dot<D, RES>(xs, x, j, j);
      bool plain = true;
      inv[j] = n2.hi > 0.f ? centroid_inv_norm(n2, n2.hi, plain) : DF{0.f, 0.f};
      kx[j] = kHasInv;
    }
    __syncthreads();
    for (int k = tid; k < D; k += T) {
      DF a{0.f, 0.f};
      for (int j = 0; j < N; ++j) a = df_add(a, df_mul(DF{element<D, RES>(xs, x, j, k), 0.f}, inv[j]));
      u[k] = a;
    }
    __syncthreads();
    double best_v = INFINITY;
    int best_i = 0x7fffffff;
    for (int c = tid; c < n_cand; c += T) {
      const int i = list[c];
      DF t{0.f, 0.f};
      if (inv[i].hi > 0.f) {
        DF a{0.f, 0.f};
        for (int k = 0; k < D; ++k) a = df_add(a, df_mul(DF{element<D, RES>(xs, x, i, k), 0.f}, u[k]));
        t = df_mul(a, inv[i]);
      }
      const double tv = df_to_double(t);
      if (tv < best_v || (tv == best_v && i < best_i)) {
        best_v = tv;
        best_i = i;
      }
    }
    double pv;
    block_argmin(best_v, best_i, red_v, red_i, pv, r);
    if (r >= N) r = n_cand > 0 ? list[0] : 0;  // no finite value at all
  }
  if (tid == 0) {
    picks[0] = r;
    kx[r] |= kPicked;
  }

  // ---- S_j = max over the picks of cos(q_j, q_pick), one pick at a time
  const uint32_t zero_chunk = smem_u32(zero_sh);
  for (int k = 1; k < nb; ++k) {
    if (!dense) {
      const float inv_r = inv32[r];
      pick_fragments<D, RES>(xs, x, r, zero_chunk, bfrag);
      if (k == 1) {
#pragma unroll
        for (int m = 0; m < MT; ++m)
#pragma unroll
          for (int h = 0; h < 2; ++h)
            S[m][h] = (lane & 3) == 0 && row0 + 16 * m * NW + 8 * h < N ? -INFINITY : INFINITY;
      }
      if (((r >> 4) & (NW - 1)) == warp) {  // r is one of this warp's rows
#pragma unroll
        for (int m = 0; m < MT; ++m)
#pragma unroll
          for (int h = 0; h < 2; ++h)
            if (row0 + 16 * m * NW + 8 * h == r && (lane & 3) == 0) {
              S[m][h] = INFINITY;
              iv[m][h] = 0.f;
            }
      }
      wmin = INFINITY;
#pragma unroll
      for (int m = 0; m < MT; ++m) {
        const int r0 = 16 * (warp + m * NW);
        if (r0 >= np) continue;  // warp-uniform
        float d[4];
        tile_products<D, RES>(xs, x, N, r0, taddr, m * kTileStep, bfrag, d);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          S[m][h] = fmaxf(S[m][h], d[2 * h] * inv_r * iv[m][h]);
          wmin = fminf(wmin, S[m][h]);
        }
      }
      n_cand = collect(2.f * kCosEps, k);
      if (n_cand > 1) n_cand = drop_repeats(n_cand);
    } else {
      __syncthreads();  // the last pick is marked
      n_cand = N - k;
    }
    if (n_cand == 1 && !dense) {
      r = list[0];
    } else {
      // exact 1 / |q| of the picks so far, then each candidate's S over the picks it does not cover yet
      auto inv_of = [&](int j) -> DF {
        if (kx[j] & kHasInv) return inv[j];
        const DF n2 = row_dot<D, RES>(xs, x, j, j);
        bool plain = true;
        return n2.hi > 0.f ? centroid_inv_norm(n2, n2.hi, plain) : DF{0.f, 0.f};
      };
      for (int m = n_pinv_sh + tid; m < k; m += T) pinv[m] = inv_of(picks[m]);
      __syncthreads();
      if (tid == 0) n_pinv_sh = k;
      auto cosine = [&](int j, DF inv_j, int m) -> double {
        if (!(inv_j.hi > 0.f && pinv[m].hi > 0.f)) return 0.0;
        return df_to_double(df_mul(df_mul(row_dot<D, RES>(xs, x, j, picks[m]), inv_j), pinv[m]));
      };
      double v = INFINITY;
      int vi = 0x7fffffff;
      if (!dense && n_cand <= 4 * NW) {  // a few: a warp per candidate, a lane per pick
        for (int c = warp; c < n_cand; c += NW) {
          const int j = list[c];
          const int k0 = kx[j] & kCovers;
          const DF inv_j = inv_of(j);
          const double cv = lane >= k0 && lane < k ? cosine(j, inv_j, lane) : 0.0;
          double Sj = k0 ? Sx[j] : 0.0;
          for (int m = k0; m < k; ++m) {
            const double cm = __shfl_sync(kFpsFull, cv, m);
            if (m == 0 || cm > Sj) Sj = cm;
          }
          __syncwarp();
          if (lane == 0) {
            Sx[j] = Sj;
            inv[j] = inv_j;
            kx[j] = static_cast<unsigned char>(kHasInv | k);
          }
          if (Sj < v || (Sj == v && j < vi)) {
            v = Sj;
            vi = j;
          }
        }
      } else {  // many: a thread per candidate
        for (int c = tid; c < (dense ? N : n_cand); c += T) {
          const int j = dense ? c : list[c];
          if (dense && (kx[j] & kPicked)) continue;
          bool has_inv = (kx[j] & kHasInv) != 0;
          DF inv_j = inv[j];
          double Sj = Sx[j];
          for (int m = kx[j] & kCovers; m < k; ++m) {
            if (!has_inv && pinv[m].hi > 0.f) {  // 0 with a zero pick: no norm is needed
              inv_j = inv_of(j);
              has_inv = true;
            }
            const double cm = has_inv ? cosine(j, inv_j, m) : 0.0;
            if (m == 0 || cm > Sj) Sj = cm;
          }
          Sx[j] = Sj;
          inv[j] = inv_j;
          kx[j] = static_cast<unsigned char>((has_inv ? kHasInv : 0) | k);
          if (Sj < v || (Sj == v && j < vi)) {
            v = Sj;
            vi = j;
          }
        }
      }
      double rv;
      block_argmin(v, vi, red_v, red_i, rv, r);
      if (r >= N) r = dense ? first_left(kx, N) : list[0];  // no finite value at all
      // rows that lie closer together than the screening can tell apart will do so for the next picks too
      dense = dense || 2 * n_cand > N - k;
    }
    if (tid == 0) {
      picks[k] = r;
      kx[r] |= kPicked;
    }
  }
  __syncthreads();

  // beacon k = k-th pick, count 1
  for (int idx = tid; idx < nb * D; idx += T) {
    const int k = idx / D, i = idx % D;
    const __nv_bfloat16 v = x[static_cast<size_t>(picks[k]) * D + i];
    cent[(static_cast<size_t>(e) * nb + k) * D + i] = __bfloat162float(v);
    if (sums) sums[(static_cast<size_t>(e) * nb + k) * D + i] = bf(v);
  }
  for (int k = tid; k < nb; k += T) counts[static_cast<size_t>(e) * nb + k] = 1;
}

template <int D, int NW, int MT, bool RES>
cudaError_t launch_fps_dr(const Shape& s, const __nv_bfloat16* q_init, int N, float* cent, double* sums,
                          long long* counts, cudaStream_t st) {
  const size_t smem = fps_layout(N, D, 32 * NW, RES).total;
  const cudaError_t e = allow_smem<fps_init_kernel<D, NW, MT, RES>>(smem);
  if (e != cudaSuccess) return e;
  fps_init_kernel<D, NW, MT, RES><<<s.n_inst, 32 * NW, smem, st>>>(q_init, N, s.nb, cent, sums, counts);
  return cudaGetLastError();
}

// Four warps up to 256 rows, with two or four tiles each (eight warps of two tiles: 233 us instead of 227 on
// 4608 instances of 256 rows of 128, call and state read: what a pick costs a warp besides its tiles is paid
// twice); eight of four tiles up to 512 rows, two CTAs per SM where sixteen warps left room for one (1152
// instances: 272 rows 154 -> 98 us, 512 rows 213 -> 175); above, up to 4096 rows, eight tiles per warp.  Rows
// that do not fit in shared memory are read from global memory (L2) in every pass.
template <int D>
cudaError_t launch_fps_d(const Shape& s, const __nv_bfloat16* q_init, int N, float* cent, double* sums,
                         long long* counts, cudaStream_t st) {
  if (N <= 128) return launch_fps_dr<D, 4, 2, true>(s, q_init, N, cent, sums, counts, st);
  if (N <= 256) return launch_fps_dr<D, 4, 4, true>(s, q_init, N, cent, sums, counts, st);
  if (N <= 512) return launch_fps_dr<D, 8, 4, true>(s, q_init, N, cent, sums, counts, st);
  if (N <= 2048 && fps_layout(N, D, 512, true).total <= kFpsResident)
    return launch_fps_dr<D, 16, 8, true>(s, q_init, N, cent, sums, counts, st);
  if (N <= 2048) return launch_fps_dr<D, 16, 8, false>(s, q_init, N, cent, sums, counts, st);
  return launch_fps_dr<D, 32, 8, false>(s, q_init, N, cent, sums, counts, st);
}

}  // namespace

cudaError_t launch_fps_init(const Shape& s, const __nv_bfloat16* q_init, int n_init, float* cent, double* sums,
                            long long* counts, cudaStream_t st) {
  const int N = s.G * n_init;
  return s.d == 128 ? launch_fps_d<128>(s, q_init, N, cent, sums, counts, st)
                    : launch_fps_d<64>(s, q_init, N, cent, sums, counts, st);
}

}  // namespace bkv
