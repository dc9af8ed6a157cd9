// Beacon maintenance (Section 3.2, Appendix D): every new query is assigned to
// the beacon of highest cosine similarity and that beacon's centroid becomes
// the running mean of the queries assigned to it.
//
// Persistent kernel, one CTA per SM; CTA k takes instances k, k + grid, ...
// An instance's queries stream through a ring of shared-memory stages in
// tiles of up to 128 (TMA, 128-byte swizzle) and are read from HBM once.
// Both contractions of a tile run on the tensor cores (tcgen05):
//
// Screening: D1 = Q x [c_hi ; c_lo]^T where c_hi = bf16(c / |c|) and c_lo =
// bf16(c / |c| - c_hi), so dot_b = D1[:, b] + D1[:, nbp + b] carries the
// unit-centroid dot to about 2^-16 |q| (bf16 x bf16 products are exact, the
// accumulation is fp32).  When best and second-best dots differ by at most
// 7e-5 |q| (kScreenMargin; the bound is 4.2e-5 |q|), the query is re-decided
// exactly: the beacon maximising (q . c_b) / |c_b| in double-float arithmetic
// (exact products, TwoSum accumulation, 1 / |c_b| from a double-float sum of
// squares and one Newton step, to about 2^-44 relative), which agrees with the
// cosine (q . c_b) / (|q| |c_b|) evaluated in fp64 except at ties below ~1e-12
// (the lowest beacon wins ties).  Only beacons screened within 1.4e-4 |q| of the
// best enter that comparison.  |q| is formed, in fp32, only where the larger
// sqrt(d) max|q_i| (exact: a packed maximum) does not rule a re-decision out (8192
// instances of 512 queries, call and state read: 534 us, with an fp32 sum for
// every query 574).  Zero queries and instances without a valid beacon give -1.
//
// Sums: Q^T x A, where A is the tile's one-hot assignment matrix (128 queries x
// beacons), exact: an element x with |x| < 2^E (E chosen per instance) goes
// whole into one of two operands, the tile itself (|x| >= 2^(E-10), a multiple
// of 2^(E-17)) or a second tile (smaller ones, multiples of 2^(E-27) for
// |x| >= 2^(E-20)), whose sums over 128 rows stay below 2^24 grid steps, so the
// fp32 accumulator never rounds.  The two sums of a (column, beacon) cell are
// integers, added up over the tiles in two registers.  The few elements outside
// [2^(E-20), 2^E) (one in ten tiles of normal data) are zeroed in the operands
// and added as a list (past 32 per instance through a global array of this CTA).
// E comes from the largest element this CTA has seen (before that from the
// centroids), never below -11, so that what the operands hold is exact in fixed
// point with 40 fractional bits; the result does not depend on it.
//
// The call's sums (int64, 40 fractional bits) and counts go to scratch.  After its
// last tile the CTA adds them once to the fp64 running sums of its instances,
// correctly rounded and without fp64 arithmetic (slow on this part), and forms
// c = fp32(sum / count) to within one fp32 ulp from double-float arithmetic on the
// sum's bits.
//
// Warp roles (23 warps): warp 0 TMA producer; warp 1 TMEM allocation and the
// screening MMAs; warp 2 the sums' MMAs; warps 3..10 two groups of four that
// take alternate tiles, one query per thread (its decision, the split of its
// elements, its column of A); warps 11..18 one column of d and half of the
// beacons per thread: they take the sums out of tensor memory; warps 19..22
// build the unit-centroid operand of the next instances.  All waits are bounded.
//
// What bounds it: a tile's chain through its group (dots, split, decision, sums:
// about 8 K clocks, two tiles in flight per SM because shared memory holds no
// third second-tile) and instruction fetch: the roles share the instruction caches,
// so loops are kept rolled and rare paths small (re-decisions and spilled elements,
// three tiles in ten, still cost a fifth of the time).  Sums formed in fp32 parts
// by CUDA cores from rows sorted by beacon took about 14 K warp instructions per
// tile.  With the fold (in a launch of its own: 255 and 485 us): 4608 instances x 512 queries of 128, 8 beacons: 393
// us, now 242 (95 at the copy rate); 8192 instances, 16 beacons: 815 us, now 476
// (178).
#include "bkv_device.cuh"
#include "bkv_internal.h"
#include "k_update_math.cuh"

namespace bkv {
namespace {

constexpr int kGroups = 2;                  // row groups of four warps, one tile each
constexpr int kGroupWarp0 = 3;              // first of the row groups' warps
constexpr int kSumWarp0 = kGroupWarp0 + 4 * kGroups;  // first of the eight warps that take the sums
constexpr int kBuildWarp0 = kSumWarp0 + 8;
constexpr int kUThreads = 32 * (kBuildWarp0 + 4);
constexpr int kQTile = 128;                 // queries per tile (MMA M of the screening, K of the sums)
constexpr uint32_t kQBox = 128 * 128;       // [128 rows][64 bf16] swizzled box slot
constexpr int kUMaxStages = 6;
constexpr int kDots = 3;                    // screening accumulators in tensor memory
constexpr int kSums = 4;                    // sum accumulators in tensor memory
constexpr int kSlots = 16;                  // per-instance words in flight between the roles (at most 11 instances)
constexpr int kSpillSlots = 8;              // instances whose spilled elements may be in flight
constexpr int kSpillList = 32;              // spilled elements per instance kept in shared memory
constexpr size_t kUSmemBudget = 220 * 1024;
// A query is re-decided exactly when its best and second-best dots differ by at most this fraction of |q|.
// A screened dot is within 2^-18 |q| (the hi / lo split) + 136 * 2^-23 |q| (17 additions in each of eight
// K = 16 steps) + 2^-21 |q| (1 / |c|) of the exact one, so a difference of two within 4.2e-5 |q|.
constexpr float kScreenMargin = 7e-5f;
// Queries whose largest element is in this range have a squared norm that fp32 holds (1e-30 < |q|^2 < 1e30).
constexpr float kTameLo = 1.7763568394002505e-15f, kTameHi = 70368744177664.f;  // 2^-49, 2^46
constexpr int kMinE = -11, kMaxE = 14;
constexpr int kLargeBits = 10;              // octaves below 2^E that the tile itself holds
constexpr int kSmallBits = 20;              // octaves below 2^E that the operands hold

struct UpdArgs {
  int n_inst, nq, nb, nbp;  // instances, queries per instance, beacons, beacons padded to 8
  int box_rows;             // rows of one TMA box of queries (<= 128)
  float* cent;
  double* sums;
  long long* counts;
  int* assign_out;
  unsigned long long* spill;  // [grid][kSpillSlots][nb][D], zero between instances
  long long* call_sum;        // [n_inst][nb][D]: this call's sums, units of 2^-40
  int* call_cnt;              // [n_inst][nb]: queries assigned
  int* err;
};

// NBO: beacons padded to 16 (the N of the sums' MMA).
template <int D, int NBO>
struct UpdCfg {
  static constexpr int kBoxes = D / 64;
  static constexpr uint32_t kStageBytes = kBoxes * kQBox;
  static constexpr uint32_t kHotBytes = 2 * NBO * 128;    // one-hot operand: two 64-query boxes of NBO rows
  static constexpr int kParts = D == 128 ? 2 : 1;         // accumulators per tile (d = 64: both operands in one)
  static constexpr uint32_t kXchg = D == 64 ? 64 * NBO * 4 : 0;  // d = 64: the small parts' sums at a fold
  __host__ __device__ static uint32_t bmat_bytes(int nbp) { return static_cast<uint32_t>(kBoxes) * 2 * nbp * 128; }
  __host__ __device__ static uint32_t fixed_bytes(int nbp) {
    return kGroups * (kStageBytes + kHotBytes) + 2 * bmat_bytes(nbp) + kXchg;
  }
  static int stages(int nbp) {
    const int n = static_cast<int>((kUSmemBudget - 1024 - fixed_bytes(nbp)) / kStageBytes);
    return n < kUMaxStages ? n : kUMaxStages;
  }
  static size_t smem_bytes(int nbp) { return 1024 + static_cast<size_t>(stages(nbp)) * kStageBytes + fixed_bytes(nbp); }
};

__device__ __forceinline__ void drain_wait(uint64_t* bar, uint32_t parity, int* err) {
  int never = 0;
  mbar_wait(bar, parity, &never, err, kDevTimeoutDrain);
}

__device__ __forceinline__ void fence_proxy_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// Brings `bytes` (a multiple of 16) at p into L2.
__device__ __forceinline__ void bulk_prefetch_l2(const void* p, uint32_t bytes) {
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(reinterpret_cast<uint64_t>(p)), "r"(bytes) : "memory");
}

// round(x * 2^40) of the bf16 value whose bits sit in the upper half of
// `hi16` (lower half zero): the scale is added to the fp32 exponent field
// (exact for |x| < 2^88; a zero or subnormal x becomes a value below 2^-80,
// which rounds to 0 as x * 2^40 would), then one round-to-nearest conversion.
__device__ __forceinline__ long long bf16_fixed40(uint32_t hi16) {
  return __float2ll_rn(__uint_as_float(hi16 + (40u << 23)));
}

// Byte offset of element (row, col) in a [rows][D] bf16 tile stored as D / 64
// boxes of [rows][64] with the 128-byte swizzle (box_bytes apart).
__device__ __forceinline__ uint32_t sw128_offset(int row, int col, uint32_t box_bytes) {
  return (col >> 6) * box_bytes + row * 128 + ((((col & 63) >> 3) ^ (row & 7)) << 4) + ((col & 7) << 1);
}

// Shared-memory descriptor of an operand read across its rows (MN-major): 64 elements of a row per
// 128-byte line, 8-row groups 1024 B apart, the next 64 elements `lbo` bytes further; 128-byte swizzle.
__device__ __forceinline__ uint64_t sdesc_mnmajor_sw128(uint32_t smem_addr, uint32_t lbo) {
  return (sdesc_kmajor_sw128(smem_addr) & ~(0x3FFFull << 16)) | (static_cast<uint64_t>((lbo >> 4) & 0x3FFFu) << 16);
}

// 16-byte shared-memory store where cond is not 0, predicated rather than branched around.
__device__ __forceinline__ void st_shared_v4_if(uint32_t cond, void* p, uint32_t x, uint32_t y, uint32_t z, uint32_t w) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.u32 p, %0, 0;\n\t"
      "@p st.shared.v4.b32 [%1], {%2, %3, %4, %5};\n\t}" ::"r"(cond),
      "r"(smem_u32(p)), "r"(x), "r"(y), "r"(z), "r"(w)
      : "memory");
}

// bf16 bits of 2^k, in both halves of a word.
__device__ __forceinline__ uint32_t pow2_bf16x2(int k) {
  const uint32_t b = static_cast<uint32_t>(k + 127) << 7;
  return b | (b << 16);
}

__device__ __forceinline__ __nv_bfloat162 as_bf162(uint32_t w) { return *reinterpret_cast<__nv_bfloat162*>(&w); }

// 8 consecutive fp32 columns of this thread's TMEM lane.
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, float* v) {
  uint32_t r[8];
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr));
#pragma unroll
  for (int i = 0; i < 8; ++i) v[i] = __uint_as_float(r[i]);
}

// Exact assignment of query n of the tile (its elements are in `raw` or, where that holds 0, in `small`)
// among the candidate beacons (warp-wide): the valid beacon
// maximising (q . c_b) * (1 / |c_b|) in double-float arithmetic, ties to the lower beacon, -1 for a zero
// query (exact_decision's result: the same operations, with a candidate's dot and norm formed together
// and the next candidate's row already loading).  Out of line: rare.
template <int D>
__device__ __noinline__ int refine_row(const unsigned char* raw, const unsigned char* small, int n, const float* cent_e,
                                       uint32_t cand) {
  const int lane = threadIdx.x & 31;
  float x[D / 32], c[D / 32];
  int b = __ffs(cand) - 1;
#pragma unroll
  for (int j = 0; j < D / 32; ++j) {
    const uint32_t off = sw128_offset(n, lane + 32 * j, kQBox);
    const uint32_t w = *reinterpret_cast<const uint16_t*>(raw + off) | *reinterpret_cast<const uint16_t*>(small + off);
    x[j] = __uint_as_float(w << 16);
    c[j] = cand ? cent_e[b * D + lane + 32 * j] : 0.f;
  }
  int nz = 0;
#pragma unroll
  for (int j = 0; j < D / 32; ++j) nz |= x[j] != 0.f;
  if (!__any_sync(0xffffffffu, nz)) return -1;
  DF best{-INFINITY, 0.f};
  int best_b = -1;
  while (cand) {
    cand &= cand - 1;
    const int b_next = __ffs(cand) - 1;
    float c_next[D / 32];
#pragma unroll
    for (int j = 0; j < D / 32; ++j) c_next[j] = cand ? cent_e[b_next * D + lane + 32 * j] : 0.f;
    float n2 = 0.f;
    DF n2d{0.f, 0.f}, dt{0.f, 0.f};
#pragma unroll
    for (int j = 0; j < D / 32; ++j) {
      n2 = fmaf(c[j], c[j], n2);
      n2d = df_add(n2d, df_two_prod(c[j], c[j]));
      dt = df_add(dt, df_two_prod(x[j], c[j]));
    }
#pragma unroll 1  // few instructions: they are fetched cold
    for (int o = 16; o > 0; o >>= 1) {
      n2 += __shfl_xor_sync(0xffffffffu, n2, o);
      n2d = df_add(n2d, DF{__shfl_xor_sync(0xffffffffu, n2d.hi, o), __shfl_xor_sync(0xffffffffu, n2d.lo, o)});
      dt = df_add(dt, DF{__shfl_xor_sync(0xffffffffu, dt.hi, o), __shfl_xor_sync(0xffffffffu, dt.lo, o)});
    }
    bool plain = true;
    const DF cs = df_mul(dt, centroid_inv_norm(n2d, n2, plain));
    if (best_b < 0 || df_gt(cs, best)) {
      best = cs;
      best_b = b;
    }
    b = b_next;
#pragma unroll
    for (int j = 0; j < D / 32; ++j) c[j] = c_next[j];
  }
  return best_b;
}

// fp32 squared norm of this thread's query: a chunk's elements sit in the raw tile or, where that holds 0, in
// the second one.  Out of line and rolled: rare.
template <int D>
__device__ __noinline__ float row_norm2(const unsigned char* raw_row, const unsigned char* small_row, uint32_t swz) {
  unsigned long long n2[4] = {0ull, 0ull, 0ull, 0ull};
#pragma unroll 2
  for (int c = 0; c < D / 8; ++c) {
    const uint32_t off = (c >> 3) * kQBox + (static_cast<uint32_t>((c & 7) << 4) ^ swz);
    const uint4 r = *reinterpret_cast<const uint4*>(raw_row + off), s = *reinterpret_cast<const uint4*>(small_row + off);
    n2[0] = add_squares(n2[0], r.x | s.x);
    n2[1] = add_squares(n2[1], r.y | s.y);
    n2[2] = add_squares(n2[2], r.z | s.z);
    n2[3] = add_squares(n2[3], r.w | s.w);
  }
  return (packed_total(n2[0]) + packed_total(n2[1])) + (packed_total(n2[2]) + packed_total(n2[3]));
}

// cnt[b] += the number of lanes whose mine == b (mine < 0: none), for every b < NB: five 6-bit counters per
// warp sum, then one conflict-free addition per beacon (one atomic per lane would serialise).
template <int NB>
__device__ __forceinline__ void add_counts(int* cnt, int mine) {
  const int lane = threadIdx.x & 31;
  constexpr int kWords = (NB + 4) / 5;
  uint32_t tot = 0u;
#pragma unroll
  for (int w = 0; w < kWords; ++w) {
    const int k = mine - 5 * w;
    const uint32_t sum = __reduce_add_sync(0xffffffffu, k >= 0 && k < 5 ? 1u << (6 * k) : 0u);
    tot = lane / 5 == w ? sum : tot;
  }
  const int n = static_cast<int>((tot >> (6 * (lane % 5))) & 63u);
  if (lane < NB && n > 0) atomicAdd(&cnt[lane], n);
}

// Spilled elements of one instance: the first kSpillList as (beacon << 8 | column, fixed point) here, more
// in the CTA's global array.
struct SpillList {
  int n;
  int key[kSpillList];
  long long val[kSpillList];
};

// The elements of one row (n of the tile) that the operands cannot hold: |x| >= 2^E (or not finite), which
// sit in the tile, and 0 < |x| < 2^(E - 20), which sit in the second one.  Each is zeroed there and noted
// for the row's beacon (b < 0: the row is not assigned).  Warp-wide; returns whether some went to the
// global array.  Out of line: rare.
template <int D>
__device__ __noinline__ bool spill_row(unsigned char* raw, unsigned char* small, int n, int E, int b, SpillList* list,
                                       unsigned long long* spill) {
  const int lane = threadIdx.x & 31;
  const uint32_t hi = pow2_bf16x2(E) & 0xffffu, lo = pow2_bf16x2(E - kSmallBits) & 0xffffu;
  constexpr int kC = D / 32;  // this lane's columns
  bool over = false;
#pragma unroll 1  // few instructions: they are fetched cold
  for (int k = 0; k < kC; ++k) {
    const int col = lane * kC + k;
    const uint32_t off = sw128_offset(n, col, kQBox);
    uint16_t* in_raw = reinterpret_cast<uint16_t*>(raw + off);
    uint16_t* in_small = reinterpret_cast<uint16_t*>(small + off);
    const uint32_t w = *in_raw | *in_small, m = w & 0x7fffu;  // one of the two is zero
    if (m == 0u || (m >= lo && m < hi)) continue;
    *in_raw = 0;
    *in_small = 0;
    if (b < 0) continue;
    const float x = __uint_as_float(w << 16);
    const long long f = fabsf(x) < 16384.f ? fixed40_one(x) : bf16_fixed40(w << 16);
    const int at = atomicAdd(&list->n, 1);
    if (at < kSpillList) {
      list->key[at] = (b << 8) | col;
      list->val[at] = f;
    } else {
      atomicAdd(spill + b * D + col, static_cast<unsigned long long>(f));
      over = true;
    }
  }
  if (!__any_sync(0xffffffffu, over)) return false;
  __threadfence();
  return true;
}

template <int D, int NBO>
__global__ void __launch_bounds__(kUThreads, 1)
    update_kernel(const __grid_constant__ CUtensorMap qmap, UpdArgs a, int n_stages) {
  using C = UpdCfg<D, NBO>;
  extern __shared__ unsigned char smem_raw[];
  __shared__ __align__(8) uint64_t full_bar[kUMaxStages], empty_bar[kUMaxStages];
  __shared__ __align__(8) uint64_t accfull[kDots], accfree[kDots], bready[2], bfree[2], drain_bar[2];
  __shared__ __align__(8) uint64_t sumready[kGroups], smallfree[kGroups], sumfull[kSums], cntready[kSums], sumfree[kSums];
  __shared__ uint32_t tmem_base_sh;
  __shared__ int abort_sh;
  __shared__ uint32_t seen_sh;               // largest element magnitude below 2^kMaxE seen so far (bf16 bits)
  // per instance in flight
  __shared__ uint32_t vmask_sh[kSlots];      // valid beacons (count > 0, nonzero centroid)
  __shared__ int exp_sh[kSlots];             // E; bit 8: a centroid norm is extreme, every query is re-decided
  __shared__ int add_cnt[kSlots][kMaxBeacons];  // queries assigned so far
  __shared__ int spilled_sh[kSlots];         // elements or sums went to the global array
  __shared__ SpillList list_sh[kSpillSlots];
  __shared__ uint32_t kv_sh[4];              // builders: each warp's valid beacons
  __shared__ uint32_t km_sh[4];              // builders: each warp's largest |c|^2 (fp32 bits), bit 31: extreme norm

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nq = a.nq, nb = a.nb, nbp = a.nbp;
  const int n_my = blockIdx.x < a.n_inst ? (a.n_inst - blockIdx.x + gridDim.x - 1) / gridDim.x : 0;
  const int T = (nq + kQTile - 1) / kQTile;  // tiles per instance
  const int n_tiles = n_my * T;
  const int ncols1 = 2 * nbp;                 // screening columns (hi, lo)
  const uint32_t bbox = static_cast<uint32_t>(ncols1) * 128;  // bytes of one 64-column box of bmat

  // 1024-byte aligned (the 128-byte swizzle pattern repeats every 1024 bytes);
  // offset from the __shared__ array itself so that accesses stay shared-space
  unsigned char* base = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  unsigned char* stage_smem = base;                                               // [n_stages][kBoxes][128 x 128 B]
  unsigned char* small_smem = base + static_cast<size_t>(n_stages) * C::kStageBytes;  // [kGroups][kBoxes][128 x 128 B]
  unsigned char* hot_smem = small_smem + kGroups * C::kStageBytes;                // [kGroups][2][NBO x 128 B]
  unsigned char* bmat = hot_smem + kGroups * C::kHotBytes;                        // [2][kBoxes][2 nbp x 128 B]
  int* xchg = reinterpret_cast<int*>(bmat + 2 * C::bmat_bytes(nbp));  // d = 64: [NBO][64]

  if (threadIdx.x == 0) {
    for (int i = 0; i < n_stages; ++i) {
      mbar_init(&full_bar[i], 1);
      mbar_init(&empty_bar[i], 1);
    }
    for (int i = 0; i < kDots; ++i) {
      mbar_init(&accfull[i], 1);
      mbar_init(&accfree[i], 4);  // the four warps of the tile's group
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&bready[i], 1);
      mbar_init(&bfree[i], 1);
    }
    for (int i = 0; i < kGroups; ++i) {
      mbar_init(&sumready[i], 4);
      mbar_init(&smallfree[i], 1);
    }
    for (int i = 0; i < kSums; ++i) {
      mbar_init(&sumfull[i], 1);
      mbar_init(&cntready[i], 1);
      mbar_init(&sumfree[i], 8);
    }
    mbar_init(&drain_bar[0], 1);
    mbar_init(&drain_bar[1], 1);
    abort_sh = 0;
    seen_sh = 0;
    fence_mbar_init();
  }
  for (uint32_t i = threadIdx.x; i < kGroups * C::kHotBytes / 16; i += kUThreads)
    reinterpret_cast<uint4*>(hot_smem)[i] = make_uint4(0u, 0u, 0u, 0u);
  for (int i = threadIdx.x; i < kSlots * kMaxBeacons; i += kUThreads) (&add_cnt[0][0])[i] = 0;
  if (threadIdx.x < kSlots) spilled_sh[threadIdx.x] = 0;
  if (threadIdx.x < kSpillSlots) list_sh[threadIdx.x].n = 0;
  if (warp == 1) {
    tmem_alloc(&tmem_base_sh, 512);
    tmem_relinquish();
  }
  fence_proxy_async_smem();  // the one-hot operands' zeros are read by the tensor cores
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  grid_dependency_wait();  // the set-up above touched no global memory
  const uint32_t tmem = tmem_base_sh;
  const uint32_t tmem_sums = tmem + kDots * ncols1;  // [kSums][kParts * NBO]
  volatile int* abort_flag = &abort_sh;

  if (warp == 0) {
    // ---------------------------------------------------------------- producer
    if (elect_one()) {
      const uint64_t once = l2_policy_evict_first();
      prefetch_tmap(&qmap);
      int st = 0, round = 0;  // stage and how often the ring has gone round
      bool ok = true;
      for (int i = 0; ok && i < n_my; ++i) {
        const int row0 = (blockIdx.x + i * gridDim.x) * nq;
        for (int t = 0; t < T; ++t) {
          if (round > 0 && !mbar_wait(&empty_bar[st], (round - 1) & 1, abort_flag, a.err, kDevTimeoutProducer)) {
            ok = false;
            break;
          }
          mbar_arrive_expect_tx(&full_bar[st], static_cast<uint32_t>(C::kBoxes * a.box_rows * 128));
          for (int b = 0; b < C::kBoxes; ++b)
            tma_load_2d(stage_smem + st * C::kStageBytes + b * kQBox, &qmap, &full_bar[st], b * 64, row0 + t * kQTile,
                        once);
          if (++st == n_stages) {
            st = 0;
            ++round;
          }
        }
      }
      if (!ok || *abort_flag) {  // let every copy already issued land before the CTA exits
        const int g = round * n_stages + st;
        for (int j = (g > n_stages ? g - n_stages : 0); j < g; ++j)
          drain_wait(&full_bar[j % n_stages], (j / n_stages) & 1, a.err);
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    // ---------------------------------------------------------------- screening MMAs
    // Their own warp, so that a tile's dots never wait behind an earlier tile whose sums are not ready.
    if (elect_one()) {
      const uint32_t idesc1 = idesc_bf16_f32(128, ncols1);
      const uint32_t stage0 = smem_u32(stage_smem);
      int si = 0, s_t = 0, s_st = 0, s_round = 0, s_ab = 0, s_use = 0;  // screening: instance, tile, stage, accumulator
      auto screen = [&]() -> bool {
        const int pb = si & 1;
        if (s_t == 0 && !mbar_wait(&bready[pb], (si >> 1) & 1, abort_flag, a.err, kDevTimeoutMma)) return false;
        if (!mbar_wait(&full_bar[s_st], s_round & 1, abort_flag, a.err, kDevTimeoutMma)) return false;
        if (s_use > 0 && !mbar_wait(&accfree[s_ab], (s_use - 1) & 1, abort_flag, a.err, kDevTimeoutMma)) return false;
        tc_fence_after();
        const uint32_t d = tmem + s_ab * ncols1;
        const uint32_t q_addr = stage0 + s_st * C::kStageBytes;
        const uint32_t b_addr = smem_u32(bmat) + pb * C::bmat_bytes(nbp);
#pragma unroll
        for (int kk = 0; kk < D / 16; ++kk)
          mma_bf16_ss(d, sdesc_kmajor_sw128(q_addr + (kk >> 2) * kQBox + (kk & 3) * 32),
                      sdesc_kmajor_sw128(b_addr + (kk >> 2) * bbox + (kk & 3) * 32), idesc1, kk > 0);
        mma_commit(&accfull[s_ab]);
        if (++s_t == T) {
          mma_commit(&bfree[pb]);  // this instance's centroid operand is no longer read
          s_t = 0;
          ++si;
        }
        if (++s_st == n_stages) {
          s_st = 0;
          ++s_round;
        }
        if (++s_ab == kDots) {
          s_ab = 0;
          ++s_use;
        }
        return true;
      };
      for (int g = 0; g < n_tiles; ++g)
        if (!screen()) break;
      mma_commit(&drain_bar[0]);
      drain_wait(&drain_bar[0], 0, a.err);
    }
    __syncwarp();
  } else if (warp == 2) {
    // ---------------------------------------------------------------- sum MMAs
    if (elect_one()) {
      const uint32_t idesc2 = idesc_bf16_f32(128, NBO) | (1u << 15);  // A is read across its rows
      const uint32_t stage0 = smem_u32(stage_smem);
      int m_st = 0;  // stage
      auto sum = [&](int g) -> bool {
        const int sb = g % kGroups, ub = g % kSums;
        if (!mbar_wait(&sumready[sb], (g / kGroups) & 1, abort_flag, a.err, kDevTimeoutMma)) return false;
        if (g >= kSums && !mbar_wait(&sumfree[ub], ((g / kSums) - 1) & 1, abort_flag, a.err, kDevTimeoutMma))
          return false;
        // passes on what the group wrote besides the operands; after the wait above, so that the barrier is
        // never two phases ahead of the warps that wait for it
        mbar_arrive(&cntready[ub]);
        tc_fence_after();
        const uint32_t d = tmem_sums + ub * (C::kParts * NBO);
        const uint32_t q_addr = stage0 + m_st * C::kStageBytes;
        const uint32_t s_addr = smem_u32(small_smem) + sb * C::kStageBytes;
        const uint32_t h_addr = smem_u32(hot_smem) + sb * C::kHotBytes;
        // A: 128 "rows" are the columns of d (d = 64: the tile's 64, then the second tile's 64)
        const uint32_t lbo = D == 128 ? kQBox : s_addr - q_addr;
        // the second tile's product first: its group waits for that buffer longest
#pragma unroll
        for (int p = C::kParts - 1; p >= 0; --p) {
#pragma unroll
          for (int kk = 0; kk < kQTile / 16; ++kk)
            mma_bf16_ss(d + p * NBO, sdesc_mnmajor_sw128((p ? s_addr : q_addr) + kk * 2048, lbo),
                        sdesc_kmajor_sw128(h_addr + (kk >> 2) * (NBO * 128) + (kk & 3) * 32), idesc2, kk > 0);
          if (p == C::kParts - 1) mma_commit(&smallfree[sb]);
        }
        mma_commit(&sumfull[ub]);
        mma_commit(&empty_bar[m_st]);  // the stage's queries are no longer read
        if (++m_st == n_stages) m_st = 0;
        return true;
      };
      for (int g = 0; g < n_tiles; ++g)
        if (!sum(g)) break;
      mma_commit(&drain_bar[1]);
      drain_wait(&drain_bar[1], 0, a.err);
    }
    __syncwarp();
  } else if (warp < kSumWarp0) {
    // ---------------------------------------------------------------- row groups: one query per thread
    const int sb = (warp - kGroupWarp0) >> 2;  // this group: tiles sb, sb + kGroups, ...
    const int quarter = warp & 3;        // TMEM lane quarter
    const uint32_t lane_addr = static_cast<uint32_t>(quarter * 32) << 16;
    const int n = quarter * 32 + lane;   // this thread's query in the tile
    const uint32_t swz = static_cast<uint32_t>(n & 7) << 4;
    unsigned char* small_row = small_smem + sb * C::kStageBytes + n * 128;
    unsigned char* hot = hot_smem + sb * C::kHotBytes + (n >> 6) * (NBO * 128) + ((n & 7) << 1);
    const uint32_t hot_chunk = static_cast<uint32_t>((n & 63) >> 3);
    int prev_b = -1;                     // beacon whose cell of the one-hot column is set
    int i = 0, t = sb;
    while (t >= T) {
      t -= T;
      ++i;
    }
    for (int g = sb; g < n_tiles; g += kGroups) {
      const int e = blockIdx.x + i * gridDim.x;
      const int st = g % n_stages, ab = g % kDots, slot = i & (kSlots - 1);
      const int rows = min(kQTile, nq - t * kQTile);
      // the tile's data and its dots (which also says that the screening has read the tile)
      bool ok = mbar_wait(&full_bar[st], (g / n_stages) & 1, abort_flag, a.err, kDevTimeoutEpilogue) &&
                mbar_wait(&accfull[ab], (g / kDots) & 1, abort_flag, a.err, kDevTimeoutEpilogue);
      if (!__all_sync(0xffffffffu, ok)) break;
      tc_fence_after();
      const int E = static_cast<signed char>(exp_sh[slot] & 0xff);
      const bool degenerate = (exp_sh[slot] & 0x100) != 0;
      const uint32_t vm = vmask_sh[slot];

      // ---- best and second best dot
      const uint32_t d = tmem + ab * ncols1 + lane_addr;
      float best = -INFINITY, second = -INFINITY;
      int bi = -1;
      for (int c0 = 0; c0 < nbp; c0 += 8) {
        float h[8], l[8];
        tmem_ld8(d + c0, h);
        tmem_ld8(d + nbp + c0, l);
        tmem_wait_ld();
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          const float dot = ((vm >> (c0 + u)) & 1u) ? h[u] + l[u] : -INFINITY;
          second = fmaxf(second, fminf(best, dot));
          if (dot > best) {
            best = dot;
            bi = c0 + u;
          }
        }
      }

      // this group's second tile is free once its previous tile's product is formed (the one-hot operand: below)
      ok = g < kGroups || mbar_wait(&smallfree[sb], ((g / kGroups) - 1) & 1, abort_flag, a.err, kDevTimeoutEpilogue);
      if (!__all_sync(0xffffffffu, ok)) break;

      // ---- the split of this query's elements and their extremes
      unsigned char* raw_row = stage_smem + st * C::kStageBytes + n * 128;
      uint32_t below = 0u;                 // bits of the elements below the operands' range
      uint32_t qmax = 0u;                  // its largest element's magnitude (bf16 bits; NaN above all)
      if (n < rows) {
        const __nv_bfloat162 lim = as_bf162(pow2_bf16x2(E - kLargeBits));
        const __nv_bfloat162 lim_lo = as_bf162(pow2_bf16x2(E - kSmallBits));
        __nv_bfloat162 mx[2] = {as_bf162(0u), as_bf162(0u)};
        // four chunks are loaded before the first store: a chunk at a time would wait out its latencies
        // (rolled in between: the roles of this kernel compete for the instruction caches)
#pragma unroll 1
        for (int c0 = 0; c0 < D / 8; c0 += 4) {
          unsigned char* box_raw = raw_row + (c0 >> 3) * kQBox;
          unsigned char* box_small = small_row + (c0 >> 3) * kQBox;
          uint4 v[4];
          uint32_t off[4];
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            off[c] = static_cast<uint32_t>(((c0 & 4) + c) << 4) ^ swz;
            v[c] = *reinterpret_cast<const uint4*>(box_raw + off[c]);
          }
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            const uint32_t w[4] = {v[c].x, v[c].y, v[c].z, v[c].w};
            uint32_t s[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
              const __nv_bfloat162 a2 = __habs2(as_bf162(w[k]));
              s[k] = w[k] & __hlt2_mask(a2, lim);
              below |= w[k] & __hlt2_mask(a2, lim_lo);
              mx[k & 1] = __hmax2_nan(mx[k & 1], a2);
            }
            *reinterpret_cast<uint4*>(box_small + off[c]) = make_uint4(s[0], s[1], s[2], s[3]);
            st_shared_v4_if((s[0] | s[1]) | (s[2] | s[3]), box_raw + off[c], w[0] ^ s[0], w[1] ^ s[1], w[2] ^ s[2],
                            w[3] ^ s[3]);
          }
        }
        const __nv_bfloat162 m2 = __hmax2_nan(mx[0], mx[1]);
        const uint32_t mw = *reinterpret_cast<const uint32_t*>(&m2);
        qmax = max(mw & 0xffffu, mw >> 16);
      } else {  // no query: nothing of a neighbour or of an earlier tile may enter the sums
        const uint4 z = make_uint4(0u, 0u, 0u, 0u);
        for (int c = 0; c < D / 8; ++c) {
          const uint32_t off = (c >> 3) * kQBox + (static_cast<uint32_t>((c & 7) << 4) ^ swz);
          *reinterpret_cast<uint4*>(raw_row + off) = z;
          *reinterpret_cast<uint4*>(small_row + off) = z;
        }
      }
      const bool special = qmax >= (pow2_bf16x2(E) & 0xffffu) || (below & 0x7fff7fffu) != 0u;
      {
        const uint32_t wmx = __reduce_max_sync(0xffffffffu, qmax < (pow2_bf16x2(kMaxE) & 0xffffu) ? qmax : 0u);
        if (lane == 0 && wmx > *reinterpret_cast<volatile uint32_t*>(&seen_sh)) atomicMax(&seen_sh, wmx);
      }

      // ---- decision
      // |q| <= sqrt(d) max|q_i| rules most queries out; where it does not, |q| is formed in fp32
      const float q_inf = __uint_as_float(qmax << 16);
      const bool wild = degenerate || !(q_inf >= kTameLo && q_inf < kTameHi);
      float margin = kScreenMargin * (D == 128 ? 11.313709f : 8.f) * q_inf;
      bool close = n < rows && vm != 0u && (wild || !(best - second > margin));
      if (__any_sync(0xffffffffu, close && !wild)) {
        margin = kScreenMargin * sqrtf(row_norm2<D>(raw_row, small_row, swz));
        close = close && (wild || !(best - second > margin));
      }
      int my_b = n < rows ? bi : -1;
      uint32_t need = __ballot_sync(0xffffffffu, close);
      if (need) {  // rare: which beacons may be the exact best, while the dots are still there
        uint32_t cand = vm;
        if (!__all_sync(0xffffffffu, !close || wild)) {
          const float floor_v = best - 2.f * margin;
          uint32_t m = 0u;
          for (int c0 = 0; c0 < nbp; c0 += 8) {
            float h[8], l[8];
            tmem_ld8(d + c0, h);
            tmem_ld8(d + nbp + c0, l);
            tmem_wait_ld();
#pragma unroll
            for (int u = 0; u < 8; ++u) m |= (h[u] + l[u] >= floor_v ? 1u : 0u) << (c0 + u);
          }
          if (!wild) cand = m & vm;
        }
        for (uint32_t m = need; m; m &= m - 1) {
          const int r = __ffs(m) - 1;
          __syncwarp();  // the rows' splits are written
          const int b = refine_row<D>(stage_smem + st * C::kStageBytes, small_smem + sb * C::kStageBytes, quarter * 32 + r,
                                      a.cent + static_cast<size_t>(e) * nb * D, __shfl_sync(0xffffffffu, cand, r));
          if (lane == r) my_b = b;
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&accfree[ab]);

      if (n < rows && a.assign_out) a.assign_out[static_cast<size_t>(e) * nq + t * kQTile + n] = my_b;
      add_counts<NBO>(add_cnt[slot], my_b);
      ok = g < kGroups || mbar_wait(&sumfull[(g - kGroups) % kSums], ((g - kGroups) / kSums) & 1, abort_flag, a.err,
                                    kDevTimeoutEpilogue);
      if (!__all_sync(0xffffffffu, ok)) break;
      // ---- this query's column of the one-hot operand: 2^(17 - E), which makes the large part's sums integers
      if (prev_b >= 0) *reinterpret_cast<uint16_t*>(hot + prev_b * 128 + ((hot_chunk ^ (prev_b & 7)) << 4)) = 0;
      if (my_b >= 0)
        *reinterpret_cast<uint16_t*>(hot + my_b * 128 + ((hot_chunk ^ (my_b & 7)) << 4)) =
            static_cast<uint16_t>(pow2_bf16x2(kLargeBits + 7 - E));
      prev_b = my_b;
      for (uint32_t m = __ballot_sync(0xffffffffu, special); m; m &= m - 1) {  // rare
        const int r = __ffs(m) - 1, b = __shfl_sync(0xffffffffu, my_b, r);
        const int si = i & (kSpillSlots - 1);
        __syncwarp();  // the rows' splits are written
        if (spill_row<D>(stage_smem + st * C::kStageBytes, small_smem + sb * C::kStageBytes, quarter * 32 + r, E, b,
                         &list_sh[si], a.spill + (static_cast<size_t>(blockIdx.x) * kSpillSlots + si) * nb * D))
          spilled_sh[slot] = 1;
      }
      fence_proxy_async_smem();  // this thread's operand writes, read next by the tensor cores
      __syncwarp();
      if (lane == 0) mbar_arrive(&sumready[sb]);
      t += kGroups;
      while (t >= T) {
        t -= T;
        ++i;
      }
    }
  } else if (warp < kBuildWarp0) {
    // ---------------------------------------------------------------- sums: a column of d and half of the beacons
    // per thread (two warps per TMEM lane quarter)
    constexpr int HB = NBO / 2;
    const int quarter = warp & 3;
    const int h0 = ((warp - kSumWarp0) >> 2) * HB;  // first beacon
    const uint32_t lane_addr = static_cast<uint32_t>(quarter * 32) << 16;
    const int col = quarter * 32 + lane;        // d = 64: 64 and more are the small parts of column col - 64
    const bool small_half = D == 64 && col >= 64;
    const bool first_warp = warp == kSumWarp0;
    for (int i = 0, g = 0; i < n_my; ++i) {
      const int e = blockIdx.x + i * gridDim.x, slot = i & (kSlots - 1);
      const size_t cells = static_cast<size_t>(nb) * D, cbase = static_cast<size_t>(e) * cells;
      // sums of the two operands, each below 2^24 per tile (d = 64: of one, by this thread's half); more than
      // kFlush tiles are passed on through the spill array
      constexpr int kFlush = 64;
      int acc_l[HB], acc_s[HB];
#pragma unroll
      for (int b = 0; b < HB; ++b) acc_l[b] = acc_s[b] = 0;
      bool ok = true;  // false after a wait gave up: the barriers below are still taken
      for (int t = 0; ok && t < T; ++t, ++g) {
        const int ub = g % kSums;
        ok = mbar_wait(&cntready[ub], (g / kSums) & 1, abort_flag, a.err, kDevTimeoutEpilogue) &&
             mbar_wait(&sumfull[ub], (g / kSums) & 1, abort_flag, a.err, kDevTimeoutEpilogue);
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
        tc_fence_after();
        const uint32_t d = tmem_sums + ub * (C::kParts * NBO) + lane_addr + h0;
        // large sums are integers (the one-hot operand's scale), small ones multiples of 2^-10
#pragma unroll
        for (int b0 = 0; b0 < HB; b0 += 8) {
          float v[C::kParts][8];
#pragma unroll
          for (int p = 0; p < C::kParts; ++p) tmem_ld8(d + p * NBO + b0, v[p]);
          tmem_wait_ld();
          if (b0 + 8 == HB) {
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&sumfree[ub]);
          }
#pragma unroll
          for (int b = 0; b < 8; ++b) {
            if constexpr (D == 128) {
              acc_l[b0 + b] += __float2int_rn(v[0][b]);
              acc_s[b0 + b] += __float2int_rn(v[C::kParts - 1][b] * 1024.f);
            } else {
              acc_l[b0 + b] += __float2int_rn(small_half ? v[0][b] * 1024.f : v[0][b]);
            }
          }
        }
        if (t + 1 < T && (t + 1) % kFlush == 0) {  // rare: more than 8192 queries per instance
          const int shift = static_cast<signed char>(exp_sh[slot] & 0xff) + 40 - (kSmallBits + 7);
          unsigned long long* sp =
              a.spill + (static_cast<size_t>(blockIdx.x) * kSpillSlots + (i & (kSpillSlots - 1))) * cells;
#pragma unroll
          for (int b = 0; b < HB; ++b) {
            const long long f = (D == 128 ? acc_l[b] * 1024ll + acc_s[b] : small_half ? acc_l[b] : acc_l[b] * 1024ll)
                                << shift;
            if (h0 + b < nb && f != 0)
              atomicAdd(sp + (h0 + b) * D + (small_half ? col - 64 : col), static_cast<unsigned long long>(f));
            acc_l[b] = acc_s[b] = 0;
          }
          spilled_sh[slot] = 1;
          __threadfence();
        }
      }
      if (T > kFlush) named_barrier(1, 256);  // what another warp passed on (d = 64) is there

      // ---- this instance's sums of the call, for the fold at the end
      const int add = lane < nb ? add_cnt[slot][lane] : 0;
      const int shift = static_cast<signed char>(exp_sh[slot] & 0xff) + 40 - (kSmallBits + 7);  // to units of 2^-40
      const bool spilled = spilled_sh[slot] != 0;
      const SpillList& list = list_sh[i & (kSpillSlots - 1)];
      const int n_list = min(list.n, kSpillList);
      unsigned long long* spill =
          a.spill + (static_cast<size_t>(blockIdx.x) * kSpillSlots + (i & (kSpillSlots - 1))) * cells;
      if constexpr (D == 64) {
        if (small_half)
#pragma unroll
          for (int b = 0; b < HB; ++b) xchg[(h0 + b) * 64 + col - 64] = acc_l[b];
        named_barrier(1, 256);
        if (!small_half)
#pragma unroll
          for (int b = 0; b < HB; ++b) acc_s[b] = xchg[(h0 + b) * 64 + col];
      }
      long long* out = a.call_sum + cbase + static_cast<size_t>(h0) * D + col;
      if (ok && !small_half) {
#pragma unroll
        for (int b = 0; b < HB; ++b)
          if (h0 + b < nb) out[b * D] = (acc_l[b] * 1024ll + acc_s[b]) << shift;
        for (int k = 0; k < n_list; ++k) {  // spilled elements of this thread's cells: rare
          const int b = (list.key[k] >> 8) - h0;
          if ((list.key[k] & 0xff) == col && b >= 0 && b < HB) out[b * D] += list.val[k];
        }
        if (spilled)
          for (int b = 0; b < HB && h0 + b < nb; ++b) {
            out[b * D] += static_cast<long long>(__ldcg(spill + (h0 + b) * D + col));
            spill[(h0 + b) * D + col] = 0ull;
          }
      }
      if (spilled) __threadfence();
      named_barrier(1, 256);  // every warp has read this slot's words (and, d = 64, the exchanged sums)
      if (ok && first_warp && lane < nb) a.call_cnt[static_cast<size_t>(e) * nb + lane] = add;
      if (first_warp) add_cnt[slot][lane] = 0;
      if (first_warp && lane == 0) {
        spilled_sh[slot] = 0;
        list_sh[i & (kSpillSlots - 1)].n = 0;
      }
    }
  } else {
    // ---------------------------------------------------------------- builders: the unit-centroid operand
    const int wk = warp - kBuildWarp0;  // 0 .. 3
    constexpr int kBatch = 1;
    for (int i = 0; i < n_my; ++i) {
      const int e = blockIdx.x + i * gridDim.x, pb = i & 1, slot = i & (kSlots - 1);
      if (wk == 0 && lane == 0 && i + 1 < n_my)
        bulk_prefetch_l2(a.cent + (static_cast<size_t>(e) + gridDim.x) * nb * D, static_cast<uint32_t>(nb * D) * 4);
      const long long cnt = lane < nb ? a.counts[static_cast<size_t>(e) * nb + lane] : 0;
      const uint32_t counted = __ballot_sync(0xffffffffu, cnt > 0);
      if (i >= 2) mbar_wait(&bfree[pb], ((i >> 1) - 1) & 1, abort_flag, a.err, kDevTimeoutEpilogue);
      unsigned char* bm = bmat + pb * C::bmat_bytes(nbp);
      uint32_t valid = 0u;
      float cmax = 0.f;
      bool extreme = false;
#pragma unroll 1
      for (int b0 = wk; b0 < nbp; b0 += 4 * kBatch) {
        float c[kBatch][D / 32];
#pragma unroll
        for (int u = 0; u < kBatch; ++u)
#pragma unroll
          for (int k = 0; k < D / 32; ++k)
            c[u][k] = b0 + 4 * u < nb ? a.cent[(static_cast<size_t>(e) * nb + b0 + 4 * u) * D + lane + 32 * k] : 0.f;
#pragma unroll
        for (int u = 0; u < kBatch; ++u) {
          const int b = b0 + 4 * u;
          if (b >= nbp) break;
          float n2 = 0.f;
#pragma unroll
          for (int k = 0; k < D / 32; ++k) n2 = fmaf(c[u][k], c[u][k], n2);
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) n2 += __shfl_xor_sync(0xffffffffu, n2, o);
          bool nz = false;
#pragma unroll
          for (int k = 0; k < D / 32; ++k) nz |= c[u][k] != 0.f;
          const bool ok = ((counted >> (b & 31)) & 1u) && b < nb && __any_sync(0xffffffffu, nz);
          if (ok) {
            valid |= 1u << b;
            cmax = fmaxf(cmax, n2);
            extreme |= !(n2 > 1e-30f && n2 < 1e30f);
          }
          const float inv = ok ? rsqrtf(n2) : 0.f;
#pragma unroll
          for (int k = 0; k < D / 32; ++k) {
            const int col = lane + 32 * k;
            const float x = c[u][k] * inv;
            const __nv_bfloat16 hi = __float2bfloat16_rn(x);
            const __nv_bfloat16 lo = __float2bfloat16_rn(x - __bfloat162float(hi));
            *reinterpret_cast<__nv_bfloat16*>(bm + sw128_offset(b, col, bbox)) = hi;
            *reinterpret_cast<__nv_bfloat16*>(bm + sw128_offset(nbp + b, col, bbox)) = lo;
          }
        }
      }
      if (lane == 0) {
        kv_sh[wk] = valid;
        km_sh[wk] = (__float_as_uint(cmax) & 0x7fffffffu) | (extreme ? 0x80000000u : 0u);
      }
      fence_proxy_async_smem();  // generic-proxy writes, read next by the tensor cores
      named_barrier(2, 128);
      if (wk == 0 && lane == 0) {
        uint32_t v = 0u, m = 0u, x = 0u;
        for (int w = 0; w < 4; ++w) {
          v |= kv_sh[w];
          m = max(m, km_sh[w] & 0x7fffffffu);
          x |= km_sh[w] >> 31;
        }
        // every element seen is below 2^E; before that a guess from the largest centroid's norm
        const uint32_t seen = *reinterpret_cast<volatile uint32_t*>(&seen_sh);
        int E = seen ? static_cast<int>(seen >> 7) - 126 : ((static_cast<int>(m >> 23) - 127) >> 1) + 2;
        E = E < kMinE ? kMinE : E > kMaxE ? kMaxE : E;
        vmask_sh[slot] = v;
        exp_sh[slot] = (E & 0xff) | (x ? 0x100 : 0);
        mbar_arrive(&bready[pb]);
      }
      named_barrier(2, 128);  // kv_sh and km_sh are free again
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, 512);
  }
  if (*abort_flag) return;  // a wait gave up: some sums are missing

  // ---- this CTA's instances: the call's sums into the running state, a warp per (instance, beacon).  After
  // the tiles, not as a role beside them: there its instructions kept the other roles waiting for theirs
  // (4608 instances of 8 beacons 298 -> 255 us, 8192 of 16 537 -> 485 us by taking it out).  What bounds it:
  // 28 bytes and about 130 instructions per cell.
  constexpr int kCells = D / 32;
  for (int unit = warp; unit < n_my * nb; unit += kUThreads / 32) {
    const int i = unit / nb, b = unit - i * nb;
    const size_t row = (static_cast<size_t>(blockIdx.x) + static_cast<size_t>(i) * gridDim.x) * nb + b;
    const int add = __ldcg(a.call_cnt + row);
    if (add == 0) continue;  // warp-uniform
    const size_t base = row * D + lane;
    double s_old[kCells], s_new[kCells];
    long long f[kCells];
    float c_new[kCells];
#pragma unroll
    for (int k = 0; k < kCells; ++k) {
      s_old[k] = a.sums[base + 32 * k];
      f[k] = __ldcg(a.call_sum + base + 32 * k);
    }
    const long long n = a.counts[row] + add;
    const DF rcp = count_reciprocal(n);
    bool plain = true;
#pragma unroll
    for (int k = 0; k < kCells; ++k) plain &= fold_and_centroid(s_old[k], f[k], rcp, s_new[k], c_new[k]);
    if (!plain) {  // a sum off the 2^-40 grid, past 2^22 or zero
#pragma unroll
      for (int k = 0; k < kCells; ++k) {
        s_new[k] = fold_sum(s_old[k], f[k]);
        c_new[k] = centroid_value(s_new[k], rcp);
      }
    }
#pragma unroll
    for (int k = 0; k < kCells; ++k) {
      a.sums[base + 32 * k] = s_new[k];
      a.cent[base + 32 * k] = c_new[k];
    }
    __syncwarp();  // every lane has read the count
    if (lane == 0) a.counts[row] = n;
  }
}

template <int D, int NBO>
cudaError_t launch_update_dn(const UpdArgs& a, const CUtensorMap& qmap, int grid, cudaStream_t st) {
  using C = UpdCfg<D, NBO>;
  const size_t smem = C::smem_bytes(a.nbp);
  const cudaError_t e = allow_smem<update_kernel<D, NBO>>(smem);
  if (e != cudaSuccess) return e;
  return launch_dependent(update_kernel<D, NBO>, static_cast<unsigned>(grid), kUThreads, smem, st, qmap, a,
                          C::stages(a.nbp));
}

}  // namespace

size_t update_spill_words(const Shape& s, int grid) {
  return static_cast<size_t>(grid) * kSpillSlots * s.nb * s.d;
}

// the call's sums, then its counts
size_t update_call_bytes(const Shape& s) {
  const size_t inst = static_cast<size_t>(s.n_inst) * s.nb;
  return inst * s.d * sizeof(long long) + inst * sizeof(int);
}

cudaError_t launch_update(const Shape& s, const CUtensorMap& qmap, int box_rows, int n_new, int grid, float* cent,
                          double* sums, long long* counts, int* assign_out, unsigned long long* spill, void* call, int* err,
                          cudaStream_t st) {
  UpdArgs a;
  a.n_inst = s.n_inst;
  a.nq = s.G * n_new;
  a.box_rows = box_rows;
  a.nb = s.nb;
  a.nbp = (s.nb + 7) / 8 * 8;
  a.cent = cent;
  a.sums = sums;
  a.counts = counts;
  a.assign_out = assign_out;
  a.spill = spill;
  a.call_sum = static_cast<long long*>(call);
  a.call_cnt = reinterpret_cast<int*>(a.call_sum + static_cast<size_t>(s.n_inst) * s.nb * s.d);
  a.err = err;
  if (s.d == 128)
    return s.nb <= 16 ? launch_update_dn<128, 16>(a, qmap, grid, st) : launch_update_dn<128, 32>(a, qmap, grid, st);
  return s.nb <= 16 ? launch_update_dn<64, 16>(a, qmap, grid, st) : launch_update_dn<64, 32>(a, qmap, grid, st);
}

}  // namespace bkv
