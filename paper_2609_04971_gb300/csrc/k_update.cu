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
// instances of 512 queries, call and state read: 527 us, some 40 less than with an
// fp32 sum for every query).  Zero queries and instances without a valid beacon give -1.
//
// Sums: Q^T x A, where A is the tile's one-hot assignment matrix (128 queries x
// beacons), exact: an element x with |x| < 2^E (E chosen per instance) goes
// whole into one of two operands, the tile itself (|x| >= 2^(E-10), a multiple
// of 2^(E-17)) or a second tile (smaller ones, multiples of 2^(E-27) for
// |x| >= 2^(E-20)), whose sums over 128 rows stay below 2^24 grid steps, so no
// addition needs rounding (that the tensor cores then add without loss is not
// documented: the tests hold it, with sums up to the limit).  The two sums of a (column, beacon) cell are
// integers, added up over the tiles in two registers.  Elements outside
// [2^(E-20), 2^E) (one in fifteen tiles of data of one scale has some) are zeroed in
// the operands and added one by one, from a list in shared memory (past its end
// through a global array of this CTA).  E follows the instance's largest centroid
// element and how far the queries of the last instances exceeded theirs; it is never
// below -11, so that what the operands hold is exact in fixed point with 40
// fractional bits, and the result does not depend on it.
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
// so loops are kept rolled and rare paths small, out of line and few.  Sums formed in
// fp32 parts by CUDA cores from rows sorted by beacon took about 14 K warp
// instructions per tile, whatever the data.  Kernel times, with those in brackets:
// 4608 instances x 512 queries of 128, 8 beacons 219 us (380; 95 at the copy rate),
// 8192 instances, 16 beacons 446 (761; 178).  Data of many scales spills in every
// tile, 4608 instances: one query of 1000 times the scale in each CTA's first 266
// (380), five columns of 300 times the rest 449 (414), elements spread by exp(1.5 N)
// 579 (381), queries so spread 595 (380), elements over 24 octaves 1430 (389).
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
constexpr int kSpillListMin = 128;          // spilled elements per instance kept in shared memory, at least
constexpr int kSpillListMax = 1024;         // and at most
constexpr int kFewRows = 2;                 // rows of a warp with spilled elements that are taken one by one
constexpr size_t kUSmemBudget = 223 * 1024;
// A query is re-decided exactly when its best and second-best dots differ by at most this fraction of |q|.
// A screened dot is within 2^-18 |q| (the hi / lo split) + 136 * 2^-23 |q| (17 additions in each of eight
// K = 16 steps) + 2^-21 |q| (1 / |c|) of the exact one, so a difference of two within 4.2e-5 |q|.
constexpr float kScreenMargin = 7e-5f;
// Queries whose largest element is in this range have a squared norm that fp32 holds (1e-30 < |q|^2 < 1e30).
constexpr float kTameLo = 1.7763568394002505e-15f, kTameHi = 70368744177664.f;  // 2^-49, 2^46
constexpr int kMinE = -11, kMaxE = 14;
constexpr int kRecent = 12;                 // instances before the one being built whose slots are still their own
constexpr int kFirstRise = 64;              // rise of the queries above the centroids before any is seen: half an octave
constexpr int kHeadroom = 32;               // and a quarter of one more (both in 1/128 octave)
constexpr int kLargeBits = 10;              // octaves below 2^E that the tile itself holds
constexpr int kSmallBits = 20;              // octaves below 2^E that the operands hold

struct UpdArgs {
  int n_inst, nq, nb, nbp;  // instances, queries per instance, beacons, beacons padded to 8
  int box_rows;             // rows of one TMA box of queries (<= 128)
  int list_cap;             // entries of an instance's list of spilled elements
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
    const int n =
        static_cast<int>((kUSmemBudget - 1024 - fixed_bytes(nbp) - kSpillSlots * kSpillListMin * 4) / kStageBytes);
    return n < kUMaxStages ? n : kUMaxStages;
  }
  static size_t smem_but_lists(int nbp) {
    return 1024 + static_cast<size_t>(stages(nbp)) * kStageBytes + fixed_bytes(nbp);
  }
  // what the stages leave goes to the lists of spilled elements
  static int list_cap(int nbp) {
    const int n = static_cast<int>((kUSmemBudget - smem_but_lists(nbp)) / (kSpillSlots * 4));
    return n < kSpillListMax ? n : kSpillListMax;
  }
  static size_t smem_bytes(int nbp) { return smem_but_lists(nbp) + static_cast<size_t>(list_cap(nbp)) * kSpillSlots * 4; }
};

// mbar_wait whose waiting loop is out of line: there are some twenty waits in the roles, which share the
// instruction caches (235 -> 230 us, 4608 instances of 512 queries).
__device__ __noinline__ bool wait_on(uint64_t* bar, uint32_t parity, volatile int* abort, int* err, int code) {
  return mbar_wait(bar, parity, abort, err, code);
}
__device__ __forceinline__ bool wait_for(uint64_t* bar, uint32_t parity, volatile int* abort, int* err, int code) {
  return mbar_try_wait(bar, parity) || wait_on(bar, parity, abort, err, code);
}

__device__ __forceinline__ void drain_wait(uint64_t* bar, uint32_t parity, int* err) {
  int never = 0;
  wait_for(bar, parity, &never, err, kDevTimeoutDrain);
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

// A spilled element (bf16 bits in the upper half) in fixed point.
__device__ __forceinline__ long long spilled_fixed40(uint32_t hi16) {
  const float x = __uint_as_float(hi16);
  return fabsf(x) < 16384.f ? fixed40_one(x) : bf16_fixed40(hi16);
}

// Elements that the operands cannot hold: 0 < |x| < 2^(E - 20), |x| >= 2^E and what is not finite.  All sit in
// the tile.  Each is zeroed there and noted for the row's beacon (b < 0: the row is not assigned) in the
// instance's list, as (element << 16 | beacon << 8 | column), or, past its end, added to the global array.
// Both functions are warp-wide, out of line and small, as rare code is fetched cold (2 - 3 K clocks a call); they
// return whether something was added to the global array.

// Where a CTA's spilled elements go (in shared memory: each argument that a call needs in a register cost the
// loops around it 2 %).
struct SpillTo {
  int* list_n;
  uint32_t* list;
  unsigned long long* spill;
  int list_cap, cells;
};

// spill_row: one row (n of the tile), a lane per column.  Data of one scale has one such row in a few tiles.
template <int D>
__device__ __noinline__ bool spill_row(unsigned char* raw, int n, int E, int b, int si, const SpillTo& to) {
  int* list_n = to.list_n + si;
  const int list_cap = to.list_cap;
  uint32_t* list = to.list + si * list_cap;
  unsigned long long* spill = to.spill + static_cast<size_t>(si) * to.cells;
  const uint32_t hi = pow2_bf16x2(E) & 0xffffu, lo = pow2_bf16x2(E - kSmallBits) & 0xffffu;
  bool over = false;
#pragma unroll 1
  for (int col = threadIdx.x & 31; col < D; col += 32) {
    uint16_t* at_x = reinterpret_cast<uint16_t*>(raw + sw128_offset(n, col, kQBox));
    const uint32_t w = *at_x, m = w & 0x7fffu;
    if (m == 0u || (m >= lo && m < hi)) continue;
    *at_x = 0;
    if (b < 0) continue;
    int at = *reinterpret_cast<volatile int*>(list_n);
    if (at < list_cap) at = atomicAdd(list_n, 1);  // a full list's length is left alone: it stays far from overflow
    if (at < list_cap) {
      list[at] = w << 16 | static_cast<uint32_t>(b << 8 | col);
    } else {
      atomicAdd(spill + b * D + col, static_cast<unsigned long long>(spilled_fixed40(w << 16)));
      over = true;
    }
  }
  if (!__any_sync(0xffffffffu, over)) return false;
  __threadfence();
  return true;
}

// spill_rows: each lane's own row (`mine`: it has some), for data of many scales, where every row has some.  The
// lanes work side by side: first each marks its row's elements (one bit each), then all take their next marked
// one at a time.
template <int D>
__device__ __noinline__ bool spill_rows(unsigned char* raw_row, uint32_t swz, int E, int b, bool mine, int si,
                                        const SpillTo& to) {
  int* list_n = to.list_n + si;
  const int list_cap = to.list_cap;
  uint32_t* list = to.list + si * list_cap;
  unsigned long long* spill = to.spill + static_cast<size_t>(si) * to.cells;
  constexpr uint32_t kAll = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  // added to |x|, these put |x| >= 2^(E - 20) and |x| >= 2^E into bit 15
  const uint32_t to_lo = 0x80008000u - pow2_bf16x2(E - kSmallBits), to_hi = 0x80008000u - pow2_bf16x2(E);
  uint32_t m[D / 32];
#pragma unroll
  for (int g = 0; g < D / 32; ++g) m[g] = 0u;
#pragma unroll 1
  for (int c = 0; c < D / 8; ++c) {
    const uint32_t off = (c >> 3) * kQBox + (static_cast<uint32_t>((c & 7) << 4) ^ swz);
    const uint4 v = *reinterpret_cast<const uint4*>(raw_row + off);
    const uint32_t w[4] = {v.x & 0x7fff7fffu, v.y & 0x7fff7fffu, v.z & 0x7fff7fffu, v.w & 0x7fff7fffu};
    uint32_t bits = 0u;  // element 2k at bit 2k, element 2k + 1 at bit 16 + 2k
#pragma unroll
    for (int k = 0; k < 4; ++k)
      bits |= ((((w[k] + 0x7fff7fffu) & ~(w[k] + to_lo)) | (w[k] + to_hi)) & 0x80008000u) >> (15 - 2 * k);
    bits = mine ? (bits & 0x55u) | ((bits >> 15) & 0xaau) : 0u;
#pragma unroll
    for (int g = 0; g + 1 < D / 32; ++g) m[g] = __funnelshift_r(m[g], m[g + 1], 8);
    m[D / 32 - 1] = (m[D / 32 - 1] >> 8) | (bits << 24);
  }
  // room for all of them at once
  uint32_t count = 0u;
#pragma unroll
  for (int g = 0; g < D / 32; ++g) count += b >= 0 ? __popc(m[g]) : 0u;
  uint32_t at = count;  // becomes the number of elements of this lane and those before it
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t u = __shfl_up_sync(kAll, at, o);
    at += lane >= o ? u : 0u;
  }
  int base = 0;
  if (lane == 31) {  // a full list's length is left alone: it stays far from overflow
    base = *reinterpret_cast<volatile int*>(list_n);
    if (base < list_cap) base = atomicAdd(list_n, static_cast<int>(at));
  }
  at += static_cast<uint32_t>(__shfl_sync(kAll, base, 31)) - count;
  bool over = false;
#pragma unroll 1
  while (__any_sync(kAll, (D == 128 ? m[0] | m[1] | m[D / 32 - 2] | m[D / 32 - 1] : m[0] | m[1]) != 0u)) {
    int g = 0;
    uint32_t cur = m[0];
#pragma unroll
    for (int k = 1; k < D / 32; ++k)
      if (cur == 0u) {
        cur = m[k];
        g = k;
      }
    if (cur != 0u) {
      const int col = 32 * g + __ffs(cur) - 1;
#pragma unroll
      for (int k = 0; k < D / 32; ++k) m[k] = k == g ? cur & (cur - 1u) : m[k];
      const uint32_t off = (col >> 6) * kQBox + ((static_cast<uint32_t>(col & 0x38) << 1) ^ swz) + ((col & 7) << 1);
      uint16_t* at_x = reinterpret_cast<uint16_t*>(raw_row + off);
      const uint32_t w = static_cast<uint32_t>(*at_x) << 16;
      *at_x = 0;
      if (b >= 0) {
        if (at < static_cast<uint32_t>(list_cap)) {
          list[at] = w | static_cast<uint32_t>(b << 8 | col);
        } else {
          atomicAdd(spill + b * D + col, static_cast<unsigned long long>(spilled_fixed40(w)));
          over = true;
        }
        ++at;
      }
    }
  }
  if (!__any_sync(kAll, over)) return false;
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
  // per instance in flight
  __shared__ uint32_t vmask_sh[kSlots];      // valid beacons (count > 0, nonzero centroid)
  __shared__ uint32_t seen_sh[kSlots];       // largest query element below 2^kMaxE seen so far (bf16 bits)
  __shared__ int cmax_sh[kSlots];            // largest centroid element (bf16 bits; 0: no valid beacon)
  __shared__ int exp_sh[kSlots];             // E; bit 8: a centroid norm is extreme, every query is re-decided
  __shared__ int add_cnt[kSlots][kMaxBeacons];  // queries assigned so far
  __shared__ int spilled_sh[kSlots];         // elements or sums went to the global array
  __shared__ SpillTo spill_to;
  __shared__ int list_n_sh[kSpillSlots];     // spilled elements so far (those past the list's end are elsewhere)
  __shared__ uint32_t kv_sh[4];              // builders: each warp's valid beacons
  __shared__ uint32_t km_sh[4];              // builders: each warp's largest centroid element (fp32 bits), bit 31: extreme norm

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
  uint32_t* list_smem = reinterpret_cast<uint32_t*>(reinterpret_cast<unsigned char*>(xchg) + C::kXchg);  // [kSpillSlots][list_cap]

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
    fence_mbar_init();
  }
  for (uint32_t i = threadIdx.x; i < kGroups * C::kHotBytes / 16; i += kUThreads)
    reinterpret_cast<uint4*>(hot_smem)[i] = make_uint4(0u, 0u, 0u, 0u);
  for (int i = threadIdx.x; i < kSlots * kMaxBeacons; i += kUThreads) (&add_cnt[0][0])[i] = 0;
  if (threadIdx.x < kSlots) spilled_sh[threadIdx.x] = 0;
  if (threadIdx.x < kSpillSlots) list_n_sh[threadIdx.x] = 0;
  if (threadIdx.x == 0) spill_to = SpillTo{list_n_sh, list_smem, a.spill + static_cast<size_t>(blockIdx.x) * kSpillSlots * nb * D, a.list_cap, nb * D};
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
          if (round > 0 && !wait_for(&empty_bar[st], (round - 1) & 1, abort_flag, a.err, kDevTimeoutProducer)) {
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
        if (s_t == 0 && !wait_for(&bready[pb], (si >> 1) & 1, abort_flag, a.err, kDevTimeoutMma)) return false;
        if (!wait_for(&full_bar[s_st], s_round & 1, abort_flag, a.err, kDevTimeoutMma)) return false;
        if (s_use > 0 && !wait_for(&accfree[s_ab], (s_use - 1) & 1, abort_flag, a.err, kDevTimeoutMma)) return false;
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
        if (!wait_for(&sumready[sb], (g / kGroups) & 1, abort_flag, a.err, kDevTimeoutMma)) return false;
        if (g >= kSums && !wait_for(&sumfree[ub], ((g / kSums) - 1) & 1, abort_flag, a.err, kDevTimeoutMma))
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
      bool ok = wait_for(&full_bar[st], (g / n_stages) & 1, abort_flag, a.err, kDevTimeoutEpilogue) &&
                wait_for(&accfull[ab], (g / kDots) & 1, abort_flag, a.err, kDevTimeoutEpilogue);
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
      ok = g < kGroups || wait_for(&smallfree[sb], ((g / kGroups) - 1) & 1, abort_flag, a.err, kDevTimeoutEpilogue);
      if (!__all_sync(0xffffffffu, ok)) break;

      // ---- the split of this query's elements and their extremes
      unsigned char* raw_row = stage_smem + st * C::kStageBytes + n * 128;
      uint32_t below = 0u;                 // bits of the elements below the operands' range
      uint32_t qmax = 0u;                  // its largest element's magnitude (bf16 bits; NaN above all)
      if (n < rows) {
        // 2^(E - 20) <= |x| < 2^(E - 10) goes to the second tile, what is below stays
        const __nv_bfloat162 hi = as_bf162(pow2_bf16x2(E - kLargeBits)), lo = as_bf162(pow2_bf16x2(E - kSmallBits));
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
              const uint32_t under = __hlt2_mask(a2, lo);
              s[k] = w[k] & __hlt2_mask(a2, hi) & ~under;
              below |= w[k] & under;
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
      const bool special = vm != 0u && ((below & 0x7fff7fffu) != 0u || qmax >= (pow2_bf16x2(E) & 0xffffu));
      {
        const uint32_t wmx = __reduce_max_sync(0xffffffffu, qmax < (pow2_bf16x2(kMaxE) & 0xffffu) ? qmax : 0u);
        if (lane == 0 && wmx > *reinterpret_cast<volatile uint32_t*>(&seen_sh[slot])) atomicMax(&seen_sh[slot], wmx);
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
      ok = g < kGroups || wait_for(&sumfull[(g - kGroups) % kSums], ((g - kGroups) / kSums) & 1, abort_flag, a.err,
                                    kDevTimeoutEpilogue);
      if (!__all_sync(0xffffffffu, ok)) break;
      // ---- this query's column of the one-hot operand: 2^(17 - E), which makes the large part's sums integers
      if (prev_b >= 0) *reinterpret_cast<uint16_t*>(hot + prev_b * 128 + ((hot_chunk ^ (prev_b & 7)) << 4)) = 0;
      if (my_b >= 0)
        *reinterpret_cast<uint16_t*>(hot + my_b * 128 + ((hot_chunk ^ (my_b & 7)) << 4)) =
            static_cast<uint16_t>(pow2_bf16x2(kLargeBits + 7 - E));
      prev_b = my_b;
      const uint32_t specials = __ballot_sync(0xffffffffu, special);
      if (specials != 0u) {  // rare on data of one scale
        const int si = i & (kSpillSlots - 1);
        bool over = false;
        if (__popc(specials) <= kFewRows) {
          for (uint32_t m = specials; m; m &= m - 1) {
            const int r = __ffs(m) - 1, b = __shfl_sync(0xffffffffu, my_b, r);
            __syncwarp();  // the rows' splits are written
            over |= spill_row<D>(stage_smem + st * C::kStageBytes, quarter * 32 + r, E, b, si, spill_to);
          }
        } else {
          over = spill_rows<D>(raw_row, swz, E, my_b, special, si, spill_to);
        }
        if (over) spilled_sh[slot] = 1;
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
        ok = wait_for(&cntready[ub], (g / kSums) & 1, abort_flag, a.err, kDevTimeoutEpilogue) &&
             wait_for(&sumfull[ub], (g / kSums) & 1, abort_flag, a.err, kDevTimeoutEpilogue);
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
      const uint32_t* list = list_smem + (i & (kSpillSlots - 1)) * a.list_cap;
      const int n_list = min(list_n_sh[i & (kSpillSlots - 1)], a.list_cap);
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
        long long f[HB];
#pragma unroll
        for (int b = 0; b < HB; ++b) f[b] = (acc_l[b] * 1024ll + acc_s[b]) << shift;
        for (int k = 0; k < n_list; k += 32) {  // rare: spilled elements, a lane each; then those of this warp's cells
          const uint32_t key = k + lane < n_list ? list[k + lane] : 0xffffu;
          const int at = static_cast<int>(key & 0xffffu);  // (beacon, column)
          const long long v = spilled_fixed40(key & 0xffff0000u);
          uint32_t m = __ballot_sync(0xffffffffu, (at & 0xff) >> 5 == quarter && at >> 8 >= h0 && at >> 8 < h0 + HB);
          for (; m; m &= m - 1) {
            const int src = __ffs(m) - 1;
            const int one = __shfl_sync(0xffffffffu, at, src);
            const long long v1 = __shfl_sync(0xffffffffu, v, src);
            const int b1 = (one & 31) == lane ? (one >> 8) - h0 : -1;
#pragma unroll
            for (int b = 0; b < HB; ++b)
              if (b == b1) f[b] += v1;
          }
        }
        if (spilled)
#pragma unroll
          for (int b = 0; b < HB; ++b)
            if (h0 + b < nb) {
              f[b] += static_cast<long long>(__ldcg(spill + (h0 + b) * D + col));
              spill[(h0 + b) * D + col] = 0ull;
            }
#pragma unroll
        for (int b = 0; b < HB; ++b)
          if (h0 + b < nb) out[b * D] = f[b];
      }
      if (spilled) __threadfence();
      named_barrier(1, 256);  // every warp has read this slot's words (and, d = 64, the exchanged sums)
      if (ok && first_warp && lane < nb) a.call_cnt[static_cast<size_t>(e) * nb + lane] = add;
      if (first_warp) add_cnt[slot][lane] = 0;
      if (first_warp && lane == 0) {
        spilled_sh[slot] = 0;
        list_n_sh[i & (kSpillSlots - 1)] = 0;
      }
    }
  } else {
    // ---------------------------------------------------------------- builders: the unit-centroid operand
    const int wk = warp - kBuildWarp0;  // 0 .. 3
    for (int i = 0; i < n_my; ++i) {
      const int e = blockIdx.x + i * gridDim.x, pb = i & 1, slot = i & (kSlots - 1);
      if (wk == 0 && lane == 0 && i + 1 < n_my)
        bulk_prefetch_l2(a.cent + (static_cast<size_t>(e) + gridDim.x) * nb * D, static_cast<uint32_t>(nb * D) * 4);
      const long long cnt = lane < nb ? a.counts[static_cast<size_t>(e) * nb + lane] : 0;
      const uint32_t counted = __ballot_sync(0xffffffffu, cnt > 0);
      if (i >= 2) wait_for(&bfree[pb], ((i >> 1) - 1) & 1, abort_flag, a.err, kDevTimeoutEpilogue);
      unsigned char* bm = bmat + pb * C::bmat_bytes(nbp);
      uint32_t valid = 0u;
      uint32_t cmax = 0u;
      bool extreme = false;
#pragma unroll 1
      for (int b = wk; b < nbp; b += 4) {
        float c[D / 32];
#pragma unroll
        for (int k = 0; k < D / 32; ++k)
          c[k] = b < nb ? a.cent[(static_cast<size_t>(e) * nb + b) * D + lane + 32 * k] : 0.f;
        float n2 = 0.f;
#pragma unroll
        for (int k = 0; k < D / 32; ++k) n2 = fmaf(c[k], c[k], n2);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) n2 += __shfl_xor_sync(0xffffffffu, n2, o);
        float big = 0.f;
#pragma unroll
        for (int k = 0; k < D / 32; ++k) big = fmaxf(big, fabsf(c[k]));
        const bool ok = ((counted >> (b & 31)) & 1u) && b < nb && __any_sync(0xffffffffu, big != 0.f || n2 != n2);
        if (ok) {
          valid |= 1u << b;
          cmax = max(cmax, __float_as_uint(big));
          extreme |= !(n2 > 1e-30f && n2 < 1e30f);
        }
        const float inv = ok ? rsqrtf(n2) : 0.f;
#pragma unroll
        for (int k = 0; k < D / 32; ++k) {
          const int col = lane + 32 * k;
          const float x = c[k] * inv;
          const __nv_bfloat16 hi = __float2bfloat16_rn(x);
          const __nv_bfloat16 lo = __float2bfloat16_rn(x - __bfloat162float(hi));
          *reinterpret_cast<__nv_bfloat16*>(bm + sw128_offset(b, col, bbox)) = hi;
          *reinterpret_cast<__nv_bfloat16*>(bm + sw128_offset(nbp + b, col, bbox)) = lo;
        }
      }
      cmax = __reduce_max_sync(0xffffffffu, cmax);
      if (lane == 0) {
        kv_sh[wk] = valid;
        km_sh[wk] = cmax | (extreme ? 0x80000000u : 0u);
      }
      fence_proxy_async_smem();  // generic-proxy writes, read next by the tensor cores
      named_barrier(2, 128);
      if (wk == 0) {
        uint32_t v = 0u, m = 0u, x = 0u;
        for (int w = 0; w < 4; ++w) {
          v |= kv_sh[w];
          m = max(m, km_sh[w] & 0x7fffffffu);
          x |= km_sh[w] >> 31;
        }
        // E: what the instance's largest centroid element is times what the queries' elements exceeded theirs
        // by in the last three instances with some (kFirstRise before that), and kHeadroom.  Scales differ by
        // head and layer, so neither a fixed E nor the largest element so far would serve: one query of 1000
        // times the scale raised E, and with it the number of spilled elements, for all that followed (3 times
        // the time).  bf16 bits are used as logarithms, in 1/128 octave.
        const int back = i - 1 - lane;  // the slots of the last instances, all of them written
        int rise = 0;
        bool some = false;
        if (lane < kRecent && back >= 0) {
          const int seen = static_cast<int>(*reinterpret_cast<volatile uint32_t*>(&seen_sh[back & (kSlots - 1)]));
          const int c0 = *reinterpret_cast<volatile int*>(&cmax_sh[back & (kSlots - 1)]);
          rise = seen - c0;
          some = seen != 0 && c0 != 0;
        }
        const uint32_t with = __ballot_sync(0xffffffffu, some);
        const bool taken = some && __popc(with & ((1u << lane) - 1u)) < 3;
        rise = __reduce_max_sync(0xffffffffu, taken ? rise : -(1 << 16));
        if (lane == 0) {
          const int c0 = static_cast<int>(m >> 16);
          int E = ((c0 + (with ? rise : kFirstRise) + kHeadroom) >> 7) - 126;
          E = E < kMinE ? kMinE : E > kMaxE ? kMaxE : E;
          vmask_sh[slot] = v;
          exp_sh[slot] = (E & 0xff) | (x ? 0x100 : 0);
          seen_sh[slot] = 0u;
          cmax_sh[slot] = v ? c0 : 0;
          mbar_arrive(&bready[pb]);
        }
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
cudaError_t launch_update_dn(UpdArgs a, const CUtensorMap& qmap, int grid, cudaStream_t st) {
  using C = UpdCfg<D, NBO>;
  a.list_cap = C::list_cap(a.nbp);
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
