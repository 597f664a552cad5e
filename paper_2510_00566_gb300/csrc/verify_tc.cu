// BF16 storage + tensor-core level-wise verification (Eq. 2-3, Algorithm 1)
// for sm_103a.
//
// Index layout (precision PANO_BF16): chunks of 128 vectors; the level-l
// slice of a chunk is a 128 x w_l bf16 tile stored exactly as the swizzled
// K-major shared-memory image a tcgen05.mma operand needs (see tcgen05.cuh),
// so one bulk-async copy stages a whole level slice and one 32/64/128-byte
// copy stages a single row.  Widths are 16, 32 or multiples of 64.  The tail
// norms, norms and error bounds are those of the dequantised vector
// x^ = bf16(x~), with e_x bounding ||x^ - T~(x - mu~)||.
//
// Work item: (list, segment of <= 4 chunks, group of <= 64 queries).  The CTA
// walks the segment level by level (the paper's batch).  Per (chunk, level)
// the partial products of all 128 candidates x the group's queries are one
// MMA chain: A = level tile of the chunk, B = the queries' level slices split
// into bf16 hi + lo parts (two MMAs into the same accumulator), accumulated
// across levels in tensor memory (4 chunks x 64 columns = 256 TMEM columns;
// two CTAs share an SM).  The margined Eq. 3 test in its separable form (three
// FMAs and a compare per (candidate, query) pair) runs at the levels of the
// bound-test schedule; a chunk whose rows are all dead is neither copied nor
// multiplied again.
#include <cuda_bf16.h>

#include <algorithm>
#include <cstring>
#include <mutex>

#include "internal.h"
#include "kernels_common.cuh"
#include "search.h"
#include "tcgen05.cuh"
#include "verify_tc.h"

namespace pano {
namespace {

constexpr int CH = TC_CHUNK;  // 128 rows (MMA M)
constexpr int QG = TC_QG;     // 64 queries per group (MMA N, padded to 16)
constexpr int S = TC_SEG;     // chunks per segment (4 x 64 = 256 TMEM columns)
// epilogue thread t < NE: TMEM lane / chunk row t % 128 and query half
// t / 128 (queries 32h .. 32h+31 are TMEM columns 32h.. of each chunk's
// accumulator); warps w and w + 4 share a lane quarter.
constexpr int NE = 256;
constexpr int kMma = NE / 32, kProdA = kMma + 1, kProdB = kMma + 2;  // the other warps' roles
constexpr int NT = NE + 3 * 32;

__device__ __forceinline__ void mbar_arrive_plain(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src)
               : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// ------------------------------------------------------------------ build
// One CTA per chunk: bf16 tiles, tail norms / norms of the dequantised
// vectors and the bound on their distance to the exact transform.
__global__ void __launch_bounds__(256) pack_bf16_kernel(
    const float* __restrict__ xt, const float* __restrict__ rows,
    const int64_t* __restrict__ perm, int64_t chunk0, int d, int L,
    const int32_t* __restrict__ level_off, const float* __restrict__ mu, double c_trans,
    uint8_t* __restrict__ slices, float* __restrict__ tails, float* __restrict__ xn2,
    float* __restrict__ ex, int32_t* __restrict__ ids) {
  __shared__ int16_t lvl_of[8192 / 8];  // level of each 8-element chunk of a row
  const int64_t lc = blockIdx.x, g = chunk0 + lc;
  const float* xblk = xt + lc * CH * d;
  const int64_t* pb = perm + lc * CH;
  uint8_t* cbase = slices + g * (int64_t)CH * d * 2;
  for (int c8 = threadIdx.x; c8 < d / 8; c8 += blockDim.x) {
    int l = 0;
    while (level_off[l + 1] <= c8 * 8) ++l;
    lvl_of[c8] = (int16_t)l;
  }
  __syncthreads();
  for (int e = threadIdx.x; e < CH * (d / 8); e += blockDim.x) {
    const int r = e / (d / 8), c8 = e % (d / 8);
    const int l = lvl_of[c8];
    const int m = level_off[l], w = level_off[l + 1] - m;
    const bool valid = pb[r] >= 0;
    __align__(16) __nv_bfloat16 v[8];
#pragma unroll
    for (int j = 0; j < 8; ++j)
      v[j] = __float2bfloat16_rn(valid ? xblk[(int64_t)r * d + c8 * 8 + j] : 0.f);
    *reinterpret_cast<uint4*>(cbase + (size_t)m * CH * 2 + tc::swz_offset(r, c8 * 8 - m, CH, w)) =
        *reinterpret_cast<const uint4*>(v);
  }
  const int warp = threadIdx.x / 32, lane = threadIdx.x & 31;
  for (int i = warp; i < CH; i += blockDim.x / 32) {
    const int64_t slot = g * CH + i;
    const bool valid = pb[i] >= 0;
    const float* x = xblk + (int64_t)i * d;
    auto stored = [](float v) { return __bfloat162float(__float2bfloat16_rn(v)); };
    const float* r = rows + (lc * CH + i) * (int64_t)d;
    const RowBounds rb = row_bounds(
        d, L, level_off, c_trans, valid, [&](int j) { return stored(x[j]); },
        [&](int j) { return (double)stored(x[j]) - (double)x[j]; },
        [&](int j) { return (double)r[j] - (double)mu[j]; },
        // (exact: xh is within a factor 2 of x[j])
        [&](Acc2& a, int j, float xh) { acc2_sq(a, __fsub_rn(xh, x[j])); },
        [&](Acc2& a, int j) { acc2_sqdiff(a, r[j], mu[j]); });
#pragma unroll
    for (int u = 0; u < 2; ++u)
      if (lane + 32 * u < L) tails[(g * (L + 1) + lane + 32 * u) * CH + i] = rb.tail[u];
    if (lane == 0) {
      tails[(g * (L + 1) + L) * CH + i] = 0.f;
      xn2[slot] = rb.xn2;
      ex[slot] = rb.ex;
      ids[slot] = valid ? (int32_t)pb[i] : -1;
    }
  }
}

// FP8 storage: each vector gets a power-of-two scale s_x = 2^e (the least with
// max |x~_j| / s_x <= 448, E4M3's largest finite value; e clamped to [-60,
// 60]) and its elements are stored as E4M3 of x~ / s_x, rounded to nearest.
// Level tiles have the byte layout of bf16 tiles of half the width; tail
// norms, norms and e_x are those of x^ = s_x e4m3(x~ / s_x).  Widths are 32,
// 64 or multiples of 128, so 16-element groups never straddle a level.
__global__ void __launch_bounds__(256) pack_fp8_kernel(
    const float* __restrict__ xt, const float* __restrict__ rows,
    const int64_t* __restrict__ perm, int64_t chunk0, int d, int L,
    const int32_t* __restrict__ level_off, const float* __restrict__ mu, double c_trans,
    uint8_t* __restrict__ slices, float* __restrict__ tails, float* __restrict__ xn2,
    float* __restrict__ ex, float* __restrict__ xscale, int32_t* __restrict__ ids) {
  __shared__ int16_t lvl_of[8192 / 16];  // level of each 16-element group of a row
  __shared__ float s_scale[CH], s_inv[CH];
  const int64_t lc = blockIdx.x, g = chunk0 + lc;
  const float* xblk = xt + lc * CH * d;
  const int64_t* pb = perm + lc * CH;
  uint8_t* cbase = slices + g * (int64_t)CH * d;
  for (int c16 = threadIdx.x; c16 < d / 16; c16 += blockDim.x) {
    int l = 0;
    while (level_off[l + 1] <= c16 * 16) ++l;
    lvl_of[c16] = (int16_t)l;
  }
  const int warp = threadIdx.x / 32, lane = threadIdx.x & 31;
  for (int i = warp; i < CH; i += blockDim.x / 32) {
    float m = 0.f;
    if (pb[i] >= 0)
      for (int j = lane; j < d; j += 32) m = fmaxf(m, fabsf(xblk[(int64_t)i * d + j]));
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, off));
    int e = 0;
    if (m > 0.f) frexpf(m / 448.f, &e);  // m / 448 < 2^e, so m / 2^e < 448
    e = max(-60, min(60, e));
    if (lane == 0) {
      s_scale[i] = ldexpf(1.f, e);
      s_inv[i] = ldexpf(1.f, -e);
    }
  }
  __syncthreads();
  for (int e = threadIdx.x; e < CH * (d / 16); e += blockDim.x) {
    const int r = e / (d / 16), c16 = e % (d / 16);
    const int l = lvl_of[c16];
    const int m = level_off[l], w = level_off[l + 1] - m;
    const bool valid = pb[r] >= 0;
    const float inv = s_inv[r];
    __align__(16) uint8_t v[16];
#pragma unroll
    for (int j = 0; j < 16; ++j)
      v[j] = tc::f32_to_e4m3(valid ? xblk[(int64_t)r * d + c16 * 16 + j] * inv : 0.f);
    *reinterpret_cast<uint4*>(cbase + (size_t)m * CH +
                              tc::swz_offset(r, (c16 * 16 - m) / 2, CH, w / 2)) =
        *reinterpret_cast<const uint4*>(v);
  }
  for (int i = warp; i < CH; i += blockDim.x / 32) {
    const int64_t slot = g * CH + i;
    const bool valid = pb[i] >= 0;
    const float* x = xblk + (int64_t)i * d;
    const float sc = s_scale[i], inv = s_inv[i];
    auto stored = [&](float v) { return tc::e4m3_to_f32(tc::f32_to_e4m3(v * inv)) * sc; };
    const float* r = rows + (lc * CH + i) * (int64_t)d;
    const RowBounds rb = row_bounds(
        d, L, level_off, c_trans, valid, [&](int j) { return stored(x[j]); },
        [&](int j) { return (double)stored(x[j]) - (double)x[j]; },
        [&](int j) { return (double)r[j] - (double)mu[j]; },
        [&](Acc2& a, int j, float xh) { acc2_sqdiff(a, xh, x[j]); },
        [&](Acc2& a, int j) { acc2_sqdiff(a, r[j], mu[j]); });
#pragma unroll
    for (int u = 0; u < 2; ++u)
      if (lane + 32 * u < L) tails[(g * (L + 1) + lane + 32 * u) * CH + i] = rb.tail[u];
    if (lane == 0) {
      tails[(g * (L + 1) + L) * CH + i] = 0.f;
      xn2[slot] = rb.xn2;
      ex[slot] = rb.ex;
      xscale[slot] = sc;
      ids[slot] = valid ? (int32_t)pb[i] : -1;
    }
  }
}

// ------------------------------------------------------------------ search
// One work item = (list, segment of S chunks, group of <= QG queries).  The
// CTA's warps have roles that meet on mbarriers only, so that the copies, the
// MMA chains and the tests of different chunks, levels and items overlap:
//
//   A producer (one thread)  claims items and streams the level tiles of their
//       chunks, panel by panel (64 bf16 or 128 E4M3 columns: 128-byte rows),
//       into a ring.  It runs ahead of the tests: a tile staged for a chunk
//       that has died since is discarded.
//   B producer (one warp)    gathers the group's query panels (the split image
//       that the query transform left in global memory) into a second ring.
//   MMA thread               one chain per (panel, chunk); at a level that is
//       tested it commits to the chunk's barrier and goes on with that chunk
//       only after the test.  Levels without a test follow each other
//       without a wait.
//   epilogue (8 warps)       candidate row t % 128 of every chunk belongs to
//       two threads, one per half of the query group.  They test, and after
//       the last level filter and defer the survivors; then the accumulators
//       go back to the MMA thread, which has the next item's tiles waiting.
//
// What bounds it: instruction issue and latency of the epilogue (44 % of the
// issue slots; tensor pipe 17 %, L2 21 %, ncu on 500k x 768), so its code is
// kept small (the roles share one instruction cache: survivors unrolled over
// 32 slots cost 15 %) and its tests run two queries per instruction.  Against
// the same work in lockstep, a CTA barrier per level and the query split redone
// per item: 4M x 768 BF16, 10,000 queries at nprobe 64, 25.4 -> 18.9 ms a
// search; 1M x 960 BF16 3.68 -> 3.32; 1M x 768 FP8, k = 100, 30.4 -> 11.4 (its
// two CTAs per SM and the insertion of large k included); 1.5M x 384 Zipf
// 60.6 -> 19.6; 4M x 128, 1,024 queries 1.33 -> 1.18.
//
// Every wait is bounded; a wait that gives up raises `fail`, on which all
// other waits end too.  The epilogue's barriers carry that flag (bar.red.or),
// so its warps leave together.
constexpr int TMEM_COLS = S * QG;  // 256: two CTAs share an SM's tensor memory
// a chunk with at most this many live rows is tested at every level: only a
// test that leaves no live row retires the chunk's copies and MMAs
constexpr int kTestRows = 16;
constexpr int kPend = 256;  // deferred re-rank entries
constexpr int UBQ = 8;      // queries per pass of the upper-bound filter
static_assert(QG == 64 && TMEM_COLS <= 256, "two query halves; two CTAs per SM");
static_assert(kPend <= NE, "the flush gives each pending pair one thread");
static_assert(UBQ == NE / 32 && QG % UBQ == 0, "one warp per query of a pass");

// Two CTAs of 113 KB share an SM: with 128-byte panel rows BF16 has 3 A stages
// of 16 KB and 2 B stages of 16 KB (hi, lo), E4M3 2 A stages and 2 B stages of
// 24 KB (three terms).  Where every level is narrower (rows of 64 or 32
// bytes), the same bytes hold twice or four times the stages: a narrow panel's
// MMAs end long before the next panel's copies would land.
// F = 128 / the widest level's row bytes: 1, 2 or 4 (compile-time: stage counts
// held in registers cost the roles 5 to 10 %).
constexpr int kMaxStages = 8;
template <bool FP8, int F>
struct Ring {
  static constexpr int PW = FP8 ? 128 : 64;  // elements of a full panel
  static constexpr int TERMS = FP8 ? 3 : 2;
  static constexpr uint32_t A_ALL = (FP8 ? 2 : 3) * CH * 128, B_ALL = 2 * TERMS * QG * 128;
  static constexpr uint32_t BYTES = A_ALL + B_ALL;
  static constexpr int NA = (FP8 ? 2 : 3) * F < kMaxStages ? (FP8 ? 2 : 3) * F : kMaxStages;
  static constexpr int NB = 2 * F;
  static constexpr uint32_t A_BYTES = CH * 128 / F, B_TERM = QG * 128 / F, B_BYTES = TERMS * B_TERM;
};

struct Item {
  int4 it;  // list (-1: no more items), segment, bucket offset, group size
  int64_t ch0;
  int nch;
};

// Per-query terms of the separable test, a pair pruned when
// p + S sx + G rx + E ex < H + Hx.  One array per term: a 16-byte read brings
// four queries' and the test runs on pairs of queries (FFMA2).
struct QTerms {
  alignas(16) float E[QG], G[QG], S[QG], H[QG];
};

struct Shared {
  float Hx[S * CH], rx[S * CH], ex[S * CH];  // candidate terms of the separable test
  uint32_t alive[S][2][CH];                  // per chunk and query half: a word per row
  QTerms qterm;                              // of the tested level
  float qnq[QG], qrq[QG], qeq[QG], qtau[QG];
  float qs[QG], qun[QG];  // E4M3: the query's scale 2^e, its split's underflow per unit of |x|_2
  int32_t qid[QG], qk[QG], bq[QG];  // bq: the B producer's copy of qid
  int scount[QG];                   // survivors of the last level per query
  uint16_t ub[UBQ][S * CH];         // bf16 upper bounds of one pass
  int64_t pslot[kPend];             // deferred pairs: slot, query; in a flush id and bounds
  int32_t pq[kPend], pid[kPend];
  float plb[kPend], pub[kPend];     // plb: the partial product, then the bound, then the distance
  uint16_t keep[kPend], rnk[kPend];
  uint32_t rowlive[2][S][NE / 32];  // by parity of the chunk's tests; one word per epilogue warp
  uint32_t tag_a[kMaxStages], tag_b[kMaxStages];  // what a stage holds: (item, panel, chunk)
  uint32_t dead[2];                 // per item slot: its chunks that died (all bits: the item)
  Item item[2];
  alignas(8) uint64_t a_full[kMaxStages], a_empty[kMaxStages], b_full[kMaxStages],
      b_empty[kMaxStages];
  uint64_t item_full[2], item_empty[2], mma_bar[S], tested[S], acc_free, fin, drain;
  unsigned long long stat[6], sec[8];
  long long tmark, tkernel;
  uint32_t gm[2];  // the group's queries with k > 0 (two halves)
  uint32_t tmem;
  int npend, fail, flush[3], issued_a, issued_b;
};

// The fail flag of the CTA, read while another thread may set it.
__device__ __forceinline__ bool failed(const int* fail) {
  return *reinterpret_cast<const volatile int*>(fail) != 0;
}

// mbarrier.try_wait that may sleep for up to `ns` before it reports an
// incomplete phase: a waiting warp polls rarely and leaves its issue slots to
// the others (polls were nearly half of the kernel's instructions).
__device__ __forceinline__ bool mbar_try_wait_for(uint64_t* bar, uint32_t parity, uint32_t ns) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n"
      " selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity), "r"(ns)
      : "memory");
  return ok != 0;
}
constexpr uint32_t kSleepNs = 20000;

// Waits for phase `parity` of `bar`; false if the wait gave up (then `fail`
// is set) or another thread's did.
__device__ __forceinline__ bool wait_or_fail(uint64_t* bar, uint32_t parity, int* fail) {
  if (mbar_try_wait_for(bar, parity, kSleepNs)) return true;
  const long long t0 = clock64();
  while (!mbar_try_wait_for(bar, parity, kSleepNs)) {
    if (failed(fail)) return false;
    if (clock64() - t0 > kWaitCycles) {
      atomicExch(fail, 1);
      return false;
    }
  }
  return true;
}

// wait_or_fail that also ends once `dead` has one of the bits `mask`: 1 the
// phase completed, 2 the bits are set, 0 failed.  (A producer must not wait
// for a stage on behalf of a chunk that died: the MMA thread discards stale
// stages only while it looks for a tile of a live one.)
__device__ __forceinline__ int wait_or_dead(uint64_t* bar, uint32_t parity, int* fail,
                                            const uint32_t* dead, uint32_t mask) {
  const volatile uint32_t* dv = dead;
  const long long t0 = clock64();
  while (true) {
    if ((*dv & mask) == mask) return 2;
    if (mbar_try_wait(bar, parity)) return (*dv & mask) == mask ? 2 : 1;
    if (failed(fail)) return 0;
    if (clock64() - t0 > kWaitCycles) {
      atomicExch(fail, 1);
      return 0;
    }
  }
}

// E4M3: the query split's underflow per unit of |x|_2, for the largest |q~_j|
// m: below the normal range of the scale 2^e each element loses at most
// 2^-10 of the scaled unit, so the partial product at most 2^-10 2^e sqrt(d)
// |x|_2.
__device__ __forceinline__ float split_underflow(float m, int d) {
  return __fmul_ru(ldexpf(1.f, min(60, tc::e4m3_exponent(m)) - 10), __fsqrt_ru((float)d));
}

// Barrier of the NE epilogue threads (named barrier 1); true if any of them
// passed p.  Every lane executes it, under conditions that are the same for the
// whole warp; like __syncthreads_or it counts threads, so lanes that arrive apart
// need no __syncwarp() before it (which cost the kernel 1.5 to 2 %).
__device__ __forceinline__ bool epi_or(bool p) {
  uint32_t r;
  asm volatile(
      "{\n .reg .pred p, q;\n setp.ne.u32 p, %1, 0;\n bar.red.or.pred q, 1, %2, p;\n"
      " selp.u32 %0, 1, 0, q;\n}\n"
      : "=r"(r)
      : "r"((uint32_t)p), "n"(NE)
      : "memory");
  return r != 0;
}

// The deferred pairs (slot, query, last-level partial product) get their Eq. 3
// bounds (C = 0), are checked against their queries' thresholds of the moment
// and against each other (below); the rest get their exact distance and top-k
// insertion, in two passes: first each query's k kept pairs of smallest lower
// bound (ties by entry), whose exact distances usually set its threshold,
// then the others that still pass the threshold.  All epilogue threads call it
// (one thread per entry at most: kPend <= NE); kept out of line so that it
// does not add to the level loop's registers.  Returns the number re-ranked
// (thread 0; 0 elsewhere), or -1 if a wait had failed.
template <bool FP8, bool LARGE>
__device__ __noinline__ int flush_pending(const VerifyTCArgs& a, Shared& sh, int np) {
  const int tid = threadIdx.x, warp = tid / 32, nw = NE / 32;
  const int32_t* pq = sh.pq;
  float* plb = sh.plb;
  int* s_cnt = sh.flush;
  auto sync_failed = [&] { return epi_or(failed(&sh.fail)); };
  if (tid < 3) s_cnt[tid] = 0;
  if (tid < QG) sh.scount[tid] = 0;
  if (sync_failed()) return -1;
  auto tau_of = [&](int q, int kk) {
    const unsigned long long key = kth_key<LARGE>(a.topk + (int64_t)q * a.k_max, kk);
    return fminf(key == kEmptyKey ? INFINITY : __fmul_ru(key_dist(key), 1.000001f),
                 __ldcg(a.tau_seed + q));
  };
  const bool mine = tid < np;
  const int q = mine ? pq[tid] : 0;
  int kk = 0;
  float lb = 0.f;
  bool keep_s = false;
  if (mine) {
    const int64_t slot = sh.pslot[tid];
    const float4 inf = a.qinfo[q];
    const float nx = a.xn2[slot], exv = a.ex[slot], rx = sqrtf(nx), p = plb[tid];
    kk = a.kq[q];
    const float tau = tau_of(q, kk);
    sh.pid[tid] = a.ids[slot];
    const float A = inf.x + nx - 2.f * p, Ss = inf.y + rx;
    const float under = FP8 ? 2.f * split_underflow(inf.w, a.d) * rx : 0.f;
    const float slack = fmaf(a.gslack * Ss, Ss, under);
    const float lr = sqrtf(fmaxf(A - slack, 0.f)) - (inf.z + exv);
    lb = lr > 0.f ? lr * lr * a.lb_scale : 0.f;
    const float ru = __fadd_ru(sqrt_up(fmaxf(A + slack, 0.f)), inf.z + exv);
    plb[tid] = lb;
    sh.pub[tid] = __fmul_ru(__fmul_ru(ru, ru), a.ub_scale);
    keep_s = !(lb > tau);
    if (keep_s) atomicAdd(&sh.scount[q & (QG - 1)], 1);
  }
  if (sync_failed()) return -1;
  // k pending pairs of the same query with upper bounds below its lower bound
  // (all k are closer) rule a pair out; with at most k pairs of the query (of
  // its hash) pending there is nothing to look for
  const bool crowded = keep_s && sh.scount[q & (QG - 1)] > kk;
  if (crowded) {
    int below = 0;
    for (int o = 0; o < np && below < kk; ++o)
      below += (pq[o] == q) & (__fmul_ru(sh.pub[o], 1.000001f) < lb);
    keep_s = below < kk;
  }
  if (keep_s && (a.d & 3) == 0)  // the kept rows head for L2 at once
    prefetch_l2(a.rows + sh.pslot[tid] * a.d, (uint32_t)a.d * 4);
  if (keep_s && crowded) sh.keep[atomicAdd(&s_cnt[0], 1)] = (uint16_t)tid;
  if (sync_failed()) return -1;
  bool first = keep_s;
  if (keep_s && crowded) {  // rank among the kept pairs of its query
    const int nc = s_cnt[0];
    int r = 0;
    for (int j = 0; j < nc; ++j) {
      const int o = sh.keep[j];
      r += (pq[o] == q) & ((plb[o] < lb) | ((plb[o] == lb) & (o < tid)));
    }
    first = r < kk;
  }
  if (first) sh.rnk[atomicAdd(&s_cnt[1], 1)] = (uint16_t)tid;
  if (sync_failed()) return -1;
  // exact distances (a warp takes two pairs at a time; they replace the lower
  // bounds), then the top-k insertions: the pairs ranked first, then the
  // others that still pass the thresholds of the moment
  const uint16_t* list = sh.rnk;
  int n = s_cnt[1];
  for (int pass = 0;; ++pass) {
    for (int i = 2 * warp; i < n; i += 2 * nw) {
      const int s0 = list[i], s1 = list[i + 1 < n ? i + 1 : i];
      float d0, d1;
      exact_sqdist_warp_pair(a.qorig + (int64_t)pq[s0] * a.d, a.rows + sh.pslot[s0] * a.d,
                             a.qorig + (int64_t)pq[s1] * a.d, a.rows + sh.pslot[s1] * a.d, a.d,
                             d0, d1);
      if ((tid & 31) == 0) {
        plb[s0] = d0;
        plb[s1] = d1;
      }
    }
    if (sync_failed()) return -1;
    topk_flush_insert<LARGE>(a.topk, a.k_max, a.kq, a.tau_seed, list, n, pq, plb, sh.pid, NE);
    if (pass) break;
    if (sync_failed()) return -1;
    if (keep_s && !first && !(lb > tau_of(q, kk)))
      sh.keep[atomicAdd(&s_cnt[2], 1)] = (uint16_t)tid;
    if (sync_failed()) return -1;
    list = sh.keep;
    n = s_cnt[2];
    if (!n) break;
  }
  if (sync_failed()) return -1;
  return tid == 0 ? s_cnt[1] + s_cnt[2] : 0;
}

// The chunks of an item as its levels pass, identical in every role: which
// live and at which level each is tested next (a byte per chunk).
struct ChunkState {
  uint32_t live, next;
  __device__ __forceinline__ void start(int nch, int first_test) {
    live = (1u << nch) - 1u;
    next = 0x01010101u * (uint32_t)first_test;
  }
  __device__ __forceinline__ int test_level(int c) const { return (int)(next >> (8 * c)) & 255; }
  // the outcome of chunk c's test at level l: n live rows
  __device__ __forceinline__ void tested(const VerifyTCArgs& a, int c, int l, int n) {
    if (n == 0) live &= ~(1u << c);
    int t = a.L - 1;
    if (a.prune && n <= kTestRows) {
      t = l + 1;
    } else if (a.prune) {
      t = min(t, (l / a.test_every + 1) * a.test_every);
    }
    next = (next & ~(255u << (8 * c))) | ((uint32_t)t << (8 * c));
  }
};

__device__ __forceinline__ int live_rows(const uint32_t (&w)[NE / 32]) {
  const volatile uint32_t* v = w;
  int n = 0;
#pragma unroll
  for (int q = 0; q < 4; ++q) n += __popc(v[q] | v[q + 4]);
  return n;
}

__device__ __forceinline__ uint32_t stage_tag(uint32_t seq, int panel, int c) {
  return (seq << 18) | ((uint32_t)panel << 2) | (uint32_t)c;
}

// FP8 = false: BF16 tiles, kind::f16 MMAs with the query split into bf16 hi +
// lo.  FP8 = true: E4M3 tiles (the byte layout of bf16 tiles of half the
// width), kind::f8f6f4 MMAs with the query split into three E4M3 terms at a
// power-of-two scale of its own; the accumulator times the row's scale s_x and
// the query's is the partial product.
// LARGE: the slots of queries with k > kChainK are unsorted (the replacements
// of the flush cost the level loop registers, so a batch without them runs
// without their code).
template <bool FP8, bool LARGE, int F>
__global__ void __launch_bounds__(NT, 2) verify_tc_kernel(const __grid_constant__ VerifyTCArgs a) {
  using R = Ring<FP8, F>;
  constexpr int EB = FP8 ? 1 : 2;  // bytes per stored element
  extern __shared__ unsigned char smem_raw[];
  unsigned char* const base = smem_raw + ((1024 - (smem_u32(smem_raw) & 1023)) & 1023);
  unsigned char* const aring = base;
  unsigned char* const bring = base + R::A_ALL;
  Shared& sh = *reinterpret_cast<Shared*>(base + R::BYTES);

  const int tid = threadIdx.x, warp = tid / 32, lane = tid & 31;
  if (warp == 0) {
    tc::tmem_alloc(&sh.tmem, TMEM_COLS);
    tc::tmem_relinquish();
  }
  if (tid == 0) {
    for (int i = 0; i < kMaxStages; ++i) {
      mbar_init(&sh.a_full[i], 1);
      mbar_init(&sh.a_empty[i], 1);
      mbar_init(&sh.b_full[i], 1);
      mbar_init(&sh.b_empty[i], 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&sh.item_full[i], 1);
      mbar_init(&sh.item_empty[i], 2 + NE / 32);
    }
    for (int c = 0; c < S; ++c) {
      mbar_init(&sh.mma_bar[c], 1);
      mbar_init(&sh.tested[c], NE / 32);
    }
    mbar_init(&sh.acc_free, NE / 32);
    mbar_init(&sh.fin, 1);
    mbar_init(&sh.drain, 1);
    fence_mbar_init();
    sh.fail = sh.npend = sh.issued_a = sh.issued_b = 0;
    for (int i = 0; i < 6; ++i) sh.stat[i] = 0;
    for (int i = 0; i < 8; ++i) sh.sec[i] = 0;
    sh.tkernel = sh.tmark = clock64();
  }
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tbase = sh.tmem;
  const int L = a.L, d = a.d;
  const int first_test = a.prune ? 0 : L - 1;
  int* const fail = &sh.fail;

  if (warp == kMma) {
    if (lane == 0) {
      int sa = 0, sb = 0, used_a = 0, used_b = 0;
      uint32_t pa = 0, pb = 0, tph = 0;
      auto next_a = [&] {
        ++used_a;
        if (++sa == R::NA) sa = 0, pa ^= 1u;
      };
      auto next_b = [&] {
        ++used_b;
        if (++sb == R::NB) sb = 0, pb ^= 1u;
      };
      const uint32_t aaddr = smem_u32(aring) >> 4, baddr = smem_u32(bring) >> 4;
      const uint32_t term = R::B_TERM / 16;
      for (uint32_t seq = 0;; ++seq) {
        const int slot = seq & 1;
        if (!wait_or_fail(&sh.item_full[slot], (seq >> 1) & 1u, fail)) goto mma_done;
        const int G = sh.item[slot].it.w, nch = sh.item[slot].nch;
        if (sh.item[slot].it.x < 0) {
          // the stages left over from tiles staged ahead go back, so that the
          // producers see every copy and commit of theirs completed
          while (used_a < sh.issued_a) {
            if (!wait_or_fail(&sh.a_full[sa], pa, fail)) goto mma_done;
            mbar_arrive_plain(&sh.a_empty[sa]);
            next_a();
          }
          if (!wait_or_fail(&sh.fin, 0, fail)) goto mma_done;
          while (used_b < sh.issued_b) {
            if (!wait_or_fail(&sh.b_full[sb], pb, fail)) goto mma_done;
            mbar_arrive_plain(&sh.b_empty[sb]);
            next_b();
          }
          goto mma_done;
        }
        const int Npad = (G + 15) & ~15;
        const uint32_t idesc = FP8 ? tc::idesc_e4m3(CH, Npad) : tc::idesc_bf16(CH, Npad);
        // the previous item's accumulators have been read for the last time
        if (seq > 0 && !wait_or_fail(&sh.acc_free, (seq - 1) & 1u, fail)) goto mma_done;
        tc::fence_after_sync();
        ChunkState cs;
        cs.start(nch, first_test);
        uint32_t pending = 0;  // chunks tested at the level before
        uint32_t want = stage_tag(seq, 0, 0);
        uint32_t acc0 = 0;  // the item's first K-step overwrites the accumulators
        for (int l = 0; l < L; ++l) {
          const int w = a.level_off[l + 1] - a.level_off[l];
          int np = 1, rb = w * EB;  // panels and their row bytes
          if (rb > 128) np = rb >> 7, rb = 128;
          const int nks = rb >> 5;  // K-steps of 32 bytes: 16 bf16 or 32 E4M3 elements
          const uint64_t desc = tc::smem_desc(0, rb);
          uint32_t test = 0;
          for (; np > 0; --np, want += 4) {
            uint64_t db = 0;
            for (uint32_t m = cs.live; m; m &= m - 1) {
              const int c = __ffs(m) - 1;
              if ((pending >> c) & 1u) {  // (first panel only)
                const uint32_t par = (tph >> c) & 1u;
                if (!wait_or_fail(&sh.tested[c], par, fail)) goto mma_done;
                tph ^= 1u << c;
                tc::fence_after_sync();
                cs.tested(a, c, l - 1, live_rows(sh.rowlive[par][c]));
                if (!((cs.live >> c) & 1u)) {
                  *reinterpret_cast<volatile uint32_t*>(&sh.dead[slot]) =
                      cs.live ? ((1u << S) - 1u) & ~cs.live : ~0u;
                  continue;
                }
              }
              if (!db) {
                while (true) {
                  if (!wait_or_fail(&sh.b_full[sb], pb, fail)) goto mma_done;
                  if (*reinterpret_cast<volatile uint32_t*>(&sh.tag_b[sb]) == want) break;
                  mbar_arrive_plain(&sh.b_empty[sb]);  // a panel of an item that died
                  next_b();
                }
                db = desc + baddr + (uint32_t)sb * (R::B_BYTES / 16);
              }
              while (true) {
                if (!wait_or_fail(&sh.a_full[sa], pa, fail)) goto mma_done;
                if (*reinterpret_cast<volatile uint32_t*>(&sh.tag_a[sa]) == want + (uint32_t)c) break;
                mbar_arrive_plain(&sh.a_empty[sa]);  // a tile of a chunk that died
                next_a();
              }
              const uint32_t dt = tbase + (uint32_t)(c * QG);
              const uint64_t da = desc + aaddr + (uint32_t)sa * (R::A_BYTES / 16);
#pragma unroll
              for (int s = 0; s < 4; ++s) {
                if (s < nks) {
                  const uint32_t acc = s > 0 ? 1u : acc0;
                  if (FP8) {
                    tc::mma_e4m3(dt, da + 2 * s, db + 2 * s, idesc, acc);
                    tc::mma_e4m3(dt, da + 2 * s, db + 2 * s + term, idesc, 1u);
                    tc::mma_e4m3(dt, da + 2 * s, db + 2 * s + 2 * term, idesc, 1u);
                  } else {
                    tc::mma_bf16(dt, da + 2 * s, db + 2 * s, idesc, acc);
                    tc::mma_bf16(dt, da + 2 * s, db + 2 * s + term, idesc, 1u);
                  }
                }
              }
              tc::mma_commit(&sh.a_empty[sa]);
              next_a();
              if (np == 1 && cs.test_level(c) == l) {
                tc::mma_commit(&sh.mma_bar[c]);
                test |= 1u << c;
              }
            }
            if (db) {
              tc::mma_commit(&sh.b_empty[sb]);
              next_b();
            }
            pending = 0;
            acc0 = 1u;
          }
          if (!cs.live) break;
          pending = test;
        }
        mbar_arrive_plain(&sh.item_empty[slot]);
      }
    mma_done:
      // no MMA may run past the tensor memory's release
      tc::mma_commit(&sh.drain);
      mbar_wait_bounded(&sh.drain, 0);
    }
  } else if (warp == kProdA) {
    if (lane == 0) {
      int sa = 0;
      uint32_t pa = 1, uses = 0;
      const int64_t n_items = *a.n_items < a.items_cap ? *a.n_items : a.items_cap;
      auto load_item = [&](int i, Item* o) {
        o->it = i < n_items ? a.items[i] : make_int4(-1, 0, 0, 0);
        o->ch0 = 0;
        o->nch = 0;
        if (o->it.x >= 0) {
          o->ch0 = a.chunk_off[o->it.x] + (int64_t)o->it.y * S;
          const int64_t n = a.chunk_off[o->it.x + 1] - o->ch0;
          o->nch = n < S ? (int)n : S;
        }
      };
      bool ok = true;
      Item cur;
      load_item(atomicAdd(a.counter, 1), &cur);
      for (uint32_t seq = 0; ok; ++seq) {
        const int slot = seq & 1;
        if (seq >= 2 && !(ok = wait_or_fail(&sh.item_empty[slot], ((seq >> 1) - 1) & 1u, fail)))
          break;
        sh.item[slot] = cur;
        sh.dead[slot] = 0u;
        mbar_arrive_plain(&sh.item_full[slot]);
        if (cur.it.x < 0) break;
        const int claimed = atomicAdd(a.counter, 1);  // the next item, one ahead
        Item nxt;
        const uint8_t* src = a.slices + cur.ch0 * (int64_t)CH * d * EB;
        int panel = 0;
        bool all_dead = false;
        for (int l = 0; l < L && ok && !all_dead; ++l) {
          const int m = a.level_off[l], w = a.level_off[l + 1] - m;
          const int np = (w + R::PW - 1) / R::PW, pw = w < R::PW ? w : R::PW;
          const uint32_t bytes = (uint32_t)(CH * pw * EB);
          for (int p = 0; p < np && ok; ++p, ++panel) {
            for (int c = 0; c < cur.nch; ++c) {
              const int r = wait_or_dead(&sh.a_empty[sa], pa, fail, &sh.dead[slot], 1u << c);
              ok = r != 0;
              if (!ok) break;
              if (r == 2) continue;
              sh.tag_a[sa] = stage_tag(seq, panel, c);
              mbar_arrive_expect_tx(&sh.a_full[sa], bytes);
              bulk_g2s(aring + sa * R::A_BYTES,
                       src + (int64_t)c * CH * d * EB + (size_t)m * CH * EB + (size_t)p * bytes,
                       bytes, &sh.a_full[sa]);
              sh.issued_a = (int)++uses;
              if (++sa == R::NA) sa = 0, pa ^= 1u;
            }
            all_dead = *reinterpret_cast<volatile uint32_t*>(&sh.dead[slot]) == ~0u;
            if (all_dead) break;
          }
          if (l == 0) load_item(claimed, &nxt);
        }
        cur = nxt;
      }
      // no copy may land after the CTA has ended; on the ordinary way out the
      // stages also came back
      for (uint32_t i = 0; i < (uint32_t)R::NA && i < uses; ++i) {
        const uint32_t par = ((uses - 1 - i) / R::NA) & 1u;
        if (ok) wait_or_fail(&sh.a_empty[i], par, fail);
        mbar_wait_bounded(&sh.a_full[i], par);
      }
    }
  } else if (warp == kProdB) {
    int sb = 0;
    uint32_t pb = 1, uses = 0;
    bool ok = true;
    for (uint32_t seq = 0; ok; ++seq) {
      const int slot = seq & 1;
      // (lane 0 waits and decides for the warp)
      ok = lane || wait_or_fail(&sh.item_full[slot], (seq >> 1) & 1u, fail);
      ok = __shfl_sync(0xffffffffu, (int)ok, 0);
      if (!ok) break;
      const int4 it = sh.item[slot].it;
      if (it.x < 0) {
        if (lane == 0) {
          sh.issued_b = (int)uses;
          mbar_arrive_plain(&sh.fin);
        }
        break;
      }
      const int G = it.w;
      if (lane < G) sh.bq[lane] = a.bucket[it.z + lane];
      if (lane + 32 < G) sh.bq[lane + 32] = a.bucket[it.z + lane + 32];
      __syncwarp();
      int panel = 0;
      bool stop = false;
      const size_t rowb = (size_t)d * 4;  // bytes of a query's image
      for (int l = 0; l < L && ok && !stop; ++l) {
        const int m = a.level_off[l], w = a.level_off[l + 1] - m;
        const int np = (w + R::PW - 1) / R::PW, pw = w < R::PW ? w : R::PW;
        const int rb = pw * EB;
        for (int p = 0; p < np; ++p, ++panel) {
          int r = lane ? 0 : wait_or_dead(&sh.b_empty[sb], pb, fail, &sh.dead[slot], ~0u);
          r = __shfl_sync(0xffffffffu, r, 0);
          ok = r != 0;
          stop = r == 2;
          if (!ok || stop) break;
          unsigned char* st = bring + sb * R::B_BYTES;
          const unsigned char* img =
              reinterpret_cast<const unsigned char*>(a.qt) + (size_t)(m + p * R::PW) * EB;
          // a lane copies one 16-byte piece of every (32 / pieces)-th row
          const int lg = __ffs(rb >> 4) - 1;  // pieces per row: 2, 4 or 8
          const int v = lane & ((1 << lg) - 1);
#pragma unroll 4
          for (int g = lane >> lg; g < G; g += 32 >> lg) {
            const unsigned char* src = img + sh.bq[g] * rowb + 16 * v;
            unsigned char* dst = st + tc::swz_offset(g, 8 * v, QG, rb / 2);
#pragma unroll
            for (int t = 0; t < R::TERMS; ++t)
              cp_async16(dst + t * R::B_TERM, src + (size_t)t * d * EB);
          }
          cp_async_wait_all();
          fence_proxy_async_smem();
          __syncwarp();
          if (lane == 0) {
            sh.tag_b[sb] = stage_tag(seq, panel, 0);
            mbar_arrive_plain(&sh.b_full[sb]);
          }
          ++uses;
          if (++sb == R::NB) sb = 0, pb ^= 1u;
        }
      }
      __syncwarp();
      if (ok && lane == 0) mbar_arrive_plain(&sh.item_empty[slot]);
    }
    if (ok && lane == 0)  // the stages came back: no commit is left in flight
      for (uint32_t i = 0; i < (uint32_t)R::NB && i < uses; ++i)
        wait_or_fail(&sh.b_empty[i], ((uses - 1 - i) / R::NB) & 1u, fail);
    __syncwarp();
  } else {
    // ---------------------------------------------------------- epilogue
    const int row = tid & (CH - 1), half = tid / CH;
    const uint32_t lane_base = (uint32_t)((warp & 3) * 32) << 16;
    const float g_slack = a.gslack;
    constexpr float kEval = 32.f * 5.9604645e-08f;  // evaluation slack of the separable test
    auto section = [&](int i) {  // charge the time since the last mark to section i
      if (a.collect && tid == 0) {
        const long long now = clock64();
        sh.sec[i] += (unsigned long long)(now - sh.tmark);
        sh.tmark = now;
      }
    };
    // threshold -> per-query terms of the separable test (thread g < QG)
    auto set_query_terms = [&](int g, float tau, float sq, QTerms& qt) {
      // sqrt(tau / lb_scale), bounded from above (a product by the rounded-up
      // reciprocal, itself rounded up, bounds the quotient from above)
      const float st = tau == INFINITY ? 1e18f : fminf(sqrt_up(__fmul_ru(tau, a.inv_lb_up)), 1e18f);
      const float E = __fadd_ru(sh.qeq[g], st);
      const float nq = sh.qnq[g], rq = sh.qrq[g];
      // E4M3: the query split's underflow error (at most qun |x|_2 on the
      // partial product) joins the g rq coefficient of rx
      qt.E[g] = E;
      qt.G[g] = FP8 ? fmaf(g_slack, rq, sh.qun[g]) : g_slack * rq;
      qt.S[g] = sq;
      qt.H[g] = 0.5f * (nq - g_slack * nq - E * E - kEval * (rq + E) * (rq + E));
      sh.qtau[g] = tau;
    };
    // bits of the 16 slots from g0 on that the margined Eq. 3 test prunes,
    // given their accumulators: two queries per instruction, the sign of each
    // comparison's difference shifted in, the last slot first
    auto pruned_bits = [&](const float (&v)[16], const QTerms& qt, int g0, float sx, float rx,
                           float ex, float Hx, float fr) {
      constexpr int N = 16;
      const uint64_t sx2 = pack2(sx, sx), rx2 = pack2(rx, rx), ex2 = pack2(ex, ex),
                     hx2 = pack2(Hx, Hx), fr2 = pack2(fr, fr);
      uint32_t bits = 0;
#pragma unroll
      for (int g = N - 4; g >= 0; g -= 4) {
        const ulonglong2 E = *reinterpret_cast<const ulonglong2*>(qt.E + g0 + g);
        const ulonglong2 G = *reinterpret_cast<const ulonglong2*>(qt.G + g0 + g);
        const ulonglong2 S2 = *reinterpret_cast<const ulonglong2*>(qt.S + g0 + g);
        const ulonglong2 H = *reinterpret_cast<const ulonglong2*>(qt.H + g0 + g);
        uint64_t p0 = pack2(v[g], v[g + 1]), p1 = pack2(v[g + 2], v[g + 3]);
        if (FP8) {
          const ulonglong2 q = *reinterpret_cast<const ulonglong2*>(sh.qs + g0 + g);
          p0 = mul2(mul2(p0, fr2), q.x);
          p1 = mul2(mul2(p1, fr2), q.y);
        }
        p1 = fma2(E.y, ex2, fma2(G.y, rx2, fma2(S2.y, sx2, p1)));
        p0 = fma2(E.x, ex2, fma2(G.x, rx2, fma2(S2.x, sx2, p0)));
        p1 = sub2(p1, add2(H.y, hx2));
        p0 = sub2(p0, add2(H.x, hx2));
        bits = __funnelshift_l((uint32_t)(p1 >> 32), bits, 1);
        bits = __funnelshift_l((uint32_t)p1, bits, 1);
        bits = __funnelshift_l((uint32_t)(p0 >> 32), bits, 1);
        bits = __funnelshift_l((uint32_t)p0, bits, 1);
      }
      return bits;
    };
    uint32_t mph = 0, tph = 0;
    bool bad = false;  // uniform over the epilogue after each epi_or
    for (uint32_t seq = 0;; ++seq) {
      const int slot = seq & 1;
      // (a failed wait goes on to the next barrier, where all warps leave)
      const bool got = wait_or_fail(&sh.item_full[slot], (seq >> 1) & 1u, fail);
      const Item im = sh.item[slot];
      const int G = im.it.w, nch = im.nch;
      if (got && im.it.x < 0) break;
      if (a.collect && tid == 0) sh.tmark = clock64();
      // ---- prologue: group, candidates, liveness
      bool valid[S] = {};
      if (got) {
#pragma unroll
        for (int c = 0; c < S; ++c)
          valid[c] = c < nch && a.ids[(im.ch0 + c) * CH + row] >= 0;
        if (tid < QG) {
          const int q = tid < G ? a.bucket[im.it.z + tid] : -1;
          sh.qid[tid] = q;
          int kk = 0;
          float4 inf = make_float4(0.f, 0.f, 0.f, 0.f);
          if (q >= 0) {
            inf = a.qinfo[q];
            kk = a.kq[q];
          }
          sh.qnq[tid] = inf.x;
          sh.qrq[tid] = inf.y;
          sh.qeq[tid] = inf.z;
          sh.qk[tid] = kk;
          sh.scount[tid] = 0;
          if (FP8) {
            const int e = tc::e4m3_exponent(inf.w);  // the split's scale is 2^e
            if (e > 60) atomicOr(a.err, kErrBadInput);
            sh.qs[tid] = ldexpf(1.f, min(60, e));
            sh.qun[tid] = split_underflow(inf.w, d);
          }
          // the group's queries with k > 0: warp 0 holds queries 0-31, warp 1 32-63
          const unsigned b = __ballot_sync(0xffffffffu, kk > 0);
          if (lane == 0) sh.gm[warp] = b;
          if (kk > 0) {
            const unsigned long long key = kth_key<LARGE>(a.topk + (int64_t)q * a.k_max, kk);
            const float tau = key == kEmptyKey ? INFINITY : __fmul_ru(key_dist(key), 1.000001f);
            set_query_terms(tid, fminf(tau, __ldcg(a.tau_seed + q)),
                            a.eps * a.qtail[(int64_t)q * (L + 1) + 1], sh.qterm);
          } else {
            sh.qterm.E[tid] = sh.qterm.G[tid] = sh.qterm.S[tid] = 0.f;
            sh.qterm.H[tid] = -INFINITY;
            sh.qtau[tid] = -1.f;
          }
        }
        for (int e = tid; e < nch * CH; e += NE) {
          const int64_t slot_e = im.ch0 * CH + e;
          const float nx = a.xn2[slot_e], rx = sqrtf(nx), exv = a.ex[slot_e];
          const float s2 = (rx + exv) * (rx + exv);
          sh.Hx[e] = 0.5f * (nx - g_slack * nx - exv * exv - kEval * s2);
          sh.rx[e] = rx;
          sh.ex[e] = exv;
        }
      }
      if ((bad = epi_or(!got || failed(fail)))) break;
      {
        const uint32_t gm = sh.gm[half], any = sh.gm[0] | sh.gm[1];
#pragma unroll
        for (int c = 0; c < S; ++c) {
          if (c < nch) sh.alive[c][half][row] = valid[c] ? gm : 0u;
          if (a.collect && half == 0) {  // live rows entering level 0
            const unsigned b = __ballot_sync(0xffffffffu, valid[c] && any);
            const int w0 = a.level_off[1];
            if (lane == 0)
              atomicAdd(&sh.stat[5], (unsigned long long)__popc(b) * (unsigned long long)(w0 * EB + 4));
          }
        }
      }
      section(0);

      // ---- the tested levels
      ChunkState cs;
      cs.start(nch, first_test);
      for (int l = first_test, l0 = 0;;) {
        uint32_t test = 0;
        for (int c = 0; c < nch; ++c)
          if (((cs.live >> c) & 1u) && cs.test_level(c) == l) test |= 1u << c;
        if (a.collect) {
          // per level since the last test: the tiles and their bytes; from
          // level 1 on the rows still live for some query of the group
          // (algorithmic bytes); the pairs and their coordinates
          for (; l0 <= l; ++l0) {
            const int w = a.level_off[l0 + 1] - a.level_off[l0];
            if (tid == 0) {
              sh.stat[2] += __popc(cs.live);
              sh.stat[3] += (unsigned long long)__popc(cs.live) * w * CH * EB;
            }
            for (int c = 0; c < nch; ++c) {
              if (!((cs.live >> c) & 1u)) continue;
              const uint32_t wm = sh.alive[c][half][row];
              const unsigned np = __reduce_add_sync(0xffffffffu, (unsigned)__popc(wm));
              if (lane == 0 && np) {
                atomicAdd(&sh.stat[0], (unsigned long long)np);
                atomicAdd(&sh.stat[1], (unsigned long long)np * w);
              }
              if (l0 > 0 && tid == 0) {
                // (the words of the chunk's last published test; of none, all its rows)
                const int n = first_test == L - 1 ? CH
                                                  : live_rows(sh.rowlive[((tph >> c) & 1u) ^ 1u][c]);
                sh.stat[5] += (unsigned long long)n * (unsigned long long)(w * EB + 4);
              }
            }
          }
        }
        // the row's tail norms after the level, a chunk ahead of their use
        const float* const tail = a.tails + (im.ch0 * (L + 1) + l + 1) * CH + row;
        auto tail_of = [&](uint32_t m) {
          return m ? __ldg(tail + (__ffs(m) - 1) * (L + 1) * CH) : 0.f;
        };
        float sx_n = tail_of(test);
        // Level 0's terms were set in the prologue.  At a level in between only
        // the query's tail norm changes: the threshold stays the item's first
        // one (an older threshold is a larger one: still valid), whose words
        // and terms were 4k of a tested level's cycles.  The last level takes
        // the threshold of the moment.
        if (l > 0 && l < L - 1 && l != first_test) {
          if (tid < QG && sh.qk[tid] > 0)
            sh.qterm.S[tid] = a.eps * a.qtail[(int64_t)sh.qid[tid] * (L + 1) + l + 1];
        } else if (l > 0 && tid < QG && sh.qk[tid] > 0) {
          const int q = sh.qid[tid];
          const unsigned long long key = kth_key<LARGE>(a.topk + (int64_t)q * a.k_max, sh.qk[tid]);
          const float tau = key == kEmptyKey ? INFINITY : __fmul_ru(key_dist(key), 1.000001f);
          set_query_terms(tid, fminf(tau, __ldcg(a.tau_seed + q)),
                          a.eps * a.qtail[(int64_t)q * (L + 1) + l + 1], sh.qterm);
        }
        if ((bad = epi_or(failed(fail)))) break;
        const QTerms& qt = sh.qterm;
#pragma unroll 1
        for (uint32_t m = test; m; m &= m - 1) {
          const int c = __ffs(m) - 1;
          const float sxc = sx_n;
          sx_n = tail_of(m & (m - 1));
          const float fr = FP8 ? a.xscale[(im.ch0 + c) * CH + row] : 1.f;
          const bool done = wait_or_fail(&sh.mma_bar[c], (mph >> c) & 1u, fail);
          mph ^= 1u << c;
          tc::fence_after_sync();
          uint32_t wm = sh.alive[c][half][row];
          const uint32_t any = __reduce_or_sync(0xffffffffu, done ? wm : 0u);
          if (any) {
            // 16 slots at a time (32 accumulators beside the terms spilled),
            // those that any of the warp's rows holds
            const float rx = sh.rx[c * CH + row], exv = sh.ex[c * CH + row];
            const float Hx = sh.Hx[c * CH + row];
            uint32_t pruned = 0;
#pragma unroll 1
            for (int h = 0; h < 32; h += 16) {
              if (!((any >> h) & 0xffffu)) continue;
              float v[16];
              tc::tmem_ld16(tbase + lane_base + (uint32_t)(c * QG + 32 * half + h), v);
              pruned |= pruned_bits(v, qt, 32 * half + h, sxc, rx, exv, Hx, fr) << h;
            }
            wm &= ~pruned;
            sh.alive[c][half][row] = wm;
          }
          if (l + 1 < L) {
            const unsigned bal = __ballot_sync(0xffffffffu, wm != 0);
            if (lane == 0) sh.rowlive[(tph >> c) & 1u][c][warp] = bal;
            // every lane's accumulator reads are complete before lane 0 tells
            // the MMA thread
            tc::fence_before_sync();
            __syncwarp();
            if (lane == 0) mbar_arrive_plain(&sh.tested[c]);
          } else if (__any_sync(0xffffffffu, wm != 0)) {
            // survivors per query
            for (uint32_t m = __reduce_or_sync(0xffffffffu, wm); m; m &= m - 1) {
              const int j = __ffs(m) - 1;
              const unsigned b = __ballot_sync(0xffffffffu, (wm >> j) & 1u);
              if (lane == 0) atomicAdd(&sh.scount[32 * half + j], __popc(b));
            }
          }
        }
        section(2);
        if (l + 1 >= L) break;
        // the outcome of the level's tests: lane c looks at chunk c
        bool ok = true;
        int n = 0;
        if (lane < S && ((test >> lane) & 1u)) {
          const uint32_t par = (tph >> lane) & 1u;
          ok = wait_or_fail(&sh.tested[lane], par, fail);
          n = live_rows(sh.rowlive[par][lane]);
        }
        __syncwarp();
        tph ^= test;
        // (after a failed wait `next` may be anything; the next barrier ends it)
        int next = L - 1;
        for (int c = 0; c < nch; ++c) {
          if ((test >> c) & 1u) cs.tested(a, c, l, __shfl_sync(0xffffffffu, n, c));
          if ((cs.live >> c) & 1u) next = min(next, cs.test_level(c));
        }
        if (!__all_sync(0xffffffffu, ok)) {
          bad = epi_or(true);
          break;
        }
        if (!cs.live) break;
        l = next;
      }
      if (bad) break;
      if (cs.live) {
        if ((bad = epi_or(failed(fail)))) break;
        // Last level done: where at least k candidates of the segment survive
        // for a query, their k-th smallest upper bound tightens its threshold
        // (at the last level UB ~ LB ~ exact) and the pairs are tested again,
        // so about k per query reach re-ranking.  Eight queries at a time; the
        // bounds are kept as bf16 rounded up (still upper bounds).
        bool tightened = false;
        for (int g0 = 0; g0 < G; g0 += UBQ) {
          bool need = false;
          for (int j = 0; j < UBQ; ++j)
            need |= sh.qk[g0 + j] > 0 && sh.scount[g0 + j] >= sh.qk[g0 + j];
          if (!need) continue;
          tightened = true;
          for (int c = half; c < S; c += 2) {
            const uint32_t wm =
                c < nch && ((cs.live >> c) & 1u) ? sh.alive[c][g0 >> 5][row] >> (g0 & 31) : 0u;
            float v[UBQ];
            const bool any_warp = __any_sync(0xffffffffu, (wm & 255u) != 0);
            if (any_warp) tc::tmem_ld8(tbase + lane_base + (uint32_t)(c * QG + g0), v);
            const int64_t slot_c = (im.ch0 + c) * CH + row;
            float nx = 0.f, fr = 1.f, rx = 0.f, exv = 0.f;
            if (wm & 255u) {
              nx = a.xn2[slot_c];
              if (FP8) fr = a.xscale[slot_c];
              rx = sh.rx[c * CH + row];
              exv = sh.ex[c * CH + row];
            }
#pragma unroll
            for (int j = 0; j < UBQ; ++j) {
              uint16_t u = 0x7f80u;
              if ((wm >> j) & 1u) {
                const int g = g0 + j;
                const float A = sh.qnq[g] + nx - 2.f * (FP8 ? (v[j] * fr) * sh.qs[g] : v[j]);
                const float Ss = sh.qrq[g] + rx;
                const float under = FP8 ? 2.f * sh.qun[g] * rx : 0.f;
                const float r = __fadd_ru(sqrt_up(fmaxf(A + fmaf(g_slack * Ss, Ss, under), 0.f)),
                                          sh.qeq[g] + exv);
                u = __bfloat16_as_ushort(
                    __float2bfloat16_ru(__fmul_ru(__fmul_ru(r, r), a.ub_scale)));
              }
              sh.ub[j][c * CH + row] = u;
            }
          }
          if ((bad = epi_or(failed(fail)))) break;
          const int g = g0 + warp;
          if (g < G && sh.qk[g] > 0 && sh.scount[g] >= sh.qk[g]) {
            const float t = warp_kth_smallest_bf16(sh.ub[warp], S * CH, sh.qk[g]);
            // k candidates with upper bounds <= t: a threshold for every later
            // work item of the query too
            if (lane == 0 && t < sh.qtau[g]) {
              sh.qtau[g] = t;
              atomicMin(reinterpret_cast<unsigned int*>(a.tau_seed) + sh.qid[g], __float_as_uint(t));
            }
          }
          if ((bad = epi_or(failed(fail)))) break;
        }
        if (bad) break;
        QTerms& qt = sh.qterm;
        if (tightened) {
          if (tid < G && sh.qk[tid] > 0) set_query_terms(tid, sh.qtau[tid], 0.f, qt);
          if ((bad = epi_or(failed(fail)))) break;
        }
        section(4);
        // survivors (of the test with the tightened threshold, C = 0 after
        // the last level) join the deferred re-rank list; a full list is checked and re-ranked by all warps at once.
        // Survivors are few: a warp walks the slots that any of its rows
        // holds and reads one accumulator column for each (code unrolled over
        // all 32 slots did not fit the instruction cache beside the rest).
        for (bool more = true; more;) {
          bool left = false;
          for (int c = 0; c < nch; ++c) {
            if (!((cs.live >> c) & 1u)) continue;
            uint32_t wm = sh.alive[c][half][row];
            uint32_t m = __reduce_or_sync(0xffffffffu, wm);
            if (!m) continue;
            const int64_t slot_c = (im.ch0 + c) * CH + row;
            const float rx = sh.rx[c * CH + row], exv = sh.ex[c * CH + row];
            const float fr = FP8 ? a.xscale[slot_c] : 1.f;
            for (; m; m &= m - 1) {
              const int j = __ffs(m) - 1, g = 32 * half + j;
              // (the lanes of the last slot's survivors rejoin; a full list
              // leaves the rest to the next round)
              if (__any_sync(0xffffffffu, *reinterpret_cast<volatile int*>(&sh.npend) >= kPend))
                break;
              float p = tc::tmem_ld1(tbase + lane_base + (uint32_t)(c * QG + g));
              if (!((wm >> j) & 1u)) continue;
              if (FP8) p = (p * fr) * sh.qs[g];
              if (tightened) {
                const float P = fmaf(qt.E[g], exv, fmaf(qt.G[g], rx, p));
                if (P < qt.H[g] + sh.Hx[c * CH + row]) {
                  wm &= ~(1u << j);
                  continue;
                }
              }
              const int pos = atomicAdd(&sh.npend, 1);
              if (pos >= kPend) continue;
              wm &= ~(1u << j);
              sh.pslot[pos] = slot_c;
              sh.pq[pos] = sh.qid[g];
              sh.plb[pos] = p;
            }
            sh.alive[c][half][row] = wm;
            left |= wm != 0;
          }
          tc::fence_before_sync();
          // (two barriers: a failed wait must not look like a survivor left)
          if ((bad = epi_or(failed(fail)))) break;
          more = epi_or(left);
          if (more) {
            const int nk = flush_pending<FP8, LARGE>(a, sh, kPend);
            if (nk < 0) {
              bad = true;
              break;
            }
            if (tid == 0) {
              if (a.collect) sh.stat[4] += nk;
              sh.npend = 0;
            }
            if ((bad = epi_or(failed(fail)))) break;
          }
        }
        if (bad) break;
        section(5);
      }
      // the accumulators and the item's slot are free
      tc::fence_before_sync();
      __syncwarp();
      if (lane == 0) {
        mbar_arrive_plain(&sh.acc_free);
        mbar_arrive_plain(&sh.item_empty[slot]);
      }
    }
    if (!bad) {  // the last deferred survivors
      const int np = sh.npend;
      const int nk = flush_pending<FP8, LARGE>(a, sh, np);
      if (tid == 0 && a.collect && nk > 0) sh.stat[4] += nk;
    }
  }
  __syncthreads();
  if (tid == 0 && sh.fail) atomicOr(a.err, kErrTimeout);
  if (a.collect && tid == 0) {
    sh.sec[6] = (unsigned long long)(clock64() - sh.tkernel);
    sh.sec[7] = 1;  // CTAs that ran
    for (int i = 0; i < 8; ++i) atomicAdd(&a.stats[8 + i], sh.sec[i]);
    if (a.phase == 0)
      for (int i = 0; i < 8; ++i) atomicAdd(&a.stats[16 + i], sh.sec[i]);
    atomicAdd(&a.stats[0], sh.stat[0]);
    atomicAdd(&a.stats[a.phase == 0 ? 6 : 7], sh.stat[1]);
    atomicAdd(&a.stats[1], sh.stat[2]);
    atomicAdd(&a.stats[2], sh.stat[3]);
    atomicAdd(&a.stats[3], sh.stat[4]);
    atomicAdd(&a.stats[25], sh.stat[5]);
  }
  tc::fence_before_sync();
  __syncthreads();
  if (warp == 0) tc::tmem_dealloc(tbase, TMEM_COLS);
}

}  // namespace

int launch_pack_bf16(const float* xt, const float* rows, const int64_t* perm, int64_t chunk0,
                     int64_t nchunks, int d, int L, const int32_t* level_off, const float* mu,
                     double c_trans, uint8_t* slices, float* tails, float* xn2, float* ex,
                     int32_t* ids, cudaStream_t st) {
  PANO_CHECK(d % 8 == 0 && d <= 8192, PANO_EINVAL, "bf16 storage needs d % 8 == 0, d <= 8192");
  pack_bf16_kernel<<<(unsigned)nchunks, 256, 0, st>>>(xt, rows, perm, chunk0, d, L, level_off,
                                                      mu, c_trans, slices, tails, xn2, ex, ids);
  PANO_CUDA(cudaGetLastError());
  return PANO_OK;
}

int launch_pack_fp8(const float* xt, const float* rows, const int64_t* perm, int64_t chunk0,
                    int64_t nchunks, int d, int L, const int32_t* level_off, const float* mu,
                    double c_trans, uint8_t* slices, float* tails, float* xn2, float* ex,
                    float* xscale, int32_t* ids, cudaStream_t st) {
  PANO_CHECK(d % 32 == 0 && d <= 8192, PANO_EINVAL, "fp8 storage needs d % 32 == 0, d <= 8192");
  pack_fp8_kernel<<<(unsigned)nchunks, 256, 0, st>>>(xt, rows, perm, chunk0, d, L, level_off, mu,
                                                     c_trans, slices, tails, xn2, ex, xscale, ids);
  PANO_CUDA(cudaGetLastError());
  return PANO_OK;
}

template <bool FP8>
constexpr size_t verify_tc_smem = 1024 + Ring<FP8, 1>::BYTES + sizeof(Shared);
static_assert(verify_tc_smem<false> <= 113 * 1024 && verify_tc_smem<true> <= 113 * 1024,
              "two CTAs per SM (228 KB, 1 KB of it reserved per CTA)");

int launch_verify_tc(const VerifyTCArgs& a, bool large, cudaStream_t st) {
  static PerDeviceOnce once;
  using Kernel = void (*)(VerifyTCArgs);
  // [format][unsorted slots above kChainK][panel rows of 128, 64 or 32 bytes at most]
  static const Kernel kernels[2][2][3] = {
      {{verify_tc_kernel<false, false, 1>, verify_tc_kernel<false, false, 2>,
        verify_tc_kernel<false, false, 4>},
       {verify_tc_kernel<false, true, 1>, verify_tc_kernel<false, true, 2>,
        verify_tc_kernel<false, true, 4>}},
      {{verify_tc_kernel<true, false, 1>, verify_tc_kernel<true, false, 2>,
        verify_tc_kernel<true, false, 4>},
       {verify_tc_kernel<true, true, 1>, verify_tc_kernel<true, true, 2>,
        verify_tc_kernel<true, true, 4>}}};
  PANO_CUDA(once.run([] {
    int dev = 0, optin = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess)
      e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    for (const auto& f : kernels)
      for (const auto& g : f)
        for (const Kernel k : g) {
          if (e == cudaSuccess)
            e = cudaFuncSetAttribute((const void*)k, cudaFuncAttributeMaxDynamicSharedMemorySize, optin);
          if (e == cudaSuccess)
            e = cudaFuncSetAttribute((const void*)k, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
        }
    return e;
  }));
  const size_t smem = a.fp8 ? verify_tc_smem<true> : verify_tc_smem<false>;
  int dev = 0, sms = 0;
  PANO_CUDA(cudaGetDevice(&dev));
  PANO_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  // the widest level an index may have (256 bytes a row)
  if (a.max_w > (a.fp8 ? 256 : 128))
    return fail(PANO_EINVAL, "tensor-core verify tile does not fit in shared memory");
  // Two CTAs x 256 TMEM columns fill an SM's tensor memory.  The grid is
  // not sized from the occupancy API: it reports the SM's current shared
  // memory carveout, which switches only when a launch asks for more.  A
  // persistent CTA that cannot be resident yet starts later and finds the
  // queue drained, so over-provisioning is harmless.
  const int rb = a.max_w * (a.fp8 ? 1 : 2);
  const Kernel kern = kernels[a.fp8 ? 1 : 0][large ? 1 : 0][rb >= 128 ? 0 : rb == 64 ? 1 : 2];
  kern<<<sms * 2, NT, smem, st>>>(a);
  PANO_CUDA(cudaGetLastError());
  return PANO_OK;
}

}  // namespace pano
