// Device helpers shared by the library's kernels: bulk-async (TMA engine)
// copies with mbarrier completion, bounded waits, (distance, id) keys and the
// two lock-free ways they enter a query's running top-k: chains through sorted
// slots, and replacement of the largest of unsorted ones.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace pano {

// Error bits written into the per-call device status word.
enum : int {
  kErrTimeout = 1,   // a bounded wait gave up
  kErrOverflow = 2,  // a capacity bound was exceeded (result still valid)
  kErrBadInput = 4,  // an out-of-range per-query value was clamped
};

// Roughly one second of spinning at GB300 clocks before a wait gives up.
constexpr long long kWaitCycles = 2000000000LL;

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)),
               "r"(count));
}

__device__ __forceinline__ void fence_mbar_init() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

__device__ __forceinline__ void fence_proxy_async_smem() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile(
      "mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)),
      "r"(bytes)
      : "memory");
}

// One bulk-async copy global -> shared completing on `bar` (TMA engine,
// non-tensor form).  dst, src and bytes must be multiples of 16.
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes,
                                         uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.shared::cta.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
          smem_u32(dst)),
      "l"(src), "r"(bytes), "r"(smem_u32(bar))
      : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
      " selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}

// Wait for phase `parity` of `bar`; false after ~kWaitCycles.
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t* bar, uint32_t parity) {
  if (mbar_try_wait(bar, parity)) return true;
  long long t0 = clock64();
  while (!mbar_try_wait(bar, parity)) {
    if (clock64() - t0 > kWaitCycles) return false;
  }
  return true;
}

// ------------------------------------------------------- (dist, id) keys
// Non-negative FP32 distances order like their bit patterns, so a 64-bit key
// (dist bits << 32 | id) orders by (distance, id).  The empty key is ~0.
constexpr unsigned long long kEmptyKey = ~0ULL;

__device__ __forceinline__ unsigned long long make_key(float dist, int32_t id) {
  dist = fmaxf(dist, 0.0f);
  return (static_cast<unsigned long long>(__float_as_uint(dist)) << 32) |
         static_cast<uint32_t>(id);
}
__device__ __forceinline__ float key_dist(unsigned long long k) {
  return __uint_as_float(static_cast<uint32_t>(k >> 32));
}
__device__ __forceinline__ int32_t key_id(unsigned long long k) {
  return static_cast<int32_t>(static_cast<uint32_t>(k & 0xffffffffULL));
}

__device__ __forceinline__ unsigned long long ld_volatile_u64(const unsigned long long* p) {
  return *reinterpret_cast<const volatile unsigned long long*>(p);
}

// Insert `key` into the ascending k-slot array `slots` shared by concurrent
// inserters.  Each step is an atomic compare-exchange between the carried
// key and one slot (atomicMin keeps the smaller, the larger moves on), so
// once all inserts have finished the slots hold the k smallest keys ever
// inserted, in ascending order.  A slot whose current value is already below
// the carried key would keep it, so those steps are skipped.
//
// By one thread: its slot reads go out in batches of eight
// independent loads (one round per eight slots, not one per slot), so that
// many threads can each insert a key at once and their compare-exchange
// chains overlap.  A read may be stale: slots only ever decrease, so the
// first slot found not below the key is never past the key's place, and
// starting early only adds steps that leave a slot unchanged.
__device__ __forceinline__ void topk_insert_thread(unsigned long long* slots, int k,
                                                   unsigned long long key) {
  int start = k;
  for (int j0 = 0; j0 < k && start == k; j0 += 8) {
    unsigned long long v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) v[u] = j0 + u < k ? ld_volatile_u64(slots + j0 + u) : kEmptyKey;
#pragma unroll
    for (int u = 7; u >= 0; --u)
      if (v[u] >= key) start = j0 + u;
  }
  for (int j = start; j < k; ++j) {
    unsigned long long old = atomicMin(slots + j, key);
    if (old == kEmptyKey || old == key) return;  // an equal key is the same pair: kept once
    key = old > key ? old : key;
  }
}

// The same by a whole warp: the slots are read once in parallel
// (one round instead of a chain of dependent reads) to find the first slot
// not below the key; lane 0 then runs the compare-exchange chain from there.
// All 32 lanes must call it with the same arguments.
__device__ __forceinline__ void topk_insert_warp(unsigned long long* slots, int k,
                                                 unsigned long long key) {
  const int lane = threadIdx.x & 31;
  int start = k;
  for (int j0 = 0; j0 < k; j0 += 32) {
    const int j = j0 + lane;
    const bool ge = j < k && ld_volatile_u64(slots + j) >= key;
    const unsigned m = __ballot_sync(0xffffffffu, ge);
    if (m) {
      start = j0 + __ffs(m) - 1;
      break;
    }
  }
  if (lane == 0)
    for (int j = start; j < k; ++j) {
      unsigned long long old = atomicMin(slots + j, key);
      if (old == kEmptyKey || old == key) return;  // an equal key is the same pair: kept once
      key = old > key ? old : key;
    }
}

// In a batch with unsorted slots (a rule on the host) a query with k above this
// keeps its slots unsorted: a new key replaces the largest one
// (topk_replace_warp), and its threshold lives in tau_seed alone.
// With sorted slots a key costs up to k dependent global atomics (about 0.7 us
// each); a replacement costs one round of loads and one of compare-exchanges
// for up to 32 keys of a query.  At k = 10 the chains of a flush end sooner (a
// warp takes its queries one after another); at k = 100 they were 84 % of the
// verify kernel (1.5M x 384 BF16, Zipf lists, 16,384 queries, k in {1, 10,
// 100}: 59 ms a search, 28 with a locked merge per flush, 20 so).  At k = 41
// and 256 to 1,024 queries both take about the same time (200k x 128 BF16, nprobe
// 8 of 128: 464 / 450 and 847 / 900 us a search).
constexpr int kChainK = 40;

// The k-th key of a query's sorted slots, kEmptyKey where they are unsorted.
template <bool LARGE>
__device__ __forceinline__ unsigned long long kth_key(const unsigned long long* slots, int k) {
  return !LARGE || k <= kChainK ? ld_volatile_u64(slots + k - 1) : kEmptyKey;
}

// Smallest / largest 64-bit value of the warp.
__device__ __forceinline__ unsigned long long warp_min_u64(unsigned long long v) {
  const uint32_t hi = __reduce_min_sync(0xffffffffu, (uint32_t)(v >> 32));
  const uint32_t lo =
      __reduce_min_sync(0xffffffffu, (uint32_t)(v >> 32) == hi ? (uint32_t)v : 0xffffffffu);
  return (unsigned long long)hi << 32 | lo;
}
__device__ __forceinline__ unsigned long long warp_max_u64(unsigned long long v) {
  const uint32_t hi = __reduce_max_sync(0xffffffffu, (uint32_t)(v >> 32));
  const uint32_t lo = __reduce_max_sync(0xffffffffu, (uint32_t)(v >> 32) == hi ? (uint32_t)v : 0u);
  return (unsigned long long)hi << 32 | lo;
}

// Enters up to 32 keys (one per lane, kEmptyKey = none) of one query into its
// k unsorted slots (k > kChainK); every lane of the warp calls it.  Once all
// concurrent calls have ended the slots hold the k smallest keys ever entered
// (an equal key is kept once).
//
// The slots are read (128 at most in registers; more in rounds, one key at a
// time), the keys ascending are given the slots descending while a key is
// below its slot, and all compare-exchanges go out at once; what fails (the
// slot was lowered meanwhile) is tried again on fresh slots.  A slot that is
// evicted while another one above it was refilled concurrently is no loss:
// slots only decrease, so at most as many slots above it remain as this call
// has smaller keys, each of which still takes the largest slot of its time or
// finds all slots below itself.
//
// The largest slot of what was read bounds the k-th distance from above (it can
// only have fallen since): tau, a pointer to the query's threshold, is lowered
// to it.
__device__ __forceinline__ void topk_replace_warp(unsigned long long* slots, int k,
                                                  unsigned long long key, float* tau) {
  const int lane = threadIdx.x & 31;
  while (true) {
    if (!__any_sync(0xffffffffu, key != kEmptyKey)) return;
    int at = -1;  // this lane's slot
    unsigned long long was = 0, top = 0;
    if (k <= 128) {
      unsigned long long v[4];
      bool dup = false;
#pragma unroll
      for (int r = 0; r < 4; ++r)
        v[r] = 32 * r + lane < k ? ld_volatile_u64(slots + 32 * r + lane) : 0ull;
      // (an absent slot reads 0: never the largest of distinct keys while k > 1.
      // It is also the key of id 0 at distance 0, so only slots that exist are
      // compared below.)
      for (uint32_t m = __ballot_sync(0xffffffffu, key != kEmptyKey); m; m &= m - 1) {
        const unsigned long long x = __shfl_sync(0xffffffffu, key, __ffs(m) - 1);
        bool same = false;
#pragma unroll
        for (int r = 0; r < 4; ++r) same |= (32 * r + lane < k) & (v[r] == x);
        if (__any_sync(0xffffffffu, same) && lane == __ffs(m) - 1) dup = true;
      }
      if (dup) key = kEmptyKey;  // the pair is held already
      bool left = key != kEmptyKey;
      while (true) {
        unsigned long long mx = v[0];
        int r = 0;
#pragma unroll
        for (int u = 1; u < 4; ++u)
          if (v[u] > mx) mx = v[u], r = u;
        top = warp_max_u64(mx);
        const unsigned long long x = warp_min_u64(left ? key : kEmptyKey);
        if (x >= top) break;
        const int owner = __ffs(__ballot_sync(0xffffffffu, mx == top)) - 1;
        const int slot = __shfl_sync(0xffffffffu, 32 * r + lane, owner);
        if (left && key == x) {  // (keys of one call are distinct: one lane)
          at = slot;
          was = top;
          left = false;
        }
        if (lane == owner) {
#pragma unroll
          for (int u = 0; u < 4; ++u)
            if (u == r) v[u] = x;
        }
      }
      if (left) key = kEmptyKey;  // not below any slot
    } else {
      // the largest slot, for the smallest key
      unsigned long long mx = 0, x = warp_min_u64(key);
      int i_mx = 0;
      bool same = false;
      for (int i = lane; i < k; i += 32) {
        const unsigned long long v = ld_volatile_u64(slots + i);
        same |= v == x;
        if (v > mx) mx = v, i_mx = i;
      }
      top = warp_max_u64(mx);
      const int owner = __ffs(__ballot_sync(0xffffffffu, mx == top)) - 1;
      const int slot = __shfl_sync(0xffffffffu, i_mx, owner);
      if (__any_sync(0xffffffffu, same)) {
        if (key == x) key = kEmptyKey;
        continue;
      }
      if (x >= top) return;
      if (key == x) {
        at = slot;
        was = top;
      }
    }
    if (top != kEmptyKey && lane == 0)
      atomicMin(reinterpret_cast<unsigned int*>(tau),
                __float_as_uint(__fmul_ru(key_dist(top), 1.000001f)));
    if (at >= 0 && atomicCAS(slots + at, was, key) == was) key = kEmptyKey;
    // a lost exchange: many warps are after the same slots; spread them out
    if (__any_sync(0xffffffffu, at >= 0 && key != kEmptyKey))
      __nanosleep(200 + ((uint32_t)clock64() & 1023u));
  }
}

// Enters the flush's pairs into their queries' top-k: entry i < n is pair
// list[i], its distance dist[], id pid[] and query pq[].  Called by all
// `nthreads` threads of the flush (tid 0 .. nthreads - 1, n <= nthreads),
// between barriers.  LARGE = false: all slots of the batch are sorted.
template <bool LARGE>
__device__ __forceinline__ void topk_flush_insert(unsigned long long* topk, int k_max,
                                                  const int32_t* __restrict__ kq, float* tau_seed,
                                                  const uint16_t* list, int n, const int32_t* pq,
                                                  const float* dist, const int32_t* pid,
                                                  int nthreads) {
  const int tid = threadIdx.x, lane = tid & 31;
  if (tid < n) {
    const int s = list[tid], q = pq[s], k = kq[q];
    if (!LARGE || k <= kChainK)
      topk_insert_thread(topk + (int64_t)q * k_max, k, make_key(dist[s], pid[s]));
  }
  if (!LARGE) return;
  __syncwarp();
  for (int i = tid >> 5; i < n; i += nthreads >> 5) {
    const int q = pq[list[i]], k = kq[q];
    if (k <= kChainK) continue;
    // the warp of a query's first entry gathers all of its entries, 32 at a
    // time (one call site: inlined where it is used, so that the flush makes
    // no nested call, which cost the level loop registers)
    bool mine = true;
    int run = 0;
    for (int base = 0; mine && (base == 0 || base < run); base += 32) {
      unsigned long long key = kEmptyKey;
      run = 0;
      for (int o0 = 0; o0 < n && mine; o0 += 32) {
        const int o = o0 + lane;
        const uint32_t b = __ballot_sync(0xffffffffu, o < n && pq[list[o]] == q);
        if (o0 < i && (b & (i - o0 >= 32 ? 0xffffffffu : (1u << (i - o0)) - 1u))) mine = false;
        for (uint32_t m = b; m; m &= m - 1, ++run)
          if (lane == run - base) {
            const int s = list[o0 + __ffs(m) - 1];
            key = make_key(dist[s], pid[s]);
          }
      }
      if (mine) topk_replace_warp(topk + (int64_t)q * k_max, k, key, tau_seed + q);
    }
  }
}

// Hint that `bytes` (a multiple of 16, 16-byte aligned) at p will be read
// soon: a bulk prefetch into L2 (no completion to wait for).
__device__ __forceinline__ void prefetch_l2(const void* p, uint32_t bytes) {
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(bytes) : "memory");
}

// sqrt(x) rounded up, for x >= 0 where only an upper bound is needed: the
// approximate square root (sqrt.approx.f32, whose relative error is a few
// units of 2^-23) times 1 + 2^-18, rounded up.  One multiply on top of the
// approximation, against the longer sequence of the IEEE directed-rounding
// square root.  Inputs below 2^-126 (zero and subnormals) are raised to it,
// so the result there is 2^-63 (times 1 + 2^-18), still an upper bound.
// panorama_debug_sqrt_up exposes it so that a test checks the bound against
// FP64 over the whole range.
__device__ __forceinline__ float sqrt_up(float x) {
  float r;
  asm("sqrt.approx.f32 %0, %1;" : "=f"(r) : "f"(fmaxf(x, 0x1p-126f)));
  return __fmul_ru(r, 1.0f + 0x1p-18f);
}

// Order-preserving map of any FP32 value to uint32.
__device__ __forceinline__ uint32_t float_ordered(float f) {
  uint32_t u = __float_as_uint(f);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

}  // namespace pano
