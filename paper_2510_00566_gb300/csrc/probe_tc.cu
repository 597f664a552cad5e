// Coarse-probe distances on the tensor cores (Section 6.1: a query probes its
// nprobe nearest IVF lists).  pd[q][c] = |q|^2 + |c|^2 - 2 q.c for a tile of
// 128 queries x 256 centroids per CTA; the dot products are three bf16
// tcgen05 MMAs per K-step (hi.hi + hi.lo + lo.hi of each operand's bf16 hi +
// lo split), accumulated in FP32 in tensor memory.  The probe selection
// re-scores exactly every centroid within the error bound of the nprobe-th
// (probe_tc_gerr), so the probe sets are those of exact distances.  The same
// products give a build the nearest centroid of every vector (assign_tc).
//
// The centroids' split is laid out once per index (cent_image): per tile of 256
// centroids and K panel of 64 the swizzled hi and lo operand images, 64 KB that
// one bulk copy brings in.  (Each CTA used to convert its 256 centroid rows
// itself, twice the work of its 128 queries: 10,000 x 1,024 x 960 took 296 us,
// now 109.)
#include <cuda_bf16.h>

#include <algorithm>

#include "internal.h"
#include "kernels_common.cuh"
#include "probe_tc.h"
#include "tcgen05.cuh"

namespace pano {
namespace {

constexpr int PM = 128;   // queries per tile (MMA M)
constexpr int PN = 256;   // centroids per tile (MMA N)
constexpr int PK = 64;    // K elements per panel (one 128-byte swizzled row)
constexpr int PT = 256;   // threads
constexpr int A_BYTES = PM * PK * 2, B_BYTES = PN * PK * 2;
constexpr int STAGE = 2 * A_BYTES + 2 * B_BYTES;  // A hi, A lo, B hi, B lo

__device__ __forceinline__ void split2(float x, __nv_bfloat16& hi, __nv_bfloat16& lo) {
  hi = __float2bfloat16_rn(x);
  lo = __float2bfloat16_rn(x - __bfloat162float(hi));
}

// Rows [r0, r0 + nr) of a row-major FP32 matrix (row length d), K panel p,
// as bf16 hi and lo tiles of R rows in the swizzled K-major image (rows
// past nr and elements past d are zeros).  A thread's loads all go out before
// the first conversion (one after another they were most of a panel's time).
// vec: 16-byte loads (d % 8 == 0 and src 16-byte aligned).
template <int R>
__device__ __forceinline__ void stage_rows(const float* __restrict__ src, int64_t r0, int nr,
                                           int d, int p, bool vec, unsigned char* hi,
                                           unsigned char* lo) {
  constexpr int kIter = R * (PK / 8) / PT, kBatch = 4;
  static_assert(R * (PK / 8) % PT == 0 && kIter % kBatch == 0, "whole rounds");
  const int c8 = threadIdx.x % (PK / 8), rr = threadIdx.x / (PK / 8);
  const int k0 = p * PK + c8 * 8;
#pragma unroll 1
  for (int i0 = 0; i0 < kIter; i0 += kBatch) {
    float f[kBatch][8];
#pragma unroll
    for (int u = 0; u < kBatch; ++u) {
      const int r = rr + (i0 + u) * (PT / (PK / 8));
      if (vec) {
        const bool in = r < nr && k0 < d;  // (d % 8 == 0: whole groups)
        const float4* s4 = reinterpret_cast<const float4*>(src + (r0 + r) * (int64_t)d + k0);
        const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
        const float4 a = in ? __ldg(s4) : z, b = in ? __ldg(s4 + 1) : z;
        f[u][0] = a.x, f[u][1] = a.y, f[u][2] = a.z, f[u][3] = a.w;
        f[u][4] = b.x, f[u][5] = b.y, f[u][6] = b.z, f[u][7] = b.w;
      } else {
#pragma unroll
        for (int j = 0; j < 8; ++j)
          f[u][j] = (r < nr && k0 + j < d) ? __ldg(src + (r0 + r) * (int64_t)d + k0 + j) : 0.f;
      }
    }
#pragma unroll
    for (int u = 0; u < kBatch; ++u) {
      const int r = rr + (i0 + u) * (PT / (PK / 8));
      __align__(16) __nv_bfloat16 h[8], l[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) split2(f[u][j], h[j], l[j]);
      const uint32_t off = tc::swz_offset(r, c8 * 8, R, PK);
      *reinterpret_cast<uint4*>(hi + off) = *reinterpret_cast<const uint4*>(h);
      *reinterpret_cast<uint4*>(lo + off) = *reinterpret_cast<const uint4*>(l);
    }
  }
}

// One CTA per (K panel, tile): the operand images of 256 centroids.
__global__ void __launch_bounds__(PT) cent_image_kernel(const float* __restrict__ C, int nlist,
                                                        int d, unsigned char* __restrict__ img) {
  unsigned char* out = img + ((size_t)blockIdx.y * gridDim.x + blockIdx.x) * (2 * B_BYTES);
  const int c0 = blockIdx.y * PN;
  stage_rows<PN>(C, c0, min(PN, nlist - c0), d, blockIdx.x,
                 (d & 7) == 0 && (reinterpret_cast<uintptr_t>(C) & 15) == 0, out, out + B_BYTES);
}

__global__ void __launch_bounds__(PT, 1) probe_tc_kernel(const float* __restrict__ Q, int64_t nq,
                                                         const unsigned char* __restrict__ cimg,
                                                         int nlist, int d,
                                                         const float* __restrict__ qn2,
                                                         const float* __restrict__ cn2,
                                                         float* __restrict__ pd, int* __restrict__ err,
                                                         bool vq) {
  extern __shared__ unsigned char smem_raw[];
  unsigned char* base = smem_raw + ((1024 - (smem_u32(smem_raw) & 1023)) & 1023);
  __shared__ __align__(8) uint64_t done[2], full[2];
  __shared__ uint32_t tmem_base;
  __shared__ int s_fail;
  const int tid = threadIdx.x, warp = tid / 32, lane = tid & 31;
  const int64_t q0 = (int64_t)blockIdx.y * PM;
  const int c0 = blockIdx.x * PN;
  const int nr_q = nq - q0 < PM ? (int)(nq - q0) : PM;
  const int nr_c = nlist - c0 < PN ? nlist - c0 : PN;
  const int N = (nr_c + 15) & ~15;  // MMA N: a multiple of 16
  if (warp == 0) {
    tc::tmem_alloc(&tmem_base, PN);
    tc::tmem_relinquish();
  }
  if (tid == 0) {
    mbar_init(&done[0], 1);
    mbar_init(&done[1], 1);
    mbar_init(&full[0], 1);
    mbar_init(&full[1], 1);
    fence_mbar_init();
    s_fail = 0;
  }
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tbase = tmem_base;
  const uint32_t idesc = tc::idesc_bf16(PM, N);
  const int np = (d + PK - 1) / PK;
  uint32_t dpar = 0;
  for (int p = 0; p < np; ++p) {
    const int s = p & 1;
    unsigned char* st = base + (size_t)s * STAGE;
    if (p >= 2) {  // the MMAs that read this stage two panels ago are done
      if (!mbar_wait_bounded(&done[s], (dpar >> s) & 1u)) atomicOr(&s_fail, 1);
      dpar ^= 1u << s;
    }
    if (tid == 0) {
      mbar_arrive_expect_tx(&full[s], 2 * B_BYTES);
      bulk_g2s(st + 2 * A_BYTES, cimg + ((size_t)blockIdx.x * np + p) * (2 * B_BYTES), 2 * B_BYTES,
               &full[s]);
    }
    stage_rows<PM>(Q, q0, nr_q, d, p, vq, st, st + A_BYTES);
    fence_proxy_async_smem();
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    if (tid == 0) {
      if (!mbar_wait_bounded(&full[s], (p >> 1) & 1)) atomicOr(&s_fail, 1);
      const uint64_t ah = tc::smem_desc(smem_u32(st), 128);
      const uint64_t al = tc::smem_desc(smem_u32(st + A_BYTES), 128);
      const uint64_t bh = tc::smem_desc(smem_u32(st + 2 * A_BYTES), 128);
      const uint64_t bl = tc::smem_desc(smem_u32(st + 2 * A_BYTES + B_BYTES), 128);
      for (int k = 0; k < PK / 16; ++k) {
        const uint64_t o = tc::kstep_off(k, 0);  // within the panel's one 128-byte row
        tc::mma_bf16(tbase, ah + o, bh + o, idesc, (p > 0 || k > 0) ? 1u : 0u);
        tc::mma_bf16(tbase, ah + o, bl + o, idesc, 1u);
        tc::mma_bf16(tbase, al + o, bh + o, idesc, 1u);
      }
      tc::mma_commit(&done[s]);
    }
  }
  // the last panel's commit covers every MMA of the tile
  {
    const int s = (np - 1) & 1;
    if (!mbar_wait_bounded(&done[s], (dpar >> s) & 1u)) atomicOr(&s_fail, 1);
  }
  tc::fence_after_sync();
  // epilogue: warp w reads TMEM lanes 32 (w % 4) .. (its 32 queries) and
  // columns 128 (w / 4) .. + 127
  const int row = (warp & 3) * 32 + lane;
  const uint32_t lane_base = (uint32_t)((warp & 3) * 32) << 16;
  const int col0 = (warp >> 2) * 128;
  const bool ok = __all_sync(0xffffffffu, s_fail == 0);
  if (ok && col0 < N) {
    const int64_t q = q0 + row;
    const float qn = row < nr_q ? qn2[q] : 0.f;
    for (int cb = col0; cb < col0 + 128 && cb < N; cb += 16) {
      float v[16];
      tc::tmem_ld16(tbase + lane_base + (uint32_t)cb, v);
      if (row < nr_q) {
        float* out = pd + q * (int64_t)nlist + c0 + cb;
        if (cb + 16 <= nr_c && ((c0 + cb) & 3) == 0 && (nlist & 3) == 0) {
#pragma unroll
          for (int j = 0; j < 16; j += 4) {
            float4 o;
            o.x = fmaf(-2.f, v[j], qn + __ldg(cn2 + c0 + cb + j));
            o.y = fmaf(-2.f, v[j + 1], qn + __ldg(cn2 + c0 + cb + j + 1));
            o.z = fmaf(-2.f, v[j + 2], qn + __ldg(cn2 + c0 + cb + j + 2));
            o.w = fmaf(-2.f, v[j + 3], qn + __ldg(cn2 + c0 + cb + j + 3));
            *reinterpret_cast<float4*>(out + j) = o;
          }
        } else {
#pragma unroll
          for (int j = 0; j < 16; ++j)
            if (cb + j < nr_c) out[j] = fmaf(-2.f, v[j], qn + __ldg(cn2 + c0 + cb + j));
        }
      }
    }
  }
  if (tid == 0 && s_fail) atomicOr(err, kErrTimeout);
  tc::fence_before_sync();
  __syncthreads();
  if (warp == 0) tc::tmem_dealloc(tbase, PN);
}

// The kBest nearest centroids, by the expansion distance without |x|^2, of each
// of a CTA's 128 rows in each of two halves of every centroid tile (row r's
// two threads each scan 128 of a tile's 256 columns): keys (ordered distance
// << 32 | id) ascending, best[row][half][kBest].
// (With four, the rows that had to be compared with every centroid because a
// half's last was within the bound, one in a thousand, were most of the pick.)
constexpr int kBest = 6;
static_assert(2 * kBest == kAssignWords && 2 * kBest <= 32, "a lane per key");

// The distance in a key.
__device__ __forceinline__ float expansion_of(unsigned long long key) {
  const uint32_t o = (uint32_t)(key >> 32);
  return __uint_as_float((o & 0x80000000u) ? (o & 0x7fffffffu) : ~o);
}

__global__ void __launch_bounds__(PT, 1) assign_tc_kernel(
    const float* __restrict__ X, int64_t m, const unsigned char* __restrict__ cimg, int nlist, int d,
    const float* __restrict__ cn2, unsigned long long* __restrict__ best, int* __restrict__ err,
    bool vx) {
  extern __shared__ unsigned char smem_raw[];
  unsigned char* base = smem_raw + ((1024 - (smem_u32(smem_raw) & 1023)) & 1023);
  __shared__ __align__(8) uint64_t done[2], full[2];
  __shared__ uint32_t tmem_base;
  __shared__ int s_fail;
  const int tid = threadIdx.x, warp = tid / 32, lane = tid & 31;
  const int64_t r0 = (int64_t)blockIdx.x * PM;
  const int nr = m - r0 < PM ? (int)(m - r0) : PM;
  if (warp == 0) {
    tc::tmem_alloc(&tmem_base, PN);
    tc::tmem_relinquish();
  }
  if (tid == 0) {
    for (int i = 0; i < 2; ++i) {
      mbar_init(&done[i], 1);
      mbar_init(&full[i], 1);
    }
    fence_mbar_init();
    s_fail = 0;
  }
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tbase = tmem_base;
  const int np = (d + PK - 1) / PK;
  const int row = (warp & 3) * 32 + lane, half = warp >> 2;
  const uint32_t lane_base = (uint32_t)((warp & 3) * 32) << 16;
  unsigned long long b[kBest];
#pragma unroll
  for (int i = 0; i < kBest; ++i) b[i] = kEmptyKey;
  float worst = INFINITY;
  uint32_t dpar = 0, it = 0;  // panels of all tiles run through the two stages
  for (int c0 = 0; c0 < nlist; c0 += PN) {
    const int nc = nlist - c0 < PN ? nlist - c0 : PN, N = (nc + 15) & ~15;
    const uint32_t idesc = tc::idesc_bf16(PM, N);
    for (int p = 0; p < np; ++p, ++it) {
      const int s = it & 1;
      unsigned char* st = base + (size_t)s * STAGE;
      if (it >= 2) {  // the MMAs that read this stage two panels ago are done
        if (!mbar_wait_bounded(&done[s], (dpar >> s) & 1u)) atomicOr(&s_fail, 1);
        dpar ^= 1u << s;
      }
      if (tid == 0) {
        mbar_arrive_expect_tx(&full[s], 2 * B_BYTES);
        bulk_g2s(st + 2 * A_BYTES, cimg + ((size_t)(c0 / PN) * np + p) * (2 * B_BYTES), 2 * B_BYTES,
                 &full[s]);
      }
      stage_rows<PM>(X, r0, nr, d, p, vx, st, st + A_BYTES);
      fence_proxy_async_smem();
      tc::fence_before_sync();
      // (and the last tile's accumulators have been read)
      const int failed = __syncthreads_or(s_fail);
      tc::fence_after_sync();
      if (failed) {  // no copy may be in flight when the CTA ends
        mbar_wait_bounded(&full[s], (it >> 1) & 1u);
        c0 = nlist;
        break;
      }
      if (tid == 0) {
        if (!mbar_wait_bounded(&full[s], (it >> 1) & 1u)) atomicOr(&s_fail, 1);
        const uint64_t ah = tc::smem_desc(smem_u32(st), 128);
        const uint64_t al = tc::smem_desc(smem_u32(st + A_BYTES), 128);
        const uint64_t bh = tc::smem_desc(smem_u32(st + 2 * A_BYTES), 128);
        const uint64_t bl = tc::smem_desc(smem_u32(st + 2 * A_BYTES + B_BYTES), 128);
        for (int k = 0; k < PK / 16; ++k) {
          const uint64_t o = tc::kstep_off(k, 0);
          tc::mma_bf16(tbase, ah + o, bh + o, idesc, (p > 0 || k > 0) ? 1u : 0u);
          tc::mma_bf16(tbase, ah + o, bl + o, idesc, 1u);
          tc::mma_bf16(tbase, al + o, bh + o, idesc, 1u);
        }
        tc::mma_commit(&done[s]);
      }
    }
    if (c0 >= nlist) break;
    // the tile's last commit (its phase is waited for again before the stage's
    // reuse: the same one, already complete)
    if (!mbar_wait_bounded(&done[(it - 1) & 1], (dpar >> ((it - 1) & 1)) & 1u)) atomicOr(&s_fail, 1);
    tc::fence_after_sync();
    for (int cb = 128 * half; cb < 128 * half + 128 && cb < N; cb += 16) {
      float v[16];
      tc::tmem_ld16(tbase + lane_base + (uint32_t)cb, v);
      // sixteen distances and their least; few batches hold one below the
      // row's kBest-th (ids ascend, so an equal one never enters)
      float least = INFINITY;
      const bool whole = c0 + cb + 16 <= nlist;
#pragma unroll
      for (int j = 0; j < 16; j += 4) {
        float4 n4 = make_float4(INFINITY, INFINITY, INFINITY, INFINITY);
        if (whole) {  // (c0 + cb is a multiple of 16)
          n4 = __ldg(reinterpret_cast<const float4*>(cn2 + c0 + cb + j));
        } else {
          if (c0 + cb + j < nlist) n4.x = __ldg(cn2 + c0 + cb + j);
          if (c0 + cb + j + 1 < nlist) n4.y = __ldg(cn2 + c0 + cb + j + 1);
          if (c0 + cb + j + 2 < nlist) n4.z = __ldg(cn2 + c0 + cb + j + 2);
          if (c0 + cb + j + 3 < nlist) n4.w = __ldg(cn2 + c0 + cb + j + 3);
        }
        v[j] = fmaf(-2.f, v[j], n4.x);
        v[j + 1] = fmaf(-2.f, v[j + 1], n4.y);
        v[j + 2] = fmaf(-2.f, v[j + 2], n4.z);
        v[j + 3] = fmaf(-2.f, v[j + 3], n4.w);
        least = fminf(least, fminf(fminf(v[j], v[j + 1]), fminf(v[j + 2], v[j + 3])));
      }
      if (!(least < worst)) continue;
#pragma unroll
      for (int j = 0; j < 16; ++j) {
        if (!(v[j] < worst)) continue;
        b[kBest - 1] = (unsigned long long)float_ordered(v[j]) << 32 | (uint32_t)(c0 + cb + j);
#pragma unroll
        for (int i = kBest - 1; i > 0; --i)
          if (b[i] < b[i - 1]) {
            const unsigned long long t = b[i];
            b[i] = b[i - 1];
            b[i - 1] = t;
          }
        if (b[kBest - 1] != kEmptyKey) worst = expansion_of(b[kBest - 1]);
      }
    }
    tc::fence_before_sync();
  }
  if (row < nr) {
#pragma unroll
    for (int i = 0; i < kBest; ++i) best[((r0 + row) * 2 + half) * kBest + i] = b[i];
  }
  __syncthreads();
  if (tid == 0 && s_fail) atomicOr(err, kErrTimeout);
  if (warp == 0) tc::tmem_dealloc(tbase, PN);
}

// The nearest centroid of each row (one warp per row): the smallest expansion
// distance unless others lie within twice its error bound of it; those are
// compared by the compensated difference form (ties to the lower id).  Where a
// half's kBest-th is within the bound there may be more: every centroid is
// compared.
__global__ void __launch_bounds__(256) assign_pick_kernel(
    const float* __restrict__ X, int64_t m, int d, const float* __restrict__ C, int nlist,
    float cmax, const unsigned long long* __restrict__ best, float gerr, int32_t* __restrict__ out) {
  const int64_t row = (int64_t)blockIdx.x * 8 + threadIdx.x / 32;
  const int lane = threadIdx.x & 31;
  if (row >= m) return;
  const float* x = X + row * d;
  const unsigned long long key = lane < 2 * kBest ? best[row * 2 * kBest + lane] : kEmptyKey;
  const unsigned long long first = warp_min_u64(key);
  float n2 = 0.f;
  for (int j = lane; j < d; j += 32) n2 = fmaf(x[j], x[j], n2);
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) n2 += __shfl_xor_sync(0xffffffffu, n2, off);
  const float s = sqrtf(n2) * 1.0001f + cmax;  // (the sum's rounding is far below 1e-4)
  const float hi = expansion_of(first) + 2.f * gerr * s * s * 1.0001f;
  const uint32_t near = __ballot_sync(0xffffffffu, key != kEmptyKey && expansion_of(key) <= hi);
  // A norm beyond FP32 (or NaN) makes the expansion the same for every centroid:
  // the lowest id, as from the FP32 products; so too where no key was kept.
  int choice = first == kEmptyKey || !(n2 < INFINITY) ? 0 : (int)(uint32_t)first;
  if (n2 < INFINITY && (near & (near - 1))) {
    float e = INFINITY;
    int c = nlist;
    auto look = [&](int ci) {
      const float ei = exact_sqdist_warp(x, C + (int64_t)ci * d, d);
      if (ei < e || (ei == e && ci < c)) e = ei, c = ci;
    };
    if (near & ((1u << (kBest - 1)) | (1u << (2 * kBest - 1)))) {
      for (int ci = 0; ci < nlist; ++ci) look(ci);
    } else {
      for (uint32_t k = near; k; k &= k - 1)
        look((int)(uint32_t)__shfl_sync(0xffffffffu, key, __ffs(k) - 1));
    }
    if (c < nlist) choice = c;  // (no distance compares where a centroid is not finite)
  }
  if (lane == 0) out[row] = choice;
}

}  // namespace

bool probe_tc_supported(int d) { return d >= 8 && d % 8 == 0; }

double probe_tc_gerr(int d) {
  // |pd - exact| <= gerr (|q| + |c|)^2: the dot product loses at most
  // 3 2^-16 sum |q_j c_j| to the split (two splits of 2^-16 each, and the
  // dropped lo.lo product) and 2^-20 of the running sum of |products| per
  // MMA (3 d / 16 MMAs; the accumulation model the verify path uses), with
  // sum |q_j c_j| <= |q| |c| <= (|q| + |c|)^2 / 4; it enters pd twice; the
  // epilogue's two roundings add 2 u of |q|^2 + |c|^2 + 2 |q.c|.  Factor 2
  // of safety on those.
  // The query and centroid norms may come from plain FP32 sums: gamma_{d+4}
  // of |q|^2 + |c|^2 <= (|q| + |c|)^2 covers them.
  const double dot = 3.0 * std::ldexp(1.0, -16) + (3.0 * std::ceil(d / 16.0)) * std::ldexp(1.0, -20);
  return 2.0 * (2.0 * dot / 4.0 + 2.0 * std::ldexp(1.0, -24)) + gamma_n(d + 4);
}

size_t cent_image_bytes(int nlist, int d) {
  return (size_t)((nlist + PN - 1) / PN) * ((d + PK - 1) / PK) * (2 * B_BYTES);
}

int build_cent_image(pano_index& I, cudaStream_t st) {
  if (!probe_tc_supported(I.d)) return PANO_OK;
  if (int rc = I.cent_img.alloc(cent_image_bytes(I.nlist, I.d))) return rc;
  const dim3 grid((unsigned)((I.d + PK - 1) / PK), (unsigned)((I.nlist + PN - 1) / PN));
  cent_image_kernel<<<grid, PT, 0, st>>>(I.cent.as<float>(), I.nlist, I.d,
                                         I.cent_img.as<unsigned char>());
  PANO_CUDA(cudaGetLastError());
  return PANO_OK;
}

int launch_probe_tc(const float* Q, int64_t nq, const pano_index& I, const float* qn2, float* pd,
                    int* err, cudaStream_t st) {
  static PerDeviceOnce once;
  const int nlist = I.nlist, d = I.d;
  const size_t smem = (size_t)2 * STAGE + 1024;
  PANO_CUDA(once.run([smem] {
    return cudaFuncSetAttribute((const void*)probe_tc_kernel,
                                cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  }));
  if (nq <= 0 || nlist <= 0) return PANO_OK;
  const dim3 grid((unsigned)((nlist + PN - 1) / PN), (unsigned)((nq + PM - 1) / PM));
  const bool vq = (d & 7) == 0 && (reinterpret_cast<uintptr_t>(Q) & 15) == 0;
  probe_tc_kernel<<<grid, PT, smem, st>>>(Q, nq, I.cent_img.as<unsigned char>(), nlist, d, qn2,
                                          I.cent_n2.as<float>(), pd, err, vq);
  PANO_CUDA(cudaGetLastError());
  return PANO_OK;
}

int launch_assign_tc(const float* X, int64_t m, const pano_index& I, unsigned long long* best,
                     int32_t* out, int* err, cudaStream_t st) {
  static PerDeviceOnce once;
  const int d = I.d, nlist = I.nlist;
  const size_t smem = (size_t)2 * STAGE + 1024;
  PANO_CUDA(once.run([smem] {
    return cudaFuncSetAttribute((const void*)assign_tc_kernel,
                                cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  }));
  if (m <= 0) return PANO_OK;
  const bool vx = (d & 7) == 0 && (reinterpret_cast<uintptr_t>(X) & 15) == 0;
  assign_tc_kernel<<<(unsigned)((m + PM - 1) / PM), PT, smem, st>>>(
      X, m, I.cent_img.as<unsigned char>(), nlist, d, I.cent_n2.as<float>(), best, err, vx);
  PANO_CUDA(cudaGetLastError());
  float gerr = (float)probe_tc_gerr(d);
  if ((double)gerr < probe_tc_gerr(d)) gerr = std::nextafter(gerr, INFINITY);
  assign_pick_kernel<<<(unsigned)((m + 7) / 8), 256, 0, st>>>(X, m, d, I.cent.as<float>(), nlist,
                                                             I.cmax, best, gerr, out);
  PANO_CUDA(cudaGetLastError());
  return PANO_OK;
}

}  // namespace pano
