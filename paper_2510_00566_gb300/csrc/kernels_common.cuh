// Warp-level helpers shared by the build and search kernels.
#pragma once

#include "device_common.cuh"

namespace pano {

__device__ __forceinline__ void kahan_add(float t, float& s, float& c) {
  float y = t - c;
  float u = s + y;
  c = (u - s) - y;
  s = u;
}

// Exact-as-FP32-allows squared distance sum_j (a_j - b_j)^2 by one warp:
// each lane keeps a Kahan-compensated sum (s, c) of its terms (the value is
// s - c); lanes are combined pairwise with an error-free TwoSum of the s
// parts.  Relative error a few FP32 units (compensated summation), far below
// the plain d-term sum's d*u.  Loads are issued in batches (several 16-byte
// loads in flight per lane) so the latency is paid a few times per row, not
// once per element.  Every lane returns the result.
__device__ __forceinline__ float exact_sqdist_warp(const float* __restrict__ a,
                                                   const float* __restrict__ b, int d) {
  const int lane = threadIdx.x & 31;
  float s = 0.f, c = 0.f;
  const bool vec = ((d & 3) == 0) && ((reinterpret_cast<uintptr_t>(a) & 15) == 0) &&
                   ((reinterpret_cast<uintptr_t>(b) & 15) == 0);
  if (vec) {
    const float4* a4 = reinterpret_cast<const float4*>(a);
    const float4* b4 = reinterpret_cast<const float4*>(b);
    const int d4 = d >> 2;
    for (int j0 = 0; j0 < d4; j0 += 4 * 32) {
      float4 av[4], bv[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int j = j0 + lane + 32 * u;
        av[u] = j < d4 ? a4[j] : make_float4(0.f, 0.f, 0.f, 0.f);
        bv[u] = j < d4 ? b4[j] : make_float4(0.f, 0.f, 0.f, 0.f);
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        float t;
        t = av[u].x - bv[u].x;
        kahan_add(t * t, s, c);
        t = av[u].y - bv[u].y;
        kahan_add(t * t, s, c);
        t = av[u].z - bv[u].z;
        kahan_add(t * t, s, c);
        t = av[u].w - bv[u].w;
        kahan_add(t * t, s, c);
      }
    }
  } else {
    for (int j0 = 0; j0 < d; j0 += 8 * 32) {
      float av[8], bv[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int j = j0 + lane + 32 * u;
        av[u] = j < d ? a[j] : 0.f;
        bv[u] = j < d ? b[j] : 0.f;
      }
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const float t = av[u] - bv[u];
        kahan_add(t * t, s, c);
      }
    }
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    float s2 = __shfl_xor_sync(0xffffffffu, s, off);
    float c2 = __shfl_xor_sync(0xffffffffu, c, off);
    float sum = s + s2;
    float bb = sum - s;
    float err = (s - (sum - bb)) + (s2 - bb);
    c = (c + c2) - err;
    s = sum;
  }
  return s - c;
}

// exact_sqdist_warp with the row fetched in batches of 8 float4 per lane per
// operand (one round of loads for d <= 1024) and two interleaved compensated
// sums per lane (half the dependent chain), combined by TwoSum at the end.
// For the re-ranking flushes, where a warp's distances are latency-bound.
__device__ __forceinline__ float exact_sqdist_warp_wide(const float* __restrict__ a,
                                                        const float* __restrict__ b, int d) {
  const int lane = threadIdx.x & 31;
  if ((d & 3) != 0 || ((reinterpret_cast<uintptr_t>(a) | reinterpret_cast<uintptr_t>(b)) & 15))
    return exact_sqdist_warp(a, b, d);
  float s0 = 0.f, c0 = 0.f, s1 = 0.f, c1 = 0.f;
  const float4* a4 = reinterpret_cast<const float4*>(a);
  const float4* b4 = reinterpret_cast<const float4*>(b);
  const int d4 = d >> 2;
  for (int j0 = 0; j0 < d4; j0 += 8 * 32) {
    float4 av[8], bv[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int j = j0 + lane + 32 * u;
      av[u] = j < d4 ? a4[j] : make_float4(0.f, 0.f, 0.f, 0.f);
      bv[u] = j < d4 ? b4[j] : make_float4(0.f, 0.f, 0.f, 0.f);
    }
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      float t;
      t = av[u].x - bv[u].x;
      kahan_add(t * t, s0, c0);
      t = av[u].y - bv[u].y;
      kahan_add(t * t, s1, c1);
      t = av[u].z - bv[u].z;
      kahan_add(t * t, s0, c0);
      t = av[u].w - bv[u].w;
      kahan_add(t * t, s1, c1);
    }
  }
  // (s0 - c0) + (s1 - c1): TwoSum of the s parts, the c parts and the error
  // term summed plainly (the same pattern as the lane tree below)
  float s = s0 + s1;
  {
    const float bb = s - s0;
    const float err = (s0 - (s - bb)) + (s1 - bb);
    c0 = (c0 + c1) - err;
  }
  float c = c0;
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    float s2 = __shfl_xor_sync(0xffffffffu, s, off);
    float c2 = __shfl_xor_sync(0xffffffffu, c, off);
    float sum = s + s2;
    float bb = sum - s;
    float err = (s - (sum - bb)) + (s2 - bb);
    c = (c + c2) - err;
    s = sum;
  }
  return s - c;
}

// Two FP32 operations per instruction (each half rounds as its scalar form).
__device__ __forceinline__ uint64_t pack2(float lo, float hi) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ float lo2(uint64_t v) { return __uint_as_float((uint32_t)v); }
__device__ __forceinline__ float hi2(uint64_t v) { return __uint_as_float((uint32_t)(v >> 32)); }
__device__ __forceinline__ uint64_t fma2(uint64_t x, uint64_t y, uint64_t z) {
  uint64_t r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(x), "l"(y), "l"(z));
  return r;
}
__device__ __forceinline__ uint64_t mul2(uint64_t x, uint64_t y) {
  uint64_t r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(x), "l"(y));
  return r;
}
__device__ __forceinline__ uint64_t add2(uint64_t x, uint64_t y) {
  uint64_t r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(x), "l"(y));
  return r;
}
__device__ __forceinline__ uint64_t sub2(uint64_t x, uint64_t y) {
  uint64_t r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(x), "l"(y));
  return r;
}

// exact_sqdist_warp_wide of two pairs at once: the same sums in the same order
// (the same bits), one pair in each half of packed FP32 operations, so that
// two pairs' loads and dependent sums overlap.  A flush's distances wait on
// latency, not on arithmetic.
__device__ __forceinline__ void exact_sqdist_warp_pair(const float* __restrict__ a0,
                                                       const float* __restrict__ b0,
                                                       const float* __restrict__ a1,
                                                       const float* __restrict__ b1, int d,
                                                       float& out0, float& out1) {
  const int lane = threadIdx.x & 31;
  if ((d & 3) != 0 || ((reinterpret_cast<uintptr_t>(a0) | reinterpret_cast<uintptr_t>(b0) |
                        reinterpret_cast<uintptr_t>(a1) | reinterpret_cast<uintptr_t>(b1)) & 15)) {
    out0 = exact_sqdist_warp_wide(a0, b0, d);
    out1 = exact_sqdist_warp_wide(a1, b1, d);
    return;
  }
  // Kahan sums of the even and odd elements; the compensations negated, so
  // that a term is y = fma(t, t, -c)
  uint64_t s0 = 0, n0 = 0, s1 = 0, n1 = 0;
  auto add = [](float t, float u, uint64_t& s, uint64_t& n) {
    const uint64_t v = pack2(t, u), y = fma2(v, v, n), w = add2(s, y);
    n = sub2(y, sub2(w, s));
    s = w;
  };
  const int d4 = d >> 2, blocks = (d4 + 255) / 256 * 4;  // (the wide form's 8-load rounds)
  const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 1
  for (int i = 0; i < blocks; ++i) {
    float4 av[2], bv[2], cv[2], dv[2];
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int j = lane + 32 * (2 * i + u);
      const bool in = j < d4;
      av[u] = in ? reinterpret_cast<const float4*>(a0)[j] : z;
      bv[u] = in ? reinterpret_cast<const float4*>(b0)[j] : z;
      cv[u] = in ? reinterpret_cast<const float4*>(a1)[j] : z;
      dv[u] = in ? reinterpret_cast<const float4*>(b1)[j] : z;
    }
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      add(av[u].x - bv[u].x, cv[u].x - dv[u].x, s0, n0);
      add(av[u].y - bv[u].y, cv[u].y - dv[u].y, s1, n1);
      add(av[u].z - bv[u].z, cv[u].z - dv[u].z, s0, n0);
      add(av[u].w - bv[u].w, cv[u].w - dv[u].w, s1, n1);
    }
  }
  // TwoSum of the s parts, the compensations and the error term summed plainly
  auto join = [](uint64_t x, uint64_t nx, uint64_t y, uint64_t ny, uint64_t& s, uint64_t& n) {
    const uint64_t t = add2(x, y), bb = sub2(t, x);
    const uint64_t err = add2(sub2(x, sub2(t, bb)), sub2(y, bb));
    n = add2(add2(nx, ny), err);
    s = t;
  };
  uint64_t s, n;
  join(s0, n0, s1, n1, s, n);
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    const uint64_t so = __shfl_xor_sync(0xffffffffu, (unsigned long long)s, off);
    const uint64_t no = __shfl_xor_sync(0xffffffffu, (unsigned long long)n, off);
    join(s, n, so, no, s, n);
  }
  s = add2(s, n);
  out0 = lo2(s);
  out1 = hi2(s);
}

// k-th smallest of the nv FP32 values vals[0..nv) (non-negative, +inf for
// absent entries) by one warp: binary search on the bit pattern for the
// least t with #{v <= t} >= k.  Returns +inf when fewer than k are finite.
__device__ __forceinline__ float warp_kth_smallest(const float* vals, int nv, int k) {
  const int lane = threadIdx.x & 31;
  int finite = 0;
  for (int i = lane; i < nv; i += 32) finite += vals[i] < INFINITY;
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) finite += __shfl_xor_sync(0xffffffffu, finite, off);
  if (k <= 0 || finite < k) return INFINITY;
  uint32_t lo = 0, hi = 0x7f800000u;
  while (lo < hi) {
    const uint32_t mid = lo + ((hi - lo) >> 1);
    int cnt = 0;
    for (int i = lane; i < nv; i += 32) cnt += __float_as_uint(vals[i]) <= mid;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) cnt += __shfl_xor_sync(0xffffffffu, cnt, off);
    if (cnt >= k) hi = mid;
    else lo = mid + 1;
  }
  return __uint_as_float(lo);
}

// k-th smallest of nv non-negative bf16 bit patterns (+inf = 0x7f80 for
// absent entries) by one warp; same search as warp_kth_smallest on 16 bits.
// Returns the value as FP32 (+inf when fewer than k are finite).
__device__ __forceinline__ float warp_kth_smallest_bf16(const uint16_t* vals, int nv, int k) {
  const int lane = threadIdx.x & 31;
  int finite = 0;
  for (int i = lane; i < nv; i += 32) finite += vals[i] < 0x7f80u;
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) finite += __shfl_xor_sync(0xffffffffu, finite, off);
  if (k <= 0 || finite < k) return INFINITY;
  uint32_t lo = 0, hi = 0x7f80u;
  while (lo < hi) {
    const uint32_t mid = (lo + hi) >> 1;
    int cnt = 0;
    for (int i = lane; i < nv; i += 32) cnt += vals[i] <= mid;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) cnt += __shfl_xor_sync(0xffffffffu, cnt, off);
    if (cnt >= k) hi = mid;
    else lo = mid + 1;
  }
  return __uint_as_float(lo << 16);
}

// Compensated FP32 sum of squares after Ogita, Rump & Oishi ("Accurate sum
// and dot product", SIAM J. Sci. Comput. 26(6), 2005): each term v*v is split
// exactly into p + e by an FMA (TwoProduct) and each addition s + p into
// t + err by TwoSum, so s + (exact sum of the error terms) is the exact sum;
// c accumulates those error terms in plain FP32.  The intrinsics keep the
// compiler from fusing the product into the addition, which would break the
// TwoSum identity.  For n terms spread over lanes, a 5-step lane tree and L
// level additions, the error of c is below (2n/32 + 2L + 12)(n/32 + L + 6) u^2
// of the sum, under 2^-30 of it for n <= 8192, L <= 64 (non-negative terms).
struct Acc2 {
  float s, c;
};

// TwoSum: t + err == x + y exactly.
__device__ __forceinline__ float two_sum(float x, float y, float& err) {
  const float t = __fadd_rn(x, y);
  const float bb = __fsub_rn(t, x);
  err = __fadd_rn(__fsub_rn(x, __fsub_rn(t, bb)), __fsub_rn(y, bb));
  return t;
}

__device__ __forceinline__ void acc2_sq(Acc2& a, float v) {
  const float p = __fmul_rn(v, v);
  const float e = __fmaf_rn(v, v, -p);
  float err;
  a.s = two_sum(a.s, p, err);
  a.c = __fadd_rn(a.c, __fadd_rn(err, e));
}

// Adds b into a.  Symmetric in a and b (TwoSum's t and err are, and so is
// a.c + b.c), so both lanes of a shuffle pair hold the same result.
__device__ __forceinline__ void acc2_add(Acc2& a, Acc2 b) {
  float err;
  a.s = two_sum(a.s, b.s, err);
  a.c = __fadd_rn(__fadd_rn(a.c, b.c), err);
}

__device__ __forceinline__ Acc2 warp_sum_acc2(Acc2 a) {
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    Acc2 b{__shfl_xor_sync(0xffffffffu, a.s, off), __shfl_xor_sync(0xffffffffu, a.c, off)};
    acc2_add(a, b);
  }
  return a;
}

// Upper bound of the exact sum held by a (relative slack 2^-23 over the
// 2^-30 error bound; FLT_MIN covers terms lost to underflow).
__device__ __forceinline__ float acc2_upper(Acc2 a, float rel) {
  return __fadd_ru(__fmul_ru(__fadd_ru(a.s, a.c), 1.0f + rel), 0x1p-126f);
}

// Adds the square of x - y, the difference split exactly into h + e (TwoSum):
// (h + e)^2 = h^2 + 2 h e + e^2, the last term below 2^-48 of the first.
__device__ __forceinline__ void acc2_sqdiff(Acc2& a, float x, float y) {
  float e;
  const float h = two_sum(x, -y, e);
  acc2_sq(a, h);
  a.c = __fmaf_rn(2.f * h, e, a.c);
}

// The warp's total as FP64, of the squares of value(j), j = lo .. hi - 1.  *ok is
// cleared where it may be off by more than the bound above and 2^-40: terms
// beyond FP32's range (elements above 1.8e19), or a total so small that the
// underflow of squares counts (2^-149 a term; not where all are zeros).
template <class F>
__device__ __forceinline__ double warp_acc2_f64(Acc2 a, int lo, int hi, F value, bool* ok) {
  a = warp_sum_acc2(a);
  if (!(a.s > 0x1p-90f && a.s < INFINITY)) {  // (the same in every lane)
    bool nonzero = false;
#pragma unroll 1
    for (int j = lo + (int)(threadIdx.x & 31); j < hi; j += 32) nonzero |= value(j) != 0.f;
    if (__any_sync(0xffffffffu, nonzero)) *ok = false;
  }
  return (double)a.s + (double)a.c;
}

// The root of the sum held by a, rounded to nearest, as FP64 would give it from
// a sum off by at most rel; NaN where that cannot be told from a.
__device__ __forceinline__ float sqrt_rn_acc2(Acc2 a, float rel) {
  float lo;
  const float hi = two_sum(a.s, a.c, lo);
  if (hi == 0.f) return 0.f;
  if (!(hi > 0x1p-80f && hi < 0x1p120f)) return NAN;
  // the exact root is r + delta up to 2^-44 of r
  const float r = __fsqrt_rn(hi);
  const float delta = __fdividef(__fadd_rn(__fmaf_rn(-r, r, hi), lo), 2.f * r);
  const float slack = r * (0.5f * rel + 0x1p-43f);
  const float up = __fadd_rn(r, delta + slack), down = __fadd_rn(r, delta - slack);
  return up == down ? up : NAN;
}

__device__ __forceinline__ double warp_sum_f64(double v) {
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
  return v;
}

// Whether the FP64 value v (normal in FP32) rounds to the same FP32 number, up
// (NEAREST false) or to nearest, wherever in v (1 -+ r 2^-53) it lies: the 29 bits
// below FP32's last one stay that far from where the rounding turns.
template <bool NEAREST>
__device__ __forceinline__ bool rounds_alike(double v, uint32_t r) {
  const uint32_t turn = NEAREST ? 1u << 28 : 0u;
  const uint32_t at = ((uint32_t)__double2loint(v) + turn) & 0x1fffffffu;
  return at - r < 0x20000000u - 2 * r;
}

// The bounds of a packed row, by one warp: rounded-up tail norms (of the stored
// vector, from level `lane` and `lane + 32` on), |x^|^2 and e_x, a bound on the
// stored vector's distance to the exact transform.
struct RowBounds {
  float tail[2], xn2, ex;
};

// stored(j): the stored element; err(j), dev(j): the storage error and (x - mu~)_j
// in FP64; add_err(acc, j, stored(j)), add_dev(acc, j): the addition of their
// squares.
//
// All results are those of FP64 sums, rounded once to FP32, but the sums are
// compensated FP32: FP64 arithmetic per element was most of the packers' time
// (a warp's FP64 instruction takes 16 cycles; 500k x 384 BF16 rows: 11.3 ms,
// 3.4 so).  Where a sum's error (a few 1e-12 of it) could move one of the
// row's results to another FP32 number, the row is summed again in FP64.
template <class Stored, class Err, class Dev, class AddErr, class AddDev>
__device__ __forceinline__ RowBounds row_bounds(int d, int L, const int32_t* __restrict__ level_off,
                                                double c_trans, bool valid, Stored stored, Err err,
                                                Dev dev, AddErr add_err, AddDev add_dev) {
  const int lane = threadIdx.x & 31;
  RowBounds out{{0.f, 0.f}, 0.f, 0.f};
  if (!valid) return out;
  constexpr double kUp = 1.0 + 1e-12, kUpE = 1.0 + 1e-9;
  // error of a sum of n terms in units of 2^-53: the bound of Acc2 with a third
  // rounding per term (acc2_sqdiff's) and no level additions (they are in
  // FP64), small terms (2^-40 = 2^13 units), FP64 roundings
  auto error = [](int n) {
    const uint32_t m = (uint32_t)(n + 31) / 32;
    return (4 * m + 16) * (m + 8) * 32 + 8192 + 256;
  };
  double tail[2] = {0.0, 0.0}, energy = 0.0;
  bool ok = true;
  Acc2 qa{0.f, 0.f}, da{0.f, 0.f};
  int widest = 0;
  for (int l = L - 1; l >= 0; --l) {
    const int lo = level_off[l], hi = level_off[l + 1];
    Acc2 e{0.f, 0.f};
    for (int j = lo + lane; j < hi; j += 32) {
      const float v = stored(j);
      acc2_sq(e, v);
      add_err(qa, j, v);
    }
    widest = max(widest, hi - lo);
    energy += warp_acc2_f64(e, lo, hi, stored, &ok);
    if (l == lane) tail[0] = energy;
    if (l == lane + 32) tail[1] = energy;
  }
  for (int j = lane; j < d; j += 32) add_dev(da, j);
  const double qe = warp_acc2_f64(qa, 0, d, err, &ok), de = warp_acc2_f64(da, 0, d, dev, &ok);
  // (lanes 0 and 1 take a root each: FP64 roots are long)
  const double root = sqrt(lane == 0 ? qe : de);
  const double e =
      (__shfl_sync(0xffffffffu, root, 0) + c_trans * __shfl_sync(0xffffffffu, root, 1)) * kUpE;
  const uint32_t r = error(widest);
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    if (32 * u >= L) break;
    const double t = sqrt(tail[u] * kUp);
    out.tail[u] = __double2float_ru(t);
    if (t > 0.0) ok &= rounds_alike<false>(t, r);
  }
  out.xn2 = (float)energy;
  out.ex = __double2float_ru(e);
  if (energy > 0.0) ok &= rounds_alike<true>(energy, r);
  if (e > 0.0) ok &= rounds_alike<false>(e, error(d));
  if (__all_sync(0xffffffffu, ok)) return out;
  double q2 = 0.0, d2 = 0.0;
  energy = 0.0;
#pragma unroll 1
  for (int l = L - 1; l >= 0; --l) {
    double s = 0.0;
#pragma unroll 1
    for (int j = level_off[l] + lane; j < level_off[l + 1]; j += 32) {
      const double v = stored(j), q = err(j);
      s += v * v;
      q2 += q * q;
    }
    energy += warp_sum_f64(s);
    const float t = __double2float_ru(sqrt(energy * kUp));
    if (l == lane) out.tail[0] = t;
    if (l == lane + 32) out.tail[1] = t;
  }
#pragma unroll 1
  for (int j = lane; j < d; j += 32) {
    const double v = dev(j);
    d2 += v * v;
  }
  out.xn2 = (float)energy;
  out.ex = __double2float_ru((sqrt(warp_sum_f64(q2)) + c_trans * sqrt(warp_sum_f64(d2))) * kUpE);
  return out;
}

}  // namespace pano
