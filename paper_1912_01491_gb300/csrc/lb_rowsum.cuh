// lb_rowsum.cuh -- FP64 arithmetic of the RK4 row sums that stays off the FP64
// pipe.  A GB300 sub-partition issues one FP64 warp instruction in about 64
// cycles whatever its active lanes (measured: 62 for a dependent add, 105 with
// the shuffle that feeds it), an integer one in two.  Combining a row's 128
// FP32 partial sums by FP64 additions took four conversions, three additions
// and five more with shuffles a row: at N = 50 more than the products.  Step
// times before and after: FP32 N = 50 44.6 -> 34.8 us, BF16 N = 50 with a
// correction every 5 steps 54.6 -> 40.8 us, BF16 N = 150 1.35 -> 1.12 ms.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace lb {

// (double)f by integer operations (the conversion is an FP64 instruction too).
__device__ __forceinline__ double widen(float f) {
  const uint32_t u = __float_as_uint(f), e = u & 0x7f800000u, s = u & 0x80000000u;
  uint32_t hi = ((u & 0x7fffffffu) >> 3) + 0x38000000u, lo = u << 29;
  if (e == 0u) {  // zero, or subnormal: shift the leading one to the implicit place
    uint32_t m = u & 0x7fffffu;
    hi = lo = 0u;
    if (m != 0u) {
      const int z = __clz((int)m) - 8;
      m = (m << z) & 0x7fffffu;
      hi = ((uint32_t)(897 - z) << 20) + (m >> 3);
      lo = m << 29;
    }
  } else if (e == 0x7f800000u) {
    hi += 0x38000000u;
  }
  return __hiloint2double((int)(hi | s), (int)lo);
}

// The warp's 128 FP32 partial sums (four per lane) as one integer: T and emax
// with sum = T 2^(emax - 180), the same in every lane.  Each partial sum is its
// 24-bit significand times a power of two up to 2^30, so T (at most 61 bits)
// is exact; false (in every lane) when a nonzero partial sum lies more than 30
// binades below the largest, is subnormal or is not finite.
__device__ __forceinline__ bool lane_sum_fixed(const float (&a)[4], int64_t& T, int& emax) {
  int e[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) e[q] = (int)((__float_as_uint(a[q]) >> 23) & 255u);
  emax = __reduce_max_sync(0xffffffffu, max(max(e[0], e[1]), max(e[2], e[3])));
  const int lo = max(emax - 30, 1);
  bool bad = emax == 255;
  int64_t s = 0;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int u = __float_as_int(a[q]);
    bad |= (u << 1) != 0 && e[q] < lo;
    int sig = e[q] == 0 ? 0 : (u & 0x7fffff) | 0x800000;
    sig = u < 0 ? -sig : sig;
    s += (int64_t)sig * (int64_t)(int)(1u << ((e[q] - emax + 30) & 31));  // one 32 x 32 + 64-bit multiply-add
  }
  if (__any_sync(0xffffffffu, bad)) return false;
  // 24 + 24 + 9 bits: sums of 32 lanes fit 32 bits
  const uint32_t s0 = __reduce_add_sync(0xffffffffu, (uint32_t)s & 0xffffffu);
  const uint32_t s1 = __reduce_add_sync(0xffffffffu, (uint32_t)(s >> 24) & 0xffffffu);
  const int s2 = __reduce_add_sync(0xffffffffu, (int)(s >> 48));
  T = (int64_t)(((uint64_t)(int64_t)s2 << 48) + ((uint64_t)s1 << 24) + s0);
  return true;
}

// T 2^(emax - 180) rounded to nearest even (|T| < 2^62; never subnormal).
__device__ __forceinline__ double fixed_to_double(int64_t T, int emax) {
  const uint64_t mag = T < 0 ? (uint64_t)0 - (uint64_t)T : (uint64_t)T;
  const int z = __clzll((long long)mag);      // 2 .. 64
  const uint64_t norm = mag << ((z - 1) & 63);  // leading bit at 62
  const uint64_t r = (norm + 0x1ffu + ((norm >> 10) & 1u)) >> 10;  // 53 bits, or a carry to 2^53
  // the leading bit's exponent is 63 - z; r carries the leading bit into the exponent field
  const uint64_t bits = ((uint64_t)(63 - z + emax - 180 + 1022) << 52) + r;
  const uint64_t sign = (uint64_t)T & 0x8000000000000000ull;
  return mag == 0 ? 0.0 : __longlong_as_double((long long)(bits | sign));
}

// The same sum by FP64 additions, (a0 + a1) + (a2 + a3) per lane and the xor
// tree over the lanes.
__device__ __forceinline__ double lane_sum_tree(const float (&a)[4]) {
  double t = (widen(a[0]) + widen(a[1])) + (widen(a[2]) + widen(a[3]));
  for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
  return t;
}

// Sum of the warp's 128 FP32 partial sums in FP64: exact and rounded once, or
// by FP64 additions where the exponents spread too far.
__device__ __forceinline__ double lane_sum(const float (&a)[4]) {
  int64_t T;
  int emax;
  if (lane_sum_fixed(a, T, emax)) return fixed_to_double(T, emax);
  return lane_sum_tree(a);
}

// The defect of a stored element, a - f or a - r q, exactly and by integer
// operations: the FP64 pipe is then left to the product with v.  The difference
// of an element and its rounded copy has few bits, so it is a short integer
// times a's unit in the last place.  False: not of that form (signs or binades
// apart, subnormal, not finite); d is then not set.
__device__ __forceinline__ bool defect(double a, float f, float, double& d) {
  const uint32_t ah = (uint32_t)__double2hiint(a), al = (uint32_t)__double2loint(a), u = __float_as_uint(f);
  // f's bits as FP64, for normal f: hi word and the top three bits of the low one
  const uint32_t fh = ((u & 0x7fffffffu) >> 3) + 0x38000000u, fl = u << 29;
  const uint32_t ea = (ah >> 20) & 0x7ffu;
  // as integers the magnitudes differ by |a| - |f| in a's last place, if f is in a's binade or the power of two above
  const uint32_t lo = al - fl;
  const int32_t hi = (int32_t)((ah & 0x7fffffffu) - fh - (al < fl ? 1u : 0u));
  const uint32_t ef = fh >> 20;
  const bool binade = ef == ea || (ef == ea + 1u && (fh & 0xfffffu) == 0u && fl == 0u);
  const bool ok = binade && ((ah ^ u) >> 31) == 0u && ea >= 64u && ea < 0x7feu && (u & 0x7f800000u) != 0u &&
                  hi == ((int32_t)lo >> 31);  // fits 32 bits
  const uint32_t m = (int32_t)lo < 0 ? 0u - lo : lo;
  const int z = __clz((int)m);
  const uint32_t t = m << (z & 31);  // leading bit at 31
  const uint32_t sign = (ah ^ lo) & 0x80000000u;
  d = m == 0u ? 0.0
              : __hiloint2double((int)(sign | (((ea - 22u - (uint32_t)z) << 20) + (t >> 11))), (int)(t << 21));
  return ok || ((ah & 0x7fffffffu) | al | (u & 0x7fffffffu)) == 0u;
}
__device__ __forceinline__ bool defect(double a, uint16_t q, float r, double& d) {
  const uint32_t ah = (uint32_t)__double2hiint(a), ur = __float_as_uint(r);
  const uint32_t ea = (ah >> 20) & 0x7ffu, er = (ur >> 23) & 0xffu, eq = ((uint32_t)q >> 7) & 0xffu;
  const uint64_t ma = ((uint64_t)__double_as_longlong(a) & 0xfffffffffffffull) | 0x10000000000000ull;
  const uint32_t p = ((ur & 0x7fffffu) | 0x800000u) * (((uint32_t)q & 0x7fu) | 0x80u);  // 24 + 8 bits
  const int k = (int)(er + eq) - (int)ea + 791;  // r q = p 2^k units of a's last place
  const bool zero = (q & 0x7fffu) == 0u;         // then d = a
  const int64_t x = (int64_t)(ma - ((uint64_t)p << (k & 31)));
  const uint64_t m = x < 0 ? (uint64_t)0 - (uint64_t)x : (uint64_t)x;
  const bool ok = (uint32_t)k <= 30u && ((ah >> 31) ^ (uint32_t)(q >> 15) ^ (ur >> 31)) == 0u && ea >= 64u &&
                  ea < 0x7feu && eq != 0u && eq != 0xffu && er != 0u && er != 0xffu && m < (1ull << 53);
  const int z = __clzll((long long)m);  // 11 .. 63, or 64
  const uint64_t t = m << (z & 63);     // leading bit at 63
  const uint64_t bits = ((uint64_t)(uint32_t)((int)ea + 10 - z) << 52) + (t >> 11);
  const uint64_t sign = ((uint64_t)__double_as_longlong(a) ^ (uint64_t)x) & 0x8000000000000000ull;
  d = zero ? a : m == 0 ? 0.0 : __longlong_as_double((long long)(bits | sign));
  return ok || zero;
}
__device__ __forceinline__ double defect_fp64(double a, float f, float) { return a - widen(f); }
__device__ __forceinline__ double defect_fp64(double a, uint16_t q, float r) {
  return fma(-widen(r), widen(__uint_as_float((uint32_t)q << 16)), a);  // r q is exact, so one rounding
}

// One lane's part of sum_n (a_n - stored_n) v_n, n = lane, lane + 32, ..; the
// whole warp calls it.  Two FP64 instructions a term (subtract and multiply, or
// for BF16 two products) were the pipe's time.  For BF16 the integer form takes
// half as long again as the FP64 product beside it, so one term of four is left
// to the FP64 pipe (M = 22499: 1.76 ms all FP64, 1.48 all integer, now
// 1.29; FP32, M = 39999: 5.5 -> 3.8).  STREAM: the stored elements are read once,
// else they may be in a cache.
template <bool STREAM, class E>
__device__ __forceinline__ double defect_dot(const double* __restrict__ a, const E* __restrict__ e, float r,
                                             const double* __restrict__ v, int M, int lane) {
  constexpr int U = 4, F = sizeof(E) == 2 ? 3 : 4;
  double t = 0.0;
  int n = lane;
  for (int n0 = 0; n0 + 32 * U <= M; n0 += 32 * U) {
    double av[U], vv[U], d[U];
    E ev[U];
    bool ok = true;
#pragma unroll
    for (int i = 0; i < U; ++i, n += 32) {
      av[i] = __ldcs(a + n);
      ev[i] = STREAM ? __ldcs(e + n) : e[n];
      vv[i] = v[n];
    }
#pragma unroll
    for (int i = 0; i < F; ++i) ok &= defect(av[i], ev[i], r, d[i]);
#pragma unroll
    for (int i = F; i < U; ++i) d[i] = defect_fp64(av[i], ev[i], r);
    if (__any_sync(0xffffffffu, !ok)) {
#pragma unroll
      for (int i = 0; i < F; ++i) d[i] = defect_fp64(av[i], ev[i], r);
    }
#pragma unroll
    for (int i = 0; i < U; ++i) t = fma(d[i], vv[i], t);
  }
  for (; n < M; n += 32) t = fma(defect_fp64(a[n], e[n], r), v[n], t);
  return t;
}

// The sum of x over the threads of the block behind the calling one (blocks of
// kSuffixThreads, sh: one value per warp).
constexpr int kSuffixThreads = 256;

template <class T>
__device__ __forceinline__ T block_suffix(T x, T* sh) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  T in = x;  // inclusive
  for (int o = 1; o < 32; o <<= 1) {
    const T u = __shfl_down_sync(0xffffffffu, in, o);
    if (lane + o < 32) in += u;
  }
  T ex = __shfl_down_sync(0xffffffffu, in, 1);
  if (lane == 31) ex = T(0);
  __syncthreads();
  if (lane == 0) sh[wid] = in;
  __syncthreads();
  T behind = T(0);
  for (int w = kSuffixThreads / 32 - 1; w > wid; --w) behind += sh[w];
  return ex + behind;
}

}  // namespace lb
