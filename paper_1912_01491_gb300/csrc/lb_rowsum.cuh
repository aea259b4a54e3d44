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
