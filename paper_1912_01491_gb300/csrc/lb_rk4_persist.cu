// lb_rk4_persist.cu -- the dense RK4 steps of small and middle systems (Sec. 4
// item 3, Table 1 step 3.1) as one cooperative launch over all steps.
//
// One launch per stage (k_stage, lb_rk4.cu) costs 4 to 6 us a stage whatever
// the size: the launch, an L2 round trip for every operand and the drain.  The
// matrix of such a system is small enough to stay on the chip, so here every
// block keeps its rows of it in shared memory for the whole call (rows that do
// not fit are read from L2), every warp keeps the state of its R rows in
// registers, and the blocks exchange only the stage vector.
//
// Exchange: an element travels as an 8-byte word {32 data bits, stage number}
// (two words for an FP64 element) in a global buffer, stored and polled with
// relaxed 64-bit accesses, so that a word carries its own flag: one L2 write
// and one L2 read per stage instead of a grid barrier (fence, atomic, poll)
// and then a read.  Two buffers alternate by stage parity.  A block
// overwrites a buffer of stage g in stage g + 2, which it computes only after
// it has polled every element of stage g + 1, and a block sends those only
// after it has read all of stage g: no reader can lag behind.  The launch is
// cooperative (all blocks are resident) and every poll is bounded (about two
// seconds of clock).  A block whose poll runs out sets *err, waits no more and
// takes NaN for every element that has not come: each row reads all of x, so all
// of its rows are NaN from the next stage on, and so are those of a block that
// still takes its words.  An element of v or of a snapshot is either right or NaN.
//
// Arithmetic: the row sums are those of k_stage (FP64: the same lane order and
// shuffle tree; FP32 and BF16: the same 128 partial sums, summed by
// lb::lane_sum), the correction that of k_correction, so the results are
// bit-identical to theirs.
#include <cuda_bf16.h>

#include <algorithm>
#include <type_traits>

#include "lb_internal.h"
#include "lb_rowsum.cuh"

namespace {

constexpr long long kPollCycles = 4000000000LL;
constexpr int kMaxWarps = 16;

thread_local long long t_poll_cycles = kPollCycles;

struct PersistArgs {
  int M, nr, rem;  // rows per block: nr, the first rem blocks one more
  int nres;        // rows a block keeps in shared memory
  int pitch;       // elements between resident rows
  int xpad;        // elements of x in shared memory
  const void* Ap;
  const float* scale;
  const double* A64;  // null: no correction
  int64_t correct_every, nsteps, snap_every, t0;
  const double* K;
  const double* keff0;  // K + correction left by an earlier launch of the same call, or null
  double* keff_out;
  double* v;
  double h;
  double* snaps;
  unsigned long long* ll;  // two buffers of bufw words
  size_t bufw;
  int* err;
  long long poll_cycles;
};

__device__ __forceinline__ void ll_store(unsigned long long* p, uint32_t data, uint32_t flag) {
  const unsigned long long w = ((unsigned long long)flag << 32) | data;
  asm volatile("st.relaxed.gpu.global.b64 [%0], %1;" ::"l"(p), "l"(w) : "memory");
}
__device__ __forceinline__ void ll_load2(const unsigned long long* p, unsigned long long& a, unsigned long long& b) {
  asm volatile("ld.relaxed.gpu.global.v2.b64 {%0, %1}, [%2];" : "=l"(a), "=l"(b) : "l"(p) : "memory");
}

__device__ __forceinline__ float bf16_float(uint16_t u) { return __uint_as_float(((uint32_t)u) << 16); }
__device__ __forceinline__ float elem32(float e) { return e; }
__device__ __forceinline__ float elem32(uint16_t e) { return bf16_float(e); }
__device__ __forceinline__ float4 vec32(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ float4 vec32(const uint16_t* p) {
  const uint2 b = *reinterpret_cast<const uint2*>(p);
  return make_float4(__uint_as_float(b.x << 16), __uint_as_float(b.x & 0xffff0000u), __uint_as_float(b.y << 16),
                     __uint_as_float(b.y & 0xffff0000u));
}

// Elements of a row in global memory before its first aligned vector of four.
template <class E>
__device__ __forceinline__ int head_of(const E* row, int M) {
  constexpr uintptr_t al = 4 * sizeof(E);
  return min((int)(((al - (reinterpret_cast<uintptr_t>(row) & (al - 1))) & (al - 1)) / sizeof(E)), M);
}

// Sum over the 32 lanes of each of R row values; lane l returns the sum of
// row l / (32 / R), every pair sum that of the xor tree 16, 8, 4, 2, 1: each
// level exchanges the rows the other half keeps, so R rows take R/2 + R/4 + ...
// FP64 additions instead of five each.
template <int R>
__device__ __forceinline__ double reduce_rows(double (&t)[R], int lane) {
  int o = 16;
#pragma unroll
  for (int n = R; n > 1; n >>= 1, o >>= 1) {
    const bool up = (lane & o) != 0;
#pragma unroll
    for (int i = 0; i < n / 2; ++i) {
      const double lo = t[i], hi = t[i + n / 2];
      const double send = up ? lo : hi;
      t[i] = (up ? hi : lo) + __shfl_xor_sync(0xffffffffu, send, o);
    }
  }
  double s = t[0];
  for (; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  return s;
}

// The 128 partial sums of one row in k_stage's lanes: lane k takes elements
// head + 4k .. head + 4k + 3 of every 128 (head: the elements before the
// row's first aligned vector in global memory, taken by the first lanes).
// Element by element: only for rows whose fixed-point sum does not apply.
template <class E>
__device__ __noinline__ double row_tree(const E* row, const float* x, int M, int head, int lane) {
  float a[4] = {0.f, 0.f, 0.f, 0.f};
  if (lane < head) a[0] = fmaf(elem32(row[lane]), x[lane], a[0]);
  const int nv = (M - head) >> 2;
  for (int k = lane; k < nv; k += 32)
#pragma unroll
    for (int c = 0; c < 4; ++c) a[c] = fmaf(elem32(row[head + 4 * k + c]), x[head + 4 * k + c], a[c]);
  for (int n = head + 4 * nv + lane; n < M; n += 32) a[0] = fmaf(elem32(row[n]), x[n], a[0]);
  return lb::lane_sum_tree(a);
}

// Row sums of R resident rows (FP32 or BF16 elements).  A thread takes the
// aligned vector 4K .. 4K + 3 of x and of each row.  Its component c belongs to
// the partial sum (lane K, c - head) for c >= head and (lane K - 1, c - head +
// 4) for c < head, in the same order as k_stage's, so the thread's four sums
// are four of k_stage's 128, in another lane: the sum of all 128 does not
// depend on where they are, and rows of any head share the loads of x.  The
// elements before head and behind the last whole vector, zero in the resident
// copy, are he and te of the first lanes: they go to the sum (lane, 0), he
// first and te last.  Lane r < R returns row r's sum.
template <class E, int R>
__device__ __forceinline__ double rows_resident(const E* const (&rows)[R], const E* const (&grow)[R],
                                                const int (&head)[R], const float (&he)[R], const float (&te)[R],
                                                const float* x, int M, int nk, int lane) {
  float a[R][4];
  const float xh = x[lane];
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const float p = he[r] * xh;
    a[r][0] = 0.f;
#pragma unroll
    for (int c = 1; c < 4; ++c) a[r][c] = head[r] == c ? p : 0.f;
  }
  const float4* xv = reinterpret_cast<const float4*>(x) + lane;
#pragma unroll 4
  for (int k = 0; k < nk; ++k) {
    const float4 w = xv[32 * k];
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const float4 u = vec32(rows[r] + 4 * lane + 128 * k);
      a[r][0] = fmaf(u.x, w.x, a[r][0]);
      a[r][1] = fmaf(u.y, w.y, a[r][1]);
      a[r][2] = fmaf(u.z, w.z, a[r][2]);
      a[r][3] = fmaf(u.w, w.w, a[r][3]);
    }
  }
  int64_t T = 0;
  int emax = 1;
  bool fixed = true;
  double y = 0.0;
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const float xt = x[head[r] + ((M - head[r]) & ~3) + lane];
#pragma unroll
    for (int c = 0; c < 4; ++c) a[r][c] = fmaf(head[r] == c ? te[r] : 0.f, xt, a[r][c]);
    int64_t Tr = 0;
    int er = 1;
    if (lb::lane_sum_fixed(a[r], Tr, er)) {
      if (lane == r) {
        T = Tr;
        emax = er;
      }
    } else {
      const double t = row_tree(grow[r], x, M, head[r], lane);
      if (lane == r) {
        y = t;
        fixed = false;
      }
    }
  }
  if (fixed) y = lb::fixed_to_double(T, emax);
  return y;
}

// The same for one row in global memory, in k_stage's lanes; lane k reads x
// from two aligned vectors.
template <class E>
__device__ __forceinline__ double row_global(const E* row, const float* x, int M, int lane) {
  float a[4] = {0.f, 0.f, 0.f, 0.f};
  const int head = head_of(row, M);
  if (lane < head) a[0] = fmaf(elem32(row[lane]), x[lane], a[0]);
  const int nv = (M - head) >> 2;
  const float4* xv = reinterpret_cast<const float4*>(x);
#pragma unroll 4
  for (int k = lane; k < nv; k += 32) {
    const float4 u = vec32(row + head + 4 * k);
    const float4 p = xv[k], q = xv[k + 1];
    const float s0 = head == 0 ? p.x : head == 1 ? p.y : head == 2 ? p.z : p.w;
    const float s1 = head == 0 ? p.y : head == 1 ? p.z : head == 2 ? p.w : q.x;
    const float s2 = head == 0 ? p.z : head == 1 ? p.w : head == 2 ? q.x : q.y;
    const float s3 = head == 0 ? p.w : head == 1 ? q.x : head == 2 ? q.y : q.z;
    a[0] = fmaf(u.x, s0, a[0]);
    a[1] = fmaf(u.y, s1, a[1]);
    a[2] = fmaf(u.z, s2, a[2]);
    a[3] = fmaf(u.w, s3, a[3]);
  }
  for (int n = head + 4 * nv + lane; n < M; n += 32) a[0] = fmaf(elem32(row[n]), x[n], a[0]);
  return lb::lane_sum(a);
}

// Row sums of R rows in FP64, in the order of k_stage: element n to sum
// (n / 32) mod 4 of its lane while the lane has all four of a chunk of 128,
// else to the first.  PAD: rows and x are zero from M to the next multiple of 32.
template <int R, bool PAD>
__device__ __forceinline__ void rows_fp64(const double* const (&rows)[R], const double* x, int M, int lane,
                                          double (&t)[R]) {
  double a[R][4];
#pragma unroll
  for (int r = 0; r < R; ++r) a[r][0] = a[r][1] = a[r][2] = a[r][3] = 0.0;
  const int full = M >> 7, rem = M & 127;
  int n = lane;
#pragma unroll 2
  for (int c = 0; c < full; ++c, n += 128) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const double xq = x[n + 32 * q];
#pragma unroll
      for (int r = 0; r < R; ++r) a[r][q] = fma(rows[r][n + 32 * q], xq, a[r][q]);
    }
  }
  const bool four = lane + 96 < rem;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    if (32 * q >= rem) break;
    const bool in = PAD || lane + 32 * q < rem;
    const double xq = in ? x[n + 32 * q] : 0.0;
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const double e = in ? rows[r][n + 32 * q] : 0.0;
      const double w = fma(e, xq, four ? a[r][q] : a[r][0]);
      a[r][q] = four ? w : a[r][q];
      a[r][0] = four && q > 0 ? a[r][0] : w;
    }
  }
#pragma unroll
  for (int r = 0; r < R; ++r) t[r] = (a[r][0] + a[r][1]) + (a[r][2] + a[r][3]);
}

template <int PREC, int R>
__global__ void __launch_bounds__(32 * kMaxWarps, 1) k_rk4_persist(PersistArgs A) {
  using E = typename std::conditional<PREC == LB_FP64, double,
                                      typename std::conditional<PREC == LB_FP32, float, uint16_t>::type>::type;
  constexpr bool F64 = PREC == LB_FP64;
  extern __shared__ __align__(16) unsigned char psm[];
  __shared__ int dead;
  const int M = A.M, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int nthr = blockDim.x, nwarps = nthr >> 5;
  const int b = blockIdx.x;
  const int r0 = b * A.nr + min(b, A.rem), nr = A.nr + (b < A.rem ? 1 : 0);
  const int nres = min(nr, A.nres);
  const bool correct = !F64 && A.A64 != nullptr;
  // shared memory: x in FP64 (FP64 form, or for the correction), x in FP32,
  // the resident rows
  double* x64 = reinterpret_cast<double*>(psm);
  float* x32 = reinterpret_cast<float*>(psm + (F64 || correct ? 8 * (size_t)A.xpad : 0));
  E* srow = reinterpret_cast<E*>(reinterpret_cast<unsigned char*>(x32) + (F64 ? 0 : 4 * (size_t)A.xpad));
  const E* Ag = static_cast<const E*>(A.Ap);
  if (tid == 0) dead = 0;
  const bool first_correct = correct && A.t0 % A.correct_every == 0;
  for (int j = tid; j < A.xpad; j += nthr) {
    const double x = j < M ? A.v[j] : 0.0;
    if (F64 || correct) x64[j] = x;
    if (!F64) x32[j] = (float)x;
  }
  for (int i = warp; i < nres; i += nwarps) {
    const E* src = Ag + (int64_t)(r0 + i) * M;
    E* dst = srow + (size_t)i * A.pitch;
    const int hd = F64 ? 0 : head_of(src, M), end = F64 ? M : hd + ((M - hd) & ~3);
#pragma unroll 4
    for (int n = lane; n < A.pitch; n += 32) dst[n] = n >= hd && n < end ? src[n] : E(0);
  }
  __syncthreads();

  // the warp's rows: i0 .. i0 + R - 1 of the block's; the lane that keeps row
  // i0 + mine: lane mine, in FP64 the first of the row's 32 / R lanes
  constexpr int kSpan = F64 ? 32 / R : 1;
  const int i0 = warp * R, mine = lane / kSpan;
  const bool active = i0 < nr, res = min(i0 + R, nr) <= nres;
  const bool holds = active && lane % kSpan == 0 && mine < R && i0 + mine < nr;
  const int s = r0 + i0 + mine;  // the held row
  const E *rows[R], *grows[R];
  int head[R];
  float he[R], te[R];
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int i = active ? min(i0 + r, nr - 1) : 0;
    const E* grow = Ag + (int64_t)(r0 + i) * M;
    rows[r] = res && active ? srow + (size_t)i * A.pitch : grow;
    grows[r] = grow;
    head[r] = F64 ? 0 : head_of(grow, M);
    he[r] = te[r] = 0.f;
    if constexpr (!F64) {
      const int end = head[r] + ((M - head[r]) & ~3);
      if (lane < head[r]) he[r] = elem32(grow[lane]);
      if (end + lane < M) te[r] = elem32(grow[end + lane]);
    }
  }
  double vs = 0.0, ac = 0.0, kf = 0.0, k0 = 0.0, sc = 1.0;
  if (holds) {
    vs = A.v[s];
    k0 = A.K[s];
    kf = A.keff0 ? A.keff0[s] : k0;
    if (PREC == LB_BF16) sc = (double)A.scale[s];
  }

  // poll every element of stage g into shared memory
  constexpr int kU = 4;  // pairs of words in flight per thread
  auto bad = [&]() { return *(volatile int*)&dead != 0; };
  auto poll = [&](uint32_t g, bool wide) {
    const unsigned long long* buf = A.ll + (size_t)(g & 1) * A.bufw;
    const int np = wide ? M : (M + 1) >> 1;
    for (int p0 = tid; p0 < np; p0 += kU * nthr) {
      unsigned long long w[kU][2] = {};
      const long long c0 = clock64();
      // a thread waits for its first pair before it asks for the others: polls
      // of words that have not come keep L2 from the stores they wait for
      // (FP64 N = 30: 17.5 -> 13.9 us a step, FP32 N = 41: 15.5 -> 14.0)
      auto ready = [&](int q) {
        return (uint32_t)(w[q][0] >> 32) == g &&
               ((!wide && 2 * (p0 + q * nthr) + 1 >= M) || (uint32_t)(w[q][1] >> 32) == g);
      };
      auto wait = [&](int q) {
        while (!ready(q) && !bad()) {
          if (clock64() - c0 > A.poll_cycles) {
            dead = 1;
            atomicExch(A.err, 1);
            break;
          }
          ll_load2(buf + 2 * (p0 + q * nthr), w[q][0], w[q][1]);
        }
        if (!ready(q)) w[q][0] = w[q][1] = 0x7ff80000u;  // NaN: FP32, and the high word of FP64
      };
      ll_load2(buf + 2 * p0, w[0][0], w[0][1]);
      wait(0);
#pragma unroll
      for (int q = 1; q < kU; ++q)
        if (p0 + q * nthr < np) ll_load2(buf + 2 * (p0 + q * nthr), w[q][0], w[q][1]);
#pragma unroll
      for (int q = 1; q < kU; ++q)
        if (p0 + q * nthr < np) wait(q);
#pragma unroll
      for (int q = 0; q < kU; ++q) {
        const int p = p0 + q * nthr;
        if (p >= np) break;
        if (wide) {
          const double x = __hiloint2double((int)(uint32_t)w[q][1], (int)(uint32_t)w[q][0]);
          x64[p] = x;
          if (!F64) x32[p] = (float)x;
        } else {
          const float f0 = __uint_as_float((uint32_t)w[q][0]);
          if (2 * p + 1 < M) *reinterpret_cast<float2*>(x32 + 2 * p) = make_float2(f0, __uint_as_float((uint32_t)w[q][1]));
          else x32[2 * p] = f0;
        }
      }
    }
  };

  // FP64 defect of the warp's rows at the v in x64: K + (A64 - A_lp) v
  auto correction = [&]() {
    if (!active) return;
#pragma unroll 1
    for (int r = 0; r < R && i0 + r < nr; ++r) {
      const int sr = r0 + i0 + r;
      double t = 0.0;
      if constexpr (!F64)
        t = lb::defect_dot<false>(A.A64 + (int64_t)sr * M, grows[0] + (size_t)r * M, PREC == LB_BF16 ? A.scale[sr] : 1.f, x64,
                           M, lane);
      for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
      if (lane == r) kf = k0 + t;
    }
  };

  const double h = A.h, h2 = 0.5 * A.h, h6 = A.h / 6.0;
  const int nk = (M + 127) >> 7;
  uint32_t g = 0;
  bool fix = first_correct;              // a correction before the next step
  int64_t since = A.t0 % A.correct_every;  // steps since the last
  for (int64_t t = 0; t < A.nsteps; ++t) {
    if (fix) {
      correction();
      fix = false;
    }
    since = since + 1 == A.correct_every ? 0 : since + 1;
    const bool next_fix = correct && since == 0;
#pragma unroll 1
    for (int stage = 1; stage <= 4; ++stage) {
      ++g;
      const bool wide = F64 || (stage == 4 && next_fix);
      unsigned long long* out = A.ll + (size_t)(g & 1) * A.bufw;
      if (active) {
        double y;
        if constexpr (F64) {
          double t_[R];
          if (res) rows_fp64<R, true>(rows, x64, M, lane, t_);
          else rows_fp64<R, false>(rows, x64, M, lane, t_);
          y = reduce_rows<R>(t_, lane);
        } else {
          if (res) {
            y = rows_resident<E, R>(rows, grows, head, he, te, x32, M, nk, lane);
          } else {
            y = 0.0;
#pragma unroll 1
            for (int r = 0; r < R && i0 + r < nr; ++r) {
              const double yr = row_global(grows[0] + (size_t)r * M, x32, M, lane);
              if (lane == r) y = yr;
            }
          }
          if (PREC == LB_BF16) y = __dmul_rn(y, sc);
        }
        if (holds) {
          const double k = y + kf;
          double nx;
          if (stage < 4) {
            nx = fma(stage == 3 ? h : h2, k, vs);
          } else {
            nx = fma(h6, ac + k, vs);
            vs = nx;
          }
          if (wide) {
            ll_store(out + 2 * (size_t)s, (uint32_t)__double2loint(nx), g);
            ll_store(out + 2 * (size_t)s + 1, (uint32_t)__double2hiint(nx), g);
          } else {
            ll_store(out + s, __float_as_uint((float)nx), g);
          }
          ac = stage == 1 ? k : fma(2.0, k, ac);
          if (stage == 4 && A.snaps && (A.t0 + t + 1) % A.snap_every == 0)
            A.snaps[((A.t0 + t + 1) / A.snap_every - 1) * (int64_t)M + s] = nx;
        }
      }
      if (stage == 4 && t + 1 == A.nsteps) break;
      __syncthreads();  // the block has read x
      poll(g, wide);
      __syncthreads();
    }
    fix = next_fix;
  }
  __syncthreads();
  if (holds) {
    A.v[s] = vs;
    A.keff_out[s] = kf;
  }
}

// Warps of a block; those without rows still poll.  No more than the rows need:
// a block of 16 takes all registers of an SM, and then the launches of several
// streams run one after the other.  us a step of all, 16 warps / now / with a
// launch per stage, 8 streams: FP32 N = 20 89 / 26 / 42, N = 30 101 / 25 / 48,
// N = 36 96 / 47 / 55, N = 44 109 / 62 / 92, FP64 N = 20 81 / 45 / 43, N = 30 137 / 92 /
// 69; one stream: FP32 N = 20 11.4 / 7.9, N = 30 13.8 / 8.8, N = 33 8.4 / 9.8, N = 44
// 13.9 / 11.4, FP64 N = 30 18.5 / 14.4 (fewer pollers leave L2 to the stores).
// FP64 rows are a warp's time each: two a warp cost more than they free (N = 40,
// one stream: 28 / 42), and so do four warps (N = 23 10.5 / 11.9) or eight for eight
// rows (N = 34 17.9 / 20.8).  Where a launch needs the registers or the shared
// memory of all SMs (FP64 N >= 33, else N >= 49) the streams still run one after
// the other: 8 streams of FP32 N = 50 128 against 119 with a launch per stage, FP64
// 532 against 389.
int block_warps(int64_t M, int nrows, bool f64) {
  if (M <= 200) return 8;
  if (f64) return nrows <= 7 ? 8 : kMaxWarps;
  return nrows <= 8 ? 4 : nrows <= 16 ? 8 : kMaxWarps;
}

template <int PREC>
const void* pick(int R) {
  return R == 1 ? (const void*)k_rk4_persist<PREC, 1> : (const void*)k_rk4_persist<PREC, 2>;
}

}  // namespace

namespace lbi {

// Measured against the stage launches (us a step, one launch / stage launches):
// FP64 N = 10: 6.6 / 25.0, N = 50: 62 / 89, N = 60: 102 / 115; FP32 N = 30:
// 12.0 / 26.5, N = 50: 25.4 / 34.8, N = 55: 31 / 43, N = 60: 40 / 43, N = 75:
// 255 / 124; BF16 N = 50: 33 / 41, N = 66: 56 / 50.  The gain ends where too
// many of a block's rows no longer fit its shared memory.
bool rk4_persist_applies(int64_t M, int precision) { return M <= (precision == LB_FP32 ? 3400 : 3600); }

cudaError_t rk4_persist(int64_t M, int precision, const void* Ap, const float* scale, const double* A64,
                        int correct_every, const double* K, double* v, double dt, int64_t nsteps, double* snaps,
                        int64_t snap_every, double* keff, void* ll, int* err, cudaStream_t st, bool* done) {
  *done = false;
  const bool f64 = precision == LB_FP64;
  const size_t esz = f64 ? 8 : precision == LB_FP32 ? 4 : 2;
  if ((reinterpret_cast<uintptr_t>(ll) & 15) || (reinterpret_cast<uintptr_t>(Ap) & (esz - 1))) return cudaSuccess;
  int dev = 0, sms = 0, optin = 0, coop = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
  if (e != cudaSuccess || !coop) return e;
  // rows per block: small systems gain more from fewer readers of the words
  // than from more blocks (N = 10: 2 rows 6.5 us a step, 1 row 7.4; N = 17: 4
  // rows 8.3, 1 row 13)
  const int rpb = M <= 128 ? 2 : 4;
  const int G = (int)std::min<int64_t>(sms, (M + rpb - 1) / rpb);
  PersistArgs a{};
  a.M = (int)M;
  a.nr = (int)(M / G);
  a.rem = (int)(M % G);
  const int nrows = a.nr + (a.rem ? 1 : 0);
  const int warps = block_warps(M, nrows, f64);
  const int R = nrows > warps ? 2 : 1;  // one round of rows: their state stays in registers
  if (nrows > R * warps) return cudaSuccess;
  a.xpad = (int)((M + 127) & ~int64_t(127)) + 32;  // the first lanes read up to 32 past the end
  a.pitch = f64 ? (int)((M + 31) & ~int64_t(31)) : (int)((M + 127) & ~int64_t(127));
  const bool correct = !f64 && correct_every > 0 && A64 != nullptr;
  const size_t fixed = (f64 || correct ? 8 : 0) * (size_t)a.xpad + (f64 ? 0 : 4) * (size_t)a.xpad;
  const size_t room = (size_t)optin - 1024;
  if (fixed > room) return cudaSuccess;
  a.nres = (int)std::min<size_t>((size_t)nrows, (room - fixed) / ((size_t)a.pitch * esz));
  const size_t smem = fixed + (size_t)a.nres * a.pitch * esz;
  a.Ap = Ap;
  a.scale = scale;
  a.A64 = correct ? A64 : nullptr;
  a.correct_every = correct ? correct_every : 1;
  a.snap_every = snap_every > 0 ? snap_every : 1;
  a.snaps = snap_every > 0 ? snaps : nullptr;
  a.K = K;
  a.keff_out = keff;
  a.v = v;
  a.h = dt;
  a.ll = static_cast<unsigned long long*>(ll);
  a.bufw = 2 * (size_t)M;
  a.err = err;
  a.poll_cycles = t_poll_cycles;
  const void* f = f64 ? pick<LB_FP64>(R) : precision == LB_FP32 ? pick<LB_FP32>(R) : pick<LB_BF16>(R);
  const int threads = 32 * warps;
  e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)room);
  int per = 0;
  if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, f, threads, smem);
  if (e != cudaSuccess) return e;
  if ((int64_t)per * sms < G) return cudaSuccess;
  const int64_t chunk = int64_t(1) << 29;  // stage numbers stay below 2^32
  for (int64_t t = 0; t < nsteps; t += chunk) {
    a.t0 = t;
    a.nsteps = std::min(chunk, nsteps - t);
    a.keff0 = t ? keff : nullptr;
    e = cudaMemsetAsync(ll, 0, 16 * a.bufw, st);
    if (e == cudaSuccess && t == 0) e = cudaMemsetAsync(err, 0, sizeof(int), st);
    if (e != cudaSuccess) return e;
    void* params[] = {&a};
    e = cudaLaunchCooperativeKernel(f, dim3((unsigned)G), dim3((unsigned)threads), params, smem, st);
    if (e == cudaErrorCooperativeLaunchTooLarge && t == 0) {  // a context with fewer SMs than the device
      cudaGetLastError();
      return cudaSuccess;
    }
    if (e != cudaSuccess) return e;
    note_launch(1);
  }
  *done = true;
  return cudaSuccess;
}

}  // namespace lbi

// For tests, not part of the ABI: the limit in clock cycles of one poll in this
// thread's later calls (negative: give up where a word has not come yet); returns the previous one.
extern "C" long long lbi_poll_cycles(long long cycles) {
  const long long before = t_poll_cycles;
  t_poll_cycles = cycles;
  return before;
}
