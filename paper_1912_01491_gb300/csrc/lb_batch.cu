// lb_batch.cu -- the batched form: many independent realizations of mixed N
// (the paper's Sec. 6 ensemble of random Lindbladians: one sample per group
// of processors, trivially parallel), assembled and then integrated by one
// persistent launch per cluster-size group.
//
// Integration: a thread-block cluster owns one realization at a time (taken
// from a global counter by the cluster's rank-0 block).  Each block of the
// cluster owns a contiguous slice of rows; as many of them as fit stay in
// shared memory for the whole 4 x nsteps stages, the others are re-read from
// global memory (L2) every stage.  Each block keeps the whole stage vector in
// its shared memory, double-buffered: while it reads one copy for the product,
// the epilogue of every row stores the row's next-stage value into the other
// copy of every block of the cluster (distributed shared memory stores, a warp
// of rows at a time), and one cluster barrier per stage orders those stores
// before the next stage reads them.  State, stage combination and the FP64
// defect correction stay FP64, as in the single-system kernels.
#include <cooperative_groups.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <type_traits>
#include <vector>

#include "lb_internal.h"
#include "lb_rowsum.cuh"

namespace cg = cooperative_groups;

namespace {

using BItem = lbi::BatchItem;

inline size_t a16(size_t x) { return (x + 15) & ~size_t(15); }

// RK4 form: shared memory of one block.  es: bytes of an element of the matrix
// and of the stage vector, 4 or 8.  room: elements of the matrix held.
struct SmemLayout {
  int64_t slice, mmax, room;
  size_t off_item, off_x, off_x64, off_v, off_acc, off_keff, off_sum, off_r, total;
};

SmemLayout layout(int64_t mmax, int C, bool resident, size_t es = sizeof(float)) {
  SmemLayout L;
  L.mmax = mmax;
  L.slice = (mmax + C - 1) / C;
  L.room = resident ? L.slice * mmax : 0;
  size_t o = 0;
  L.off_item = o; o = a16(o + 16);
  L.off_x = o; o = a16(o + es * 2 * mmax);
  L.off_x64 = o; if (es == sizeof(float)) o = a16(o + sizeof(double) * mmax);
  L.off_v = o; o = a16(o + sizeof(double) * L.slice);
  L.off_acc = o; o = a16(o + sizeof(double) * L.slice);
  L.off_keff = o; o = a16(o + sizeof(double) * L.slice);
  L.off_sum = o; o = a16(o + es * L.slice);
  L.off_r = o; o = a16(o + es * L.room);
  L.total = o;
  return L;
}

// Classical RK4 stage epilogue for one row (Table 1 step 3.1): k = A x + K,
// acc and the next stage input as in the single-system kernels.
// (dt6 = dt / 6).
__device__ __forceinline__ double stage_update(int stage, double k, double vi, double acci, double dt, double dt6,
                                               double* acc_out, double* v_out) {
  if (stage == 1) {
    *acc_out = k;
    return vi + 0.5 * dt * k;
  }
  if (stage == 2) {
    *acc_out = acci + 2.0 * k;
    return vi + 0.5 * dt * k;
  }
  if (stage == 3) {
    *acc_out = acci + 2.0 * k;
    return vi + dt * k;
  }
  const double nx = vi + dt6 * (acci + k);
  *v_out = nx;
  return nx;
}

// Lanes per row: small rows are shared by fewer lanes so that one warp
// instruction of the FP64 epilogue serves 32 / W rows.
__device__ __forceinline__ int row_group_width(int64_t M) {
  return M >= 256 ? 32 : M >= 96 ? 16 : M >= 32 ? 8 : 4;
}

// Multiply-add in the element type (an explicit FP32 FMA for float, so that
// no operand is promoted to FP64).
__device__ __forceinline__ float mad(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double mad(double a, double b, double c) { return fma(a, b, c); }

// Partial dot product of one lane of a W-lane row group.  Full-warp rows use
// a compile-time stride, which the compiler unrolls with the loads of several
// iterations in flight (long rows stream from L2); short rows use W lanes.
template <class T>
__device__ __forceinline__ T group_dot(const T* __restrict__ row, const T* __restrict__ x, int64_t M, int sub,
                                       int W) {
  T a = T(0);
  if (W == 32) {
    for (int64_t n = sub; n < M; n += 32) a = mad(row[n], x[n], a);
  } else {
    for (int64_t n = sub; n < M; n += W) a = mad(row[n], x[n], a);
  }
  return a;
}

// Partial dot products of one lane for R rows, each in the order of group_dot;
// the rows share the loads of x.
template <class T, int W, int R>
__device__ __forceinline__ void rows_dot(const T* const (&row)[R], const T* __restrict__ x, int M, int sub, T (&a)[R]) {
#pragma unroll
  for (int r = 0; r < R; ++r) a[r] = T(0);
#pragma unroll(R > 2 ? 4 : 8)
  for (int n = sub; n < M; n += W) {
    const T xn = x[n];
#pragma unroll
    for (int r = 0; r < R; ++r) a[r] = mad(row[r][n], xn, a[r]);
  }
}

// The same for long rows that are streamed: eight elements of every row are asked
// for before the first is used.
template <class T, int W, int R>
__device__ __forceinline__ void rows_dot_ahead(const T* const (&row)[R], const T* __restrict__ x, int M, int sub,
                                               T (&a)[R]) {
  constexpr int U = 8;
#pragma unroll
  for (int r = 0; r < R; ++r) a[r] = T(0);
  int n = sub;
  for (; n + (U - 1) * W < M; n += U * W) {
    T e[R][U];
#pragma unroll
    for (int u = 0; u < U; ++u)
#pragma unroll
      for (int r = 0; r < R; ++r) e[r][u] = __ldg(row[r] + n + u * W);
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const T xn = x[n + u * W];
#pragma unroll
      for (int r = 0; r < R; ++r) a[r] = mad(e[r][u], xn, a[r]);
    }
  }
  for (; n < M; n += W) {
    const T xn = x[n];
#pragma unroll
    for (int r = 0; r < R; ++r) a[r] = mad(row[r][n], xn, a[r]);
  }
}

// Sums of R rows over the W lanes of each group.  The additions of a row are
// those of the xor tree from W / 2 down; halves of the group take different
// rows, so four rows cost 6 shuffles in place of 20.  Row r is then with the
// lane r (W / R') of the group (R' = 1, 2 or 4).
template <class T, int W>
__device__ __forceinline__ T rows_sum(const T (&a)[1], int) {
  T t = a[0];
#pragma unroll
  for (int o = W / 2; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
  return t;
}
template <class T, int W>
__device__ __forceinline__ T rows_sum(const T (&a)[2], int sub) {
  const bool up = (sub & (W / 2)) != 0;
  T t = up ? a[1] : a[0];
  t += __shfl_xor_sync(0xffffffffu, up ? a[0] : a[1], W / 2);
#pragma unroll
  for (int o = W / 4; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
  return t;
}
template <class T, int W>
__device__ __forceinline__ T rows_sum(const T (&a)[4], int sub) {
  const bool up = (sub & (W / 2)) != 0, up2 = (sub & (W / 4)) != 0;
  T t0 = up ? a[2] : a[0], t1 = up ? a[3] : a[1];
  t0 += __shfl_xor_sync(0xffffffffu, up ? a[0] : a[2], W / 2);
  t1 += __shfl_xor_sync(0xffffffffu, up ? a[1] : a[3], W / 2);
  T t = up2 ? t1 : t0;
  t += __shfl_xor_sync(0xffffffffu, up2 ? t0 : t1, W / 4);
#pragma unroll
  for (int o = W / 8; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
  return t;
}
template <class T, int W>
__device__ __forceinline__ T rows_sum(const T (&a)[3], int sub) {
  const T b[4] = {a[0], a[1], a[2], T(0)};
  return rows_sum<T, W>(b, sub);
}

// Sums A x of the rows u G + g, u = u0, u0 + step, .. (R of them) of n, into sums.
template <class T, int W, int R, bool AHEAD = false>
__device__ __forceinline__ void rows_batch(const T* __restrict__ mat, int n, int u0, int step,
                                           const T* __restrict__ x, int M, int lane, T* __restrict__ sums) {
  constexpr int G = 32 / W, parts = R == 1 ? 1 : R == 2 ? 2 : 4;
  const int sub = lane % W, g = lane / W;
  const T* row[R];
#pragma unroll
  for (int r = 0; r < R; ++r) row[r] = mat + (int64_t)min((u0 + r * step) * G + g, n - 1) * M;
  T a[R];
  if constexpr (AHEAD) rows_dot_ahead<T, W, R>(row, x, M, sub, a);
  else rows_dot<T, W, R>(row, x, M, sub, a);
  const T t = rows_sum<T, W>(a, sub);
  const int r = sub / (W / parts), i = (u0 + r * step) * G + g;
  if (sub % (W / parts) == 0 && r < R && i < n) sums[i] = t;
}

// Sums A x of n rows, mat their first element (shared memory or global): the
// warps (w of nw) take every nw-th unit of 32 / W rows, up to four at a time.
template <class T, int W>
__device__ __forceinline__ void rows_stage(const T* __restrict__ mat, int n, const T* __restrict__ x, int M, int w,
                                           int nw, int lane, T* __restrict__ sums) {
  constexpr int G = 32 / W;
  const int units = (n + G - 1) / G;
  int left = (units - w + nw - 1) / nw;
  for (int u = w; left > 0;) {
    const int r = left >= 6 || left == 4 ? 4 : left >= 3 ? 3 : left;
    if (r == 4) rows_batch<T, W, 4>(mat, n, u, nw, x, M, lane, sums);
    else if (r == 3) rows_batch<T, W, 3>(mat, n, u, nw, x, M, lane, sums);
    else if (r == 2) rows_batch<T, W, 2>(mat, n, u, nw, x, M, lane, sums);
    else rows_batch<T, W, 1>(mat, n, u, nw, x, M, lane, sums);
    u += r * nw;
    left -= r;
  }
}

// The same for streamed rows of systems from M = kLongRow on: at most two rows a
// warp, eight elements of each ahead.  From N = 48 on the matrices of the clusters
// under way exceed L2, and four rows a warp with what the compiler asks for ahead
// left too few loads under way (30 steps, four rows / now: 16 of N = 64 69.7 /
// 42.1 ms, 24 of N = 48, 50 22.8 / 18.6; FP64, 16 of N = 64 126 / 100); below N = 44
// they are in L2, where four rows are quicker (48 of N = 40 8.6 / 9.4).
constexpr int kLongRow = 1900;

template <class T, int W>
__device__ __forceinline__ void rows_far(const T* __restrict__ mat, int n, const T* __restrict__ x, int M, int w, int nw,
                                         int lane, T* __restrict__ sums) {
  constexpr int G = 32 / W;
  int left = ((n + G - 1) / G - w + nw - 1) / nw;
  for (int u = w; left > 0; u += 2 * nw, left -= 2) {
    if (left >= 2) rows_batch<T, W, 2, true>(mat, n, u, nw, x, M, lane, sums);
    else rows_batch<T, W, 1, true>(mat, n, u, nw, x, M, lane, sums);
  }
}

// Takes the next realization for this cluster; every block returns the same
// queue position.
__device__ __forceinline__ int next_item(cg::cluster_group& cluster, int rank, int* item_slot, int* counter) {
  if (rank == 0 && threadIdx.x == 0) *item_slot = atomicAdd(counter, 1);
  cluster.sync();
  const int qi = *cluster.map_shared_rank(item_slot, 0);
  cluster.sync();  // every block has read the slot before rank 0 may overwrite it
  return qi;
}

__device__ __forceinline__ double wide(float x) { return lb::widen(x); }
__device__ __forceinline__ double wide(double x) { return x; }
__device__ __forceinline__ const float* matrix_of(const BItem& it, float) { return it.A32; }
__device__ __forceinline__ const double* matrix_of(const BItem& it, double) { return it.A64; }

// T = float: FP32 products of the FP32-rounded stage vector, state FP64, with
// the FP64 correction.  T = double: matrix, stage vector and products FP64, no
// correction.
// What bounds it: rows held, the shared memory reads (5 bytes a product, the
// matrix element and a quarter of x); rows streamed, L2.  At 40 levels a third
// of the matrix fits a cluster of 16.  FP32, 100 steps at the best cluster size:
// 48 of N = 39, 40 47.8 -> 23.1 ms, 64 of N = 33 .. 35 34.1 -> 18.1 ms, 128 of
// N = 26 .. 28 29.5 -> 13.2 ms, 256 of N = 10 .. 12 3.2 -> 1.0 ms; FP64, 30 steps,
// 64 of N = 33, 35 28.1 -> 21.9 ms, 256 of N = 18, 20 14.9 -> 9.9 ms (with one row a
// warp, its epilogue on every lane, and a slice held whole or not at all).
// LONG: for groups with a system of M >= kLongRow (a kernel of its own: with both
// forms in one, the others lost 4-7%).
template <class T, bool LONG>
__global__ void __launch_bounds__(512, 2) k_rk4_batch(const BItem* __restrict__ items, const int* __restrict__ order,
                                                      int nitems, int* __restrict__ counter, int64_t nsteps, double dt,
                                                      int correct_every, SmemLayout L) {
  constexpr bool kF32 = sizeof(T) == sizeof(float);
  extern __shared__ __align__(16) unsigned char smem[];
  cg::cluster_group cluster = cg::this_cluster();
  const int C = (int)cluster.num_blocks();
  const int rank = (int)cluster.block_rank();
  int* item_slot = reinterpret_cast<int*>(smem + L.off_item);
  T* x = reinterpret_cast<T*>(smem + L.off_x);  // [2][mmax]
  double* x64 = reinterpret_cast<double*>(smem + L.off_x64);  // FP32 only
  double* vv = reinterpret_cast<double*>(smem + L.off_v);
  double* acc = reinterpret_cast<double*>(smem + L.off_acc);
  double* keff = reinterpret_cast<double*>(smem + L.off_keff);
  T* sums = reinterpret_cast<T*>(smem + L.off_sum);
  T* Rs = reinterpret_cast<T*>(smem + L.off_r);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  const double dt6 = dt / 6.0;
  while (true) {
    const int qi = next_item(cluster, rank, item_slot, counter);
    if (qi >= nitems) break;
    const BItem it = items[order[qi]];
    const int M = (int)it.M;
    const int slice = (M + C - 1) / C;
    const int r0 = min(rank * slice, M), nrow = min(slice, M - r0);
    const int held = (int)min((int64_t)nrow, L.room / M);  // rows [0, held) of the slice
    const T* mat = matrix_of(it, T(0)) + (int64_t)r0 * M;
    const bool correct = kF32 && correct_every > 0 && it.A64 != nullptr;
    for (int i = threadIdx.x; i < nrow; i += blockDim.x) {
      vv[i] = it.v[r0 + i];
      keff[i] = it.K[r0 + i];
    }
    for (int e = threadIdx.x; e < held * M; e += blockDim.x) Rs[e] = mat[e];
    for (int n = threadIdx.x; n < M; n += blockDim.x) {
      x[n] = (T)it.v[n];
      if (kF32) x64[n] = it.v[n];
    }
    __syncthreads();
    for (int64_t t = 0; t < nsteps; ++t) {
      if (correct && t % correct_every == 0) {
        // FP64 defect c = (A64 - A32) v on own rows, with the full current v in x64
        for (int i = warp; i < nrow; i += nw) {
          const int64_t s = r0 + i;
          double c = lb::defect_dot<false>(it.A64 + s * M, it.A32 + s * M, 1.f, x64, M, lane);
          for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
          if (lane == 0) keff[i] = it.K[s] + c;
        }
        __syncthreads();
      }
      const bool push64 = correct && (t + 1) % correct_every == 0;
      for (int stage = 1; stage <= 4; ++stage) {
        const T* xc = x + ((stage - 1) & 1) * L.mmax;
        T* xn = x + (stage & 1) * L.mmax;
        auto products = [&](auto width) {
          constexpr int W = decltype(width)::value;
          auto streamed = [&] {
            const T* far = mat + (int64_t)held * M;
            if constexpr (LONG) rows_far<T, W>(far, nrow - held, xc, M, warp, nw, lane, sums + held);
            else rows_stage<T, W>(far, nrow - held, xc, M, warp, nw, lane, sums + held);
          };
          // every second warp begins with the streamed rows, so that shared memory and L2 are both busy
          if (warp & 1) streamed();
          rows_stage<T, W>(Rs, held, xc, M, nw - 1 - warp, nw, lane, sums);
          if (!(warp & 1)) streamed();
        };
        switch (row_group_width(M)) {
          case 32: products(std::integral_constant<int, 32>{}); break;
          case 16: products(std::integral_constant<int, 16>{}); break;
          case 8: products(std::integral_constant<int, 8>{}); break;
          default: products(std::integral_constant<int, 4>{}); break;
        }
        __syncthreads();
        // the epilogue with a thread a row: the FP64 pipe takes a warp instruction in some 60 cycles whatever its
        // active lanes, and with one row a warp it was a third of the time
        for (int i = threadIdx.x; i < nrow; i += blockDim.x) {
          const double vi = vv[i], ai = acc[i];
          double acc_new = ai, v_new = vi;
          const double nx = stage_update(stage, wide(sums[i]) + keff[i], vi, ai, dt, dt6, &acc_new, &v_new);
          acc[i] = acc_new;
          vv[i] = v_new;
          const T xv = (T)nx;
          for (int q = 0; q < C; ++q) {
            *cluster.map_shared_rank(xn + r0 + i, q) = xv;
            if (kF32 && stage == 4 && push64) *cluster.map_shared_rank(x64 + r0 + i, q) = nx;
          }
        }
        cluster.sync();  // every block's copy of the next stage vector is complete
      }
    }
    for (int i = threadIdx.x; i < nrow; i += blockDim.x) it.v[r0 + i] = vv[i];
    cluster.sync();  // all blocks are done with this realization's buffers
  }
}

// ---------------------------------------------------------------------------
// Propagator form (lb_prop.cu): one step is v <- v + h (D' v + c'), one
// product with the matrix and one exchange of the state per step.  The
// cluster layout is that of k_rk4_batch: each block owns a slice of rows and
// keeps its slice of D' in shared memory when it fits.
//   FP32: D' stored in FP32 (D32 = fl(A32 + R32), R32 = D' - A in FP32),
//     products FP32 FMAs of the FP32-rounded state, state FP64.  Every
//     correct_every steps the FP64 defect d = (A64 + R32 - D32) v is formed
//     from the FP64 state and added to c' until the next one: A64 - A32 is
//     the storage error of A and A32 + R32 - D32 the rounding of the sum,
//     the two FP32 errors of D' to first order (R32's own rounding is h|A|
//     times smaller).
//   FP64: D' in FP64, FP64 products, no correction.
struct PItem {
  int64_t M;
  const float* D32;   // FP32 form: D' (M x M)
  const float* R32;   // FP32 form: D' - A in FP32, for the correction
  const double* A64;  // FP32 form with correction: A; FP64 form: D' (FP64)
  const double* cp;   // c' (M)
  double* v;          // M, in/out
};

struct SmemLayoutP {
  int64_t slice, mmax;
  bool resident;
  size_t off_item, off_x32, off_x64, off_v, off_keff, off_r, total;
};

SmemLayoutP layoutP(int64_t mmax, int C, bool resident, bool f64) {
  SmemLayoutP L;
  L.mmax = mmax;
  L.slice = (mmax + C - 1) / C;
  L.resident = resident;
  size_t o = 0;
  L.off_item = o; o = a16(o + 16);
  L.off_x32 = o; o = a16(o + (f64 ? 0 : sizeof(float) * 2 * mmax));
  L.off_x64 = o; o = a16(o + sizeof(double) * (f64 ? 2 : 1) * mmax);
  L.off_v = o; o = a16(o + sizeof(double) * L.slice);
  L.off_keff = o; o = a16(o + sizeof(double) * L.slice);
  L.off_r = o;
  if (resident) o = a16(o + (f64 ? sizeof(double) : sizeof(float)) * L.slice * mmax);
  L.total = o;
  return L;
}

__global__ void __launch_bounds__(256, 4) k_prop_batch(const PItem* __restrict__ items, const int* __restrict__ order,
                                                    int nitems, int* __restrict__ counter, int64_t nsteps, double h,
                                                    int correct_every, SmemLayoutP L) {
  extern __shared__ __align__(16) unsigned char smem[];
  cg::cluster_group cluster = cg::this_cluster();
  const int C = (int)cluster.num_blocks();
  const int rank = (int)cluster.block_rank();
  int* item_slot = reinterpret_cast<int*>(smem + L.off_item);
  float* x32 = reinterpret_cast<float*>(smem + L.off_x32);  // [2][mmax]
  double* x64 = reinterpret_cast<double*>(smem + L.off_x64);
  double* vv = reinterpret_cast<double*>(smem + L.off_v);
  double* keff = reinterpret_cast<double*>(smem + L.off_keff);
  float* Ds = reinterpret_cast<float*>(smem + L.off_r);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  const int64_t mmax = L.mmax;
  while (true) {
    const int qi = next_item(cluster, rank, item_slot, counter);
    if (qi >= nitems) break;
    const PItem it = items[order[qi]];
    const int64_t M = it.M;
    const int64_t slice = (M + C - 1) / C;
    const int64_t r0 = rank * slice, r1 = r0 + slice < M ? r0 + slice : M;
    const int64_t nrow = r1 > r0 ? r1 - r0 : 0;
    const bool resident = L.resident;
    const bool correct = correct_every > 0 && it.A64 != nullptr && it.R32 != nullptr;
    for (int64_t i = threadIdx.x; i < nrow; i += blockDim.x) {
      vv[i] = it.v[r0 + i];
      keff[i] = it.cp[r0 + i];
    }
    if (resident)
      for (int64_t e = threadIdx.x; e < nrow * M; e += blockDim.x) Ds[e] = it.D32[r0 * M + e];
    for (int64_t n = threadIdx.x; n < M; n += blockDim.x) {
      x32[n] = (float)it.v[n];
      x64[n] = it.v[n];
    }
    __syncthreads();
    const int W = row_group_width(M), G = 32 / W, g = lane / W, sub = lane % W;
    for (int64_t t = 0; t < nsteps; ++t) {
      if (correct && t % correct_every == 0) {
        // FP64 defect d = (A64 + R32 - D32) v on own rows
        for (int64_t i = warp; i < nrow; i += nw) {
          const int64_t s = r0 + i;
          double d = 0.0;
          for (int64_t n = lane; n < M; n += 32) {
            const int64_t q = s * M + n;
            d = fma((it.A64[q] + (double)it.R32[q]) - (double)it.D32[q], x64[n], d);
          }
          for (int o = 16; o > 0; o >>= 1) d += __shfl_xor_sync(0xffffffffu, d, o);
          if (lane == 0) keff[i] = it.cp[s] + d;
        }
        __syncthreads();
      }
      const bool push64 = correct && (t + 1) % correct_every == 0;
      const float* xc = x32 + (t & 1) * mmax;
      float* xn = x32 + ((t + 1) & 1) * mmax;
      for (int64_t i0 = (int64_t)warp * G; i0 < nrow; i0 += (int64_t)nw * G) {
        const int64_t i = i0 + g;
        const bool valid = i < nrow;  // every lane reaches the shuffles
        float a = 0.f;
        if (valid) {
          const float* row = resident ? Ds + i * M : it.D32 + (r0 + i) * M;
          a = group_dot(row, xc, M, sub, W);
        }
        for (int o = W >> 1; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
        const double vi = valid ? vv[i] : 0.0, ki = valid ? keff[i] : 0.0;
        __syncwarp();
        if (valid) {
          const double nx = fma(h, (double)a + ki, vi);
          if (sub == 0) vv[i] = nx;
          for (int q = sub; q < C; q += W) {
            *cluster.map_shared_rank(xn + r0 + i, q) = (float)nx;
            if (push64) *cluster.map_shared_rank(x64 + r0 + i, q) = nx;
          }
        }
      }
      cluster.sync();  // every block's copy of the next state is complete
    }
    for (int64_t i = threadIdx.x; i < nrow; i += blockDim.x) it.v[r0 + i] = vv[i];
    cluster.sync();  // all blocks are done with this realization's buffers
  }
}

__global__ void __launch_bounds__(256, 4) k_prop_batch64(const PItem* __restrict__ items,
                                                      const int* __restrict__ order, int nitems,
                                                      int* __restrict__ counter, int64_t nsteps, double h,
                                                      SmemLayoutP L) {
  extern __shared__ __align__(16) unsigned char smem[];
  cg::cluster_group cluster = cg::this_cluster();
  const int C = (int)cluster.num_blocks();
  const int rank = (int)cluster.block_rank();
  int* item_slot = reinterpret_cast<int*>(smem + L.off_item);
  double* x = reinterpret_cast<double*>(smem + L.off_x64);  // [2][mmax]
  double* vv = reinterpret_cast<double*>(smem + L.off_v);
  double* keff = reinterpret_cast<double*>(smem + L.off_keff);
  double* Ds = reinterpret_cast<double*>(smem + L.off_r);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  const int64_t mmax = L.mmax;
  while (true) {
    const int qi = next_item(cluster, rank, item_slot, counter);
    if (qi >= nitems) break;
    const PItem it = items[order[qi]];
    const int64_t M = it.M;
    const int64_t slice = (M + C - 1) / C;
    const int64_t r0 = rank * slice, r1 = r0 + slice < M ? r0 + slice : M;
    const int64_t nrow = r1 > r0 ? r1 - r0 : 0;
    const bool resident = L.resident;
    for (int64_t i = threadIdx.x; i < nrow; i += blockDim.x) {
      vv[i] = it.v[r0 + i];
      keff[i] = it.cp[r0 + i];
    }
    if (resident)
      for (int64_t e = threadIdx.x; e < nrow * M; e += blockDim.x) Ds[e] = it.A64[r0 * M + e];
    for (int64_t n = threadIdx.x; n < M; n += blockDim.x) x[n] = it.v[n];
    __syncthreads();
    const int W = row_group_width(M), G = 32 / W, g = lane / W, sub = lane % W;
    for (int64_t t = 0; t < nsteps; ++t) {
      const double* xc = x + (t & 1) * mmax;
      double* xn = x + ((t + 1) & 1) * mmax;
      for (int64_t i0 = (int64_t)warp * G; i0 < nrow; i0 += (int64_t)nw * G) {
        const int64_t i = i0 + g;
        const bool valid = i < nrow;
        double a = 0.0;
        if (valid) {
          const double* row = resident ? Ds + i * M : it.A64 + (r0 + i) * M;
          a = group_dot(row, xc, M, sub, W);
        }
        for (int o = W >> 1; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
        const double vi = valid ? vv[i] : 0.0, ki = valid ? keff[i] : 0.0;
        __syncwarp();
        if (valid) {
          const double nx = fma(h, a + ki, vi);
          if (sub == 0) vv[i] = nx;
          for (int q = sub; q < C; q += W) *cluster.map_shared_rank(xn + r0 + i, q) = nx;
        }
      }
      cluster.sync();
    }
    for (int64_t i = threadIdx.x; i < nrow; i += blockDim.x) it.v[r0 + i] = vv[i];
    cluster.sync();
  }
}
}  // namespace

struct lb_batch {
  int count = 0;
  std::vector<int> N;
  std::vector<int64_t> M;
  std::vector<const double*> a, h;  // caller-owned device inputs
  std::vector<double*> v;           // caller-owned device state
  std::vector<lb_basis_t*> basis;   // one per distinct N (owned)
  std::vector<int> basis_of;
  std::vector<double*> A64, K;
  std::vector<float*> A32;
  std::vector<int> cluster;  // chosen cluster size per realization
  int precision = LB_FP32;   // storage and arithmetic of the integration
  int form = LB_FORM_RK4;    // stage-by-stage RK4 or the propagator form
  // propagator form, made for step prop_dt and precision prop_prec
  double prop_dt = 0.0;
  int prop_prec = -1;
  std::vector<float*> D32, R32;  // FP32: D' and D' - A
  std::vector<double*> D64, cp;  // FP64: D'; both: c'
  float prop_ms = 0.f;           // device time of the last formation
  BItem* d_items = nullptr;
  int* d_order = nullptr;
  int* d_counter = nullptr;
  void* d_prop_items = nullptr;
  cudaStream_t side[lbi::kBatchSide] = {};  // made at first use
  cudaEvent_t fork = nullptr, join[lbi::kBatchSide] = {};
};

namespace lbi {

cudaError_t batch_alloc(lb_batch* b) {
  for (int r = 0; r < b->count; ++r) {
    const size_t mm = (size_t)b->M[r] * (size_t)b->M[r];
    cudaError_t e;
    if ((e = cudaMalloc(&b->A64[r], 8 * mm)) != cudaSuccess) return e;
    if ((e = cudaMalloc(&b->A32[r], 4 * mm)) != cudaSuccess) return e;
    if ((e = cudaMalloc(&b->K[r], 8 * (size_t)b->M[r])) != cudaSuccess) return e;
  }
  cudaError_t e;
  if ((e = cudaMalloc(&b->d_items, sizeof(BItem) * b->count)) != cudaSuccess) return e;
  if ((e = cudaMalloc(&b->d_order, sizeof(int) * b->count)) != cudaSuccess) return e;
  return cudaMalloc(&b->d_counter, sizeof(int) * 8);
}

void prop_free(lb_batch* b) {
  for (auto* p : b->D32) cudaFree(p);
  for (auto* p : b->R32) cudaFree(p);
  for (auto* p : b->D64) cudaFree(p);
  for (auto* p : b->cp) cudaFree(p);
  b->D32.clear();
  b->R32.clear();
  b->D64.clear();
  b->cp.clear();
  cudaFree(b->d_prop_items);
  b->d_prop_items = nullptr;
  b->prop_prec = -1;
}

void batch_free(lb_batch* b) {
  prop_free(b);
  for (int r = 0; r < b->count; ++r) {
    cudaFree(b->A64[r]);
    cudaFree(b->A32[r]);
    cudaFree(b->K[r]);
  }
  cudaFree(b->d_items);
  cudaFree(b->d_order);
  cudaFree(b->d_counter);
  for (int i = 0; i < kBatchSide; ++i) {
    if (b->side[i]) cudaStreamDestroy(b->side[i]);
    if (b->join[i]) cudaEventDestroy(b->join[i]);
  }
  if (b->fork) cudaEventDestroy(b->fork);
}

// The batch's side streams behind what is queued on st ..
cudaError_t batch_fork(lb_batch* b, cudaStream_t st) {
  cudaError_t e = cudaSuccess;
  if (!b->fork && (e = cudaEventCreateWithFlags(&b->fork, cudaEventDisableTiming)) != cudaSuccess) return e;
  if ((e = cudaEventRecord(b->fork, st)) != cudaSuccess) return e;
  for (int i = 0; i < kBatchSide; ++i) {
    if (!b->side[i] && (e = cudaStreamCreateWithFlags(&b->side[i], cudaStreamNonBlocking)) != cudaSuccess) return e;
    if (!b->join[i] && (e = cudaEventCreateWithFlags(&b->join[i], cudaEventDisableTiming)) != cudaSuccess) return e;
    if ((e = cudaStreamWaitEvent(b->side[i], b->fork, 0)) != cudaSuccess) return e;
  }
  return cudaSuccess;
}

// .. and st behind the side streams, whatever `before` says; the first error.
cudaError_t batch_join(lb_batch* b, cudaStream_t st, cudaError_t before) {
  for (int i = 0; i < kBatchSide; ++i) {
    if (!b->side[i] || !b->join[i]) continue;
    cudaError_t e = cudaEventRecord(b->join[i], b->side[i]);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(st, b->join[i], 0);
    if (before == cudaSuccess) before = e;
  }
  return before;
}

// Realizations are independent, and the kernels of one assembly at N <= 64 are
// chains of a few microseconds on a part of the chip: they go round the side
// streams (256 of N = 4 .. 40: 29 -> 11 ms).
cudaError_t batch_assemble(lb_batch* b, const std::vector<lb::BasisView>& views, int algorithm, cudaStream_t st) {
  cudaError_t e = batch_fork(b, st);
  for (int r = 0; r < b->count && e == cudaSuccess; ++r) {
    const lb::BasisView& B = views[b->basis_of[r]];
    cudaStream_t s = b->side[r % kBatchSide];
    e = assemble_dense(B, b->h[r], reinterpret_cast<const double2*>(b->a[r]), b->A64[r], nullptr, nullptr, b->K[r],
                       algorithm, s);
    if (e == cudaSuccess) e = pack_fp32(b->M[r], b->A64[r], b->A32[r], s);
  }
  if ((e = batch_join(b, st, e)) != cudaSuccess) return e;
  return cudaGetLastError();
}

// D' and c' of every realization for step h in the batch's precision
// (lb_prop.cu): G0 = A + (h/4) A A, G1 = A + (h/3) A G0, R' = (h/2) A G1,
// D' = A + R' (FP32 from A32, or FP64 from A64); c' from A64 in FP64.
cudaError_t batch_form_propagator(lb_batch* b, double h, cudaStream_t st) {
  const bool f64 = b->precision == LB_FP64;
  if (b->prop_prec != -1 && b->prop_prec == b->precision && b->prop_dt == h) return cudaSuccess;
  prop_free(b);
  const int n = b->count;
  cudaError_t e = cudaSuccess;
  b->cp.assign(n, nullptr);
  if (f64) {
    b->D64.assign(n, nullptr);
  } else {
    b->D32.assign(n, nullptr);
    b->R32.assign(n, nullptr);
  }
  std::vector<void*> tmp;
  auto scratch_free = [&]() {
    for (auto* p : tmp) cudaFree(p);
    tmp.clear();
  };
  for (int r = 0; r < n && e == cudaSuccess; ++r) {
    const size_t mm = (size_t)b->M[r] * (size_t)b->M[r];
    e = cudaMalloc(&b->cp[r], 8 * (size_t)b->M[r]);
    if (e == cudaSuccess) e = f64 ? cudaMalloc(&b->D64[r], 8 * mm) : cudaMalloc(&b->D32[r], 4 * mm);
    if (e == cudaSuccess && !f64) e = cudaMalloc(&b->R32[r], 4 * mm);
  }
  if (e == cudaSuccess) e = cudaMalloc(&b->d_prop_items, sizeof(PItem) * n);
  // scratch: G0, G1 per realization, the job lists, the GEMV vectors
  std::vector<void*> G0(n, nullptr), G1(n, nullptr), u(n, nullptr);
  const size_t esz = f64 ? 8 : 4;
  for (int r = 0; r < n && e == cudaSuccess; ++r) {
    const size_t mm = (size_t)b->M[r] * (size_t)b->M[r];
    if ((e = cudaMalloc(&G0[r], esz * mm)) == cudaSuccess) tmp.push_back(G0[r]);
    if (e == cudaSuccess && (e = cudaMalloc(&G1[r], esz * mm)) == cudaSuccess) tmp.push_back(G1[r]);
    if (e == cudaSuccess && (e = cudaMalloc(&u[r], 16 * (size_t)b->M[r])) == cudaSuccess) tmp.push_back(u[r]);
  }
  const size_t sb = std::max(batch_gemm_scratch_bytes(b->M), sizeof(GemvJob) * (size_t)n + 256);
  void* js = nullptr;
  if (e == cudaSuccess && (e = cudaMalloc(&js, sb)) == cudaSuccess) tmp.push_back(js);
  cudaEvent_t t0 = nullptr, t1 = nullptr;
  if (e == cudaSuccess) e = cudaEventCreate(&t0);
  if (e == cudaSuccess) e = cudaEventCreate(&t1);
  if (e == cudaSuccess) e = cudaEventRecord(t0, st);
  // the three products
  for (int step = 0; step < 3 && e == cudaSuccess; ++step) {
    const double alpha = step == 0 ? h / 4.0 : step == 1 ? h / 3.0 : h / 2.0;
    if (f64) {
      std::vector<GemmJob<double>> jobs;
      for (int r = 0; r < n; ++r) {
        const double* A = b->A64[r];
        const double* G = step == 0 ? A : step == 1 ? static_cast<double*>(G0[r]) : static_cast<double*>(G1[r]);
        double* Y = step == 0 ? static_cast<double*>(G0[r]) : step == 1 ? static_cast<double*>(G1[r]) : b->D64[r];
        jobs.push_back(GemmJob<double>{b->M[r], A, G, step == 2 ? nullptr : A, Y, alpha});
      }
      e = batch_gemm<double>(jobs, js, sb, st);
    } else {
      std::vector<GemmJob<float>> jobs;
      for (int r = 0; r < n; ++r) {
        const float* A = b->A32[r];
        const float* G = step == 0 ? A : step == 1 ? static_cast<float*>(G0[r]) : static_cast<float*>(G1[r]);
        float* Y = step == 0 ? static_cast<float*>(G0[r]) : step == 1 ? static_cast<float*>(G1[r]) : b->R32[r];
        jobs.push_back(GemmJob<float>{b->M[r], A, G, step == 2 ? nullptr : A, Y, (float)alpha});
      }
      e = batch_gemm<float>(jobs, js, sb, st);
    }
  }
  // D' = A + R'
  for (int r = 0; r < n && e == cudaSuccess; ++r) {
    const int64_t mm = b->M[r] * b->M[r];
    e = f64 ? add64(b->A64[r], b->D64[r], b->D64[r], mm, st) : add32(b->A32[r], b->R32[r], b->D32[r], mm, st);
  }
  // c' = K + (h/2) A (K + (h/3) A (K + (h/4) A K)) in FP64
  for (int step = 0; step < 3 && e == cudaSuccess; ++step) {
    const double alpha = step == 0 ? h / 4.0 : step == 1 ? h / 3.0 : h / 2.0;
    std::vector<GemvJob> jobs;
    for (int r = 0; r < n; ++r) {
      double* ua = static_cast<double*>(u[r]);
      double* ub = ua + b->M[r];
      const double* x = step == 0 ? b->K[r] : step == 1 ? ua : ub;
      double* y = step == 0 ? ua : step == 1 ? ub : b->cp[r];
      jobs.push_back(GemvJob{b->M[r], b->A64[r], x, b->K[r], y, alpha});
    }
    e = batch_gemv64(jobs, js, sb, st);
  }
  if (e == cudaSuccess) e = cudaEventRecord(t1, st);
  if (e == cudaSuccess) e = cudaEventSynchronize(t1);
  if (e == cudaSuccess) e = cudaEventElapsedTime(&b->prop_ms, t0, t1);
  if (t0) cudaEventDestroy(t0);
  if (t1) cudaEventDestroy(t1);
  scratch_free();
  if (e != cudaSuccess) {
    prop_free(b);
    return e;
  }
  b->prop_dt = h;
  b->prop_prec = b->precision;
  return cudaSuccess;
}

int smem_optin() {
  int dev = 0, v = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&v, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  return v;
}

// Shared-memory layout for (mmax, C): as many rows as fit; total 0 if not even
// the vectors do.  FP64 slices that do not fit whole leave room for a second
// block on the SM (an SM then takes two realizations, and one's FP64 sums run
// beside the other's loads and barriers): 30 steps, one block / two, the best
// cluster size, 32 of N = 33, 35 14.5 / 12.3 ms, 48 of N = 36 26.4 / 20.8, 48 of
// N = 40 43.0 / 31.3, 16 of N = 64 equal.  In FP32 the rows held are worth more
// (48 of N = 40 8.6 / 13.3).
SmemLayout pick_layout(int64_t mmax, int C, size_t es) {
  constexpr size_t kReserved = 1024;  // of an SM's shared memory, a block
  size_t cap = (size_t)smem_optin();
  SmemLayout L = layout(mmax, C, true, es);
  if (L.total <= cap) return L;
  L = layout(mmax, C, false, es);
  if (L.total > cap) {
    L.total = 0;
    return L;
  }
  const size_t half = (cap + kReserved) / 2 - kReserved;
  if (es == sizeof(double) && L.total <= half) cap = half;
  L.room = (int64_t)((cap - L.total) / es);
  L.total = cap;
  return L;
}

SmemLayoutP pick_layoutP(int64_t mmax, int C, bool f64) {
  const size_t cap = (size_t)smem_optin();
  SmemLayoutP L = layoutP(mmax, C, true, f64);
  if (L.total > cap) L = layoutP(mmax, C, false, f64);
  if (L.total > cap) L.total = 0;
  return L;
}

template <class T>
auto rk4_kernel(int64_t mmax) {
  return mmax >= kLongRow ? k_rk4_batch<T, true> : k_rk4_batch<T, false>;
}

// Threads of a block of k_rk4_batch: where the shared memory leaves room for
// one block an SM, or rows are streamed, 16 warps keep enough loads under way.
int rk4_threads(const SmemLayout& L) {
  return 2 * L.total > (size_t)smem_optin() || L.room < L.slice * L.mmax ? 512 : 256;
}

// Launch configuration of a batched kernel (func) for n items at cluster size
// C with smem bytes of dynamic shared memory; the number of clusters is what
// the device can hold at once, capped at n.  The dynamic shared-memory limit
// is raised to the device maximum (the same value from every thread), so
// concurrent launches never see a smaller limit.
cudaError_t configure(const void* func, int C, size_t smem, int n, int threads, cudaStream_t st, cudaLaunchConfig_t* cfg,
                      cudaLaunchAttribute* attr) {
  cudaError_t e = cudaFuncSetAttribute(func, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_optin());
  if (e != cudaSuccess) return e;
  if (C > 8) {
    e = cudaFuncSetAttribute(func, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
  }
  *cfg = cudaLaunchConfig_t{};
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = C;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg->blockDim = dim3((unsigned)threads, 1, 1);
  cfg->dynamicSmemBytes = smem;
  cfg->stream = st;
  cfg->attrs = attr;
  cfg->numAttrs = 1;
  cfg->gridDim = dim3((unsigned)C, 1, 1);
  int clusters = 0;
  e = cudaOccupancyMaxActiveClusters(&clusters, func, cfg);
  if (e != cudaSuccess) return e;
  if (clusters < 1) return cudaErrorInvalidConfiguration;
  clusters = std::min<int>(clusters, n);
  cfg->gridDim = dim3((unsigned)(clusters * C), 1, 1);
  return cudaSuccess;
}

// The propagator form of batch_run_group (formed for dt beforehand).
cudaError_t batch_run_group_prop(lb_batch* b, const std::vector<int>& ids, int C, int64_t mmax, int64_t nsteps,
                                 double dt, int correct_every, cudaStream_t st, float* ms) {
  const bool f64 = b->precision == LB_FP64;
  cudaError_t e = batch_form_propagator(b, dt, st);
  if (e != cudaSuccess) return e;
  const SmemLayoutP L = pick_layoutP(mmax, C, f64);
  if (L.total == 0) return cudaErrorInvalidConfiguration;
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute attr[1];
  e = f64 ? configure((const void*)k_prop_batch64, C, L.total, (int)ids.size(), 256, st, &cfg, attr)
          : configure((const void*)k_prop_batch, C, L.total, (int)ids.size(), 256, st, &cfg, attr);
  if (e != cudaSuccess) return e;
  std::vector<int> ord(ids.begin(), ids.end());
  std::sort(ord.begin(), ord.end(), [&](int x, int y) { return b->M[x] > b->M[y]; });
  std::vector<PItem> host(b->count);
  for (int r = 0; r < b->count; ++r) {
    if (f64)
      host[r] = PItem{b->M[r], nullptr, nullptr, b->D64[r], b->cp[r], b->v[r]};
    else
      host[r] = PItem{b->M[r], b->D32[r], b->R32[r], correct_every > 0 ? b->A64[r] : nullptr, b->cp[r], b->v[r]};
  }
  if ((e = cudaMemcpyAsync(b->d_prop_items, host.data(), sizeof(PItem) * b->count, cudaMemcpyHostToDevice, st)) !=
      cudaSuccess)
    return e;
  if ((e = cudaMemcpyAsync(b->d_order, ord.data(), sizeof(int) * ord.size(), cudaMemcpyHostToDevice, st)) !=
      cudaSuccess)
    return e;
  if ((e = cudaMemsetAsync(b->d_counter, 0, sizeof(int), st)) != cudaSuccess) return e;
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  if (ms) {
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    cudaEventRecord(e0, st);
  }
  const PItem* items = static_cast<const PItem*>(b->d_prop_items);
  if (f64)
    e = cudaLaunchKernelEx(&cfg, k_prop_batch64, items, (const int*)b->d_order, (int)ord.size(), b->d_counter, nsteps,
                           dt, L);
  else
    e = cudaLaunchKernelEx(&cfg, k_prop_batch, items, (const int*)b->d_order, (int)ord.size(), b->d_counter, nsteps,
                           dt, correct_every, L);
  note_launch(1);
  if (ms) {
    cudaEventRecord(e1, st);
    cudaEventSynchronize(e1);
    cudaEventElapsedTime(ms, e0, e1);
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
  }
  if (e != cudaSuccess) return e;
  // the item list is read by the kernel: keep it until the launch is done
  return cudaStreamSynchronize(st);
}

// The RK4 form's item list (for every group).
cudaError_t batch_upload_items(lb_batch* b, int correct_every, cudaStream_t st) {
  const bool a64 = correct_every > 0 || b->precision == LB_FP64;
  std::vector<BItem> host(b->count);
  for (int r = 0; r < b->count; ++r)
    host[r] = BItem{b->M[r], b->A32[r], a64 ? b->A64[r] : nullptr, b->K[r], b->v[r]};
  return cudaMemcpyAsync(b->d_items, host.data(), sizeof(BItem) * b->count, cudaMemcpyHostToDevice, st);
}

// Launch the RK4 form for the realizations `ids` (one cluster size C), the item
// list uploaded; `at`: their place in the order list, `slot`: their counter.
// A cluster size the device cannot place with the needed shared memory fails
// with cudaErrorInvalidConfiguration before any launch.
cudaError_t batch_launch_group(lb_batch* b, const std::vector<int>& ids, int C, size_t at, int slot, int64_t nsteps,
                               double dt, int correct_every, cudaStream_t st) {
  int64_t mmax = 0;
  for (int r : ids) mmax = std::max<int64_t>(mmax, b->M[r]);
  const bool f64 = b->precision == LB_FP64;
  const SmemLayout L = pick_layout(mmax, C, f64 ? sizeof(double) : sizeof(float));
  if (L.total == 0) return cudaErrorInvalidConfiguration;
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute attr[1];
  auto kernel = f64 ? rk4_kernel<double>(mmax) : rk4_kernel<float>(mmax);
  cudaError_t e = configure((const void*)kernel, C, L.total, (int)ids.size(), rk4_threads(L), st, &cfg, attr);
  if (e != cudaSuccess) return e;
  // items in decreasing order of work (largest first)
  std::vector<int> ord(ids.begin(), ids.end());
  std::sort(ord.begin(), ord.end(), [&](int x, int y) { return b->M[x] > b->M[y]; });
  if ((e = cudaMemcpyAsync(b->d_order + at, ord.data(), sizeof(int) * ord.size(), cudaMemcpyHostToDevice, st)) !=
      cudaSuccess)
    return e;
  if ((e = cudaMemsetAsync(b->d_counter + slot, 0, sizeof(int), st)) != cudaSuccess) return e;
  e = cudaLaunchKernelEx(&cfg, kernel, (const BItem*)b->d_items, (const int*)(b->d_order + at), (int)ord.size(),
                         b->d_counter + slot, nsteps, dt, correct_every, L);
  note_launch(1);
  return e;
}

// Run the realizations `ids` (one cluster size C) for nsteps; synchronous when
// ms is requested.
cudaError_t batch_run_group(lb_batch* b, const std::vector<int>& ids, int C, int64_t nsteps, double dt,
                            int correct_every, cudaStream_t st, float* ms) {
  if (ids.empty()) {
    if (ms) *ms = 0.f;
    return cudaSuccess;
  }
  if (b->form == LB_FORM_PROPAGATOR) {
    int64_t mmax = 0;
    for (int r : ids) mmax = std::max<int64_t>(mmax, b->M[r]);
    return batch_run_group_prop(b, ids, C, mmax, nsteps, dt, correct_every, st, ms);
  }
  cudaError_t e = batch_upload_items(b, correct_every, st);
  if (e != cudaSuccess) return e;
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  if (ms) {
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    cudaEventRecord(e0, st);
  }
  e = batch_launch_group(b, ids, C, 0, 0, nsteps, dt, correct_every, st);
  if (ms) {
    cudaEventRecord(e1, st);
    cudaEventSynchronize(e1);
    cudaEventElapsedTime(ms, e0, e1);
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
  }
  if (e != cudaSuccess) return e;
  return cudaGetLastError();
}

// All realizations in the RK4 form, a group per cluster size, the groups on the
// side streams: they share nothing, and one after the other each would leave
// the chip half empty for the length of its last realizations (256 of N = 4 ..
// 40, 100 steps: 33.5 -> 28.1 ms).  Large clusters first, they need whole GPCs;
// but a group of far lighter blocks goes behind the heavier one: placed first, the
// light blocks keep the heavy ones off their SMs, which then crowd the rest (FP64,
// 128 of N = 9 with clusters of 1 and 128 of N = 4 with clusters of 2, 300 steps:
// light first 12.2 ms, one after the other 5.5).
cudaError_t batch_run_groups(lb_batch* b, int64_t nsteps, double dt, int correct_every, cudaStream_t st, float* ms) {
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  cudaError_t e = cudaSuccess;
  if (ms) {
    if ((e = cudaEventCreate(&e0)) == cudaSuccess) e = cudaEventCreate(&e1);
    if (e == cudaSuccess) e = cudaEventRecord(e0, st);
  }
  if (e == cudaSuccess) e = batch_upload_items(b, correct_every, st);
  if (e == cudaSuccess) {
    e = batch_fork(b, st);
    struct Group {
      int C;
      double work;  // of a block, the largest realization
      std::vector<int> ids;
    };
    std::vector<Group> groups;
    for (int C : {16, 8, 4, 2, 1}) {
      Group g{C, 0.0, {}};
      for (int r = 0; r < b->count; ++r)
        if (b->cluster[r] == C) {
          g.ids.push_back(r);
          g.work = std::max(g.work, (double)b->M[r] * (double)b->M[r] / C);
        }
      if (!g.ids.empty()) groups.push_back(std::move(g));
    }
    for (size_t n = groups.size(); n > 1; --n)
      for (size_t i = 0; i + 1 < n; ++i)
        if (groups[i + 1].work > 8.0 * groups[i].work) std::swap(groups[i], groups[i + 1]);
    size_t at = 0;
    int slot = 0;
    for (const Group& g : groups) {
      if (e == cudaSuccess)
        e = batch_launch_group(b, g.ids, g.C, at, slot, nsteps, dt, correct_every, b->side[slot % kBatchSide]);
      at += g.ids.size();
      ++slot;
    }
    e = batch_join(b, st, e);
  }
  if (ms) {
    *ms = 0.f;
    if (e == cudaSuccess) e = cudaEventRecord(e1, st);
    if (e == cudaSuccess) e = cudaEventSynchronize(e1);
    if (e == cudaSuccess) e = cudaEventElapsedTime(ms, e0, e1);
    if (e0) cudaEventDestroy(e0);
    if (e1) cudaEventDestroy(e1);
  }
  return e == cudaSuccess ? cudaGetLastError() : e;
}

int batch_default_cluster(int64_t M) {
  const size_t cap = (size_t)smem_optin();
  for (int C : {1, 2, 4, 8, 16})
    if (layout(M, C, true).total <= cap) return C;
  return 16;
}

cudaError_t batch_launch_async(const BatchItem* items, int n, int C, int64_t nsteps, double dt, int correct_every,
                               cudaMemPool_t pool, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  int64_t mmax = 0;
  for (int i = 0; i < n; ++i) mmax = std::max<int64_t>(mmax, items[i].M);
  const SmemLayout L = pick_layout(mmax, C, sizeof(float));
  if (L.total == 0) return cudaErrorInvalidConfiguration;
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute attr[1];
  auto kernel = rk4_kernel<float>(mmax);
  cudaError_t e = configure((const void*)kernel, C, L.total, n, rk4_threads(L), st, &cfg, attr);
  if (e != cudaSuccess) return e;
  std::vector<int> ord(n);
  for (int i = 0; i < n; ++i) ord[i] = i;
  std::sort(ord.begin(), ord.end(), [&](int x, int y) { return items[x].M > items[y].M; });
  // one block: items, then order, then the counter
  const size_t bi = sizeof(BItem) * (size_t)n, bo = sizeof(int) * (size_t)n;
  const size_t off_o = (bi + 255) & ~size_t(255), off_c = (off_o + bo + 255) & ~size_t(255);
  std::vector<unsigned char> host(off_c + sizeof(int), 0);
  std::memcpy(host.data(), items, bi);
  std::memcpy(host.data() + off_o, ord.data(), bo);
  void* d = nullptr;
  if ((e = cudaMallocFromPoolAsync(&d, host.size(), pool, st)) != cudaSuccess) return e;
  unsigned char* db = static_cast<unsigned char*>(d);
  e = cudaMemcpyAsync(d, host.data(), host.size(), cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess)
    e = cudaLaunchKernelEx(&cfg, kernel, reinterpret_cast<const BItem*>(db),
                           reinterpret_cast<const int*>(db + off_o), n, reinterpret_cast<int*>(db + off_c), nsteps,
                           dt, correct_every, L);
  note_launch(1);
  const cudaError_t ef = cudaFreeAsync(d, st);
  if (e != cudaSuccess) return e;
  if (ef != cudaSuccess) return ef;
  return cudaGetLastError();
}

}  // namespace lbi

// ------------------------------------------------------------------ ABI

extern "C" {

int lb_batch_create(int count, const int* Ns, lb_batch_t** out) {
  if (!out || !Ns || count <= 0) {
    lbi::set_error("lb_batch_create: bad arguments");
    return LB_EINVAL;
  }
  *out = nullptr;
  lb_batch* b = new lb_batch;
  b->count = count;
  b->N.assign(Ns, Ns + count);
  b->M.resize(count);
  b->a.assign(count, nullptr);
  b->h.assign(count, nullptr);
  b->v.assign(count, nullptr);
  b->A64.assign(count, nullptr);
  b->A32.assign(count, nullptr);
  b->K.assign(count, nullptr);
  b->cluster.assign(count, 1);
  b->basis_of.assign(count, -1);
  std::vector<int> distinct;
  for (int r = 0; r < count; ++r) {
    if (Ns[r] < 2 || Ns[r] > lbi::kBatchMaxN) {
      lbi::set_error("lb_batch_create: N = %d outside [2, %d]", Ns[r], lbi::kBatchMaxN);
      delete b;
      return LB_EINVAL;
    }
    b->M[r] = (int64_t)Ns[r] * Ns[r] - 1;
    auto it = std::find(distinct.begin(), distinct.end(), Ns[r]);
    if (it == distinct.end()) {
      distinct.push_back(Ns[r]);
      b->basis_of[r] = (int)distinct.size() - 1;
    } else {
      b->basis_of[r] = (int)(it - distinct.begin());
    }
  }
  for (int n : distinct) {
    lb_basis_t* bb = nullptr;
    int rc = lb_basis_create(n, nullptr, &bb);
    if (rc != LB_OK) {
      for (auto* x : b->basis) lb_basis_destroy(x);
      delete b;
      return rc;
    }
    b->basis.push_back(bb);
  }
  cudaError_t e = lbi::batch_alloc(b);
  if (e != cudaSuccess) {
    lbi::batch_free(b);
    for (auto* x : b->basis) lb_basis_destroy(x);
    delete b;
    cudaGetLastError();
    lbi::set_error("lb_batch_create: device allocation failed (%s)", cudaGetErrorString(e));
    return e == cudaErrorMemoryAllocation ? LB_ENOMEM : LB_ECUDA;
  }
  *out = b;
  return LB_OK;
}

int lb_batch_set(lb_batch_t* b, int r, const double* a, const double* h, double* v) {
  if (!b || r < 0 || r >= b->count || !a || !v) {
    lbi::set_error("lb_batch_set: bad arguments");
    return LB_EINVAL;
  }
  b->a[r] = a;
  b->h[r] = h;
  b->v[r] = v;
  return LB_OK;
}

int lb_batch_assemble(lb_batch_t* b, int algorithm, void* stream) {
  if (!b) {
    lbi::set_error("lb_batch_assemble: NULL batch");
    return LB_EINVAL;
  }
  for (int r = 0; r < b->count; ++r)
    if (!b->a[r] || !b->v[r]) {
      lbi::set_error("lb_batch_assemble: realization %d has no inputs (lb_batch_set)", r);
      return LB_EINVAL;
    }
  std::vector<lb::BasisView> views;
  for (auto* x : b->basis) views.push_back(x->view());
  cudaError_t e = lbi::batch_assemble(b, views, algorithm, static_cast<cudaStream_t>(stream));
  if (e == cudaSuccess) e = cudaStreamSynchronize(static_cast<cudaStream_t>(stream));
  if (e != cudaSuccess) return lbi::cuda_fail(e, "lb_batch_assemble");
  return LB_OK;
}

int lb_batch_set_cluster(lb_batch_t* b, int r, int C) {
  if (!b || r < 0 || r >= b->count || !(C == 1 || C == 2 || C == 4 || C == 8 || C == 16)) {
    lbi::set_error("lb_batch_set_cluster: bad arguments");
    return LB_EINVAL;
  }
  b->cluster[r] = C;
  return LB_OK;
}

int lb_batch_set_precision(lb_batch_t* b, int precision) {
  if (!b || (precision != LB_FP32 && precision != LB_FP64)) {
    lbi::set_error("lb_batch_set_precision: bad arguments (LB_FP32 or LB_FP64)");
    return LB_EINVAL;
  }
  b->precision = precision;
  return LB_OK;
}

int lb_batch_set_form(lb_batch_t* b, int form) {
  if (!b || (form != LB_FORM_RK4 && form != LB_FORM_PROPAGATOR)) {
    lbi::set_error("lb_batch_set_form: bad arguments (LB_FORM_RK4 or LB_FORM_PROPAGATOR)");
    return LB_EINVAL;
  }
  b->form = form;
  return LB_OK;
}

int lb_batch_form_propagator(lb_batch_t* b, double dt, void* stream, float* ms) {
  if (!b || !(dt > 0.0) || !std::isfinite(dt)) {
    lbi::set_error("lb_batch_form_propagator: bad arguments");
    return LB_EINVAL;
  }
  cudaError_t e = lbi::batch_form_propagator(b, dt, static_cast<cudaStream_t>(stream));
  if (e != cudaSuccess) {
    if (e == cudaErrorMemoryAllocation) {
      cudaGetLastError();
      lbi::set_error("lb_batch_form_propagator: device memory exhausted");
      return LB_ENOMEM;
    }
    return lbi::cuda_fail(e, "lb_batch_form_propagator");
  }
  if (ms) *ms = b->prop_ms;
  return LB_OK;
}

int lb_batch_integrate(lb_batch_t* b, int correct_every, double dt, int64_t nsteps, void* stream, float* ms) {
  if (!b || nsteps < 0 || correct_every < 0) {
    lbi::set_error("lb_batch_integrate: bad arguments");
    return LB_EINVAL;
  }
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  float total = 0.f;
  if (b->form == LB_FORM_RK4) {
    cudaError_t e = lbi::batch_run_groups(b, nsteps, dt, correct_every, st, ms ? &total : nullptr);
    const cudaError_t es = cudaStreamSynchronize(st);
    if (e == cudaSuccess) e = es;
    if (e != cudaSuccess) return lbi::cuda_fail(e, "lb_batch_integrate");
    if (ms) *ms = total;
    return LB_OK;
  }
  for (int C : {16, 8, 4, 2, 1}) {
    std::vector<int> ids;
    for (int r = 0; r < b->count; ++r)
      if (b->cluster[r] == C) ids.push_back(r);
    float m = 0.f;
    cudaError_t e = lbi::batch_run_group(b, ids, C, nsteps, dt, correct_every, st, ms ? &m : nullptr);
    if (e != cudaSuccess) return lbi::cuda_fail(e, "lb_batch_integrate");
    total += m;
  }
  if (ms) *ms = total;
  cudaError_t e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) return lbi::cuda_fail(e, "lb_batch_integrate");
  return LB_OK;
}

// Autotuner: realizations are bucketed by N (bucket width `width`); for each
// bucket every cluster size of {1, 2, 4, 8, 16} that the device can place
// runs the bucket's realizations for probe_steps steps (timed with CUDA
// events), the states are restored, and the size with the shortest time is
// kept.  choice (optional, one per realization) receives the result.
int lb_batch_tune(lb_batch_t* b, int width, int probe_steps, double dt, void* stream, int* choice) {
  if (!b || width < 1 || probe_steps < 1) {
    lbi::set_error("lb_batch_tune: bad arguments");
    return LB_EINVAL;
  }
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  // save the states
  std::vector<double*> saved(b->count, nullptr);
  cudaError_t e = cudaSuccess;
  for (int r = 0; r < b->count && e == cudaSuccess; ++r) {
    if (!b->v[r]) {
      lbi::set_error("lb_batch_tune: realization %d has no state (lb_batch_set)", r);
      for (auto* p : saved) cudaFree(p);
      return LB_EINVAL;
    }
    e = cudaMalloc(&saved[r], 8 * (size_t)b->M[r]);
    if (e == cudaSuccess) e = cudaMemcpyAsync(saved[r], b->v[r], 8 * (size_t)b->M[r], cudaMemcpyDeviceToDevice, st);
  }
  int nmax = 0;
  for (int n : b->N) nmax = std::max(nmax, n);
  for (int lo = 2; lo <= nmax && e == cudaSuccess; lo += width) {
    std::vector<int> ids;
    for (int r = 0; r < b->count; ++r)
      if (b->N[r] >= lo && b->N[r] < lo + width) ids.push_back(r);
    if (ids.empty()) continue;
    float best = 3.4e38f;
    int bestC = 1;
    for (int C : {1, 2, 4, 8, 16}) {
      float ms = 0.f;
      cudaError_t ec = lbi::batch_run_group(b, ids, C, probe_steps, dt, 0, st, &ms);
      if (ec != cudaSuccess) {  // size not placeable with this shared memory: skip it
        cudaGetLastError();
        continue;
      }
      if (ms < best) {
        best = ms;
        bestC = C;
      }
      for (int r : ids)
        e = cudaMemcpyAsync(b->v[r], saved[r], 8 * (size_t)b->M[r], cudaMemcpyDeviceToDevice, st);
    }
    for (int r : ids) b->cluster[r] = bestC;
  }
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  for (auto* p : saved) cudaFree(p);
  if (e != cudaSuccess) return lbi::cuda_fail(e, "lb_batch_tune");
  if (choice)
    for (int r = 0; r < b->count; ++r) choice[r] = b->cluster[r];
  return LB_OK;
}

int lb_batch_system(const lb_batch_t* b, int r, const double** A64, const float** A32, const double** K,
                    int64_t* M) {
  if (!b || r < 0 || r >= b->count) {
    lbi::set_error("lb_batch_system: bad arguments");
    return LB_EINVAL;
  }
  if (A64) *A64 = b->A64[r];
  if (A32) *A32 = b->A32[r];
  if (K) *K = b->K[r];
  if (M) *M = b->M[r];
  return LB_OK;
}

int lb_batch_copy_system(const lb_batch_t* b, int r, double* A64, double* K, void* stream) {
  if (!b || r < 0 || r >= b->count) {
    lbi::set_error("lb_batch_copy_system: bad arguments");
    return LB_EINVAL;
  }
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const size_t M = (size_t)b->M[r];
  cudaError_t e = cudaSuccess;
  if (A64) e = cudaMemcpyAsync(A64, b->A64[r], 8 * M * M, cudaMemcpyDefault, st);
  if (K && e == cudaSuccess) e = cudaMemcpyAsync(K, b->K[r], 8 * M, cudaMemcpyDefault, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) return lbi::cuda_fail(e, "lb_batch_copy_system");
  return LB_OK;
}

int lb_batch_destroy(lb_batch_t* b) {
  if (!b) return LB_OK;
  lbi::batch_free(b);
  for (auto* x : b->basis) lb_basis_destroy(x);
  delete b;
  return LB_OK;
}

}  // extern "C"
