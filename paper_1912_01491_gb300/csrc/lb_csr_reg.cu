// lb_csr_reg.cu -- RK4 stages of sparse systems laid out by groups of 32 rows
// (Table 1 step 3.1 on CSR; the ladder and dimer models).
//
// The element s of a pair block couples to s + (a few offsets), the same for
// every s of one vertex a but for its ends, because the pair index is linear in
// the second vertex.  32 consecutive rows form a group, which a warp takes:
//   regular   all rows have L entries and column j of every row is the row plus
//             one offset delta_j.  Kept: the L offsets, and the values
//             transposed (entry j of the 32 rows together) in the place of the
//             group's values in the CSR arrays.
//   explicit  any other group: columns and values transposed, padded to its
//             longest row, with the rows' lengths.
//   long rows (more than 8 + 5/4 of the mean) belong to no group: a warp each,
//             from the CSR arrays.
// So values and columns are read in whole lines, a regular group reads 1/32 of
// its columns and no row pointers, and x is gathered in whole lines.  Entries of
// a row are summed in CSR order, those of a long row in FP64 by 32 lanes.
//
// What bounds it: the latency of HBM at N = 2000 (the ladder's FP32 stage moves
// 273 MB instead of 408 MB with columns and row pointers: 71 -> 54-57 us, 5.0
// TB/s; FP64 115 -> 107 us, where the FP64 pipe alone takes 82), latency and
// the FP64 pipe where the system fits L2 (dimer at N = 400: 35 -> 14 us).
// Measured slower at N = 2000: chunks of 256 rows staged two ahead by bulk
// copies (69 us FP32), warps that loop over groups with the next one's loads in
// flight (102 registers: 75 us), bulk prefetches into L2 (65 us).
//
// Consecutive stages use programmatic dependent launch: a stage's blocks start
// while the last ones of the stage before drain, and load what no stage writes
// before they wait for it.
#include <algorithm>
#include <type_traits>

#include "lb_internal.h"
#include "lb_rowsum.cuh"

namespace {

using lbi::CsrRegView;

constexpr int kSkip = 255;  // length of a row that belongs to no group

// A group's record: base (two words: the place of its values in the CSR arrays,
// explicit: of its slots), L entries, kind (0 regular, 1 explicit).
constexpr int kRec = 4;
__device__ __forceinline__ int64_t desc_base(const int4& d) { return ((int64_t)d.y << 32) | (uint32_t)d.x; }
__device__ __forceinline__ int4 desc_of(const int32_t* rec, int64_t g) {
  return __ldg(reinterpret_cast<const int4*>(rec + kRec * g));
}

// One warp per group.  FILL = false: count[0] += its padded slots and count[2]
// += 1 if explicit, count[1] += its long rows.  FILL = true: its descriptor,
// offsets, lengths and columns; slots, long rows and the list of explicit
// groups are taken from the same counters.
template <bool FILL>
__global__ void __launch_bounds__(256) k_reg_desc(int64_t M, int longer, const int64_t* __restrict__ rowptr,
                                                  const int32_t* __restrict__ col, unsigned long long* count,
                                                  int32_t* rec, int32_t* delta, uint8_t* len8, int32_t* ecol,
                                                  int32_t* longrow, int32_t* egroup) {
  const int64_t g = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (g * 32 >= M) return;  // whole warps leave together
  const int64_t s = g * 32 + lane;
  const bool in = s < M;
  const int64_t b = in ? rowptr[s] : 0, e = in ? rowptr[s + 1] : 0;
  const int64_t b0 = __shfl_sync(0xffffffffu, b, 0);
  const bool isl = e - b > longer;
  const int L = isl ? 0 : (int)(e - b), L0 = __shfl_sync(0xffffffffu, L, 0);
  bool reg = __all_sync(0xffffffffu, in && !isl && L == L0);
  for (int j = 0; reg && j < L0; ++j) {
    const int64_t d = (int64_t)col[b + j] - s;
    reg = __all_sync(0xffffffffu, d == __shfl_sync(0xffffffffu, d, 0));
    if (FILL && lane == 0) {
      delta[(b0 >> 5) + j] = (int32_t)d;
    }
  }
  const unsigned lm = __ballot_sync(0xffffffffu, isl);
  const int Lm = __reduce_max_sync(0xffffffffu, L);
  unsigned long long off = 0, lo = 0;
  if (lane == 0) {
    if (!reg) {
      off = atomicAdd(count, 32ull * Lm);
      const unsigned long long k = atomicAdd(count + 2, 1ull);
      if (FILL) egroup[k] = (int32_t)g;
    }
    if (lm) lo = atomicAdd(count + 1, (unsigned long long)__popc(lm));
  }
  if (!FILL) return;
  off = __shfl_sync(0xffffffffu, off, 0);
  lo = __shfl_sync(0xffffffffu, lo, 0);
  if (lane == 0) {
    const int64_t base = reg ? b0 : (int64_t)off;
    *reinterpret_cast<int4*>(rec + kRec * g) =
        make_int4((int)(base & 0xffffffff), (int)(base >> 32), reg ? L0 : Lm, reg ? 0 : 1);
  }
  if (isl) longrow[lo + __popc(lm & ((1u << lane) - 1u))] = (int32_t)s;
  if (in) len8[s] = (uint8_t)(isl ? kSkip : L);
  if (!reg)
    for (int j = 0; j < Lm; ++j) ecol[off + 32 * j + lane] = j < L ? col[b + j] : 0;
}

// Transposed values: regular groups into out (the CSR places), explicit ones into eout.
template <class T>
__global__ void __launch_bounds__(256) k_reg_values(int64_t M, const int32_t* __restrict__ rec,
                                                    const uint8_t* __restrict__ len8,
                                                    const int64_t* __restrict__ rowptr,
                                                    const double* __restrict__ val, T* __restrict__ out,
                                                    T* __restrict__ eout) {
  const int64_t g = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (g * 32 >= M) return;
  const int4 d = desc_of(rec, g);
  const int64_t base = desc_base(d), s = g * 32 + lane;
  if (d.w == 0) {
    for (int j = 0; j < d.z; ++j) out[base + 32 * j + lane] = (T)val[base + (int64_t)d.z * lane + j];
  } else {
    const int L = s < M && len8[s] != kSkip ? len8[s] : 0;
    const int64_t b = s < M ? rowptr[s] : 0;
    for (int j = 0; j < d.z; ++j) eout[base + 32 * j + lane] = j < L ? (T)val[b + j] : T(0);
  }
}

__device__ __forceinline__ double mad(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ float mad(float a, float b, float c) { return fmaf(a, b, c); }

// A group as its warp holds it: of a regular one its first PRE entries and the
// offsets of its first 32, which no stage writes.
template <class V, int PRE>
struct Group {
  int L;       // entries a row of a regular group, else -1
  int32_t dl;  // offset of entry `lane` of the current 32
  int64_t base;
  V pv[PRE];
  __device__ __forceinline__ void fetch(const CsrRegView& A, int j0, int lane) {
    const V* vp = static_cast<const V*>(A.val) + base + lane;
#pragma unroll
    for (int j = 0; j < PRE; ++j)
      if (j0 + j < L) pv[j] = __ldcs(vp + 32 * (j0 + j));
    if ((j0 & 31) == 0) dl = j0 + lane < L ? __ldg(A.delta + (base >> 5) + j0 + lane) : 0;
  }
  __device__ __forceinline__ void load(const CsrRegView& A, int64_t g, int lane) {
    const int4 d = desc_of(A.rec, g);
    base = desc_base(d);
    L = d.w == 0 ? d.z : -1;
    fetch(A, 0, lane);
  }
  // Sum over row s of a regular group of the matrix times x, in CSR order.
  __device__ __forceinline__ V sum(const CsrRegView& A, int64_t s, int lane, const V* x) {
    V t = V(0);
    for (int j0 = 0; j0 < L; j0 += PRE) {
      if (j0 > 0) fetch(A, j0, lane);
      V xv[PRE];
#pragma unroll
      for (int j = 0; j < PRE; ++j) {
        const int32_t o = __shfl_sync(0xffffffffu, dl, (j0 + j) & 31);
        if (j0 + j < L) xv[j] = __ldca(x + s + o);
      }
#pragma unroll
      for (int j = 0; j < PRE; ++j)
        if (j0 + j < L) t = mad(pv[j], xv[j], t);
    }
    return t;
  }
};

// The sum over row s (len entries) of an explicit group, in CSR order.
template <class V>
__device__ __forceinline__ V explicit_sum(const CsrRegView& A, const int4& d, int len, int lane, const V* x) {
  const V* vp = static_cast<const V*>(A.eval) + desc_base(d) + lane;
  const int32_t* cp = A.ecol + desc_base(d) + lane;
  V t = V(0);
  for (int j0 = 0; j0 < d.z; j0 += 4) {
    V a[4], xv[4];
    int32_t c[4];
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (j0 + j < len) {
        c[j] = __ldcs(cp + 32 * (j0 + j));
        a[j] = __ldcs(vp + 32 * (j0 + j));
      }
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (j0 + j < len) xv[j] = __ldca(x + c[j]);
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (j0 + j < len) t = mad(a[j], xv[j], t);
  }
  return t;
}

// Sum over row s from the CSR arrays by one warp, the same in every lane: FP64
// by 32 lanes and the xor tree; FP32 in CSR order.
template <class V>
__device__ __forceinline__ V long_row(const CsrRegView& A, int64_t s, int lane, const V* x) {
  const int64_t b = __ldg(A.rowptr + s), e = __ldg(A.rowptr + s + 1);
  V t = V(0);
  if constexpr (sizeof(V) == 8) {
#pragma unroll 4
    for (int64_t q = b + lane; q < e; q += 32) t = fma(__ldg(A.val64 + q), __ldca(x + __ldg(A.col + q)), t);
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
  } else {
    for (int64_t q0 = b; q0 < e; q0 += 32) {
      const int64_t q = q0 + lane;
      const V a = q < e ? (V)__ldg(A.val64 + q) : V(0), xv = q < e ? __ldca(x + __ldg(A.col + q)) : V(0);
      const int n = (int)min(e - q0, (int64_t)32);
      for (int j = 0; j < n; ++j)
        t = fmaf(__shfl_sync(0xffffffffu, a, j), __shfl_sync(0xffffffffu, xv, j), t);
    }
  }
  return t;
}

// The sum over row s of a matrix whose groups are whatever they are there (Q1
// of the driven form), by the thread of row s of a group.
template <class V>
__device__ __forceinline__ V any_row(const CsrRegView& A, int64_t s, int lane, bool valid, const V* x) {
  const int4 d = desc_of(A.rec, s >> 5);
  V t = V(0);
  if (d.w == 0) {
    const V* vp = static_cast<const V*>(A.val) + desc_base(d) + lane;
    const int32_t* dp = A.delta + (desc_base(d) >> 5);
#pragma unroll 2
    for (int j = 0; j < d.z; ++j) t = mad(__ldcs(vp + 32 * j), __ldca(x + s + __ldg(dp + j)), t);
  } else if (valid) {
    const int len = __ldg(A.len8 + s);
    if (len != kSkip) return explicit_sum<V>(A, d, len, lane, x);
    const int64_t b = __ldg(A.rowptr + s), e = __ldg(A.rowptr + s + 1);
#pragma unroll 4
    for (int64_t q = b; q < e; ++q) t = mad((V)__ldg(A.val64 + q), __ldca(x + __ldg(A.col + q)), t);
  }
  return t;
}

// The stage update of row s from the row sum y (in FP64).
template <int STAGE, class V>
__device__ __forceinline__ void stage_row(int64_t s, double y, double kf, double vs, double ac, double h, V* xn,
                                          double* acc, double* v) {
  const double k = y + kf;
  double nx;
  if (STAGE < 4) {
    __stcs(acc + s, STAGE == 1 ? k : fma(2.0, k, ac));
    nx = fma(h, k, vs);
  } else {
    nx = fma(h, ac + k, vs);
    __stcs(v + s, nx);
  }
  xn[s] = (V)nx;
}

__device__ __forceinline__ double as_double(double x) { return x; }
__device__ __forceinline__ double as_double(float x) { return lb::widen(x); }

// Threads of a block: how fast blocks turn over against how many must be
// launched.  Ladder at N = 2000, us a step of four stages with 64 / 128 / 256 /
// 512 threads: FP32 275 / 222 / 233 / 285, FP64 428 / 447 / 496 / 540.
constexpr int stage_threads(int prec, bool td) { return prec == LB_FP64 && !td ? 64 : 128; }
// Blocks per SM the registers must allow (48, 64 and 72 of them a thread).
constexpr int stage_blocks(int prec, bool td) { return td ? 7 : prec == LB_FP64 ? 16 : 10; }

// One RK4 stage (Keff: K + correction; h: dt / 2, dt / 2, dt, dt / 6): a warp per
// long row, then one per explicit group, then one per group of the matrix (the
// regular ones of them).  TD: the matrix is A + eps Q1.
template <int PREC, int STAGE, bool TD>
__global__ void __launch_bounds__(stage_threads(PREC, TD), stage_blocks(PREC, TD))
    k_stage_reg(int64_t M, CsrRegView A, CsrRegView Q1, double eps, const double* Keff, const void* xv, void* xnv,
                double* acc, double* v, double h) {
  using V = typename std::conditional<PREC == LB_FP64, double, float>::type;
  const int64_t w = (blockIdx.x * (int64_t)stage_threads(PREC, TD) + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  const V* x = static_cast<const V*>(xv);
  V* xn = static_cast<V*>(xnv);
  lb::grid_release();
  if (w < A.nlong) {
    const int64_t s = __ldg(A.longrow + w);
    lb::grid_wait();
    double y = as_double(long_row<V>(A, s, lane, x));
    if constexpr (TD) y = fma(eps, long_row<V>(Q1, s, lane, x), y);
    if (lane == 0) stage_row<STAGE>(s, y, Keff[s], v[s], STAGE > 1 ? acc[s] : 0.0, h, xn, acc, v);
    return;
  }
  if (w < A.nlong + A.nexp) {
    const int64_t s = (int64_t)__ldg(A.egroup + (w - A.nlong)) * 32 + lane;
    const bool valid = s < M;
    const int4 d = desc_of(A.rec, s >> 5);
    int len = valid ? (int)__ldg(A.len8 + s) : 0;
    const bool mine = valid && len != kSkip;
    if (!mine) len = 0;
    lb::grid_wait();
    double kf = 0.0, vs = 0.0, ac = 0.0;
    if (mine) {
      kf = __ldcs(Keff + s);
      vs = __ldcs(v + s);
      if (STAGE > 1) ac = __ldcs(acc + s);
    }
    double y = as_double(explicit_sum<V>(A, d, len, lane, x));
    if constexpr (TD) y = fma(eps, any_row<V>(Q1, s, lane, mine, x), y);
    if (mine) stage_row<STAGE>(s, y, kf, vs, ac, h, xn, acc, v);
    return;
  }
  const int64_t s = (w - A.nlong - A.nexp) * 32 + lane;
  if (s - lane >= M) return;  // whole warps leave together
  Group<V, 8> G;
  G.load(A, s >> 5, lane);
  lb::grid_wait();
  double kf = 0.0, vs = 0.0, ac = 0.0;
  if (s < M) {  // asked for before the group's kind is known; a regular group's rows all exist
    kf = __ldcs(Keff + s);
    vs = __ldcs(v + s);
    if (STAGE > 1) ac = __ldcs(acc + s);
  }
  if (G.L < 0) return;
  double y = as_double(G.sum(A, s, lane, x));
  if constexpr (TD) y = fma(eps, any_row<V>(Q1, s, lane, true, x), y);
  stage_row<STAGE>(s, y, kf, vs, ac, h, xn, acc, v);
}

// c = (A64 - A32) v;  Keff = K + c.  One thread per row.
__global__ void __launch_bounds__(256) k_correction_reg(int64_t M, CsrRegView A, const double* x, const double* K,
                                                        double* Keff) {
  const int64_t s = blockIdx.x * (int64_t)256 + threadIdx.x;
  if (s >= M) return;
  const int4 d = desc_of(A.rec, s >> 5);
  const int64_t b = A.rowptr[s], e = A.rowptr[s + 1];
  const int32_t* dl = A.delta + (desc_base(d) >> 5);
  const bool reg = d.w == 0;
  double t = 0.0;
#pragma unroll 4
  for (int64_t q = b; q < e; ++q) {
    const double a = A.val64[q];
    const int64_t c = reg ? s + __ldg(dl + (q - b)) : (int64_t)__ldg(A.col + q);
    t = fma(a - lb::widen((float)a), x[c], t);
  }
  Keff[s] = K[s] + t;
}

inline unsigned nblk(int64_t n) { return (unsigned)((n + 255) / 256); }

template <int PREC, bool TD>
cudaError_t launch(int stage, const cudaLaunchConfig_t& cfg, int64_t M, const CsrRegView& A, const CsrRegView& Q1,
                   double eps, const double* Keff, const void* x, void* xn, double* acc, double* v, double h) {
  switch (stage) {
    case 1: return cudaLaunchKernelEx(&cfg, k_stage_reg<PREC, 1, TD>, M, A, Q1, eps, Keff, x, xn, acc, v, h);
    case 2: return cudaLaunchKernelEx(&cfg, k_stage_reg<PREC, 2, TD>, M, A, Q1, eps, Keff, x, xn, acc, v, h);
    case 3: return cudaLaunchKernelEx(&cfg, k_stage_reg<PREC, 3, TD>, M, A, Q1, eps, Keff, x, xn, acc, v, h);
    default: return cudaLaunchKernelEx(&cfg, k_stage_reg<PREC, 4, TD>, M, A, Q1, eps, Keff, x, xn, acc, v, h);
  }
}

}  // namespace

namespace lbi {

void csr_plan_free(CsrPlan* p) {
  cudaFree(p->rec);  // with the arrays behind it
  for (int q = 0; q < 2; ++q) cudaFree(p->val[q]);
  *p = CsrPlan{};
}

cudaError_t csr_plan(CsrPlan* p, int64_t M, int64_t nnz, const int64_t* rowptr, const int32_t* col, const double* val,
                     int precision, cudaStream_t st, CsrRegView* view, bool* usable) {
  *usable = false;
  if (p->state < 0) return cudaSuccess;
  cudaError_t e = cudaSuccess;
  const int64_t groups = (M + 31) / 32;
  const unsigned grid = nblk(groups * 32);
  auto pad = [](size_t n) { return (n + 255) & ~size_t(255); };
  // without memory for it the caller takes the kernels that need no layout
  auto refused = [&]() {
    if (e != cudaErrorMemoryAllocation) return e;
    cudaGetLastError();
    return cudaSuccess;
  };
  if (p->state == 0) {
    unsigned long long *cnt = nullptr, hc[3] = {0, 0, 0};
    const int longer = (int)std::min<int64_t>(200, 8 + 5 * nnz / (4 * M));
    cudaMemPool_t pool = nullptr;
    if ((e = scratch_pool(&pool)) != cudaSuccess) return e;
    if ((e = cudaMallocFromPoolAsync((void**)&cnt, sizeof(hc), pool, st)) != cudaSuccess) return refused();
    e = cudaMemsetAsync(cnt, 0, sizeof(hc), st);
    if (e == cudaSuccess) {
      k_reg_desc<false><<<grid, 256, 0, st>>>(M, longer, rowptr, col, cnt, nullptr, nullptr, nullptr, nullptr, nullptr,
                                              nullptr);
      note_launch(1);
      e = cudaMemcpyAsync(hc, cnt, sizeof(hc), cudaMemcpyDeviceToHost, st);
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    // padding or long rows without end: the CSR kernels
    const bool fits = 2 * hc[0] <= 3ull * (unsigned long long)nnz + 4096 && 8 * (int64_t)hc[1] <= M;
    if (e == cudaSuccess && fits) {
      // one allocation: each takes some ten microseconds whatever its size
      const size_t rec = pad(sizeof(int32_t) * kRec * (size_t)groups), delta = pad(sizeof(int32_t) * (size_t)(nnz / 32 + 1)),
                   len8 = pad((size_t)M), ecol = pad(sizeof(int32_t) * (size_t)(hc[0] + 1)),
                   longrow = pad(sizeof(int32_t) * (size_t)(hc[1] + 1)), egroup = sizeof(int32_t) * (size_t)(hc[2] + 1);
      char* m = nullptr;
      e = cudaMalloc((void**)&m, rec + delta + len8 + ecol + longrow + egroup);
      if (e == cudaSuccess) {
        p->rec = reinterpret_cast<int32_t*>(m);
        p->delta = reinterpret_cast<int32_t*>(m += rec);
        p->len8 = reinterpret_cast<uint8_t*>(m += delta);
        p->ecol = reinterpret_cast<int32_t*>(m += len8);
        p->longrow = reinterpret_cast<int32_t*>(m += ecol);
        p->egroup = reinterpret_cast<int32_t*>(m += longrow);
        e = cudaMemsetAsync(cnt, 0, sizeof(hc), st);
      }
      if (e == cudaSuccess) {
        k_reg_desc<true><<<grid, 256, 0, st>>>(M, longer, rowptr, col, cnt, p->rec, p->delta, p->len8, p->ecol,
                                               p->longrow, p->egroup);
        note_launch(1);
        e = cudaStreamSynchronize(st);
      }
    }
    cudaFreeAsync(cnt, st);
    if (e != cudaSuccess || !fits) {
      csr_plan_free(p);
      if (e == cudaSuccess) p->state = -1;
      return refused();
    }
    p->state = 1;
    p->slots = (int64_t)hc[0];
    p->nlong = (int64_t)hc[1];
    p->nexp = (int64_t)hc[2];
  }
  const int q = precision == LB_FP64 ? 0 : 1;
  if (!p->val[q]) {
    const size_t esz = q == 0 ? 8 : 4, first = pad(esz * (size_t)(nnz + 8));
    char* a = nullptr;
    e = cudaMalloc((void**)&a, first + esz * (size_t)(p->slots + 1));
    if (e == cudaSuccess) {
      if (q == 0)
        k_reg_values<double><<<grid, 256, 0, st>>>(M, p->rec, p->len8, rowptr, val, (double*)a, (double*)(a + first));
      else
        k_reg_values<float><<<grid, 256, 0, st>>>(M, p->rec, p->len8, rowptr, val, (float*)a, (float*)(a + first));
      note_launch(1);
      e = cudaStreamSynchronize(st);  // other streams use it from here on
    }
    if (e != cudaSuccess) {
      cudaFree(a);
      return refused();
    }
    p->val[q] = a;
    p->eval[q] = a + first;
  }
  *view = CsrRegView{p->rec, p->delta, p->len8, p->ecol, p->longrow, p->egroup, p->nlong, p->nexp,
                     p->val[q], p->eval[q], nnz,
                     rowptr, col, val};
  *usable = true;
  return cudaSuccess;
}

cudaError_t csr_reg_stage(int precision, int stage, int64_t M, const CsrRegView& A, const CsrRegView* Q1, double eps,
                          const double* Keff, const void* x, void* xn, double* acc, double* v, double h,
                          cudaStream_t st) {
  cudaLaunchConfig_t cfg{};
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  const int threads = stage_threads(precision, Q1 != nullptr);
  cfg.gridDim = dim3((unsigned)(((A.nlong + A.nexp + (M + 31) / 32) * 32 + threads - 1) / threads), 1, 1);
  cfg.blockDim = dim3((unsigned)threads, 1, 1);
  cfg.stream = st;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  note_launch(1);
  if (Q1) return launch<LB_FP64, true>(stage, cfg, M, A, *Q1, eps, Keff, x, xn, acc, v, h);
  if (precision == LB_FP64) return launch<LB_FP64, false>(stage, cfg, M, A, A, 0.0, Keff, x, xn, acc, v, h);
  return launch<LB_FP32, false>(stage, cfg, M, A, A, 0.0, Keff, x, xn, acc, v, h);
}

cudaError_t csr_reg_correction(int64_t M, const CsrRegView& A, const double* v, const double* K, double* Keff,
                               cudaStream_t st) {
  k_correction_reg<<<nblk(M), 256, 0, st>>>(M, A, v, K, Keff);
  note_launch(1);
  return cudaGetLastError();
}

}  // namespace lbi
