// lb_csr_bulk.cu -- rows of a sparse A = Q + R in closed form (Eqs. (07), (09)
// with a = sum_p gamma_p l_p l_p^dagger, sparse L_p = sum_j l_pj F_j and H).
//
// For far-apart vertices c, d the rows S_cd and J_cd need no sum over the
// structure constants.  Applied to the matrix unit E_ab the generator has the
// coefficient
//   t_(cd),(ab) = sum_p gamma_p (L_p)_ca conj((L_p)_db) + G_ca [d = b] +
//                 [c = a] conj(G_db),   G = -i H - 1/2 sum_p gamma_p L_p^+ L_p
// of E_cd, and with the units written in S_ab and J_ab
//   A(S_cd, S_ab) = A(J_cd, J_ab) = Re t,  A(S_cd, J_ab) = -A(J_cd, S_ab) = Im t
// for a < b; for a > b (column pair (b, a)) the J columns change sign.  This is
// the whole row when no diagonal element takes part in the join of Eq. (09),
// i.e. when d is more than two steps from c on the graph of the edges of the
// l_p, not a neighbour on that of H, and out of reach of the rows of G: for the
// banded models all rows but O(N).  The join adds 143 terms to each row of the
// ladder at N = 2000, most of which cancel; here a row costs 9 candidates.
//
// An entry of the join is kept when |value| > 1e-12 sum |terms|.  The sums of
// magnitudes are bounded for the whole matrix by one number, smax (each term is
// a W term times a U term; see k_bulk_limit): an entry above 1e-12 smax is kept
// by both, one that is zero up to the rounding of t's own terms is kept by
// neither, and a row with an entry in between goes the general way.
//
// What bounds it: the FP64 and the integer pipe (47% and 42% busy) and the loads
// from the vertices' lists between (k_bulk_rows runs once over the pairs to count
// and once to fill, 1.0 and 0.65 ms at N = 2000, 1.4 and 1.25 ms with complex
// products and FP64 comparisons throughout).  Whole assembly, with the scratch
// kept between calls and the join's passes free of FP64 work for entries that
// are only counted or dropped: ladder N = 2000 40.9 -> 6.5 ms, N = 1000 12.0 ->
// 2.3 ms; dimer N = 400 6.2 -> 1.2 ms.
#include <algorithm>

#include "lb_internal.h"
#include "lb_rowsum.cuh"

namespace {

using namespace lb;
using lbi::CsrBulk;

constexpr int kMaxDeg = 16;   // candidates per vertex
constexpr int kMaxNear = 24;  // neighbours on the l graph

// The pair elements of the channels: L_p (dense N x N), per edge and channel
// the sum of |l|, and the number of list entries on the edge (both orders).
__global__ void k_bulk_scatter(BasisView B, int nP, const int64_t* lp_ptr, const int64_t* lp_idx,
                               const double2* lp_val, int64_t nu, CsrBulk b) {
  const int64_t u = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (u >= nu) return;
  const int64_t k = lp_idx[u];
  if (k >= 2 * B.P) return;
  int p = 0;
  while (p + 1 < nP && lp_ptr[p + 1] <= u) ++p;
  const Elem e = decode(B, k);
  const double2 l = lp_val[u];
  const int N = B.N;
  const int64_t nn = (int64_t)N * N, ab = (int64_t)e.a * N + e.b, ba = (int64_t)e.b * N + e.a;
  // S: 1/sqrt2 both ways; J: -i/sqrt2 at (a, b), +i/sqrt2 at (b, a)
  double2 x = make_double2(kInvSqrt2 * l.x, kInvSqrt2 * l.y), y = x;
  if (e.kind == kJ) {
    x = make_double2(kInvSqrt2 * l.y, -kInvSqrt2 * l.x);
    y = make_double2(-x.x, -x.y);
  }
  double2* L = b.L + p * nn;
  atomicAdd(&L[ab].x, x.x);
  atomicAdd(&L[ab].y, x.y);
  atomicAdd(&L[ba].x, y.x);
  atomicAdd(&L[ba].y, y.y);
  const double m = sqrt(l.x * l.x + l.y * l.y);
  atomicAdd(b.mag + p * nn + ab, m);
  atomicAdd(b.mag + p * nn + ba, m);
  atomicAdd(b.cnt + ab, 1);
  atomicAdd(b.cnt + ba, 1);
}

// Components that are rounding residue (the S and J parts of an edge cancel)
// become zero.
__global__ void k_bulk_clean(int64_t n, double2* L, const double* mag) {
  const int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (q >= n) return;
  const double m = mag[q];
  if (m == 0.0) return;
  double2 x = L[q];
  if (fabs(x.x) <= 1e-15 * m) x.x = 0.0;
  if (fabs(x.y) <= 1e-15 * m) x.y = 0.0;
  L[q] = x;
}

// Sum over the block's threads; every thread gets it.
__device__ double block_sum(double x, double* sh) {
  for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = x;
  __syncthreads();
  double t = 0.0;
  for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += sh[w];
  return t;
}
__device__ double block_max(double x, double* sh) {
  for (int o = 16; o > 0; o >>= 1) x = fmax(x, __shfl_xor_sync(0xffffffffu, x, o));
  __syncthreads();
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = x;
  __syncthreads();
  double t = 0.0;
  for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t = fmax(t, sh[w]);
  return t;
}

// Diagonals, block p < nP: channel p, block nP: H.
//   x_kk = sum_{nu > k} x_nu c_nu + x_k lc_k   (x_0 = 0)
// Each thread sums a contiguous run of nu; the sums of the runs behind it come
// from the block.  gd[p] = 4 sum |x_nu| c_nu + 2 max |x_nu lc_nu|: above every
// diagonal sum of an edge, summed by magnitude.  npd[p N + k]: the nonzero ones
// of D_1 .. D_k.
__global__ void __launch_bounds__(kSuffixThreads) k_bulk_diag(BasisView B, int nP, const double2* dl, const int* hasD,
                                                              const double* h, CsrBulk b) {
  __shared__ double sh[kSuffixThreads / 32];
  const int p = blockIdx.x, N = B.N, t = threadIdx.x;
  const bool isH = p == nP;
  const int64_t nn = (int64_t)N * N;
  auto at = [&](int nu) {  // component of D_nu
    if (nu < 1) return make_double2(0.0, 0.0);
    if (isH) return make_double2(h ? h[2 * B.P - 1 + nu] : 0.0, 0.0);
    return hasD[p] ? dl[(int64_t)p * N + nu] : make_double2(0.0, 0.0);
  };
  const int per = (N + kSuffixThreads - 1) / kSuffixThreads, k0 = min(t * per, N), k1 = min(k0 + per, N);
  double sr = 0.0, si = 0.0, sm = 0.0, mlc = 0.0;
  int n = 0;
  for (int nu = max(k0, 1); nu < k1; ++nu) {
    const double2 x = at(nu);
    const double c = ld_c(B, nu), m = sqrt(x.x * x.x + x.y * x.y);
    sr += x.x * c;
    si += x.y * c;
    sm += m * c;
    mlc = fmax(mlc, m * fabs(ld_lc(B, nu)));
    n += x.x != 0.0 || x.y != 0.0;
  }
  const double gsum = block_sum(sm, sh), glc = block_max(mlc, sh);
  double ar = block_suffix(sr, sh), ai = block_suffix(si, sh);  // sum over nu > the element at hand
  const int behind = block_suffix(n, reinterpret_cast<int*>(sh));
  __shared__ int total;
  if (t == 0) total = n + behind;
  __syncthreads();
  int upto = total - behind;  // nonzero ones of D_1 .. D_k
  for (int k = k1 - 1; k >= k0; --k) {
    const double2 x = at(k);
    const double lc = k > 0 ? ld_lc(B, k) : 0.0, c = k > 0 ? ld_c(B, k) : 0.0;
    const double2 d = make_double2(ar + x.x * lc, ai + x.y * lc);
    if (isH) b.hdiag[k] = d.x;
    else b.L[p * nn + (int64_t)k * N + k] = d;
    ar += x.x * c;
    ai += x.y * c;
    b.npd[(int64_t)p * N + k] = upto;
    upto -= x.x != 0.0 || x.y != 0.0;
  }
  if (t == 0) b.gd[p] = 4.0 * gsum + 2.0 * glc;
}

// smax.  A W term of a row is l_k f, |f| <= 1/sqrt2, or a diagonal sum of an
// edge, a U term l_j z or a diagonal sum likewise, each at most once per (l, n);
// with mx the largest sum of |l| over the edges of a vertex
//   sum |terms| <= 1/2 gamma (2 mx / sqrt2 + gd) max(mx / sqrt2, gd)
// per channel, and a Q term is at most max |h| / sqrt2 or the diagonal sum of h.
// A negative gamma gives the join a negative bound, a value that is not finite
// none: those matrices go the general way (smax infinite or NaN).
__global__ void k_bulk_limit(int nP, CsrBulk b) {
  double s = kInvSqrt2 * b.mx[nP] + b.gd[nP];
  for (int p = 0; p < nP; ++p) {
    const double m = kInvSqrt2 * b.mx[p], g = b.gd[p];
    s += 0.5 * b.gamma[p] * (2.0 * m + g) * fmax(m, g);
    if (!(b.gamma[p] >= 0.0)) s = 1.0 / 0.0;
  }
  *b.smax = s;
}

// Positive doubles order as their bits.
__device__ __forceinline__ void max_double(double* at, double x) {
  atomicMax(reinterpret_cast<unsigned long long*>(at), (unsigned long long)__double_as_longlong(x));
}

// The zeros of H: H_cw for w != c from the pair coefficients.
__device__ __forceinline__ double2 h_entry(const BasisView& B, const double* h, int c, int w) {
  const int64_t e = pair_index_any(B.N, c, w);
  const double s = kInvSqrt2 * h[e], j = kInvSqrt2 * h[B.P + e];
  return make_double2(s, c < w ? -j : j);
}

// One warp per vertex c: its neighbours on the l graph with their counts, the
// rows that go the general way for its sake (near[c][w] = 1), and its
// candidates a in ascending order with G_ca, (L_p)_ca and gamma_p (L_p)_ca.
__global__ void __launch_bounds__(128) k_bulk_vertex(BasisView B, int nP, const double* h, const double* gamma,
                                                     CsrBulk b) {
  constexpr int kList = 64;
  __shared__ int s_n1[4][kMaxNear], s_k[4][kMaxNear], s_col[4][kList];
  __shared__ double2 s_g[4][kList];
  __shared__ double s_m[4][kList];
  const int N = B.N, lane = threadIdx.x & 31, wq = threadIdx.x >> 5;
  const int c = blockIdx.x * 4 + wq;
  if (c >= N) return;
  int *n1 = s_n1[wq], *kl = s_k[wq], *col = s_col[wq];
  double2* g = s_g[wq];
  double* gm = s_m[wq];
  const int64_t nn = (int64_t)N * N;
  uint8_t* near = b.near + (int64_t)c * N;
  int nn1 = 0, nk = 0, ncol = 1, nh = 0;
  double mh = 0.0;
  bool over = false;
  if (lane == 0) {
    col[0] = c;
    const double hd = h ? b.hdiag[c] : 0.0;
    g[0] = make_double2(0.0, -hd);
    gm[0] = fabs(hd);
    near[c] = 1;
  }
  __syncwarp();
  auto nz = [&](double2 x) { return x.x != 0.0 || x.y != 0.0; };
  for (int w0 = 0; w0 < N; w0 += 32) {
    const int w = w0 + lane;
    bool isn = false, isk = false, row = false, ish = false;
    double2 hv = make_double2(0.0, 0.0);
    if (w < N && w != c) {
      isn = b.cnt[(int64_t)c * N + w] > 0;
      if (isn)
        for (int p = 0; p < nP; ++p) {
          row |= nz(b.L[p * nn + (int64_t)c * N + w]);
          isk |= nz(b.L[p * nn + (int64_t)w * N + c]);
        }
      if (h) {
        hv = h_entry(B, h, c, w);
        ish = nz(hv);
        if (ish) near[w] = 1;
        const int64_t e = pair_index_any(N, c, w);
        nh += (h[e] != 0.0) + (h[B.P + e] != 0.0);
        mh = fmax(mh, fmax(fabs(h[e]), fabs(h[B.P + e])));
      }
      if (isn) near[w] = 1;
    } else if (w == c) {
      for (int p = 0; p < nP; ++p) isk |= nz(b.L[p * nn + (int64_t)c * N + c]);
    }
    unsigned m = __ballot_sync(0xffffffffu, isn);
    while (m) {
      const int q = __ffs(m) - 1;
      m &= m - 1;
      if (nn1 < kMaxNear) {
        if (lane == 0) n1[nn1] = w0 + q;
        ++nn1;
      } else {
        over = true;
      }
    }
    m = __ballot_sync(0xffffffffu, isk);
    while (m) {
      const int q = __ffs(m) - 1;
      m &= m - 1;
      if (nk < kMaxNear) {
        if (lane == 0) kl[nk] = w0 + q;
        ++nk;
      } else {
        over = true;
      }
    }
    m = __ballot_sync(0xffffffffu, row || ish);
    while (m) {
      const int q = __ffs(m) - 1;
      m &= m - 1;
      const double hr = __shfl_sync(0xffffffffu, hv.x, q), hi = __shfl_sync(0xffffffffu, hv.y, q);
      if (ncol < kList) {
        if (lane == 0) {
          col[ncol] = w0 + q;
          g[ncol] = make_double2(hi, -hr);  // -i H
          gm[ncol] = fabs(hr) + fabs(hi);
        }
        ++ncol;
      } else {
        over = true;
      }
    }
  }
  for (int o = 16; o > 0; o >>= 1) {
    nh += __shfl_xor_sync(0xffffffffu, nh, o);
    mh = fmax(mh, __shfl_xor_sync(0xffffffffu, mh, o));
  }
  __syncwarp();
  if (lane == 0) {
    max_double(b.mx + nP, mh);
    for (int p = 0; p < nP && !over; ++p) {
      double m = 0.0;
      for (int i = 0; i < nn1; ++i) m += b.mag[p * nn + (int64_t)c * N + n1[i]];
      max_double(b.mx + p, m);
    }
    if (over) max_double(b.mx + nP, 1.0 / 0.0);  // a list cut short: no bound
  }
  __syncwarp();
  // two steps on the l graph
  for (int i = 0; i < nn1; ++i)
    for (int w = lane; w < N; w += 32)
      if (b.cnt[(int64_t)n1[i] * N + w] > 0) near[w] = 1;
  // G_ca -= 1/2 gamma_p conj((L_p)_kc) (L_p)_ka
  for (int i = 0; i < nk && !over; ++i) {
    const int k = kl[i];
    for (int w0 = 0; w0 < N; w0 += 32) {
      const int w = w0 + lane;
      bool any = false;
      if (w < N)
        for (int p = 0; p < nP; ++p) any |= nz(b.L[p * nn + (int64_t)k * N + w]);
      unsigned m = __ballot_sync(0xffffffffu, any);
      while (m) {
        const int a = w0 + __ffs(m) - 1;
        m &= m - 1;
        int f = -1;
        for (int q0 = 0; q0 < ncol; q0 += 32) {
          const unsigned hit = __ballot_sync(0xffffffffu, q0 + lane < ncol && col[q0 + lane] == a);
          if (hit) f = q0 + __ffs(hit) - 1;
        }
        if (f < 0) {
          if (ncol == kList) {
            over = true;
            break;
          }
          f = ncol++;
          if (lane == 0) {
            col[f] = a;
            g[f] = make_double2(0.0, 0.0);
            gm[f] = 0.0;
          }
          __syncwarp();
        }
        if (lane == 0)
          for (int p = 0; p < nP; ++p) {
            const double2 x = b.L[p * nn + (int64_t)k * N + c], y = b.L[p * nn + (int64_t)k * N + a];
            const double q = -0.5 * gamma[p];
            const double rr = x.x * y.x, ii = x.y * y.y, ri = x.x * y.y, ir = x.y * y.x;
            g[f].x += q * (rr + ii);
            g[f].y += q * (ri - ir);
            gm[f] += fabs(q) * (fabs(rr) + fabs(ii) + fabs(ri) + fabs(ir));
          }
        __syncwarp();
      }
      if (over) break;
    }
  }
  __syncwarp();
  // drop residues, keep what is left in ascending order
  int kept = 0;
  for (int q0 = 0; q0 < ncol && !over; q0 += 32) {
    const int q = q0 + lane;
    bool keep = false;
    if (q < ncol) {
      const double tiny = 1e-15 * gm[q];
      if (fabs(g[q].x) <= tiny) g[q].x = 0.0;
      if (fabs(g[q].y) <= tiny) g[q].y = 0.0;
      keep = nz(g[q]) || q == 0;
      for (int p = 0; p < nP && !keep; ++p) keep = nz(b.L[p * nn + (int64_t)c * N + col[q]]);
    }
    __syncwarp();
    if (q < ncol && !keep) col[q] = N;  // sorts behind the kept ones
    kept += __popc(__ballot_sync(0xffffffffu, keep));
  }
  __syncwarp();
  if (kept > kMaxDeg) over = true;
  if (!over) {
    for (int q = lane; q < ncol; q += 32) {
      const int a = col[q];
      if (a == N) continue;
      int rank = 0;
      for (int r = 0; r < ncol; ++r) rank += col[r] < a;
      const int at = c * kMaxDeg + rank;
      near[a] = 1;
      b.ucol[at] = a;
      b.G[at] = g[q];
      for (int p = 0; p < nP; ++p) {
        const double2 x = b.L[p * nn + (int64_t)c * N + a];
        b.Lu[((int64_t)p * N + c) * kMaxDeg + rank] = x;
        if (x.y != 0.0) *b.cplx = 1;
      }
    }
    for (int i = lane; i < nn1; i += 32) {
      b.nbr[c * kMaxNear + i] = n1[i];
      b.nbc[c * kMaxNear + i] = b.cnt[(int64_t)c * N + n1[i]];
    }
  }
  if (lane == 0) {
    b.deg[c] = over ? -1 : kept;
    b.nn1[c] = nn1;
    b.nh[c] = nh;
    int d = 0;
    for (int i = 0; i < nn1; ++i) d += b.cnt[(int64_t)c * N + n1[i]];
    b.d1[c] = d;
    if (!over) atomicMax(b.maxdeg, kept);
  }
}

// exponent of |x|, 0 for zero
__device__ __forceinline__ int expo(double x) { return (__double2hiint(x) >> 20) & 0x7ff; }
// |x| bit for bit: orders as the value does, NaN above all; -x.  Integer work: a warp instruction of the FP64 pipe
// takes some 60 cycles whatever it computes.
__device__ __forceinline__ unsigned long long mag_bits(double x) {
  return (unsigned long long)__double_as_longlong(x) & 0x7fffffffffffffffull;
}
__device__ __forceinline__ double minus(double x, bool neg) {
  return __longlong_as_double(__double_as_longlong(x) ^ (neg ? (long long)0x8000000000000000ull : 0ll));
}

// The rows of pair (c, d) by GW lanes, candidate e = i deg(d) + j: a = ucol[c][i],
// b = ucol[d][j].  FILL = false: rowc of both rows, slow[row] = 1 for the rows of
// the general way, the number of join terms of the others; FILL = true: the
// entries at rowptr.  Real l_p (the usual ladder) take two products of a term's
// six; comparisons and signs are integer work.
template <bool FILL, int GW>
__global__ void __launch_bounds__(256) k_bulk_rows(BasisView B, int nP, CsrBulk b, unsigned long long* rowc,
                                                   unsigned long long* terms, const int64_t* rowptr, int32_t* col,
                                                   double* val) {
  const int N = B.N, lane = threadIdx.x & 31, sub = lane & (GW - 1), g0 = lane & ~(GW - 1);
  const unsigned gmask = (GW == 32 ? 0xffffffffu : ((1u << GW) - 1u)) << g0;
  // candidate counts of at most 4 x 4 take 16 lanes a pair
  if ((*b.maxdeg <= 4) != (GW == 16)) return;
  const unsigned long long lim = mag_bits(1e-12 * *b.smax);
  // no bound: every row goes the general way, those whose entries all cancel too (under a negative bound the join
  // keeps even zeros)
  const bool bounded = lim < 0x7ff0000000000000ull, cplx = *b.cplx != 0;
  unsigned long long nterm = 0;
  for (int64_t w0 = (blockIdx.x * (int64_t)256 + (threadIdx.x & ~31)) / GW; w0 < B.P;
       w0 += gridDim.x * (int64_t)256 / GW) {
  const int64_t pr = w0 + lane / GW;
  const bool in = pr < B.P;
  int c = 0, d = 1;
  if (in) {
    const Elem e = decode(B, pr);
    c = e.a;
    d = e.b;
  }
  const int dc = b.deg[c], dd = b.deg[d];
  bool bulk = in && (FILL ? !b.slow[pr] : bounded && !b.near[(int64_t)c * N + d] && !b.near[(int64_t)d * N + c] &&
                                              dc > 0 && dd > 0 && dc * dd <= GW);
  double re = 0.0, im = 0.0;
  bool kre = false, kim = false, unsure = false, flip = false;
  int32_t pi = 0x7fffffff;
  if (bulk && sub < dc * dd) {
    const int i = sub / dd, j = sub - i * dd;
    const int ac = b.ucol[c * kMaxDeg + i], bc = b.ucol[d * kMaxDeg + j];
    int mr = 0, mi = 0;  // largest exponent of the terms
    for (int p = 0; p < nP; ++p) {
      const double2 x = b.Lu[((int64_t)p * N + c) * kMaxDeg + i], y = b.Lu[((int64_t)p * N + d) * kMaxDeg + j];
      // explicit rounding: the count and the fill have to see the same bits
      const double gx = __dmul_rn(b.gamma[p], x.x), t0 = __dmul_rn(gx, y.x);
      mr = max(mr, expo(t0));
      if (!cplx) {
        re = p ? __dadd_rn(re, t0) : t0;
        continue;
      }
      const double gy = __dmul_rn(b.gamma[p], x.y);
      const double t1 = __dmul_rn(gy, y.y), t2 = __dmul_rn(gy, y.x), t3 = __dmul_rn(gx, y.y);
      mr = max(mr, expo(t1));
      mi = max(mi, max(expo(t2), expo(t3)));
      re = __dadd_rn(re, __dadd_rn(t0, t1));
      im = __dadd_rn(im, __dadd_rn(t2, -t3));
    }
    if (bc == d) {
      const double2 x = b.G[c * kMaxDeg + i];
      mr = max(mr, expo(x.x));
      mi = max(mi, expo(x.y));
      re = __dadd_rn(re, x.x);
      im = __dadd_rn(im, x.y);
    }
    if (ac == c) {
      const double2 x = b.G[d * kMaxDeg + j];
      mr = max(mr, expo(x.x));
      mi = max(mi, expo(x.y));
      re = __dadd_rn(re, x.x);
      im = __dadd_rn(im, -x.y);
    }
    // zero up to the rounding of the terms; kept; or not certain
    const unsigned long long ur = mag_bits(re), ui = mag_bits(im), inf = 0x7ff0000000000000ull;
    kre = expo(re) + 49 > mr && ur != 0;
    kim = expo(im) + 49 > mi && ui != 0;
    unsure = (kre && (ur <= lim || ur > inf)) || (kim && (ui <= lim || ui > inf));
    flip = ac > bc;
    pi = (int32_t)pair_index_any(N, ac, bc);
  }
  if (!FILL) {
    const bool bad = (__ballot_sync(0xffffffffu, unsure) & gmask) != 0;
    if (bad) bulk = false;
  }
  const unsigned br = __ballot_sync(0xffffffffu, bulk && kre) & gmask;
  const unsigned bi = __ballot_sync(0xffffffffu, bulk && kim) & gmask;
  const int nre = __popc(br), nim = __popc(bi);
  if (!FILL) {
    if (in && sub == 0) {
      b.slow[pr] = b.slow[B.P + pr] = bulk ? 0 : 1;
      rowc[pr] = rowc[B.P + pr] = bulk ? (unsigned long long)(nre + nim) : 0ull;
      if (bulk) {
        // join terms of a row: over its W terms the U terms of their rows, and Q
        auto diag = [&](int p, int x, int y) {  // a nonzero D_nu with max(x, 1) <= nu <= y
          const int* n = b.npd + (int64_t)p * N;
          return n[y] - (x > 1 ? n[x - 1] : 0) > 0;
        };
        auto utot = [&](int u, int w) {
          const int x = min(u, w), y = max(u, w);
          long long t = 2ll * (b.d1[u] + b.d1[w]);
          for (int p = 0; p < nP; ++p) {
            t += diag(p, x, y);
            // H: any nu >= max(x, 1), but for nu = y = 1 (coefficient zero)
            const int* n = b.npd + (int64_t)p * N;
            t += n[N - 1] - (x > 1 ? n[x - 1] : 0) - (y == 1 ? n[1] : 0) > 0;
          }
          return t;
        };
        long long t = 0;
        for (int i = 0; i < b.nn1[c]; ++i) t += b.nbc[c * kMaxNear + i] * utot(b.nbr[c * kMaxNear + i], d);
        for (int i = 0; i < b.nn1[d]; ++i) t += b.nbc[d * kMaxNear + i] * utot(c, b.nbr[d * kMaxNear + i]);
        for (int p = 0; p < nP; ++p)
          if (diag(p, c, d)) t += utot(c, d);
        t += b.nh[c] + b.nh[d] + (diag(nP, c, d) ? 1 : 0);
        nterm += 2ull * (unsigned long long)t;
      }
    }
    continue;
  }
  // ranks among the kept columns of each kind: lanes are in column order unless a pair is flipped
  int rr = __popc(br & ((1u << lane) - 1u)), ri = __popc(bi & ((1u << lane) - 1u));
  if (__any_sync(0xffffffffu, bulk && flip && (kre || kim))) {
    rr = ri = 0;
    for (int q = 0; q < GW; ++q) {
      const int32_t o = __shfl_sync(0xffffffffu, pi, g0 + q);
      rr += ((br >> (g0 + q)) & 1u) && o < pi;
      ri += ((bi >> (g0 + q)) & 1u) && o < pi;
    }
  }
  if (!bulk) continue;
  const int64_t rs = rowptr[pr], rj = rowptr[B.P + pr];
  const int32_t P = (int32_t)B.P;
  if (kre) {  // A(S, S) and A(J, J)
    col[rs + rr] = pi;
    val[rs + rr] = re;
    col[rj + nim + rr] = P + pi;
    val[rj + nim + rr] = minus(re, flip);
  }
  if (kim) {  // A(S, J) and A(J, S)
    col[rs + nre + ri] = P + pi;
    val[rs + nre + ri] = minus(im, flip);
    col[rj + ri] = pi;
    val[rj + ri] = minus(im, true);
  }
  }
  if (!FILL) {
    for (int o = 16; o > 0; o >>= 1) nterm += __shfl_xor_sync(0xffffffffu, nterm, o);
    if (lane == 0 && nterm) atomicAdd(terms, nterm);
  }
}

// The rows of the general way, and slow = 1 on the D rows.
__global__ void k_bulk_list(int64_t M, int64_t P2, uint8_t* slow, int64_t* list, unsigned long long* count) {
  const int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  bool take = false;
  if (s < M) {
    if (s >= P2) slow[s] = 1;
    take = s >= P2 || slow[s];
  }
  const unsigned m = __ballot_sync(0xffffffffu, take);
  const int lane = threadIdx.x & 31;
  unsigned long long k = 0;
  if (lane == 0 && m) k = atomicAdd(count, (unsigned long long)__popc(m));
  k = __shfl_sync(0xffffffffu, k, 0);
  if (take) list[k + __popc(m & ((1u << lane) - 1u))] = s;
}

inline unsigned nb(int64_t n, int bs) { return (unsigned)((n + bs - 1) / bs); }

}  // namespace

namespace lbi {

size_t csr_bulk_bytes(int N, int nP) {
  const size_t nn = (size_t)N * N, a = 256;
  auto r = [&](size_t x) { return (x + a - 1) & ~(a - 1); };
  return r(16 * nn * nP) + r(8 * nn * nP) + r(4 * nn) + r(nn) + r(8 * (size_t)N) + r(4 * (size_t)N * kMaxDeg) +
         r(16 * (size_t)N * kMaxDeg) + r(16 * (size_t)N * kMaxDeg * nP) + 2 * r(4 * (size_t)N * kMaxNear) +
         4 * r(4 * (size_t)N) + r(4 * (size_t)N * (nP + 1)) + 5 * a + r(nn) + 2 * r(8 * (size_t)(nP + 1));
}

CsrBulk csr_bulk_carve(void* mem, int N, int nP, const double* gamma) {
  char* p = static_cast<char*>(mem);
  auto take = [&](size_t n) {
    char* q = p;
    p += (n + 255) & ~size_t(255);
    return static_cast<void*>(q);
  };
  const size_t nn = (size_t)N * N;
  CsrBulk b{};
  // zeroed by csr_bulk_count: L, mag, cnt, near, smax, maxdeg, cplx, mx, gd
  b.L = static_cast<double2*>(take(16 * nn * nP));
  b.mag = static_cast<double*>(take(8 * nn * nP));
  b.cnt = static_cast<int*>(take(4 * nn));
  b.near = static_cast<uint8_t*>(take(nn));
  b.smax = static_cast<double*>(take(8));
  b.maxdeg = static_cast<int*>(take(4));
  b.cplx = static_cast<int*>(take(4));
  b.mx = static_cast<double*>(take(8 * (size_t)(nP + 1)));
  b.gd = static_cast<double*>(take(8 * (size_t)(nP + 1)));
  b.zeroed = (size_t)(p - static_cast<char*>(mem));
  b.hdiag = static_cast<double*>(take(8 * (size_t)N));
  b.ucol = static_cast<int*>(take(4 * (size_t)N * kMaxDeg));
  b.G = static_cast<double2*>(take(16 * (size_t)N * kMaxDeg));
  b.Lu = static_cast<double2*>(take(16 * (size_t)N * kMaxDeg * nP));
  b.nbr = static_cast<int*>(take(4 * (size_t)N * kMaxNear));
  b.nbc = static_cast<int*>(take(4 * (size_t)N * kMaxNear));
  b.deg = static_cast<int*>(take(4 * (size_t)N));
  b.nn1 = static_cast<int*>(take(4 * (size_t)N));
  b.nh = static_cast<int*>(take(4 * (size_t)N));
  b.d1 = static_cast<int*>(take(4 * (size_t)N));
  b.npd = static_cast<int*>(take(4 * (size_t)N * (nP + 1)));
  b.slow = static_cast<uint8_t*>(take(nn));
  b.gamma = gamma;
  return b;
}

// Tables, then the count pass: slow, rowc of the rows in closed form (0 for the
// others) and their join terms, and the list of the other rows.
cudaError_t csr_bulk_count(const lb::BasisView& B, const CsrBulk& b, int nP, const int64_t* lp_ptr,
                           const int64_t* lp_idx, const double2* lp_val, int64_t nu, const double2* dl, const int* hasD,
                           const double* h, unsigned long long* rowc, unsigned long long* terms, int64_t* list,
                           unsigned long long* nlist, cudaStream_t st) {
  const int N = B.N;
  cudaError_t e = cudaMemsetAsync(b.L, 0, b.zeroed, st);
  if (e != cudaSuccess) return e;
  const int64_t nn = (int64_t)N * N * nP;
  if (nu > 0) {
    k_bulk_scatter<<<nb(nu, 256), 256, 0, st>>>(B, nP, lp_ptr, lp_idx, lp_val, nu, b);
    k_bulk_clean<<<nb(nn, 256), 256, 0, st>>>(nn, b.L, b.mag);
    note_launch(2);
  }
  k_bulk_diag<<<nP + 1, kSuffixThreads, 0, st>>>(B, nP, dl, hasD, h, b);
  k_bulk_vertex<<<nb(N, 4), 128, 0, st>>>(B, nP, h, b.gamma, b);
  k_bulk_limit<<<1, 1, 0, st>>>(nP, b);
  const unsigned grid = (unsigned)std::min<int64_t>(nb(B.P * 16, 256), 152 * 16);
  k_bulk_rows<false, 16><<<grid, 256, 0, st>>>(B, nP, b, rowc, terms, nullptr, nullptr, nullptr);
  k_bulk_rows<false, 32><<<grid, 256, 0, st>>>(B, nP, b, rowc, terms, nullptr, nullptr, nullptr);
  k_bulk_list<<<nb(B.M, 256), 256, 0, st>>>(B.M, 2 * B.P, b.slow, list, nlist);
  note_launch(6);
  return cudaGetLastError();
}

cudaError_t csr_bulk_fill(const lb::BasisView& B, const CsrBulk& b, int nP, const int64_t* rowptr, int32_t* col,
                          double* val, cudaStream_t st) {
  const unsigned grid = (unsigned)std::min<int64_t>(nb(B.P * 16, 256), 152 * 16);
  k_bulk_rows<true, 16><<<grid, 256, 0, st>>>(B, nP, b, nullptr, nullptr, rowptr, col, val);
  k_bulk_rows<true, 32><<<grid, 256, 0, st>>>(B, nP, b, nullptr, nullptr, rowptr, col, val);
  note_launch(2);
  return cudaGetLastError();
}

}  // namespace lbi
