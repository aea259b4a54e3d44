// lb_basis.cu -- kernel (a): index-arithmetic enumeration of the nonzero
// structure constants f_mns, d_mns (Eq. (05); Table 1 step 2.2), plus the
// basis index tables, the expansion of Eq. (02) and the reconstruction of
// Eq. (rho).
//
// Canonical lists hold each unordered triple once as m <= n <= s, sorted by
// (m, n, s).  The nonzero triples fall into three classes:
//   * three pair elements whose edges form a triangle a-b-c: for given
//     types of two of them the type of the third is fixed by parity (f: odd
//     number of J's, d: even);
//   * two pair elements on one edge (a,b) and D_l: f(S_ab, J_ab, D_l) != 0
//     for max(a,1) <= l <= b; d(S_ab, S_ab, D_l) = d(J_ab, J_ab, D_l) != 0
//     for l >= max(a,1) except (a,b,l) = (0,1,1);
//   * d(D_l, D_l, D_r) for r >= l except l = r = 1 (canonical form of the
//     "two smallest equal" rule).
// The number of triples of a row m and of all rows before it are polynomials
// in the row's vertices, so one pass writes the list: no count, no scan.
#include "lb_internal.h"

namespace {

using namespace lb;

__global__ void k_tables(int N, int32_t* pair_ab, double* tab) {
  int64_t P = (int64_t)N * (N - 1) / 2;
  int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t < P) {
    // invert the lexicographic pair index
    int a = 0;
    int64_t p = t;
    // rows have N-1-a entries; a linear walk is O(N) but runs once per basis
    while (p >= N - 1 - a) {
      p -= N - 1 - a;
      ++a;
    }
    pair_ab[t] = (a << 16) | (a + 1 + (int)p);
  }
  double* c = tab;
  double* lc = tab + N;
  double* c2 = tab + 2 * N;
  double* inv = tab + 3 * N;
  if (t <= N) {
    if (t >= 1) inv[t] = 1.0 / (double)t;
    else inv[0] = 0.0;
  }
  if (t < N) {
    if (t == 0) {
      c[0] = lc[0] = c2[0] = 0.0;
    } else {
      double l = (double)t;
      double cl = 1.0 / sqrt(l * (l + 1.0));
      c[t] = cl;
      lc[t] = -l * cl;
      c2[t] = 1.0 / (l * (l + 1.0));
    }
  }
}

// ------------------------------------------------ places of the rows
// tri(n) = 1 + .. + n, tet(n) = tri(1) + .. + tri(n), sqr(n) = 1 + 4 + .. + n^2.
LB_HD int64_t tri(int64_t n) { return n * (n + 1) / 2; }
LB_HD int64_t tet(int64_t n) { return n * (n + 1) * (n + 2) / 6; }
LB_HD int64_t sqr(int64_t n) { return n * (n + 1) * (2 * n + 1) / 6; }

// Canonical triples of the S_ab rows before (a, b), of the J_ab rows before
// (a, b), and of the D_l rows before l, with lo = max(a, 1) and e = 1 on the
// edge (0, 1).  A row holds
//   f: S  2 (N-1-b) + (b-a-1) triangles and b - lo + 1 D_l;  J  N-1-b triangles
//   d: S  (N-1-b) + (N-2) triangles and N - lo - e D_l;  J  N - lo - e D_l;
//      D  N - l - [l = 1].
// (a, b) = (N-1, N) and l = N give the totals.
LB_HD int64_t rows_s(int64_t N, int which, int64_t a, int64_t b) {
  const int64_t n = N - 1, lo = a > 1 ? a : 1, in = b - a - 1;
  if (which == LB_F) {
    const int64_t before = a == 0 ? 0 : n * (2 * N - 3) + 2 * (sqr(N - 2) - sqr(n - a));
    return before + in * (2 * N - 2 - a - lo);
  }
  int64_t before = 0;
  if (a > 0) {
    const int64_t k = a - 1;  // rows a' = 1 .. k, each 3n^2 - 4n a' + a'^2 - tri(n) + tri(a')
    before = n * (3 * n - 1) - tri(n) - 1 + k * (3 * n * n - tri(n)) - 4 * n * tri(k) + sqr(k) + tet(k);
  }
  return before + in * (3 * n - lo) - (tri(b - 1) - tri(a)) - (a == 0 && b > 1 ? 1 : 0);
}
LB_HD int64_t rows_j(int64_t N, int which, int64_t a, int64_t b) {
  const int64_t n = N - 1, lo = a > 1 ? a : 1;
  if (which == LB_F) return tet(N - 2) - tet(N - 2 - a) + tri(N - 2 - a) - tri(n - b);
  const int64_t before = a == 0 ? 0 : n * n - 1 + 2 * (tet(N - 2) - tet(n - a));
  return before + (b - a - 1) * (N - lo) - (a == 0 && b > 1 ? 1 : 0);
}
LB_HD int64_t rows_d(int64_t N, int which, int64_t l) {
  return which == LB_F ? 0 : tri(N - 1) - tri(N - l) - (l > 1 ? 1 : 0);
}

// One warp per row m: lane by lane the row's triples in canonical order, a
// run of partners n for each class (below, w is the third vertex of a
// triangle; every triangle's value is 1/sqrt2 up to the stated sign):
//   f, S_ab: n = S_aw (w > b), S_wb (a < w < b), S_bw (w > b) with the J of
//            the third edge; then n = J_ab with D_l
//   f, J_ab: n = J_aw, s = J_bw, w > b
//   d, S_ab: n = S_ab with D_l; n = S_aw, s = S_bw, w > b; then, w ascending,
//            the J of the edges to a and to b (minus for a < w < b)
//   d, J_ab: n = J_ab with D_l
//   d, D_l:  n = D_l, s = D_r, r >= l
// Bound by the stores: 20 bytes a triple.  The three indices of 32 triples are
// 96 consecutive words, which the lanes exchange and write as three runs.  At
// N = 200 (1.7e7 triples of f and d, both calls) 0.66 ms with a count pass over all
// candidate partners, a scan and a fill pass, 0.135 ms so (2.5 TB/s).
__global__ void __launch_bounds__(256) k_rows(BasisView B, int which, int32_t* __restrict__ idx,
                                              double* __restrict__ val) {
  const int lane = threadIdx.x & 31;
  const int64_t m = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  if (m >= B.M) return;  // whole warps leave together
  const Elem em = decode(B, m);
  const int N = B.N, a = em.a, b = em.b, k = em.kind;
  const int32_t P = (int32_t)B.P;
  const double c = 2.0 * kInv2Sqrt2;
  auto edge = [&](int u, int v) {  // pair index (int32: M is)
    const int x = imin(u, v), y = imax(u, v);
    return (int32_t)((uint32_t)x * (uint32_t)(2 * N - x - 1) / 2u) + (y - x - 1);
  };
  int64_t off = 0;
  int cnt = 0, n1 = 0, n2 = 0, lo = 0;
  const int up = N - 1 - b;  // vertices above b
  if (k == kD) {
    if (which == LB_D) {
      lo = a == 1 ? 2 : a;
      cnt = N - lo;
      off = rows_s(N, which, N - 1, N) + rows_j(N, which, N - 1, N) + rows_d(N, which, a);
    }
  } else {
    lo = imax(a, 1);
    if (which == LB_F) {
      if (k == kS) {
        n1 = up;
        n2 = up + b - a - 1;
        cnt = n2 + up + b - lo + 1;
        off = rows_s(N, which, a, b);
      } else {
        cnt = up;
        off = rows_s(N, which, N - 1, N) + rows_j(N, which, a, b);
      }
    } else {
      if (a == 0 && b == 1) lo = 2;
      n1 = N - lo;
      if (k == kS) {
        n2 = n1 + up;
        cnt = n2 + N - 2;
        off = rows_s(N, which, a, b);
      } else {
        cnt = n1;
        off = rows_s(N, which, N - 1, N) + rows_j(N, which, a, b);
      }
    }
  }
  const int32_t eab = k == kD ? 0 : edge(a, b);
  for (int e0 = 0; e0 < cnt; e0 += 32) {
    const int e = e0 + lane;
    int32_t n = (int32_t)m, s = 0;
    double v = c;
    if (e < cnt) {
      if (k == kD) {
        const int r = lo + e;
        s = 2 * P + r - 1;
        v = 2.0 * (r == a ? (double)(1 - a) * ld_c(B, a) : ld_c(B, r));
      } else if (which == LB_F) {
        if (k == kJ) {
          const int w = b + 1 + e;
          n = P + edge(a, w);
          s = P + edge(b, w);
        } else if (e < n1) {
          const int w = b + 1 + e;
          n = edge(a, w);
          s = P + edge(b, w);
        } else if (e < n2) {
          const int w = a + 1 + (e - n1);
          n = edge(w, b);
          s = P + edge(a, w);
        } else if (e < n2 + up) {
          const int w = b + 1 + (e - n2);
          n = edge(b, w);
          s = P + edge(a, w);
        } else {
          const int l = lo + (e - n2 - up);
          n = P + eab;
          s = 2 * P + l - 1;
          v = delta(B, a, l) - delta(B, b, l);
        }
      } else {
        if (e < n1) {
          const int l = lo + e;
          s = 2 * P + l - 1;
          v = delta(B, a, l) + delta(B, b, l);
        } else if (e < n2) {
          const int w = b + 1 + (e - n1);
          n = edge(a, w);
          s = edge(b, w);
        } else {
          const int i = e - n2, w = i < a ? i : i < b - 1 ? i + 1 : i + 2;
          n = P + edge(a, w);
          s = P + edge(b, w);
          if (a < w && w < b) v = -c;
        }
      }
      val[off + e] = v;
    }
#pragma unroll
    for (int t = 0; t < 3; ++t) {
      const int word = 32 * t + lane, src = word / 3, q = word - 3 * src;
      const int32_t nn = __shfl_sync(0xffffffffu, n, src), ss = __shfl_sync(0xffffffffu, s, src);
      if (e0 + src < cnt) idx[3 * (off + e0) + word] = q == 0 ? (int32_t)m : q == 1 ? nn : ss;
    }
  }
}

// Eq. (02): coef_j = Tr(F_j A) = sum_pq (F_j)_pq A_qp.
__global__ void k_expand(BasisView B, const double2* A, double2* coef) {
  int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (j >= B.M) return;
  const int N = B.N;
  const Elem e = decode(B, j);
  double2 r;
  if (e.kind == kD) {
    const int l = e.a;
    double sr = 0.0, si = 0.0;
    for (int k = 0; k <= l; ++k) {
      const double w = delta(B, k, l);
      const double2 x = A[(int64_t)k * N + k];
      sr += w * x.x;
      si += w * x.y;
    }
    r = make_double2(sr, si);
  } else {
    const double2 ab = A[(int64_t)e.a * N + e.b];  // A_ab
    const double2 ba = A[(int64_t)e.b * N + e.a];  // A_ba
    if (e.kind == kS) {
      // (A_ba + A_ab)/sqrt2
      r = make_double2(kInvSqrt2 * (ba.x + ab.x), kInvSqrt2 * (ba.y + ab.y));
    } else {
      // (-i A_ba + i A_ab)/sqrt2
      r = make_double2(kInvSqrt2 * (ba.y - ab.y), kInvSqrt2 * (ab.x - ba.x));
    }
  }
  coef[j] = r;
}

// Eq. (rho): rho = 1/N + sum_i v_i F_i.
__global__ void k_rho(BasisView B, const double* v, double2* out, double id) {
  const int N = B.N;
  int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t >= (int64_t)N * N) return;
  const int p = (int)(t / N), q = (int)(t % N);
  double2 r;
  if (p == q) {
    double s = id;
    for (int l = imax(p, 1); l < N; ++l) s += v[d_index(B, l)] * delta(B, p, l);
    r = make_double2(s, 0.0);
  } else {
    const int64_t pi = pair_index_any(N, p, q);
    const double vs = v[pi], vj = v[B.P + pi];
    // S contributes v_S/sqrt2 at (p,q) and (q,p); J_ab contributes -i v_J/sqrt2 at (a,b), +i at (b,a)
    const double sg = p < q ? -1.0 : 1.0;
    r = make_double2(kInvSqrt2 * vs, sg * kInvSqrt2 * vj);
  }
  out[t] = r;
}

inline unsigned nblocks(int64_t n, int bs) { return (unsigned)((n + bs - 1) / bs); }

}  // namespace

namespace lbi {

cudaError_t build_tables(int N, int32_t* pair_ab, double* tab, cudaStream_t st) {
  int64_t P = (int64_t)N * (N - 1) / 2;
  int64_t n = P > N + 1 ? P : N + 1;
  k_tables<<<nblocks(n, 256), 256, 0, st>>>(N, pair_ab, tab);
  note_launch(1);
  return cudaGetLastError();
}

int64_t structure_total(int N, int which) {
  return rows_s(N, which, N - 1, N) + rows_j(N, which, N - 1, N) + rows_d(N, which, N);
}

cudaError_t structure_fill(const lb::BasisView& B, int which, int32_t* idx3, double* val, cudaStream_t st) {
  k_rows<<<nblocks(B.M * 32, 256), 256, 0, st>>>(B, which, idx3, val);
  note_launch(1);
  return cudaGetLastError();
}

cudaError_t expand(const lb::BasisView& B, const double2* A, double2* coef, cudaStream_t st) {
  k_expand<<<nblocks(B.M, 256), 256, 0, st>>>(B, A, coef);
  note_launch(1);
  return cudaGetLastError();
}

cudaError_t rho(const lb::BasisView& B, const double* v, double2* out, cudaStream_t st) {
  k_rho<<<nblocks((int64_t)B.N * B.N, 256), 256, 0, st>>>(B, v, out, 1.0 / B.N);
  note_launch(1);
  return cudaGetLastError();
}

cudaError_t synth(const lb::BasisView& B, const double* v, double2* out, cudaStream_t st) {
  k_rho<<<nblocks((int64_t)B.N * B.N, 256), 256, 0, st>>>(B, v, out, 0.0);
  note_launch(1);
  return cudaGetLastError();
}

}  // namespace lbi
