// Near-field precorrection and local terms as a sparse Galerkin matrix.
//
// The precorrection of the precorrected-FFT method (Appendix B's near data at
// the target quadrature points, exact minus grid moments) reaches the rows
// only through the Galerkin testing of Eqs. 1-3, 13 and 14, and its sources
// only through the RWG expansion.  Both are linear and fixed while the
// conductivity is, so the product of testing, near records and expansion is
// formed once (set-up, and again for the absorber rows on every
// scabem_set_sigma): one small block per pair of edges of which some pair of
// triangles is near, together with the side-limit terms of the triangles the
// two edges share.  With J_i = -J_e on plain (L) edges and the same panel
// moments in the rows of E and H, the block of an edge pair holds
//
//   row L, col L (3):  U  G  V
//     E: U xJ - G xM                     H: G xJ + V xM
//   row L, col R (5):  Ue Ui ge gi V
//     E: Ue Je - Ui Ji - (ge + gi) M     H: ge Je - gi Ji + V M
//   row R, col L (6):  U  G  G13 V13 P Q
//     Eq. 3: U xJ - G xM   Eq. 13: G13 xJ + V13 xM   Eq. 14: P xJ + Q xM
//   row R, col R (8):  Ue Ui e13 i13 G V13 P Q
//     Eq. 3: Ue Je - Ui Ji - G M   Eq. 13: e13 Je + i13 Ji + V13 M
//     Eq. 14: P Ji + Q M (+ <X, X'> Je of edges sharing a triangle)
//
// where U = j (z/k phi - z k alpha), V = j (phi/(k z) - (k/z) alpha),
// alpha = <X, A>, phi = <div X, phi>, g = <X, curl A> of the unit current
// of the column edge, summed over media without a subscript, and the 13 / P /
// Q entries carry the sigma-weighted and side-limit terms of their rows.
//
// Edges are numbered by class here: row or column r < nL is the plain edge of
// class index r, r >= nL the absorber edge r - nL.
#include <cuda_runtime.h>

#include <algorithm>
#include <vector>

#include "device.cuh"

namespace {

using cd = cx<double>;

// values per edge pair, by (row class, column class)
__host__ __device__ constexpr int nm_words(bool rowR, bool colR) {
  return rowR ? (colR ? 8 : 6) : (colR ? 5 : 3);
}

// index of near pair (t, s) in t's ascending source list, -1 if absent
__device__ __forceinline__ int find_pair(const int32_t* __restrict__ noff, const int32_t* __restrict__ nsrc, int t,
                                         int s) {
  int lo = noff[t], hi = noff[t + 1];
  const int end = hi;
  while (lo < hi) {
    const int mid = (lo + hi) >> 1;
    if (nsrc[mid] < s)
      lo = mid + 1;
    else
      hi = mid;
  }
  return lo < end && nsrc[lo] == s ? lo : -1;
}
__device__ __forceinline__ bool near_or_same(const int32_t* __restrict__ noff, const int32_t* __restrict__ nsrc, int t,
                                             int s) {
  return t == s || find_pair(noff, nsrc, t, s) >= 0;
}

// Columns of every row, one warp per row: the edges of the near (or same)
// triangles s of the row's two triangles.  An edge met through several
// triangle pairs is kept at the first of them (T+ before T-, then the lower
// source triangle), which needs two look-ups and no sorting.  cnt != null
// counts (cnt[r] all, nl[r] plain columns); else the columns are written,
// plain ones first.
__global__ void __launch_bounds__(128) k_near_pattern(const int32_t* __restrict__ rtk, const int32_t* __restrict__ tedge,
                                                      const int32_t* __restrict__ noff,
                                                      const int32_t* __restrict__ nsrc, int64_t ne, int64_t nL,
                                                      int32_t* __restrict__ cnt, int32_t* __restrict__ nl,
                                                      const int32_t* __restrict__ off, int32_t* __restrict__ col) {
  const int64_t r = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  if (r >= ne) return;
  const int lane = threadIdx.x & 31;
  const unsigned below = (1u << lane) - 1;
  const int T0 = rtk[4 * r];
  int cl = 0, cr = 0;
  const int64_t bl = cnt ? 0 : off[r], br = cnt ? 0 : bl + nl[r];
  for (int it = 0; it < 2; ++it) {
    const int t = rtk[4 * r + 2 * it];
    const int n0 = noff[t], len = noff[t + 1] - n0;
    const int total = len > 0 ? 3 * len : 3;  // without near data: the triangle itself
    for (int i0 = 0; i0 < total; i0 += 32) {
      const int i = i0 + lane;
      bool keep = i < total;
      int m = 0;
      if (keep) {
        const int s = len > 0 ? nsrc[n0 + i / 3] : t;
        m = tedge[3 * (int64_t)s + i % 3];
        const int s2 = rtk[4 * (int64_t)m] == s ? rtk[4 * (int64_t)m + 2] : rtk[4 * (int64_t)m];
        if (s2 < s && near_or_same(noff, nsrc, t, s2)) keep = false;
        if (keep && it == 1 && (near_or_same(noff, nsrc, T0, s) || near_or_same(noff, nsrc, T0, s2))) keep = false;
      }
      const unsigned ml = __ballot_sync(0xffffffffu, keep && m < nL), mr = __ballot_sync(0xffffffffu, keep && m >= nL);
      if (!cnt && keep) {
        if (m < nL)
          col[bl + cl + __popc(ml & below)] = m;
        else
          col[br + cr + __popc(mr & below)] = m;
      }
      cl += __popc(ml);
      cr += __popc(mr);
    }
  }
  if (cnt && lane == 0) {
    cnt[r] = cl + cr;
    nl[r] = cl;
  }
}

// Sorts each class segment of a row's columns by edge number, one warp per row
// (rank by counting): neighbouring lanes of the products then gather from
// neighbouring unknowns.  Segments longer than NM_SORT stay as they are.
constexpr int NM_SORT = 1024;
__global__ void __launch_bounds__(128) k_near_sort(const int32_t* __restrict__ off, const int32_t* __restrict__ nl,
                                                   int64_t ne, const int32_t* __restrict__ in,
                                                   int32_t* __restrict__ out) {
  const int64_t r = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  if (r >= ne) return;
  for (int seg = 0; seg < 2; ++seg) {
    const int b = off[r] + (seg ? nl[r] : 0), n = (seg ? off[r + 1] : off[r] + nl[r]) - b;
    for (int j = threadIdx.x & 31; j < n; j += 32) {
      const int m = in[b + j];
      int rank = n > NM_SORT ? j : 0;
      if (n <= NM_SORT)
        for (int k = 0; k < n; ++k) rank += in[b + k] < m;
      out[b + rank] = m;
    }
  }
}

// tpos[i] = position of row r among the columns of row m = col[i] (the
// pattern is symmetric), one warp per row r
__global__ void __launch_bounds__(128) k_near_tpos(const int32_t* __restrict__ off, const int32_t* __restrict__ nl,
                                                   const int32_t* __restrict__ col, int64_t ne, int64_t nL,
                                                   int32_t* __restrict__ tpos) {
  const int64_t r = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  if (r >= ne) return;
  for (int i = off[r] + (threadIdx.x & 31); i < off[r + 1]; i += 32) {
    const int m = col[i];
    const int b = off[m], e0 = r < nL ? b : b + nl[m], e1 = r < nL ? b + nl[m] : off[m + 1];
    int p = 0;
    for (int k = e0; k < e1; ++k)
      if (col[k] == r) p = k - b;
    tpos[i] = p;
  }
}

// Values of the rows r0 .. ne - 1, one warp per row, one lane per column (bound by
// the FP64 pipe and divergent lanes: 9 ms for the 5 um guide, 4 for its absorber
// rows, once per conductivity):
// sums over the (at most four) near triangle pairs of the edge pair and the
// target points, in FP64, from the near records of type RG.  Written to the
// row-wise (f) and the transposed (t) copies of each precision that is built.
template <typename RG>
__global__ void __launch_bounds__(128)
    k_near_values(int64_t r0, int64_t ne, int64_t nL, const int32_t* __restrict__ off, const int32_t* __restrict__ nl,
                  const int32_t* __restrict__ col, const int32_t* __restrict__ tpos, const int64_t* __restrict__ vo,
                  const int64_t* __restrict__ vt, const int32_t* __restrict__ rtk, const int32_t* __restrict__ noff,
                  const int32_t* __restrict__ nsrc, const cx<RG>* __restrict__ rec, const double* __restrict__ tri,
                  const double* __restrict__ cX, const double* __restrict__ tp, const double* __restrict__ sig, int q,
                  double ke, double ki, double ze, double zi, cd* __restrict__ fd, cd* __restrict__ td,
                  cx<float>* __restrict__ ff, cx<float>* __restrict__ tf) {
  const int64_t r = r0 + ((blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5);
  if (r >= ne) return;
  const bool rowR = r >= nL;
  const int cl = nl[r], c0 = off[r], cnt = off[r + 1] - c0;
  for (int j = threadIdx.x & 31; j < cnt; j += 32) {
    const int m = col[c0 + j];
    const bool colR = m >= nL;
    cd al[2], ph[2], ga[2];  // alpha, phi, gamma per medium
    for (int i = 0; i < 2; ++i) al[i] = ph[i] = ga[i] = mk(0.0, 0.0);
    cd s13J = mk(0.0, 0.0), s13M = s13J, s14J = s13J, s14M = s13J;  // sigma-weighted, without the factor j of J
    double xx = 0.0, xnx = 0.0, sxx = 0.0, sxnx = 0.0;              // shared-triangle terms
    for (int pr = 0; pr < 4; ++pr) {
      const int t = rtk[4 * r + 2 * (pr >> 1)], k = rtk[4 * r + 2 * (pr >> 1) + 1];
      const int s = rtk[4 * (int64_t)m + 2 * (pr & 1)], l = rtk[4 * (int64_t)m + 2 * (pr & 1) + 1];
      const int p = find_pair(noff, nsrc, t, s);
      if (p < 0 && t != s) continue;
      const double* n = tri + 16 * (int64_t)t + 12;
      const double* gs = tri + 16 * (int64_t)s;
      const double a0 = cX[3 * (int64_t)s + l];
      const double be[3] = {a0 * (gs[3 * l] - gs[9]), a0 * (gs[3 * l + 1] - gs[10]), a0 * (gs[3 * l + 2] - gs[11])};
      for (int a = 0; a < q; ++a) {
        const int64_t Qa = (int64_t)t * q + a;
        const double* tq = tp + 16 * Qa;
        const double w = tq[3], sg = rowR ? w * sig[Qa] : 0.0, dv = w * tq[13 + k];
        const double X[3] = {tq[4 + 3 * k], tq[5 + 3 * k], tq[6 + 3 * k]};
        const double nX[3] = {n[1] * X[2] - n[2] * X[1], n[2] * X[0] - n[0] * X[2], n[0] * X[1] - n[1] * X[0]};
        if (t == s) {
          const double* Y = tq + 4 + 3 * l;
          const double d = X[0] * Y[0] + X[1] * Y[1] + X[2] * Y[2];
          const double c = -(nX[0] * Y[0] + nX[1] * Y[1] + nX[2] * Y[2]);  // X . (n x Y)
          xx += w * d;
          xnx += w * c;
          sxx += sg * d;
          sxnx += sg * c;
        }
        if (p < 0) continue;
        // X . (Q x be) = Q . (be x X)
        const double bX[3] = {be[1] * X[2] - be[2] * X[1], be[2] * X[0] - be[0] * X[2], be[0] * X[1] - be[1] * X[0]};
        const double Xb = X[0] * be[0] + X[1] * be[1] + X[2] * be[2];
#pragma unroll
        for (int med = 0; med < 2; ++med) {
          const cx<RG>* dp = rec + (((int64_t)p * q + a) * 2 + med) * NCORR;
          cd d[NCORR];
#pragma unroll
          for (int c = 0; c < NCORR; ++c) d[c] = mk((double)dp[c].re, (double)dp[c].im);
          cd xa = mk(0.0, 0.0), xc = xa;
#pragma unroll
          for (int c = 0; c < 3; ++c) {
            axpy(xa, a0 * X[c], d[1 + c]);
            axpy(xc, a0 * X[c], d[7 + c]);
            axpy(xc, -bX[c], d[4 + c]);
          }
          axpy(xa, -Xb, d[0]);
          axpy(al[med], w, xa);
          axpy(ph[med], 2.0 * a0 * dv, d[0]);
          axpy(ga[med], w, xc);
          if (rowR) {
            const double k_ = med ? ki : ke, z = med ? zi : ze;
            if (med == 0) {
              const double nb = nX[0] * be[0] + nX[1] * be[1] + nX[2] * be[2];
              const double bn[3] = {be[1] * nX[2] - be[2] * nX[1], be[2] * nX[0] - be[0] * nX[2],
                                    be[0] * nX[1] - be[1] * nX[0]};
              cd na = mk(0.0, 0.0), ng = na, nc = na;
#pragma unroll
              for (int c = 0; c < 3; ++c) {
                axpy(na, a0 * nX[c], d[1 + c]);
                axpy(ng, 2.0 * a0 * nX[c], d[4 + c]);
                axpy(nc, a0 * nX[c], d[7 + c]);
                axpy(nc, -bn[c], d[4 + c]);
              }
              axpy(na, -nb, d[0]);
              axpy(s13J, sg * z * k_, na);
              axpy(s13J, sg * z / k_, ng);
              axpy(s13M, sg, nc);
            } else {
              cd xg = mk(0.0, 0.0);
#pragma unroll
              for (int c = 0; c < 3; ++c) axpy(xg, 2.0 * a0 * X[c], d[4 + c]);
              axpy(s14J, sg * z * k_, xa);
              axpy(s14J, sg * z / k_, xg);
              axpy(s14M, -sg, xc);
            }
          }
        }
      }
    }
    const cd Ue = mulj((ze / ke) * ph[0] - (ze * ke) * al[0]), Ui = mulj((zi / ki) * ph[1] - (zi * ki) * al[1]);
    const cd V = mulj((1.0 / (ke * ze)) * ph[0] - (ke / ze) * al[0] + (1.0 / (ki * zi)) * ph[1] - (ki / zi) * al[1]);
    const cd G = ga[0] + ga[1];
    cd v[8];
    if (!rowR) {
      if (!colR) {
        v[0] = Ue + Ui;
        v[1] = G;
        v[2] = V;
      } else {
        v[0] = Ue;
        v[1] = Ui;
        v[2] = ga[0];
        v[3] = ga[1];
        v[4] = V;
      }
    } else {
      const cd V13 = V + s13M - mk(0.5 * sxx, 0.0), Q = s14M - mk(0.5 * sxnx, 0.0);
      if (!colR) {
        v[0] = Ue + Ui;
        v[1] = G;
        v[2] = G + mulj(s13J);
        v[3] = V13;
        v[4] = -mulj(s14J);
        v[5] = Q;
      } else {
        v[0] = Ue;
        v[1] = Ui;
        v[2] = ga[0] + mulj(s13J) - mk(0.5 * xnx, 0.0);
        v[3] = -ga[1] - mk(0.5 * xnx, 0.0);
        v[4] = G;
        v[5] = V13;
        v[6] = mulj(s14J) + mk(xx, 0.0);
        v[7] = Q;
      }
    }
    const int words = nm_words(rowR, colR);
    // row-wise: [plain columns][word][column], [absorber columns][word][column]
    const int64_t fb = vo[r] + (colR ? (int64_t)nm_words(rowR, false) * cl + (j - cl) : j);
    const int fs = colR ? cnt - cl : cl;
    // transposed: row m, its neighbours' position of r
    const int tl = nl[m], tc = off[m + 1] - off[m], tj = tpos[c0 + j];
    const int64_t tb = vt[m] + (rowR ? (int64_t)nm_words(false, colR) * tl + (tj - tl) : tj);
    const int ts = rowR ? tc - tl : tl;
    for (int e = 0; e < words; ++e) {
      if (fd) fd[fb + (int64_t)e * fs] = v[e];
      if (ff) ff[fb + (int64_t)e * fs] = cvt<float>(v[e]);
      if (td) td[tb + (int64_t)e * ts] = v[e];
      if (tf) tf[tb + (int64_t)e * ts] = cvt<float>(v[e]);
    }
  }
}

// <X_r, X_m> of absorber edge r with the absorber edges m of its two
// triangles (at most five): the Eq. 14 coefficient of J_e
__global__ void k_near_gram(const int32_t* __restrict__ rtk, const int32_t* __restrict__ tedge,
                            const double* __restrict__ tp, int64_t ne, int64_t nL, int q, int32_t* __restrict__ gcol,
                            double* __restrict__ gd, float* __restrict__ gf) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= ne - nL) return;
  const int64_t r = nL + i;
  int col[5];
  double val[5];
  int n = 0;
  for (int it = 0; it < 2; ++it) {
    const int64_t t = rtk[4 * r + 2 * it];
    const int k = rtk[4 * r + 2 * it + 1];
    for (int l = 0; l < 3; ++l) {
      const int m = tedge[3 * t + l];
      if (m < nL) continue;
      double s = 0.0;
      for (int a = 0; a < q; ++a) {
        const double* tq = tp + 16 * (t * q + a);
        for (int c = 0; c < 3; ++c) s += tq[3] * tq[4 + 3 * k + c] * tq[4 + 3 * l + c];
      }
      int f = 0;
      while (f < n && col[f] != m) ++f;
      if (f == n) {
        if (n == 5) continue;
        col[n] = m;
        val[n++] = 0.0;
      }
      val[f] += s;
    }
  }
  for (int f = 0; f < 5; ++f) {
    gcol[5 * i + f] = f < n ? col[f] : -1;
    gd[5 * i + f] = f < n ? val[f] : 0.0;
    gf[5 * i + f] = f < n ? (float)val[f] : 0.f;
  }
}

// ---------------------------------------------------------------- products
// f(m, v) for the columns m = col[j] of one segment of a row, with values v[e]
// = val[e n + j], j = lane, lane + LANES, ..: the next column's values and the
// index after it are loaded before the current column's gathers of x.
template <typename R, int W, int LANES, class F>
__device__ __forceinline__ void near_segment(const int32_t* __restrict__ col, const cx<R>* __restrict__ val, int n,
                                             int lane, const F& f) {
  int j = lane;
  if (j >= n) return;
  int m = col[j], mn = j + LANES < n ? col[j + LANES] : 0;
  cx<R> v[W];
#pragma unroll
  for (int e = 0; e < W; ++e) v[e] = ldstream(val + (int64_t)e * n + j);
  while (true) {
    const int jn = j + LANES;
    const bool more = jn < n;
    cx<R> vn[W];
    int m2 = 0;
    if (more) {
      if (jn + LANES < n) m2 = col[jn + LANES];
#pragma unroll
      for (int e = 0; e < W; ++e) vn[e] = ldstream(val + (int64_t)e * n + jn);
    }
    f(m, v);
    if (!more) break;
    j = jn;
    m = mn;
    mn = m2;
#pragma unroll
    for (int e = 0; e < W; ++e) v[e] = vn[e];
  }
}

// One row of the matrix (T = false) or of its transpose (T = true) against
// the kc <= K columns of x: the row's three (two for a plain edge) sums in
// acc, each of the LANES lanes sharing the row taking every LANES-th column.
// x holds the unknowns (or, transposed, the rows) of an edge m at m, nL + m
// (plain) or nL + m, nL + m + nR, nL + m + 2 nR (absorber).
constexpr int NM_THREADS = 128;

// Where a row's data lie: near columns off .. off + cnt (nl plain ones), near
// values from vo, stencil entries xoff .. xoff + nx.
struct __align__(16) RowDesc {
  int32_t off, nl, cnt, xoff;
  int64_t vo;
  int32_t nx, pad;
};
__device__ __forceinline__ RowDesc load_desc(const RowDesc* p) {
  const int4 a = __ldg(reinterpret_cast<const int4*>(p)), b = __ldg(reinterpret_cast<const int4*>(p) + 1);
  RowDesc d;
  d.off = a.x;
  d.nl = a.y;
  d.cnt = a.z;
  d.xoff = a.w;
  d.vo = (int64_t)(((uint64_t)(uint32_t)b.y << 32) | (uint32_t)b.x);
  d.nx = b.z;
  d.pad = 0;
  return d;
}

template <typename R, int K, bool T, int LANES>
__device__ __forceinline__ void near_row(const RowDesc& D, bool isR, int64_t nL, int64_t nR,
                                         const int32_t* __restrict__ col, const cx<R>* __restrict__ val,
                                         const cx<R>* __restrict__ x, int64_t xst, int lane, cx<R> acc[3][K]) {
  const int cl = D.nl, cr = D.cnt - cl;
  const cx<R>* v0 = val + D.vo;
  const int32_t *colL = col + D.off, *colR = colL + cl;
  // the entries of x of column m: J, M of a plain edge; J_e, J_i, M of an absorber edge
#define COLUMNS2(...)                                       \
  cx<R> xa[K], xb[K];                                       \
  load_cols<R, K>(x + m * xst, xa);                \
  load_cols<R, K>(x + (m + nL) * xst, xb);                  \
  _Pragma("unroll") for (int c = 0; c < K; ++c) {           \
    const cx<R> a = xa[c], b = xb[c];                       \
    __VA_ARGS__                                             \
  }
#define COLUMNS3(...)                                       \
  cx<R> xa[K], xb[K], xd[K];                                \
  load_cols<R, K>(x + (m + nL) * xst, xa);                  \
  load_cols<R, K>(x + (m + nL + nR) * xst, xb);             \
  load_cols<R, K>(x + (m + nL + 2 * nR) * xst, xd);         \
  _Pragma("unroll") for (int c = 0; c < K; ++c) {           \
    const cx<R> a = xa[c], b = xb[c], d = xd[c];            \
    __VA_ARGS__                                             \
  }
  if (!isR) {
    near_segment<R, 3, LANES>(colL, v0, cl, lane, [&](int64_t m, const cx<R>* v) {
      COLUMNS2(  // U G V
          cmac(acc[0][c], v[0], a); cmac(acc[0][c], T ? v[1] : -v[1], b); cmac(acc[1][c], T ? -v[1] : v[1], a);
          cmac(acc[1][c], v[2], b);)
    });
    near_segment<R, T ? 6 : 5, LANES>(colR, v0 + (int64_t)nm_words(false, false) * cl, cr, lane,
                                            [&](int64_t m, const cx<R>* v) {
      if constexpr (!T) {  // Ue Ui ge gi V
        COLUMNS3(cmac(acc[0][c], v[0], a); cmac(acc[0][c], -v[1], b); cmac(acc[0][c], -(v[2] + v[3]), d);
                 cmac(acc[1][c], v[2], a); cmac(acc[1][c], -v[3], b); cmac(acc[1][c], v[4], d);)
      } else {  // U G G13 V13 P Q against the rows of Eqs. 3, 13, 14
        COLUMNS3(cmac(acc[0][c], v[0], a); cmac(acc[0][c], v[2], b); cmac(acc[0][c], v[4], d);
                 cmac(acc[1][c], -v[1], a); cmac(acc[1][c], v[3], b); cmac(acc[1][c], v[5], d);)
      }
    });
  } else {
    near_segment<R, T ? 5 : 6, LANES>(colL, v0, cl, lane,
                                            [&](int64_t m, const cx<R>* v) {
      if constexpr (!T) {  // U G G13 V13 P Q
        COLUMNS2(cmac(acc[0][c], v[0], a); cmac(acc[0][c], -v[1], b); cmac(acc[1][c], v[2], a);
                cmac(acc[1][c], v[3], b); cmac(acc[2][c], v[4], a); cmac(acc[2][c], v[5], b);)
      } else {  // Ue Ui ge gi V
        COLUMNS2(cmac(acc[0][c], v[0], a); cmac(acc[0][c], v[2], b); cmac(acc[1][c], -v[1], a);
                cmac(acc[1][c], -v[3], b); cmac(acc[2][c], -(v[2] + v[3]), a); cmac(acc[2][c], v[4], b);)
      }
    });
    near_segment<R, 8, LANES>(colR, v0 + (int64_t)(T ? 5 : 6) * cl, cr, lane,
                                    [&](int64_t m, const cx<R>* v) {
      if constexpr (!T) {  // Ue Ui e13 i13 G V13 P Q
        COLUMNS3(cmac(acc[0][c], v[0], a); cmac(acc[0][c], -v[1], b); cmac(acc[0][c], -v[4], d);
                 cmac(acc[1][c], v[2], a); cmac(acc[1][c], v[3], b); cmac(acc[1][c], v[5], d);
                 cmac(acc[2][c], v[6], b); cmac(acc[2][c], v[7], d);)
      } else {
        COLUMNS3(cmac(acc[0][c], v[0], a); cmac(acc[0][c], v[2], b); cmac(acc[1][c], -v[1], a);
                 cmac(acc[1][c], v[3], b); cmac(acc[1][c], v[6], d); cmac(acc[2][c], -v[4], a);
                 cmac(acc[2][c], v[5], b); cmac(acc[2][c], v[7], d);)
      }
    });
  }
#undef COLUMNS3
#undef COLUMNS2
}

// Sums over the LANES lanes of a row, in every lane (within a warp), or over
// the CTA's four warps in the first warp's lanes (LANES = NM_THREADS).
template <typename R, int K, int LANES>
__device__ __forceinline__ void near_reduce(cx<R> acc[3][K]) {
  constexpr int W = LANES < 32 ? LANES : 32;
#pragma unroll
  for (int o = W / 2; o > 0; o >>= 1)
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int c = 0; c < K; ++c) {
        acc[i][c].re += __shfl_xor_sync(0xffffffffu, acc[i][c].re, o);
        acc[i][c].im += __shfl_xor_sync(0xffffffffu, acc[i][c].im, o);
      }
  if constexpr (LANES > 32) {
    __shared__ cx<R> sm[LANES / 32][3 * K];
    const int w = threadIdx.x >> 5;
    if ((threadIdx.x & 31) == 0)
#pragma unroll
      for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int c = 0; c < K; ++c) sm[w][i * K + c] = acc[i][c];
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int c = 0; c < K; ++c) {
        cx<R> v = sm[0][i * K + c];
#pragma unroll
        for (int u = 1; u < LANES / 32; ++u) v += sm[u][i * K + c];
        acc[i][c] = v;
      }
  }
}

// Grid part of an edge's rows: sums over the edge's n covered grid points
// (compact points xpt) of the entry's weight blocks (stencil.cu) and the
// potential groups there.  Lane = slot * H + half group, H = 8 half groups of
// a plain edge, 16 of an absorber edge: each lane sums two complex values of
// a point against two weights into ga[c], so that a warp's loads are
// contiguous (the 128 or 256 bytes of a point in complex64).  Entries go in
// blocks of GR_IF slots: a block's point indices are loaded by the lanes one
// block ahead and handed out by shuffles, and all of its weights and (one
// right-hand side) potentials are loaded before the first is used.  AHEAD hands
// out the whole block's indices before its loads (a plain load does not move across
// a shuffle); rows_ahead says where not.
constexpr int GR_IF = 4;

__device__ __forceinline__ void load_two(const float* p, float* v) {
  const float2 u = __ldg(reinterpret_cast<const float2*>(p));
  v[0] = u.x;
  v[1] = u.y;
}
__device__ __forceinline__ void load_two(const double* p, double* v) {
  const double2 u = __ldg(reinterpret_cast<const double2*>(p));
  v[0] = u.x;
  v[1] = u.y;
}
// two potentials, by plain loads (pdl_wait)
__device__ __forceinline__ void load_pot(const cx<float>* p, cx<float>* v) {
  const float4 u = *reinterpret_cast<const float4*>(p);
  v[0] = mk(u.x, u.y);
  v[1] = mk(u.z, u.w);
}
__device__ __forceinline__ void load_pot(const cx<double>* p, cx<double>* v) {
  const double2 a = *reinterpret_cast<const double2*>(p), b = *(reinterpret_cast<const double2*>(p) + 1);
  v[0] = mk(a.x, a.y);
  v[1] = mk(b.x, b.y);
}

template <typename R, int K, int H, int STRIDE, int LANES, bool AHEAD>
__device__ __forceinline__ void grid_rows(const int32_t* __restrict__ xpt, int n, const R* __restrict__ w,
                                          const cx<R>* pot, int64_t cs_g, int kc, int lane, cx<R> ga[K]) {
  constexpr int S = 32 / H, BLK = GR_IF * S, STEP = BLK * (LANES / 32);
  const int wl = lane & 31, slot = wl / H;
  int b = BLK * (lane >> 5);  // the warps of a wide row take the blocks in turn
  int id = wl < BLK && b + wl < n ? xpt[b + wl] : 0;
  for (; b < n; b += STEP) {
    const int cur = id;
    if (b + STEP + wl < n && wl < BLK) id = xpt[b + STEP + wl];
    R a[GR_IF][2];
    cx<R> g[GR_IF][2];
    const cx<R>* pp[GR_IF];
    auto point = [&](int u) { return pot + (int64_t)__shfl_sync(0xffffffffu, cur, u * S + slot) * NPOT; };
    if constexpr (AHEAD)
#pragma unroll
      for (int u = 0; u < GR_IF; ++u) pp[u] = point(u);
#pragma unroll
    for (int u = 0; u < GR_IF; ++u) {
      const int j = b + u * S + slot;
      if constexpr (!AHEAD) pp[u] = point(u);
      a[u][0] = a[u][1] = R(0);
      g[u][0] = g[u][1] = czero<R>();
      if (j < n) {
        load_two(w + (int64_t)STRIDE * j, a[u]);
        if constexpr (K == 1) load_pot(pp[u], g[u]);
      }
    }
#pragma unroll
    for (int u = 0; u < GR_IF; ++u) {
      if constexpr (K == 1) {
        axpy2(ga[0], a[u][0], g[u][0]);
        axpy2(ga[0], a[u][1], g[u][1]);
      } else if (b + u * S + slot < n) {
#pragma unroll
        for (int c = 0; c < K; ++c)
          if (c < kc) {
            load_pot(pp[u] + c * cs_g, g[u]);
            axpy2(ga[c], a[u][0], g[u][0]);
            axpy2(ga[c], a[u][1], g[u][1]);
          }
      }
    }
  }
}

// Requests the lines of n bytes at p into L2, shared between the LANES lanes of a row
template <int LANES>
__device__ __forceinline__ void prefetch_l2(const void* p, int64_t n, int lane) {
  for (int64_t o = 128 * (int64_t)lane; o < n; o += 128 * LANES)
    asm volatile("prefetch.global.L2 [%0];\n" ::"l"(static_cast<const char*>(p) + o));
}
// The whole row at its start: near values, weights and points, so
// that the passes over them, which follow one another, wait for L2 and not HBM
// (apply on the 12 um guide 122 -> 115 us: the requests run under the
// predecessor's tail).  Operators with few rows hold all of it in L2 (sphere of
// 320 triangles 20.4 -> 20.6 us), complex128 is bound by the FP64 pipe (771 ->
// 775 us), and a batch's groups would request it twice: they go without.
template <typename R, int LANES>
__device__ __forceinline__ void prefetch_row(const RowDesc& D, int wl, int wr, const cx<R>* val,
                                             const int32_t* xpt, const R* w, int wn, int lane) {
  prefetch_l2<LANES>(val + D.vo, (int64_t)(wl * D.nl + wr * (D.cnt - D.nl)) * sizeof(cx<R>), lane);
  prefetch_l2<LANES>(w, (int64_t)wn * D.nx * sizeof(R), lane);
  prefetch_l2<LANES>(xpt, (int64_t)D.nx * sizeof(int32_t), lane);
}

struct RowTables {
  const RowDesc* desc;
  const int32_t *col, *gcol, *xpt;
  int64_t ne, nL, nxl;
};

// K4: y = grid part + near part of every row, the last launch of an apply:
// LANES lanes per edge.  The testing of the potentials and the near-field
// matrix of an edge meet in one reduction, and every row is written once,
// from sums in a fixed order.  Bound by the stream of near values and
// weights (HBM on large operators) and by load latency: the near values are
// loaded a column ahead, the weights a block of entries ahead of their use.  The
// form before (near records per triangle pair and target point, 706 MB per product
// instead of 230, tested per triangle) took 145 us in complex64 and 5.0 ms in
// complex128 on the 12 um guide; this one 62 and 321 us.
template <typename R, int K, int LANES, bool AHEAD>
__global__ void __launch_bounds__(NM_THREADS, sizeof(R) == 8 ? 1 : K == 1 ? 8 : K == 2 ? 7 : 6)
    k_rows(RowTables T, const cx<R>* __restrict__ nmv, const R* __restrict__ gval, const R* __restrict__ xw,
           const cx<R>* pot, int64_t cs_g, const cx<R>* __restrict__ x, int xst, cx<R>* __restrict__ y, int64_t ldy,
           int kc) {
  // unit = (row, group of K right-hand sides): a row's groups sit in
  // neighbouring warps and share its values and weights through L1
  const int64_t unit = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) / LANES;
  const int ng = (kc + K - 1) / K;
  const int64_t r = K == 1 ? unit : unit / ng;
  const int lane = threadIdx.x % LANES, c0 = K == 1 ? 0 : (int)(unit - r * ng) * K;
  x += c0 / K * group_pad(K);
  y += c0 * ldy;
  pot += c0 * cs_g;
  kc = min(K, kc - c0);
  const int64_t nL = T.nL, nR = T.ne - nL;
  cx<R> acc[3][K];
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int c = 0; c < K; ++c) acc[i][c] = czero<R>();
  if (r < T.ne) {
    const RowDesc D = load_desc(T.desc + r);
    const int64_t x0 = D.xoff;
    const int64_t st = K == 1 ? 1 : xst;
    if constexpr (K == 1 && LANES == 32 && sizeof(R) == 4)
      prefetch_row<R, LANES>(D, r < nL ? 3 : 6, r < nL ? 5 : 8, nmv, T.xpt + x0,
                             r < nL ? xw + 8 * x0 : xw + 8 * T.nxl + 24 * (x0 - T.nxl), r < nL ? 8 : 24, lane);
    near_row<R, K, false, LANES>(D, r >= nL, nL, nR, T.col, nmv, x, st, lane, acc);
    // the near part needs x only, which was complete before the predecessor
    // (the last stage of the convolution) started: it runs beside that stage
    pdl_wait();
    cx<R> ga[K];
#pragma unroll
    for (int c = 0; c < K; ++c) ga[c] = czero<R>();
    int i;
    if (r < nL) {
      const int h = lane & 7;
      grid_rows<R, K, 8, 8, LANES, AHEAD>(T.xpt + x0, D.nx, xw + 8 * x0 + 2 * (h & 3), pot + 2 * h, cs_g, kc, lane, ga);
      i = h >> 2;  // groups 0, 1 -> E row; 2, 3 -> H row
    } else {
      const int h = lane & 15, g = h >> 1;
      grid_rows<R, K, 16, 24, LANES, AHEAD>(T.xpt + x0, D.nx,
                                            xw + 8 * T.nxl + 24 * (x0 - T.nxl) + 2 * (g < 4 ? h & 3 : h - 4),
                                            pot + 2 * h, cs_g, kc, lane, ga);
      i = (g + 2) >> 2;  // groups 0, 1 -> Eq. 3; 2 .. 5 -> Eq. 13; 6, 7 -> Eq. 14
      if (lane < 5) {
        const int g = T.gcol[5 * (r - nL) + lane];
        if (g >= 0) {
          const R s = gval[5 * (r - nL) + lane];
#pragma unroll
          for (int c = 0; c < K; ++c) axpy2(acc[2][c], s, x[(nL + g) * st + c]);
        }
      }
    }
#pragma unroll
    for (int c = 0; c < K; ++c)
#pragma unroll
      for (int u = 0; u < 3; ++u)
        if (u == i) acc[u][c] += ga[c];
  }
  near_reduce<R, K, LANES>(acc);
  if (r >= T.ne || lane >= kc) return;
  // lane c finishes column c
  cx<R>* yc = y + lane * ldy;
  cx<R> s[3];
#pragma unroll
  for (int c = 0; c < K; ++c)
    if (c == lane)
#pragma unroll
      for (int i = 0; i < 3; ++i) s[i] = acc[i][c];
  if (r < nL) {
    yc[r] = s[0];
    yc[nL + r] = s[1];
  } else {
    yc[nL + r] = s[0];
    yc[nL + r + nR] = s[1];
    yc[nL + r + 2 * nR] = s[2];
  }
}

// The same for the transposed apply: x = near part (transposed matrix) +
// projection transposed (the value blocks Q0 against the convolved adjoint
// fields of J_e, M outside, J_i, M inside: groups 4 .. 7 of pot).
template <typename R, int LANES, bool AHEAD>
__global__ void __launch_bounds__(NM_THREADS, sizeof(R) == 4 ? 8 : 1)
    k_rows_adj(RowTables T, const cx<R>* __restrict__ nmt, const R* __restrict__ gval, const R* __restrict__ xw,
               const cx<R>* pot, const cx<R>* __restrict__ y, cx<R>* __restrict__ x) {
  const int64_t r = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) / LANES;
  const int lane = threadIdx.x % LANES;
  const int64_t nL = T.nL, nR = T.ne - nL;
  cx<R> acc[3][1] = {{czero<R>()}, {czero<R>()}, {czero<R>()}};
  if (r < T.ne) {
    const RowDesc D = load_desc(T.desc + r);
    const int64_t x0 = D.xoff;
    if constexpr (LANES == 32 && sizeof(R) == 4)
      prefetch_row<R, LANES>(D, r < nL ? 3 : 5, r < nL ? 6 : 8, nmt, T.xpt + x0,
                             r < nL ? xw + 8 * x0 : xw + 8 * T.nxl + 24 * (x0 - T.nxl), r < nL ? 8 : 24, lane);
    near_row<R, 1, true, LANES>(D, r >= nL, nL, nR, T.col, nmt, y, 1, lane, acc);
    pdl_wait();  // as in k_rows
    const int h = lane & 7, grp = h >> 1;
    cx<R> gs[1] = {czero<R>()};
    if (r < nL)
      grid_rows<R, 1, 8, 8, LANES, AHEAD>(T.xpt + x0, D.nx, xw + 8 * x0 + 2 * (h & 1), pot + 16 + 2 * h, 0, 1, lane, gs);
    else
      grid_rows<R, 1, 8, 24, LANES, AHEAD>(T.xpt + x0, D.nx, xw + 8 * T.nxl + 24 * (x0 - T.nxl) + 2 * (h & 1),
                                           pot + 16 + 2 * h, 0, 1, lane, gs);
    const cx<R> ga = gs[0];
    // groups J_e, M, J_i, -M; on plain edges J_i = -J_e
    if (r < nL) {
      if (grp == 0) acc[0][0] += ga;
      if (grp == 2) acc[0][0] -= ga;
      if (grp == 1) acc[1][0] += ga;
      if (grp == 3) acc[1][0] -= ga;
    } else {
      if (grp == 0) acc[0][0] += ga;
      if (grp == 2) acc[1][0] += ga;
      if (grp == 1) acc[2][0] += ga;
      if (grp == 3) acc[2][0] -= ga;
      if (lane < 5) {
        const int g = T.gcol[5 * (r - nL) + lane];
        if (g >= 0) axpy2(acc[0][0], gval[5 * (r - nL) + lane], y[nL + g + 2 * nR]);
      }
    }
  }
  near_reduce<R, 1, LANES>(acc);
  if (r >= T.ne || lane != 0) return;
  if (r < nL) {
    x[r] = acc[0][0];
    x[nL + r] = acc[1][0];
  } else {
    x[nL + r] = acc[0][0];
    x[nL + r + nR] = acc[1][0];
    x[nL + r + 2 * nR] = acc[2][0];
  }
}

template <typename R>
PrecData<R>& pdata(scabem_op* op);
template <>
PrecData<float>& pdata<float>(scabem_op* op) {
  return op->f;
}
template <>
PrecData<double>& pdata<double>(scabem_op* op) {
  return op->d;
}

RowTables row_tables(const scabem_op* op, const void* desc) {
  return {(const RowDesc*)desc, op->nm_col, op->nm_gcol, op->xpt, op->ne, op->nL, op->nxl};
}
// A warp per row and group of right-hand sides; a whole CTA where these are few
// and the rows long, so that warps would leave the chip idle.  Products of guides and
// spheres, warps and CTAs, us, complex64 (rows of 71 to 105 columns): 624 rows
// 19.9 and 18.4, 1188 rows 20.1 and 18.8, 1992 rows 25.2 and 25.7, 2268 rows 24.0
// and 25.2, 3900 rows 30.4 and 35.1; eight columns (two groups) of 624 rows 48.7 and
// 44.4, 1020 rows 53.1 and 53.2, 1188 rows 51.3 and 53.0, 1992 rows 71.9 and 78.2: they
// meet at 14 rows and groups per SM.  Complex128 keeps the FP64 units busy sooner: 480
// rows 115.6 and 113.2, 624 rows 87.3 and 89.4, 1020 rows 96.0 and 102.9, 3900 rows
// 209 and 244: 6 per SM.
template <typename R>
bool wide_rows(const scabem_op* op, int groups) {
  return op->ne * groups < 152 * (sizeof(R) == 4 ? 14 : 6) && op->nm_nnz > 64 * op->ne;
}

// Whether a warp's row of one complex128 column hands out its point indices ahead
// of the loads: 104 registers and 16 rows per SM at a time, against 134 and 12.
// Large operators gain by it (4368 rows 208 us against 216, 29,130 rows 755 and 778).
// Up to about two waves of rows the last wave, nearly empty, decides, for either
// form at its own sizes (1776 rows 151 and 148 us, 2208 rows 160 and 166, 3072 rows
// 199 and 191, 3648 rows 204 and 202): there the form with fewer rows in flight stays.
bool rows_ahead(const scabem_op* op) { return op->ne >= 152 * 28; }

template <typename R, int K>
int launch_rows(scabem_op* op, const cx<R>* x, cx<R>* y, int64_t ldy, int kc, cudaStream_t s) {
  PrecData<R>& pd = pdata<R>(op);
  const bool wide = wide_rows<R>(op, (int)cdiv(kc, K));
  auto fn = wide ? k_rows<R, K, NM_THREADS, true> : k_rows<R, K, 32, true>;
  if constexpr (sizeof(R) == 8 && K == 1)
    if (!wide && !rows_ahead(op)) fn = k_rows<R, K, 32, false>;
  const int64_t units = op->ne * cdiv(kc, K);
  CK(launch_pdl(fn, dim3((unsigned)cdiv(units * (wide ? NM_THREADS : 32), NM_THREADS)), NM_THREADS, 0, s,
                row_tables(op, op->rdesc), pd.nmv, pd.gram, pd.xw, pd.grid, col_stride_pot(op), x, batch_stride(kc),
                y, ldy, kc));
  return SCABEM_OK;
}

}  // namespace

// y_c = A x_c from the potentials pd.grid (column c) and the near matrix, c <
// kc <= KBATCH, x in the layout of load_cols.  At most four right-hand sides
// per warp: eight hold 126 registers and half the warps (325 us for 8 columns
// of the 12 um guide; 300 us with four; 274 us with x interleaved; 249 us with a
// block's point indices handed out before its loads).
template <typename R>
int rows_apply(scabem_op* op, const cx<R>* x, cx<R>* y, int64_t ldy, int kc, cudaStream_t s) {
  switch (batch_group(kc)) {
    case 1: return launch_rows<R, 1>(op, x, y, ldy, kc, s);
    case 2: return launch_rows<R, 2>(op, x, y, ldy, kc, s);
    case 3: return launch_rows<R, 3>(op, x, y, ldy, kc, s);
    default: return launch_rows<R, 4>(op, x, y, ldy, kc, s);
  }
}
template int rows_apply<float>(scabem_op*, const cx<float>*, cx<float>*, int64_t, int, cudaStream_t);
template int rows_apply<double>(scabem_op*, const cx<double>*, cx<double>*, int64_t, int, cudaStream_t);

// x = A^T y from the convolved adjoint fields and the transposed near matrix
template <typename R>
int rows_adjoint(scabem_op* op, const cx<R>* y, cx<R>* x, cudaStream_t s) {
  PrecData<R>& pd = pdata<R>(op);
  const bool wide = wide_rows<R>(op, 1);
  auto fn = wide ? k_rows_adj<R, NM_THREADS, true> : k_rows_adj<R, 32, true>;
  if constexpr (sizeof(R) == 8)
    if (!wide && !rows_ahead(op)) fn = k_rows_adj<R, 32, false>;
  CK(launch_pdl(fn, dim3((unsigned)cdiv(op->ne * (wide ? NM_THREADS : 32), NM_THREADS)), NM_THREADS, 0, s,
                row_tables(op, op->rdesc_t), pd.nmt, pd.gram, pd.xw, pd.grid, y, x));
  return SCABEM_OK;
}
template int rows_adjoint<float>(scabem_op*, const cx<float>*, cx<float>*, cudaStream_t);
template int rows_adjoint<double>(scabem_op*, const cx<double>*, cx<double>*, cudaStream_t);

// Pattern and storage of the matrix (after the near list); its values follow
// with the first conductivity.
int setup_near_matrix(scabem_op* op, cudaStream_t s) {
  const int64_t ne = op->ne, nL = op->nL, nR = op->nR;
  const unsigned gw = (unsigned)cdiv(ne * 32, 128);
  int32_t* cnt = nullptr;
  CK(cudaMalloc(&op->nm_nl, sizeof(int32_t) * ne));
  CK(cudaMalloc(&op->nm_off, sizeof(int32_t) * (ne + 1)));
  CK(cudaMalloc(&op->nm_vo, sizeof(int64_t) * (ne + 1)));
  CK(cudaMalloc(&op->nm_vt, sizeof(int64_t) * (ne + 1)));
  cnt = op->nm_off;  // counts first, offsets afterwards
  k_near_pattern<<<gw, 128, 0, s>>>(op->rtk, op->tedge, op->noff, op->nsrc, ne, nL, cnt, op->nm_nl, nullptr, nullptr);
  CK(cudaGetLastError());
  std::vector<int32_t> hc(ne + 1), hl(ne);
  CK(cudaMemcpyAsync(hc.data(), cnt, sizeof(int32_t) * ne, cudaMemcpyDeviceToHost, s));
  CK(cudaMemcpyAsync(hl.data(), op->nm_nl, sizeof(int32_t) * ne, cudaMemcpyDeviceToHost, s));
  CK(cudaStreamSynchronize(s));
  std::vector<int64_t> vo(ne + 1), vt(ne + 1);
  int64_t acc = 0, av = 0, at = 0;
  for (int64_t r = 0; r < ne; ++r) {
    const int64_t n = hc[r], l = hl[r];
    hc[r] = (int32_t)acc;
    vo[r] = av;
    vt[r] = at;
    acc += n;
    av += nm_words(r >= nL, false) * l + nm_words(r >= nL, true) * (n - l);
    at += nm_words(false, r >= nL) * l + nm_words(true, r >= nL) * (n - l);
    if (acc > INT32_MAX) {
      set_error("near list too long: reduce r_near");
      return SCABEM_E_ARG;
    }
  }
  hc[ne] = (int32_t)acc;
  vo[ne] = av;
  vt[ne] = at;
  op->nm_nnz = acc;
  CK(cudaMemcpyAsync(op->nm_off, hc.data(), sizeof(int32_t) * (ne + 1), cudaMemcpyHostToDevice, s));
  CK(cudaMemcpyAsync(op->nm_vo, vo.data(), sizeof(int64_t) * (ne + 1), cudaMemcpyHostToDevice, s));
  CK(cudaMemcpyAsync(op->nm_vt, vt.data(), sizeof(int64_t) * (ne + 1), cudaMemcpyHostToDevice, s));
  std::vector<RowDesc> rd(ne), rt(ne);
  for (int64_t r = 0; r < ne; ++r) {
    rd[r] = {hc[r], hl[r], hc[r + 1] - hc[r], op->h_xoff[r], vo[r], op->h_xoff[r + 1] - op->h_xoff[r], 0};
    rt[r] = rd[r];
    rt[r].vo = vt[r];
  }
  std::vector<int32_t>().swap(op->h_xoff);
  CK(cudaMalloc(&op->rdesc, sizeof(RowDesc) * ne));
  CK(cudaMalloc(&op->rdesc_t, sizeof(RowDesc) * ne));
  CK(cudaMemcpyAsync(op->rdesc, rd.data(), sizeof(RowDesc) * ne, cudaMemcpyHostToDevice, s));
  CK(cudaMemcpyAsync(op->rdesc_t, rt.data(), sizeof(RowDesc) * ne, cudaMemcpyHostToDevice, s));
  CK(cudaMalloc(&op->nm_col, sizeof(int32_t) * acc));
  CK(cudaMalloc(&op->nm_tpos, sizeof(int32_t) * acc));
  k_near_pattern<<<gw, 128, 0, s>>>(op->rtk, op->tedge, op->noff, op->nsrc, ne, nL, nullptr, op->nm_nl, op->nm_off,
                                    op->nm_col);
  CK(cudaGetLastError());
  // sorted through the position table's storage
  k_near_sort<<<gw, 128, 0, s>>>(op->nm_off, op->nm_nl, ne, op->nm_col, op->nm_tpos);
  CK(cudaGetLastError());
  std::swap(op->nm_col, op->nm_tpos);
  k_near_tpos<<<gw, 128, 0, s>>>(op->nm_off, op->nm_nl, op->nm_col, ne, nL, op->nm_tpos);
  CK(cudaGetLastError());
  if (op->f.built) {
    CK(cudaMalloc(&op->f.nmv, sizeof(cx<float>) * av));
    CK(cudaMalloc(&op->f.nmt, sizeof(cx<float>) * at));
  }
  if (op->d.built) {
    CK(cudaMalloc(&op->d.nmv, sizeof(cd) * av));
    CK(cudaMalloc(&op->d.nmt, sizeof(cd) * at));
  }
  const int64_t ng = std::max<int64_t>(nR, 1) * 5;
  CK(cudaMalloc(&op->nm_gcol, sizeof(int32_t) * ng));
  CK(cudaMalloc(&op->d.gram, sizeof(double) * ng));
  CK(cudaMalloc(&op->f.gram, sizeof(float) * ng));
  if (nR > 0) {
    k_near_gram<<<(unsigned)cdiv(nR, 128), 128, 0, s>>>(op->rtk, op->tedge, op->d.tp, ne, nL, op->q, op->nm_gcol,
                                                        op->d.gram, op->f.gram);
    CK(cudaGetLastError());
  }
  CK(cudaStreamSynchronize(s));
  op->nm_ready = false;
  return SCABEM_OK;
}

// Values for the operator's current conductivity: all rows the first time,
// the absorber rows (the only ones that hold it) after that.
int near_matrix_update(scabem_op* op, cudaStream_t s) {
  const int64_t r0 = op->nm_ready ? op->nL : 0, nr = op->ne - r0;
  if (nr > 0) {
    const unsigned g = (unsigned)cdiv(nr * 32, 128);
    if (op->d.near)
      k_near_values<double><<<g, 128, 0, s>>>(r0, op->ne, op->nL, op->nm_off, op->nm_nl, op->nm_col, op->nm_tpos,
                                              op->nm_vo, op->nm_vt, op->rtk, op->noff, op->nsrc, op->d.near, op->tri,
                                              op->cX, op->d.tp, op->sig64, op->q, op->ke, op->ki, op->ze, op->zi,
                                              op->d.nmv, op->d.nmt, op->f.nmv, op->f.nmt);
    else
      k_near_values<float><<<g, 128, 0, s>>>(r0, op->ne, op->nL, op->nm_off, op->nm_nl, op->nm_col, op->nm_tpos,
                                             op->nm_vo, op->nm_vt, op->rtk, op->noff, op->nsrc, op->f.near, op->tri,
                                             op->cX, op->d.tp, op->sig64, op->q, op->ke, op->ki, op->ze, op->zi,
                                             op->d.nmv, op->d.nmt, op->f.nmv, op->f.nmt);
    CK(cudaGetLastError());
  }
  op->nm_ready = true;
  return SCABEM_OK;
}
