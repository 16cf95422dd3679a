// Right-hand side, GMRES with iterative refinement, fields
// at interior points and the reflection fit.
//
// * rhs: tested incident field b (Appendix A): per row type <X, E_inc>,
//   <X, H_inc>, <X, H_inc> (Eq. 13), <sigma X, E_inc> (Eq. 14) for an
//   interior source (Eqs. 8-9); the mirrored combination, with
//   <sigma n x X, E_inc> in Eq. 13, for an exterior source.
// * solve: restarted GMRES (the paper's iterative solver, Appendix B) with
//   classical Gram-Schmidt on the device, its second pass where the DGKS
//   test asks, on Krylov vectors held as FP32 (hi, lo) pairs (about 48
//   bits, products and sums on the FP32 units); Hessenberg least squares by
//   Givens rotations in FP64; right-preconditioned by the inverse per-edge
//   diagonal blocks (the block-diagonal preconditioner of Appendix B).  In
//   complex64 mode only the operator runs in complex64.  An outer FP64
//   residual r = b - A x drives iterative refinement in both modes.
// * fields / reflection: total interior field E_inc + E_i(J_i, M_i) (Eq. 8) at
//   probe points by the triangle quadrature, and a least-squares split of the
//   on-axis field into forward and backward waves (Table 1's reflection).
#include <cuda_runtime.h>

#include <algorithm>
#include <climits>
#include <cmath>
#include <mutex>
#include <string>
#include <type_traits>
#include <vector>

#include "device.cuh"

template <typename R>
int compute_summ(scabem_op* op, const cx<R>* x, cx<R>* summ, cudaStream_t s);

namespace {

using cd = cx<double>;

__device__ __forceinline__ cd cexpd(cd z) {
  double s, c;
  sincos(z.im, &s, &c);
  const double e = exp(z.re);
  return mk(e * c, e * s);
}
__device__ __forceinline__ cd cdivd(cd a, cd b) {
  const double d = b.re * b.re + b.im * b.im;
  return mk((a.re * b.re + a.im * b.im) / d, (a.im * b.re - a.re * b.im) / d);
}
__device__ __forceinline__ cd csqrtd(cd z) {
  const double r = hypot(z.re, z.im);
  if (r == 0.0) return mk(0.0, 0.0);
  const double s = sqrt(0.5 * (r + fabs(z.re)));
  if (z.re >= 0.0) return mk(s, z.im / (2.0 * s));
  return mk(fabs(z.im) / (2.0 * s), copysign(s, z.im));
}

// Incident E and H (eta0 = 1 units) of source S in a medium (k, z).
__device__ void incident(const scabem_source& S, double k, double z, const double* r, cd* E, cd* H) {
  if (S.kind == 0) {
    const double ph = k * (S.dir[0] * r[0] + S.dir[1] * r[1] + S.dir[2] * r[2]);
    double sn, cs;
    sincos(ph, &sn, &cs);
    const cd e = mk(cs, -sn);
    const double dxp[3] = {S.dir[1] * S.pol[2] - S.dir[2] * S.pol[1], S.dir[2] * S.pol[0] - S.dir[0] * S.pol[2],
                           S.dir[0] * S.pol[1] - S.dir[1] * S.pol[0]};
    for (int c = 0; c < 3; ++c) {
      E[c] = S.pol[c] * e;
      H[c] = (dxp[c] / z) * e;
    }
    return;
  }
  const double b = S.kind == 2 ? S.b : 0.0;
  cd D[3];
  for (int c = 0; c < 3; ++c) D[c] = mk(r[c] - S.pos[c], b * S.dir[c]);  // r - (pos - j b dir)
  const cd R2 = D[0] * D[0] + D[1] * D[1] + D[2] * D[2];
  const cd R = csqrtd(R2);
  const cd iR = cdivd(mk(1.0, 0.0), R);
  cd Rh[3];
  for (int c = 0; c < 3; ++c) Rh[c] = D[c] * iR;
  const cd G = (1.0 / (4.0 * M_PI)) * (cexpd(mk(0.0, -k) * R) * iR);
  const cd u = mk(0.0, k) + iR;
  const cd G1 = -(u * G);
  const cd G2 = (u * u + iR * iR) * G;
  const cd rp = S.pol[0] * Rh[0] + S.pol[1] * Rh[1] + S.pol[2] * Rh[2];
  const cd G1R = G1 * iR;
  for (int c = 0; c < 3; ++c) {
    const cd hess = (G2 * rp) * Rh[c] + G1R * (mk(S.pol[c], 0.0) - rp * Rh[c]);
    const cd L = mk(0.0, k) * (S.pol[c] * G + (1.0 / (k * k)) * hess);
    E[c] = -z * L;
  }
  H[0] = G1 * (Rh[1] * S.pol[2] - Rh[2] * S.pol[1]);
  H[1] = G1 * (Rh[2] * S.pol[0] - Rh[0] * S.pol[2]);
  H[2] = G1 * (Rh[0] * S.pol[1] - Rh[1] * S.pol[0]);
}

__global__ void k_rhs(scabem_source S, const double* __restrict__ tri, const double* __restrict__ cX,
                      const double* __restrict__ qp, const double* __restrict__ qw, const double* __restrict__ sig,
                      int64_t nt, int q, double k, double z, cd* __restrict__ val) {
  int64_t gid = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (gid >= nt * 3) return;
  const int64_t t = gid / 3;
  const int kk = (int)(gid - t * 3);
  const double* g = tri + 16 * t;
  const double cxk = cX[gid];
  cd tE = mk(0.0, 0.0), tH = tE, tnsE = tE, tsE = tE;
  for (int a = 0; a < q; ++a) {
    const int64_t Qa = t * q + a;
    const double r[3] = {qp[3 * Qa], qp[3 * Qa + 1], qp[3 * Qa + 2]};
    cd E[3], H[3];
    incident(S, k, z, r, E, H);
    double X[3];
    for (int c = 0; c < 3; ++c) X[c] = cxk * (r[c] - g[3 * kk + c]);
    const double* n = g + 12;
    const double nX[3] = {n[1] * X[2] - n[2] * X[1], n[2] * X[0] - n[0] * X[2], n[0] * X[1] - n[1] * X[0]};
    const double w = qw[Qa];
    const cd xe = X[0] * E[0] + X[1] * E[1] + X[2] * E[2];
    tE += w * xe;
    tH += w * (X[0] * H[0] + X[1] * H[1] + X[2] * H[2]);
    tnsE += (w * sig[Qa]) * (nX[0] * E[0] + nX[1] * E[1] + nX[2] * E[2]);
    tsE += (w * sig[Qa]) * xe;
  }
  // rows: <X,E>, <X,H>, Eq. 13 (<X,H> and <sigma n x X, E>), Eq. 14
  cd* o = val + gid * 4;
  if (S.side == 0) {
    o[0] = tE;
    o[1] = tH;
    o[2] = tH;
    o[3] = tsE;
  } else {
    o[0] = -tE;
    o[1] = -tH;
    o[2] = tnsE - tH;
    o[3] = mk(0.0, 0.0);
  }
}

// Right-hand-side part of the conductivity sensitivity, one thread per
// quadrature point: hs[p] -= eta0 sum_kk lam_row d(rhs_row)/d sg, the
// sigma-weighted incident-field terms of k_rhs (Eq. 14 rows for an interior
// source, Eq. 13 rows for an exterior one).
__global__ void k_rhs_sens(scabem_source S, const double* __restrict__ tri, const double* __restrict__ cX,
                           const double* __restrict__ qp, const double* __restrict__ qw, const int32_t* __restrict__ valrow,
                           const cd* __restrict__ lam, int64_t Q, int q, double k, double z, cd* __restrict__ hs) {
  const int64_t Qa = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (Qa >= Q) return;
  const int64_t t = Qa / q;
  const double* g = tri + 16 * t;
  const double r[3] = {qp[3 * Qa], qp[3 * Qa + 1], qp[3 * Qa + 2]};
  cd E[3], H[3];
  incident(S, k, z, r, E, H);
  const double w = qw[Qa];
  const double* n = g + 12;
  cd acc = mk(0.0, 0.0);
  for (int kk = 0; kk < 3; ++kk) {
    double X[3];
    for (int c = 0; c < 3; ++c) X[c] = cX[3 * t + kk] * (r[c] - g[3 * kk + c]);
    const int row = valrow[(t * 3 + kk) * 4 + (S.side == 0 ? 3 : 2)];
    if (row < 0) continue;
    cd d;
    if (S.side == 0) {
      d = X[0] * E[0] + X[1] * E[1] + X[2] * E[2];
    } else {
      const double nX[3] = {n[1] * X[2] - n[2] * X[1], n[2] * X[0] - n[0] * X[2], n[0] * X[1] - n[1] * X[0]};
      d = nX[0] * E[0] + nX[1] * E[1] + nX[2] * E[2];
    }
    acc += lam[row] * (w * d);
  }
  hs[Qa] -= ETA0 * acc;
}

// Gradient reductions over the quadrature points (one block per parameter,
// fixed tree order): g[i] = sum_p dsigma_p/dc_i hs[p].
constexpr int GRAD_THREADS = 256;
__device__ void block_sum_store(cd v, cd* out) {
  __shared__ double sr[GRAD_THREADS], si[GRAD_THREADS];
  sr[threadIdx.x] = v.re;
  si[threadIdx.x] = v.im;
  __syncthreads();
  for (int st = GRAD_THREADS / 2; st > 0; st >>= 1) {
    if (threadIdx.x < st) {
      sr[threadIdx.x] += sr[threadIdx.x + st];
      si[threadIdx.x] += si[threadIdx.x + st];
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) *out = mk(sr[0], si[0]);
}

// B-spline coefficient i: dsigma_p/dc_i = N_i(s_p), by de Boor's scheme on
// the unit coefficient vector (the same knots as k_sigma_bspline).
__global__ void k_grad_bspline(const double* __restrict__ qp, int64_t Q, double x0, double L, int axis, int ncoef,
                               const cd* __restrict__ hs, cd* __restrict__ g) {
  const int ci = blockIdx.x;
  const int nspan = ncoef - 3;
  cd acc = mk(0.0, 0.0);
  for (int64_t p = threadIdx.x; p < Q; p += GRAD_THREADS) {
    const double s = (qp[3 * p + axis] - x0) / L;
    if (s < 0.0 || s > 1.0) continue;
    int j = (int)(s * nspan);
    if (j >= nspan) j = nspan - 1;
    if (ci < j || ci > j + 3) continue;  // N_i vanishes outside its four spans
    auto knot = [&](int m) {
      const int v = m - 3;
      return v <= 0 ? 0.0 : (v >= nspan ? 1.0 : (double)v / nspan);
    };
    const int sp = j + 3;
    double d[4];
    for (int r = 0; r < 4; ++r) d[r] = (sp - 3 + r == ci) ? 1.0 : 0.0;
    for (int lvl = 1; lvl <= 3; ++lvl)
      for (int r = 3; r >= lvl; --r) {
        const int m = sp - 3 + r;
        const double den = knot(m + 4 - lvl) - knot(m);
        const double al = den > 0.0 ? (s - knot(m)) / den : 0.0;
        d[r] = (1.0 - al) * d[r - 1] + al * d[r];
      }
    acc += d[3] * hs[p];
  }
  block_sum_store(acc, g + ci);
}

// Monomial segment i: dsigma_p/dsigma0_i = u(s_p)^d of that segment.
__global__ void k_grad_monomial(const double* __restrict__ qp, int64_t Q, const double* __restrict__ seg,
                                const cd* __restrict__ hs, cd* __restrict__ g) {
  const double* sg = seg + 6 * blockIdx.x;
  const int ax = (int)sg[4];
  cd acc = mk(0.0, 0.0);
  for (int64_t p = threadIdx.x; p < Q; p += GRAD_THREADS) {
    const double s = sg[5] * (qp[3 * p + ax] - sg[0]) / sg[1];
    if (s < 0.0) continue;
    acc += pow(s > 1.0 ? 1.0 : s, sg[3]) * hs[p];
  }
  block_sum_store(acc, g + blockIdx.x);
}

template <typename R>
__global__ void k_rows_out(const cd* __restrict__ val, const int32_t* __restrict__ rowsrc, int64_t N,
                           cx<R>* __restrict__ y) {
  int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= N) return;
  const cd v = val[rowsrc[2 * i]] + val[rowsrc[2 * i + 1]];
  y[i] = mk((R)v.re, (R)v.im);
}

// E and H of one current set at points (Eqs. 15-16 evaluated off the
// surface, Eq. 8): side 0 = the interior set (J_i, -M) radiating in the
// interior medium, plus the interior incident field when asked; side 1 =
// the exterior set (J_e, M) in the exterior medium.  With A, phi of J and F,
// psi of M (point-source quadrature over every source point):
//   E = -z (jk A + (j/k) grad phi) - curl F,   H = curl A - (jk F + (j/k) grad psi) / z.
//
// k_point_currents forms each source point's weighted currents once:
// pc[b] = { position (3), J w / 4 pi (3), M w / 4 pi (3), r1, r2, 0 } with r1 = -(z j / k) div J
// and r2 = -(j / (k z)) div M (weighted alike), 20 doubles.  k_point_fields then
// sums, with G = exp(-jkR) / R and grad G = g D (D = r - r', g = -(1/R + jk) G / R),
//   E += -jzk G J + g (r1 D - D x M),   H += -(jk/z) G M + g (D x J + r2 D)
// over a slice of the sources for FP_PTS points per CTA.  It is bound by the
// FP64 units (about 180 operations per point and source, a third of them the
// sincos), so the sources are split over enough CTAs to fill the chip
// (one CTA per point left 63 points on 63 of 152 SMs: 7.6 ms against 1.8 ms
// on the 12 um guide); the slices' partial sums are added in order.
__global__ void k_point_currents(const cd* __restrict__ summ, const double* __restrict__ tri,
                                 const double* __restrict__ qp, const double* __restrict__ qw, int64_t Q, int q,
                                 double k, double z, int side, double* __restrict__ pc) {
  const int64_t b = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (b >= Q) return;
  const int64_t t = b / q;
  const double* g = tri + 16 * t;
  const cd* sj = summ + (3 * t + (side ? 0 : 1)) * 4;
  const cd* sm = summ + (3 * t + 2) * 4;
  const double w = qw[b] / (4.0 * M_PI), wm = side ? w : -w;
  double o[20];
  for (int c = 0; c < 3; ++c) {
    const double rel = qp[3 * b + c] - g[9 + c];
    const cd J = w * (rel * sj[0] - sj[1 + c]), M = wm * (rel * sm[0] - sm[1 + c]);
    o[c] = qp[3 * b + c];
    o[3 + 2 * c] = J.re;
    o[4 + 2 * c] = J.im;
    o[9 + 2 * c] = M.re;
    o[10 + 2 * c] = M.im;
  }
  const cd r1 = (-2.0 * w * z / k) * mulj(sj[0]), r2 = (-2.0 * wm / (k * z)) * mulj(sm[0]);
  o[15] = r1.re;
  o[16] = r1.im;
  o[17] = r2.re;
  o[18] = r2.im;
  o[19] = 0.0;
  for (int c = 0; c < 20; c += 2) reinterpret_cast<double2*>(pc + 20 * b)[c / 2] = make_double2(o[c], o[c + 1]);
}

constexpr int FP_PTS = 2;
constexpr int FP_THREADS = 256;

// part[(slice * npts + point) * 12 + {E (3 complex), H (3 complex)}], bound by the
// FP64 pipe (one CTA per point left most of the chip idle: 7.6 ms for 63 points of
// the 12 um guide; fields, fits and decay together 13.7 -> 3.7 ms)
template <bool WITH_H>
__global__ void __launch_bounds__(FP_THREADS) k_point_fields(const double* __restrict__ pc, int64_t Q,
                                                             const double* __restrict__ pts, int npts, double k,
                                                             double z, double* __restrict__ part) {
  constexpr int NV = WITH_H ? 12 : 6;
  const int p0 = blockIdx.x * FP_PTS;
  double r[FP_PTS][3], acc[FP_PTS][NV];
#pragma unroll
  for (int u = 0; u < FP_PTS; ++u) {
    const int p = min(p0 + u, npts - 1);
#pragma unroll
    for (int c = 0; c < 3; ++c) r[u][c] = pts[3 * p + c];
#pragma unroll
    for (int v = 0; v < NV; ++v) acc[u][v] = 0.0;
  }
  const double zk = -z * k, kz = -k / z;
  for (int64_t b = blockIdx.y * (int64_t)FP_THREADS + threadIdx.x; b < Q; b += (int64_t)gridDim.y * FP_THREADS) {
    double s[20];
#pragma unroll
    for (int c = 0; c < 10; ++c) {
      const double2 v = __ldg(reinterpret_cast<const double2*>(pc + 20 * b) + c);
      s[2 * c] = v.x;
      s[2 * c + 1] = v.y;
    }
    const cd J[3] = {mk(s[3], s[4]), mk(s[5], s[6]), mk(s[7], s[8])};
    const cd M[3] = {mk(s[9], s[10]), mk(s[11], s[12]), mk(s[13], s[14])};
    const cd r1 = mk(s[15], s[16]), r2 = mk(s[17], s[18]);
#pragma unroll
    for (int u = 0; u < FP_PTS; ++u) {
      const double D[3] = {r[u][0] - s[0], r[u][1] - s[1], r[u][2] - s[2]};
      const double d2 = D[0] * D[0] + D[1] * D[1] + D[2] * D[2];
      const double iR = rsqrt(d2), R = d2 * iR;
      double sn, cs;
      sincos(k * R, &sn, &cs);
      const cd G = mk(iR * cs, -iR * sn);
      const cd g = (-iR) * (mk(iR, k) * G);
      const cd jG = mulj(G), GE = zk * jG, GH = kz * jG;
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const int c1 = (c + 1) % 3, c2 = (c + 2) % 3;
        cd T = D[c] * r1;
        axpy(T, -D[c1], M[c2]);
        axpy(T, D[c2], M[c1]);
        cd a = mk(acc[u][2 * c], acc[u][2 * c + 1]);
        cfma(a, GE, J[c]);
        cfma(a, g, T);
        acc[u][2 * c] = a.re;
        acc[u][2 * c + 1] = a.im;
        if constexpr (WITH_H) {
          cd U = D[c] * r2;
          axpy(U, D[c1], J[c2]);
          axpy(U, -D[c2], J[c1]);
          cd h = mk(acc[u][6 + 2 * c], acc[u][7 + 2 * c]);
          cfma(h, GH, M[c]);
          cfma(h, g, U);
          acc[u][6 + 2 * c] = h.re;
          acc[u][7 + 2 * c] = h.im;
        }
      }
    }
  }
  __shared__ double red[FP_THREADS / 32][FP_PTS * NV];
  const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
#pragma unroll
  for (int u = 0; u < FP_PTS; ++u)
#pragma unroll
    for (int v = 0; v < NV; ++v) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) acc[u][v] += __shfl_xor_sync(0xffffffffu, acc[u][v], o);
      if (lane == 0) red[wp][u * NV + v] = acc[u][v];
    }
  __syncthreads();
  for (int i = threadIdx.x; i < FP_PTS * NV; i += FP_THREADS) {
    const int u = i / NV, v = i - u * NV;
    if (p0 + u >= npts) continue;
    double t = 0.0;
    for (int w = 0; w < FP_THREADS / 32; ++w) t += red[w][i];
    part[((int64_t)blockIdx.y * npts + p0 + u) * 12 + v] = t;
  }
}

// the slices' sums in order, plus the incident field; H may be null
__global__ void k_point_finish(const double* __restrict__ part, int nsl, const double* __restrict__ pts, int npts,
                               double k, double z, scabem_source inc, int has_inc, cd* __restrict__ E,
                               cd* __restrict__ H) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= npts) return;
  cd Ei[3], Hi[3];
  for (int c = 0; c < 3; ++c) Ei[c] = Hi[c] = mk(0.0, 0.0);
  if (has_inc) incident(inc, k, z, pts + 3 * p, Ei, Hi);
  double v[12];
  for (int c = 0; c < 12; ++c) v[c] = 0.0;
  for (int s = 0; s < nsl; ++s)
    for (int c = 0; c < (H ? 12 : 6); ++c) v[c] += part[((int64_t)s * npts + p) * 12 + c];
  for (int c = 0; c < 3; ++c) {
    E[3 * p + c] = Ei[c] + mk(v[2 * c], v[2 * c + 1]);
    if (H) H[3 * p + c] = Hi[c] + mk(v[6 + 2 * c], v[7 + 2 * c]);
  }
}

// Device scratch of the field evaluation at npts points
struct FieldScratch {
  double *pc = nullptr, *part = nullptr;
  int nsl = 1;
  ~FieldScratch() {
    cudaFree(pc);
    cudaFree(part);
  }
  int init(const scabem_op* op, int npts) {
    // four CTAs per SM, at least 512 source points each
    const int64_t tiles = cdiv(npts, FP_PTS);
    nsl = (int)std::max<int64_t>(1, std::min<int64_t>(cdiv(4 * 152, tiles), cdiv(op->Q, 2 * FP_THREADS)));
    CK(cudaMalloc(&pc, sizeof(double) * 20 * op->Q));
    CK(cudaMalloc(&part, sizeof(double) * 12 * npts * nsl));
    return SCABEM_OK;
  }
};

// Perimeter loss of a band of the surface (Sec. III-B): part[b] = sum over the
// quadrature points of block b with |x_axis - xc| < slab of sigma eta0 w |M|^2
// (|E_tan| = |n x M| = |M| on the sheet).
__global__ void k_band_loss(const cd* __restrict__ summ, const double* __restrict__ tri, const double* __restrict__ qp,
                            const double* __restrict__ qw, const double* __restrict__ sig, int64_t Q, int q, int axis,
                            double xc, double slab, double* __restrict__ part) {
  __shared__ double sm[256];
  double v = 0.0;
  for (int64_t b = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; b < Q; b += (int64_t)gridDim.x * blockDim.x) {
    if (fabs(qp[3 * b + axis] - xc) >= slab) continue;
    const int64_t t = b / q;
    const double* g = tri + 16 * t;
    const cd* m = summ + (3 * t + 2) * 4;
    double m2 = 0.0;
    for (int c = 0; c < 3; ++c) {
      const cd M = (qp[3 * b + c] - g[9 + c]) * m[0] - m[1 + c];
      m2 += M.re * M.re + M.im * M.im;
    }
    v += sig[b] * qw[b] * m2;
  }
  sm[threadIdx.x] = v;
  __syncthreads();
  for (int st = blockDim.x / 2; st > 0; st >>= 1) {
    if (threadIdx.x < st) sm[threadIdx.x] += sm[threadIdx.x + st];
    __syncthreads();
  }
  if (threadIdx.x == 0) part[blockIdx.x] = sm[0];
}

// ---------------------------------------------------------------- batched GMRES (FP64 Krylov work)
// K <= KBATCH right-hand sides run in lockstep.  One batched operator apply
// per Arnoldi step serves all K (the rows read the near matrix once per group of
// up to four); everything else in the step stays on the device: the
// norms, classical Gram-Schmidt whose second pass runs per column only when
// the first one cancels most of w (|w'| < |w| / sqrt 2, the Daniel-Gragg-
// Kaufman-Stewart test), the Givens update of the Hessenberg least squares
// and the convergence test.  The host reads one host-mapped word per step,
// one step behind the device, so the GPU never waits for it.  Column c of
// every K-column work array starts at c * N; the basis of column c holds
// m + 1 vectors of N from c * (m + 1) * N.
constexpr int BG_THREADS = 256;
constexpr int BG_BLOCKS = 4 * 152;  // row blocks per column of the reductions (four per SM)
constexpr int BG_TC = 4;        // basis vectors per tile of the dot products
constexpr int BG_WAVE = 3 * 152;  // dot-product blocks in one wave (4 resident per SM)
constexpr int FLAG_NONFINITE = 1, FLAG_BREAKDOWN = 2;

// Error-free transformations in round-to-nearest intrinsics, which the
// compiler neither contracts nor reassociates: Knuth's two-sum (s + e = a + b
// exactly) and the product's rounding error by FMA (a b = p + e exactly).
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
  s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}
struct dfa {  // h + l
  float h, l;
};
// acc += a b: the product exactly, the sum compensated
__device__ __forceinline__ void df_mac(dfa& acc, float a, float b) {
  const float p = __fmul_rn(a, b);
  const float e = __fmaf_rn(a, b, -p);
  float sh, t;
  two_sum(acc.h, p, sh, t);
  acc.h = sh;
  acc.l = __fadd_rn(acc.l, __fadd_rn(t, e));
}
// acc += a b for a term below the precision of acc.h (a cross term with a lo part)
__device__ __forceinline__ void df_small(dfa& acc, float a, float b) { acc.l = __fmaf_rn(a, b, acc.l); }
__device__ __forceinline__ dfa df_renorm(dfa a) {
  dfa r;
  two_sum(a.h, a.l, r.h, r.l);
  return r;
}
__device__ __forceinline__ dfa df_add(dfa a, dfa b) {
  float sh, e;
  two_sum(a.h, b.h, sh, e);
  dfa r;
  two_sum(sh, __fadd_rn(e, __fadd_rn(a.l, b.l)), r.h, r.l);
  return r;
}
__device__ __forceinline__ dfa df_shfl_xor(dfa a, int o) {
  dfa r;
  r.h = __shfl_xor_sync(0xffffffffu, a.h, o);
  r.l = __shfl_xor_sync(0xffffffffu, a.l, o);
  return r;
}
__device__ __forceinline__ double df_d(dfa a) { return (double)a.h + (double)a.l; }
// a vector element in its storage precision as (hi, lo) pairs
__device__ __forceinline__ cdf ld_df(const cx<float>* p) {
  const cx<float> v = *p;
  cdf o;
  o.rh = v.re;
  o.ih = v.im;
  o.rl = 0.f;
  o.il = 0.f;
  return o;
}
__device__ __forceinline__ cdf ld_df(const cx<double>* p) { return df_split(*p); }
__device__ __forceinline__ cdf ld_df(const cdf* p) { return *p; }

// Counts this block at *done; true in the last of n blocks, which sees the
// others' writes (and resets the counter for the next launch).
__device__ __forceinline__ bool last_block(int* done, int n) {
  __shared__ int s_last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) {
    s_last = atomicAdd(done, 1) == n - 1;
    if (s_last) *done = 0;
  }
  __syncthreads();
  if (s_last) __threadfence();
  return s_last;
}

// part[(c * rb + b) * ldp + col] = sum over row block b of conj(V_c[:, col]) . w_c,
// col in the tile blockIdx.y; with self_col, column nv is w_c itself (its
// squared norm); skipped for columns with need[c] == 0.  The basis is held
// as FP32 (hi, lo) pairs and w is read in its own precision WT (the
// complex64 operator's output in the first pass, exact as a hi part); every
// product is formed on the FP32 units with its rounding error and summed
// with compensation, so that the sums keep about 48 bits.  The last row block
// of a tile adds the parts into hout[c * ldh + col] (a separate reduction launch
// cost 3.3 us of every Arnoldi step).
template <typename WT>
__global__ void __launch_bounds__(BG_THREADS) k_bdots(const cdf* __restrict__ V, int64_t csV, int nv,
                                                      const WT* w, int64_t N, cd* __restrict__ part, int ldp,
                                                      const int* need, int self_col,
                                                      cd* __restrict__ hout, int ldh, int* __restrict__ done) {
  constexpr bool WLO = !std::is_same<WT, cx<float>>::value;  // w has lo parts
  const int c = blockIdx.z;
  pdl_wait();
  if (need && !need[c]) return;  // the whole block
  V += c * csV;
  w += c * N;
  __shared__ dfa sm[BG_THREADS / 32][2 * BG_TC];
  const int c0 = blockIdx.y * BG_TC;
  const int nc = min(BG_TC, nv + self_col - c0);
  dfa v[2 * BG_TC];  // v[2k]: real part of column c0 + k, v[2k + 1]: imaginary part
#pragma unroll
  for (int k = 0; k < 2 * BG_TC; ++k) v[k] = dfa{0.f, 0.f};
  // two rows per step (their loads in flight together)
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i0 < N; i0 += 2 * stride) {
    const int64_t i1 = i0 + stride;
    const bool two = i1 < N;
    const cdf b0 = ld_df(w + i0);
    cdf b1 = b0;
    if (two) b1 = ld_df(w + i1);
    cdf a0[BG_TC], a1[BG_TC];
#pragma unroll
    for (int k = 0; k < BG_TC; ++k) {
      const bool basis = c0 + k < nv;
      a0[k] = basis && k < nc ? V[(int64_t)(c0 + k) * N + i0] : b0;
      a1[k] = basis && k < nc && two ? V[(int64_t)(c0 + k) * N + i1] : b1;
    }
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      if (r == 1 && !two) break;
      const cdf b = r ? b1 : b0;
#pragma unroll
      for (int k = 0; k < BG_TC; ++k)
        if (k < nc) {
          const cdf a = r ? a1[k] : a0[k];
          // conj(a) b = (a.re b.re + a.im b.im) + j (a.re b.im - a.im b.re)
          df_mac(v[2 * k], a.rh, b.rh);
          df_mac(v[2 * k], a.ih, b.ih);
          df_mac(v[2 * k + 1], a.rh, b.ih);
          df_mac(v[2 * k + 1], -a.ih, b.rh);
          df_small(v[2 * k], a.rl, b.rh);
          df_small(v[2 * k], a.il, b.ih);
          df_small(v[2 * k + 1], a.rl, b.ih);
          df_small(v[2 * k + 1], -a.il, b.rh);
          if (WLO) {
            df_small(v[2 * k], a.rh, b.rl);
            df_small(v[2 * k], a.ih, b.il);
            df_small(v[2 * k + 1], a.rh, b.il);
            df_small(v[2 * k + 1], -a.ih, b.rl);
          }
        }
    }
  }
  // warp sums of the NV = 2 BG_TC values by halving exchanges: at offset
  // o = NV, NV / 2, .., 2 each lane keeps half of its values, sends the other
  // half to lane ^ o and adds what it receives, so that NV additions (not 5
  // per value) leave lane l with a value whose index is given by those bits
  // of l; plain exchanges over the remaining lane bits complete the sums.
  const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
  constexpr int NV = 2 * BG_TC;
  static_assert(NV >= 2 && NV <= 16 && (NV & (NV - 1)) == 0, "halving exchanges need a power of two");
  int idx = 0;
#pragma unroll
  for (int half = NV / 2; half >= 1; half >>= 1) {
    const int o = 2 * half;
    const bool upper = (lane & o) != 0;
    if (upper) idx += half;
#pragma unroll
    for (int t = 0; t < half; ++t) {
      const dfa send = upper ? v[t] : v[t + half];
      const dfa keep = upper ? v[t + half] : v[t];
      v[t] = df_add(keep, df_shfl_xor(send, o));
    }
  }
#pragma unroll
  for (int o = 2 * NV; o < 32; o <<= 1) v[0] = df_add(v[0], df_shfl_xor(v[0], o));
  v[0] = df_add(v[0], df_shfl_xor(v[0], 1));
  if ((lane & ~(2 * NV - 2)) == 0) sm[wp][idx] = v[0];  // one lane per value index
  __syncthreads();
  if (threadIdx.x < 2 * nc) {
    dfa t = sm[0][threadIdx.x];
    for (int k = 1; k < BG_THREADS / 32; ++k) t = df_add(t, sm[k][threadIdx.x]);
    double* o = reinterpret_cast<double*>(part + ((int64_t)c * gridDim.x + blockIdx.x) * ldp + c0);
    o[threadIdx.x] = df_d(t);
  }
  if (!last_block(done + c * gridDim.y + blockIdx.y, gridDim.x)) return;
  // the tile's last block adds the row blocks' parts, in a fixed order
  __shared__ double sr[BG_THREADS];
  const int v2 = threadIdx.x % (2 * BG_TC), g = threadIdx.x / (2 * BG_TC);
  double t = 0.0;
  if (v2 < 2 * nc)
    for (int b = g; b < gridDim.x; b += BG_THREADS / (2 * BG_TC))
      t += __ldcg(reinterpret_cast<const double*>(part + ((int64_t)c * gridDim.x + b) * ldp + c0) + v2);
  sr[threadIdx.x] = t;
  __syncthreads();
  for (int st = BG_THREADS / 2; st >= 2 * BG_TC; st >>= 1) {
    if (threadIdx.x < st) sr[threadIdx.x] += sr[threadIdx.x + st];
    __syncthreads();
  }
  if (threadIdx.x < 2 * nc) reinterpret_cast<double*>(hout + (int64_t)c * ldh + c0)[threadIdx.x] = sr[threadIdx.x];
}

// Squared norm of each column of an FP64 vector per row block (grid:
// BG_BLOCKS x K), for the residual norms at the start and the restarts.
__global__ void __launch_bounds__(BG_THREADS) k_bnorm_parts(const cd* __restrict__ x, int64_t N,
                                                            double* __restrict__ nparts) {
  const int c = blockIdx.y;
  x += c * N;
  __shared__ double sm[BG_THREADS / 32];
  double nn = 0.0;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < N; i += (int64_t)gridDim.x * blockDim.x) {
    const cd v = x[i];
    nn = fma(v.re, v.re, nn);
    nn = fma(v.im, v.im, nn);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) nn += __shfl_xor_sync(0xffffffffu, nn, o);
  if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5] = nn;
  __syncthreads();
  if (threadIdx.x == 0) {
    double v = 0.0;
    for (int k = 0; k < BG_THREADS / 32; ++k) v += sm[k];
    nparts[(int64_t)c * gridDim.x + blockIdx.x] = v;
  }
}

// wout_c = win_c - V_c h_c over nv basis vectors, stored as (hi, lo) pairs,
// and the squared norm of the new w_c per row block (grid: at most
// BG_BLOCKS x K; nparts gets gridDim.x values per column).  win is read in
// its own precision WT and may be wout itself (in place).  BV_KS lanes share
// a row and take every BV_KS-th basis vector, so that each thread's chain of
// dependent loads is BV_KS times shorter; their partial sums meet by
// shuffles.  The coefficients h (FP64) are split into (hi, lo) pairs once
// per block; every product is formed with its rounding error and summed
// with compensation.
constexpr int GM_MAXM = 200;  // largest restart length (checked by the C ABI)
// Short vectors (all K right-hand sides together) take 16 lanes per row, so that
// the chip fills and the chains shorten; long ones are bound by the basis stream
// and take 4 (8 x 5500 unknowns: 23 us with 16, 13.5 us with 4).
constexpr int BV_KS_LONG = 4, BV_KS_SHORT = 16;
inline bool bv_short(int64_t NK) { return NK * BV_KS_LONG < (int64_t)BG_BLOCKS * BG_THREADS / 2; }
inline unsigned bv_blocks(int64_t N, int K) {
  const int ks = bv_short(N * K) ? BV_KS_SHORT : BV_KS_LONG;
  return (unsigned)std::max<int64_t>(1, std::min<int64_t>(BG_BLOCKS, cdiv(N * ks, BG_THREADS)));
}
template <typename WT, int BV_KS>
__global__ void __launch_bounds__(BG_THREADS) k_bvsub_norm(const cdf* __restrict__ V, int64_t csV, int nv,
                                                           const cd* h, int ldh, const WT* win, cdf* wout, int64_t N,
                                                           double* __restrict__ nparts, const int* need,
                                                           double* __restrict__ nrm, int* __restrict__ set_need,
                                                           int* __restrict__ done) {
  const int c = blockIdx.y;
  pdl_wait();
  if (need && !need[c]) return;
  V += c * csV;
  win += c * N;
  wout += c * N;
  h += (int64_t)c * ldh;
  __shared__ cdf hs[GM_MAXM + 1];
  __shared__ dfa sm[BG_THREADS / 32];
  for (int k = threadIdx.x; k < nv; k += blockDim.x) hs[k] = df_split(h[k]);
  __syncthreads();
  const int sub = threadIdx.x & (BV_KS - 1);
  dfa nn = {0.f, 0.f};
  const int64_t rows_per_pass = (int64_t)gridDim.x * (blockDim.x / BV_KS);
  for (int64_t i0 = (int64_t)blockIdx.x * (blockDim.x / BV_KS); i0 < N; i0 += rows_per_pass) {
    const int64_t i = i0 + threadIdx.x / BV_KS;  // uniform trip count: every lane reaches the shuffles
    const bool row = i < N;
    dfa xr = {0.f, 0.f}, xi = {0.f, 0.f};
    if (row && sub == 0) {
      const cdf x0 = ld_df(win + i);
      xr = dfa{x0.rh, x0.rl};
      xi = dfa{x0.ih, x0.il};
    }
    if (row) {
      int n = 0;
#pragma unroll 4
      for (int k = sub; k < nv; k += BV_KS, ++n) {
        const cdf a = V[(int64_t)k * N + i], b = hs[k];
        // x -= a b: re += -a.re b.re + a.im b.im, im += -a.re b.im - a.im b.re
        df_mac(xr, -a.rh, b.rh);
        df_mac(xr, a.ih, b.ih);
        df_mac(xi, -a.rh, b.ih);
        df_mac(xi, -a.ih, b.rh);
        df_small(xr, -a.rh, b.rl);
        df_small(xr, -a.rl, b.rh);
        df_small(xr, a.ih, b.il);
        df_small(xr, a.il, b.ih);
        df_small(xi, -a.rh, b.il);
        df_small(xi, -a.rl, b.ih);
        df_small(xi, -a.ih, b.rl);
        df_small(xi, -a.il, b.rh);
        if ((n & 7) == 7) {
          xr = df_renorm(xr);
          xi = df_renorm(xi);
        }
      }
    }
#pragma unroll
    for (int o = 1; o < BV_KS; o <<= 1) {
      xr = df_add(xr, df_shfl_xor(xr, o));
      xi = df_add(xi, df_shfl_xor(xi, o));
    }
    if (row && sub == 0) {
      xr = df_renorm(xr);
      xi = df_renorm(xi);
      cdf o;
      o.rh = xr.h;
      o.ih = xi.h;
      o.rl = xr.l;
      o.il = xi.l;
      wout[i] = o;
      // |x|^2 = h^2 + 2 h l + l^2 per part
      df_mac(nn, xr.h, xr.h);
      df_small(nn, 2.f * xr.h, xr.l);
      df_mac(nn, xi.h, xi.h);
      df_small(nn, 2.f * xi.h, xi.l);
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) nn = df_add(nn, df_shfl_xor(nn, o));
  if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5] = nn;
  __syncthreads();
  if (threadIdx.x == 0) {
    dfa v = sm[0];
    for (int k = 1; k < BG_THREADS / 32; ++k) v = df_add(v, sm[k]);
    nparts[(int64_t)c * gridDim.x + blockIdx.x] = df_d(v);
  }
  if (!last_block(done + c, gridDim.x)) return;
  // the column's last block: |w| after the pass into nrm[4c] (pass 1: with |w|
  // before it, from the self column of the dot products, and the DGKS test)
  __shared__ double sr[BG_THREADS];
  double v = 0.0;
  for (int b = threadIdx.x; b < gridDim.x; b += BG_THREADS) v += __ldcg(nparts + (int64_t)c * gridDim.x + b);
  sr[threadIdx.x] = v;
  __syncthreads();
  for (int st = BG_THREADS / 2; st > 0; st >>= 1) {
    if (threadIdx.x < st) sr[threadIdx.x] += sr[threadIdx.x + st];
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    const double n = sqrt(fmax(sr[0], 0.0));
    nrm[4 * c] = n;
    if (set_need) {
      const double before = sqrt(fmax(h[nv].re, 0.0));
      nrm[4 * c - 1] = before;
      set_need[c] = !(n >= 0.70710678118654752 * before);
    }
  }
}

// out[c * ostride] = sqrt(sum of column c's row-block parts) (grid: K)
__global__ void k_bnorm_fin(const double* __restrict__ nparts, int nb, double* __restrict__ out, int ostride) {
  const int c = blockIdx.x;
  __shared__ double sm[BG_THREADS];
  double v = 0.0;
  for (int b = threadIdx.x; b < nb; b += blockDim.x) v += nparts[(int64_t)c * nb + b];
  sm[threadIdx.x] = v;
  __syncthreads();
  for (int st = blockDim.x / 2; st > 0; st >>= 1) {
    if (threadIdx.x < st) sm[threadIdx.x] += sm[threadIdx.x + st];
    __syncthreads();
  }
  if (threadIdx.x == 0) out[(int64_t)c * ostride] = sqrt(fmax(sm[0], 0.0));
}

// Per-column state of the lockstep solver, on the device.
struct BState {
  cd* H;        // K * m * (m + 1): column j of column c's Hessenberg at (c m + j) (m + 1)
  cd* cs;       // K * m Givens cosines
  cd* sn;       // K * m Givens sines
  cd* g;        // K * (m + 1) rotated right-hand side of the least squares
  cd* y;        // K * m least-squares solution
  cd* h1;       // K * (m + 1) first Gram-Schmidt pass
  cd* h2;       // K * (m + 1) second pass
  double* nrm;  // K * 4: |w| before, after pass 1, after pass 2; beta of the cycle
  double* rn0;  // K initial residual norms
  double* est;  // K residual estimates |g_{j+1}| / rn0
  int* need;    // K second pass wanted
  int* act;     // K still iterating in this cycle
  int* jc;      // K basis vectors in this cycle's least squares
  int* iters;   // K iterations so far
  int* col;     // K the right-hand side (column of r, d, u, t) that slot c works on
};

__device__ __forceinline__ cd shfl_up_cd(cd v, int d) {
  return mk(__shfl_up_sync(0xffffffffu, v.re, d), __shfl_up_sync(0xffffffffu, v.im, d));
}
__device__ __forceinline__ cd shfl_cd(cd v, int src) {
  return mk(__shfl_sync(0xffffffffu, v.re, src), __shfl_sync(0xffffffffu, v.im, src));
}

// The Givens step of Arnoldi column j for every active column (warp c for
// right-hand side c): Hessenberg column j = h1 + h2 (the second pass when
// taken) and |w|, the previous rotations, a new rotation, the rotated
// right-hand side and the residual estimate; a column stops when the
// estimate reaches tol or w vanishes.  word[0] = columns still active,
// word[1] |= flags (host-mapped).
//
// Rotation i maps (e_i, e_i+1) to (conj(c_i) e_i + conj(s_i) e_i+1,
// c_i e_i+1 - s_i e_i), so the entry it carries on obeys the first-order
// recurrence r_i+1 = a_i r_i + b_i with a_i = -s_i and b_i = c_i e_i+1.  The
// warp takes 32 rotations at a time and forms the prefix compositions
// (a, b) o (a', b') = (a a', a b' + b) by a shuffle scan (5 steps), which
// gives every r_i of the chunk at once: a sequential chain of FP64
// operations in one lane would pay the full issue cost of an FP64 warp
// instruction for every step on this GPU's narrow FP64 units.
__global__ void __launch_bounds__(KBATCH * 32) k_givens(BState S, int j, int m, int K, double tol,
                                                        int* __restrict__ word) {
  const int c = threadIdx.x >> 5, lane = threadIdx.x & 31;
  bool on = false;
  if (c < K && S.act[c]) {  // warp-uniform
    const cd* a1 = S.h1 + (int64_t)c * (m + 1);
    const cd* a2 = S.h2 + (int64_t)c * (m + 1);
    const bool two = S.need[c] != 0;
    const double hn = two ? S.nrm[4 * c + 2] : S.nrm[4 * c + 1];
    cd* col = S.H + ((int64_t)c * m + j) * (m + 1);
    cd* cs = S.cs + (int64_t)c * m;
    cd* sn = S.sn + (int64_t)c * m;
    cd* g = S.g + (int64_t)c * (m + 1);
    cd r = two ? a1[0] + a2[0] : a1[0];  // r_i0: entry i0 after rotations 0 .. i0 - 1
    for (int i0 = 0; i0 < j; i0 += 32) {
      const int n = min(32, j - i0);  // rotations i0 .. i0 + n - 1 (lane l: rotation i0 + l)
      const bool v = lane < n;
      cd cl = mk(1.0, 0.0), sl = mk(0.0, 0.0), e = mk(0.0, 0.0);
      if (v) {
        const int k = i0 + 1 + lane;
        cl = cs[i0 + lane];
        sl = sn[i0 + lane];
        e = two ? a1[k] + a2[k] : a1[k];
      }
      cd A = v ? -sl : mk(1.0, 0.0), B = v ? cl * e : mk(0.0, 0.0);
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const cd Ap = shfl_up_cd(A, d), Bp = shfl_up_cd(B, d);
        if (lane >= d) {
          B = A * Bp + B;
          A = A * Ap;
        }
      }
      // r_i0+l = (prefix of lanes 0 .. l - 1) applied to r_i0
      const cd Al = shfl_up_cd(A, 1), Bl = shfl_up_cd(B, 1);
      const cd ri = lane == 0 ? r : Al * r + Bl;
      if (v) col[i0 + lane] = conj(cl) * ri + conj(sl) * e;
      r = shfl_cd(A, n - 1) * r + shfl_cd(B, n - 1);
    }
    // the new rotation, computed by every lane alike, written by lane 0
    const double r2 = r.re * r.re + r.im * r.im + hn * hn;
    on = true;
    if (!isfinite(hn) || !isfinite(r2)) {
      if (lane == 0) atomicOr(word + 1, FLAG_NONFINITE);
      on = false;
    } else if (r2 == 0.0) {
      if (lane == 0) atomicOr(word + 1, FLAG_BREAKDOWN);
      on = false;
    } else {
      const double inv = rsqrt(r2), den = r2 * inv;
      const cd cj = mk(r.re * inv, r.im * inv), sj = mk(hn * inv, 0.0);
      const cd gj = g[j];
      const cd g1 = -(sj * gj);
      const double e = sqrt(g1.re * g1.re + g1.im * g1.im) / S.rn0[c];
      if (lane == 0) {
        cs[j] = cj;
        sn[j] = sj;
        col[j] = mk(den, 0.0);
        col[j + 1] = mk(0.0, 0.0);
        g[j] = conj(cj) * gj;
        g[j + 1] = g1;
        S.est[c] = e;
        S.jc[c] = j + 1;
        S.iters[c] += 1;
      }
      if (hn <= 1e-300 || e <= tol) on = false;
    }
    if (!on && lane == 0) S.act[c] = 0;
    on = on && lane == 0;
  }
  const int n = __syncthreads_count(on);
  if (threadIdx.x == 0) word[0] = n;
}

// x / |w| in (hi, lo) pairs, 1 / |w| = sh + sl: each product with its rounding error
__device__ __forceinline__ cdf df_scale(cdf x, float sh, float sl) {
  dfa r = {0.f, 0.f}, m = {0.f, 0.f};
  df_mac(r, x.rh, sh);
  df_small(r, x.rh, sl);
  df_small(r, x.rl, sh);
  df_mac(m, x.ih, sh);
  df_small(m, x.ih, sl);
  df_small(m, x.il, sh);
  r = df_renorm(r);
  m = df_renorm(m);
  cdf o;
  o.rh = r.h;
  o.ih = m.h;
  o.rl = r.l;
  o.il = m.l;
  return o;
}
// 1 / |w| of slot c (|w| after the last pass; zero when it vanishes) as (hi, lo)
__device__ __forceinline__ void inv_norm(const double* nrm, const int* need, int c, float& sh, float& sl) {
  const double n = need[c] ? nrm[4 * c + 2] : nrm[4 * c + 1];
  const double sd = n > 1e-300 ? 1.0 / n : 0.0;
  sh = __double2float_rn(sd);
  sl = __double2float_rn(sd - (double)sh);
}

// v_c,j+1 = w_c / |w_c|
__global__ void k_bscale(const cdf* __restrict__ w, cdf* __restrict__ V, int64_t csV, int j1,
                         const double* __restrict__ nrm, const int* __restrict__ need, int64_t N) {
  const int c = blockIdx.y;
  float sh, sl;
  inv_norm(nrm, need, c, sh, sl);
  w += c * N;
  V += c * csV + (int64_t)j1 * N;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < N; i += (int64_t)gridDim.x * blockDim.x)
    V[i] = df_scale(w[i], sh, sl);
}

// The same and z_c = P^-1 v_c,j+1 in one launch, for the block-diagonal
// preconditioner: one thread per (edge, row) scales the edge's entries, keeps
// its own and forms its row of the block (P^-T when transposed), written in the
// operator's precision.  One launch instead of two (4.4 + 9.3 us).
template <typename TO>
__global__ void __launch_bounds__(128) k_bscale_precond(const cdf* w, cdf* __restrict__ V, int64_t csV, int j1,
                                                        const double* nrm, const int* need, int64_t N,
                                                        const cd* __restrict__ pinv, const int32_t* __restrict__ eunk,
                                                        int64_t ne, int transposed, cx<TO>* __restrict__ z) {
  const int64_t u = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (u >= 3 * ne) return;
  const int c = blockIdx.y;
  const int64_t e = u / 3;
  const int i = (int)(u - 3 * e);
  int id[3];
  for (int l = 0; l < 3; ++l) id[l] = eunk[3 * e + l];
  const int nb = id[2] < 0 ? 2 : 3;
  if (i >= nb) return;
  cd P[3];
  for (int l = 0; l < nb; ++l) P[l] = pinv[9 * e + (transposed ? 3 * l + i : 3 * i + l)];
  pdl_wait();
  w += c * N;
  V += c * csV + (int64_t)j1 * N;
  z += c * N;
  float sh, sl;
  inv_norm(nrm, need, c, sh, sl);
  cd acc = mk(0.0, 0.0);
  for (int l = 0; l < nb; ++l) {
    const cdf v = df_scale(w[id[l]], sh, sl);
    if (l == i) V[id[l]] = v;
    acc += P[l] * df_join(v);
  }
  z[id[i]] = cvt<TO>(acc);
}

// start of a cycle in slot c (the slot's right-hand side is column col[c]
// of t): v_c,0 = t / beta_c, g_c = beta_c e_1
__global__ void k_bstart(const cd* __restrict__ t, const int* __restrict__ col, cdf* __restrict__ V, int64_t csV,
                         BState S, int m, int64_t N) {
  const int c = blockIdx.y;
  const double beta = S.nrm[4 * c + 3];
  const double s = beta > 1e-300 ? 1.0 / beta : 0.0;
  t += col[c] * N;
  V += c * csV;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < N; i += (int64_t)gridDim.x * blockDim.x)
    V[i] = df_split(s * t[i]);
  if (blockIdx.x == 0) {
    for (int i = threadIdx.x; i <= m; i += blockDim.x) S.g[(int64_t)c * (m + 1) + i] = mk(i == 0 ? beta : 0.0, 0.0);
    if (threadIdx.x == 0) S.jc[c] = 0;
  }
}

// out (column c, leading dimension N) = v_c,j in FP64, for the preconditioners
// that take FP64 input (the circulant block)
__global__ void k_bjoin(const cdf* __restrict__ V, int64_t csV, cd* __restrict__ out, int64_t N) {
  const int c = blockIdx.y;
  V += c * csV;
  out += c * N;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < N; i += (int64_t)gridDim.x * blockDim.x)
    out[i] = df_join(V[i]);
}

// least squares of the cycle: y_c = R^-1 g_c over its jc[c] columns, block c for
// right-hand side c.  Thread k holds row k's remaining right-hand side and takes
// each solved entry out of it as it becomes known: one barrier and a short FP64
// chain per entry (the pivots' reciprocals are formed before), and the columns
// of R, contiguous over the rows, are loaded a block of entries ahead.  A warp
// per column with a sum per entry took 350 us for 120 entries; 56 us now.
constexpr int BS_THREADS = 256, BS_IF = 4;
__global__ void __launch_bounds__(BS_THREADS) k_backsub(BState S, int m) {
  __shared__ cd ys[2];  // alternating: a thread is at most one entry ahead
  const int c = blockIdx.x, k = threadIdx.x, j = S.jc[c];
  const cd* H = S.H + (int64_t)c * m * (m + 1);
  cd r = mk(0.0, 0.0), inv = r, h[BS_IF];
  if (k < j) {
    r = S.g[(int64_t)c * (m + 1) + k];
    const cd hd = H[(int64_t)k * (m + 1) + k];
    const double dd = hd.re * hd.re + hd.im * hd.im;
    inv = mk(hd.re / dd, -hd.im / dd);
  }
  auto fetch = [&](int i0) {
#pragma unroll
    for (int u = 0; u < BS_IF; ++u) h[u] = k < i0 - u ? H[(int64_t)(i0 - u) * (m + 1) + k] : mk(0.0, 0.0);
  };
  fetch(j - 1);
  for (int i0 = j - 1; i0 >= 0; i0 -= BS_IF) {
    cd a[BS_IF];
#pragma unroll
    for (int u = 0; u < BS_IF; ++u) a[u] = h[u];
    fetch(i0 - BS_IF);
#pragma unroll
    for (int u = 0; u < BS_IF; ++u) {
      const int i = i0 - u;
      if (i < 0) break;  // the whole block
      if (k == i) {
        const cd y = r * inv;
        ys[i & 1] = y;
        S.y[(int64_t)c * m + i] = y;
      }
      __syncthreads();
      const cd y = ys[i & 1];
      cfma(r, -a[u], y);
    }
  }
}
static_assert(BS_THREADS >= GM_MAXM, "a thread per row");

// u (column col[c]) += V_c y_c over slot c's jc[c] basis vectors; eight lanes
// share a row, so that short vectors fill the chip (one thread per row took
// 81 us for 1572 rows and 120 vectors; 17 us now)
constexpr int BU_ROWS = 4;  // rows per warp: 64 contiguous bytes of a basis vector
__global__ void __launch_bounds__(256) k_bupdate(const cdf* __restrict__ V, int64_t csV, BState S, int m,
                                                 const int* __restrict__ col, cd* __restrict__ u, int64_t N) {
  const int c = blockIdx.y;
  const int j = S.jc[c];
  if (j == 0) return;
  V += c * csV;
  u += col[c] * N;
  const cd* y = S.y + (int64_t)c * m;
  const int lane = threadIdx.x & 31, sub = lane / BU_ROWS;
  const int64_t step = (int64_t)gridDim.x * 8 * BU_ROWS;
  for (int64_t i0 = ((int64_t)blockIdx.x * 8 + (threadIdx.x >> 5)) * BU_ROWS; i0 < N; i0 += step) {  // per warp
    const int64_t i = i0 + lane % BU_ROWS;
    cd acc = mk(0.0, 0.0);
    if (i < N)
#pragma unroll 4
      for (int l = sub; l < j; l += 32 / BU_ROWS) cfma(acc, df_join(V[(int64_t)l * N + i]), y[l]);
#pragma unroll
    for (int o = BU_ROWS; o < 32; o <<= 1) acc = xadd(acc, o);
    if (i < N && sub == 0) u[i] += acc;
  }
}

__global__ void k_sub(const cd* __restrict__ a, const cd* __restrict__ b, cd* __restrict__ o, int64_t n) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    o[i] = a[i] - b[i];
}
__global__ void k_add(cd* __restrict__ x, const cd* __restrict__ d, int64_t n) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    x[i] += d[i];
}
__global__ void k_to_f(const cd* __restrict__ a, cx<float>* __restrict__ o, int64_t n) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    o[i] = mk((float)a[i].re, (float)a[i].im);
}
__global__ void k_from_f(const cx<float>* __restrict__ a, cd* __restrict__ o, int64_t n) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    o[i] = mk((double)a[i].re, (double)a[i].im);
}

constexpr int EW_BLOCKS = 4 * 152;  // element-wise kernels: 4 blocks of 256 threads per SM

struct BWork {
  int K = 0, Kcap = 0, m = 0;
  int64_t N = 0;
  bool tr = false;
  cdf* V = nullptr;          // K (m + 1) N basis, (hi, lo) pairs
  cdf* wdf = nullptr;        // K N vector under orthogonalisation, (hi, lo) pairs
  cd* w = nullptr;           // K N FP64 operator output
  cd* z = nullptr;           // K N preconditioned basis vector
  cd* u = nullptr;           // K N solution in the preconditioned variables
  cd* t = nullptr;           // K N working residual
  cx<float>* zf = nullptr;   // K N complex64 operator input / output
  cx<float>* wf = nullptr;
  cd* part = nullptr;        // K BG_BLOCKS (m + 1)
  double* nparts = nullptr;  // K BG_BLOCKS
  BState S;
  // the Givens step of a column reads the step's h1, h2, norms and DGKS flags on
  // a stream of its own, beside the next operator apply, so these alternate
  // between two copies (BState points at the first)
  cd *h1[2] = {nullptr, nullptr}, *h2[2] = {nullptr, nullptr};
  double* nrm[2] = {nullptr, nullptr};
  int* need[2] = {nullptr, nullptr};
  int* done = nullptr;       // last-block counters of the Gram-Schmidt kernels
  int* word_h = nullptr;     // host-mapped {active columns, flags}
  int* word_d = nullptr;
  cudaStream_t side = nullptr;
  cudaEvent_t ev[2] = {nullptr, nullptr}, gs[2] = {nullptr, nullptr};
  std::vector<void*> owned;
  template <typename T>
  int get(T** p, int64_t count) {
    cudaError_t e = cudaMalloc(reinterpret_cast<void**>(p), sizeof(T) * (size_t)(count > 0 ? count : 1));
    if (e != cudaSuccess) return cuda_fail(e, "cudaMalloc (GMRES workspace)");
    owned.push_back(*p);
    return SCABEM_OK;
  }
  ~BWork() {
    if (side) {
      cudaStreamSynchronize(side);
      cudaStreamDestroy(side);
    }
    for (auto& e : gs)
      if (e) cudaEventDestroy(e);
    for (void* p : owned) cudaFree(p);
    if (word_h) cudaFreeHost(word_h);
    for (auto& e : ev)
      if (e) cudaEventDestroy(e);
  }
  int init(int k, int mm, int64_t n, bool c64, cudaStream_t s) {
    K = Kcap = k;
    m = mm;
    N = n;
    int rc;
    if ((rc = get(&V, (int64_t)K * (m + 1) * N)) || (rc = get(&wdf, K * N)) || (rc = get(&w, K * N)) || (rc = get(&z, K * N)) ||
        (rc = get(&u, K * N)) || (rc = get(&t, K * N)) || (rc = get(&part, (int64_t)K * BG_BLOCKS * (m + 1))) ||
        (rc = get(&nparts, (int64_t)K * BG_BLOCKS)) || (rc = get(&S.H, (int64_t)K * m * (m + 1))) ||
        (rc = get(&S.cs, K * m)) || (rc = get(&S.sn, K * m)) || (rc = get(&S.g, K * (m + 1))) ||
        (rc = get(&S.y, K * m)) || (rc = get(&S.rn0, K)) || (rc = get(&S.est, K)) || (rc = get(&S.act, K)) || (rc = get(&S.jc, K)) || (rc = get(&S.iters, K)) || (rc = get(&S.col, K)))
      return rc;
    for (int b = 0; b < 2; ++b)
      if ((rc = get(&h1[b], K * (m + 1))) || (rc = get(&h2[b], K * (m + 1))) || (rc = get(&nrm[b], 4 * K)) ||
          (rc = get(&need[b], K)))
        return rc;
    S.h1 = h1[0];
    S.h2 = h2[0];
    S.nrm = nrm[0];
    S.need = need[0];
    const int64_t nd = K * (cdiv(m + 1, BG_TC) + 2);
    if ((rc = get(&done, nd))) return rc;
    CK(cudaMemsetAsync(done, 0, sizeof(int) * nd, s));  // before the kernels of s that count
    CK(cudaStreamCreateWithFlags(&side, cudaStreamNonBlocking));
    for (auto& e : gs) CK(cudaEventCreateWithFlags(&e, cudaEventDisableTiming));
    if (c64 && ((rc = get(&zf, K * N)) || (rc = get(&wf, K * N)))) return rc;
    CK(cudaHostAlloc(reinterpret_cast<void**>(&word_h), 2 * sizeof(int), cudaHostAllocMapped));
    CK(cudaHostGetDevicePointer(reinterpret_cast<void**>(&word_d), word_h, 0));
    for (auto& e : ev) CK(cudaEventCreateWithFlags(&e, cudaEventDisableTiming));
    return SCABEM_OK;
  }
};

// out[c * ostride] = |x_c| for the K columns of x (c * N apart)
int bnorms(const cd* x, BWork& W, double* out, int ostride, cudaStream_t s) {
  k_bnorm_parts<<<dim3(BG_BLOCKS, W.K), BG_THREADS, 0, s>>>(x, W.N, W.nparts);
  CK(cudaGetLastError());
  k_bnorm_fin<<<W.K, BG_THREADS, 0, s>>>(W.nparts, BG_BLOCKS, out, ostride);
  CK(cudaGetLastError());
  return SCABEM_OK;
}

// wf = A zf for the K columns with the complex64 operator (the transposed
// operator when solving A^T)
int bapply_f32(scabem_op* op, BWork& W, cudaStream_t s) {
  const int64_t N = W.N;
  const int K = W.K;
  if (W.tr) {
    for (int c = 0; c < K; ++c)
      if (int rc = apply_adjoint_one<float>(op, W.zf + c * N, W.wf + c * N, s)) return rc;
    return SCABEM_OK;
  }
  return K == 1 ? apply_one<float>(op, W.zf, W.wf, s) : apply_batch<float>(op, W.zf, N, W.wf, N, K, s);
}

// w = A z for the K columns (FP64 storage, operator arithmetic in prec; the
// transposed operator when solving A^T)
int bapply(scabem_op* op, const cd* z, cd* w, int prec, BWork& W, cudaStream_t s) {
  const int64_t N = W.N;
  const int K = W.K;
  if (prec == SCABEM_C128) {
    if (W.tr) {
      for (int c = 0; c < K; ++c)
        if (int rc = apply_adjoint_one<double>(op, z + c * N, w + c * N, s)) return rc;
      return SCABEM_OK;
    }
    return K == 1 ? apply_one<double>(op, z, w, s) : apply_batch<double>(op, z, N, w, N, K, s);
  }
  k_to_f<<<EW_BLOCKS, 256, 0, s>>>(z, W.zf, K * N);
  CK(cudaGetLastError());
  if (int rc = bapply_f32(op, W, s)) return rc;
  k_from_f<<<EW_BLOCKS, 256, 0, s>>>(W.wf, w, K * N);
  CK(cudaGetLastError());
  return SCABEM_OK;
}

// Restarted GMRES for A d_c = r_c, c < K in lockstep, from d = 0 (r, d: K N
// on the device).  use[c] = false leaves column c out (d_c = 0).  iters[c]
// accumulates column c's inner iterations; est[c] is its last relative
// residual (estimate, or true residual at a restart).  Every restart cycle
// runs only the columns still above tol, packed into the first slots (the
// Krylov work of slot s belongs to column col[s]), so that converged
// columns cost nothing in the batched apply.
int gmres_batch(scabem_op* op, const cd* r, cd* d, const std::vector<char>& use, int prec, double tol, int maxit,
                BWork& W, cudaStream_t s, std::vector<int>& iters, std::vector<double>& est) {
  const int64_t N = W.N;
  const int K = W.K, m = W.m;
  const int64_t csV = (int64_t)(m + 1) * N;
  BState& S = W.S;
  CK(cudaMemsetAsync(d, 0, sizeof(cd) * K * N, s));
  CK(cudaMemsetAsync(W.u, 0, sizeof(cd) * K * N, s));
  if (int rc = bnorms(r, W, S.rn0, 1, s)) return rc;
  std::vector<double> rn0(K), beta(K);
  CK(cudaMemcpyAsync(rn0.data(), S.rn0, sizeof(double) * K, cudaMemcpyDeviceToHost, s));
  CK(cudaStreamSynchronize(s));
  std::vector<int> act(K);
  for (int c = 0; c < K; ++c) {
    if (use[c] && !std::isfinite(rn0[c])) {
      set_error("non-finite residual");
      return SCABEM_E_NONFINITE;
    }
    act[c] = use[c] && rn0[c] > 0.0;
    est[c] = 0.0;
    beta[c] = rn0[c];
  }
  // the first cycle starts from t = r, beta = |r|
  CK(cudaMemcpyAsync(W.t, r, sizeof(cd) * K * N, cudaMemcpyDeviceToDevice, s));
  int lock = 0;  // lockstep iterations
  std::vector<int> col, h_int(4 * K);
  std::vector<double> h_slot(4 * K);
  while (true) {
    col.clear();
    for (int c = 0; c < K; ++c)
      if (act[c]) col.push_back(c);
    const int Ka = (int)col.size();
    if (Ka == 0) break;
    // slot state: column map, initial norms (rn0 for the estimate, beta for the start)
    for (int a = 0; a < Ka; ++a) {
      h_int[a] = col[a];
      h_int[K + a] = 1;  // act
      h_int[2 * K + a] = 0;  // iters
      h_slot[a] = rn0[col[a]];
      h_slot[K + a] = beta[col[a]];
    }
    CK(cudaMemcpyAsync(S.col, h_int.data(), sizeof(int) * Ka, cudaMemcpyHostToDevice, s));
    CK(cudaMemcpyAsync(S.act, h_int.data() + K, sizeof(int) * Ka, cudaMemcpyHostToDevice, s));
    CK(cudaMemcpyAsync(S.iters, h_int.data() + 2 * K, sizeof(int) * Ka, cudaMemcpyHostToDevice, s));
    CK(cudaMemcpyAsync(S.rn0, h_slot.data(), sizeof(double) * Ka, cudaMemcpyHostToDevice, s));
    for (int a = 0; a < Ka; ++a)
      CK(cudaMemcpyAsync(S.nrm + 4 * a + 3, h_slot.data() + K + a, sizeof(double), cudaMemcpyHostToDevice, s));
    CK(cudaStreamSynchronize(s));  // the pageable sources above are read before they change
    W.word_h[0] = Ka;
    W.word_h[1] = 0;
    W.K = Ka;
    k_bstart<<<dim3(EW_BLOCKS / 4, Ka), 256, 0, s>>>(W.t, S.col, W.V, csV, S, m, N);
    CK(cudaGetLastError());
    for (int j = 0; j < m && lock < maxit; ++j, ++lock) {
      // z = P^-1 v_j (right preconditioning), w = A z.  The block-diagonal
      // preconditioner reads v_j as (hi, lo) pairs and, for the complex64
      // operator, writes its complex64 input directly; the first pass then
      // reads the complex64 output.  A circulant block takes v_j in FP64
      // (t is free during a cycle: it is read at the cycle's start only).
      const cdf* vj = W.V + (int64_t)j * N;
      const bool bd = precond_is_block_diagonal(op, W.tr);
      const bool f32 = prec == SCABEM_C64 && bd;
      const int cur = j & 1;
      if (bd) {  // steps after the first: the previous step's last launch left P^-1 v_j
        if (j == 0)
          if (int rc = precond_apply_df(op, vj, f32 ? W.zf : nullptr, f32 ? nullptr : W.z, s, W.tr, Ka, csV, N))
            return rc;
      } else {
        k_bjoin<<<dim3(EW_BLOCKS / 4, Ka), 256, 0, s>>>(vj, csV, W.t, N);
        CK(cudaGetLastError());
        if (int rc = precond_apply(op, W.t, W.z, s, W.tr, Ka, N, N)) return rc;
      }
      if (int rc = f32 ? bapply_f32(op, W, s) : bapply(op, W.z, W.w, prec, W, s)) return rc;
      // first pass h1 = V^H w with |w|^2 in its column j + 1, w -= V h1, |w|; the
      // DGKS test; the second pass only where it asks
      const int tiles = (int)cdiv(j + 2, BG_TC);
      // row blocks of the dot products: one wave over all columns, two rows per thread at least
      const int64_t rmax = cdiv(N, 2 * BG_THREADS);
      auto row_blocks = [&](int t) { return (int)std::max<int64_t>(1, std::min<int64_t>(rmax, BG_WAVE / (t * Ka))); };
      if (j >= 2) CK(cudaStreamWaitEvent(s, W.ev[cur], 0));  // the Givens step that read this copy
      for (int pass = 0; pass < 2; ++pass) {
        const int* need = pass ? W.need[cur] : nullptr;
        cd* h = pass ? W.h2[cur] : W.h1[cur];
        const int tl = pass ? (int)cdiv(j + 1, BG_TC) : tiles;
        const dim3 gd(row_blocks(tl), tl, Ka), gv(bv_blocks(N, Ka), Ka);
        int* nd = W.done + (int64_t)W.Kcap * cdiv(m + 1, BG_TC);  // counters of the updates
        if (pass == 0 && f32)
          CK(launch_pdl(k_bdots<cx<float>>, gd, BG_THREADS, 0, s, W.V, csV, j + 1, W.wf, N, W.part, m + 1, need, 1, h,
                        m + 1, W.done));
        else if (pass == 0)
          CK(launch_pdl(k_bdots<cx<double>>, gd, BG_THREADS, 0, s, W.V, csV, j + 1, W.w, N, W.part, m + 1, need, 1, h,
                        m + 1, W.done));
        else
          CK(launch_pdl(k_bdots<cdf>, gd, BG_THREADS, 0, s, W.V, csV, j + 1, W.wdf, N, W.part, m + 1, need, 0, h, m + 1,
                        W.done));
        double* nr = W.nrm[cur] + 1 + pass;
        int* sn = pass ? nullptr : W.need[cur];
        auto update = [&](auto* in) {
          using WT = std::remove_const_t<std::remove_pointer_t<decltype(in)>>;
          auto fn = bv_short(N * Ka) ? k_bvsub_norm<WT, BV_KS_SHORT> : k_bvsub_norm<WT, BV_KS_LONG>;
          return launch_pdl(fn, gv, BG_THREADS, 0, s, W.V, csV, j + 1, h, m + 1, in, W.wdf, N, W.nparts, need, nr, sn,
                            nd);
        };
        CK(pass ? update(W.wdf) : f32 ? update(W.wf) : update(W.w));
      }
      // the Givens step on its own stream (10 us of one CTA), beside the next apply
      BState St = S;
      St.h1 = W.h1[cur];
      St.h2 = W.h2[cur];
      St.nrm = W.nrm[cur];
      St.need = W.need[cur];
      CK(cudaEventRecord(W.gs[cur], s));
      CK(cudaStreamWaitEvent(W.side, W.gs[cur], 0));
      k_givens<<<1, KBATCH * 32, 0, W.side>>>(St, j, m, Ka, tol, W.word_d);
      CK(cudaGetLastError());
      if (j + 1 < m) {
        const dim3 gp((unsigned)cdiv(3 * op->ne, 128), Ka);
        if (f32)
          CK(launch_pdl(k_bscale_precond<float>, gp, 128, 0, s, W.wdf, W.V, csV, j + 1, W.nrm[cur], W.need[cur], N,
                        op->pinv, op->eunk, op->ne, W.tr ? 1 : 0, W.zf));
        else if (bd)
          CK(launch_pdl(k_bscale_precond<double>, gp, 128, 0, s, W.wdf, W.V, csV, j + 1, W.nrm[cur], W.need[cur], N,
                        op->pinv, op->eunk, op->ne, W.tr ? 1 : 0, W.z));
        else
          k_bscale<<<dim3(EW_BLOCKS / 4, Ka), 256, 0, s>>>(W.wdf, W.V, csV, j + 1, W.nrm[cur], W.need[cur], N);
        CK(cudaGetLastError());
      }
      // the host stays one step ahead: wait for the previous step, read its word
      CK(cudaEventRecord(W.ev[cur], W.side));
      if (j > 0) {
        CK(cudaEventSynchronize(W.ev[(j - 1) & 1]));
        const int flags = reinterpret_cast<volatile int*>(W.word_h)[1];
        if (flags & FLAG_NONFINITE) {
          set_error("non-finite Krylov vector");
          return SCABEM_E_NONFINITE;
        }
        if (flags & FLAG_BREAKDOWN) {
          set_error("GMRES breakdown");
          return SCABEM_E_BREAKDOWN;
        }
        if (reinterpret_cast<volatile int*>(W.word_h)[0] == 0) {
          ++lock;
          break;
        }
      }
    }
    // the cycle's Givens steps are complete, on this stream too
    CK(cudaStreamWaitEvent(s, W.ev[0], 0));
    CK(cudaStreamWaitEvent(s, W.ev[1], 0));
    // least squares of the cycle into u (at each slot's column), then d = P^-1 u for all columns
    k_backsub<<<Ka, BS_THREADS, 0, s>>>(S, m);
    CK(cudaGetLastError());
    k_bupdate<<<dim3((unsigned)std::min<int64_t>(EW_BLOCKS, cdiv(N, 8 * BU_ROWS)), Ka), 256, 0, s>>>(W.V, csV, S, m, S.col, W.u, N);
    CK(cudaGetLastError());
    W.K = K;
    if (int rc = precond_apply(op, W.u, d, s, W.tr, K, N, N)) return rc;
    // slots that stopped inside the cycle (estimate at tol) are done; the
    // others restart from their true residual
    std::vector<int> still(Ka), nit(Ka);
    std::vector<double> e(Ka);
    CK(cudaMemcpyAsync(still.data(), S.act, sizeof(int) * Ka, cudaMemcpyDeviceToHost, s));
    CK(cudaMemcpyAsync(nit.data(), S.iters, sizeof(int) * Ka, cudaMemcpyDeviceToHost, s));
    CK(cudaMemcpyAsync(e.data(), S.est, sizeof(double) * Ka, cudaMemcpyDeviceToHost, s));
    CK(cudaStreamSynchronize(s));
    if (W.word_h[1] & FLAG_NONFINITE) {
      set_error("non-finite Krylov vector");
      return SCABEM_E_NONFINITE;
    }
    if (W.word_h[1] & FLAG_BREAKDOWN) {
      set_error("GMRES breakdown");
      return SCABEM_E_BREAKDOWN;
    }
    int nact = 0;
    for (int a = 0; a < Ka; ++a) {
      const int c = col[a];
      iters[c] += nit[a];
      est[c] = e[a];
      act[c] = still[a];
      nact += act[c];
    }
    if (nact == 0 || lock >= maxit) break;
    if (int rc = bapply(op, d, W.w, prec, W, s)) return rc;
    k_sub<<<EW_BLOCKS, 256, 0, s>>>(r, W.w, W.t, K * N);
    CK(cudaGetLastError());
    if (int rc = bnorms(W.t, W, S.nrm + 3, 4, s)) return rc;
    std::vector<double> nb(4 * K);
    CK(cudaMemcpyAsync(nb.data(), S.nrm, sizeof(double) * 4 * K, cudaMemcpyDeviceToHost, s));
    CK(cudaStreamSynchronize(s));
    for (int c = 0; c < K; ++c) {
      if (!act[c]) continue;
      beta[c] = nb[4 * c + 3];
      est[c] = beta[c] / rn0[c];
      act[c] = est[c] > tol;
    }
  }
  W.K = K;
  return SCABEM_OK;
}

// ---------------------------------------------------------------- fits
// The scans of both fits: one warp per candidate, lanes over the samples, with
// the explicit residual of each candidate's least-squares amplitudes.  Each CTA
// keeps its best candidate (ties to the lowest index); the finishing kernel
// takes the best of the CTAs and forms the results.  (One CTA with a thread
// per candidate took 0.8 ms for 601 candidates of 48 samples.)
constexpr int FIT_WARPS = 8;
constexpr int FIT_BLOCKS = 4 * 152;

__device__ __forceinline__ double wsum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ cd wsum(cd v) { return mk(wsum(v.re), wsum(v.im)); }
__device__ __forceinline__ bool better(double r, int i, double rb, int ib) {
  return i >= 0 && (r < rb || (r == rb && i < ib));
}

// E(t) = a exp(-j beta t) + c exp(j beta t): the amplitudes for one beta (a warp)
__device__ void two_wave(const cd* __restrict__ E, const double* __restrict__ tt, int npts, double beta, int lane, cd& a,
                         cd& c) {
  cd a12 = mk(0.0, 0.0), r1 = a12, r2 = a12;
  for (int i = lane; i < npts; i += 32) {
    double sn, cs;
    sincos(beta * tt[i], &sn, &cs);
    const cd ep = mk(cs, sn), em = mk(cs, -sn);
    a12 += ep * ep;   // conj(em) * ep
    r1 += ep * E[i];  // conj(em) * E
    r2 += em * E[i];  // conj(ep) * E
  }
  a12 = wsum(a12);
  r1 = wsum(r1);
  r2 = wsum(r2);
  const double n = npts;
  const double det = n * n - (a12.re * a12.re + a12.im * a12.im);
  a = (1.0 / det) * (n * r1 - a12 * r2);
  c = (1.0 / det) * (n * r2 - conj(a12) * r1);
}

// Decay-rate fit (Sec. III): least squares for E(t) = a exp(-g tau) +
// c exp(g tau), g = alpha + j beta, tau = t - tm with tm the midpoint of the
// samples (both waves decay along their direction of travel).  With
// phi1 = exp(-g tau), phi2 = exp(g tau) the normal equations are
//   [g11 g12; conj(g12) g22] [a; c] = [r1; r2],
//   g11 = sum exp(-2 alpha tau), g22 = sum exp(2 alpha tau),
//   g12 = sum exp(2 j beta tau), r1 = sum conj(phi1) E, r2 = sum conj(phi2) E.
__device__ void decay_amplitudes(const cd* __restrict__ E, const double* __restrict__ tt, int npts, double tm,
                                 double al, double be, int lane, cd& a, cd& c) {
  double g11 = 0.0, g22 = 0.0;
  cd g12 = mk(0.0, 0.0), r1 = g12, r2 = g12;
  for (int i = lane; i < npts; i += 32) {
    const double tau = tt[i] - tm;
    const double em = exp(-al * tau), ep = exp(al * tau);
    double sn, cs;
    sincos(be * tau, &sn, &cs);
    g11 += em * em;
    g22 += ep * ep;
    g12 += mk(cs * cs - sn * sn, 2.0 * sn * cs);
    r1 += mk(em * cs, em * sn) * E[i];   // conj(phi1) = exp(-alpha tau) exp(+j beta tau)
    r2 += mk(ep * cs, -ep * sn) * E[i];  // conj(phi2) = exp(alpha tau) exp(-j beta tau)
  }
  g11 = wsum(g11);
  g22 = wsum(g22);
  g12 = wsum(g12);
  r1 = wsum(r1);
  r2 = wsum(r2);
  const double det = g11 * g22 - (g12.re * g12.re + g12.im * g12.im);
  a = (1.0 / det) * (g22 * r1 - g12 * r2);
  c = (1.0 / det) * (g11 * r2 - conj(g12) * r1);
}

struct FitGrid {  // candidates alpha-major: index = ia * nb + ib; na = 0: the two-wave fit
  double alo, ahi;
  int na;
  double blo, bhi;
  int nb;
  __device__ double alpha(int i) const { return na > 1 ? alo + (ahi - alo) * (i / nb) / (na - 1) : alo; }
  __device__ double beta(int i) const {
    const int ib = na > 0 ? i - (i / nb) * nb : i;
    return nb > 1 ? blo + (bhi - blo) * ib / (nb - 1) : blo;
  }
};

__global__ void __launch_bounds__(FIT_WARPS * 32) k_fit_scan(const cd* __restrict__ E, const double* __restrict__ tt,
                                                             int npts, FitGrid F, double* __restrict__ bres,
                                                             int* __restrict__ bidx) {
  const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
  const int ncand = F.na > 0 ? F.na * F.nb : F.nb;
  const double tm = 0.5 * (tt[0] + tt[npts - 1]);
  double best = 1e300;
  int bi = -1;
  for (int ic = blockIdx.x * FIT_WARPS + wp; ic < ncand; ic += gridDim.x * FIT_WARPS) {
    const double be = F.beta(ic);
    cd a, c;
    double res = 0.0;
    if (F.na > 0) {
      const double al = F.alpha(ic);
      decay_amplitudes(E, tt, npts, tm, al, be, lane, a, c);
      for (int i = lane; i < npts; i += 32) {
        const double tau = tt[i] - tm, em = exp(-al * tau), ep = exp(al * tau);
        double sn, cs;
        sincos(be * tau, &sn, &cs);
        const cd f = a * mk(em * cs, -em * sn) + c * mk(ep * cs, ep * sn) - E[i];
        res += f.re * f.re + f.im * f.im;
      }
    } else {
      two_wave(E, tt, npts, be, lane, a, c);
      for (int i = lane; i < npts; i += 32) {
        double sn, cs;
        sincos(be * tt[i], &sn, &cs);
        const cd f = a * mk(cs, -sn) + c * mk(cs, sn) - E[i];
        res += f.re * f.re + f.im * f.im;
      }
    }
    res = wsum(res);
    if (res < best) {
      best = res;
      bi = ic;
    }
  }
  __shared__ double sr[FIT_WARPS];
  __shared__ int si[FIT_WARPS];
  if (lane == 0) {
    sr[wp] = best;
    si[wp] = bi;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < FIT_WARPS; ++w)
      if (better(sr[w], si[w], best, bi < 0 ? INT_MAX : bi)) {
        best = sr[w];
        bi = si[w];
      }
    bres[blockIdx.x] = best;
    bidx[blockIdx.x] = bi;
  }
}

// out: {Re r, Im r, beta, residual, SWR, r_swr} (two-wave fit) or {alpha, beta,
// residual, Re c/a, Im c/a, |a|} (decay fit); one warp
__global__ void k_fit_finish(const cd* __restrict__ E, const double* __restrict__ tt, int npts, FitGrid F,
                             const double* __restrict__ bres, const int* __restrict__ bidx, int nblk,
                             double* __restrict__ out) {
  const int lane = threadIdx.x;
  double r = 1e300;
  int b = -1;
  for (int i = lane; i < nblk; i += 32)
    if (better(bres[i], bidx[i], r, b < 0 ? INT_MAX : b)) {
      r = bres[i];
      b = bidx[i];
    }
  for (int o = 16; o > 0; o >>= 1) {
    const double r2 = __shfl_xor_sync(0xffffffffu, r, o);
    const int b2 = __shfl_xor_sync(0xffffffffu, b, o);
    if (better(r2, b2, r, b < 0 ? INT_MAX : b)) {
      r = r2;
      b = b2;
    }
  }
  double en = 0.0, emax = 0.0, emin = 1e300;
  for (int i = lane; i < npts; i += 32) {
    const double m2 = E[i].re * E[i].re + E[i].im * E[i].im, m = sqrt(m2);
    en += m2;
    emax = fmax(emax, m);
    emin = fmin(emin, m);
  }
  en = wsum(en);
  for (int o = 16; o > 0; o >>= 1) {
    emax = fmax(emax, __shfl_xor_sync(0xffffffffu, emax, o));
    emin = fmin(emin, __shfl_xor_sync(0xffffffffu, emin, o));
  }
  const double be = F.beta(b);
  cd a, c;
  if (F.na > 0)
    decay_amplitudes(E, tt, npts, 0.5 * (tt[0] + tt[npts - 1]), F.alpha(b), be, lane, a, c);
  else
    two_wave(E, tt, npts, be, lane, a, c);
  if (lane != 0) return;
  const cd rr = cdivd(c, a);
  if (F.na > 0) {
    out[0] = F.alpha(b);
    out[1] = be;
    out[2] = sqrt(r / en);
    out[3] = rr.re;
    out[4] = rr.im;
    out[5] = sqrt(a.re * a.re + a.im * a.im);
  } else {
    const double swr = emax / emin;
    out[0] = rr.re;
    out[1] = rr.im;
    out[2] = be;
    out[3] = sqrt(r / en);
    out[4] = swr;
    out[5] = (swr - 1.0) / (swr + 1.0);
  }
}

// scan and finish on device samples; scratch: FIT_BLOCKS doubles, then FIT_BLOCKS ints
constexpr size_t FIT_SCRATCH = FIT_BLOCKS * (sizeof(double) + sizeof(int));
int fit_dev(const cd* E, const double* tt, int npts, const FitGrid& F, void* scratch, double* out, cudaStream_t s) {
  const int64_t ncand = F.na > 0 ? (int64_t)F.na * F.nb : F.nb;
  const int nblk = (int)std::min<int64_t>(FIT_BLOCKS, cdiv(ncand, FIT_WARPS));
  double* bres = (double*)scratch;
  int* bidx = (int*)(bres + FIT_BLOCKS);
  k_fit_scan<<<nblk, FIT_WARPS * 32, 0, s>>>(E, tt, npts, F, bres, bidx);
  CK(cudaGetLastError());
  k_fit_finish<<<1, 32, 0, s>>>(E, tt, npts, F, bres, bidx, nblk, out);
  CK(cudaGetLastError());
  return SCABEM_OK;
}

}  // namespace

int rhs_impl(scabem_op* op, const scabem_source* src, int nsrc, void* b, int64_t ld, int prec, cudaStream_t s) {
  cd* val = nullptr;
  CK(cudaMalloc(&val, sizeof(cd) * op->nt * 12));
  for (int i = 0; i < nsrc; ++i) {
    const scabem_source S = src[i];
    const double k = S.side == 0 ? op->ki : op->ke;
    const double z = S.side == 0 ? op->zi : op->ze;
    k_rhs<<<(int)cdiv(op->nt * 3, 128), 128, 0, s>>>(S, op->tri, op->cX, op->qp, op->qw, op->sig64, op->nt, op->q, k,
                                                     z, val);
    CK(cudaGetLastError());
    if (prec == SCABEM_C128)
      k_rows_out<double><<<(int)cdiv(op->N, 256), 256, 0, s>>>(val, op->rowsrc, op->N, (cd*)b + (int64_t)i * ld);
    else
      k_rows_out<float><<<(int)cdiv(op->N, 256), 256, 0, s>>>(val, op->rowsrc, op->N,
                                                              (cx<float>*)b + (int64_t)i * ld);
    CK(cudaGetLastError());
  }
  CK(cudaStreamSynchronize(s));
  cudaFree(val);
  return SCABEM_OK;
}

// Gradient of lam^T (A x - b) with respect to the parameters of `basis`
// (x, lam: device complex128, N each).  g_out: host, 2 * entries doubles.
int sigma_gradient_impl(scabem_op* op, const cd* x, const cd* lam, const scabem_source* src, int nsrc,
                        const scabem_sigma* basis, double* g_out, cudaStream_t s) {
  const int64_t Q = op->Q;
  cd *hs = nullptr, *g = nullptr;
  double* dseg = nullptr;
  int64_t ng = basis->kind == SCABEM_SIGMA_PER_QPOINT ? Q
               : basis->kind == SCABEM_SIGMA_BSPLINE   ? basis->ncoef
                                                       : basis->nseg;
  int rc = SCABEM_OK;
  auto fail = [&](cudaError_t e, const char* what) { rc = cuda_fail(e, what); };
  cudaError_t e;
  if ((e = cudaMalloc(&hs, sizeof(cd) * Q)) != cudaSuccess) fail(e, "cudaMalloc");
  if (!rc && (e = cudaMalloc(&g, sizeof(cd) * (ng > 0 ? ng : 1))) != cudaSuccess) fail(e, "cudaMalloc");
  if (!rc) rc = sigma_sensitivity_op(op, x, lam, hs, s);
  for (int i = 0; !rc && i < nsrc; ++i) {
    const double k = src[i].side == 0 ? op->ki : op->ke, z = src[i].side == 0 ? op->zi : op->ze;
    k_rhs_sens<<<(int)cdiv(Q, 256), 256, 0, s>>>(src[i], op->tri, op->cX, op->qp, op->qw, op->valrow, lam, Q,
                                                 op->q, k, z, hs);
    if ((e = cudaGetLastError()) != cudaSuccess) fail(e, "k_rhs_sens");
  }
  if (!rc && basis->kind == SCABEM_SIGMA_PER_QPOINT) {
    if ((e = cudaMemcpyAsync(g_out, hs, sizeof(cd) * Q, cudaMemcpyDeviceToHost, s)) != cudaSuccess) fail(e, "copy");
  } else if (!rc && basis->kind == SCABEM_SIGMA_BSPLINE) {
    k_grad_bspline<<<basis->ncoef, GRAD_THREADS, 0, s>>>(op->qp, Q, basis->x0, basis->L, basis->axis, basis->ncoef,
                                                         hs, g);
    if ((e = cudaGetLastError()) != cudaSuccess) fail(e, "k_grad_bspline");
    if (!rc && (e = cudaMemcpyAsync(g_out, g, sizeof(cd) * ng, cudaMemcpyDeviceToHost, s)) != cudaSuccess)
      fail(e, "copy");
  } else if (!rc && ng > 0) {
    if ((e = cudaMalloc(&dseg, sizeof(double) * 6 * ng)) != cudaSuccess) fail(e, "cudaMalloc");
    if (!rc && (e = cudaMemcpyAsync(dseg, basis->seg, sizeof(double) * 6 * ng, cudaMemcpyHostToDevice, s)) !=
                   cudaSuccess)
      fail(e, "copy");
    if (!rc) {
      k_grad_monomial<<<(int)ng, GRAD_THREADS, 0, s>>>(op->qp, Q, dseg, hs, g);
      if ((e = cudaGetLastError()) != cudaSuccess) fail(e, "k_grad_monomial");
    }
    if (!rc && (e = cudaMemcpyAsync(g_out, g, sizeof(cd) * ng, cudaMemcpyDeviceToHost, s)) != cudaSuccess)
      fail(e, "copy");
  }
  if (!rc && (e = cudaStreamSynchronize(s)) != cudaSuccess) fail(e, "cudaStreamSynchronize");
  cudaFree(hs);
  cudaFree(g);
  cudaFree(dseg);
  return rc;
}

int solve_impl(scabem_op* op, const void* bv, void* xv, int nrhs, int64_t ld, const scabem_solve_opts* o,
               cudaStream_t s, scabem_solve_info* info) {
  const int64_t N = op->N;
  const int m = o->restart;
  const int prec = o->prec;
  const bool tr = o->transpose != 0;
  if (nrhs == 0) return SCABEM_OK;
  const int KB = nrhs < KBATCH ? nrhs : KBATCH;
  if (KB > 1 && !tr) {
    if (int rc = ensure_batch<double>(op, KB, s)) return rc;
    if (prec == SCABEM_C64)
      if (int rc = ensure_batch<float>(op, KB, s)) return rc;
  }
  BWork W;
  W.tr = tr;
  if (int rc = W.init(KB, m, N, prec == SCABEM_C64, s)) return rc;
  cd *B = nullptr, *X = nullptr, *R = nullptr, *D = nullptr;
  if (int rc = W.get(&B, KB * N)) return rc;
  if (int rc = W.get(&X, KB * N)) return rc;
  if (int rc = W.get(&R, KB * N)) return rc;
  if (int rc = W.get(&D, KB * N)) return rc;
  const int outer = o->max_refine > 0 ? o->max_refine : 1;
  const double tol_out = o->refine_tol > 0 ? o->refine_tol : o->tol;
  int status = SCABEM_OK;
  for (int c0 = 0; c0 < nrhs; c0 += KB) {
    const int k = nrhs - c0 < KB ? nrhs - c0 : KB;
    W.K = k;
    for (int c = 0; c < k; ++c) {
      CK(cudaMemcpyAsync(B + c * N, (const cd*)bv + (c0 + c) * ld, sizeof(cd) * N, cudaMemcpyDeviceToDevice, s));
      CK(cudaMemcpyAsync(X + c * N, (const cd*)xv + (c0 + c) * ld, sizeof(cd) * N, cudaMemcpyDeviceToDevice, s));
    }
    std::vector<double> bn(k), rn(k), relres(k, 0.0), est(k, 0.0);
    if (int rc = bnorms(B, W, W.S.rn0, 1, s)) return rc;
    CK(cudaMemcpyAsync(bn.data(), W.S.rn0, sizeof(double) * k, cudaMemcpyDeviceToHost, s));
    std::vector<int> iters(k, 0), refs(k, 0), st(k, SCABEM_E_NOCONV);
    std::vector<char> done(k, 0), use(k, 0);
    for (int it = 0; it <= outer; ++it) {
      // FP64 residual r = b - A x with the complex128 operator
      if (int rc = bapply(op, X, W.w, SCABEM_C128, W, s)) return rc;
      k_sub<<<EW_BLOCKS, 256, 0, s>>>(B, W.w, R, k * N);
      CK(cudaGetLastError());
      if (int rc = bnorms(R, W, W.S.nrm + 3, 4, s)) return rc;
      std::vector<double> nb(4 * k);
      CK(cudaMemcpyAsync(nb.data(), W.S.nrm, sizeof(double) * 4 * k, cudaMemcpyDeviceToHost, s));
      CK(cudaStreamSynchronize(s));
      int left = 0;
      for (int c = 0; c < k; ++c) {
        if (done[c]) continue;
        relres[c] = bn[c] > 0 ? nb[4 * c + 3] / bn[c] : 0.0;
        if (!std::isfinite(relres[c])) {
          st[c] = SCABEM_E_NONFINITE;
          done[c] = 1;
        } else if (relres[c] <= tol_out) {
          st[c] = SCABEM_OK;
          done[c] = 1;
        } else if (it == outer || iters[c] >= o->maxit) {
          done[c] = 1;
        }
        use[c] = !done[c];
        left += use[c];
      }
      if (left == 0) break;
      int budget = 0;
      for (int c = 0; c < k; ++c)
        if (use[c]) budget = std::max(budget, o->maxit - iters[c]);
      if (int rc = gmres_batch(op, R, D, use, prec, o->tol, budget, W, s, iters, est)) return rc;
      k_add<<<EW_BLOCKS, 256, 0, s>>>(X, D, k * N);
      CK(cudaGetLastError());
      for (int c = 0; c < k; ++c) refs[c] += use[c];
    }
    for (int c = 0; c < k; ++c)
      CK(cudaMemcpyAsync((cd*)xv + (c0 + c) * ld, X + c * N, sizeof(cd) * N, cudaMemcpyDeviceToDevice, s));
    for (int c = 0; c < k; ++c) {
      if (info) {
        info[c0 + c].iters = iters[c];
        info[c0 + c].refinements = refs[c];
        info[c0 + c].relres = relres[c];
        info[c0 + c].status = st[c];
      }
      if (st[c] != SCABEM_OK && status == SCABEM_OK) status = st[c];
    }
  }
  CK(cudaStreamSynchronize(s));
  if (status != SCABEM_OK) set_error("solver did not reach the requested residual");
  return status;
}

// E (and H unless null) of one current set of x at device points
static int fields_dev(scabem_op* op, const cd* x, const double* dpts, int npts, int side, const scabem_source* inc,
                      FieldScratch& W, cd* dE, cd* dH, cudaStream_t s) {
  if (int rc = compute_summ<double>(op, x, op->d.summ, s)) return rc;
  const double k = side ? op->ke : op->ki, z = side ? op->ze : op->zi;
  k_point_currents<<<(int)cdiv(op->Q, 128), 128, 0, s>>>(op->d.summ, op->tri, op->qp, op->qw, op->Q, op->q, k, z, side,
                                                         W.pc);
  CK(cudaGetLastError());
  const dim3 g((unsigned)cdiv(npts, FP_PTS), W.nsl);
  if (dH)
    k_point_fields<true><<<g, FP_THREADS, 0, s>>>(W.pc, op->Q, dpts, npts, k, z, W.part);
  else
    k_point_fields<false><<<g, FP_THREADS, 0, s>>>(W.pc, op->Q, dpts, npts, k, z, W.part);
  CK(cudaGetLastError());
  scabem_source S{};
  if (inc) S = *inc;
  k_point_finish<<<(int)cdiv(npts, 64), 64, 0, s>>>(W.part, W.nsl, dpts, npts, k, z, S, inc && side == 0 ? 1 : 0, dE, dH);
  CK(cudaGetLastError());
  return SCABEM_OK;
}

int fields_impl(scabem_op* op, const void* x, int nrhs, int64_t ld, const double* pts, int npts,
                const scabem_source* inc, double* E, cudaStream_t s) {
  double* dpts = nullptr;
  cd* dE = nullptr;
  FieldScratch W;
  if (int rc = W.init(op, npts)) return rc;
  CK(cudaMalloc(&dpts, sizeof(double) * 3 * npts));
  CK(cudaMalloc(&dE, sizeof(cd) * 3 * npts));
  CK(cudaMemcpyAsync(dpts, pts, sizeof(double) * 3 * npts, cudaMemcpyHostToDevice, s));
  for (int col = 0; col < nrhs; ++col) {
    int rc = fields_dev(op, (const cd*)x + (int64_t)col * ld, dpts, npts, 0, inc, W, dE, nullptr, s);
    if (rc) return rc;
    CK(cudaMemcpyAsync(E + (int64_t)col * 6 * npts, dE, sizeof(cd) * 3 * npts, cudaMemcpyDeviceToHost, s));
  }
  CK(cudaStreamSynchronize(s));
  cudaFree(dpts);
  cudaFree(dE);
  return SCABEM_OK;
}

// E and H of one current set at host points, per right-hand side.
int fields_eh_impl(scabem_op* op, const void* x, int nrhs, int64_t ld, const double* pts, int npts, int side,
                   const scabem_source* inc, double* E, double* H, cudaStream_t s) {
  double* dpts = nullptr;
  cd* dE = nullptr;
  FieldScratch W;
  if (int rc = W.init(op, npts)) return rc;
  CK(cudaMalloc(&dpts, sizeof(double) * 3 * npts));
  CK(cudaMalloc(&dE, sizeof(cd) * 6 * npts));
  CK(cudaMemcpyAsync(dpts, pts, sizeof(double) * 3 * npts, cudaMemcpyHostToDevice, s));
  for (int col = 0; col < nrhs; ++col) {
    int rc = fields_dev(op, (const cd*)x + (int64_t)col * ld, dpts, npts, side, inc, W, dE, dE + 3 * npts, s);
    if (rc) return rc;
    CK(cudaMemcpyAsync(E + (int64_t)col * 6 * npts, dE, sizeof(cd) * 3 * npts, cudaMemcpyDeviceToHost, s));
    CK(cudaMemcpyAsync(H + (int64_t)col * 6 * npts, dE + 3 * npts, sizeof(cd) * 3 * npts, cudaMemcpyDeviceToHost, s));
  }
  CK(cudaStreamSynchronize(s));
  cudaFree(dpts);
  cudaFree(dE);
  return SCABEM_OK;
}

namespace {
// Gauss-Legendre rule on [-1, 1]: the roots of P_n by Newton's method from
// the estimate cos(pi (i - 1/4) / (n + 1/2)), weights 2 / ((1 - x^2) P_n'(x)^2).
void gauss_legendre(int n, std::vector<double>& x, std::vector<double>& w) {
  x.assign(n, 0.0);
  w.assign(n, 0.0);
  for (int i = 0; i < n; ++i) {
    double t = std::cos(M_PI * (i + 0.75) / (n + 0.5)), dp = 1.0;
    for (int it = 0; it < 100; ++it) {
      double p0 = 1.0, p1 = t;
      for (int m = 2; m <= n; ++m) {
        const double p2 = ((2.0 * m - 1.0) * t * p1 - (m - 1.0) * p0) / m;
        p0 = p1;
        p1 = p2;
      }
      dp = n * (t * p1 - p0) / (t * t - 1.0);  // p1 = P_n(t), p0 = P_{n-1}(t)
      const double dt = p1 / dp;
      t -= dt;
      if (std::fabs(dt) < 1e-16) break;
    }
    x[i] = t;
    w[i] = 2.0 / ((1.0 - t * t) * dp * dp);
  }
}

struct QPoint {
  double y, z, w;
};
// n x n Gauss-Legendre points of the rectangle [y0, y1] x [z0, z1]
void gl_rect(double y0, double y1, double z0, double z1, int n, std::vector<QPoint>& out) {
  std::vector<double> u, wu;
  gauss_legendre(n, u, wu);
  for (int i = 0; i < n; ++i)
    for (int j = 0; j < n; ++j)
      out.push_back({0.5 * (y1 - y0) * u[i] + 0.5 * (y1 + y0), 0.5 * (z1 - z0) * u[j] + 0.5 * (z1 + z0),
                     wu[i] * wu[j] * 0.25 * (y1 - y0) * (z1 - z0)});
}
}  // namespace

// Decay rate by Poynting's theorem (Sec. III-B) at the cross-section
// x = xc of a guide along x centred on y = z = 0.
int poynting_impl(scabem_op* op, const void* x, int nrhs, int64_t ld, const scabem_poynting* P,
                  const scabem_source* inc, double* out, cudaStream_t s) {
  const int n = P->n;
  const double hy = P->core[0], hz = P->core[1], Y = P->box[0], Z = P->box[1];
  // cross-section: the core (interior field) and the eight rectangles around it (exterior field)
  std::vector<QPoint> core, outer;
  gl_rect(-hy, hy, -hz, hz, n, core);
  const double ys[4] = {-Y, -hy, hy, Y}, zs[4] = {-Z, -hz, hz, Z};
  for (int a = 0; a < 3; ++a)
    for (int b = 0; b < 3; ++b)
      if (!(a == 1 && b == 1)) gl_rect(ys[a], ys[a + 1], zs[b], zs[b + 1], n, outer);
  // outer boundary: lines y = +-Y (z in [-Z, Z]) and z = +-Z (y in [-Y, Y]), 2n points each;
  // weight = Gauss weight x half length x the sign of the outward normal
  std::vector<double> u, wu;
  gauss_legendre(2 * n, u, wu);
  std::vector<QPoint> side;
  std::vector<int> side_comp;
  for (int ax = 0; ax < 2; ++ax)
    for (int sg = 1; sg >= -1; sg -= 2) {
      const double half = ax == 0 ? Z : Y;
      for (int i = 0; i < 2 * n; ++i) {
        const double l = u[i] * half;
        side.push_back(ax == 0 ? QPoint{sg * Y, l, wu[i] * half * sg} : QPoint{l, sg * Z, wu[i] * half * sg});
        side_comp.push_back(1 + ax);
      }
    }
  const int ni = (int)core.size(), ne = (int)(outer.size() + side.size());
  std::vector<double> pi(3 * ni), pe(3 * ne);
  for (int i = 0; i < ni; ++i) {
    pi[3 * i] = P->xc;
    pi[3 * i + 1] = core[i].y;
    pi[3 * i + 2] = core[i].z;
  }
  for (int i = 0; i < ne; ++i) {
    const QPoint& qq = i < (int)outer.size() ? outer[i] : side[i - outer.size()];
    pe[3 * i] = P->xc;
    pe[3 * i + 1] = qq.y;
    pe[3 * i + 2] = qq.z;
  }
  std::vector<double> Ei(6 * ni), Hi(6 * ni), Ee(6 * ne), He(6 * ne);
  const int nb = 152;
  double* part = nullptr;
  CK(cudaMalloc(&part, sizeof(double) * nb));
  std::vector<double> hp(nb);
  for (int col = 0; col < nrhs; ++col) {
    const void* xcol = (const cd*)x + (int64_t)col * ld;
    int rc = fields_eh_impl(op, xcol, 1, ld, pi.data(), ni, 0, inc, Ei.data(), Hi.data(), s);
    if (rc) return rc;
    rc = fields_eh_impl(op, xcol, 1, ld, pe.data(), ne, 1, nullptr, Ee.data(), He.data(), s);
    if (rc) return rc;
    auto sx = [](const double* E, const double* H) {  // Re (E x H*) . x
      return (E[2] * H[4] + E[3] * H[5]) - (E[4] * H[2] + E[5] * H[3]);
    };
    double flux = 0.0, sidef = 0.0;
    for (int i = 0; i < ni; ++i) flux += core[i].w * sx(&Ei[6 * i], &Hi[6 * i]);
    for (int i = 0; i < (int)outer.size(); ++i) flux += outer[i].w * sx(&Ee[6 * i], &He[6 * i]);
    for (int i = 0; i < (int)side.size(); ++i) {
      const int j = (int)outer.size() + i;
      const double* E = &Ee[6 * j];
      const double* H = &He[6 * j];
      // Re (E x H*) component 1 (y) or 2 (z)
      const int c = side_comp[i], c1 = (c + 1) % 3, c2 = (c + 2) % 3;
      const double S = (E[2 * c1] * H[2 * c2] + E[2 * c1 + 1] * H[2 * c2 + 1]) -
                       (E[2 * c2] * H[2 * c1] + E[2 * c2 + 1] * H[2 * c1 + 1]);
      sidef += side[i].w * S;
    }
    // the sheet's loss around the perimeter: the band |x - xc| < slab over its width
    rc = compute_summ<double>(op, (const cd*)xcol, op->d.summ, s);
    if (rc) return rc;
    k_band_loss<<<nb, 256, 0, s>>>(op->d.summ, op->tri, op->qp, op->qw, op->sig64, op->Q, op->q, 0, P->xc, P->slab,
                                   part);
    CK(cudaGetLastError());
    CK(cudaMemcpyAsync(hp.data(), part, sizeof(double) * nb, cudaMemcpyDeviceToHost, s));
    CK(cudaStreamSynchronize(s));
    double loss = 0.0;
    for (double v : hp) loss += v;
    loss /= 2.0 * P->slab;
    double* o = out + 4 * col;
    o[0] = (loss + sidef) / (2.0 * flux);
    o[1] = loss;
    o[2] = sidef;
    o[3] = flux;
  }
  cudaFree(part);
  return SCABEM_OK;
}

int reflection_impl(scabem_op* op, const void* x, int nrhs, int64_t ld, const scabem_probe* pr,
                    const scabem_source* inc, double* out, cudaStream_t s) {
  const int npts = pr->npts;
  std::vector<double> pts(3 * npts), tt(npts);
  for (int i = 0; i < npts; ++i) {
    const double t = npts > 1 ? pr->t0 + (pr->t1 - pr->t0) * i / (npts - 1) : pr->t0;
    tt[i] = t;
    for (int c = 0; c < 3; ++c) pts[3 * i + c] = pr->p0[c] + (c == pr->axis ? t : 0.0);
  }
  double *dpts = nullptr, *dtt = nullptr, *dout = nullptr;
  cd *dE = nullptr, *dc = nullptr;
  CK(cudaMalloc(&dpts, sizeof(double) * 3 * npts));
  CK(cudaMalloc(&dtt, sizeof(double) * npts));
  CK(cudaMalloc(&dE, sizeof(cd) * 3 * npts));
  CK(cudaMalloc(&dc, sizeof(cd) * npts));
  CK(cudaMalloc(&dout, sizeof(double) * 6 + FIT_SCRATCH));
  FieldScratch W;
  if (int rc = W.init(op, npts)) return rc;
  CK(cudaMemcpyAsync(dpts, pts.data(), sizeof(double) * 3 * npts, cudaMemcpyHostToDevice, s));
  CK(cudaMemcpyAsync(dtt, tt.data(), sizeof(double) * npts, cudaMemcpyHostToDevice, s));
  for (int col = 0; col < nrhs; ++col) {
    int rc = fields_dev(op, (const cd*)x + (int64_t)col * ld, dpts, npts, 0, inc, W, dE, nullptr, s);
    if (rc) return rc;
    CK(cudaMemcpy2DAsync(dc, sizeof(cd), (const char*)dE + sizeof(cd) * pr->comp, 3 * sizeof(cd), sizeof(cd), npts,
                         cudaMemcpyDeviceToDevice, s));
    const FitGrid F{0.0, 0.0, 0, pr->beta_lo, pr->beta_hi, pr->nbeta};
    if ((rc = fit_dev(dc, dtt, npts, F, dout + 6, dout, s))) return rc;
    CK(cudaMemcpyAsync(out + 6 * col, dout, sizeof(double) * 6, cudaMemcpyDeviceToHost, s));
  }
  CK(cudaStreamSynchronize(s));
  cudaFree(dpts);
  cudaFree(dtt);
  cudaFree(dE);
  cudaFree(dc);
  cudaFree(dout);
  return SCABEM_OK;
}

// Decay-rate fit of given samples (host t, host complex128 E).
int decay_fit_impl(const double* t, const double* E, int npts, double alo, double ahi, int na, double blo, double bhi,
                   int nb, double* out, cudaStream_t s) {
  double *dt = nullptr, *dout = nullptr;
  cd* dE = nullptr;
  CK(cudaMalloc(&dt, sizeof(double) * npts));
  CK(cudaMalloc(&dE, sizeof(cd) * npts));
  CK(cudaMalloc(&dout, sizeof(double) * 6 + FIT_SCRATCH));
  CK(cudaMemcpyAsync(dt, t, sizeof(double) * npts, cudaMemcpyHostToDevice, s));
  CK(cudaMemcpyAsync(dE, E, sizeof(cd) * npts, cudaMemcpyHostToDevice, s));
  if (int rc = fit_dev(dE, dt, npts, FitGrid{alo, ahi, na, blo, bhi, nb}, dout + 6, dout, s)) return rc;
  CK(cudaMemcpyAsync(out, dout, sizeof(double) * 6, cudaMemcpyDeviceToHost, s));
  CK(cudaStreamSynchronize(s));
  cudaFree(dt);
  cudaFree(dE);
  cudaFree(dout);
  return SCABEM_OK;
}

// Decay rate along a probe line: the total interior field component there
// (as for the reflection), then the decay-rate fit.
int decay_rate_impl(scabem_op* op, const void* x, int nrhs, int64_t ld, const scabem_probe* pr, double alo,
                    double ahi, int na, const scabem_source* inc, double* out, cudaStream_t s) {
  const int npts = pr->npts;
  std::vector<double> pts(3 * npts), tt(npts);
  for (int i = 0; i < npts; ++i) {
    const double t = npts > 1 ? pr->t0 + (pr->t1 - pr->t0) * i / (npts - 1) : pr->t0;
    tt[i] = t;
    for (int c = 0; c < 3; ++c) pts[3 * i + c] = pr->p0[c] + (c == pr->axis ? t : 0.0);
  }
  double *dpts = nullptr, *dtt = nullptr, *dout = nullptr;
  cd *dE = nullptr, *dc = nullptr;
  CK(cudaMalloc(&dpts, sizeof(double) * 3 * npts));
  CK(cudaMalloc(&dtt, sizeof(double) * npts));
  CK(cudaMalloc(&dE, sizeof(cd) * 3 * npts));
  CK(cudaMalloc(&dc, sizeof(cd) * npts));
  CK(cudaMalloc(&dout, sizeof(double) * 6 + FIT_SCRATCH));
  FieldScratch W;
  if (int rc = W.init(op, npts)) return rc;
  CK(cudaMemcpyAsync(dpts, pts.data(), sizeof(double) * 3 * npts, cudaMemcpyHostToDevice, s));
  CK(cudaMemcpyAsync(dtt, tt.data(), sizeof(double) * npts, cudaMemcpyHostToDevice, s));
  for (int col = 0; col < nrhs; ++col) {
    int rc = fields_dev(op, (const cd*)x + (int64_t)col * ld, dpts, npts, 0, inc, W, dE, nullptr, s);
    if (rc) return rc;
    CK(cudaMemcpy2DAsync(dc, sizeof(cd), (const char*)dE + sizeof(cd) * pr->comp, 3 * sizeof(cd), sizeof(cd), npts,
                         cudaMemcpyDeviceToDevice, s));
    const FitGrid F{alo, ahi, na, pr->beta_lo, pr->beta_hi, pr->nbeta};
    if ((rc = fit_dev(dc, dtt, npts, F, dout + 6, dout, s))) return rc;
    CK(cudaMemcpyAsync(out + 6 * col, dout, sizeof(double) * 6, cudaMemcpyDeviceToHost, s));
  }
  CK(cudaStreamSynchronize(s));
  cudaFree(dpts);
  cudaFree(dtt);
  cudaFree(dE);
  cudaFree(dc);
  cudaFree(dout);
  return SCABEM_OK;
}

// ---------------------------------------------------------------- right-hand side without allocation
// Some callers cannot allocate device memory while they run: code that lives
// inside another framework's memory pool (which has already reserved the
// device), real-time loops that cannot afford the device-wide
// synchronisation a cudaFree implies, and services that must not meet an
// out-of-memory error halfway through a run.  scabem_rhs allocates its
// per-call row-value scratch; scabem_rhs_noalloc runs the same two kernels
// with that scratch in the fixed device array below instead.
constexpr int64_t NOALLOC_MAX_TRIANGLES = 32768;
// nt * 3 local edges * 4 row types complex128 values: 6 MiB, held by every
// GPU that loads this library until the process exits.
static __device__ __align__(256) cd g_rhs_scratch[NOALLOC_MAX_TRIANGLES * 12];

namespace {
constexpr int NOALLOC_MAX_DEVICES = 256;
std::mutex g_noalloc_mu;
cd* g_noalloc_ptr[NOALLOC_MAX_DEVICES] = {};

// Device address of the scratch array on the current device, looked up once
// per device (the array's name is only a host-side stand-in in host code).
int noalloc_scratch(int dev, cd** out) {
  if (dev < 0 || dev >= NOALLOC_MAX_DEVICES) {
    set_error("scabem_rhs_noalloc: device ordinal out of range");
    return SCABEM_E_DEVICE;
  }
  std::lock_guard<std::mutex> lock(g_noalloc_mu);
  if (!g_noalloc_ptr[dev]) {
    void* p = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&p, g_rhs_scratch);
    if (e != cudaSuccess) return cuda_fail(e, "cudaGetSymbolAddress(g_rhs_scratch)");
    g_noalloc_ptr[dev] = static_cast<cd*>(p);
  }
  *out = g_noalloc_ptr[dev];
  return SCABEM_OK;
}
}  // namespace

extern "C" int scabem_rhs_noalloc(scabem_op_t op, const scabem_source* src, int32_t nsrc, void* b, int64_t ld,
                                  int32_t prec, void* stream) {
  if (!op || !src || !b || nsrc < 0 || ld < op->N || (prec != SCABEM_C64 && prec != SCABEM_C128)) {
    set_error("scabem_rhs_noalloc: bad argument");
    return SCABEM_E_ARG;
  }
  if (op->nt > NOALLOC_MAX_TRIANGLES) {
    set_error("scabem_rhs_noalloc: mesh has " + std::to_string(op->nt) + " triangles; the fixed scratch holds at most " +
              std::to_string(NOALLOC_MAX_TRIANGLES) + " (use scabem_rhs)");
    return SCABEM_E_ARG;
  }
  for (int i = 0; i < nsrc; ++i)
    if (src[i].kind < 0 || src[i].kind > 2 || src[i].side < 0 || src[i].side > 1) {
      set_error("scabem_rhs_noalloc: source kind must be 0..2 and side 0..1");
      return SCABEM_E_ARG;
    }
  int dev = 0;
  CK(cudaGetDevice(&dev));
  if (dev != op->device) {
    set_error("scabem_rhs_noalloc: the operator's device is not the current device");
    return SCABEM_E_ARG;
  }
  cudaPointerAttributes at;
  if (cudaPointerGetAttributes(&at, b) != cudaSuccess ||
      (at.type != cudaMemoryTypeDevice && at.type != cudaMemoryTypeManaged)) {
    cudaGetLastError();
    set_error("scabem_rhs_noalloc: b must be device memory (host buffers would need staging)");
    return SCABEM_E_ARG;
  }
  cd* val = nullptr;
  int rc = noalloc_scratch(dev, &val);
  if (rc) return rc;
  cudaStream_t s = (cudaStream_t)stream;
  for (int i = 0; i < nsrc; ++i) {
    const scabem_source S = src[i];
    const double k = S.side == 0 ? op->ki : op->ke;
    const double z = S.side == 0 ? op->zi : op->ze;
    // k_rhs writes all nt*12 entries that k_rows_out reads, so the previous
    // call's contents never leak into this one.
    k_rhs<<<(int)cdiv(op->nt * 3, 128), 128, 0, s>>>(S, op->tri, op->cX, op->qp, op->qw, op->sig64, op->nt, op->q, k,
                                                     z, val);
    CK(cudaGetLastError());
    if (prec == SCABEM_C128)
      k_rows_out<double><<<(int)cdiv(op->N, 256), 256, 0, s>>>(val, op->rowsrc, op->N, (cd*)b + (int64_t)i * ld);
    else
      k_rows_out<float><<<(int)cdiv(op->N, 256), 256, 0, s>>>(val, op->rowsrc, op->N,
                                                              (cx<float>*)b + (int64_t)i * ld);
    CK(cudaGetLastError());
  }
  return SCABEM_OK;
}
