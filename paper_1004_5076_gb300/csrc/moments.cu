// Set-up of the triangle moments of the grid stencils.
//
// The RWG currents and test functions are linear on a triangle, so the grid
// sees a triangle only through quadrature moments of the stencils.  For
// every grid point g that a stencil of one of the triangle's quadrature
// points covers, with W_a(g) the stencil weight of point a, w_a its
// quadrature weight and rel_a = r_a - centroid:
//
//   wA = { m0, m1 }:   m0 = sum_a w_a W_a,       m1 = sum_a w_a W_a rel_a
//   wB, wC = { n0, c1 }: n0 = sum_a w_a grad W_a, c1 = sum_a w_a rel_a x grad W_a
//
// Projection: a current J = a (r - c) - beta puts a m1 - beta m0 and the
// charge 2 a m0 on g.  Testing: <V>, <rel . V> of an interpolated potential
// V are sums of m0 V(g) and m1 . V(g); <curl V> and <rel . curl V> of n0 x V(g)
// and c1 . V(g).  A triangle covers about 48 points where its 6 x 27 stencil
// entries overlap, and each entry serves all fields at once.
//
// The conductivity-weighted rows (Eqs. 13, 14) use the same moments with
// sigma_a w_a in place of w_a, on triangles with an absorber edge only:
//   sA = { s0, t0 }:  sum w, sum w grad W        sB = { s1, g1 }: sum w W rel, sum w rel . grad W
//   sC = { k1 }:      sum w rel x grad W
//   sD, sE = the same as sB, sC with n x rel in place of rel.
// They are formed again on every scabem_set_sigma.
#include <cuda_runtime.h>

#include <algorithm>
#include <vector>

#include "common.cuh"

namespace {

__device__ __forceinline__ bool covers(const int32_t* __restrict__ base, int64_t Qi, int i0, int i1, int i2, int p) {
  const int a = i0 - base[3 * Qi], b = i1 - base[3 * Qi + 1], c = i2 - base[3 * Qi + 2];
  return (unsigned)a < (unsigned)p && (unsigned)b < (unsigned)p && (unsigned)c < (unsigned)p;
}

// The grid points of each triangle, one warp per triangle, in (point, slot)
// order of the first stencil that covers them; cnt != null only counts.
__global__ void __launch_bounds__(128) k_tri_points(const int32_t* __restrict__ base, int64_t nt, int q, int p, int n1,
                                                    int n2, int32_t* __restrict__ cnt, const int32_t* __restrict__ toff,
                                                    int32_t* __restrict__ tgi) {
  const int64_t t = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  if (t >= nt) return;
  const int lane = threadIdx.x & 31, p2 = p * p, p3 = p2 * p;
  int n = 0;
  for (int b = 0; b < q * p3; b += 32) {
    const int u = b + lane;
    bool keep = u < q * p3;
    int i0 = 0, i1 = 0, i2 = 0;
    if (keep) {
      const int a = u / p3, sl = u - a * p3;
      const int64_t Qi = t * q + a;
      i0 = base[3 * Qi] + sl / p2;
      i1 = base[3 * Qi + 1] + (sl / p) % p;
      i2 = base[3 * Qi + 2] + sl % p;
      for (int c = 0; c < a && keep; ++c) keep = !covers(base, t * q + c, i0, i1, i2, p);
    }
    const unsigned m = __ballot_sync(0xffffffffu, keep);
    if (keep && !cnt) tgi[toff[t] + n + __popc(m & ((1u << lane) - 1))] = (i0 * n1 + i1) * n2 + i2;
    n += __popc(m);
  }
  if (cnt && lane == 0) cnt[t] = n;
}

template <typename R>
struct Tables {
  R *A, *B, *C;
};
template <typename R>
struct SigTables {
  R *A, *B, *C, *D, *E;
};

template <typename R>
__device__ __forceinline__ void put4(R* p, int64_t e, const double* v) {
  for (int c = 0; c < 4; ++c) p[4 * e + c] = (R)v[c];
}

// Weights of every (triangle, grid point) entry, one warp per triangle, lanes
// over its entries; sums over the quadrature points in FP64.
__global__ void __launch_bounds__(128)
    k_tri_weights(const int32_t* __restrict__ toff, const int32_t* __restrict__ tgi, const int32_t* __restrict__ base,
                  const double* __restrict__ L, const double* __restrict__ dL, const double* __restrict__ tp, int64_t nt,
                  int q, int p, int n1, int n2, Tables<double> d, Tables<float> f) {
  const int64_t t = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  if (t >= nt) return;
  for (int64_t e = toff[t] + (threadIdx.x & 31); e < toff[t + 1]; e += 32) {
    const int g = tgi[e], i2 = g % n2, i1 = (g / n2) % n1, i0 = g / (n1 * n2);
    double A[4] = {0, 0, 0, 0}, B[4] = {0, 0, 0, 0}, c1[3] = {0, 0, 0};
    for (int a = 0; a < q; ++a) {
      const int64_t Qi = t * q + a;
      if (!covers(base, Qi, i0, i1, i2, p)) continue;
      const int x = i0 - base[3 * Qi], y = i1 - base[3 * Qi + 1], z = i2 - base[3 * Qi + 2];
      const double lx = L[(3 * Qi + 0) * p + x], ly = L[(3 * Qi + 1) * p + y], lz = L[(3 * Qi + 2) * p + z];
      const double dx = dL[(3 * Qi + 0) * p + x], dy = dL[(3 * Qi + 1) * p + y], dz = dL[(3 * Qi + 2) * p + z];
      const double* r = tp + 16 * Qi;
      const double w = r[3], W = w * lx * ly * lz;
      const double G[3] = {w * dx * ly * lz, w * lx * dy * lz, w * lx * ly * dz};
      A[0] += W;
      for (int c = 0; c < 3; ++c) {
        A[1 + c] += W * r[c];
        B[c] += G[c];
      }
      c1[0] += r[1] * G[2] - r[2] * G[1];
      c1[1] += r[2] * G[0] - r[0] * G[2];
      c1[2] += r[0] * G[1] - r[1] * G[0];
    }
    B[3] = c1[0];
    if (d.A) {
      put4(d.A, e, A);
      put4(d.B, e, B);
      d.C[2 * e] = c1[1];
      d.C[2 * e + 1] = c1[2];
    }
    if (f.A) {
      put4(f.A, e, A);
      put4(f.B, e, B);
      f.C[2 * e] = (float)c1[1];
      f.C[2 * e + 1] = (float)c1[2];
    }
  }
}

// The conductivity-weighted weights, for the triangles with an absorber edge
__global__ void __launch_bounds__(128)
    k_tri_sigma(const int32_t* __restrict__ soff, const int32_t* __restrict__ toff, const int32_t* __restrict__ tgi,
                const int32_t* __restrict__ base, const double* __restrict__ L, const double* __restrict__ dL,
                const double* __restrict__ tp, const double* __restrict__ sig, const double* __restrict__ tri,
                int64_t nt, int q, int p, int n1, int n2, SigTables<double> d, SigTables<float> f) {
  const int64_t t = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  if (t >= nt || soff[t] < 0) return;
  const double* n = tri + 16 * t + 12;
  const int len = toff[t + 1] - toff[t];
  for (int j = threadIdx.x & 31; j < len; j += 32) {
    const int64_t e = soff[t] + j;
    const int g = tgi[toff[t] + j], i2 = g % n2, i1 = (g / n2) % n1, i0 = g / (n1 * n2);
    double A[4] = {0, 0, 0, 0}, B[4] = {0, 0, 0, 0}, C[4] = {0, 0, 0, 0}, D[4] = {0, 0, 0, 0}, E[4] = {0, 0, 0, 0};
    for (int a = 0; a < q; ++a) {
      const int64_t Qi = t * q + a;
      if (!covers(base, Qi, i0, i1, i2, p)) continue;
      const int x = i0 - base[3 * Qi], y = i1 - base[3 * Qi + 1], z = i2 - base[3 * Qi + 2];
      const double lx = L[(3 * Qi + 0) * p + x], ly = L[(3 * Qi + 1) * p + y], lz = L[(3 * Qi + 2) * p + z];
      const double dx = dL[(3 * Qi + 0) * p + x], dy = dL[(3 * Qi + 1) * p + y], dz = dL[(3 * Qi + 2) * p + z];
      const double* r = tp + 16 * Qi;
      const double w = r[3] * sig[Qi], W = w * lx * ly * lz;
      const double G[3] = {w * dx * ly * lz, w * lx * dy * lz, w * lx * ly * dz};
      const double m[3] = {n[1] * r[2] - n[2] * r[1], n[2] * r[0] - n[0] * r[2], n[0] * r[1] - n[1] * r[0]};
      A[0] += W;
      for (int c = 0; c < 3; ++c) {
        const int c1 = (c + 1) % 3, c2 = (c + 2) % 3;
        A[1 + c] += G[c];
        B[c] += W * r[c];
        B[3] += r[c] * G[c];
        C[c] += r[c1] * G[c2] - r[c2] * G[c1];
        D[c] += W * m[c];
        D[3] += m[c] * G[c];
        E[c] += m[c1] * G[c2] - m[c2] * G[c1];
      }
    }
    if (d.A) {
      put4(d.A, e, A);
      put4(d.B, e, B);
      put4(d.C, e, C);
      put4(d.D, e, D);
      put4(d.E, e, E);
    }
    if (f.A) {
      put4(f.A, e, A);
      put4(f.B, e, B);
      put4(f.C, e, C);
      put4(f.D, e, D);
      put4(f.E, e, E);
    }
  }
}

// geo[t] = {cX_k, v_k - c} for k < 3, then the normal
__global__ void k_tri_geo(const double* __restrict__ tri, const double* __restrict__ cX, int64_t nt,
                          double* __restrict__ gd, float* __restrict__ gf) {
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t >= nt) return;
  const double* g = tri + 16 * t;
  double v[16];
  for (int k = 0; k < 3; ++k) {
    v[4 * k] = cX[3 * t + k];
    for (int c = 0; c < 3; ++c) v[4 * k + 1 + c] = g[3 * k + c] - g[9 + c];
  }
  for (int c = 0; c < 3; ++c) v[12 + c] = g[12 + c];
  v[15] = 0.0;
  for (int i = 0; i < 16; ++i) {
    if (gd) gd[16 * t + i] = v[i];
    if (gf) gf[16 * t + i] = (float)v[i];
  }
}

// projection weights in grid-point order
__global__ void k_grid_order(const int32_t* __restrict__ ge, int64_t n, const double* __restrict__ Ad,
                             const float* __restrict__ Af, double* __restrict__ od, float* __restrict__ of) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int64_t e = ge[i];
  for (int c = 0; c < 4; ++c) {
    if (od) od[4 * i + c] = Ad[4 * e + c];
    if (of) of[4 * i + c] = Af[4 * e + c];
  }
}

template <typename R>
int alloc_tables(PrecData<R>& pd, int64_t ne, int64_t ns, int64_t nt) {
  if (!pd.built) return SCABEM_OK;
  CK(cudaMalloc(&pd.wA, sizeof(R) * 4 * ne));
  CK(cudaMalloc(&pd.wB, sizeof(R) * 4 * ne));
  CK(cudaMalloc(&pd.wC, sizeof(R) * 2 * ne));
  CK(cudaMalloc(&pd.gA, sizeof(R) * 4 * ne));
  CK(cudaMalloc(&pd.sW, sizeof(R) * 20 * std::max<int64_t>(ns, 1)));
  CK(cudaMalloc(&pd.geo, sizeof(R) * 16 * nt));
  return SCABEM_OK;
}
template <typename R>
SigTables<R> sig_tables(const PrecData<R>& pd, int64_t ns) {
  if (!pd.built) return {nullptr, nullptr, nullptr, nullptr, nullptr};
  return {pd.sW, pd.sW + 4 * ns, pd.sW + 8 * ns, pd.sW + 12 * ns, pd.sW + 16 * ns};
}

}  // namespace

// Entry lists and conductivity-free weights (after the stencils and the
// covered points gpt of setup_gather).
int setup_moments(scabem_op* op, cudaStream_t s) {
  const int64_t nt = op->nt;
  const unsigned gw = (unsigned)cdiv(nt * 32, 128);
  const int n1 = op->n[1], n2 = op->n[2];
  CK(cudaMalloc(&op->toff, sizeof(int32_t) * (nt + 1)));
  CK(cudaMalloc(&op->soff, sizeof(int32_t) * nt));
  k_tri_points<<<gw, 128, 0, s>>>(op->base, nt, op->q, op->p, n1, n2, op->toff, nullptr, nullptr);
  CK(cudaGetLastError());
  std::vector<int32_t> off(nt + 1), soff(nt);
  std::vector<int32_t> te(3 * nt);
  CK(cudaMemcpyAsync(off.data(), op->toff, sizeof(int32_t) * nt, cudaMemcpyDeviceToHost, s));
  CK(cudaMemcpyAsync(te.data(), op->tedge, sizeof(int32_t) * 3 * nt, cudaMemcpyDeviceToHost, s));
  CK(cudaStreamSynchronize(s));
  int64_t acc = 0, ns = 0;  // at most Q p^3 < 2^31 entries (setup_gather)
  for (int64_t t = 0; t < nt; ++t) {
    const int32_t c = off[t];
    const bool hasR = te[3 * t] >= op->nL || te[3 * t + 1] >= op->nL || te[3 * t + 2] >= op->nL;
    soff[t] = hasR ? (int32_t)ns : -1;
    if (hasR) ns += c;
    off[t] = (int32_t)acc;
    acc += c;
  }
  off[nt] = (int32_t)acc;
  op->ntent = acc;
  op->nsent = ns;
  CK(cudaMemcpyAsync(op->toff, off.data(), sizeof(int32_t) * (nt + 1), cudaMemcpyHostToDevice, s));
  CK(cudaMemcpyAsync(op->soff, soff.data(), sizeof(int32_t) * nt, cudaMemcpyHostToDevice, s));
  CK(cudaMalloc(&op->tgi, sizeof(int32_t) * acc));
  k_tri_points<<<gw, 128, 0, s>>>(op->base, nt, op->q, op->p, n1, n2, nullptr, op->toff, op->tgi);
  CK(cudaGetLastError());
  if (int rc = alloc_tables(op->d, acc, ns, nt)) return rc;
  if (int rc = alloc_tables(op->f, acc, ns, nt)) return rc;
  k_tri_weights<<<gw, 128, 0, s>>>(op->toff, op->tgi, op->base, op->d.L, op->d.dL, op->d.tp, nt, op->q, op->p, n1, n2,
                                   Tables<double>{op->d.wA, op->d.wB, op->d.wC},
                                   Tables<float>{op->f.wA, op->f.wB, op->f.wC});
  CK(cudaGetLastError());
  k_tri_geo<<<(unsigned)cdiv(nt, 128), 128, 0, s>>>(op->tri, op->cX, nt, op->d.geo, op->f.geo);
  CK(cudaGetLastError());
  // the entries of every covered grid point, in triangle order (counting sort on the host)
  std::vector<int32_t> gi(acc), gpt(op->ngnz);
  CK(cudaMemcpyAsync(gi.data(), op->tgi, sizeof(int32_t) * acc, cudaMemcpyDeviceToHost, s));
  CK(cudaMemcpyAsync(gpt.data(), op->gpt, sizeof(int32_t) * op->ngnz, cudaMemcpyDeviceToHost, s));
  CK(cudaStreamSynchronize(s));
  const int64_t ng = (int64_t)op->n[0] * n1 * n2;
  std::vector<int32_t> pos(ng, -1), eoff(op->ngnz + 1, 0), gt(acc), ge(acc);
  for (int64_t i = 0; i < op->ngnz; ++i) pos[gpt[i]] = (int32_t)i;
  for (int64_t e = 0; e < acc; ++e) ++eoff[pos[gi[e]] + 1];
  for (int64_t i = 0; i < op->ngnz; ++i) eoff[i + 1] += eoff[i];
  std::vector<int32_t> cur(eoff.begin(), eoff.end() - 1);
  for (int64_t t = 0; t < nt; ++t)
    for (int64_t e = off[t]; e < off[t + 1]; ++e) {
      const int32_t k = cur[pos[gi[e]]]++;
      gt[k] = (int32_t)t;
      ge[k] = (int32_t)e;
    }
  CK(cudaMalloc(&op->eoff, sizeof(int32_t) * (op->ngnz + 1)));
  CK(cudaMalloc(&op->gtri, sizeof(int32_t) * acc));
  CK(cudaMalloc(&op->gent2, sizeof(int32_t) * acc));
  CK(cudaMemcpyAsync(op->eoff, eoff.data(), sizeof(int32_t) * (op->ngnz + 1), cudaMemcpyHostToDevice, s));
  CK(cudaMemcpyAsync(op->gtri, gt.data(), sizeof(int32_t) * acc, cudaMemcpyHostToDevice, s));
  CK(cudaMemcpyAsync(op->gent2, ge.data(), sizeof(int32_t) * acc, cudaMemcpyHostToDevice, s));
  k_grid_order<<<(unsigned)cdiv(acc, 256), 256, 0, s>>>(op->gent2, acc, op->d.wA, op->f.wA, op->d.gA, op->f.gA);
  CK(cudaGetLastError());
  CK(cudaStreamSynchronize(s));
  return SCABEM_OK;
}

int moments_update(scabem_op* op, cudaStream_t s) {
  if (op->nsent == 0) return SCABEM_OK;
  k_tri_sigma<<<(unsigned)cdiv(op->nt * 32, 128), 128, 0, s>>>(
      op->soff, op->toff, op->tgi, op->base, op->d.L, op->d.dL, op->d.tp, op->sig64, op->tri, op->nt, op->q, op->p,
      op->n[1], op->n[2], sig_tables(op->d, op->nsent), sig_tables(op->f, op->nsent));
  CK(cudaGetLastError());
  return SCABEM_OK;
}
