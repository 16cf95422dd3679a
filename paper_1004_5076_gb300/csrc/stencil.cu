// Set-up of the edge stencils: the grid's weights folded with the RWG test
// functions.
//
// The grid acts on the unknowns and rows of an edge only through quadrature
// sums of its function X over the edge's two triangles, so these sums are
// formed once per (edge, covered grid point g).  With W_a(g) the stencil weight
// of quadrature point a and w_a its quadrature weight:
//
//   Q0 = { x, d }   x = sum_a w_a X W_a,  d = sum_a w_a div X W_a
//   Q1 = { c, 0 }   c = sum_a w_a X x grad W_a   (<X, curl V> = sum_g c . V(g))
//
// Projection puts x J and d J on g; testing is x . V + d v and c . V of the
// potentials there.  Absorber edges carry four more blocks with sigma_a w_a in
// place of w_a and strong-form gradients, for Eq. 13 (n x X) and Eq. 14 (X):
//
//   S4 = { n x X W, (n x X) . grad W },  S5 = { (n x X) x grad W, 0 }
//   S6 = { X W, X . grad W },            S7 = { X x grad W, 0 }
//
// formed again on every scabem_set_sigma.  Entries of an edge are in class
// order (near.cu: plain edges first), 8 reals per entry of a plain edge, 24 per
// entry of an absorber edge.  An edge of the 12 um guide has about 45 entries,
// where the stencils of its 12 quadrature points hold 324.
#include <cuda_runtime.h>

#include <algorithm>
#include <vector>

#include "common.cuh"

namespace {

__device__ __forceinline__ bool covers(const int32_t* __restrict__ base, int64_t Qi, int i0, int i1, int i2, int p) {
  const int a = i0 - base[3 * Qi], b = i1 - base[3 * Qi + 1], c = i2 - base[3 * Qi + 2];
  return (unsigned)a < (unsigned)p && (unsigned)b < (unsigned)p && (unsigned)c < (unsigned)p;
}

// The grid points of each edge, one warp per edge, in (point, slot) order of
// the first stencil that covers them; as compact indices i0 nac + column.
// cnt != null only counts.
__global__ void __launch_bounds__(128) k_edge_points(const int32_t* __restrict__ rtk, const int32_t* __restrict__ base,
                                                     const int32_t* __restrict__ cmap, int64_t ne, int q, int p, int n2,
                                                     int nac, int32_t* __restrict__ cnt,
                                                     const int32_t* __restrict__ xoff, int32_t* __restrict__ xpt) {
  const int64_t r = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  if (r >= ne) return;
  const int lane = threadIdx.x & 31, p2 = p * p, p3 = p2 * p;
  const int64_t T[2] = {rtk[4 * r], rtk[4 * r + 2]};
  int n = 0;
  for (int b = 0; b < 2 * q * p3; b += 32) {
    const int u = b + lane;
    bool keep = u < 2 * q * p3;
    int i0 = 0, i1 = 0, i2 = 0;
    if (keep) {
      const int a = u / p3, sl = u - a * p3;
      const int64_t Qi = a < q ? T[0] * q + a : T[1] * q + a - q;
      i0 = base[3 * Qi] + sl / p2;
      i1 = base[3 * Qi + 1] + (sl / p) % p;
      i2 = base[3 * Qi + 2] + sl % p;
      for (int c = 0; c < a && keep; ++c) keep = !covers(base, c < q ? T[0] * q + c : T[1] * q + c - q, i0, i1, i2, p);
    }
    const unsigned m = __ballot_sync(0xffffffffu, keep);
    if (keep && !cnt) xpt[xoff[r] + n + __popc(m & ((1u << lane) - 1))] = i0 * nac + cmap[i1 * n2 + i2];
    n += __popc(m);
  }
  if (cnt && lane == 0) cnt[r] = n;
}

// Weights of the entries, one warp per edge, lanes over its entries (0.3 ms per call
// on the 5 um guide, FP64; once per operator and, SIG, per conductivity); sums over
// the quadrature points in FP64.  SIG: blocks S4 .. S7 of the absorber edges,
// else Q0, Q1 of all edges.
template <bool SIG>
__global__ void __launch_bounds__(128)
    k_edge_weights(const int32_t* __restrict__ rtk, const int32_t* __restrict__ xoff, const int32_t* __restrict__ xpt,
                   const int32_t* __restrict__ base, const int32_t* __restrict__ acol, const double* __restrict__ L,
                   const double* __restrict__ dL, const double* __restrict__ tp, const double* __restrict__ sig,
                   const double* __restrict__ tri, int64_t r0, int64_t ne, int64_t nL, int64_t nxl, int q, int p, int n2,
                   int nac, double* __restrict__ wd, float* __restrict__ wf) {
  const int64_t r = r0 + ((blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5);
  if (r >= ne) return;
  for (int64_t e = xoff[r] + (threadIdx.x & 31); e < xoff[r + 1]; e += 32) {
    const int i0 = xpt[e] / nac, cc = acol[xpt[e] - i0 * nac], i1 = cc / n2, i2 = cc - i1 * n2;
    double v[16] = {0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0};
    for (int side = 0; side < 2; ++side) {
      const int64_t t = rtk[4 * r + 2 * side];
      const int k = rtk[4 * r + 2 * side + 1];
      const double* n = tri + 16 * t + 12;
      for (int a = 0; a < q; ++a) {
        const int64_t Qi = t * q + a;
        if (!covers(base, Qi, i0, i1, i2, p)) continue;
        const int x = i0 - base[3 * Qi], y = i1 - base[3 * Qi + 1], z = i2 - base[3 * Qi + 2];
        const double lx = L[(3 * Qi + 0) * p + x], ly = L[(3 * Qi + 1) * p + y], lz = L[(3 * Qi + 2) * p + z];
        const double dx = dL[(3 * Qi + 0) * p + x], dy = dL[(3 * Qi + 1) * p + y], dz = dL[(3 * Qi + 2) * p + z];
        const double* tq = tp + 16 * Qi;
        const double w = SIG ? tq[3] * sig[Qi] : tq[3], W = w * lx * ly * lz;
        const double G[3] = {w * dx * ly * lz, w * lx * dy * lz, w * lx * ly * dz};
        const double X[3] = {tq[4 + 3 * k], tq[5 + 3 * k], tq[6 + 3 * k]};
        const double N[3] = {n[1] * X[2] - n[2] * X[1], n[2] * X[0] - n[0] * X[2], n[0] * X[1] - n[1] * X[0]};
        for (int c = 0; c < 3; ++c) {
          const int c1 = (c + 1) % 3, c2 = (c + 2) % 3;
          if (!SIG) {
            v[c] += W * X[c];
            v[4 + c] += X[c1] * G[c2] - X[c2] * G[c1];
          } else {
            v[c] += W * N[c];
            v[3] += N[c] * G[c];
            v[4 + c] += N[c1] * G[c2] - N[c2] * G[c1];
            v[8 + c] += W * X[c];
            v[11] += X[c] * G[c];
            v[12 + c] += X[c1] * G[c2] - X[c2] * G[c1];
          }
        }
        if (!SIG) v[3] += W * tq[13 + k];
      }
    }
    const int64_t o = (r < nL ? 8 * e : 8 * nxl + 24 * (e - nxl)) + (SIG ? 8 : 0);
    for (int c = 0; c < (SIG ? 16 : 8); ++c) {
      if (wd) wd[o + c] = v[c];
      if (wf) wf[o + c] = (float)v[c];
    }
  }
}

// Q0 in grid-point order, for the projection
__global__ void k_grid_order(const int32_t* __restrict__ ge, int64_t n, int64_t nxl, const double* __restrict__ wd,
                             const float* __restrict__ wf, double* __restrict__ od, float* __restrict__ of) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int64_t e = ge[i], o = e < nxl ? 8 * e : 8 * nxl + 24 * (e - nxl);
  for (int c = 0; c < 4; ++c) {
    if (od) od[4 * i + c] = wd[o + c];
    if (of) of[4 * i + c] = wf[o + c];
  }
}

template <typename R>
int alloc_tables(PrecData<R>& pd, int64_t nx, int64_t nxl) {
  if (!pd.built) return SCABEM_OK;
  CK(cudaMalloc(&pd.xw, sizeof(R) * (8 * nxl + 24 * (nx - nxl))));
  CK(cudaMalloc(&pd.gq, sizeof(R) * 4 * nx));
  return SCABEM_OK;
}

}  // namespace

// Entry lists and conductivity-free weights (after the stencils, the active
// columns and the covered points of setup_gather).
int setup_stencils(scabem_op* op, cudaStream_t s) {
  const int64_t ne = op->ne;
  const unsigned gw = (unsigned)cdiv(ne * 32, 128);
  const int n2 = op->n[2], nac = (int)op->nac;
  const int64_t npt = (int64_t)op->n[0] * nac;
  CK(cudaMalloc(&op->xoff, sizeof(int32_t) * (ne + 1)));
  k_edge_points<<<gw, 128, 0, s>>>(op->rtk, op->base, op->cmap, ne, op->q, op->p, n2, nac, op->xoff, nullptr, nullptr);
  CK(cudaGetLastError());
  std::vector<int32_t> off(ne + 1);
  CK(cudaMemcpyAsync(off.data(), op->xoff, sizeof(int32_t) * ne, cudaMemcpyDeviceToHost, s));
  CK(cudaStreamSynchronize(s));
  int64_t acc = 0;
  for (int64_t r = 0; r < ne; ++r) {
    if (r == op->nL) op->nxl = acc;
    const int32_t c = off[r];
    off[r] = (int32_t)acc;
    acc += c;
    if (acc > INT32_MAX) {
      set_error("mesh too large for the projection map");
      return SCABEM_E_ARG;
    }
  }
  if (op->nL == ne) op->nxl = acc;
  off[ne] = (int32_t)acc;
  op->nx = acc;
  CK(cudaMemcpyAsync(op->xoff, off.data(), sizeof(int32_t) * (ne + 1), cudaMemcpyHostToDevice, s));
  CK(cudaMalloc(&op->xpt, sizeof(int32_t) * acc));
  k_edge_points<<<gw, 128, 0, s>>>(op->rtk, op->base, op->cmap, ne, op->q, op->p, n2, nac, nullptr, op->xoff, op->xpt);
  CK(cudaGetLastError());
  if (int rc = alloc_tables(op->d, acc, op->nxl)) return rc;
  if (int rc = alloc_tables(op->f, acc, op->nxl)) return rc;
  k_edge_weights<false><<<gw, 128, 0, s>>>(op->rtk, op->xoff, op->xpt, op->base, op->acol, op->d.L, op->d.dL, op->d.tp,
                                           nullptr, op->tri, 0, ne, op->nL, op->nxl, op->q, op->p, n2, nac, op->d.xw,
                                           op->f.xw);
  CK(cudaGetLastError());
  // the entries of every covered grid point, in edge order (counting sort on the host)
  std::vector<int32_t> pt(acc);
  CK(cudaMemcpyAsync(pt.data(), op->xpt, sizeof(int32_t) * acc, cudaMemcpyDeviceToHost, s));
  CK(cudaStreamSynchronize(s));
  std::vector<int32_t> cnt(npt + 1, 0), cntl(npt, 0);
  for (int64_t e = 0; e < acc; ++e) ++cnt[pt[e]];
  for (int64_t e = 0; e < op->nxl; ++e) ++cntl[pt[e]];
  std::vector<int32_t> list, goff, gl, cur(npt);
  goff.push_back(0);
  for (int64_t i = 0; i < npt; ++i) {
    if (!cnt[i]) continue;
    cur[i] = goff.back();
    list.push_back((int32_t)i);
    gl.push_back(cntl[i]);
    goff.push_back(goff.back() + cnt[i]);
  }
  std::vector<int32_t> gr(acc), ge(acc);
  for (int64_t r = 0; r < ne; ++r)
    for (int64_t e = off[r]; e < off[r + 1]; ++e) {
      const int32_t k = cur[pt[e]]++;
      gr[k] = (int32_t)r;
      ge[k] = (int32_t)e;
    }
  op->ngp = (int64_t)list.size();
  CK(cudaMalloc(&op->gp, sizeof(int32_t) * op->ngp));
  CK(cudaMalloc(&op->gpoff, sizeof(int32_t) * (op->ngp + 1)));
  CK(cudaMalloc(&op->gpl, sizeof(int32_t) * op->ngp));
  CK(cudaMalloc(&op->gpr, sizeof(int32_t) * acc));
  CK(cudaMalloc(&op->gpe, sizeof(int32_t) * acc));
  CK(cudaMemcpyAsync(op->gp, list.data(), sizeof(int32_t) * op->ngp, cudaMemcpyHostToDevice, s));
  CK(cudaMemcpyAsync(op->gpoff, goff.data(), sizeof(int32_t) * (op->ngp + 1), cudaMemcpyHostToDevice, s));
  CK(cudaMemcpyAsync(op->gpl, gl.data(), sizeof(int32_t) * op->ngp, cudaMemcpyHostToDevice, s));
  CK(cudaMemcpyAsync(op->gpr, gr.data(), sizeof(int32_t) * acc, cudaMemcpyHostToDevice, s));
  CK(cudaMemcpyAsync(op->gpe, ge.data(), sizeof(int32_t) * acc, cudaMemcpyHostToDevice, s));
  k_grid_order<<<(unsigned)cdiv(acc, 256), 256, 0, s>>>(op->gpe, acc, op->nxl, op->d.xw, op->f.xw, op->d.gq, op->f.gq);
  CK(cudaGetLastError());
  CK(cudaStreamSynchronize(s));
  op->h_xoff = std::move(off);
  return SCABEM_OK;
}

// The conductivity-weighted blocks for the operator's current conductivity
int stencils_update(scabem_op* op, cudaStream_t s) {
  if (op->nR == 0) return SCABEM_OK;
  k_edge_weights<true><<<(unsigned)cdiv(op->nR * 32, 128), 128, 0, s>>>(
      op->rtk, op->xoff, op->xpt, op->base, op->acol, op->d.L, op->d.dL, op->d.tp, op->sig64, op->tri, op->nL, op->ne,
      op->nL, op->nxl, op->q, op->p, op->n[2], (int)op->nac, op->d.xw, op->f.xw);
  CK(cudaGetLastError());
  return SCABEM_OK;
}
