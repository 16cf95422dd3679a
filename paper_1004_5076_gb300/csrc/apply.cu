// The matvec y = A x of the grid-accelerated operator (one right-hand side).
//
//  K1 k_summ     RWG coefficients -> per-triangle current summaries
//                J(r) = a (r - c_t) - beta for the exterior J, interior J and
//                exterior M sets (current reduction, Eqs. 10-12)
//  K2 k_project  summaries spread onto the grid by the triangles' stencil
//                moments (moments.cu; 12 fields), as a gather over the covered
//                grid points
//  K3-5          fft_conv (fft.cu): 12 -> 16 grid potentials (A, phi, F, psi
//                of each medium, Eqs. 15-16)
//  K6 k_test     the potentials, gradients and curls tested per triangle by the
//                same moments: Galerkin rows of Eqs. 1-3 (weak form), Eq. 13 and
//                Eq. 14 (sigma-weighted)
//  K7 k_near_rows  (near.cu) near-field precorrection (exact minus grid panel
//                interaction) and side-limit terms as a sparse matrix over
//                edges, plus the row sums of the tested values
#include <cuda_runtime.h>

#include "common.cuh"

namespace {

template <typename R>
__device__ __forceinline__ cx<R> coef_of(const cx<R>* __restrict__ x, int32_t code) {
  if (code > 0) return x[code - 1];
  if (code < 0) return -x[-code - 1];
  return czero<R>();
}

// a += s * b on (re, im) as one packed FP32x2 FMA in complex64.
__device__ __forceinline__ void axpy2(cx<float>& a, float s, cx<float> b) {
  const float2 r = __ffma2_rn(make_float2(s, s), make_float2(b.re, b.im), make_float2(a.re, a.im));
  a = mk(r.x, r.y);
}
__device__ __forceinline__ void axpy2(cx<double>& a, double s, cx<double> b) { axpy(a, s, b); }

// The four potentials of one (grid point, medium, group), or the summary (a,
// beta) of one (triangle, set): 32 contiguous bytes in complex64.
__device__ __forceinline__ void load_group(const cx<float>* p, cx<float>* v) {
  const float4 u0 = __ldg(reinterpret_cast<const float4*>(p));
  const float4 u1 = __ldg(reinterpret_cast<const float4*>(p) + 1);
  v[0] = mk(u0.x, u0.y);
  v[1] = mk(u0.z, u0.w);
  v[2] = mk(u1.x, u1.y);
  v[3] = mk(u1.z, u1.w);
}
__device__ __forceinline__ void load_group(const cx<double>* p, cx<double>* v) {
#pragma unroll
  for (int f = 0; f < 4; ++f) {
    const double2 u = __ldg(reinterpret_cast<const double2*>(p) + f);
    v[f] = mk(u.x, u.y);
  }
}
// Four reals starting on a 16-byte boundary
__device__ __forceinline__ void load4(const float* p, float* v) {
  const float4 u = __ldg(reinterpret_cast<const float4*>(p));
  v[0] = u.x;
  v[1] = u.y;
  v[2] = u.z;
  v[3] = u.w;
}
__device__ __forceinline__ void load4(const double* p, double* v) {
  const double2 a = __ldg(reinterpret_cast<const double2*>(p)), b = __ldg(reinterpret_cast<const double2*>(p) + 1);
  v[0] = a.x;
  v[1] = a.y;
  v[2] = b.x;
  v[3] = b.y;
}
__device__ __forceinline__ void load2(const float* p, float* v) {
  const float2 u = __ldg(reinterpret_cast<const float2*>(p));
  v[0] = u.x;
  v[1] = u.y;
}
__device__ __forceinline__ void load2(const double* p, double* v) {
  const double2 u = __ldg(reinterpret_cast<const double2*>(p));
  v[0] = u.x;
  v[1] = u.y;
}

// v[t] of a pair of lanes that differ in lane bit `o`: the lower one keeps
// v[0 .. half), the upper one v[half .. 2 half), each adding the other's part
// (the halving step of a reduction over several values).
template <typename R>
__device__ __forceinline__ void halve(cx<R>* v, int half, int lane, int o) {
  const bool up = (lane & o) != 0;
#pragma unroll
  for (int t = 0; t < half; ++t) {
    const cx<R> send = up ? v[t] : v[t + half], keep = up ? v[t + half] : v[t];
    v[t] = keep + mk(__shfl_xor_sync(0xffffffffu, send.re, o), __shfl_xor_sync(0xffffffffu, send.im, o));
  }
}
template <typename R>
__device__ __forceinline__ cx<R> xadd(cx<R> v, int o) {
  return v + mk(__shfl_xor_sync(0xffffffffu, v.re, o), __shfl_xor_sync(0xffffffffu, v.im, o));
}

// K1: one thread per (triangle, set): the current summary
// summ[(t*3+set)*4 + {a, bx, by, bz}], J(r) = a (r - c_t) - beta, of the
// exterior J, interior J and exterior M sets.
template <typename R>
__global__ void k_summ(const cx<R>* __restrict__ x, const int32_t* __restrict__ unk, const R* __restrict__ geo,
                       int64_t nt, cx<R>* __restrict__ summ, int64_t ldx) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= 3 * nt) return;
  x += blockIdx.y * ldx;  // right-hand side blockIdx.y of a batch
  summ += blockIdx.y * 12 * nt;
  const int64_t t = i / 3;
  const int set = (int)(i - 3 * t);
  cx<R> a = czero<R>(), b0 = a, b1 = a, b2 = a;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    R g[4];
    load4(geo + 16 * t + 4 * k, g);
    const cx<R> j = g[0] * coef_of(x, unk[(3 * t + k) * 3 + set]);
    a += j;
    axpy2(b0, g[1], j);
    axpy2(b1, g[2], j);
    axpy2(b2, g[3], j);
  }
  cx<R>* o = summ + 4 * i;
  o[0] = a;
  o[1] = b0;
  o[2] = b1;
  o[3] = b2;
}

// K2: projection as a gather over the triangles.  One warp per grid point
// that some stencil covers: lane = set * 8 + slot takes entries slot, slot + 8,
// ... of the point, each one triangle's summary of that set (32 bytes in
// complex64) against its moments m0, m1: a m1 - beta m0 and 2 a m0.  The slot
// sums meet by halving exchanges.  Points no stencil covers stay zero from
// set-up.  The sum order is fixed, so the result does not depend on thread
// timing.  Bound by the latency of the (triangle -> summary) loads out of L2:
// two entries per lane are in flight.
constexpr int PJ_INFLIGHT = 2;

template <typename R>
__global__ void __launch_bounds__(256) k_project(const cx<R>* __restrict__ summ, const int32_t* __restrict__ gpt,
                                                 const int32_t* __restrict__ eoff, const int32_t* __restrict__ gtri,
                                                 const R* __restrict__ gA, int64_t ngnz, int64_t ng,
                                                 cx<R>* __restrict__ grids, int64_t cs_s, int64_t cs_g) {
  summ += blockIdx.y * cs_s;  // right-hand side blockIdx.y of a batch
  grids += blockIdx.y * cs_g;
  const int64_t i = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  if (i >= ngnz) return;  // whole warp
  const int lane = threadIdx.x & 31, set = min(lane >> 3, 2), slot = lane & 7;
  cx<R> acc[4];
#pragma unroll
  for (int c = 0; c < 4; ++c) acc[c] = czero<R>();
  const int e1 = lane < 24 ? eoff[i + 1] : 0;
  for (int e = eoff[i] + slot; e < e1; e += 8 * PJ_INFLIGHT) {
    R w[PJ_INFLIGHT][4];
    cx<R> v[PJ_INFLIGHT][4];
#pragma unroll
    for (int u = 0; u < PJ_INFLIGHT; ++u) {
      const int eu = e + 8 * u < e1 ? e + 8 * u : e;
      load4(gA + 4 * (int64_t)eu, w[u]);
      load_group(summ + (3 * (int64_t)gtri[eu] + set) * 4, v[u]);
    }
#pragma unroll
    for (int u = 0; u < PJ_INFLIGHT; ++u) {
      const R on = e + 8 * u < e1 ? R(1) : R(0);
      const R m0 = on * w[u][0];
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        axpy2(acc[c], on * w[u][1 + c], v[u][0]);
        axpy2(acc[c], -m0, v[u][1 + c]);
      }
      axpy2(acc[3], m0 + m0, v[u][0]);
    }
  }
  halve(acc, 2, lane, 4);
  halve(acc, 1, lane, 2);
  acc[0] = xadd(acc[0], 1);
  if (lane < 24 && !(lane & 1)) grids[(int64_t)(set * 4 + ((lane >> 1) & 1) + ((lane >> 1) & 2)) * ng + gpt[i]] = acc[0];
}

template <typename R>
const R* gather_dweights(scabem_op* op);
template <>
const float* gather_dweights<float>(scabem_op* op) {
  return op->gdf;
}
template <>
const double* gather_dweights<double>(scabem_op* op) {
  return op->gdd;
}

template <typename R>
const R* gather_weights(scabem_op* op);
template <>
const float* gather_weights<float>(scabem_op* op) {
  return op->gwf;
}
template <>
const double* gather_weights<double>(scabem_op* op) {
  return op->gwd;
}

// Two consecutive complex values of shared memory on a 16-byte boundary.
__device__ __forceinline__ void load_pair_smem(const cx<float>* p, cx<float>* v) {
  const float4 u = *reinterpret_cast<const float4*>(p);
  v[0] = mk(u.x, u.y);
  v[1] = mk(u.z, u.w);
}
__device__ __forceinline__ void load_pair_smem(const cx<double>* p, cx<double>* v) {
  v[0] = p[0];
  v[1] = p[1];
}

// Two consecutive complex values starting on a 16-byte boundary.
__device__ __forceinline__ void load_pair(const cx<float>* p, cx<float>* v) {
  const float4 u = __ldg(reinterpret_cast<const float4*>(p));
  v[0] = mk(u.x, u.y);
  v[1] = mk(u.z, u.w);
}
__device__ __forceinline__ void load_pair(const cx<double>* p, cx<double>* v) {
  v[0] = p[0];
  v[1] = p[1];
}

// Interpolated potentials of one medium at quadrature point Qi, group h of
// the record (NREC = 2 x 10): h = 0 A(3) phi grad phi(3) curl A(3) from the
// J fields, h = 1 F(3) psi grad psi(3) curl F(3) from the M fields.  The
// grid is point-major: point g holds its 16 potentials at grids[16 g ..].
template <typename R, int p>
__device__ __forceinline__ void interp_group(const cx<R>* __restrict__ grids, const int32_t* __restrict__ base,
                                             const R* __restrict__ L, const R* __restrict__ dL, int64_t Qi, int med,
                                             int h, int n1, int n2, cx<R>* r) {
  R Lx[p], Ly[p], Lz[p], dx[p], dy[p], dz[p];
#pragma unroll
  for (int i = 0; i < p; ++i) {
    Lx[i] = L[(3 * Qi + 0) * p + i];
    Ly[i] = L[(3 * Qi + 1) * p + i];
    Lz[i] = L[(3 * Qi + 2) * p + i];
    dx[i] = dL[(3 * Qi + 0) * p + i];
    dy[i] = dL[(3 * Qi + 1) * p + i];
    dz[i] = dL[(3 * Qi + 2) * p + i];
  }
  const int b0 = base[3 * Qi], b1 = base[3 * Qi + 1], b2 = base[3 * Qi + 2];
  cx<R> v[4], gx[4], gy[4], gz[4];
  for (int f = 0; f < 4; ++f) v[f] = gx[f] = gy[f] = gz[f] = czero<R>();
  const cx<R>* gm = grids + 4 * (med * 2 + h);
#pragma unroll
  for (int i = 0; i < p; ++i)
#pragma unroll
    for (int j = 0; j < p; ++j) {
      const R wxy = Lx[i] * Ly[j], dxy = dx[i] * Ly[j], xdy = Lx[i] * dy[j];
      const int64_t rowi = ((int64_t)(b0 + i) * n1 + (b1 + j)) * n2 + b2;
#pragma unroll
      for (int k = 0; k < p; ++k) {
        const R w = wxy * Lz[k], wx = dxy * Lz[k], wy = xdy * Lz[k], wz = wxy * dz[k];
        cx<R> gv[4];
        load_group(gm + (rowi + k) * NFIELD_OUT, gv);
#pragma unroll
        for (int f = 0; f < 4; ++f) {
          axpy2(v[f], w, gv[f]);
          axpy2(gx[f], wx, gv[f]);
          axpy2(gy[f], wy, gv[f]);
          axpy2(gz[f], wz, gv[f]);
        }
      }
    }
  r[0] = v[0];
  r[1] = v[1];
  r[2] = v[2];
  r[3] = v[3];
  r[4] = gx[3];
  r[5] = gy[3];
  r[6] = gz[3];
  r[7] = gy[2] - gz[1];
  r[8] = gz[0] - gx[2];
  r[9] = gx[1] - gy[0];
}

// One near record (dP0, dP1, dQ, dC) applied to source summary sv (a, beta):
// A += a dP1 - beta dP0, phi += 2a dP0, grad phi += 2a dQ,
// curl A += a dC - dQ x beta (the same for F, psi of an M source).
template <typename R>
__device__ __forceinline__ void near_part(const cx<R>* d, const cx<R>* sv, cx<R>* acc) {
  const cx<R> d0 = d[0];
  const cx<R> al = sv[0], al2 = R(2) * al;
  const cx<R> be[3] = {sv[1], sv[2], sv[3]};
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    cfma(acc[c], al, d[1 + c]);
    acc[c] -= be[c] * d0;
    cfma(acc[4 + c], al2, d[4 + c]);
    cfma(acc[7 + c], al, d[7 + c]);
  }
  cfma(acc[3], al2, d0);
  acc[7] -= d[5] * be[2] - d[6] * be[1];
  acc[8] -= d[6] * be[0] - d[4] * be[2];
  acc[9] -= d[4] * be[1] - d[5] * be[0];
}

template <typename R>
__device__ __forceinline__ cx<R> dot3(const R* X, const cx<R>* V) {
  return X[0] * V[0] + X[1] * V[1] + X[2] * V[2];
}

// d out / d sg of the Eq. 13 and Eq. 14 tested values of local edge kk at
// point a (sg the normalised conductivity): d2 = w (-(n x X) . E_e - X . M / 2),
// d3 = w (-X . E_i - X . (n x M) / 2), from the point's records.
template <typename R>
__device__ __forceinline__ void test_point_sigma(const cx<R>* recs, const cx<R>* __restrict__ summ,
                                                 const double* __restrict__ tri, const R* __restrict__ tp, int64_t t,
                                                 int kk, int a, int q, R ke, R ki, R ze, R zi, cx<R>& d2,
                                                 cx<R>& d3) {
  const double* g = tri + 16 * t;
  const R nrm[3] = {(R)g[12], (R)g[13], (R)g[14]};
  const cx<R>* sM = summ + (3 * t + 2) * 4;
  const R* tq = tp + 16 * (t * q + a);
  const R w = tq[3];
  R X[3], rel[3];
  for (int c = 0; c < 3; ++c) {
    X[c] = tq[4 + 3 * kk + c];
    rel[c] = tq[c];
  }
  const R kl[2] = {ke, ki}, zl[2] = {ze, zi};
  cx<R> E[2][3];
  for (int m = 0; m < 2; ++m) {
    const cx<R>* r = recs + m * NREC;
    const R k = kl[m], z = zl[m];
    for (int c = 0; c < 3; ++c)
      E[m][c] = -z * (k * mulj(r[c]) + (R(1) / k) * mulj(r[4 + c])) - r[17 + c];
  }
  cx<R> M[3], nM[3];
  for (int c = 0; c < 3; ++c) M[c] = rel[c] * sM[0] - sM[1 + c];
  nM[0] = nrm[1] * M[2] - nrm[2] * M[1];
  nM[1] = nrm[2] * M[0] - nrm[0] * M[2];
  nM[2] = nrm[0] * M[1] - nrm[1] * M[0];
  const R nX[3] = {nrm[1] * X[2] - nrm[2] * X[1], nrm[2] * X[0] - nrm[0] * X[2], nrm[0] * X[1] - nrm[1] * X[0]};
  d2 = -w * (dot3(nX, E[0]) + R(0.5) * dot3(X, M));
  d3 = -w * (dot3(X, E[1]) + R(0.5) * dot3(X, nM));
}

// Bulk asynchronous global -> shared copies (the TMA unit, cp.async.bulk)
// completing on an mbarrier, and bounded waits on it.
__device__ __forceinline__ unsigned smem_u32(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mbar_init(uint64_t* bar, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_init_fence() {
  asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
}
__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory"); }
// The near records are read once per apply: their copies carry an L2
// evict-first policy, so that the stream of records does not push the
// apply's reused data (grids, sources, geometry) and the caller's vectors out
// of L2.
__device__ __forceinline__ void bulk_copy(void* dst, const void* src, unsigned bytes, uint64_t* bar) {
  uint64_t pol;
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;\n" : "=l"(pol));
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], %4;\n" ::"r"(
          smem_u32(dst)),
      "l"(src), "r"(bytes), "r"(smem_u32(bar)), "l"(pol)
      : "memory");
}
// The arrival of one thread that expects `bytes` of copies on `bar`, and one
// bulk copy completing its bytes there (several copies may share one arrival).
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(smem_u32(bar)), "r"(bytes)
               : "memory");
}
// one arrival that also expects `bytes` of transaction, then the copy
__device__ __forceinline__ void bulk_load(void* dst, const void* src, unsigned bytes, uint64_t* bar) {
  mbar_expect_tx(bar, bytes);
  bulk_copy(dst, src, bytes, bar);
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, unsigned parity) {
  unsigned ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ uint64_t gtimer_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;\n" : "=l"(t));
  return t;
}
// Wait for the phase of the given parity; false after about a second.
constexpr uint64_t WAIT_LIMIT_NS = 1000000000ull;
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, unsigned parity) {
  if (mbar_try_wait(bar, parity)) return true;
  const uint64_t t0 = gtimer_ns();
  for (;;) {
    for (int i = 0; i < 64; ++i)
      if (mbar_try_wait(bar, parity)) return true;
    if (gtimer_ns() - t0 > WAIT_LIMIT_NS) return false;
  }
}

// Self-test of the bounded waits: one warp waits on an mbarrier that no
// arrival or copy ever completes, through the same mbar_wait as the record
// rings; when the wait gives up it reports through *tmo exactly as they do.
__global__ void k_wait_selftest(int* __restrict__ tmo) {
  __shared__ uint64_t bar;
  if (threadIdx.x == 0) {
    mbar_init(&bar, 1);
    mbar_init_fence();
  }
  __syncwarp();
  const bool ok = __all_sync(0xffffffffu, mbar_wait(&bar, 0));
  if (!ok && threadIdx.x == 0) atomicOr(tmo, 1);
}

// Conductivity sensitivity, one warp per target triangle t, PT_WARPS triangles
// per CTA; warps never wait on one another.
//  Phase 1: lane (point a, medium, record group h), 4q lanes, interpolates
//    its 10 record values, then adds the near corrections.  The triangle's
//    near records are one contiguous run (pairs noff[t] .. noff[t+1]); they
//    stream through a per-warp ring of PT_NSTG stages of PT_KP pairs, one
//    bulk copy per stage issued by lane 0, the next stages in flight while
//    one is consumed (the first ones during the interpolation).  A stage
//    that does not arrive within the wait limit sets *tmo and ends the
//    triangle's near loop after its copies in flight have landed.
//  Phase 2: lane (local edge kk, point a), 3q lanes, differentiates the point's
//    sigma-weighted tested values; they are summed over kk into
//    hs[t q + a] = eta0 sum_kk (lam_row2 d2 + lam_row3 d3), the derivative of
//    lam^T A x with respect to the conductivity [S] at the point.
constexpr int PT_WARPS = 4;
constexpr int PT_NSTG = 2;  // 2 stages of 4 pairs: the bytes in flight of 4 stages of 2, with half the
constexpr int PT_KP = 4;    // stages' waits, fences and copy issues per pair

// complex values of per-warp shared memory: the ring, which the records and
// point parts of phases 2-3 reuse once the near loop is done
__host__ __device__ constexpr int pt_warp_complex(int q) {
  return PT_NSTG * PT_KP * NCORR * 2 * q > 2 * q * NREC + 3 * q * 4 ? PT_NSTG * PT_KP * NCORR * 2 * q
                                                                     : 2 * q * NREC + 3 * q * 4;
}
// bytes of shared memory per CTA: rings, then one mbarrier per stage and warp
__host__ __device__ constexpr size_t pt_smem_bytes(int q, size_t csize) {
  return (size_t)PT_WARPS * pt_warp_complex(q) * csize + (size_t)PT_WARPS * PT_NSTG * sizeof(uint64_t);
}

// Lanes past the 4q of phase 1 repeat lane 4q - 4 .. 4q - 1's work without
// storing it, so that the near loop runs without divergence.
template <typename R, int P>
__global__ void __launch_bounds__(PT_WARPS * 32, 3) k_points_sens(
    const cx<R>* __restrict__ grids, const int32_t* __restrict__ base, const R* __restrict__ L,
    const R* __restrict__ dL, const cx<R>* __restrict__ corr, const int32_t* __restrict__ noff,
    const int32_t* __restrict__ nsrc, const cx<R>* __restrict__ summ, const double* __restrict__ tri,
    const R* __restrict__ tp, int64_t nt, int q, int n1, int n2, R ke, R ki, R ze, R zi, int has_near,
    const int32_t* __restrict__ valrow, int* __restrict__ tmo, const cx<R>* __restrict__ lam, cx<R>* __restrict__ hs) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t t = (int64_t)blockIdx.x * PT_WARPS + warp;
  if (t >= nt) return;  // whole warp; no CTA-wide barrier below
  const int pairc = NCORR * 2 * q;  // complex per pair: [point][medium][component]
  cx<R>* ring = reinterpret_cast<cx<R>*>(smem_raw) + (int64_t)warp * pt_warp_complex(q);
  uint64_t* bars = reinterpret_cast<uint64_t*>(reinterpret_cast<cx<R>*>(smem_raw) + PT_WARPS * pt_warp_complex(q)) +
                   warp * PT_NSTG;
  cx<R>* recs = ring;                 // [q][2][NREC], after the near loop
  cx<R>* part = recs + 2 * q * NREC;  // [3][q][4]

  const bool act = lane < 4 * q;
  const int a = min(lane >> 2, q - 1), med = (lane >> 1) & 1, h = lane & 1;
  const int j0 = has_near ? noff[t] : 0, j1 = has_near ? noff[t + 1] : 0;
  const int nst = (j1 - j0 + PT_KP - 1) / PT_KP;
  const unsigned pair_bytes = (unsigned)(pairc * sizeof(cx<R>));
  // stage st -> slot st % PT_NSTG, issued by lane 0
  auto issue = [&](int st) {
    const int pj = j0 + st * PT_KP;
    const int np = min(PT_KP, j1 - pj);
    fence_proxy_async();  // earlier reads of the slot come before the copy
    bulk_load(ring + (st % PT_NSTG) * PT_KP * pairc, corr + (int64_t)pj * pairc, np * pair_bytes,
              bars + st % PT_NSTG);
  };
  if (nst > 0) {
    if (lane == 0) {
#pragma unroll
      for (int i = 0; i < PT_NSTG; ++i) mbar_init(bars + i, 1);
      mbar_init_fence();
      for (int st = 0; st < PT_NSTG - 1 && st < nst; ++st) issue(st);
    }
    __syncwarp();
  }
  // source triangles of the pairs, 32 at a time in the lanes (one block ahead)
  const int npair = j1 - j0;
  int src_nxt = lane < npair ? nsrc[j0 + lane] : 0, src_cur = 0;
  cx<R> acc[NREC / 2];
  interp_group<R, P>(grids, base, L, dL, t * q + a, med, h, n1, n2, acc);
  if (nst > 0) {
    const int set = h ? 2 : med;  // source J of this medium, or M
    // the interior medium sees -M: accumulate -acc + sum, then negate back
    const bool neg = h && med;
    if (neg)
#pragma unroll
      for (int c = 0; c < NREC / 2; ++c) acc[c] = -acc[c];
    int st = 0;
    bool ok = true;
    for (; st < nst; ++st) {
      if (lane == 0 && st + PT_NSTG - 1 < nst) issue(st + PT_NSTG - 1);  // slot consumed at st - 1
      ok = __all_sync(0xffffffffu, mbar_wait(bars + st % PT_NSTG, (st / PT_NSTG) & 1));
      if (!ok) break;
      const cx<R>* rs = ring + (st % PT_NSTG) * PT_KP * pairc + (a * 2 + med) * NCORR;
#pragma unroll
      for (int k = 0; k < PT_KP; ++k) {
        const int jj = st * PT_KP + k;  // pair within the triangle (warp-uniform)
        if (jj < npair) {
          if ((jj & 31) == 0) {
            src_cur = src_nxt;
            src_nxt = jj + 32 + lane < npair ? nsrc[j0 + jj + 32 + lane] : 0;
          }
          const int64_t sj = __shfl_sync(0xffffffffu, src_cur, jj & 31);
          cx<R> d[NCORR], sv[4];
          load_group(summ + (3 * sj + set) * 4, sv);
#pragma unroll
          for (int c = 0; c < NCORR; c += 2) load_pair_smem(rs + k * pairc + c, d + c);
          near_part(d, sv, acc);
        }
      }
      __syncwarp();
    }
    if (!ok) {
      // stages st .. min(st + PT_NSTG - 1, nst - 1) were issued: let them land
      for (int s2 = st; s2 < nst && s2 < st + PT_NSTG; ++s2) (void)mbar_wait(bars + s2 % PT_NSTG, (s2 / PT_NSTG) & 1);
      if (lane == 0) atomicOr(tmo, 1);
    }
    __syncwarp();  // every lane is done with the ring before it holds records
    if (neg)
#pragma unroll
      for (int c = 0; c < NREC / 2; ++c) acc[c] = -acc[c];
  }
  if (act) {
    cx<R>* o = recs + (a * 2 + med) * NREC + 10 * h;
#pragma unroll
    for (int c = 0; c < NREC / 2; ++c) o[c] = acc[c];
  }
  __syncwarp();
  if (lane < 3 * q) {
    const int kk = lane / q, pa = lane - kk * q;
    cx<R> d2, d3;
    test_point_sigma(recs + pa * 2 * NREC, summ, tri, tp, t, kk, pa, q, ke, ki, ze, zi, d2, d3);
    const int r2 = valrow[(t * 3 + kk) * 4 + 2], r3 = valrow[(t * 3 + kk) * 4 + 3];
    cx<R> c = czero<R>();
    if (r2 >= 0) c += lam[r2] * d2;
    if (r3 >= 0) c += lam[r3] * d3;
    part[kk * q + pa] = c;
  }
  __syncwarp();
  if (lane < q) hs[t * q + lane] = R(ETA0) * (part[lane] + part[q + lane] + part[2 * q + lane]);
}

// K6-7: interpolation and testing by the triangle moments (moments.cu), one
// warp per triangle.  Lane = slot * 4 + group takes entries slot, slot + 8, ...
// of the triangle's grid points and the four potentials of its (medium, J or
// M set) group there (32 bytes in complex64): the value sums V = <pot>, S =
// <rel . pot> - 2/k^2 <charge potential> and the curl sums C = <curl pot>,
// D = <rel . curl pot>; on triangles with an absorber edge also Z, Y, the
// sigma-weighted strong-form E sums of its medium (rel -> n x rel in the
// exterior one, for Eq. 13).  The slots meet by halving exchanges, and lane (kk,
// type) forms the tested value of local edge kk:
//   type 0 <X, E_e - E_i>, 1 <X, H_e - H_i> (weak forms), 2 Eq. 13, 3 Eq. 14,
// with X_kk = cX_kk (rel - rel_kk).
constexpr int TS_WARPS = 4;

template <typename R>
__global__ void __launch_bounds__(TS_WARPS * 32)
    k_test(const cx<R>* __restrict__ grids, const int32_t* __restrict__ toff, const int32_t* __restrict__ tgi,
           const int32_t* __restrict__ soff, const R* __restrict__ wA, const R* __restrict__ wB,
           const R* __restrict__ wC, const R* __restrict__ sW, int64_t ns, const R* __restrict__ geo, int64_t nt, R ke,
           R ki, R ze, R zi, cx<R>* __restrict__ val, int64_t cs_g, int64_t cs_v) {
  __shared__ cx<R> red[TS_WARPS][48];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t t = (int64_t)blockIdx.x * TS_WARPS + warp;
  if (t >= nt) return;  // whole warp; no CTA-wide barrier below
  grids += blockIdx.y * cs_g;  // right-hand side blockIdx.y of a batch
  const int grp = lane & 3, slot = lane >> 2;
  const bool isM = grp & 1, inner = grp & 2;
  const int e0 = toff[t], e1 = toff[t + 1], s0 = soff[t];
  const R k = inner ? ki : ke, ik2 = R(1) / (k * k), kap = R(-2) * ik2;
  cx<R> v[8], z[4];  // V, S, C, D; Z, Y
#pragma unroll
  for (int i = 0; i < 8; ++i) v[i] = czero<R>();
#pragma unroll
  for (int i = 0; i < 4; ++i) z[i] = czero<R>();
  const R* sA = sW + 4 * (int64_t)(s0 - e0);
  // sigma block of this lane: J exterior D, interior B; M exterior E, interior C
  const R* sB = sA + 4 * ns * (isM ? (inner ? 2 : 4) : (inner ? 1 : 3));
  const cx<R>* gb = grids + 4 * grp;
#pragma unroll 2
  for (int e = e0 + slot; e < e1; e += 8) {
    cx<R> g[4];
    R a[4], b[4], c[2];
    load_group(gb + (int64_t)tgi[e] * NFIELD_OUT, g);
    load4(wA + 4 * (int64_t)e, a);
    load4(wB + 4 * (int64_t)e, b);
    load2(wC + 2 * (int64_t)e, c);
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      axpy2(v[i], a[0], g[i]);
      axpy2(v[3], a[1 + i], g[i]);
    }
    axpy2(v[3], kap * a[0], g[3]);
    axpy2(v[4], b[1], g[2]);
    axpy2(v[4], -b[2], g[1]);
    axpy2(v[5], b[2], g[0]);
    axpy2(v[5], -b[0], g[2]);
    axpy2(v[6], b[0], g[1]);
    axpy2(v[6], -b[1], g[0]);
    axpy2(v[7], b[3], g[0]);
    axpy2(v[7], c[0], g[1]);
    axpy2(v[7], c[1], g[2]);
    if (s0 >= 0) {
      R p[4], r[4];
      load4(sA + 4 * (int64_t)e, p);
      load4(sB + 4 * (int64_t)e, r);
      if (!isM) {  // A + grad phi / k^2
        const R f = ik2;
#pragma unroll
        for (int i = 0; i < 3; ++i) {
          axpy2(z[i], p[0], g[i]);
          axpy2(z[i], f * p[1 + i], g[3]);
          axpy2(z[3], r[i], g[i]);
        }
        axpy2(z[3], f * r[3], g[3]);
      } else {  // curl F
        axpy2(z[0], p[2], g[2]);
        axpy2(z[0], -p[3], g[1]);
        axpy2(z[1], p[3], g[0]);
        axpy2(z[1], -p[1], g[2]);
        axpy2(z[2], p[1], g[1]);
        axpy2(z[2], -p[2], g[0]);
#pragma unroll
        for (int i = 0; i < 3; ++i) axpy2(z[3], r[i], g[i]);
      }
    }
  }
  halve(v, 4, lane, 16);
  halve(v, 2, lane, 8);
  halve(v, 1, lane, 4);
  cx<R>* rw = red[warp];
  rw[grp * 12 + ((lane >> 2) & 4) + ((lane >> 2) & 2) + ((lane >> 2) & 1)] = v[0];
  if (s0 >= 0) {
    halve(z, 2, lane, 16);
    halve(z, 1, lane, 8);
    z[0] = xadd(z[0], 4);
    if (!(lane & 4)) rw[grp * 12 + 8 + ((lane >> 3) & 2) + ((lane >> 3) & 1)] = z[0];
  }
  __syncwarp();
  if (lane < 12) {
    const int kk = lane >> 2, ty = lane & 3;
    R gk[4], nr[4];
    load4(geo + 16 * t + 4 * kk, gk);
    load4(geo + 16 * t + 12, nr);
    const cx<R>*eJ = rw, *eM = rw + 12, *iJ = rw + 24, *iM = rw + 36;
    cx<R> o = czero<R>();
    if (ty < 3) {
      cx<R> f[4];
#pragma unroll
      for (int c = 0; c < 4; ++c)
        f[c] = ty == 0 ? mulj((zi * ki) * iJ[c] - (ze * ke) * eJ[c]) - eM[4 + c] + iM[4 + c]
                       : eJ[4 + c] - iJ[4 + c] + mulj((ki / zi) * iM[c] - (ke / ze) * eM[c]);
      o = gk[0] * (f[3] - (gk[1] * f[0] + gk[2] * f[1] + gk[3] * f[2]));
    }
    if (ty >= 2 && s0 >= 0) {
      const bool in = ty == 3;
      const R zk = in ? zi * ki : ze * ke;
      const cx<R>*J = (in ? iJ : eJ) + 8, *M = (in ? iM : eM) + 8;
      cx<R> f[4];
#pragma unroll
      for (int c = 0; c < 4; ++c) f[c] = -(zk * mulj(J[c])) - M[c];
      R x[3] = {gk[1], gk[2], gk[3]};
      if (!in) {  // n x rel_kk
        x[0] = nr[1] * gk[3] - nr[2] * gk[2];
        x[1] = nr[2] * gk[1] - nr[0] * gk[3];
        x[2] = nr[0] * gk[2] - nr[1] * gk[1];
      }
      o -= gk[0] * (f[3] - (x[0] * f[0] + x[1] * f[1] + x[2] * f[2]));
    }
    val[blockIdx.y * cs_v + t * 12 + lane] = o;
  }
}

// ================================================================ transposed apply
// x_bar = A^T y_bar: the stages of the apply in reverse order, each the
// transpose of its forward map (no conjugation):
//   T1 k_points_adj   rows -> tested values -> record adjoints at every point
//                     (Eqs. 1-3, 13, 14 testing transposed) and the
//                     triangle's own side-limit terms -> its summary adjoints
//   T2 k_near_adj_*   record adjoints of the targets -> summary adjoints of
//                     the source triangles (near records transposed): per
//                     pair over each target's record run, then per source
//                     over its reverse pair list (no atomics)
//   T3 k_interp_adj   record adjoints -> 16 grid fields (value and derivative
//                     stencils transposed), as a gather over covered points
//   T4 fft_conv(adjoint): each field with its medium's Green function
//   T5 k_proj_adj     grid -> point-source adjoints (value stencils
//                     transposed) -> summary adjoints (source expansion
//                     transposed), plus T1 + T2
//   T6 k_x_adj        summary adjoints -> unknowns (current expansion transposed)

// T1: one warp per triangle t.  Phase 1, lane (kk, a): the adjoints of the
// point-a quantities that the tested values of local edge kk read
// (u_type = w * ybar of the row, X = X_kk):
//   WE: X u0, wE: divX u0, WH: X (u1 + u2), wH: divX (u1 + u2),
//   E_e: -sg (n x X) u2, E_i: -sg X u3,
//   J_e + J_i: (n x X) u2 / 2 + X u3, M: sg (-X u2 + (n x X) u3) / 2.
// Phase 2, lane (a, medium, group): summed over kk, mapped to the 10 record
// values of the group (the transposes of medium_fields' combinations).
// Phase 3, lane (set, a | beta component): the own-summary adjoints summed
// over the points.
template <typename R>
__global__ void __launch_bounds__(PT_WARPS * 32)
    k_points_adj(const cx<R>* __restrict__ ybar, const int32_t* __restrict__ valrow, const double* __restrict__ tri,
                 const R* __restrict__ tp, const R* __restrict__ sig, int64_t nt, int q, R ke, R ki, R ze, R zi,
                 cx<R>* __restrict__ recb, cx<R>* __restrict__ sdir) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  constexpr int NA = 20;  // adjoint quantities per (kk, point)
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t t = (int64_t)blockIdx.x * PT_WARPS + warp;
  if (t >= nt) return;
  cx<R>* part = reinterpret_cast<cx<R>*>(smem_raw) + (int64_t)warp * 3 * q * NA;  // [kk][a][NA]
  const double* g = tri + 16 * t;
  const R nrm[3] = {(R)g[12], (R)g[13], (R)g[14]};
  if (lane < 3 * q) {
    const int kk = lane / q, pa = lane - kk * q;
    const int64_t Qa = t * q + pa;
    const R* tq = tp + 16 * Qa;
    const R w = tq[3], sg = sig[Qa], divX = tq[13 + kk];
    const R X[3] = {tq[4 + 3 * kk], tq[5 + 3 * kk], tq[6 + 3 * kk]};
    const R nX[3] = {nrm[1] * X[2] - nrm[2] * X[1], nrm[2] * X[0] - nrm[0] * X[2], nrm[0] * X[1] - nrm[1] * X[0]};
    cx<R> u[4];
#pragma unroll
    for (int ty = 0; ty < 4; ++ty) {
      const int row = valrow[(t * 3 + kk) * 4 + ty];
      u[ty] = row >= 0 ? w * ybar[row] : czero<R>();
    }
    const cx<R> u12 = u[1] + u[2];
    cx<R>* o = part + (int64_t)(kk * q + pa) * NA;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      o[c] = X[c] * u[0];
      o[4 + c] = X[c] * u12;
      o[8 + c] = (-sg * nX[c]) * u[2];
      o[11 + c] = (-sg * X[c]) * u[3];
      o[14 + c] = (R(0.5) * nX[c]) * u[2] + X[c] * u[3];
      o[17 + c] = (R(0.5) * sg) * (nX[c] * u[3] - X[c] * u[2]);
    }
    o[3] = divX * u[0];
    o[7] = divX * u12;
  }
  __syncwarp();
  if (lane < 4 * q) {
    const int pa = lane >> 2, m = (lane >> 1) & 1, h = lane & 1;
    cx<R> ag[NA];
#pragma unroll
    for (int i = 0; i < NA; ++i) ag[i] = czero<R>();
    for (int kk = 0; kk < 3; ++kk) {
      const cx<R>* o = part + (int64_t)(kk * q + pa) * NA;
#pragma unroll
      for (int i = 0; i < 14; ++i) ag[i] += o[i];
    }
    const R k = m ? ki : ke, z = m ? zi : ze, sgm = m ? R(-1) : R(1);
    const cx<R>* Eb = ag + (m ? 11 : 8);
    cx<R> r[10];
    if (h == 0) {  // A, phi, grad phi, curl A
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        r[c] = (sgm * (-z * k)) * mulj(ag[c]) + (-z * k) * mulj(Eb[c]);
        r[4 + c] = (-z / k) * mulj(Eb[c]);
        r[7 + c] = sgm * ag[4 + c];
      }
      r[3] = (sgm * z / k) * mulj(ag[3]);
    } else {  // F, psi, grad psi (unused by the rows), curl F
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        r[c] = (-sgm * k / z) * mulj(ag[4 + c]);
        r[4 + c] = czero<R>();
        r[7 + c] = -(sgm * ag[c]) - Eb[c];
      }
      r[3] = (sgm / (k * z)) * mulj(ag[7]);
    }
    cx<R>* dst = recb + ((t * q + pa) * 2 + m) * NREC + 10 * h;
#pragma unroll
    for (int c = 0; c < 10; ++c) dst[c] = r[c];
  }
  __syncwarp();
  if (lane < 12) {
    const int set = lane >> 2, comp = lane & 3;
    const int base = set < 2 ? 14 : 17;  // J_e + J_i feeds sets 0 and 1, M set 2
    cx<R> acc = czero<R>();
    for (int pa = 0; pa < q; ++pa) {
      cx<R> v[3];
#pragma unroll
      for (int c = 0; c < 3; ++c)
        v[c] = part[(0 * q + pa) * NA + base + c] + part[(1 * q + pa) * NA + base + c] +
               part[(2 * q + pa) * NA + base + c];
      const R* tq = tp + 16 * (t * q + pa);
      if (comp == 0)
        acc += tq[0] * v[0] + tq[1] * v[1] + tq[2] * v[2];  // a: J = a (r - c) - beta
      else
        acc -= v[comp - 1];
    }
    sdir[(t * 3 + set) * 4 + comp] = acc;
  }
}

// T2a: one warp per target triangle t over its own near pairs (one
// contiguous run of records).  The pairs stream through a per-warp ring of
// NA_NSTG stages of NA_KP pairs (one bulk copy per pair into a slot padded to
// na_slot(q) complex values, so that the 16 (pair, point, medium) rows a warp
// load touches fall in distinct banks; bounded waits).  The target's record
// adjoints (q points x 2 media x 20) sit in shared memory.  Lane (pair k,
// point half ah, medium m, group h) forms, for pair k of the stage, the
// transpose of near_part summed over its points a = ah, ah + NA_AH, ...:
//   a_bar = sum_a r . dP1 + 2 phi_r dP0 + 2 grad_r . dQ + curl_r . dC,
//   beta_bar = sum_a -A_r dP0 - (the dQ x beta term transposed);
// the point halves are summed by one xor shuffle, and the pair's 12
// contributions are the per-set values J_e = (exterior, J), J_i = (interior,
// J), M = (exterior, M) - (interior, M).
constexpr int NA_AH = 2;  // lanes sharing one pair's points (1 or 2)
constexpr int NA_KP = 8 / NA_AH;
constexpr int NA_NSTG = 2;
__host__ __device__ __forceinline__ int na_slot(int q) {
  const int pc = NCORR * 2 * q;
  return pc + (((2 * NA_AH - pc) % 16) + 16) % 16;
}
__host__ __device__ __forceinline__ int na_warp_cx(int q) { return NA_NSTG * NA_KP * na_slot(q) + 40 * q; }
template <typename R>
__global__ void __launch_bounds__(PT_WARPS * 32, 4)
    k_near_adj_pairs(const cx<R>* __restrict__ corr, const int32_t* __restrict__ noff, const cx<R>* __restrict__ recb,
                     int64_t nt, int q, cx<R>* __restrict__ contrib, int* __restrict__ tmo) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t t = (int64_t)blockIdx.x * PT_WARPS + warp;
  if (t >= nt) return;  // whole warp
  const int pairc = NCORR * 2 * q, slot = na_slot(q), wcx = na_warp_cx(q);
  cx<R>* ring = reinterpret_cast<cx<R>*>(smem_raw) + (int64_t)warp * wcx;
  cx<R>* rt = ring + NA_NSTG * NA_KP * slot;
  uint64_t* bars = reinterpret_cast<uint64_t*>(reinterpret_cast<cx<R>*>(smem_raw) + PT_WARPS * wcx) + warp * NA_NSTG;
  const int j0 = noff[t], j1 = noff[t + 1];
  const int nst = (j1 - j0 + NA_KP - 1) / NA_KP;
  if (nst == 0) return;
  const unsigned pair_bytes = (unsigned)(pairc * sizeof(cx<R>));
  auto issue = [&](int st) {
    const int pj = j0 + st * NA_KP;
    const int np = min(NA_KP, j1 - pj);
    uint64_t* b = bars + st % NA_NSTG;
    fence_proxy_async();
    mbar_expect_tx(b, np * pair_bytes);
    for (int k = 0; k < np; ++k)
      bulk_copy(ring + ((st % NA_NSTG) * NA_KP + k) * slot, corr + (int64_t)(pj + k) * pairc, pair_bytes, b);
  };
  if (lane == 0) {
#pragma unroll
    for (int i = 0; i < NA_NSTG; ++i) mbar_init(bars + i, 1);
    mbar_init_fence();
    for (int st = 0; st < NA_NSTG - 1 && st < nst; ++st) issue(st);
  }
  {
    const cx<R>* rs = recb + t * q * 40;
    for (int u = lane; u < 40 * q; u += 32) rt[u] = rs[u];
  }
  __syncwarp();
  const int k = lane / (4 * NA_AH), ah = (lane >> 2) & (NA_AH - 1), m = (lane >> 1) & 1, h = lane & 1;
  const cx<R>* rl = rt + m * NREC + 10 * h;
  int st = 0;
  bool ok = true;
  for (; st < nst; ++st) {
    if (lane == 0 && st + NA_NSTG - 1 < nst) issue(st + NA_NSTG - 1);
    ok = __all_sync(0xffffffffu, mbar_wait(bars + st % NA_NSTG, (st / NA_NSTG) & 1));
    if (!ok) break;
    const int j = j0 + st * NA_KP + k;
    const cx<R>* dp = ring + ((st % NA_NSTG) * NA_KP + k) * slot + m * NCORR;
    cx<R> al = czero<R>(), be[3] = {czero<R>(), czero<R>(), czero<R>()};
    if (j < j1) {
      for (int a = ah; a < q; a += NA_AH) {
        cx<R> r[10], d[NCORR];
#pragma unroll
        for (int c = 0; c < 10; c += 2) load_pair_smem(rl + a * 40 + c, r + c);
#pragma unroll
        for (int c = 0; c < NCORR; c += 2) load_pair_smem(dp + a * 2 * NCORR + c, d + c);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          cfma(al, r[c], d[1 + c]);
          cfma(al, R(2) * r[4 + c], d[4 + c]);
          cfma(al, r[7 + c], d[7 + c]);
          be[c] -= r[c] * d[0];
        }
        cfma(al, R(2) * r[3], d[0]);
        be[0] += r[9] * d[5] - r[8] * d[6];
        be[1] += r[7] * d[6] - r[9] * d[4];
        be[2] += r[8] * d[4] - r[7] * d[5];
      }
    }
    cx<R> v[4] = {al, be[0], be[1], be[2]};
    if (NA_AH == 2)  // the two point halves (lane bit 2)
#pragma unroll
      for (int c = 0; c < 4; ++c)
        v[c] += mk(__shfl_xor_sync(0xffffffffu, v[c].re, 4), __shfl_xor_sync(0xffffffffu, v[c].im, 4));
    // (exterior, M) - (interior, M): lanes h = 1 differ in bit 1 (medium)
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const cx<R> o = mk(__shfl_xor_sync(0xffffffffu, v[c].re, 2), __shfl_xor_sync(0xffffffffu, v[c].im, 2));
      if (h) v[c] -= o;
    }
    if (j < j1 && ah == 0 && (h == 0 || m == 0)) {
      cx<R>* cj = contrib + (int64_t)j * 12 + (h ? 8 : 4 * m);
#pragma unroll
      for (int c = 0; c < 4; ++c) cj[c] = v[c];
    }
    __syncwarp();
  }
  if (!ok) {
    for (int s2 = st; s2 < nst && s2 < st + NA_NSTG; ++s2) (void)mbar_wait(bars + s2 % NA_NSTG, (s2 / NA_NSTG) & 1);
    if (lane == 0) atomicOr(tmo, 1);
  }
}

// T2b: thread per (source triangle s, set, component): sdir plus the pair
// contributions of the pairs whose source is s, in reverse-list order.
template <typename R>
__global__ void k_near_adj_sum(const int32_t* __restrict__ roff, const int32_t* __restrict__ rpair,
                               const cx<R>* __restrict__ contrib, const cx<R>* __restrict__ sdir, int64_t nt,
                               cx<R>* __restrict__ snear) {
  const int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (idx >= nt * 12) return;
  const int64_t sidx = idx / 12;
  const int c = (int)(idx - sidx * 12);
  cx<R> acc = sdir[idx];
  for (int rp = roff[sidx]; rp < roff[sidx + 1]; ++rp) acc += contrib[(int64_t)rpair[rp] * 12 + c];
  snear[idx] = acc;
}

// T3: one warp per covered grid point i.  Lane pr < 20 reads the 16-byte
// portion pr of the 320-byte record-adjoint row of every entry of the point
// (records 2 pr, 2 pr + 1 of the 40 = 2 media x 2 groups x 10; one coalesced
// row per load instruction, IADJ_INFLIGHT rows in flight) and accumulates
// each record against all four entry weights (value W, derivatives Wx, Wy,
// Wz).  The transposed interpolation of one group (records r0..r9) is then a
// fixed combination of those sums:
//   f0 = W r0 + Wz r8 - Wy r9,  f1 = W r1 - Wz r7 + Wx r9,
//   f2 = W r2 + Wy r7 - Wx r8,  f3 = W r3 + Wx r4 + Wy r5 + Wz r6,
// formed by lanes 0..15 (group g4, field f) and written field-major.
constexpr int IADJ_INFLIGHT = 4;
template <typename R>
__global__ void __launch_bounds__(256) k_interp_adj(const cx<R>* __restrict__ recb, const int32_t* __restrict__ gpt,
                                                    const int32_t* __restrict__ goff, const int32_t* __restrict__ gq,
                                                    const R* __restrict__ gw, const R* __restrict__ gd,
                                                    int64_t ngnz, int64_t ng, cx<R>* __restrict__ grids) {
  __shared__ cx<R> red[8][20][8];  // [warp in CTA][portion][record k * 4 + weight]
  const int64_t i = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31, wl = threadIdx.x >> 5;
  const bool act = lane < 20 && i < ngnz;
  cx<R> acc[8];
#pragma unroll
  for (int c = 0; c < 8; ++c) acc[c] = czero<R>();
  if (act) {
    const int e1 = goff[i + 1];
    for (int e = goff[i]; e < e1; e += IADJ_INFLIGHT) {
      int qe[IADJ_INFLIGHT];
      R w[IADJ_INFLIGHT][4];
#pragma unroll
      for (int u = 0; u < IADJ_INFLIGHT; ++u) {
        const int eu = e + u < e1 ? e + u : e;
        const R on = e + u < e1 ? R(1) : R(0);
        qe[u] = gq[eu];
        w[u][0] = on * gw[eu];
#pragma unroll
        for (int c = 0; c < 3; ++c) w[u][1 + c] = on * gd[3 * (int64_t)eu + c];
      }
      cx<R> v[IADJ_INFLIGHT][2];
#pragma unroll
      for (int u = 0; u < IADJ_INFLIGHT; ++u) load_pair(recb + (int64_t)qe[u] * (2 * NREC) + 2 * lane, v[u]);
#pragma unroll
      for (int u = 0; u < IADJ_INFLIGHT; ++u)
#pragma unroll
        for (int k = 0; k < 2; ++k)
#pragma unroll
          for (int c = 0; c < 4; ++c) axpy2(acc[k * 4 + c], w[u][c], v[u][k]);
    }
  }
  if (lane < 20)
#pragma unroll
    for (int c = 0; c < 8; ++c) red[wl][lane][c] = acc[c];
  __syncwarp();
  if (lane < 16 && i < ngnz) {
    // record 10 h + r of group g4 = 2 m + h sits in portion 5 g4 + r / 2,
    // slot (r & 1) * 4 + weight; weights 0 W, 1 Wx, 2 Wy, 3 Wz
    const int g4 = lane >> 2, f = lane & 3;
    const cx<R>(*rp)[8] = red[wl] + 5 * g4;
#define RW(r, wt) rp[(r) >> 1][((r) & 1) * 4 + (wt)]
    cx<R> o;
    switch (f) {
      case 0: o = RW(0, 0) + RW(8, 3) - RW(9, 2); break;
      case 1: o = RW(1, 0) - RW(7, 3) + RW(9, 1); break;
      case 2: o = RW(2, 0) + RW(7, 2) - RW(8, 1); break;
      default: o = RW(3, 0) + RW(4, 1) + RW(5, 2) + RW(6, 3); break;
    }
#undef RW
    grids[(int64_t)lane * ng + gpt[i]] = o;
  }
}

// T5: one warp per triangle t; lane (point a, set): the transposed value
// interpolation of the convolved adjoint grid (point-major; J_e from fields
// 0..3, J_i from 8..11, M from 4..7 minus 12..15), then the transposed point
// sources (a_bar += w (r - c) . qb + 2 w qb_div, beta_bar -= w qb), summed
// over the points in point order and added to snear.
template <typename R, int P>
__global__ void __launch_bounds__(PT_WARPS * 32)
    k_proj_adj(const cx<R>* __restrict__ grids, const int32_t* __restrict__ base, const R* __restrict__ L,
               const R* __restrict__ tp, const cx<R>* __restrict__ snear, int64_t nt, int q, int n1, int n2,
               cx<R>* __restrict__ stot) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t t = (int64_t)blockIdx.x * PT_WARPS + warp;
  if (t >= nt) return;
  cx<R>* red = reinterpret_cast<cx<R>*>(smem_raw) + (int64_t)warp * 32 * 4;  // [lane][4]
  if (lane < 3 * q) {
    const int pa = lane / 3, set = lane - pa * 3;
    const int64_t Qi = t * q + pa;
    R Lx[P], Ly[P], Lz[P];
#pragma unroll
    for (int i = 0; i < P; ++i) {
      Lx[i] = L[(3 * Qi + 0) * P + i];
      Ly[i] = L[(3 * Qi + 1) * P + i];
      Lz[i] = L[(3 * Qi + 2) * P + i];
    }
    const int b0 = base[3 * Qi], b1 = base[3 * Qi + 1], b2 = base[3 * Qi + 2];
    const int fa = set == 0 ? 0 : (set == 1 ? 8 : 4);
    cx<R> qb[4] = {czero<R>(), czero<R>(), czero<R>(), czero<R>()};
#pragma unroll
    for (int i = 0; i < P; ++i)
#pragma unroll
      for (int j = 0; j < P; ++j) {
        const R wxy = Lx[i] * Ly[j];
        const int64_t rowi = ((int64_t)(b0 + i) * n1 + (b1 + j)) * n2 + b2;
#pragma unroll
        for (int k = 0; k < P; ++k) {
          const R W = wxy * Lz[k];
          cx<R> gv[4];
          load_group(grids + (rowi + k) * NFIELD_OUT + fa, gv);
          if (set == 2) {
            cx<R> gi[4];
            load_group(grids + (rowi + k) * NFIELD_OUT + 12, gi);
#pragma unroll
            for (int f = 0; f < 4; ++f) gv[f] -= gi[f];
          }
#pragma unroll
          for (int f = 0; f < 4; ++f) axpy(qb[f], W, gv[f]);
        }
      }
    const R* tq = tp + 16 * Qi;
    const R w = tq[3];
    red[lane * 4 + 0] = w * (tq[0] * qb[0] + tq[1] * qb[1] + tq[2] * qb[2]) + (R(2) * w) * qb[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) red[lane * 4 + 1 + c] = -(w * qb[c]);
  }
  __syncwarp();
  if (lane < 12) {
    const int set = lane >> 2, comp = lane & 3;
    cx<R> acc = snear[(t * 3 + set) * 4 + comp];
    for (int pa = 0; pa < q; ++pa) acc += red[(pa * 3 + set) * 4 + comp];
    stot[(t * 3 + set) * 4 + comp] = acc;
  }
}

// T6: thread per unknown: x_bar = sum over its uses (triangle t, local edge k,
// set, sign) of sign cX_k (a_bar + (v_k - c) . beta_bar).
template <typename R>
__global__ void k_x_adj(const cx<R>* __restrict__ stot, const int32_t* __restrict__ xsrc,
                        const double* __restrict__ tri, const double* __restrict__ cX, int64_t N,
                        cx<R>* __restrict__ xbar) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= N) return;
  cx<R> acc = czero<R>();
  for (int u = 0; u < 4; ++u) {
    const int32_t code = xsrc[4 * i + u];
    if (code == 0) break;
    const int64_t c = (code > 0 ? code : -code) - 1;
    const int set = (int)(c % 3);
    const int64_t tk = c / 3, t = tk / 3;
    const int k = (int)(tk - t * 3);
    const double* g = tri + 16 * t;
    const cx<R>* sb = stot + (t * 3 + set) * 4;
    cx<R> v = sb[0];
#pragma unroll
    for (int cc = 0; cc < 3; ++cc) v += (R)(g[3 * k + cc] - g[9 + cc]) * sb[1 + cc];
    const R f = (R)cX[3 * t + k] * (code > 0 ? R(1) : R(-1));
    acc += f * v;
  }
  xbar[i] = acc;
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

}  // namespace

// The grid part up to the potentials, for k right-hand sides: summaries,
// projection, convolution.
template <typename R>
int grid_potentials(scabem_op* op, const cx<R>* x, int64_t ldx, int k, cudaStream_t s) {
  PrecData<R>& pd = pdata<R>(op);
  const int64_t ng = (int64_t)op->n[0] * op->n[1] * op->n[2];
  prof_mark(op, s);
  k_summ<R><<<dim3((unsigned)cdiv(3 * op->nt, 128), k), 128, 0, s>>>(x, op->unk, pd.geo, op->nt, pd.summ, ldx);
  CK(cudaGetLastError());
  prof_mark(op, s);
  k_project<R><<<dim3((unsigned)cdiv(op->ngnz * 32, 256), k), 256, 0, s>>>(
      pd.summ, op->gpt, op->eoff, op->gtri, pd.gA, op->ngnz, ng, pd.src, col_stride_summ(op), col_stride_grid(op));
  CK(cudaGetLastError());
  prof_mark(op, s);
  return fft_conv<R>(op, pd, s, false, k);
}

template <typename R>
int apply_batch(scabem_op* op, const cx<R>* x, int64_t ldx, cx<R>* y, int64_t ldy, int k, cudaStream_t s) {
  PrecData<R>& pd = pdata<R>(op);
  if (k < 1 || k > KBATCH || k > pd.kcap) {
    set_error("apply_batch: batch size outside the workspace capacity");
    return SCABEM_E_ARG;
  }
  if (int rc = grid_potentials<R>(op, x, ldx, k, s)) return rc;
  prof_mark(op, s);
  k_test<R><<<dim3((unsigned)cdiv(op->nt, TS_WARPS), k), TS_WARPS * 32, 0, s>>>(
      pd.grid, op->toff, op->tgi, op->soff, pd.wA, pd.wB, pd.wC, pd.sW, op->nsent, pd.geo, op->nt, (R)op->ke, (R)op->ki,
      (R)op->ze, (R)op->zi, pd.val, col_stride_grid(op), col_stride_val(op));
  CK(cudaGetLastError());
  if (int rc = near_rows<R>(op, x, ldx, y, ldy, k, s)) return rc;
  prof_mark(op, s);
  return SCABEM_OK;
}

template <typename R>
int apply_one(scabem_op* op, const cx<R>* x, cx<R>* y, cudaStream_t s) {
  return apply_batch<R>(op, x, op->N, y, op->N, 1, s);
}

template <typename R>
using ProjAdjFn = void (*)(const cx<R>*, const int32_t*, const R*, const R*, const cx<R>*, int64_t, int, int, int,
                           cx<R>*);

// x_bar = A^T y_bar (one right-hand side), stages T1-T6.
template <typename R>
int apply_adjoint_one(scabem_op* op, const cx<R>* ybar, cx<R>* xbar, cudaStream_t s) {
  PrecData<R>& pd = pdata<R>(op);
  const int64_t nt = op->nt;
  const int q = op->q;
  const int64_t ng = (int64_t)op->n[0] * op->n[1] * op->n[2];
  cx<R>* sdir = pd.sbar;
  cx<R>* snear = pd.sbar + nt * 12;
  const int blocks = (int)cdiv(nt, PT_WARPS);
  {
    const size_t sm = (size_t)PT_WARPS * 3 * q * 20 * sizeof(cx<R>);
    if (int rc_ = set_max_smem(op->device, (const void*)k_points_adj<R>, (int)sm)) return rc_;
    k_points_adj<R><<<blocks, PT_WARPS * 32, sm, s>>>(ybar, op->valrow, op->tri, pd.tp, pd.sig, nt, q, (R)op->ke,
                                                      (R)op->ki, (R)op->ze, (R)op->zi, pd.recb, sdir);
    CK(cudaGetLastError());
  }
  const cx<R>* s_after_near = sdir;
  if (op->npairs > 0) {
    const size_t sm = (size_t)PT_WARPS * na_warp_cx(q) * sizeof(cx<R>) + (size_t)PT_WARPS * NA_NSTG * sizeof(uint64_t);
    if (int rc_ = set_max_smem(op->device, (const void*)k_near_adj_pairs<R>, (int)sm)) return rc_;
    k_near_adj_pairs<R><<<blocks, PT_WARPS * 32, sm, s>>>(pd.near, op->noff, pd.recb, nt, q, pd.nadj, op->tmo_d);
    CK(cudaGetLastError());
    k_near_adj_sum<R><<<(int)cdiv(nt * 12, 256), 256, 0, s>>>(op->roff, op->rpair, pd.nadj, sdir, nt, snear);
    CK(cudaGetLastError());
    s_after_near = snear;
  }
  if (op->ngnz > 0) {
    k_interp_adj<R><<<(int)cdiv(op->ngnz * 32, 256), 256, 0, s>>>(pd.recb, op->gpt, op->goff, op->gent,
                                                                 gather_weights<R>(op), gather_dweights<R>(op),
                                                                 op->ngnz, ng, pd.src);
    CK(cudaGetLastError());
  }
  int rc = fft_conv<R>(op, pd, s, true);
  if (rc) return rc;
  {
    const size_t sm = (size_t)PT_WARPS * 32 * 4 * sizeof(cx<R>);
    ProjAdjFn<R> fn = op->p == 2 ? k_proj_adj<R, 2> : op->p == 3 ? k_proj_adj<R, 3> : k_proj_adj<R, 4>;
    fn<<<blocks, PT_WARPS * 32, sm, s>>>(pd.grid, op->base, pd.L, pd.tp, s_after_near, nt, q, op->n[1], op->n[2],
                                         sdir);
    CK(cudaGetLastError());
  }
  k_x_adj<R><<<(int)cdiv(op->N, 256), 256, 0, s>>>(sdir, op->xsrc, op->tri, op->cX, op->N, xbar);
  CK(cudaGetLastError());
  return SCABEM_OK;
}

// hs[p] = d(lam^T A x)/d sigma_p [per S] at every quadrature point
// (complex128): the apply's stages up to the records, then the derivative
// of the sigma-weighted testing (k_points in its sensitivity mode).
int sigma_sensitivity_op(scabem_op* op, const cx<double>* x, const cx<double>* lam, cx<double>* hs,
                         cudaStream_t s) {
  PrecData<double>& pd = op->d;
  if (int rc = grid_potentials<double>(op, x, op->N, 1, s)) return rc;
  prof_mark(op, s);
  const size_t sm = pt_smem_bytes(op->q, sizeof(cx<double>));
  auto fn = op->p == 2 ? k_points_sens<double, 2> : op->p == 3 ? k_points_sens<double, 3> : k_points_sens<double, 4>;
  if (int rc_ = set_max_smem(op->device, (const void*)fn, (int)sm)) return rc_;
  fn<<<(int)cdiv(op->nt, PT_WARPS), PT_WARPS * 32, sm, s>>>(
      pd.grid, op->base, pd.L, pd.dL, pd.near, op->noff, op->nsrc, pd.summ, op->tri, pd.tp, op->nt, op->q, op->n[1],
      op->n[2], op->ke, op->ki, op->ze, op->zi, op->npairs > 0 ? 1 : 0, op->valrow, op->tmo_d, lam, hs);
  CK(cudaGetLastError());
  prof_mark(op, s);
  return SCABEM_OK;
}

int selftest_wait(scabem_op* op, cudaStream_t s) {
  k_wait_selftest<<<1, 32, 0, s>>>(op->tmo_d);
  CK(cudaGetLastError());
  CK(cudaStreamSynchronize(s));
  return SCABEM_OK;
}

// Current summaries only (used by the field evaluation at probe points).
template <typename R>
int compute_summ(scabem_op* op, const cx<R>* x, cx<R>* summ, cudaStream_t s) {
  k_summ<R><<<(int)cdiv(3 * op->nt, 128), 128, 0, s>>>(x, op->unk, pdata<R>(op).geo, op->nt, summ, op->N);
  CK(cudaGetLastError());
  return SCABEM_OK;
}

template int compute_summ<double>(scabem_op*, const cx<double>*, cx<double>*, cudaStream_t);
template int apply_one<float>(scabem_op*, const cx<float>*, cx<float>*, cudaStream_t);
template int apply_adjoint_one<float>(scabem_op*, const cx<float>*, cx<float>*, cudaStream_t);
template int apply_adjoint_one<double>(scabem_op*, const cx<double>*, cx<double>*, cudaStream_t);
template int apply_one<double>(scabem_op*, const cx<double>*, cx<double>*, cudaStream_t);
template int apply_batch<float>(scabem_op*, const cx<float>*, int64_t, cx<float>*, int64_t, int, cudaStream_t);
template int apply_batch<double>(scabem_op*, const cx<double>*, int64_t, cx<double>*, int64_t, int, cudaStream_t);
