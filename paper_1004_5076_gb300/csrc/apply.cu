// The matvec y = A x of the grid-accelerated operator, for one right-hand side or
// a batch of up to eight, and its transpose.
//
//  K1 k_project  RWG coefficients -> point sources on the grid (12 fields: the
//                exterior J, interior J and exterior M sets, current reduction
//                of Eqs. 10-12), through the edge stencils (stencil.cu), as a
//                gather over the covered grid points
//  K2-3          fft_conv (fft.cu): 12 -> 16 grid potentials (A, phi, F, psi
//                of each medium, Eqs. 15-16), written as the combinations that
//                the rows test
//  K4 k_rows     (near.cu) Galerkin rows of Eqs. 1-3 (weak form), Eq. 13 and
//                Eq. 14 (sigma-weighted): the potentials tested through the same
//                edge stencils, plus the near-field precorrection (exact minus
//                grid panel interaction) and the side-limit terms as a sparse
//                matrix over edges
#include <cuda_runtime.h>

#include "device.cuh"

namespace {

template <typename R>
__device__ __forceinline__ cx<R> coef_of(const cx<R>* __restrict__ x, int32_t code) {
  if (code > 0) return x[code - 1];
  if (code < 0) return -x[-code - 1];
  return czero<R>();
}

// One thread per (triangle, set): the current summary
// summ[(t*3+set)*4 + {a, bx, by, bz}], J(r) = a (r - c_t) - beta, of the
// exterior J, interior J and exterior M sets (current reduction, Eqs. 10-12).
template <typename R>
__global__ void k_summ(const cx<R>* __restrict__ x, const int32_t* __restrict__ unk, const double* __restrict__ cX,
                       const double* __restrict__ tri, int64_t nt, cx<R>* __restrict__ summ) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= 3 * nt) return;
  const int64_t t = i / 3;
  const int set = (int)(i - 3 * t);
  const double* g = tri + 16 * t;
  cx<R> a = czero<R>(), b[3] = {a, a, a};
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const cx<R> j = (R)cX[3 * t + k] * coef_of(x, unk[(3 * t + k) * 3 + set]);
    a += j;
#pragma unroll
    for (int c = 0; c < 3; ++c) axpy(b[c], (R)(g[3 * k + c] - g[9 + c]), j);
  }
  cx<R>* o = summ + 4 * i;
  o[0] = a;
#pragma unroll
  for (int c = 0; c < 3; ++c) o[1 + c] = b[c];
}

// K1: projection, as a gather over the edges.  One warp per covered grid
// point: lane = slot * 4 + component takes entries slot, slot + 8, ... of the
// point, the component (x, y, z, div) of the edge's value block Q0 (stencil.cu)
// against the edge's unknowns.  Plain edges come first and feed J_e and J_i =
// -J_e with one sum.  The slots meet by halving exchanges.  Points no stencil
// covers stay zero from set-up.  The sum order is fixed, so the result does not
// depend on thread timing.  Bound by the latency of the (edge -> unknown)
// loads out of L2.
// A warp takes K right-hand sides, which share the entries' weights and indices.
// 12 um guide: 24 us, 76 for 8 columns (33 and 188 as a gather of point sources
// behind a kernel that formed them in 13 and 56).
// LANES = 128 puts four warps on a point, for operators with few points
// (project_wide).
constexpr int PJ_THREADS = 128;

template <typename R, int K, int LANES>
__global__ void __launch_bounds__(PJ_THREADS) k_project(const cx<R>* x, int xst,
                                                        const int32_t* __restrict__ gp,
                                                        const int32_t* __restrict__ gpoff,
                                                        const int32_t* __restrict__ gpl,
                                                        const int32_t* __restrict__ gpr, const R* __restrict__ gq,
                                                        int64_t ngp, int64_t npt, int64_t nL, int64_t nR,
                                                        cx<R>* __restrict__ src, int64_t cs, int kc) {
  constexpr int ST = LANES / 4;  // slots
  const int64_t st = K == 1 ? 1 : xst;
  x += blockIdx.y * group_pad(K);  // group blockIdx.y of a batch of kc
  src += blockIdx.y * K * cs;
  kc = min(K, kc - (int)blockIdx.y * K);
  const int64_t i = (blockIdx.x * (int64_t)PJ_THREADS + threadIdx.x) / LANES;
  if (i >= ngp) return;  // whole warp; LANES = 128: no CTA
  const int lane = threadIdx.x & 31, comp = lane & 3, slot = (threadIdx.x % LANES) >> 2;
  const int e0 = gpoff[i], el = e0 + gpl[i], e1 = gpoff[i + 1];
  pdl_wait();
  cx<R> v[K][4];  // plain J, absorber J_e, absorber J_i, M
#pragma unroll
  for (int k = 0; k < K; ++k)
#pragma unroll
    for (int c = 0; c < 4; ++c) v[k][c] = czero<R>();
  auto plain = [&](R w, const cx<R>* a, const cx<R>* b) {
#pragma unroll
    for (int k = 0; k < K; ++k) {
      axpy2(v[k][0], w, a[k]);
      axpy2(v[k][3], w, b[k]);
    }
  };
  auto absorber = [&](R w, const cx<R>* a, const cx<R>* b, const cx<R>* d) {
#pragma unroll
    for (int k = 0; k < K; ++k) {
      axpy2(v[k][1], w, a[k]);
      axpy2(v[k][2], w, b[k]);
      axpy2(v[k][3], w, d[k]);
    }
  };
  if constexpr (LANES == 32) {  // many warps: few registers
    constexpr int UN = K == 1 ? 4 : K < 4 ? 2 : 1;
#pragma unroll UN
    for (int e = e0 + slot; e < el; e += ST) {
      const int64_t m = gpr[e];
      const R w = gq[4 * (int64_t)e + comp];
      cx<R> a[K], b[K];
      load_cols<R, K>(x + m * st, a);
      load_cols<R, K>(x + (m + nL) * st, b);
      plain(w, a, b);
    }
#pragma unroll UN
    for (int e = el + slot; e < e1; e += ST) {
      const int64_t m = nL + gpr[e];
      const R w = gq[4 * (int64_t)e + comp];
      cx<R> a[K], b[K], d[K];
      load_cols<R, K>(x + m * st, a);
      load_cols<R, K>(x + (m + nR) * st, b);
      load_cols<R, K>(x + (m + 2 * nR) * st, d);
      absorber(w, a, b, d);
    }
  } else {  // few entries per lane: all of a block's loads before the first use
    constexpr int IF = K == 1 ? 4 : 2;
    for (int e = e0 + slot; e < el; e += IF * ST) {
      cx<R> a[IF][K], b[IF][K];
      R w[IF];
#pragma unroll
      for (int u = 0; u < IF; ++u) {
        w[u] = R(0);
#pragma unroll
        for (int k = 0; k < K; ++k) a[u][k] = b[u][k] = czero<R>();
        if (e + u * ST < el) {
          const int64_t m = gpr[e + u * ST];
          w[u] = gq[4 * (int64_t)(e + u * ST) + comp];
          load_cols<R, K>(x + m * st, a[u]);
          load_cols<R, K>(x + (m + nL) * st, b[u]);
        }
      }
#pragma unroll
      for (int u = 0; u < IF; ++u) plain(w[u], a[u], b[u]);
    }
    for (int e = el + slot; e < e1; e += IF * ST) {
      cx<R> a[IF][K], b[IF][K], d[IF][K];
      R w[IF];
#pragma unroll
      for (int u = 0; u < IF; ++u) {
        w[u] = R(0);
#pragma unroll
        for (int k = 0; k < K; ++k) a[u][k] = b[u][k] = d[u][k] = czero<R>();
        if (e + u * ST < e1) {
          const int64_t m = nL + gpr[e + u * ST];
          w[u] = gq[4 * (int64_t)(e + u * ST) + comp];
          load_cols<R, K>(x + m * st, a[u]);
          load_cols<R, K>(x + (m + nR) * st, b[u]);
          load_cols<R, K>(x + (m + 2 * nR) * st, d[u]);
        }
      }
#pragma unroll
      for (int u = 0; u < IF; ++u) absorber(w[u], a[u], b[u], d[u]);
    }
  }
#pragma unroll
  for (int k = 0; k < K; ++k) {
    halve(v[k], 2, lane, 16);
    halve(v[k], 1, lane, 8);
    v[k][0] = xadd(v[k][0], 4);
  }
  if constexpr (LANES > 32) {
    __shared__ cx<R> sm[3][K][32];
    const int wp = threadIdx.x >> 5;
    if (wp > 0)
#pragma unroll
      for (int k = 0; k < K; ++k) sm[wp - 1][k][lane] = v[k][0];
    __syncthreads();
    if (wp > 0) return;
#pragma unroll
    for (int k = 0; k < K; ++k)
#pragma unroll
      for (int u = 0; u < 3; ++u) v[k][0] += sm[u][k][lane];
  }
  const int set = (lane >> 3) - 1;
#pragma unroll
  for (int k = 0; k < K; ++k) {
    // lane bits (4, 3) hold plain J, J_e, J_i, M: add the plain part to J_e and -J_i
    const cx<R> pe = shfl_xor_cx(v[k][0], 8), pi = shfl_xor_cx(v[k][0], 16);
    if (set < 0 || (lane & 4) || k >= kc) continue;
    const cx<R> o = set == 0 ? v[k][0] + pe : set == 1 ? v[k][0] - pi : v[k][0];
    src[k * cs + (int64_t)(4 * set + comp) * npt + gp[i]] = o;
  }
}

// x of a batch of k in the layout of load_cols: out[u][group][column], st = batch_stride(k)
template <typename R>
__global__ void __launch_bounds__(256) k_interleave(const cx<R>* x, int64_t ldx, int64_t N, int k, int K,
                                                    int st, cx<R>* __restrict__ out) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  pdl_wait();
  if (i >= N * st) return;
  const int64_t u = i / st;
  const int l = (int)(i - u * st), kp = group_pad(K), c = l / kp * K + l % kp;
  out[i] = l % kp < K && c < k ? x[c * ldx + u] : czero<R>();
}

// Two consecutive complex values of shared memory on a 16-byte boundary.
__device__ __forceinline__ void load_pair_smem(const cx<double>* p, cx<double>* v) {
  v[0] = p[0];
  v[1] = p[1];
}

// Interpolated potentials of one medium at quadrature point Qi, group h of
// the record (NREC = 2 x 10): h = 0 A(3) phi grad phi(3) curl A(3) from the
// J fields, h = 1 F(3) 0 0(3) curl F(3) from the M fields.  The potential grid
// is point-major, groups 4 .. 7 of a point hold the sets (fft.cu), [A, phi] with
// the factors j z k and j z / k, which are taken out again.
template <typename R, int p>
__device__ __forceinline__ void interp_group(const cx<R>* __restrict__ grids, const int32_t* __restrict__ base,
                                             const R* __restrict__ L, const R* __restrict__ dL, int64_t Qi, int med,
                                             int h, const int32_t* __restrict__ cmap, int n2, int nac, R k, R z,
                                             cx<R>* r) {
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
  const cx<R>* gm = grids + 16 + 4 * (med * 2 + h);
#pragma unroll
  for (int i = 0; i < p; ++i)
#pragma unroll
    for (int j = 0; j < p; ++j) {
      const R wxy = Lx[i] * Ly[j], dxy = dx[i] * Ly[j], xdy = Lx[i] * dy[j];
      const int32_t* cj = cmap + (b1 + j) * n2 + b2;
#pragma unroll
      for (int k = 0; k < p; ++k) {
        const R w = wxy * Lz[k], wx = dxy * Lz[k], wy = xdy * Lz[k], wz = wxy * dz[k];
        cx<R> gv[4];
        load_group(gm + ((int64_t)(b0 + i) * nac + cj[k]) * NPOT, gv);
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
  if (h == 0) {
    const R sa = R(1) / (z * k), sp = k / z;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      r[c] = -(sa * mulj(r[c]));
      r[4 + c] = -(sp * mulj(r[4 + c]));
      r[7 + c] = -(sa * mulj(r[7 + c]));
    }
    r[3] = -(sp * mulj(r[3]));
  }
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
// The near records are read once per conductivity gradient, the only reader
// besides set-up: their copies carry an L2 evict-first policy, so that the
// stream of records does not push the reused data (potentials, summaries,
// geometry) and the caller's vectors out of L2.
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
    const R* __restrict__ tp, const int32_t* __restrict__ cmap, int64_t nt, int q, int n2, int nac, R ke, R ki, R ze,
    R zi, int has_near,
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
  interp_group<R, P>(grids, base, L, dL, t * q + a, med, h, cmap, n2, nac, med ? ki : ke, med ? zi : ze, acc);
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

// ================================================================ transposed apply
// x_bar = A^T y_bar: the stages of the apply in reverse order, each the
// transpose of its forward map (no conjugation):
//   T1 k_grid_adj  rows -> 16 grid fields (the edge stencils transposed)
//   T2 fft_conv(adjoint): each field with its medium's Green function
//   T3 k_rows_adj  (near.cu) projection transposed, plus the transposed near
//                  matrix -> unknowns

// T1 (replaces a 180 us gather of 320-byte point adjoints on the 12 um guide):
// one warp (WPP = 8: a CTA, for operators with few points, project_wide) per
// covered grid point, a gather over its (edge, entry) pairs:
// lane = slot * 8 + group takes the group's weight block (four reals) of an
// entry against the edge's row that reads the group (groups 0, 1: E rows; 2, 3:
// H rows and Eq. 13; 4, 5: Eq. 13; 6, 7: Eq. 14); entries of plain edges have
// the first four groups only and use the spare lane bit as a slot.  The
// groups' adjoints are then combined into the 16 fields, as the transpose of
// the combination that stage C of the convolution forms.
template <typename R, int WPP>
__global__ void __launch_bounds__(256) k_grid_adj(const cx<R>* y, const int32_t* __restrict__ gp,
                                                  const int32_t* __restrict__ gpoff, const int32_t* __restrict__ gpl,
                                                  const int32_t* __restrict__ gpr, const int32_t* __restrict__ gpe,
                                                  const R* __restrict__ xw, int64_t nxl, int64_t ngp, int64_t npt,
                                                  int64_t nL, int64_t nR, R ke, R ki, R ze, R zi,
                                                  cx<R>* __restrict__ src) {
  __shared__ cx<R> red[8][32];  // [warp in CTA][group * 4 + component]
  const int64_t i = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) / (32 * WPP);
  if (i >= ngp) return;  // whole warp; WPP = 8: no CTA
  const int lane = threadIdx.x & 31, wl = threadIdx.x >> 5, wp = wl % WPP;
  const int e0 = gpoff[i], el = e0 + gpl[i], e1 = gpoff[i + 1];
  pdl_wait();
  cx<R> v[4], u[4];
#pragma unroll
  for (int c = 0; c < 4; ++c) v[c] = u[c] = czero<R>();
  {
    const R* w = xw + 4 * (lane & 1);
    const cx<R>* yr = y + ((lane & 2) ? nL : 0);
#pragma unroll 2
    for (int e = e0 + (lane >> 2) + 8 * wp; e < el; e += 8 * WPP) {
      R a[4];
      load4(w + 8 * (int64_t)gpe[e], a);
      const cx<R> b = yr[gpr[e]];
#pragma unroll
      for (int c = 0; c < 4; ++c) axpy2(u[c], a[c], b);
    }
  }
  {
    const int g = lane & 7;
    const R* w = xw + 8 * nxl + 4 * (g < 4 ? g & 1 : g - 2);
    const cx<R>* yr = y + nL + nR * ((g + 2) >> 2);
#pragma unroll 2
    for (int e = el + (lane >> 3) + 4 * wp; e < e1; e += 4 * WPP) {
      R a[4];
      load4(w + 24 * (int64_t)(gpe[e] - nxl), a);
      const cx<R> b = yr[gpr[e]];
#pragma unroll
      for (int c = 0; c < 4; ++c) axpy2(v[c], a[c], b);
    }
  }
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    u[c] = xadd(u[c], 4);
    if (!(lane & 4)) v[c] += u[c];
  }
  halve(v, 2, lane, 16);
  halve(v, 1, lane, 8);
  cx<R>* rw = red[wl];
  rw[(lane & 7) * 4 + ((lane >> 3) & 2) + ((lane >> 3) & 1)] = v[0];
  if constexpr (WPP > 1) {
    __syncthreads();
    if (wl > 0) return;
    cx<R> t = rw[lane];
#pragma unroll
    for (int w = 1; w < WPP; ++w) t += red[w][lane];
    rw[lane] = t;
  }
  __syncwarp();
  if (lane < 16) {
    const int f = lane >> 2, c = lane & 3;  // field group (medium, set), component
    const bool inner = f & 2;
    const R k = inner ? ki : ke, z = inner ? zi : ze, sg = inner ? R(-1) : R(1);
    cx<R> o;
    if (!(f & 1)) {  // A, phi: groups 0, 3 and 4 or 6
      const cx<R> g0 = rw[c], g4 = rw[16 + 4 * f + c];
      if (c < 3)
        o = mulj((z * k) * g4 - (sg * z * k) * g0) + sg * rw[12 + c];
      else
        o = mulj((z / k) * g4 + (sg * z / k) * g0);
    } else {  // F, psi: groups 1, 2 and 5 or 7
      const cx<R> g2 = rw[8 + c];
      if (c < 3)
        o = rw[16 + 4 * f + c] - sg * rw[4 + c] - (sg * k / z) * mulj(g2);
      else
        o = (sg / (k * z)) * mulj(g2);
    }
    src[(int64_t)lane * npt + gp[i]] = o;
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

}  // namespace

// Four warps per grid point where one per point and group leaves less than 32
// per SM (2 um guide, 1800 points: 13.3 -> 8.0 us)
static bool project_wide(const scabem_op* op, int groups) { return op->ngp * groups < (int64_t)152 * 32; }

// The grid part up to the potentials, for k right-hand sides: projection and
// convolution.  x in the layout of load_cols (k = 1: as it is).
template <typename R>
int grid_potentials(scabem_op* op, const cx<R>* x, int k, cudaStream_t s) {
  PrecData<R>& pd = pdata<R>(op);
  prof_mark(op, s);
  prof_mark(op, s);  // (the summaries stage is part of the projection)
  const int K = batch_group(k), groups = (int)cdiv(k, K);
  const bool wide = project_wide(op, groups);
  auto fn = K == 1   ? (wide ? k_project<R, 1, 128> : k_project<R, 1, 32>)
            : K == 2 ? (wide ? k_project<R, 2, 128> : k_project<R, 2, 32>)
            : K == 3 ? (wide ? k_project<R, 3, 128> : k_project<R, 3, 32>)
                     : (wide ? k_project<R, 4, 128> : k_project<R, 4, 32>);
  CK(launch_pdl(fn, dim3((unsigned)cdiv(op->ngp * (wide ? 128 : 32), PJ_THREADS), groups), PJ_THREADS, 0, s, x,
                batch_stride(k), op->gp, op->gpoff, op->gpl, op->gpr, pd.gq, op->ngp, (int64_t)op->n[0] * op->nac,
                op->nL, op->nR, pd.src, col_stride_src(op), k));
  prof_mark(op, s);
  return fft_conv<R>(op, pd, s, false, k);
}

// The last kernel of a product still reads its input while it writes the result:
// an input column that overlaps the result is copied first, into pd.xi.
template <typename R>
static int apart(scabem_op* op, const cx<R>*& in, const cx<R>* out, cudaStream_t s) {
  const auto a = reinterpret_cast<uintptr_t>(in), b = reinterpret_cast<uintptr_t>(out);
  const uintptr_t len = sizeof(cx<R>) * (uintptr_t)op->N;
  if (a >= b + len || b >= a + len) return SCABEM_OK;
  cx<R>* xi = pdata<R>(op).xi;
  CK(launch_pdl(k_interleave<R>, dim3((unsigned)cdiv(op->N, 256)), 256, 0, s, in, op->N, op->N, 1, 1, 1, xi));
  in = xi;
  return SCABEM_OK;
}

template <typename R>
int apply_batch(scabem_op* op, const cx<R>* x, int64_t ldx, cx<R>* y, int64_t ldy, int k, cudaStream_t s) {
  PrecData<R>& pd = pdata<R>(op);
  if (k < 1 || k > KBATCH || k > pd.kcap) {
    set_error("apply_batch: batch size outside the workspace capacity");
    return SCABEM_E_ARG;
  }
  if (k > 1) {
    const int st = batch_stride(k);
    CK(launch_pdl(k_interleave<R>, dim3((unsigned)cdiv(op->N * st, 256)), 256, 0, s, x, ldx, op->N, k, batch_group(k),
                  st, pd.xi));
    x = pd.xi;
  } else if (int rc = apart<R>(op, x, y, s)) {
    return rc;
  }
  if (int rc = grid_potentials<R>(op, x, k, s)) return rc;
  prof_mark(op, s);
  if (int rc = rows_apply<R>(op, x, y, ldy, k, s)) return rc;
  prof_mark(op, s);
  return SCABEM_OK;
}

template <typename R>
int apply_one(scabem_op* op, const cx<R>* x, cx<R>* y, cudaStream_t s) {
  return apply_batch<R>(op, x, op->N, y, op->N, 1, s);
}

// x_bar = A^T y_bar (one right-hand side), stages T1-T3.
template <typename R>
int apply_adjoint_one(scabem_op* op, const cx<R>* ybar, cx<R>* xbar, cudaStream_t s) {
  PrecData<R>& pd = pdata<R>(op);
  if (int rc = apart<R>(op, ybar, xbar, s)) return rc;
  const bool wide = project_wide(op, 1);
  CK(launch_pdl(wide ? k_grid_adj<R, 8> : k_grid_adj<R, 1>, dim3((unsigned)cdiv(op->ngp * (wide ? 256 : 32), 256)), 256, 0, s, ybar, op->gp, op->gpoff, op->gpl,
                op->gpr, op->gpe, pd.xw, op->nxl, op->ngp, (int64_t)op->n[0] * op->nac, op->nL, op->nR, (R)op->ke,
                (R)op->ki, (R)op->ze, (R)op->zi, pd.src));
  if (int rc = fft_conv<R>(op, pd, s, true)) return rc;
  return rows_adjoint<R>(op, ybar, xbar, s);
}

// Current summaries only (used by the field evaluation at probe points).
template <typename R>
int compute_summ(scabem_op* op, const cx<R>* x, cx<R>* summ, cudaStream_t s) {
  k_summ<R><<<(int)cdiv(3 * op->nt, 128), 128, 0, s>>>(x, op->unk, op->cX, op->tri, op->nt, summ);
  CK(cudaGetLastError());
  return SCABEM_OK;
}

// hs[p] = d(lam^T A x)/d sigma_p [per S] at every quadrature point
// (complex128): the apply's stages up to the records, then the derivative
// of the sigma-weighted testing (k_points_sens).
int sigma_sensitivity_op(scabem_op* op, const cx<double>* x, const cx<double>* lam, cx<double>* hs,
                         cudaStream_t s) {
  PrecData<double>& pd = op->d;
  if (int rc = compute_summ<double>(op, x, pd.summ, s)) return rc;
  if (int rc = grid_potentials<double>(op, x, 1, s)) return rc;
  prof_mark(op, s);
  const size_t sm = pt_smem_bytes(op->q, sizeof(cx<double>));
  auto fn = op->p == 2 ? k_points_sens<double, 2> : op->p == 3 ? k_points_sens<double, 3> : k_points_sens<double, 4>;
  if (int rc_ = set_max_smem(op->device, (const void*)fn, (int)sm)) return rc_;
  fn<<<(int)cdiv(op->nt, PT_WARPS), PT_WARPS * 32, sm, s>>>(
      pd.grid, op->base, pd.L, pd.dL, pd.near, op->noff, op->nsrc, pd.summ, op->tri, pd.tp, op->cmap, op->nt, op->q,
      op->n[2], (int)op->nac, op->ke, op->ki, op->ze, op->zi, op->npairs > 0 ? 1 : 0, op->valrow, op->tmo_d, lam, hs);
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

template int compute_summ<double>(scabem_op*, const cx<double>*, cx<double>*, cudaStream_t);
template int apply_one<float>(scabem_op*, const cx<float>*, cx<float>*, cudaStream_t);
template int apply_adjoint_one<float>(scabem_op*, const cx<float>*, cx<float>*, cudaStream_t);
template int apply_adjoint_one<double>(scabem_op*, const cx<double>*, cx<double>*, cudaStream_t);
template int apply_one<double>(scabem_op*, const cx<double>*, cx<double>*, cudaStream_t);
template int apply_batch<float>(scabem_op*, const cx<float>*, int64_t, cx<float>*, int64_t, int, cudaStream_t);
template int apply_batch<double>(scabem_op*, const cx<double>*, int64_t, cx<double>*, int64_t, int, cudaStream_t);
