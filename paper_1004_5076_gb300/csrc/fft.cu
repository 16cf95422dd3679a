// Grid convolution by zero-padded 3-D FFT, fused with the Green's-function
// multiply (the FFT acceleration of Appendix B, on the uniform grid of the
// precorrected-FFT method).
//
// Layout: physical grids are [field][i0][active column] (n0 points along axis 0,
// the (i1, i2) columns that some stencil covers); the transform size is P = 2n
// per axis.  The convolution runs in three kernels:
//   stage A: forward FFT along axis 0 of the 12 source fields, input pruned
//            to i0 < n0, output [field][k0][column];
//   stage B: per k0, the (y, z) convolution with the Green function of the
//            medium, 12 -> 16 fields: zero-padded 2-D FFTs over whole planes
//            (n1 n2 columns), direct sums over the active columns, or those sums
//            block-diagonalised by parity;
//   stage C: inverse FFT along axis 0, keep i0 < n0, written point-major
//            [i0][active column][32] for the testing gathers.
// Every FFT is an in-place shared-memory Stockham transform (radix 8, then 4
// or 2) with compile-time power-of-two lengths: each pass loads its
// butterflies into registers, synchronises, and stores them at their sorted
// positions.  One CTA owns whole lines, so each field makes one HBM round trip
// per stage.  The 1/(P0 P1 P2) scale is folded into the stored spectra.
#include <cuda_runtime.h>

#include <algorithm>

#include "device.cuh"

namespace {

constexpr int FFT_THREADS = 512;
constexpr int FFT_LTHREADS = 9;

template <typename R, int DIR>
__device__ __forceinline__ cx<R> rot(cx<R> a) {  // multiply by DIR * j
  return DIR < 0 ? mk(a.im, -a.re) : mk(-a.im, a.re);
}

// complex add / subtract; complex64 as one packed FP32x2 add
__device__ __forceinline__ cx<float> padd(cx<float> a, cx<float> b) {
  const float2 r = __fadd2_rn(make_float2(a.re, a.im), make_float2(b.re, b.im));
  return mk(r.x, r.y);
}
__device__ __forceinline__ cx<float> psub(cx<float> a, cx<float> b) {
  const float2 r = __fadd2_rn(make_float2(a.re, a.im), make_float2(-b.re, -b.im));
  return mk(r.x, r.y);
}
__device__ __forceinline__ cx<double> padd(cx<double> a, cx<double> b) { return a + b; }
__device__ __forceinline__ cx<double> psub(cx<double> a, cx<double> b) { return a - b; }

template <typename R, int DIR>
__device__ __forceinline__ void dft4(cx<R>& a0, cx<R>& a1, cx<R>& a2, cx<R>& a3) {
  cx<R> t0 = padd(a0, a2), t1 = psub(a0, a2), t2 = padd(a1, a3), u = rot<R, DIR>(psub(a1, a3));
  a0 = padd(t0, t2);
  a2 = psub(t0, t2);
  a1 = padd(t1, u);
  a3 = psub(t1, u);
}

template <typename R, int RAD, int DIR>
__device__ __forceinline__ void dft(cx<R>* v) {
  if constexpr (RAD == 2) {
    const cx<R> t = v[0];
    v[0] = t + v[1];
    v[1] = t - v[1];
  } else if constexpr (RAD == 4) {
    dft4<R, DIR>(v[0], v[1], v[2], v[3]);
  } else {
    // 8 = 2 x 4: even / odd 4-point transforms, then combine with w8^k
    cx<R> e0 = v[0], e1 = v[2], e2 = v[4], e3 = v[6];
    cx<R> o0 = v[1], o1 = v[3], o2 = v[5], o3 = v[7];
    dft4<R, DIR>(e0, e1, e2, e3);
    dft4<R, DIR>(o0, o1, o2, o3);
    const R s = R(0.70710678118654752440);
    // w8^1 = (1 + DIR j)/sqrt2, w8^2 = DIR j, w8^3 = (-1 + DIR j)/sqrt2
    const cx<R> w1 = s * (o1 + rot<R, DIR>(o1));
    const cx<R> w2 = rot<R, DIR>(o2);
    const cx<R> w3 = s * (rot<R, DIR>(o3) - o3);
    v[0] = padd(e0, o0);
    v[4] = psub(e0, o0);
    v[1] = padd(e1, w1);
    v[5] = psub(e1, w1);
    v[2] = padd(e2, w2);
    v[6] = psub(e2, w2);
    v[3] = padd(e3, w3);
    v[7] = psub(e3, w3);
  }
}

// One in-place Stockham pass of radix 2^LR over the 2^lnl lines of length
// N = 2^LN; element j of line l lives at buf[l*ls + j*es].  2^LNS is the
// product of the radices of the previous passes.  Consecutive threads take
// consecutive lines.  TOTL = log2 of the largest element count a caller
// passes, which bounds the butterflies each thread holds.
template <typename R, int LN, int LR, int LNS, int DIR, int TOTL>
__device__ __forceinline__ void pass_ip(cx<R>* buf, int lnl, int ls, int es, const cx<R>* tw) {
  constexpr int RAD = 1 << LR;
  constexpr int LPER = LN - LR;
  constexpr int NSM = (1 << LNS) - 1;
  constexpr int LTS = LN - LNS - LR;
  constexpr int MB0 = TOTL - LR - FFT_LTHREADS;
  constexpr int MAXB = MB0 > 0 ? (1 << MB0) : 1;
  const int nb = 1 << (lnl + LPER);
  const int lmask = (1 << lnl) - 1;
  cx<R> v[MAXB][RAD];
  int dst[MAXB];
#pragma unroll
  for (int i = 0; i < MAXB; ++i) {
    const int b = threadIdx.x + i * FFT_THREADS;
    if (b < nb) {
      const int line = b & lmask;
      const int j = b >> lnl;
      const cx<R>* s = buf + line * ls;
#pragma unroll
      for (int r = 0; r < RAD; ++r) v[i][r] = s[(j + (r << LPER)) * es];
      if (LNS > 0) {
        const int k = j & NSM;
#pragma unroll
        for (int r = 1; r < RAD; ++r) {
          cx<R> t = tw[(r * k) << LTS];
          if (DIR > 0) t = conj(t);
          v[i][r] = v[i][r] * t;
        }
      }
      dft<R, RAD, DIR>(v[i]);
      dst[i] = line * ls + ((((j >> LNS) << (LNS + LR)) + (j & NSM)) * es);
    }
  }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < MAXB; ++i) {
    const int b = threadIdx.x + i * FFT_THREADS;
    if (b < nb) {
#pragma unroll
      for (int r = 0; r < RAD; ++r) buf[dst[i] + ((r << LNS) * es)] = v[i][r];
    }
  }
  __syncthreads();
}

template <typename R, int LN, int LNS, int DIR, int TOTL>
__device__ __forceinline__ void fft_ip(cx<R>* buf, int lnl, int ls, int es, const cx<R>* tw) {
  if constexpr (LNS < LN) {
    constexpr int REM = LN - LNS;
    constexpr int LR = REM >= 3 ? 3 : REM;
    pass_ip<R, LN, LR, LNS, DIR, TOTL>(buf, lnl, ls, es, tw);
    fft_ip<R, LN, LNS + LR, DIR, TOTL>(buf, lnl, ls, es, tw);
  }
}

// FFT of 2^lnl lines of length 2^ln (3 <= ln <= 10), all threads of the CTA.
template <typename R, int DIR, int TOTL>
__device__ __forceinline__ void fft_lines(cx<R>* buf, int ln, int lnl, int ls, int es, const cx<R>* tw) {
  switch (ln) {
    case 3: fft_ip<R, 3, 0, DIR, TOTL>(buf, lnl, ls, es, tw); break;
    case 4: fft_ip<R, 4, 0, DIR, TOTL>(buf, lnl, ls, es, tw); break;
    case 5: fft_ip<R, 5, 0, DIR, TOTL>(buf, lnl, ls, es, tw); break;
    case 6: fft_ip<R, 6, 0, DIR, TOTL>(buf, lnl, ls, es, tw); break;
    case 7: fft_ip<R, 7, 0, DIR, TOTL>(buf, lnl, ls, es, tw); break;
    case 8: fft_ip<R, 8, 0, DIR, TOTL>(buf, lnl, ls, es, tw); break;
    case 9: fft_ip<R, 9, 0, DIR, TOTL>(buf, lnl, ls, es, tw); break;
    default: fft_ip<R, 10, 0, DIR, TOTL>(buf, lnl, ls, es, tw); break;
  }
}

__host__ __device__ inline int ilog2(int v) {
  int l = 0;
  while ((1 << l) < v) ++l;
  return l;
}

// largest element count (log2) one CTA transforms: complex64 8192, complex128 4096
template <typename R>
struct Tot {
  static constexpr int L = sizeof(R) == 4 ? 13 : 12;
};

// ---------------------------------------------------------------- stage A / C
// Stage A on the nac active columns, [field][i0][active column]; one CTA owns
// CB of them for one field over the whole axis 0 (smem: [P0][CB], lines =
// columns).  Inputs i0 >= n_in are zero.
// The output has Cout columns per (field, k0): active column j goes to
// column j (compact, Cout = nac) or to acol[j] (whole planes, Cout = C).
template <typename R>
__global__ void __launch_bounds__(FFT_THREADS) k_axis0(const cx<R>* in, cx<R>* __restrict__ out,
                                                       int n_in, int P0, const int32_t* __restrict__ acol, int nac,
                                                       int CB, const cx<R>* __restrict__ tw,
                                                       int64_t cs_in, int64_t cs_out, int64_t Cout, int compact) {
  extern __shared__ unsigned char smem_raw[];
  cx<R>* tws = reinterpret_cast<cx<R>*>(smem_raw);
  cx<R>* b0 = tws + P0;
  in += blockIdx.z * cs_in;  // right-hand side blockIdx.z
  out += blockIdx.z * cs_out;
  const int f = blockIdx.y;
  const int a0 = blockIdx.x * CB;
  const int lcb = ilog2(CB);
  for (int i = threadIdx.x; i < P0; i += FFT_THREADS) tws[i] = tw[i];
  pdl_wait();
  const int64_t fin = (int64_t)f * n_in * nac;
  for (int idx = threadIdx.x; idx < P0 * CB; idx += FFT_THREADS) {
    const int i0 = idx >> lcb, l = idx & (CB - 1);
    cx<R> v = czero<R>();
    if (i0 < n_in && a0 + l < nac) v = in[fin + (int64_t)i0 * nac + a0 + l];
    b0[idx] = v;
  }
  __syncthreads();
  fft_lines<R, -1, Tot<R>::L>(b0, ilog2(P0), lcb, 1, CB, tws);
  const int64_t fout = (int64_t)f * P0 * Cout;
  for (int idx = threadIdx.x; idx < P0 * CB; idx += FFT_THREADS) {
    const int k0 = idx >> lcb, l = idx & (CB - 1);
    if (a0 + l < nac) out[fout + (int64_t)k0 * Cout + (compact ? a0 + l : acol[a0 + l])] = b0[idx];
  }
}

// Stage C with point-major output, on the nac active columns only (the
// potentials are read nowhere else; the input is [k0][active column][16 fields]
// from the direct sums (compact), [field][k0][Cin columns] from the FFT planes):
// one CTA owns NC of them
// for the eight fields of one set (bound by latency and shared-memory passes: 13 us
// on the 12 um guide, 57 for 8 columns; 71 with the input fields 8 bytes apart) (J: A, phi of both media; M: F, psi of both)
// over axis 0, line l = field * NC + column, and writes groups of four complex
// values, whole 32-byte sectors in complex64, at out[(i0 * nac + column) * 32]
// for i0 < n_out.
//
// The groups are what the rows read (near.cu).  Groups 4 .. 7 (exterior J, M,
// interior J, M): [A, phi] scaled by j z k and j z / k (the strong-form E of
// Eqs. 13, 14) and [F, 0].  Groups 0 .. 3: the weak-form differences of the two
// media, E from [A, phi] and from [F], H from [F, psi] and from [A], which
// halve the products of the testing; a set's two media meet in its CTA.
// COMB = false (transposed apply): the fields themselves in groups 4 .. 7.
template <typename R, bool COMB, int TOTL>
__global__ void __launch_bounds__(FFT_THREADS)
    k_axis0_pm(const cx<R>* in, cx<R>* __restrict__ out, int n_out, int P0,
               const int32_t* __restrict__ acol, int nac, int NC, const cx<R>* __restrict__ tw, int64_t cs_in,
               int64_t cs_out, int64_t Cin, int compact, R ke, R ki, R ze, R zi) {
  extern __shared__ unsigned char smem_raw[];
  cx<R>* tws = reinterpret_cast<cx<R>*>(smem_raw);
  cx<R>* b0 = tws + P0;
  in += blockIdx.z * cs_in;  // right-hand side blockIdx.z
  out += blockIdx.z * cs_out;
  const int set = blockIdx.y;
  const int a0 = blockIdx.x * NC;
  const int CB = 8 * NC;
  const int lcb = ilog2(CB), lnc = ilog2(NC);
  for (int i = threadIdx.x; i < P0; i += FFT_THREADS) tws[i] = tw[i];
  pdl_wait();
  for (int idx = threadIdx.x; idx < P0 * CB; idx += FFT_THREADS) {
    const int i0 = idx >> lcb, l = idx & (CB - 1);
    const int fl = compact ? l & 7 : l >> lnc, cl = compact ? l >> 3 : l & (NC - 1);  // in the input's order
    const int field = (fl & 3) + 4 * set + 2 * (fl & 4);
    cx<R> v = czero<R>();
    if (a0 + cl < nac)
      v = compact ? in[((int64_t)i0 * nac + a0 + cl) * NFIELD_OUT + field]
                  : in[((int64_t)field * P0 + i0) * Cin + acol[a0 + cl]];
    b0[(i0 << lcb) + fl * NC + cl] = v;
  }
  __syncthreads();
  fft_lines<R, 1, TOTL>(b0, ilog2(P0), lcb, 1, CB, tws);
  const R wE = ze * ke, wI = zi * ki, pE = ze / ke, pI = zi / ki, yE = ke / ze, yI = ki / zi;
  const R qE = R(1) / (ke * ze), qI = R(1) / (ki * zi);
  for (int idx = threadIdx.x; idx < 4 * n_out * NC; idx += FFT_THREADS) {
    const int fl = idx & 3, cl = (idx >> 2) & (NC - 1), k0 = idx >> (2 + lnc);  // component fastest: whole sectors
    if (a0 + cl >= nac) continue;
    const cx<R> e = b0[(k0 << lcb) + fl * NC + cl], i = b0[(k0 << lcb) + (fl + 4) * NC + cl];
    cx<R>* o = out + ((int64_t)k0 * nac + a0 + cl) * NPOT + fl;
    if (!COMB) {
      o[16 + 4 * set] = e;
      o[24 + 4 * set] = i;
    } else if (set == 0) {  // A, phi
      o[0] = fl < 3 ? mulj(wI * i - wE * e) : mulj(pE * e - pI * i);
      o[12] = fl < 3 ? e - i : czero<R>();
      o[16] = mulj((fl < 3 ? wE : pE) * e);
      o[24] = mulj((fl < 3 ? wI : pI) * i);
    } else {  // F, psi (the interior M set carries its sign)
      o[4] = fl < 3 ? i - e : czero<R>();
      o[8] = fl < 3 ? mulj(yI * i - yE * e) : mulj(qE * e - qI * i);
      o[20] = fl < 3 ? e : czero<R>();
      o[28] = fl < 3 ? i : czero<R>();
    }
  }
}

// ---------------------------------------------------------------- warp-owned lines
// FFT of one line of length 2^LN owned by T = 2^(LN-3) consecutive lanes of a
// warp (lane tl of the group).  The first pass reads element j through
// ld(j), the last pass writes element j through st(j, v); the passes in
// between exchange through the line's shared-memory storage line[j*es]
// with warp-level synchronisation only.
template <typename R, int LN, int LNS, int DIR, class LD, class ST>
__device__ __forceinline__ void wline_fft(cx<R>* line, int es, int tl, bool act, const cx<R>* tw, const LD& ld,
                                          const ST& st) {
  if constexpr (LNS < LN) {
    constexpr int REM = LN - LNS;
    constexpr int LR = REM >= 3 ? 3 : REM;
    constexpr int RAD = 1 << LR;
    constexpr int LT = LN - 3;
    constexpr int LPER = LN - LR;
    constexpr int NBT = 1 << (LPER - LT);  // butterflies per lane
    constexpr int NSM = (1 << LNS) - 1;
    constexpr int LTS = LN - LNS - LR;
    constexpr bool FIRST = LNS == 0, LAST = LNS + LR == LN;
    cx<R> v[NBT][RAD];
    int dst[NBT];
    if (act) {
#pragma unroll
      for (int i = 0; i < NBT; ++i) {
        const int j = tl + (i << LT);
#pragma unroll
        for (int r = 0; r < RAD; ++r) {
          const int e = j + (r << LPER);
          v[i][r] = FIRST ? ld(e) : line[e * es];
        }
        if (LNS > 0) {
          const int k = j & NSM;
#pragma unroll
          for (int r = 1; r < RAD; ++r) {
            cx<R> t = tw[(r * k) << LTS];
            if (DIR > 0) t = conj(t);
            v[i][r] = v[i][r] * t;
          }
        }
        dft<R, RAD, DIR>(v[i]);
        dst[i] = ((j >> LNS) << (LNS + LR)) + (j & NSM);
      }
    }
    if (!LAST) __syncwarp();
    if (act) {
#pragma unroll
      for (int i = 0; i < NBT; ++i)
#pragma unroll
        for (int r = 0; r < RAD; ++r) {
          const int e = dst[i] + (r << LNS);
          if (LAST)
            st(e, v[i][r]);
          else
            line[e * es] = v[i][r];
        }
    }
    if (!LAST) {
      __syncwarp();
      wline_fft<R, LN, LNS + LR, DIR>(line, es, tl, act, tw, ld, st);
    }
  }
}

// Runs f(l, line, tl, act) for lines l < nlines spread over the warps of the
// CTA (2^(5-LT) lines per warp); trip counts are uniform within a warp.
template <int LN, class F>
__device__ __forceinline__ void for_warp_lines(int nlines, const F& f) {
  constexpr int LT = LN - 3;
  constexpr int LPW = 32 >> LT;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  const int tl = lane & ((1 << LT) - 1), sub = lane >> LT;
  for (int l0 = warp * LPW; l0 < nlines; l0 += nw * LPW) {
    const int l = l0 + sub;
    f(l < nlines ? l : 0, tl, l < nlines);
  }
}

// ---------------------------------------------------------------- stage B
// One CTA per (k0 plane, source field).  Source fields:
//   0..3  exterior J (x, y, z, div)  -> outputs 0..3 with G_e
//   4..7  interior J                 -> outputs 8..11 with G_i
//   8..11 exterior M                 -> outputs 4..7 with G_e and 12..15 with -G_i
// The plane lives in shared memory with row stride P2 + 2; S holds the
// forward spectrum, W the working plane of one output.  The forward row pass
// reads the physical n1 x n2 corner straight from global memory, the forward
// column pass skips the zero rows, the Green multiply is applied as the
// inverse column pass loads S, only the n1 physical rows are kept, and the
// inverse row pass writes the physical corner straight to global memory.
constexpr int PLANE_THREADS = 256;

template <typename R, int L1, int L2>
__global__ void __launch_bounds__(PLANE_THREADS) k_planes(const cx<R>* A, cx<R>* __restrict__ B,
                                                          const cx<R>* __restrict__ ghE,
                                                          const cx<R>* __restrict__ ghI, int P0, int n1, int n2,
                                                          const cx<R>* __restrict__ tw1,
                                                          const cx<R>* __restrict__ tw2, int ident, int64_t cs) {
  extern __shared__ unsigned char smem_raw[];
  constexpr int P1 = 1 << L1, P2 = 1 << L2;
  A += blockIdx.z * cs;  // right-hand side blockIdx.z
  B += blockIdx.z * cs;
  constexpr int LS = P2 + 2;
  constexpr int plane = P1 * LS;
  cx<R>* t1 = reinterpret_cast<cx<R>*>(smem_raw);
  cx<R>* t2 = t1 + P1;
  cx<R>* S = t2 + P2;
  cx<R>* W = S + plane;
  const int k0 = blockIdx.x;
  const int f = blockIdx.y;
  for (int i = threadIdx.x; i < P1; i += PLANE_THREADS) t1[i] = tw1[i];
  for (int i = threadIdx.x; i < P2; i += PLANE_THREADS) t2[i] = tw2[i];
  pdl_wait();
  __syncthreads();
  const int64_t C = (int64_t)n1 * n2;
  const cx<R>* src = A + ((int64_t)f * P0 + k0) * C;
  // forward rows (axis 2): the n1 non-zero rows, read from global memory
  for_warp_lines<L2>(n1, [&](int i1, int tl, bool act) {
    cx<R>* row = S + i1 * LS;
    wline_fft<R, L2, 0, -1>(
        row, 1, tl, act, t2, [&](int e) { return e < n2 ? src[i1 * n2 + e] : czero<R>(); },
        [&](int e, cx<R> v) { row[e] = v; });
  });
  __syncthreads();
  // forward columns (axis 1): rows >= n1 are zero and are not read
  for_warp_lines<L1>(P2, [&](int k2, int tl, bool act) {
    cx<R>* col = S + k2;
    wline_fft<R, L1, 0, -1>(
        col, LS, tl, act, t1, [&](int e) { return e < n1 ? col[e * LS] : czero<R>(); },
        [&](int e, cx<R> v) { col[e * LS] = v; });
  });
  __syncthreads();

  const int h1 = P1 / 2 + 1, h2 = P2 / 2 + 1;
  const int q0 = min(k0, P0 - k0);
  const int nout = (!ident && f >= 8) ? 2 : 1;
  for (int which = 0; which < nout; ++which) {
    int fo;
    const cx<R>* gh;
    R sgn = R(1);
    if (ident) {  // transposed apply: each of the 16 fields with its medium's function
      fo = f;
      gh = f < 8 ? ghE : ghI;
    } else if (f < 4) {
      fo = f;
      gh = ghE;
    } else if (f < 8) {
      fo = 8 + (f - 4);
      gh = ghI;
    } else if (which == 0) {
      fo = 4 + (f - 8);
      gh = ghE;
    } else {
      fo = 12 + (f - 8);
      gh = ghI;
      sgn = R(-1);
    }
    const cx<R>* g0 = gh + (int64_t)q0 * h1 * h2;
    // inverse columns: load S times the Green spectrum, keep rows < n1 in W
    for_warp_lines<L1>(P2, [&](int k2, int tl, bool act) {
      const cx<R>* scol = S + k2;
      cx<R>* wcol = W + k2;
      const cx<R>* gcol = g0 + min(k2, P2 - k2) * h1;
      wline_fft<R, L1, 0, 1>(
          wcol, LS, tl, act, t1,
          [&](int e) { return sgn * (scol[e * LS] * gcol[min(e, P1 - e)]); },
          [&](int e, cx<R> v) {
            if (e < n1) wcol[e * LS] = v;
          });
    });
    __syncthreads();
    // inverse rows: the n1 physical rows, written straight to global memory
    cx<R>* dst = B + ((int64_t)fo * P0 + k0) * C;
    for_warp_lines<L2>(n1, [&](int i1, int tl, bool act) {
      cx<R>* row = W + i1 * LS;
      wline_fft<R, L2, 0, 1>(
          row, 1, tl, act, t2, [&](int e) { return row[e]; },
          [&](int e, cx<R> v) {
            if (e < n2) dst[i1 * n2 + e] = v;
          });
    });
    __syncthreads();
  }
}

template <typename R>
using PlanesFn = void (*)(const cx<R>*, cx<R>*, const cx<R>*, const cx<R>*, int, int, int, const cx<R>*,
                          const cx<R>*, int, int64_t);

template <typename R, int L1, int L2>
PlanesFn<R> planes_fn() {
  if constexpr (L1 + L2 <= 12) return k_planes<R, L1, L2>;
  else return nullptr;
}

template <typename R, int L1>
PlanesFn<R> planes_row(int l2) {
  switch (l2) {
    case 3: return planes_fn<R, L1, 3>();
    case 4: return planes_fn<R, L1, 4>();
    case 5: return planes_fn<R, L1, 5>();
    case 6: return planes_fn<R, L1, 6>();
    case 7: return planes_fn<R, L1, 7>();
    default: return nullptr;
  }
}

// ---------------------------------------------------------------- stage B, 64 x 64 planes
// The same plane step specialised to P1 = P2 = 64 (n1 = n2 = 32), the usual
// cross-section of a guide grid.  A 64-point line belongs to eight lanes:
// lane t holds elements t + 8r, transforms over r (radix 8), multiplies by
// w64^(t k) and swaps through a per-line scratch so that lane k then holds
// index k of every t; a second radix-8 transform leaves elements k + 8m in
// lane k.  That is the layout the inverse transform starts from, so the
// forward column transform, the Green multiply of each output and the
// inverse column transform run back to back in registers.  Half-zero inputs
// and half-kept outputs use pruned radix-8 transforms.
//
// Shared memory (8-byte words, 16 banks of 8 bytes per half-warp): a plane
// holds rows 0..31 with row i, column k at i*64 + (k ^ g(i)), g(i) =
// 2(i mod 8) ^ 8(i mod 2); row accesses (two rows per half-warp) and column
// accesses (eight rows of two columns per half-warp) are then free of bank
// conflicts.  The per-line scratch puts element (t, k) at 8t + (k + t) mod 8,
// 72 words per line, for the same reason.
constexpr int P64_THREADS = 256;  // 8 warps x 4 lines of 8 lanes: one pass over 32 rows
constexpr int P64_SCR = 72;

__device__ __forceinline__ int swz64(int i, int k) { return i * 64 + (k ^ ((2 * (i & 7)) ^ ((i & 1) << 3))); }

// radix-8 transform of v[0..3] with v[4..7] = 0
template <typename R, int DIR>
__device__ __forceinline__ void dft8_hin(cx<R>* v) {
  const R s = R(0.70710678118654752440);
  cx<R> e0 = v[0], e1 = v[1], e2 = v[2], e3 = v[3];
  cx<R> o0 = v[0], o1 = s * (v[1] + rot<R, DIR>(v[1])), o2 = rot<R, DIR>(v[2]), o3 = s * (rot<R, DIR>(v[3]) - v[3]);
  dft4<R, DIR>(e0, e1, e2, e3);
  dft4<R, DIR>(o0, o1, o2, o3);
  v[0] = e0;
  v[2] = e1;
  v[4] = e2;
  v[6] = e3;
  v[1] = o0;
  v[3] = o1;
  v[5] = o2;
  v[7] = o3;
}

// radix-8 transform keeping outputs 0..3
template <typename R, int DIR>
__device__ __forceinline__ void dft8_hout(cx<R>* v) {
  cx<R> e0 = v[0], e1 = v[2], e2 = v[4], e3 = v[6];
  cx<R> o0 = v[1], o1 = v[3], o2 = v[5], o3 = v[7];
  dft4<R, DIR>(e0, e1, e2, e3);
  dft4<R, DIR>(o0, o1, o2, o3);
  const R s = R(0.70710678118654752440);
  v[0] = padd(e0, o0);
  v[1] = padd(e1, s * (o1 + rot<R, DIR>(o1)));
  v[2] = padd(e2, rot<R, DIR>(o2));
  v[3] = padd(e3, s * (rot<R, DIR>(o3) - o3));
}

// 64-point transform of one line over its eight lanes (lane t, v[r] =
// element t + 8r on entry, element t + 8m in v[m] on exit); w[k] = w64^(t k).
template <typename R, int DIR, bool HALF_IN, bool HALF_OUT>
__device__ __forceinline__ void line64(cx<R>* v, const cx<R>* w, cx<R>* scr, int t) {
  if (HALF_IN)
    dft8_hin<R, DIR>(v);
  else
    dft<R, 8, DIR>(v);
#pragma unroll
  for (int k = 1; k < 8; ++k) v[k] = v[k] * (DIR < 0 ? w[k] : conj(w[k]));
#pragma unroll
  for (int k = 0; k < 8; ++k) scr[t * 8 + ((k + t) & 7)] = v[k];
  __syncwarp();
#pragma unroll
  for (int i = 0; i < 8; ++i) v[i] = scr[i * 8 + ((t + i) & 7)];
  __syncwarp();
  if (HALF_OUT)
    dft8_hout<R, DIR>(v);
  else
    dft<R, 8, DIR>(v);
}

template <typename R>
__global__ void __launch_bounds__(P64_THREADS, sizeof(R) == 4 ? 3 : 1)
    k_planes64(const cx<R>* A, cx<R>* __restrict__ B, const cx<R>* __restrict__ ghE,
               const cx<R>* __restrict__ ghI, int P0, const cx<R>* __restrict__ tw64, uint64_t rowmask, int ident,
               int64_t cs) {
  constexpr int NP = 32, H = 33;
  A += blockIdx.z * cs;  // right-hand side blockIdx.z
  B += blockIdx.z * cs;
  extern __shared__ unsigned char smem_raw[];
  cx<R>* W0 = reinterpret_cast<cx<R>*>(smem_raw);  // forward rows, then output 0
  cx<R>* W1 = W0 + NP * 64;                        // output 1
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int t = lane & 7, sub = lane >> 3;
  cx<R>* scr = W1 + NP * 64 + (warp * 4 + sub) * P64_SCR;
  cx<R> w[8];
  w[0] = mk(R(1), R(0));
#pragma unroll
  for (int k = 1; k < 8; ++k) w[k] = tw64[t * k];
  pdl_wait();
  const int k0 = blockIdx.x, f = blockIdx.y;
  const int i1 = warp * 4 + sub;  // the row this lane works on in the row passes
  // rows no stencil covers are zero in and unused out; the test is per warp
  // (its four rows) so that the line transforms' warp barriers see all lanes
  const bool row_on = ((rowmask >> (warp * 4)) & 0xF) != 0;
  {
    // forward rows: the 32 physical rows, elements >= 32 are zero
    cx<R> v[8];
    if (row_on) {
      const cx<R>* src = A + ((int64_t)f * P0 + k0) * (NP * NP) + i1 * NP;
#pragma unroll
      for (int r = 0; r < 4; ++r) v[r] = src[t + 8 * r];
      line64<R, -1, true, false>(v, w, scr, t);
    } else {
#pragma unroll
      for (int m = 0; m < 8; ++m) v[m] = czero<R>();
    }
#pragma unroll
    for (int m = 0; m < 8; ++m) W0[swz64(i1, t + 8 * m)] = v[m];
  }
  __syncthreads();

  // source field -> output fields, media and signs (as in k_planes)
  // transposed apply (ident): each of the 16 fields with its medium's function
  const int nout = (!ident && f >= 8) ? 2 : 1;
  const int q0 = min(k0, P0 - k0);
  const cx<R>* ga = ident ? (f < 8 ? ghE : ghI) : ((f >= 4 && f < 8) ? ghI : ghE);  // output 0
  const int foa = ident ? f : (f < 4 ? f : (f < 8 ? 8 + (f - 4) : 4 + (f - 8)));
  const int fob = 12 + (f - 8);  // output 1 (f >= 8), interior medium, sign -1
  ga += (int64_t)q0 * H * H;
  const cx<R>* gb = ghI + (int64_t)q0 * H * H;

  // columns: forward transform (rows >= 32 zero), Green multiply, inverse
  // transform, rows < 32 kept in W0 / W1 (a column is read and rewritten by
  // the same eight lanes)
#pragma unroll 1
  for (int it = 0; it < 2; ++it) {
    const int c = it * 32 + warp * 4 + sub;
    cx<R> x[8];
#pragma unroll
    for (int r = 0; r < 4; ++r) x[r] = W0[swz64(t + 8 * r, c)];
    line64<R, -1, true, false>(x, w, scr, t);
    const int cg = min(c, 64 - c) * H;
#pragma unroll 1
    for (int o = 0; o < nout; ++o) {
      const cx<R>* gp = (o ? gb : ga) + cg;
      cx<R> v[8];
#pragma unroll
      for (int m = 0; m < 8; ++m) {
        const int e = t + 8 * m;
        v[m] = x[m] * gp[min(e, 64 - e)];
        if (o) v[m] = -v[m];
      }
      line64<R, 1, false, true>(v, w, scr, t);
      cx<R>* Wo = o ? W1 : W0;
#pragma unroll
      for (int m = 0; m < 4; ++m) Wo[swz64(t + 8 * m, c)] = v[m];
    }
  }
  __syncthreads();

  // inverse rows, the 32 physical columns written to global memory
#pragma unroll 1
  for (int o = 0; o < nout && row_on; ++o) {
    const cx<R>* Wo = o ? W1 : W0;
    cx<R> v[8];
#pragma unroll
    for (int r = 0; r < 8; ++r) v[r] = Wo[swz64(i1, t + 8 * r)];
    line64<R, 1, false, true>(v, w, scr, t);
    cx<R>* dst = B + ((int64_t)(o ? fob : foa) * P0 + k0) * (NP * NP) + i1 * NP;
#pragma unroll
    for (int m = 0; m < 4; ++m) dst[t + 8 * m] = v[m];
  }
}

// ---------------------------------------------------------------- stage B, direct
// (In the transposed apply, ident = 1, medium m takes fields 8m .. 8m+7 to
// the same fields, no sign.)
// Stage B as a direct sum over the active (i1, i2) columns: per (k0 plane,
// medium) the 8 source fields of that medium (its J set and the M set) are
// convolved with gt[q0][|d1|][|d2|] (the axis-0 transform of the spatial
// Green table):  out_v(i) = sum over active j of gt(|i1 - j1|, |i2 - j2|)
// src_v(j).  This is the linear convolution that the zero-padded 2-D FFTs
// compute (offsets never reach the padding), evaluated only on the columns
// that are read.  Medium 0: J_e (0..3), M (8..11) -> outputs 0..3, 4..7;
// medium 1: J_i (4..7), M (8..11) -> outputs 8..11 and -(12..15).  One
// thread per output column, 8 accumulators; each table value serves the 8
// fields, and the source values are shared-memory broadcasts.
constexpr int PD_THREADS = 128;

// acc[v] += t * s[v], v < 8; complex64 keeps P + j Q parts (packed FP32x2)
template <typename R>
struct Acc8;
template <>
struct Acc8<float> {
  float2 P[8], Q[8];
  __device__ __forceinline__ void zero() {
#pragma unroll
    for (int v = 0; v < 8; ++v) P[v] = Q[v] = make_float2(0.f, 0.f);
  }
  __device__ __forceinline__ void mac(cx<float> t, const cx<float>* s) {
    const float2 tr = make_float2(t.re, t.re), ti = make_float2(t.im, t.im);
    const float4* s4 = reinterpret_cast<const float4*>(s);
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const float4 w = s4[u];
      const float2 a = make_float2(w.x, w.y), b = make_float2(w.z, w.w);
      P[2 * u] = __ffma2_rn(tr, a, P[2 * u]);
      Q[2 * u] = __ffma2_rn(ti, a, Q[2 * u]);
      P[2 * u + 1] = __ffma2_rn(tr, b, P[2 * u + 1]);
      Q[2 * u + 1] = __ffma2_rn(ti, b, Q[2 * u + 1]);
    }
  }
  __device__ __forceinline__ cx<float> get(int v) const { return mk(P[v].x - Q[v].y, P[v].y + Q[v].x); }
};
template <>
struct Acc8<double> {
  cx<double> a[8];
  __device__ __forceinline__ void zero() {
#pragma unroll
    for (int v = 0; v < 8; ++v) a[v] = czero<double>();
  }
  __device__ __forceinline__ void mac(cx<double> t, const cx<double>* s) {
#pragma unroll
    for (int v = 0; v < 8; ++v) cfma(a[v], t, s[v]);
  }
  __device__ __forceinline__ cx<double> get(int v) const { return a[v]; }
};

template <typename R>
__global__ void __launch_bounds__(PD_THREADS) k_planes_direct(const cx<R>* A, cx<R>* __restrict__ B,
                                                              const cx<R>* __restrict__ gtE,
                                                              const cx<R>* __restrict__ gtI, int P0,
                                                              const int32_t* __restrict__ acoord, int nac, int R1,
                                                              int R2, int ident, int64_t cs) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  A += blockIdx.z * cs;  // right-hand side blockIdx.z
  B += blockIdx.z * cs;
  cx<R>* src = reinterpret_cast<cx<R>*>(smem_raw);  // [nac][8]
  cx<R>* T = src + (int64_t)nac * 8;                 // [R1][R2]
  int32_t* crd = reinterpret_cast<int32_t*>(T + R1 * R2);
  const int k0 = blockIdx.x, med = blockIdx.y;
  const int q0 = min(k0, P0 - k0);
  const cx<R>* gt = (med ? gtI : gtE) + (int64_t)q0 * R1 * R2;
  for (int i = threadIdx.x; i < R1 * R2; i += PD_THREADS) T[i] = gt[i];
  pdl_wait();
  for (int idx = threadIdx.x; idx < nac * 8; idx += PD_THREADS) {
    const int v = idx / nac, j = idx - v * nac;  // consecutive threads: consecutive columns of one field
    const int f = ident ? 8 * med + v : (v < 4 ? (med ? 4 + v : v) : 8 + (v - 4));
    src[j * 8 + v] = A[((int64_t)f * P0 + k0) * nac + j];
  }
  for (int i = threadIdx.x; i < nac; i += PD_THREADS) crd[i] = acoord[i];
  __syncthreads();
  for (int i = threadIdx.x; i < nac; i += PD_THREADS) {
    const int ci = crd[i];
    const int i1 = ci >> 16, i2 = ci & 0xffff;
    Acc8<R> acc;
    acc.zero();
    for (int j = 0; j < nac; ++j) {
      const int cj = crd[j];
      const int d1 = abs(i1 - (cj >> 16)), d2 = abs(i2 - (cj & 0xffff));
      acc.mac(T[d1 * R2 + d2], src + j * 8);
    }
#pragma unroll
    for (int v = 0; v < 8; ++v) {
      const cx<R> val = acc.get(v);
      B[((int64_t)k0 * nac + i) * NFIELD_OUT + 8 * med + v] = (!ident && med && v >= 4) ? -val : val;
    }
  }
}

// ---------------------------------------------------------------- stage B, direct, by parity
// The direct sum over the box R1 x R2 of the active columns, block
// diagonalised by its reflection symmetry: gt depends on |i1 - j1| and |i2 - j2|
// only, so sums and differences of mirrored columns along either axis do not
// mix.  The four parity blocks need a quarter of the products of the whole box
// (guide: 3,136 per field against 104^2 = 10,816 over the active columns).
// Positions keep their place: e = x_i + x_(n-1-i) lies at i (the middle one as
// it is), o = x_i - x_(n-1-i) at n - 1 - i.  The tables hold, per axis-0
// frequency and block, M[j][i] = (1/4) sum of gt over the direct and mirrored
// offsets with the block's signs (setup.cu: k_parity_tables), so that the
// same butterflies lead back.
//
// One CTA per (q0, medium): the planes k0 = q0 and P0 - q0 share the table.
// One thread per (plane, position), 8 fields each; a table value serves 8
// fields, the sources are shared-memory broadcasts.  In complex64 the products
// take a few microseconds, so the rest is kept short: the table is copied to
// shared memory while the sources arrive (STAGE), the sources of all rows are in
// flight at once, and the two axes' butterflies are one pass.  The CTA takes
// every gridDim.z-th right-hand side of a batch in turn.
constexpr int PS_THREADS = 256;
constexpr int PS_W = 10;  // words per position: 8 fields, padded so that a row's stores spread over the banks

// butterflies of both axes over the planes s [plane][i1][i2][PS_W], in place
template <typename R>
__device__ __forceinline__ void parity_pass(cx<R>* s, int R1, int R2, int npl) {
  const int E1 = (R1 + 1) / 2, E2 = (R2 + 1) / 2;
  for (int u = threadIdx.x; u < npl * E1 * E2 * 8; u += PS_THREADS) {
    const int v = u & 7, w = u >> 3, q = w / E2, i2 = w - q * E2, pl = q >= E1, i1 = q - pl * E1;
    const int m1 = R1 - 1 - i1, m2 = R2 - 1 - i2;
    cx<R>* b = s + (int64_t)pl * R1 * R2 * PS_W + v;
    cx<R>*p00 = b + (i1 * R2 + i2) * PS_W, *p10 = b + (m1 * R2 + i2) * PS_W, *p01 = b + (i1 * R2 + m2) * PS_W,
         *p11 = b + (m1 * R2 + m2) * PS_W;
    cx<R> x00 = *p00, x10 = *p10, x01 = *p01, x11 = *p11;
    if (m1 != i1) {
      const cx<R> a = x00 - x10, c = x01 - x11;
      x00 = x00 + x10;
      x01 = x01 + x11;
      x10 = a;
      x11 = c;
    }
    if (m2 != i2) {
      const cx<R> a = x00 - x01, c = x10 - x11;
      x00 = x00 + x01;
      x10 = x10 + x11;
      x01 = a;
      x11 = c;
    }
    *p00 = x00;
    if (m1 != i1) *p10 = x10;
    if (m2 != i2) *p01 = x01;
    if (m1 != i1 && m2 != i2) *p11 = x11;
  }
}

__device__ __forceinline__ cx<float> ldg_cx(const cx<float>* p) {
  const float2 u = __ldg(reinterpret_cast<const float2*>(p));
  return mk(u.x, u.y);
}
__device__ __forceinline__ cx<double> ldg_cx(const cx<double>* p) {
  const double2 u = __ldg(reinterpret_cast<const double2*>(p));
  return mk(u.x, u.y);
}

template <typename R, bool STAGE>
__global__ void __launch_bounds__(PS_THREADS, sizeof(R) == 4 ? 3 : 2)
    k_planes_parity(const cx<R>* A, cx<R>* __restrict__ B, const cx<R>* __restrict__ mE,
                    const cx<R>* __restrict__ mI, int P0, const int32_t* __restrict__ acoord, int nac, int R1, int R2,
                    int words, int ident, int64_t cs, int ncol) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int q0 = blockIdx.x, med = blockIdx.y, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nb = R1 * R2, npl = (q0 == 0 || 2 * q0 == P0) ? 1 : 2, tot = npl * nb;
  const bool onepass = 2 * nb <= PS_THREADS;  // every result waits in its thread's registers
  cx<R>* src = reinterpret_cast<cx<R>*>(smem_raw);  // [plane][i1][i2][PS_W]
  cx<R>* res = onepass ? src : src + 2 * nb * PS_W;
  cx<R>* Ms = res + 2 * nb * PS_W;
  int32_t* crd = reinterpret_cast<int32_t*>(Ms + (STAGE ? words + (words & 1) : 0));
  const cx<R>* Mg = (med ? mI : mE) + (int64_t)q0 * words;
  if (STAGE) {  // 8 bytes per copy in complex64 (a table may start on an odd value), 16 in complex128
    for (int i = threadIdx.x; i < words; i += PS_THREADS)
      asm volatile("cp.async.ca.shared.global [%0], [%1], %2;\n" ::"r"((unsigned)__cvta_generic_to_shared(Ms + i)),
                   "l"(Mg + i), "n"((int)sizeof(cx<R>))
                   : "memory");
  }
  const cx<R>* M0 = STAGE ? Ms : Mg;
  const int E1 = (R1 + 1) / 2, E2 = (R2 + 1) / 2, O1 = R1 - E1, O2 = R2 - E2;
  for (int i = threadIdx.x; i < nac; i += PS_THREADS) {
    const int c = acoord[i];
    crd[i] = (c >> 16) * R2 + (c & 0xffff);
  }
  // rows (plane, field) warp and warp + 8; four columns per lane in flight
  const cx<R>* rp[2];
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int v = warp, pl = h, k0 = pl ? P0 - q0 : q0;
    const int f = ident ? 8 * med + v : (v < 4 ? (med ? 4 + v : v) : 8 + (v - 4));
    rp[h] = A + (int64_t)(f * P0 + k0) * nac;
  }
  pdl_wait();
  bool first = true;
  for (int col = blockIdx.z; col < ncol; col += gridDim.z, first = false) {
    for (int i = threadIdx.x; i < 2 * nb * PS_W; i += PS_THREADS) src[i] = czero<R>();
    __syncthreads();
    for (int jb = 0; jb < nac; jb += 128) {
      cx<R> x[2][4];
#pragma unroll
      for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int j = jb + 32 * u + lane;
          if (h < npl && j < nac) x[h][u] = rp[h][col * cs + j];
        }
#pragma unroll
      for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int j = jb + 32 * u + lane;
          if (h < npl && j < nac) src[(h * nb + crd[j]) * PS_W + warp] = x[h][u];
        }
    }
    __syncthreads();
    parity_pass<R>(src, R1, R2, npl);
    if (STAGE && first) asm volatile("cp.async.wait_all;\n" ::: "memory");
    __syncthreads();
    for (int u = threadIdx.x; u < (onepass ? PS_THREADS : tot); u += PS_THREADS) {
      Acc8<R> acc;
      acc.zero();
      int at = 0;
      if (u < tot) {
        // block (odd along axis 1, odd along axis 2) and index in it; blocks in
        // the order (even, even), (even, odd), (odd, even), (odd, odd)
        const int pl = u >= nb;
        int a = u - pl * nb;
        const bool s1 = a >= E1 * R2;
        a -= s1 ? E1 * R2 : 0;
        const int n1 = s1 ? O1 : E1;
        const bool s2 = a >= n1 * E2;
        a -= s2 ? n1 * E2 : 0;
        const int n2 = s2 ? O2 : E2, n = n1 * n2, a1 = a / n2, a2 = a - a1 * n2;
        at = pl * nb + (s1 ? R1 - 1 - a1 : a1) * R2 + (s2 ? R2 - 1 - a2 : a2);
        const cx<R>* M = M0 + (s1 ? E1 * E1 * (E2 * E2 + O2 * O2) : 0) + (s2 ? n1 * n1 * E2 * E2 : 0) + a;
        const cx<R>* sp = src + (pl * nb + (s1 ? (R1 - 1) * R2 : 0) + (s2 ? R2 - 1 : 0)) * PS_W;
        const int st1 = (s1 ? -R2 : R2) * PS_W, st2 = s2 ? -PS_W : PS_W;
        for (int j1 = 0; j1 < n1; ++j1) {
          const cx<R>* sj = sp + j1 * st1;
#pragma unroll 4
          for (int j2 = 0; j2 < n2; ++j2) {
            acc.mac(STAGE ? *M : ldg_cx(M), sj);
            M += n;
            sj += st2;
          }
        }
      }
      if (onepass) __syncthreads();  // the sources are read before the results replace them
      if (u < tot)
#pragma unroll
        for (int v = 0; v < 8; ++v) res[(int64_t)at * PS_W + v] = acc.get(v);
    }
    __syncthreads();
    parity_pass<R>(res, R1, R2, npl);
    __syncthreads();
    for (int u = threadIdx.x; u < npl * nac * 8; u += PS_THREADS) {  // fields fastest: 64 bytes in complex64
      const int v = u & 7, w = u >> 3, h = w >= nac, j = w - h * nac;
      const cx<R> val = res[(h * nb + crd[j]) * PS_W + v];
      B[col * cs + ((int64_t)(h ? P0 - q0 : q0) * nac + j) * NFIELD_OUT + 8 * med + v] =
          (!ident && med && v >= 4) ? -val : val;
    }
    __syncthreads();
  }
}

// Shared memory of the parity form: the two planes, a second pair for the
// results when the positions outnumber the threads, the table when staged, the
// columns' positions.
size_t parity_smem(int nb, int64_t nac, int64_t staged, size_t csz) {
  return (size_t)2 * nb * PS_W * csz * (2 * nb <= PS_THREADS ? 1 : 2) + (size_t)(staged + (staged & 1)) * csz +
         sizeof(int32_t) * nac;
}

// Compiled plane sizes: (2^l1) x (2^l2) with 3 <= l1, l2 <= 7 and l1 + l2 <= 12.
template <typename R>
PlanesFn<R> planes_kernel(int l1, int l2) {
  switch (l1) {
    case 3: return planes_row<R, 3>(l2);
    case 4: return planes_row<R, 4>(l2);
    case 5: return planes_row<R, 5>(l2);
    case 6: return planes_row<R, 6>(l2);
    case 7: return planes_row<R, 7>(l2);
    default: return nullptr;
  }
}

// ---------------------------------------------------------------- generic 3-D FFT (set-up, complex128)
template <typename R, int DIR>
__global__ void __launch_bounds__(FFT_THREADS) k_fft_axis(cx<R>* data, int len, int inner, int64_t nlines, int CB,
                                                          const cx<R>* __restrict__ tw) {
  extern __shared__ unsigned char smem_raw[];
  cx<R>* tws = reinterpret_cast<cx<R>*>(smem_raw);
  cx<R>* b0 = tws + len;
  const int64_t L0 = (int64_t)blockIdx.x * CB;
  const int lcb = ilog2(CB);
  for (int i = threadIdx.x; i < len; i += FFT_THREADS) tws[i] = tw[i];
  for (int idx = threadIdx.x; idx < len * CB; idx += FFT_THREADS) {
    const int j = idx >> lcb, l = idx & (CB - 1);
    const int64_t L = L0 + l;
    cx<R> v = czero<R>();
    if (L < nlines) v = data[(L / inner) * ((int64_t)len * inner) + (L % inner) + (int64_t)j * inner];
    b0[idx] = v;
  }
  __syncthreads();
  fft_lines<R, DIR, Tot<R>::L>(b0, ilog2(len), lcb, 1, CB, tws);
  for (int idx = threadIdx.x; idx < len * CB; idx += FFT_THREADS) {
    const int j = idx >> lcb, l = idx & (CB - 1);
    const int64_t L = L0 + l;
    if (L < nlines) data[(L / inner) * ((int64_t)len * inner) + (L % inner) + (int64_t)j * inner] = b0[idx];
  }
}

template <typename R>
__global__ void k_twiddles(cx<R>* tw, int len) {
  int m = blockIdx.x * blockDim.x + threadIdx.x;
  if (m >= len) return;
  double s, c;
  sincospi(2.0 * (double)m / (double)len, &s, &c);
  tw[m] = mk(R(c), R(-s));
}

// Lines per CTA for a transform of length len: up to 2^Tot<R>::L elements,
// at most 16 lines.
template <typename R>
int lines_per_cta(int len) {
  int cb = (1 << Tot<R>::L) / len;
  if (cb > 16) cb = 16;
  if (cb < 1) cb = 1;
  return cb;
}

}  // namespace

template <typename R>
int make_twiddles(cx<R>* tw, int len, cudaStream_t s) {
  k_twiddles<R><<<(int)cdiv(len, 256), 256, 0, s>>>(tw, len);
  CK(cudaGetLastError());
  return SCABEM_OK;
}

// Full-length transform along one axis of a P0 x P1 x P2 array (set-up).
template <typename R>
int fft_axis_full(scabem_op* op, cx<R>* data, int a, const cx<R>* tw, int dir, cudaStream_t s) {
  const int64_t total = (int64_t)op->P[0] * op->P[1] * op->P[2];
  const int len = op->P[a];
  int inner = 1;
  for (int b = a + 1; b < 3; ++b) inner *= op->P[b];
  const int64_t nlines = total / len;
  const int cb = lines_per_cta<R>(len);
  const size_t sm = (size_t)len * (cb + 1) * sizeof(cx<R>);
  const int blocks = (int)cdiv(nlines, cb);
  if (dir < 0) {
    CK(cudaFuncSetAttribute(k_fft_axis<R, -1>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
    k_fft_axis<R, -1><<<blocks, FFT_THREADS, sm, s>>>(data, len, inner, nlines, cb, tw);
  } else {
    CK(cudaFuncSetAttribute(k_fft_axis<R, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
    k_fft_axis<R, 1><<<blocks, FFT_THREADS, sm, s>>>(data, len, inner, nlines, cb, tw);
  }
  CK(cudaGetLastError());
  return SCABEM_OK;
}

template <typename R>
int fft3d_full(scabem_op* op, cx<R>* data, const cx<R>* const tw[3], int dir, cudaStream_t s) {
  for (int a = 0; a < 3; ++a) {
    int rc = fft_axis_full<R>(op, data, a, tw[a], dir, s);
    if (rc) return rc;
  }
  return SCABEM_OK;
}

// Lines per CTA of the pruned axis-0 stages for `units` lines (field, column):
// 8, so that the few active columns of a long guide still spread over the
// SMs; more for short transforms, up to the eight elements per thread that
// the radix-8 passes take, while a CTA per SM remains (a 64-point transform
// of 8 lines keeps 64 of 512 threads busy).
template <typename R>
int pruned_lines(int P0, int64_t units) {
  int l = lines_per_cta<R>(P0);
  l = l < 8 ? l : 8;
  while (P0 * l < 8 * FFT_THREADS && units / (2 * l) >= 152) l *= 2;
  return l;
}

// stage C: 16 fields [field][k0][c] -> point-major groups, active columns
template <typename R>
static int axis0_inverse(scabem_op* op, PrecData<R>& pd, cudaStream_t s, bool adjoint, int ncol) {
  const int P0 = op->P[0];
  const int lines = op->a0_lines > 0 ? op->a0_lines : pruned_lines<R>(P0, 16 * op->nac * ncol);
  const int nc = lines >= 8 ? lines / 8 : 1;  // eight lines of P0 <= 1024 always fit
  const size_t sm = (size_t)P0 * (8 * nc + 1) * sizeof(cx<R>);
  const bool big = P0 * 8 * nc > (1 << Tot<R>::L);
  auto fn = big ? (adjoint ? k_axis0_pm<R, false, 13> : k_axis0_pm<R, true, 13>)
                : (adjoint ? k_axis0_pm<R, false, Tot<R>::L> : k_axis0_pm<R, true, Tot<R>::L>);
  if (int rc_ = set_max_smem(op->device, (const void*)fn, (int)sm)) return rc_;
  CK(launch_pdl(fn, dim3((unsigned)cdiv(op->nac, nc), 2, ncol), FFT_THREADS, sm, s, pd.stB, pd.grid, op->n[0], P0,
      op->acol, (int)op->nac, nc, pd.tw[0], col_stride_st(op), col_stride_pot(op), op->cst, op->tdirect ? 1 : 0,
      (R)op->ke, (R)op->ki, (R)op->ze, (R)op->zi));
  return SCABEM_OK;
}

template <typename R>
int fft_conv(scabem_op* op, PrecData<R>& pd, cudaStream_t s, bool adjoint, int ncol) {
  const int n0 = op->n[0], n1 = op->n[1], n2 = op->n[2];
  const int nf = adjoint ? NFIELD_OUT : NFIELD_IN;  // fields transformed along axis 0
  const int id = adjoint ? 1 : 0;
  const int P0 = op->P[0], P1 = op->P[1], P2 = op->P[2];
  if (op->nac == 0) {
    set_error("grid: no grid point is covered by a stencil");
    return SCABEM_E_ARG;
  }
  const int cb = op->a0_lines > 0 ? op->a0_lines : pruned_lines<R>(P0, nf * op->nac * ncol);
  const size_t sm0 = (size_t)P0 * (cb + 1) * sizeof(cx<R>);
  // stage A
  if (int rc_ = set_max_smem(op->device, (const void*)k_axis0<R>, (int)sm0)) return rc_;
  CK(launch_pdl(k_axis0<R>, dim3((unsigned)cdiv(op->nac, cb), nf, ncol), FFT_THREADS, sm0, s, pd.src, pd.stA, n0,
      P0, op->acol, (int)op->nac, cb, pd.tw[0], col_stride_src(op), col_stride_st(op), op->cst, op->tdirect ? 1 :
      0));
  prof_mark(op, s);
  // stage B
  if (op->tdirect && op->parity) {
    const int words = (int)parity_words(op), nb = op->R1 * op->R2;
    const bool stage = parity_smem(nb, op->nac, words, sizeof(cx<R>)) <= 100 * 1024;  // two CTAs per SM and more
    const size_t sm = parity_smem(nb, op->nac, stage ? words : 0, sizeof(cx<R>));
    auto fn = stage ? k_planes_parity<R, true> : k_planes_parity<R, false>;
    if (int rc_ = set_max_smem(op->device, (const void*)fn, (int)sm)) return rc_;
    // two CTAs per SM from the columns of a batch where the frequencies are few
    const unsigned zs = (unsigned)std::min<int64_t>(ncol, cdiv(2 * 152, P0 + 2));
    CK(launch_pdl(fn, dim3(P0 / 2 + 1, 2, zs), PS_THREADS, sm, s, pd.stA, pd.stB, pd.gt[0], pd.gt[1], P0, op->acoord,
      (int)op->nac, op->R1, op->R2, words, id, col_stride_st(op), ncol));
    prof_mark(op, s);
    return axis0_inverse(op, pd, s, adjoint, ncol);
  }
  if (op->tdirect) {
    const size_t sm = ((size_t)op->nac * 8 + (size_t)op->R1 * op->R2) * sizeof(cx<R>) + sizeof(int32_t) * op->nac;
    if (int rc_ = set_max_smem(op->device, (const void*)k_planes_direct<R>, (int)sm)) return rc_;
    CK(launch_pdl(k_planes_direct<R>, dim3(P0, 2, ncol), PD_THREADS, sm, s, pd.stA, pd.stB, pd.gt[0], pd.gt[1], P0,
                  op->acoord, (int)op->nac, op->R1, op->R2, id, col_stride_st(op)));
    prof_mark(op, s);
    return axis0_inverse(op, pd, s, adjoint, ncol);
  }
  if (P1 == 64 && P2 == 64) {
    const size_t sm = ((size_t)2 * 32 * 64 + (size_t)(P64_THREADS / 8) * P64_SCR) * sizeof(cx<R>);
    if (int rc_ = set_max_smem(op->device, (const void*)k_planes64<R>, (int)sm)) return rc_;
    CK(launch_pdl(k_planes64<R>, dim3(P0, nf, ncol), P64_THREADS, sm, s, pd.stA, pd.stB, pd.ghat[0], pd.ghat[1], P0,
      pd.tw[1], op->rowmask, id, col_stride_st(op)));
    prof_mark(op, s);
    return axis0_inverse(op, pd, s, adjoint, ncol);
  }
  const size_t sm1 = ((size_t)P1 + P2 + 2 * (size_t)P1 * (P2 + 2)) * sizeof(cx<R>);
  PlanesFn<R> fn = planes_kernel<R>(ilog2(P1), ilog2(P2));
  if (!fn) {
    set_error("grid: the y and z transform sizes must be in [8, 128]");
    return SCABEM_E_ARG;
  }
  if (int rc_ = set_max_smem(op->device, (const void*)fn, (int)sm1)) return rc_;
  CK(launch_pdl(fn, dim3(P0, nf, ncol), PLANE_THREADS, sm1, s, pd.stA, pd.stB, pd.ghat[0], pd.ghat[1], P0, n1, n2,
      pd.tw[1], pd.tw[2], id, col_stride_st(op)));
  prof_mark(op, s);
  return axis0_inverse(op, pd, s, adjoint, ncol);
}

// The parity form where its products, (E1^2 + O1^2)(E2^2 + O2^2) per field and
// frequency against nac^2, are fewer (they are not when the box holds few
// active columns: two guides far apart; 12 um guide 18 us against 29 for the
// direct sums, complex128 219 against 733), its planes fit in shared memory and
// its tables stay below 1 GiB.
void choose_parity(scabem_op* op) {
  const int64_t nb = (int64_t)op->R1 * op->R2;
  const size_t csz = (op->prec_mask & 2) ? sizeof(cx<double>) : sizeof(cx<float>);
  const int64_t w = parity_words(op);
  op->parity = w < op->nac * op->nac && w <= INT32_MAX && nb < (1 << 16) && parity_smem((int)nb, op->nac, 0, csz) <= 227 * 1024 &&
               2 * w * (op->P[0] / 2 + 1) * (int64_t)csz <= (1ll << 30);
}

template int make_twiddles<float>(cx<float>*, int, cudaStream_t);
template int make_twiddles<double>(cx<double>*, int, cudaStream_t);
template int fft3d_full<double>(scabem_op*, cx<double>*, const cx<double>* const[3], int, cudaStream_t);
template int fft_axis_full<double>(scabem_op*, cx<double>*, int, const cx<double>*, int, cudaStream_t);
template int fft_conv<float>(scabem_op*, PrecData<float>&, cudaStream_t, bool, int);
template int fft_conv<double>(scabem_op*, PrecData<double>&, cudaStream_t, bool, int);
