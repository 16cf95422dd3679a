// Small device helpers shared by the kernels of the product.
#pragma once

#include "common.cuh"

// a += s * b on (re, im) as one packed FP32x2 FMA in complex64.
__device__ __forceinline__ void axpy2(cx<float>& a, float s, cx<float> b) {
  const float2 r = __ffma2_rn(make_float2(s, s), make_float2(b.re, b.im), make_float2(a.re, a.im));
  a = mk(r.x, r.y);
}
__device__ __forceinline__ void axpy2(cx<double>& a, double s, cx<double> b) { axpy(a, s, b); }

// a += v * x (complex); complex64 as two packed FP32x2 FMAs
__device__ __forceinline__ void cmac(cx<double>& a, cx<double> v, cx<double> x) { cfma(a, v, x); }
__device__ __forceinline__ void cmac(cx<float>& a, cx<float> v, cx<float> x) {
  float2 r = __ffma2_rn(make_float2(v.re, v.re), make_float2(x.re, x.im), make_float2(a.re, a.im));
  r = __ffma2_rn(make_float2(v.im, v.im), make_float2(-x.im, x.re), r);
  a = mk(r.x, r.y);
}

// Four consecutive complex values from a 16-byte boundary (32 bytes in complex64)
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
// Four reals from a 16-byte boundary
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
// streaming loads of values read once per product, which should not push the
// reused tables and grids out of L2
__device__ __forceinline__ cx<float> ldstream(const cx<float>* p) {
  const float2 u = __ldcs(reinterpret_cast<const float2*>(p));
  return mk(u.x, u.y);
}
__device__ __forceinline__ cx<double> ldstream(const cx<double>* p) {
  const double2 u = __ldcs(reinterpret_cast<const double2*>(p));
  return mk(u.x, u.y);
}

// Right-hand sides of a batch of k go in groups of K, what one warp takes; the
// kernels that gather x read it as [unknown][group][column of the group], the
// columns padded to a power of two with zeros, so that an unknown's entries
// come with one or two 16-byte loads (k_interleave, apply.cu).
inline int batch_group(int k) { return k <= 3 ? k : k == 5 || k == 6 ? 3 : 4; }
__host__ __device__ constexpr int group_pad(int K) { return K == 3 ? 4 : K; }
inline int batch_stride(int k) { return (int)cdiv(k, batch_group(k)) * group_pad(batch_group(k)); }

template <typename R, int K>
__device__ __forceinline__ void load_cols(const cx<R>* p, cx<R>* v) {
  if constexpr (K == 1) {
    v[0] = *p;
  } else if constexpr (sizeof(R) == 8) {
#pragma unroll
    for (int c = 0; c < K; ++c) {
      const double2 u = *(reinterpret_cast<const double2*>(p) + c);
      v[c] = mk((R)u.x, (R)u.y);
    }
  } else {
#pragma unroll
    for (int c = 0; c < K; c += 2) {
      const float4 u = *reinterpret_cast<const float4*>(p + c);
      v[c] = mk((R)u.x, (R)u.y);
      if (c + 1 < K) v[c + 1] = mk((R)u.z, (R)u.w);
    }
  }
}

template <typename R>
__device__ __forceinline__ cx<R> shfl_xor_cx(cx<R> v, int o) {
  return mk(__shfl_xor_sync(0xffffffffu, v.re, o), __shfl_xor_sync(0xffffffffu, v.im, o));
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
    v[t] = keep + shfl_xor_cx(send, o);
  }
}
template <typename R>
__device__ __forceinline__ cx<R> xadd(cx<R> v, int o) {
  return v + shfl_xor_cx(v, o);
}

// Programmatic dependent launch: a kernel of the product starts while its
// predecessor in the stream still runs, sets itself up from data that no kernel
// of the stream writes, and waits here for the predecessor's completion.  Only
// then does it let its own successor start, so a kernel that is running knows
// that everything before its direct predecessor has completed.  Every kernel
// launched with launch_pdl comes through pdl_wait before it reads or writes
// what the stream's kernels share.
//
// What the direct predecessor writes is therefore written during this kernel's
// lifetime, and the read-only path (__ldg, or const with __restrict__) is defined
// only for memory that nobody writes meanwhile.  These kernels read it with plain loads
// through pointers without __restrict__, which the "memory" clobber keeps below
// the wait; const __restrict__ is for set-up tables and for vectors that were
// complete before the predecessor started.
__device__ __forceinline__ void pdl_wait() {
  asm volatile("griddepcontrol.wait;\n" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
}
template <typename... KA, typename... A>
inline cudaError_t launch_pdl(void (*kernel)(KA...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, A&&... args) {
  cudaLaunchConfig_t c = {};
  c.gridDim = grid;
  c.blockDim = block;
  c.dynamicSmemBytes = smem;
  c.stream = s;
  cudaLaunchAttribute a = {};
  a.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  a.val.programmaticStreamSerializationAllowed = 1;
  c.attrs = &a;
  c.numAttrs = 1;
  return cudaLaunchKernelEx(&c, kernel, static_cast<KA>(args)...);
}
