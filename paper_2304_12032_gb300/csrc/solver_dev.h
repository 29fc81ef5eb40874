// Device types and small device functions shared by the linear-algebra kernels (solver.cu) and the
// persistent Krylov cycle (cycle.cu): vector records, BF16 unpacking, matrix blocks, the sub-block
// and CSR views, row dot products.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "kernels.h"
#include "solver.h"

namespace lfx {

template <class T> struct Vec4T;
template <> struct Vec4T<double> { using type = D4; };
template <> struct Vec4T<float> { using type = F4; };

// Arithmetic type of the vector kernels: FP32 vectors (the inner solve) are combined in FP32 and
// only per-thread partial sums are widened to FP64 for the cross-thread reduction; FP64 vectors
// stay FP64 throughout.  (FP64 instructions issue at 1/61 of the FP32 rate on this part, so an
// FP64 accumulator would make the FP32 Krylov kernels arithmetic-bound.)
template <class T, class X = T> struct AccT { using type = double; };
template <> struct AccT<float, float> { using type = float; };

template <class T>
__device__ __forceinline__ typename Vec4T<T>::type ld4(const T *p, int64_t i) {
  return reinterpret_cast<const typename Vec4T<T>::type *>(p)[i];
}
template <class T>
__device__ __forceinline__ void st4(T *p, int64_t i, const typename Vec4T<T>::type &v) {
  reinterpret_cast<typename Vec4T<T>::type *>(p)[i] = v;
}

// Two packed BF16 values to FP32 (exact: a BF16 value is the top half of its FP32 value).  Bit
// operations on the integer pipe; the conversion instruction would take FP64-pipe issue slots.
__device__ __forceinline__ void bf16x2_to_f32(uint32_t w, float &lo, float &hi) {
  lo = __uint_as_float(w << 16);
  hi = __uint_as_float(w & 0xffff0000u);
}

template <class S, class A>
__device__ __forceinline__ void ld_block(const S *vals, int64_t k, A b[16]);
template <>
__device__ __forceinline__ void ld_block<double, double>(const double *vals, int64_t k, double b[16]) {
  const double2 *p = reinterpret_cast<const double2 *>(vals + 16 * k);
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    double2 v = __ldg(p + i);
    b[2 * i] = v.x;
    b[2 * i + 1] = v.y;
  }
}
template <>
__device__ __forceinline__ void ld_block<float, float>(const float *vals, int64_t k, float b[16]) {
  const float4 *p = reinterpret_cast<const float4 *>(vals + 16 * k);
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    float4 v = __ldg(p + i);
    b[4 * i] = v.x;
    b[4 * i + 1] = v.y;
    b[4 * i + 2] = v.z;
    b[4 * i + 3] = v.w;
  }
}
template <>
__device__ __forceinline__ void ld_block<__nv_bfloat16, float>(const __nv_bfloat16 *vals, int64_t k, float b[16]) {
  const uint4 *p = reinterpret_cast<const uint4 *>(vals + 16 * k);
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    uint4 v = __ldg(p + i);
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int q = 0; q < 4; ++q) bf16x2_to_f32(w[q], b[8 * i + 2 * q], b[8 * i + 2 * q + 1]);
  }
}
template <>
__device__ __forceinline__ void ld_block<float, double>(const float *vals, int64_t k, double b[16]) {
  const float4 *p = reinterpret_cast<const float4 *>(vals + 16 * k);
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    float4 v = __ldg(p + i);
    b[4 * i] = v.x;
    b[4 * i + 1] = v.y;
    b[4 * i + 2] = v.z;
    b[4 * i + 3] = v.w;
  }
}

// a smoothing coefficient in the arithmetic type T (the FP32 kernels read the FP32 copy)
template <class T>
__device__ __forceinline__ T coef_t(const double &d, const float &) {
  return (T)d;
}
template <>
__device__ __forceinline__ float coef_t<float>(const double &, const float &f) {
  return f;
}

__device__ __forceinline__ bool finished(const KState *st) {
  return st != nullptr && *(volatile const int *)&st->done != 0;
}

template <class S>
struct SplitView {
  int64_t V;
  const int32_t *rowptr, *col, *diag, *trans;
  const S *F;    // [nnzb][12]: F00 F01 F02 F10 F11 F12 F20 F21 F22 0 0 0
  const S *G;    // [nnzb][4]:  G0 G1 G2 0
  const S *DC;   // [nnzb][4]:  D0 D1 D2 C
};

// N consecutive values (N a multiple of 4) from an aligned record
template <int N>
__device__ __forceinline__ void ld_rec(const double *p, double *o) {
#pragma unroll
  for (int i = 0; i < N / 2; ++i) {
    const double2 v = __ldg(reinterpret_cast<const double2 *>(p) + i);
    o[2 * i] = v.x;
    o[2 * i + 1] = v.y;
  }
}
template <int N>
__device__ __forceinline__ void ld_rec(const float *p, float *o) {
#pragma unroll
  for (int i = 0; i < N / 4; ++i) {
    const float4 v = __ldg(reinterpret_cast<const float4 *>(p) + i);
    o[4 * i] = v.x;
    o[4 * i + 1] = v.y;
    o[4 * i + 2] = v.z;
    o[4 * i + 3] = v.w;
  }
}
template <int N>
__device__ __forceinline__ void ld_rec(const __nv_bfloat16 *p, float *o) {
#pragma unroll
  for (int i = 0; i < N / 4; ++i) {
    const uint2 v = __ldg(reinterpret_cast<const uint2 *>(p) + i);
    bf16x2_to_f32(v.x, o[4 * i], o[4 * i + 1]);
    bf16x2_to_f32(v.y, o[4 * i + 2], o[4 * i + 3]);
  }
}

// ---- explicit CSR levels of the Schur AMG (scalar unknowns).  Values are stored in the
// preconditioner's vector type T (FP32 for the mixed-precision inner solve, FP64 otherwise).
template <class VT>
struct CsrV {
  int64_t n;
  const int32_t *rp, *ci;
  const VT *v;
};

// sum_k v[k] x[ci[k]*is + io] over the row, G lanes per row (lane = position in the group),
// four nonzeros per lane in flight; the group's total is returned in every lane of the group.
// Lanes with valid == false add nothing but take part in the shuffles.
template <int G, class T>
__device__ __forceinline__ typename AccT<T>::type csr_row_dot(const int32_t *__restrict__ rp,
                                                              const int32_t *__restrict__ ci,
                                                              const T *__restrict__ v, const T *x, int is, int io,
                                                              int64_t row, int lane, bool valid) {
  using A = typename AccT<T>::type;
  A s = A(0);
  if (valid) {
    const int32_t k1 = __ldg(rp + row + 1);
    int32_t k = __ldg(rp + row) + lane;
    for (; k + 3 * G < k1; k += 4 * G) {
      int32_t c[4];
      T w[4], xv[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        c[u] = __ldg(ci + k + u * G);
        w[u] = __ldg(v + k + u * G);
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) xv[u] = x[(int64_t)c[u] * is + io];
#pragma unroll
      for (int u = 0; u < 4; ++u) s += (A)w[u] * (A)xv[u];
    }
    for (; k < k1; k += G) s += (A)__ldg(v + k) * (A)x[(int64_t)__ldg(ci + k) * is + io];
  }
#pragma unroll
  for (int o = G / 2; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  return s;
}

// sum_k Minv[row][k] b[k*is+io] over one warp (eight columns per lane in flight)
template <class T>
__device__ __forceinline__ typename AccT<T>::type dense_row_dot(int64_t n, const T *__restrict__ Minv, const T *b,
                                                                int is, int io, int64_t row, int lane, bool valid) {
  using A = typename AccT<T>::type;
  A s = A(0);
  if (valid) {
    const T *m = Minv + row * n;
    int64_t k = lane;
    for (; k + 7 * 32 < n; k += 8 * 32) {
      T w[8], xv[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        w[u] = __ldg(m + k + u * 32);
        xv[u] = b[(k + u * 32) * is + io];
      }
#pragma unroll
      for (int u = 0; u < 8; ++u) s += (A)w[u] * (A)xv[u];
    }
    for (; k < n; k += 32) s += (A)__ldg(m + k) * (A)b[k * is + io];
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  return s;
}

template <class T>
struct CoarseLevel {
  int64_t n, nnext;
  const int32_t *rp, *ci;
  const T *v, *dinv;
  const int32_t *Prp, *Pci;
  const T *Pv;
  const int32_t *Rrp, *Rci;
  const T *Rv;
  T *x, *b, *r, *d0, *d1, *rr;
  T *xo;   // where the level's final iterate is left (d1 when one smoothing step is fused, else x)
  typename AccT<T>::type init, c1[kMaxSmooth], c2[kMaxSmooth];   // (converted on the host)
};
constexpr int kMaxCoarse = 8;
template <class T>
struct CoarseArgs {
  int L;            // levels in amg[] (level 0 is matrix-free and not part of this launch)
  int s_steps;
  typename AccT<T>::type alpha;
  const T *coarse_inv;
  int64_t nc;
  CoarseLevel<T> lv[kMaxCoarse];
};

}  // namespace lfx
