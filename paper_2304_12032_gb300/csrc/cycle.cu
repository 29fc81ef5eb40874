// One GMRES cycle as one cooperative launch: the aSIMPLE preconditioner (velocity Chebyshev passes,
// Schur multigrid cycle), the product with the operator, Gram-Schmidt and the stopping test of every
// Arnoldi step, then the update of the iterate.
//
// Why one launch.  A step is about twenty dependent passes.  As separate kernels each costs 4-5 us at
// every size (launch, three dependent loads from L2, drain), so a 19k-tetrahedron solve and a 150k one
// took nearly the same time and the host had to poll a stop flag per step.  Here each CTA owns a fixed
// range of block rows for the whole cycle: their vectors (residual, iterate, diagonals, Krylov vector)
// stay in its shared memory, velocity records too as far as they fit, and a pass costs one grid
// barrier.  Vectors read at neighbour rows go through global memory: at the start of a pass the CTA
// copies its own entries and those of its halo (each neighbour once) into shared memory, and the blocks
// address them by 16-bit local indices (in the padding of the velocity and gradient records).  A node is read by about fifteen rows, so gathering from L2 row
// by row moved seven times the bytes of the copy (17 us a velocity pass at 1M tetrahedra, L2-bound).
//
// Measured (ms per time step, step-by-step launches and this): 3k tetrahedra FP64 2.87 and 1.54 (1.11 with
// the gathered assembly), 19k mixed 4.98 and 3.28, 100k FP64 15.4 and 7.7, 150k mixed with Newton 21.3 and 15.7,
// 500k mixed 16.1 and 10.9, 600k FP64 48.4 and 33.2, 1.02M mixed 24.1 and 17.9.  A pass costs 1.4 us for the
// barrier (waiting for the halo's CTAs only: 2 us, their flags arrive one by one), 1.1 to 1.7 us of latency
// (neighbour copy, records, sums) at 32 rows per CTA, and then grows with the rows: at 1M tetrahedra 14 us per
// velocity pass and 7 us per gradient or divergence pass.  No unit is full there (over a launch at 818k the L1 data
// pipe is 46 % busy, issue 28 %, DRAM 21 %): barrier, halo copy and the first record loads follow one another.
// FP64 passes run at the FP64 pipe's rate (a velocity pass at 108k nodes: 45 us, 37 us of it FP64 issue); with the
// barriers the pipe is 50 % busy over a launch at 102k tetrahedra.  A system within amg_coarse_size has 11 passes
// per step, the dense inverse among them (729 nodes, FP64: 3.9 us each).
//
// A batch of independent meshes runs the same way, each piece with CTAs, basis, sums and stopping test of its
// own (16 meshes of 10k to 40k tetrahedra in one launch: 13.3 -> 8.0 ms a step).
//
// One extra CTA owns no rows.  It runs the FP64 recurrences of a step (Hessenberg column, rotations,
// stopping test, back substitution) while the others are already in the next step's velocity passes,
// and they read its verdict after the first of those passes.
//
// Every wait is bounded: a CTA that gives up sets the error word and returns, the others then run into
// their own limits.  The CTA without rows, or the next cycle's at its start, flags the solve's status, and the
// host ends the solve with LFX_ERR_TIMEOUT.
#include <algorithm>
#include <cstddef>
#include <type_traits>

#include "cycle.h"
#include "dd.h"
#include "grid_wait.h"

namespace lfx {

namespace {

constexpr int kSmemCap = 220 * 1024, kExtraCap = 190 * 1024;
constexpr int kDots = 8;                  // shares of one dot product in a CTA

template <class T, int LPR> struct Shape { static constexpr int threads = sizeof(T) == 8 ? 512 : 1024; };

// sums of T: FP64 values, or FP32 pairs whose low word gathers the rounding errors.  (Pairs all the way: the
// launches summed in FP32 per thread and warp and in FP64 between warps.  Error of a product of two vectors
// against 64 bits, relative to their norms, largest of 10 to 40 draws, launches and this: 17k rows 7e-8 and 5e-8,
// 175k 3e-8 and 8e-9, 690k 3e-8 and 1.3e-8; of the summation alone 1e-8 to 9e-8 and below 3e-14.)
template <class T> struct Sum;
template <> struct Sum<double> {
  using type = double;
  static __device__ __forceinline__ double zero() { return 0.0; }
  static __device__ __forceinline__ void add(double &s, double v) { s += v; }
  static __device__ __forceinline__ double shfl(double s, int o) { return __shfl_xor_sync(0xffffffffu, s, o); }
  static __device__ __forceinline__ void join(double &s, double v) { s += v; }
  static __device__ __forceinline__ double value(double s) { return s; }
  static __device__ __forceinline__ double rounded(double s) { return s; }
  static __device__ __forceinline__ double inv_sqrt(double s) { return s > 0.0 ? 1.0 / sqrt(s) : 0.0; }
};
template <> struct Sum<float> {
  using type = float2;
  static __device__ __forceinline__ float2 zero() { return make_float2(0.f, 0.f); }
  static __device__ __forceinline__ void add(float2 &s, float v) {
    const dd t = two_sum(s.x, v);
    s = make_float2(t.hi, f_add(s.y, t.lo));
  }
  static __device__ __forceinline__ float2 shfl(float2 s, int o) {
    return make_float2(__shfl_xor_sync(0xffffffffu, s.x, o), __shfl_xor_sync(0xffffffffu, s.y, o));
  }
  static __device__ __forceinline__ void join(float2 &s, float2 v) {
    const dd t = two_sum(s.x, v.x);
    s = make_float2(t.hi, f_add(f_add(s.y, v.y), t.lo));
  }
  static __device__ __forceinline__ double value(float2 s) { return (double)s.x + (double)s.y; }
  static __device__ __forceinline__ float rounded(float2 s) { return f_add(s.x, s.y); }
  static __device__ __forceinline__ float inv_sqrt(float2 s) { return inv_sqrt_once(s.x, s.y); }
};

__device__ __forceinline__ unsigned long long now_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
  return t;
}

// matrix values read once per step: the preconditioner's sub-blocks, read up to five times, keep the L2
__device__ __forceinline__ uint64_t stream_policy() {
  uint64_t p;
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
  return p;
}
__device__ __forceinline__ float4 ld_stream(const float4 *p, uint64_t policy) {
  float4 v;
  asm volatile("ld.global.nc.L2::cache_hint.v4.f32 {%0, %1, %2, %3}, [%4], %5;"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
               : "l"(p), "l"(policy));
  return v;
}

// The thread index, opaque to the compiler: index arithmetic derived from it stays inside its pass.
// Hoisted out of the step loop, the twenty passes' addresses overflow the registers, and spills are
// dear here (shared memory leaves little L1 for them).
__device__ __forceinline__ int pass_tid() {
  int t = threadIdx.x;
  asm volatile("" : "+r"(t));
  return t;
}

template <int N, class T>
__device__ __forceinline__ T lanes_sum(T v) {
#pragma unroll
  for (int o = N / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// A velocity record as loaded, its use (acc += F v) and the block's local index in its padding.
struct FRecBf {
  uint2 a, b, c;
  __device__ __forceinline__ void load(const __nv_bfloat16 *rec) {
    const uint2 *p = reinterpret_cast<const uint2 *>(rec);
    a = p[0];
    b = p[1];
    c = p[2];
  }
  __device__ __forceinline__ uint32_t local() const { return c.y >> 16; }
  __device__ __forceinline__ void apply(const F4 &v, float acc[3]) const {
    float f[10];
    bf16x2_to_f32(a.x, f[0], f[1]);
    bf16x2_to_f32(a.y, f[2], f[3]);
    bf16x2_to_f32(b.x, f[4], f[5]);
    bf16x2_to_f32(b.y, f[6], f[7]);
    f[8] = __uint_as_float(c.x << 16);
#pragma unroll
    for (int i = 0; i < 3; ++i) acc[i] += f[3 * i] * v.x + f[3 * i + 1] * v.y + f[3 * i + 2] * v.z;
  }
};
struct FRecF32 {
  float4 a, b, c;
  __device__ __forceinline__ void load(const float *rec) {
    const float4 *p = reinterpret_cast<const float4 *>(rec);
    a = p[0];
    b = p[1];
    c = p[2];
  }
  __device__ __forceinline__ uint32_t local() const { return __float_as_uint(c.w); }
  __device__ __forceinline__ void apply(const F4 &v, float acc[3]) const {
    acc[0] += a.x * v.x + a.y * v.y + a.z * v.z;
    acc[1] += a.w * v.x + b.x * v.y + b.y * v.z;
    acc[2] += b.z * v.x + b.w * v.y + c.x * v.z;
  }
};
// a four-value record as loaded
struct Rec4Bf {
  uint2 v;
  __device__ __forceinline__ void load(const __nv_bfloat16 *p) { v = __ldg(reinterpret_cast<const uint2 *>(p)); }
  __device__ __forceinline__ uint32_t local() const { return v.y >> 16; }   // (G records)
  __device__ __forceinline__ F4 get() const {
    F4 o;
    bf16x2_to_f32(v.x, o.x, o.y);
    bf16x2_to_f32(v.y, o.z, o.w);
    return o;
  }
};
struct Rec4F32 {
  float4 v;
  __device__ __forceinline__ void load(const float *p) { v = __ldg(reinterpret_cast<const float4 *>(p)); }
  __device__ __forceinline__ uint32_t local() const { return __float_as_uint(v.w); }
  __device__ __forceinline__ F4 get() const { return F4{v.x, v.y, v.z, v.w}; }
};
template <class S> struct Rec4;
template <> struct Rec4<__nv_bfloat16> { using type = Rec4Bf; };
template <> struct Rec4<float> { using type = Rec4F32; };
template <class S> struct FRec;
template <> struct FRec<__nv_bfloat16> { using type = FRecBf; };
template <> struct FRec<float> { using type = FRecF32; };

// The CTA's own rows: everything read and written by this CTA alone.
template <class T>
struct Own {
  int32_t r0, n;         // first row, rows
  int32_t *rp;           // [n + 1] row pointers
  const int32_t *halo;   // [loc - n] neighbour rows of other CTAs
  int32_t loc;           // rows and halo together
  T *sv;                 // [4 (loc + 1)] the vector of the pass, then a zero entry
  T *vb;                 // [nb][4 n] the first nb basis vectors' own rows (the others in global memory)
  T *r, *x;              // velocity residual and iterate, df: 1 / diag(F); three values per row, or four in
  const T *df;           // the global vectors that take their place where shared memory is short
  T *t, *xp;             // [n] Schur residual, pressure iterate
  const T *ds;           // [n] 1 / diag(S)
  T *w;                  // [4 n] Krylov vector
};


// ---- row products.  FP32: a row's blocks are dealt to LPR lanes, the lanes' sums joined by shuffles,
// and lane 0 applies the result.  FP64: the FP64 pipe issues one warp instruction per about 19 cycles
// of an SM whatever the number of active lanes, so lanes are dealt to components instead (lane i of a
// row forms component i of every block: no shuffles, and the row's update uses all lanes too).
template <class T, int LPR>
struct Rows;

// three sums over LPR lanes, component i of them on lane i of the group (i < 3)
template <int LPR>
__device__ __forceinline__ float spread3(float acc[3], int lane) {
#pragma unroll
  for (int o = LPR / 2; o >= 4; o >>= 1)
#pragma unroll
    for (int i = 0; i < 3; ++i) acc[i] += __shfl_xor_sync(0xffffffffu, acc[i], o);
  // lanes 4q .. 4q + 3: swap with the odd (even) neighbour, then with the pair
  const bool odd = lane & 1, high = lane & 2;
  const float p = __shfl_xor_sync(0xffffffffu, odd ? acc[0] : acc[1], 1);
  const float q = __shfl_xor_sync(0xffffffffu, acc[2], 1);
  const float mine = (odd ? acc[1] : acc[0]) + p, third = acc[2] + q;
  const float r = __shfl_xor_sync(0xffffffffu, high ? mine : third, 2);
  return (high ? third : mine) + r;
}

template <int LPR>
struct Rows<float, LPR> {
  static constexpr int NT = Shape<float, LPR>::threads;
  static constexpr int U = LPR <= 4 ? 4 : (LPR <= 8 ? 2 : 1);   // blocks in flight per lane
  // sum_k F_k v(col k): use(row, i, sum) on lane i of the row's group.  rec(row): the row's records.
  // (Slots past the row's end load its last block again and multiply the zero entry at sv[loc].)
  template <class S, class Rec, class Use>
  static __device__ __forceinline__ void velocity(const Own<float> &o, const uint16_t *, Rec rec, Use use) {
    const int tid = pass_tid(), g = tid / LPR, lane = tid % LPR;
#pragma unroll 1
    for (int base = 0; base < o.n; base += NT / LPR) {
      const int row = base + g;
      const bool has = row < o.n;
      float acc[3] = {0.f, 0.f, 0.f};
      if (has) {
        const int32_t n = o.rp[row + 1] - o.rp[row];
        const S *q = rec(row);
#pragma unroll 1
        for (int32_t k = lane; k < n; k += U * LPR) {
          typename FRec<S>::type f[U];
#pragma unroll
          for (int u = 0; u < U; ++u) f[u].load(q + 12 * min(k + u * LPR, n - 1));
#pragma unroll
          for (int u = 0; u < U; ++u) f[u].apply(ld4(o.sv, k + u * LPR < n ? f[u].local() : (uint32_t)o.loc), acc);
        }
      }
      const float a = spread3<LPR>(acc, lane);
      if (has && lane < 3) use(row, lane, a);
    }
  }
  // sum_k G_k p(col k)
  template <class S, class Use>
  static __device__ __forceinline__ void gradient(const Own<float> &o, const S *G, const uint16_t *, Use use) {
    const int tid = pass_tid(), g = tid / LPR, lane = tid % LPR;
#pragma unroll 1
    for (int base = 0; base < o.n; base += NT / LPR) {
      const int row = base + g;
      const bool has = row < o.n;
      float acc[3] = {0.f, 0.f, 0.f};
      if (has) {
        const int32_t n = o.rp[row + 1] - o.rp[row];
        const S *q = G + 4 * (int64_t)o.rp[row];
#pragma unroll 1
        for (int32_t k = lane; k < n; k += U * LPR) {
          typename Rec4<S>::type b[U];
#pragma unroll
          for (int u = 0; u < U; ++u) b[u].load(q + 4 * min(k + u * LPR, n - 1));
#pragma unroll
          for (int u = 0; u < U; ++u) {
            const float p = o.sv[k + u * LPR < n ? b[u].local() : (uint32_t)o.loc];
            const F4 v = b[u].get();
            acc[0] += v.x * p;
            acc[1] += v.y * p;
            acc[2] += v.z * p;
          }
        }
      }
      const float a = spread3<LPR>(acc, lane);
      if (has && lane < 3) use(row, lane, a);
    }
  }
  // sum_k D_k v.xyz(col k) (kFull: C_k v.w - D_k v.xyz): use(row, sum) on lane 0
  template <bool kFull, class S, class Use>
  static __device__ __forceinline__ void divergence(const Own<float> &o, const S *DC, const uint16_t *lcol, Use use) {
    const int tid = pass_tid(), g = tid / LPR, lane = tid % LPR;
#pragma unroll 1
    for (int base = 0; base < o.n; base += NT / LPR) {
      const int row = base + g;
      const bool has = row < o.n;
      float acc = 0.f;
      if (has) {
        const int32_t n = o.rp[row + 1] - o.rp[row];
        const S *q = DC + 4 * (int64_t)o.rp[row];
        const uint16_t *lc = lcol + o.rp[row];
#pragma unroll 1
        for (int32_t k = lane; k < n; k += U * LPR) {
          typename Rec4<S>::type b[U];
          uint32_t c[U];
#pragma unroll
          for (int u = 0; u < U; ++u) {
            const int32_t kk = min(k + u * LPR, n - 1);
            b[u].load(q + 4 * kk);
            c[u] = __ldg(lc + kk);
          }
#pragma unroll
          for (int u = 0; u < U; ++u) {
            const F4 v = ld4(o.sv, k + u * LPR < n ? c[u] : (uint32_t)o.loc);
            const F4 d = b[u].get();
            const float s = d.x * v.x + d.y * v.y + d.z * v.z;
            acc += kFull ? d.w * v.w - s : s;
          }
        }
      }
      acc = lanes_sum<LPR>(acc);
      if (has && lane == 0) use(row, acc);
    }
  }
  // o.w = A v: lane i of a row reads row i of each block (a block is one 64-byte segment of four lanes;
  // whole blocks per lane would use half of every sector per load)
  static __device__ __forceinline__ void product(const Own<float> &o, const float *A, const uint16_t *lcol) {
    constexpr int SUB = LPR / 4, U = 4;
    const int tid = pass_tid(), lane = tid % LPR, comp = lane & 3, sub = lane >> 2;
    const uint64_t policy = stream_policy();
#pragma unroll 1
    for (int base = 0; base < o.n; base += NT / LPR) {
      const int row = base + tid / LPR;
      const bool has = row < o.n;
      float acc = 0.f;
      if (has) {
        const int32_t k1 = o.rp[row + 1];
#pragma unroll 1
        for (int32_t k = o.rp[row] + sub; k < k1; k += U * SUB) {
          float4 a[U];
          uint16_t c[U];
#pragma unroll
          for (int u = 0; u < U; ++u)
            {
              const int32_t kk = min(k + u * SUB, k1 - 1);
              a[u] = ld_stream(reinterpret_cast<const float4 *>(A) + 4 * (int64_t)kk + comp, policy);
              c[u] = __ldg(lcol + kk);
            }
#pragma unroll
          for (int u = 0; u < U; ++u)
            {
              const F4 q = ld4(o.sv, k + u * SUB < k1 ? c[u] : o.loc);
              acc += a[u].x * q.x + a[u].y * q.y + a[u].z * q.z + a[u].w * q.w;
            }
        }
      }
#pragma unroll
      for (int s = 4; s < LPR; s <<= 1) acc += __shfl_xor_sync(0xffffffffu, acc, s);
      if (has && sub == 0) o.w[4 * row + comp] = acc;
    }
  }
};


template <int LPR>
struct Rows<double, LPR> {
  static constexpr int NT = Shape<double, LPR>::threads;
  static constexpr int SUB = LPR / 4;                    // lanes that share a component's blocks
  static constexpr int U = SUB == 1 ? 3 : 2;             // blocks in flight per lane
  // The lanes of a three-component product: ten rows of three lanes per warp, or LPR lanes per row
  // with every fourth idle when there are too few rows to fill the CTA.
  struct Three {
    int row, comp, sub, step;
    bool on;
    __device__ __forceinline__ Three() {
      const int t = pass_tid(), lane = t & 31;
      if (SUB == 1) {
        row = (t >> 5) * 10 + lane / 3;
        comp = lane % 3;
        sub = 0;
        step = NT / 32 * 10;
        on = lane < 30;
      } else {
        row = t / LPR;
        comp = lane & 3;
        sub = (lane % LPR) >> 2;
        step = NT / LPR;
        on = comp < 3;
      }
    }
  };
  static __device__ __forceinline__ double over_sub(double a) {
#pragma unroll
    for (int o = 4; o < LPR; o <<= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
    return a;
  }
  template <class S, class Rec, class Use>
  static __device__ __forceinline__ void velocity(const Own<double> &o, const uint16_t *lcol, Rec rec, Use use) {
    const Three l;
#pragma unroll 1
    for (int base = 0; base < o.n; base += l.step) {
      const int row = base + l.row;
      const bool has = l.on && row < o.n;
      double acc = 0.0;
      if (has) {
        const int32_t k0 = o.rp[row], k1 = o.rp[row + 1];
        const S *q = rec(row) + 3 * l.comp;
#pragma unroll 1
        for (int32_t k = k0 + l.sub; k < k1; k += U * SUB) {
          double f[U][3];
          uint16_t c[U];
#pragma unroll
          for (int u = 0; u < U; ++u)
            {
              const int32_t kk = min(k + u * SUB, k1 - 1);
              const S *p = q + 12 * (int64_t)(kk - k0);
              f[u][0] = __ldg(p);
              f[u][1] = __ldg(p + 1);
              f[u][2] = __ldg(p + 2);
              c[u] = __ldg(lcol + kk);
            }
#pragma unroll
          for (int u = 0; u < U; ++u)
            if (k + u * SUB < k1) {
              const double *v = o.sv + 4 * c[u];
              acc += f[u][0] * v[0] + f[u][1] * v[1] + f[u][2] * v[2];
            }
        }
      }
      acc = over_sub(acc);
      if (has && l.sub == 0) use(row, l.comp, acc);
    }
  }
  template <class S, class Use>
  static __device__ __forceinline__ void gradient(const Own<double> &o, const S *G, const uint16_t *lcol, Use use) {
    const Three l;
#pragma unroll 1
    for (int base = 0; base < o.n; base += l.step) {
      const int row = base + l.row;
      const bool has = l.on && row < o.n;
      double acc = 0.0;
      if (has) {
        const int32_t k1 = o.rp[row + 1];
#pragma unroll 1
        for (int32_t k = o.rp[row] + l.sub; k < k1; k += U * SUB) {
          double g[U];
          uint16_t c[U];
#pragma unroll
          for (int u = 0; u < U; ++u)
            {
              const int32_t kk = min(k + u * SUB, k1 - 1);
              g[u] = __ldg(G + 4 * (int64_t)kk + l.comp);
              c[u] = __ldg(lcol + kk);
            }
#pragma unroll
          for (int u = 0; u < U; ++u)
            if (k + u * SUB < k1) acc += g[u] * o.sv[c[u]];
        }
      }
      acc = over_sub(acc);
      if (has && l.sub == 0) use(row, l.comp, acc);
    }
  }
  template <bool kFull, class S, class Use>
  static __device__ __forceinline__ void divergence(const Own<double> &o, const S *DC, const uint16_t *lcol, Use use) {
    const int tid = pass_tid(), lane = tid % LPR, comp = lane & 3, sub = lane >> 2;
#pragma unroll 1
    for (int base = 0; base < o.n; base += NT / LPR) {
      const int row = base + tid / LPR;
      const bool has = row < o.n;
      double acc = 0.0;
      if (has && (kFull || comp < 3)) {
        const int32_t k1 = o.rp[row + 1];
#pragma unroll 1
        for (int32_t k = o.rp[row] + sub; k < k1; k += U * SUB) {
          double d[U];
          uint16_t c[U];
#pragma unroll
          for (int u = 0; u < U; ++u)
            {
              const int32_t kk = min(k + u * SUB, k1 - 1);
              d[u] = __ldg(DC + 4 * (int64_t)kk + comp);
              c[u] = __ldg(lcol + kk);
            }
#pragma unroll
          for (int u = 0; u < U; ++u)
            if (k + u * SUB < k1) acc += d[u] * o.sv[4 * c[u] + comp];
        }
      }
      if (kFull && comp < 3) acc = -acc;
#pragma unroll
      for (int s = 1; s < LPR; s <<= 1) acc += __shfl_xor_sync(0xffffffffu, acc, s);
      if (has && lane == 0) use(row, acc);
    }
  }
  static __device__ __forceinline__ void product(const Own<double> &o, const double *A, const uint16_t *lcol) {
    constexpr int W = 2;   // blocks in flight per lane
    const int tid = pass_tid(), lane = tid % LPR, comp = lane & 3, sub = lane >> 2;
#pragma unroll 1
    for (int base = 0; base < o.n; base += NT / LPR) {
      const int row = base + tid / LPR;
      const bool has = row < o.n;
      double acc = 0.0;
      if (has) {
        const int32_t k1 = o.rp[row + 1];
#pragma unroll 1
        for (int32_t k = o.rp[row] + sub; k < k1; k += W * SUB) {
          double2 a[W][2];
          uint16_t c[W];
#pragma unroll
          for (int u = 0; u < W; ++u)
            {
              const int32_t kk = min(k + u * SUB, k1 - 1);
              const double2 *p = reinterpret_cast<const double2 *>(A + 16 * (int64_t)kk + 4 * comp);
              a[u][0] = __ldg(p);
              a[u][1] = __ldg(p + 1);
              c[u] = __ldg(lcol + kk);
            }
#pragma unroll
          for (int u = 0; u < W; ++u)
            if (k + u * SUB < k1) {
              const double *v = o.sv + 4 * c[u];
              acc += a[u][0].x * v[0] + a[u][0].y * v[1] + a[u][1].x * v[2] + a[u][1].y * v[3];
            }
        }
      }
      acc = over_sub(acc);
      if (has && sub == 0) o.w[4 * row + comp] = acc;
    }
  }
};

// shared memory of the CTA's own data: the pass's vector, 16 values per row, halo, row pointers
// (spill 1: w, t, xp and 1 / diag(S) stay in global memory, seven values per row; spill 2: r, x and 1 / diag(F)
// too)
__host__ __device__ inline size_t own_bytes(size_t t, int rows, int loc, int spill) {
  const size_t n = (size_t)((rows + 3) & ~3), per = spill == 0 ? 16 : (spill == 1 ? 9 : 0);
  return ((size_t)(loc + 1) * (4 * t + 4) + n * (per * t + 4) + 4 + 127) & ~(size_t)127;
}

// grid barriers of one Arnoldi step
__host__ __device__ inline int step_barriers(int f_steps, int L, bool fp64) {
  return (f_steps - 1) + 1 + (L == 1 ? 1 : 7 + 4 * (L - 2)) + 1 + (fp64 ? 3 : 2);
}

// one thread of the CTA without rows: a wait ran out, which ends the solve and the one that it preconditions
// (the host reads the flag with the status of the cycle)
template <class S, class T>
__device__ __forceinline__ void gave_up(const CycleArgs<S, T> &A) {
  atomicExch(&A.sync->error, 1);
  A.ks->flag = kFlagTimeout;
  A.ks->done = 1;
  if (A.parent) {
    A.parent->flag = kFlagTimeout;
    A.parent->done = 1;
  }
}

// The CTA without rows: Hessenberg columns, rotations, stopping test, back substitution (FP64).
template <class S, class T, int LPR>
__device__ __forceinline__ void dense_algebra(const CycleArgs<S, T> &A, unsigned char *sm, unsigned rows_ctas) {
  using Sm = Sum<T>;
  constexpr int NW = Shape<T, LPR>::threads / 32;
  double *h = reinterpret_cast<double *>(sm), *cs = h + kMaxRestart + 2, *sn = cs + kMaxRestart, *y = sn + kMaxRestart,
         *g = y + kMaxRestart + 2, *R = g + kMaxRestart + 2;   // R [m][m + 1], columns of the rotated Hessenberg matrix
  __shared__ int go;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const typename Sm::type *part = static_cast<const typename Sm::type *>(A.part);
  const typename Sm::type *pn = static_cast<const typename Sm::type *>(A.part_n);
  const unsigned B = step_barriers(A.f_steps, A.L, sizeof(T) == 8);
  KState *ks = A.ks;
  const double tol = ks->tol_abs;
  int total = ks->total;
  if (threadIdx.x == 0) g[0] = ks->g[0];
  auto reached = [&](unsigned barriers) {
    __syncthreads();
    if (threadIdx.x == 0) go = wait_for(&A.sync->arrived, barriers * rows_ctas + A.unreachable, A.polls);
    __syncthreads();
    if (!go && threadIdx.x == 0) gave_up(A);
    return go != 0;
  };
  for (int j = 0;; ++j) {
    if (!reached(1 + j * B + B - (sizeof(T) == 8 ? 2 : 1))) return;
    for (int i = warp; i <= j; i += NW) {
      double s = 0.0;
      for (unsigned c = lane; c < rows_ctas; c += 32) s += Sm::value(part[(size_t)i * rows_ctas + c]);
      s = lanes_sum<32>(s);
      if (lane == 0) h[i] = s;
    }
    if (!reached(1 + (j + 1) * B)) return;
    int done = 0;
    if (warp == 0) {
      double s = 0.0;
      for (unsigned c = lane; c < rows_ctas; c += 32) s += Sm::value(pn[c]);
      s = lanes_sum<32>(s);
      if (lane == 0) {
        const double hn = sqrt(s);
        double a = h[0];
        double *col = R + (size_t)j * (kMaxRestart + 1);
        for (int i = 0; i < j; ++i) {
          const double b = h[i + 1];
          col[i] = cs[i] * a + sn[i] * b;
          a = -sn[i] * a + cs[i] * b;
        }
        const double den = hypot(a, hn);
        double c = 1.0, q = 0.0;
        if (den > 0.0) {
          c = a / den;
          q = hn / den;
        }
        cs[j] = c;
        sn[j] = q;
        col[j] = den;
        g[j + 1] = -q * g[j];
        g[j] = c * g[j];
        const double res = fabs(g[j + 1]);
        ++total;
        int flag = 0;
        if (!isfinite(res) || !isfinite(hn)) {
          flag = 2;
          done = 1;
        } else if (res <= tol || hn == 0.0) {
          flag = 1;
          done = 1;
        } else if (j + 1 >= A.m || total >= A.maxit) {
          done = 1;
        }
        ks->j = j + 1;
        ks->total = total;
        ks->res = res;
        ks->flag = flag;
        if (done) ks->done = 1;
        fence_gpu();
        atomicExch(&A.sync->progress, 2u * (unsigned)(j + 1) + (unsigned)done);
      }
      done = __shfl_sync(0xffffffffu, done, 0);
      if (done) {
        for (int i = j; i >= 0; --i) {
          double p = 0.0;
          for (int k = i + 1 + lane; k <= j; k += 32) p += R[(size_t)k * (kMaxRestart + 1) + i] * y[k];
          p = lanes_sum<32>(p);
          if (lane == 0) {
            const double d = R[(size_t)i * (kMaxRestart + 1) + i];
            y[i] = d != 0.0 ? (g[i] - p) / d : 0.0;   // d = 0 only after a breakdown (w = 0)
          }
          __syncwarp();
        }
        for (int i = lane; i <= j; i += 32) ks->y[i] = y[i];
        __syncwarp();
        if (lane == 0) {
          fence_gpu();
          atomicExch(&A.sync->solved, 1u);
        }
      }
    }
    if (__syncthreads_or(done)) return;
  }
}

// The same for several segments in lockstep, a warp per segment, with the Hessenberg matrix and rotations in
// the segments' status structs.  A segment that has converged keeps its count and solution; its rows meet the
// others at their barriers with basis vectors of zeros until every segment has.
template <class S, class T, int LPR>
__device__ __forceinline__ void dense_algebra_seg(const CycleArgs<S, T> &A, unsigned rows_ctas) {
  using Sm = Sum<T>;
  constexpr int NW = Shape<T, LPR>::threads / 32;
  __shared__ int go;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const typename Sm::type *part = static_cast<const typename Sm::type *>(A.part);
  const typename Sm::type *pn = static_cast<const typename Sm::type *>(A.part_n);
  const unsigned B = step_barriers(A.f_steps, A.L, sizeof(T) == 8);
  int total = A.ks->total;
  auto reached = [&](unsigned barriers) {
    __syncthreads();
    if (threadIdx.x == 0) go = wait_for(&A.sync->arrived, barriers * rows_ctas + A.unreachable, A.polls);
    __syncthreads();
    if (!go && threadIdx.x == 0) gave_up(A);
    return go != 0;
  };
  for (int j = 0;; ++j) {
    if (!reached(1 + j * B + B - (sizeof(T) == 8 ? 2 : 1))) return;
    for (int c = warp; c < A.n_seg; c += NW) {
      KState &k = A.kseg[c];
      if (k.done) continue;
      double *col = k.H + (size_t)j * (kMaxRestart + 1);
      for (int i = 0; i <= j; ++i) {
        double s = 0.0;
        for (int b = A.seg_off[c] + lane; b < A.seg_off[c + 1]; b += 32) s += Sm::value(part[(size_t)i * rows_ctas + b]);
        s = lanes_sum<32>(s);
        if (lane == 0) col[i] = s;
      }
    }
    if (!reached(1 + (j + 1) * B)) return;
    ++total;
    int running = 0, bad = 0;
    for (int c = warp; c < A.n_seg; c += NW) {
      KState &k = A.kseg[c];
      if (k.done) continue;
      double s = 0.0;
      for (int b = A.seg_off[c] + lane; b < A.seg_off[c + 1]; b += 32) s += Sm::value(pn[b]);
      s = lanes_sum<32>(s);
      if (lane == 0) {
        const double hn = sqrt(s);
        double *col = k.H + (size_t)j * (kMaxRestart + 1);
        double a = col[0];
        for (int i = 0; i < j; ++i) {
          const double b = col[i + 1];
          col[i] = k.cs[i] * a + k.sn[i] * b;
          a = -k.sn[i] * a + k.cs[i] * b;
        }
        const double den = hypot(a, hn);
        double cc = 1.0, q = 0.0;
        if (den > 0.0) {
          cc = a / den;
          q = hn / den;
        }
        k.cs[j] = cc;
        k.sn[j] = q;
        col[j] = den;
        k.g[j + 1] = -q * k.g[j];
        k.g[j] = cc * k.g[j];
        const double res = fabs(k.g[j + 1]);
        k.j = j + 1;
        k.total += 1;
        k.res = res;
        if (!isfinite(res) || !isfinite(hn)) {
          k.flag = 2;
          k.done = 1;
          bad = 1;
        } else if (res <= k.tol_abs || hn == 0.0) {
          k.flag = 1;
          k.done = 1;
        }
        if (!k.done) running = 1;
      }
      __syncwarp();
    }
    bad = __syncthreads_or(bad);
    running = __syncthreads_or(running);
    const int done = !running || bad || j + 1 >= A.m || total >= A.maxit;
    if (threadIdx.x == 0) {
      A.ks->j = j + 1;
      A.ks->total = total;
      A.ks->flag = bad ? 2 : (running ? 0 : 1);
      if (done) A.ks->done = 1;
      fence_gpu();
      atomicExch(&A.sync->progress, 2u * (unsigned)(j + 1) + (unsigned)done);
    }
    if (!done) continue;
    for (int c = warp; c < A.n_seg; c += NW) {
      KState &k = A.kseg[c];
      for (int i = k.j - 1; i >= 0; --i) {
        double p = 0.0;
        for (int q = i + 1 + lane; q < k.j; q += 32) p += k.H[(size_t)q * (kMaxRestart + 1) + i] * k.y[q];
        p = lanes_sum<32>(p);
        if (lane == 0) {
          const double d = k.H[(size_t)i * (kMaxRestart + 1) + i];
          k.y[i] = d != 0.0 ? (k.g[i] - p) / d : 0.0;   // d = 0 only after a breakdown (w = 0)
        }
        __syncwarp();
      }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      fence_gpu();
      atomicExch(&A.sync->solved, 1u);
    }
    return;
  }
}

// kFar: r, x and 1 / diag(F) in global memory (spill 2)
template <class S, class T, int LPR, bool kFar = false>
__global__ void __launch_bounds__(Shape<T, LPR>::threads, 1) cycle_kernel(const __grid_constant__ CycleArgs<S, T> A) {
  using Sm = Sum<T>;
  using SumT = typename Sm::type;
  using V4 = typename Vec4T<T>::type;
  using R = Rows<T, LPR>;
  constexpr int NT = Shape<T, LPR>::threads, NW = NT / 32;
  constexpr bool fp64 = sizeof(T) == 8;
  constexpr int st = kFar ? 4 : 3;   // values per row of r, x, df
  extern __shared__ __align__(16) unsigned char sm[];
  __shared__ T hs[kMaxRestart + 1];
  __shared__ SumT red[(kMaxRestart + 1) * kDots];
  __shared__ unsigned long long t0, ns_f;   // thread 0's clock and sum (in registers they would be every thread's)
  __shared__ int verdict, resident, solved, over;   // over: this CTA's segment has converged (thread 0's)
  if (finished(A.ks)) return;
  const unsigned rows_ctas = gridDim.x - 1, cta = blockIdx.x;
  if (*(volatile const int *)&A.sync->error) {   // a wait of an earlier cycle gave up
    if (cta == rows_ctas && threadIdx.x == 0) gave_up(A);
    return;
  }
  if (cta == rows_ctas) {
    if (A.n_seg > 1) dense_algebra_seg<S, T, LPR>(A, rows_ctas);
    else dense_algebra<S, T, LPR>(A, sm, rows_ctas);
    return;
  }
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  Own<T> o;
  o.r0 = A.row_off[cta];
  o.n = A.row_off[cta + 1] - o.r0;
  // the CTAs of this one's segment: their rows are one system with its own basis, sums and scale (looked up
  // where it is needed rather than held in registers)
  const int seg = A.cta_seg[cta];
  const unsigned cta0 = A.seg_off[seg], cta1 = A.seg_off[seg + 1];
  {
    const int n = (A.max_rows + 3) & ~3;   // (four-value records stay aligned)
    const int64_t r = o.r0;
    T *at = reinterpret_cast<T *>(sm);
    o.sv = at;
    at += 4 * (size_t)(A.max_loc + 1);
    if (!kFar) {
      o.r = at;
      o.x = at + 3 * n;
      o.df = at + 6 * n;
      at += 9 * n;
    } else {   // W4 is free during the velocity passes; X ends up holding the iterate anyway
      o.r = A.W4 + 4 * r;
      o.x = A.X + 4 * r;
      o.df = A.dinvF + 4 * r;
    }
    if (A.spill < 1) {
      o.w = at;
      o.t = at + 4 * n;
      o.xp = o.t + n;
      o.ds = o.xp + n;
      at += 7 * n;
    } else {
      o.w = A.wk + 4 * r;
      o.t = A.t + r;
      o.xp = A.xp + r;
      o.ds = A.dinvS + r;
    }
    o.rp = reinterpret_cast<int32_t *>(at);
    o.loc = o.n + A.halo_off[cta + 1] - A.halo_off[cta];
    int32_t *h = o.rp + n + 1;
    o.halo = h;
    for (int i = threadIdx.x; i < o.loc - o.n; i += NT) h[i] = A.halo[A.halo_off[cta] + i];
  }
  o.vb = reinterpret_cast<T *>(sm + own_bytes(sizeof(T), A.max_rows, A.max_loc, A.spill));
  S *own_f = reinterpret_cast<S *>(reinterpret_cast<unsigned char *>(o.vb) + A.vb_bytes);
  const int vstride = 4 * A.max_rows, nb = (int)(A.vb_bytes / (vstride * sizeof(T)));
  const int64_t r0 = o.r0;
  // ---- the CTA's own data
  for (int i = tid; i <= o.n; i += NT) o.rp[i] = A.rowptr[r0 + i];
  for (int i = tid; i < o.n; i += NT) {
    const V4 d = ld4(A.dinvF, r0 + i), v = ld4(A.Vb, r0 + i);
    if (!kFar) {
      T *df = const_cast<T *>(o.df);
      df[3 * i] = d.x;
      df[3 * i + 1] = d.y;
      df[3 * i + 2] = d.z;
    }
    if (A.spill < 1) const_cast<T *>(o.ds)[i] = A.dinvS[r0 + i];
    st4(o.w, i, v);
    if (nb > 0) st4(o.vb, i, v);
    V4 q;
    q.x = d.x * v.x;
    q.y = d.y * v.y;
    q.z = d.z * v.z;
    q.w = T(0);
    st4(A.Q, r0 + i, q);
  }
  __syncthreads();
  if (tid == 0) {   // rows whose velocity records fit
    over = 0;
    ns_f = 0;
    const int64_t most = A.f_bytes / (12 * sizeof(S));
    int lo = 0, hi = o.n;
    while (lo < hi) {
      const int mid = (lo + hi + 1) / 2;
      if (o.rp[mid] - o.rp[0] <= most) lo = mid;
      else hi = mid - 1;
    }
    resident = lo;
  }
  __syncthreads();
  const int64_t words = (int64_t)(o.rp[resident] - o.rp[0]) * (12 * sizeof(S) / 8);
  const uint2 *src = reinterpret_cast<const uint2 *>(A.F + 12 * (int64_t)o.rp[0]);
  for (int64_t i = tid; i < words; i += NT) reinterpret_cast<uint2 *>(own_f)[i] = src[i];
  // the pass's vector into shared memory: own rows, then the halo
  auto load4 = [&](const T *v) {
#pragma unroll 2
    for (int i = pass_tid(); i < o.loc; i += NT) st4(o.sv, i, ld4(v, i < o.n ? r0 + i : (int64_t)o.halo[i - o.n]));
    if (tid < 4) o.sv[4 * o.loc + tid] = T(0);
    __syncthreads();
  };
  auto load1 = [&](const T *v) {
#pragma unroll 2
    for (int i = pass_tid(); i < o.loc; i += NT) o.sv[i] = v[i < o.n ? r0 + i : (int64_t)o.halo[i - o.n]];
    if (tid == 0) o.sv[o.loc] = T(0);
    __syncthreads();
  };
  unsigned target = A.unreachable;   // (0 but in tests)
  // grid barrier; with decide >= 0 also the verdict on that step: 0 go on, 1 a wait gave up, 2 the cycle has ended
  auto barrier = [&](int decide) -> int {
    __syncthreads();
    target += rows_ctas;
    if (tid == 0) {
      arrive(&A.sync->arrived);
      int v = wait_for(&A.sync->arrived, target, A.polls) ? 0 : 1;
      if (v == 0 && decide > 0) {
        if (!wait_for(&A.sync->progress, 2u * (unsigned)decide, A.polls)) v = 1;
        else if (ld_relaxed(&A.sync->progress) & 1u) v = 2;
        // (not written again before this CTA has arrived at the end of the step)
        if (v == 0 && A.n_seg > 1) over = *(volatile const int *)&A.kseg[A.cta_seg[cta]].done;
      }
      if (v == 1) atomicExch(&A.sync->error, 1);
      verdict = v;
    }
    __syncthreads();
    return verdict;
  };
#define LFX_CYCLE_SYNC()  \
  do {                    \
    if (barrier(0)) return; \
  } while (0)
  LFX_CYCLE_SYNC();
  const int64_t n4 = 4 * A.V;
  auto basis = [&](int i) -> T * { return i < nb ? o.vb + (size_t)i * vstride : A.Vb + (int64_t)i * n4 + 4 * r0; };
  auto rec = [&](int row) -> const S * {
    if constexpr (fp64) return A.F + 12 * (int64_t)o.rp[row];
    return row < resident ? own_f + 12 * (int64_t)(o.rp[row] - o.rp[0]) : A.F + 12 * (int64_t)o.rp[row];
  };
  const T s0 = coef_t<T>(A.cf->f_init, A.cf->f_initf), ss0 = coef_t<T>(A.cf->s_init, A.cf->s_initf);
  T *const dbuf[2] = {A.D0, A.D1};
  const int decide_at = min(3, A.f_steps - 1);
  T s = T(1);                        // 1 / norm of the Krylov vector held in w
  int j = 0;
  for (;; ++j) {
    // ---- z_u* ~= F^-1 v_u: Chebyshev steps; the first one reads diag(F)^-1 w
    for (int k = 1; k < A.f_steps; ++k) {
      const bool first = k == 1, last = k == A.f_steps - 1;
      const T c1 = coef_t<T>(A.cf->f_c1[k], A.cf->f_c1f[k]), c2 = coef_t<T>(A.cf->f_c2[k], A.cf->f_c2f[k]);
      const T *src = first ? A.Q : dbuf[(k - 1) & 1];
      T *dst = last ? A.X : dbuf[k & 1];
      T *vj = first && j > 0 ? basis(j) : nullptr;
      const T sa = s * s0;
      // one component: residual, step and iterate of the row
      auto update = [&](int row, int i, T a) -> T {
        const int e = st * row + i;
        T rv, d0, xv;
        if (first) {
          rv = s * (o.df[e] * o.w[4 * row + i]);
          d0 = s0 * rv;
          a = sa * a;
          xv = d0;
        } else {
          rv = o.r[e];
          d0 = o.sv[4 * row + i];
          xv = o.x[e];
        }
        rv -= o.df[e] * a;
        const T dn = c1 * d0 + c2 * rv;
        xv += dn;
        o.r[e] = rv;
        o.x[e] = xv;
        return last ? xv : dn;
      };
      load4(src);
      auto use = [&](int row, int i, T a) {
        dst[4 * (r0 + row) + i] = update(row, i, a);
        if (vj) {
          vj[4 * row + i] = s * o.w[4 * row + i];
          if (i == 0) vj[4 * row + 3] = s * o.w[4 * row + 3];
        }
      };
      R::template velocity<S>(o, A.lcol, rec, use);
      const int v = barrier(k == decide_at ? j : 0);
      if (v == 1) return;
      if (v == 2) goto ended;
      if (cta == 0 && tid == 0) {
        const unsigned long long t = now_ns();
        if (!first) ns_f += t - t0;
        t0 = t;
      }
    }
    // ---- z_p ~= S^-1 (v_p - D z_u*)
    load4(A.X);
    auto start = [&](int row, T a) {
      const T t = s * o.w[4 * row + 3] - a;
      o.t[row] = t;
      if (A.L == 1) {
        A.rr[r0 + row] = t;
      } else {
        const T x = ss0 * (o.ds[row] * t);
        o.xp[row] = x;
        A.xp[r0 + row] = x;
      }
    };
    R::template divergence<false>(o, A.DC, A.lcol, start);
    LFX_CYCLE_SYNC();
    const int64_t gwarp = (int64_t)cta * NW + warp, nwarps = (int64_t)rows_ctas * NW;
    if (A.L == 1) {
      for (int64_t row = gwarp; row < A.V; row += nwarps) {
        const T a = dense_row_dot(A.V, A.coarse_inv, A.rr, 1, 0, row, lane, true);
        if (lane == 0) A.pf[row] = a;
      }
      LFX_CYCLE_SYNC();
    } else {
      // diag(F)^-1 G x_p with x_p beside it, then the Schur residual of x_p
      auto scaled_gradient = [&]() {
        load1(A.xp);
        auto use = [&](int row, int i, T a) {
          A.W4[4 * (r0 + row) + i] = o.df[st * row + i] * a;
          if (i == 0) A.W4[4 * (r0 + row) + 3] = o.xp[row];
        };
        R::gradient(o, A.G, A.lcol, use);
      };
      scaled_gradient();
      LFX_CYCLE_SYNC();
      load4(A.W4);
      auto residual = [&](int row, T a) { A.rr[r0 + row] = o.t[row] - a; };
      R::template divergence<true>(o, A.DC, A.lcol, residual);
      LFX_CYCLE_SYNC();
      for (int64_t row = gwarp; row < A.R0.n; row += nwarps) {
        const T a = csr_row_dot<32>(A.R0.rp, A.R0.ci, A.R0.v, A.rr, 1, 0, row, lane, true);
        if (lane == 0) A.b1[row] = a;
      }
      LFX_CYCLE_SYNC();
      // levels 1 .. L-1, a warp per row
      const CoarseArgs<T> &C = *A.coarse;
      for (int l = 1; l < A.L - 1; ++l) {
        const CoarseLevel<T> &D = C.lv[l];
        // x = init dinv b and rr = b - A x in one pass (x of a neighbour is formed from its b)
        for (int64_t row = gwarp; row < D.n; row += nwarps) {
          T a = T(0);
          const int32_t k1 = __ldg(D.rp + row + 1);
          for (int32_t k = __ldg(D.rp + row) + lane; k < k1; k += 32) {
            const int32_t c = __ldg(D.ci + k);
            a += __ldg(D.v + k) * (__ldg(D.dinv + c) * D.b[c]);
          }
          a = lanes_sum<32>(a);
          if (lane == 0) {
            const T b = D.b[row];
            D.x[row] = D.init * D.dinv[row] * b;
            D.rr[row] = b - D.init * a;
          }
        }
        LFX_CYCLE_SYNC();
        for (int64_t row = gwarp; row < D.nnext; row += nwarps) {
          const T a = csr_row_dot<32>(D.Rrp, D.Rci, D.Rv, D.rr, 1, 0, row, lane, true);
          if (lane == 0) C.lv[l + 1].b[row] = a;
        }
        LFX_CYCLE_SYNC();
      }
      for (int64_t row = gwarp; row < C.nc; row += nwarps) {
        const T a = dense_row_dot(C.nc, C.coarse_inv, C.lv[A.L - 1].b, 1, 0, row, lane, true);
        if (lane == 0) C.lv[A.L - 1].x[row] = a;
      }
      LFX_CYCLE_SYNC();
      for (int l = A.L - 2; l >= 1; --l) {
        const CoarseLevel<T> &D = C.lv[l];
        const T *xc = l + 1 == A.L - 1 ? C.lv[l + 1].x : C.lv[l + 1].xo;
        for (int64_t row = gwarp; row < D.n; row += nwarps) {
          const T a = csr_row_dot<32>(D.Prp, D.Pci, D.Pv, xc, 1, 0, row, lane, true);
          if (lane == 0) D.x[row] = D.x[row] + C.alpha * a;
        }
        LFX_CYCLE_SYNC();
        for (int64_t row = gwarp; row < D.n; row += nwarps) {
          const T a = csr_row_dot<32>(D.rp, D.ci, D.v, D.x, 1, 0, row, lane, true);
          if (lane == 0) D.xo[row] = D.x[row] + D.init * D.dinv[row] * (D.b[row] - a);
        }
        LFX_CYCLE_SYNC();
      }
      // correction, post-smoothing
#pragma unroll 1
      for (int base = 0; base < o.n; base += NT / LPR) {
        const int row = base + tid / LPR;
        const T a = csr_row_dot<LPR>(A.P0.rp + r0, A.P0.ci, A.P0.v, A.x1, 1, 0, row, tid % LPR, row < o.n);
        if (row < o.n && tid % LPR == 0) {
          const T x = o.xp[row] + A.alpha * a;
          o.xp[row] = x;
          A.xp[r0 + row] = x;
        }
      }
      LFX_CYCLE_SYNC();
      scaled_gradient();
      LFX_CYCLE_SYNC();
      load4(A.W4);
      auto smooth = [&](int row, T a) {
        const T x = o.xp[row] + ss0 * (o.ds[row] * (o.t[row] - a));
        o.xp[row] = x;
        A.pf[r0 + row] = x;
      };
      R::template divergence<true>(o, A.DC, A.lcol, smooth);
      LFX_CYCLE_SYNC();
    }
    // ---- z_u = z_u* - diag(F)^-1 G z_p
    T *zj = A.Zb + (int64_t)j * n4;
    load1(A.pf);
    {
      auto use = [&](int row, int i, T a) {
        zj[4 * (r0 + row) + i] = o.x[st * row + i] - o.df[st * row + i] * a;
        if (i == 0) zj[4 * (r0 + row) + 3] = o.sv[row];
      };
      R::gradient(o, A.G, A.lcol, use);
    }
    LFX_CYCLE_SYNC();
    // ---- w = A z, then its products with the basis (own rows only: no barrier between)
    if (tid == 0) t0 = now_ns();
    load4(zj);
    R::product(o, A.A, A.lcol);
    __syncthreads();
    if (tid == 0) atomicMax(&A.sync->product_ns[j], (unsigned)(now_ns() - t0));
    const int nv = j + 1;
    {
      const int shares = max(1, min(kDots, NW / nv));
      for (int task = warp; task < nv * shares; task += NW) {
        const int i = task % nv, sh = task / nv;
        const V4 *b = reinterpret_cast<const V4 *>(basis(i));
        SumT a = Sm::zero();
        const int e1 = o.n * (sh + 1) / shares;
#pragma unroll (LPR == 4 ? 4 : 2)
        for (int e = o.n * sh / shares + lane; e < e1; e += 32) {
          const V4 bv = b[e], wv = ld4(o.w, e);
          Sm::add(a, bv.x * wv.x + bv.y * wv.y + bv.z * wv.z + bv.w * wv.w);
        }
#pragma unroll
        for (int q = 16; q > 0; q >>= 1) Sm::join(a, Sm::shfl(a, q));
        if (lane == 0) red[i * kDots + sh] = a;
      }
      __syncthreads();
      for (int i = tid; i < nv; i += NT) {
        SumT a = red[i * kDots];
        for (int q = 1; q < shares; ++q) Sm::join(a, red[i * kDots + q]);
        static_cast<SumT *>(A.part)[(size_t)i * rows_ctas + cta] = a;
      }
    }
    LFX_CYCLE_SYNC();
    {
      const SumT *part = static_cast<const SumT *>(A.part);
      auto total = [&](int i) {
        SumT a = Sm::zero();
        for (unsigned c = cta0 + lane; c < cta1; c += 32) Sm::join(a, part[(size_t)i * rows_ctas + c]);
#pragma unroll
        for (int q = 16; q > 0; q >>= 1) Sm::join(a, Sm::shfl(a, q));
        return a;
      };
      if constexpr (fp64) {
        // FP64 sums are dear: each vector's by one warp of the grid
        T *fin = static_cast<T *>(A.part) + (size_t)(kMaxRestart + 1) * (rows_ctas + seg);
        for (int i = warp * (int)(cta1 - cta0) + (int)(cta - cta0); i < nv; i += NW * (int)(cta1 - cta0)) {
          const T a = total(i);
          if (lane == 0) fin[i] = a;
        }
        LFX_CYCLE_SYNC();
        for (int q = tid; q < nv; q += NT) hs[q] = fin[q];
      } else {
        for (int i = warp; i < nv; i += NW) {
          const SumT a = total(i);
          if (lane == 0) hs[i] = Sm::rounded(a);
        }
      }
      __syncthreads();
    }
    // ---- w -= sum_i h_i v_i, |w|^2, and diag(F)^-1 w for the next first pass
    SumT nrm = Sm::zero();
    for (int e = tid; e < o.n; e += NT) {
      V4 a = ld4(o.w, e);
#pragma unroll 4
      for (int i = 0; i < nv; ++i) {
        const V4 b = ld4(basis(i), e);
        const T h = hs[i];
        a.x -= h * b.x;
        a.y -= h * b.y;
        a.z -= h * b.z;
        a.w -= h * b.w;
      }
      st4(o.w, e, a);
      st4(A.Q, r0 + e, V4{o.df[st * e] * a.x, o.df[st * e + 1] * a.y, o.df[st * e + 2] * a.z, T(0)});
      Sm::add(nrm, a.x * a.x + a.y * a.y + a.z * a.z + a.w * a.w);
    }
#pragma unroll
    for (int q = 16; q > 0; q >>= 1) Sm::join(nrm, Sm::shfl(nrm, q));
    if (lane == 0) red[warp] = nrm;
    __syncthreads();
    if (warp == 0) {
      SumT a = lane < NW ? red[lane] : Sm::zero();
#pragma unroll
      for (int q = 16; q > 0; q >>= 1) Sm::join(a, Sm::shfl(a, q));
      if (lane == 0) static_cast<SumT *>(A.part_n)[cta] = a;
    }
    LFX_CYCLE_SYNC();
    if (warp == 0) {
      SumT a = Sm::zero();
      for (unsigned c = cta0 + lane; c < cta1; c += 32) Sm::join(a, static_cast<const SumT *>(A.part_n)[c]);
#pragma unroll
      for (int q = 16; q > 0; q >>= 1) Sm::join(a, Sm::shfl(a, q));
      if (lane == 0) hs[0] = over ? T(0) : Sm::inv_sqrt(a);
    }
    __syncthreads();
    s = hs[0];
  }
ended:
  // ---- x += sum_i y_i z_i over the steps taken (j of them)
  // (a word of its own: other warps may still be reading the verdict that sent them here)
  if (tid == 0) {
    solved = wait_for(&A.sync->solved, 1u, A.polls);
    if (!solved) atomicExch(&A.sync->error, 1);
  }
  __syncthreads();
  if (!solved) return;
  if (cta == 0 && tid == 0) {
    unsigned long long ns_p = 0;
    for (int i = 0; i < j; ++i) ns_p += A.sync->product_ns[i];
    A.sync->t_f += ns_f;
    A.sync->n_f += (A.f_steps - 2) * j + max(decide_at - 2, 0);   // (with those of the step the verdict interrupted)
    A.sync->t_spmv += ns_p;
    A.sync->n_spmv += j;
  }
  const KState *own = A.n_seg > 1 ? A.kseg + A.cta_seg[cta] : A.ks;
  if (A.n_seg > 1) j = own->j;   // (steps until this segment had converged)
  for (int i = tid; i < j; i += NT) hs[i] = (T)own->y[i];
  __syncthreads();
  for (int e = tid; e < o.n; e += NT) {
    V4 a = ld4(A.x, r0 + e);
#pragma unroll 4
    for (int i = 0; i < j; ++i) {
      const V4 z = ld4(A.Zb + (int64_t)i * n4, r0 + e);
      const T y = hs[i];
      a.x += y * z.x;
      a.y += y * z.y;
      a.z += y * z.z;
      a.w += y * z.w;
    }
    st4(A.x, r0 + e, a);
  }
#undef LFX_CYCLE_SYNC
}

constexpr size_t kDenseSmem = sizeof(double) * (4 * (kMaxRestart + 2) + (size_t)kMaxRestart * (kMaxRestart + 1) + 64);

template <class T>
constexpr int threads_of(int lanes) {
  return lanes > 8 ? Shape<T, 16>::threads : (lanes > 4 ? Shape<T, 8>::threads : Shape<T, 4>::threads);
}
template <class S, class T>
using CycleKernel = void (*)(const CycleArgs<S, T>);
template <class S, class T>
CycleKernel<S, T> kernel_of(int lanes, bool far) {
  if (far) return cycle_kernel<S, T, 4, true>;
  if constexpr (sizeof(T) == 8) return lanes > 4 ? cycle_kernel<S, T, 16> : cycle_kernel<S, T, 4>;
  else return lanes > 8 ? cycle_kernel<S, T, 16> : (lanes > 4 ? cycle_kernel<S, T, 8> : cycle_kernel<S, T, 4>);
}

}  // namespace

size_t cycle_part_norm_offset(const CyclePlan &p) {
  return (size_t)(kMaxRestart + 1) * (p.rows_ctas + p.map->n_seg) + 2;
}
size_t cycle_part_bytes(const CyclePlan &p) {
  // [vector][CTA], the FP64 totals [segment][vector], [CTA] of the norm
  return sizeof(double) * (cycle_part_norm_offset(p) + (size_t)p.rows_ctas);
}

template <class T>
lfx_status cycle_ctas(int64_t V, int *ctas) {
  *ctas = 0;
  int dev = 0, sms = 0, coop = 0;
  LFX_CUDA_TRY(cudaGetDevice(&dev));
  LFX_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  LFX_CUDA_TRY(cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev));
  // small systems: 32 rows per CTA in FP32 (fewer CTAs meet sooner), 8 in FP64 (the FP64 pipes of more SMs)
  const int min_rows = sizeof(T) == 8 ? 8 : 32;
  if (coop && sms >= 2 && V >= 1) *ctas = (int)std::max<int64_t>(1, std::min<int64_t>(sms - 1, V / min_rows));
  return LFX_OK;
}

template <class S, class T>
lfx_status plan_cycle(int64_t V, int64_t nnzb, const CycleMap &map, CyclePlan *p) {
  *p = CyclePlan{};
  LFX_CUDA_TRY(cudaGetDevice(&p->device));
  if (map.ctas < 1 || map.max_loc > 65535) return LFX_OK;
  const int rows = map.max_rows;
  // as many lanes per row as the rows of a CTA leave free
  p->lanes = 4;
  if (rows * 16 <= threads_of<T>(16)) p->lanes = 16;
  else if (sizeof(T) == 4 && rows * 8 <= threads_of<T>(8)) p->lanes = 8;
  // Large systems leave some or all of a row's sixteen values in global memory: 4.0M tetrahedra, 2: 95.3 ms a
  // step against 111.6 step by step.  (Where they fit, shared memory serves them better: 1.02M, 0: 18.0 ms, 1: 18.5.)
  for (p->spill = 0; p->spill <= 2; ++p->spill)
    if (own_bytes(sizeof(T), rows, map.max_loc, p->spill) <= (size_t)kSmemCap) break;
  if (p->spill > 2) return LFX_OK;
  const size_t own = own_bytes(sizeof(T), rows, map.max_loc, p->spill);
  // velocity records (FP32): this CTA's share with some slack, as far as they fit; then basis vectors.  Only
  // up to kExtraCap in all: what shared memory leaves is L1, which holds the lines of the records and of the
  // operator between a row's loads.
  const size_t room = own < (size_t)kExtraCap ? kExtraCap - own : 0;
  const size_t want = sizeof(T) == 4 ? (size_t)(((double)nnzb / (double)V) * 1.15 * (double)rows + 64) * 12 * sizeof(S) : 0;
  p->f_bytes = std::min<size_t>(want, room) & ~(size_t)15;
  const size_t vec = 4 * sizeof(T) * (size_t)rows;
  p->vb_bytes = vec * std::min<size_t>(kMaxRestart + 1, (room - p->f_bytes) / vec);
  p->map = &map;
  p->smem = std::max(own + p->vb_bytes + p->f_bytes, kDenseSmem);
  CycleKernel<S, T> k = kernel_of<S, T>(p->lanes, p->spill == 2);
  int per = 0;
  LFX_CUDA_TRY(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemCap));
  LFX_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k, threads_of<T>(p->lanes), p->smem));
  if (per < 1) return LFX_OK;
  p->rows_ctas = map.ctas;
  return LFX_OK;
}

template <class S, class T>
lfx_status launch_cycle(cudaStream_t st, const CyclePlan &p, const CycleArgs<S, T> &args) {
  CycleArgs<S, T> a = args;
  a.max_rows = p.map->max_rows;
  a.max_loc = p.map->max_loc;
  a.row_off = p.map->row_off.as<int32_t>();
  a.cta_seg = p.map->cta_seg.as<int32_t>();
  a.seg_off = p.map->seg_off.as<int32_t>();
  a.n_seg = p.map->n_seg;
  a.halo_off = p.map->halo_off.as<int32_t>();
  a.halo = p.map->halo.as<int32_t>();
  a.lcol = p.map->lcol.as<uint16_t>();
  a.f_bytes = (uint32_t)p.f_bytes;
  a.vb_bytes = (uint32_t)p.vb_bytes;
  a.spill = p.spill;
  if (a.polls == 0) a.polls = kWaitPolls;
  LFX_CUDA_TRY(cudaMemsetAsync(a.sync, 0, offsetof(CycleSync, error), st));
  void *kargs[] = {&a};
  LFX_CUDA_TRY(cudaLaunchCooperativeKernel((const void *)kernel_of<S, T>(p.lanes, p.spill == 2), dim3(p.rows_ctas + 1),
                                           dim3(threads_of<T>(p.lanes)), kargs, p.smem, st));
  note_launches(1);
  return LFX_OK;
}

template lfx_status cycle_ctas<double>(int64_t, int *);
template lfx_status cycle_ctas<float>(int64_t, int *);
template lfx_status plan_cycle<double, double>(int64_t, int64_t, const CycleMap &, CyclePlan *);
template lfx_status plan_cycle<float, float>(int64_t, int64_t, const CycleMap &, CyclePlan *);
template lfx_status plan_cycle<__nv_bfloat16, float>(int64_t, int64_t, const CycleMap &, CyclePlan *);
template lfx_status launch_cycle<double, double>(cudaStream_t, const CyclePlan &, const CycleArgs<double, double> &);
template lfx_status launch_cycle<float, float>(cudaStream_t, const CyclePlan &, const CycleArgs<float, float> &);
template lfx_status launch_cycle<__nv_bfloat16, float>(cudaStream_t, const CyclePlan &,
                                                       const CycleArgs<__nv_bfloat16, float> &);

}  // namespace lfx
