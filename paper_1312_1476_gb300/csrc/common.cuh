// common.cuh -- device helpers shared by the Lanczos kernels.
//
// * compensated FP32 ("double-float") sums for the dot products of the
//   Lanczos recurrence: GB300's FP64 rate is a small fraction of its FP32
//   rate, so every per-element and per-warp reduction of the FP32 path runs
//   on pairs of floats and only the final per-vector sums are FP64;
// * the per-vector iteration state and the end-of-step logic shared by the
//   stencil and the preconditioned step kernels: alpha_j, beta_j
//   (Algorithm 1), the LDL^T recurrence of T_m, and the stopping rule built
//   on the a-posteriori bound of Theorem 1 (eq. krylov_bound);
// * Philox-4x32-10 (Salmon et al., SC'11) for z and the Rademacher probes.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/gmrf.h"

namespace gmrf {

// ----------------------------------------------------------------- status codes
enum : int { VS_RUNNING = 1, VS_DONE = 0 };  // other values: negative gmrf error codes

// --------------------------------------------------------- compensated float sums
struct df {
  float hi, lo;
};

__device__ __forceinline__ df two_sum(float a, float b) {
  float s = __fadd_rn(a, b);
  float bb = __fsub_rn(s, a);
  float e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
  return {s, e};
}
__device__ __forceinline__ df fast_two_sum(float a, float b) {  // |a| >= |b|
  float s = __fadd_rn(a, b);
  float e = __fsub_rn(b, __fsub_rn(s, a));
  return {s, e};
}
__device__ __forceinline__ df df_add(df a, df b) {
  df s = two_sum(a.hi, b.hi);
  float e = __fadd_rn(s.lo, __fadd_rn(a.lo, b.lo));
  return fast_two_sum(s.hi, e);
}
// exact product a*b as an unevaluated pair
__device__ __forceinline__ df two_prod(float a, float b) {
  float p = __fmul_rn(a, b);
  float e = __fmaf_rn(a, b, -p);
  return {p, e};
}
__device__ __forceinline__ df df_shfl_down(df v, int off) {
  return {__shfl_down_sync(0xffffffffu, v.hi, off), __shfl_down_sync(0xffffffffu, v.lo, off)};
}
__device__ __forceinline__ double df_to_double(df v) { return (double)v.hi + (double)v.lo; }

__device__ __forceinline__ df sum_add(df a, df b) { return df_add(a, b); }
__device__ __forceinline__ double sum_add(double a, double b) { return a + b; }
__device__ __forceinline__ df sum_xor(df v, int m) {
  return {__shfl_xor_sync(0xffffffffu, v.hi, m), __shfl_xor_sync(0xffffffffu, v.lo, m)};
}
__device__ __forceinline__ double sum_xor(double v, int m) { return __shfl_xor_sync(0xffffffffu, v, m); }
__device__ __forceinline__ df sum_from(df v, int lane) {
  return {__shfl_sync(0xffffffffu, v.hi, lane), __shfl_sync(0xffffffffu, v.lo, lane)};
}
__device__ __forceinline__ double sum_from(double v, int lane) { return __shfl_sync(0xffffffffu, v, lane); }

// Accumulator of the three dot products of one Lanczos step:
//   s1 = v_j . q, s2 = q . q, s3 = v_j . v_j  (all for one vector).
template <typename T>
struct Dots;

template <>
struct Dots<float> {
  typedef df S;
  df s1, s2, s3;
  __device__ __forceinline__ void zero() { s1 = s2 = s3 = {0.f, 0.f}; }
  __device__ __forceinline__ void add(float v, float q) {
    s1 = df_add(s1, two_prod(v, q));
    s2 = df_add(s2, two_prod(q, q));
    s3 = df_add(s3, two_prod(v, v));
  }
  // Dot2 of Ogita, Rump and Oishi (SIAM J. Sci. Comput. 2005): exact product
  // (TwoProd), TwoSum into hi, the rounding errors summed into lo without
  // renormalising; as accurate as summing in twice the working precision.
  __device__ __forceinline__ static void dot2(df& a, float x, float y) {
    const float p = __fmul_rn(x, y);
    const float pe = __fmaf_rn(x, y, -p);
    const df t = two_sum(a.hi, p);
    a.hi = t.hi;
    a.lo = __fadd_rn(a.lo, __fadd_rn(t.lo, pe));
  }
  __device__ __forceinline__ void add_dot2(float v, float q) {
    dot2(s1, v, q);
    dot2(s2, q, q);
    dot2(s3, v, v);
  }
  __device__ __forceinline__ void merge(const Dots& o) {
    s1 = df_add(s1, o.s1);
    s2 = df_add(s2, o.s2);
    s3 = df_add(s3, o.s3);
  }
  __device__ __forceinline__ Dots shfl_down(int off) const {
    Dots r;
    r.s1 = df_shfl_down(s1, off);
    r.s2 = df_shfl_down(s2, off);
    r.s3 = df_shfl_down(s3, off);
    return r;
  }
  __device__ __forceinline__ void get(double& a, double& b, double& c) const {
    a = df_to_double(s1);
    b = df_to_double(s2);
    c = df_to_double(s3);
  }
};

// ---- paired FP32 arithmetic (Blackwell f32x2): one issue slot for two
// lane-wise FP32 operations, each with the IEEE round-to-nearest result of
// the scalar operation.
__device__ __forceinline__ unsigned long long x2_pk(float2 a) {
  unsigned long long r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a.x), "f"(a.y));
  return r;
}
__device__ __forceinline__ float2 x2_upk(unsigned long long r) {
  float2 a;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a.x), "=f"(a.y) : "l"(r));
  return a;
}
__device__ __forceinline__ float2 x2_add(float2 a, float2 b) {
  unsigned long long d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(x2_pk(a)), "l"(x2_pk(b)));
  return x2_upk(d);
}
__device__ __forceinline__ float2 x2_sub(float2 a, float2 b) {
  unsigned long long d;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(x2_pk(a)), "l"(x2_pk(b)));
  return x2_upk(d);
}
__device__ __forceinline__ float2 x2_mul(float2 a, float2 b) {
  unsigned long long d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(x2_pk(a)), "l"(x2_pk(b)));
  return x2_upk(d);
}
__device__ __forceinline__ float2 x2_fma(float2 a, float2 b, float2 c) {
  unsigned long long d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(x2_pk(a)), "l"(x2_pk(b)), "l"(x2_pk(c)));
  return x2_upk(d);
}

// The three sums of Dots<float> in Dot2 form over pairs of elements, on the
// paired instructions: two accumulators per sum (the pair's halves), merged
// into a Dots<float> at the end.  Per pair and sum: the product and its
// exact error (TwoProd by FMA), TwoSum into hi, the errors summed into lo.
struct Dot2x2 {
  float2 h1, l1, h2, l2, h3, l3;  // v.q, q.q, v.v
  __device__ __forceinline__ void zero() { h1 = l1 = h2 = l2 = h3 = l3 = make_float2(0.f, 0.f); }
  // (h, l) += x * y; xn = -x
  __device__ __forceinline__ static void acc(float2& h, float2& l, float2 x, float2 xn, float2 y) {
    const float2 p = x2_mul(x, y);
    const float2 pen = x2_fma(xn, y, p);  // p - x y = -(rounding error of p), exact
    const float2 s = x2_add(h, p);
    const float2 bb = x2_sub(s, h);
    const float2 e = x2_add(x2_sub(h, x2_sub(s, bb)), x2_sub(p, bb));
    l = x2_add(l, x2_sub(e, pen));
    h = s;
  }
  __device__ __forceinline__ void add(float2 v, float2 q) {
    const float2 vn = make_float2(-v.x, -v.y), qn = make_float2(-q.x, -q.y);
    acc(h1, l1, v, vn, q);
    acc(h2, l2, q, qn, q);
    acc(h3, l3, v, vn, v);
  }
  __device__ __forceinline__ Dots<float> merged() const {
    Dots<float> d;
    d.s1 = df_add({h1.x, l1.x}, {h1.y, l1.y});
    d.s2 = df_add({h2.x, l2.x}, {h2.y, l2.y});
    d.s3 = df_add({h3.x, l3.x}, {h3.y, l3.y});
    return d;
  }
};

template <>
struct Dots<double> {
  typedef double S;
  double s1, s2, s3;
  __device__ __forceinline__ void zero() { s1 = s2 = s3 = 0.0; }
  __device__ __forceinline__ void add(double v, double q) {
    s1 = fma(v, q, s1);
    s2 = fma(q, q, s2);
    s3 = fma(v, v, s3);
  }
  __device__ __forceinline__ void merge(const Dots& o) {
    s1 += o.s1;
    s2 += o.s2;
    s3 += o.s3;
  }
  __device__ __forceinline__ Dots shfl_down(int off) const {
    Dots r;
    r.s1 = __shfl_down_sync(0xffffffffu, s1, off);
    r.s2 = __shfl_down_sync(0xffffffffu, s2, off);
    r.s3 = __shfl_down_sync(0xffffffffu, s3, off);
    return r;
  }
  __device__ __forceinline__ void get(double& a, double& b, double& c) const {
    a = s1;
    b = s2;
    c = s3;
  }
};

// Fixed-order block reduction (result valid in thread 0).  `scratch` must
// hold blockDim/32 entries.  The tree depends only on the block shape.
template <typename A>
__device__ __forceinline__ A block_reduce(A v, A* scratch) {
  const int tid = threadIdx.x + blockDim.x * (threadIdx.y + blockDim.y * threadIdx.z);
  const int lane = tid & 31;
  const int warp = tid >> 5;
  const int nwarps = (blockDim.x * blockDim.y * blockDim.z) >> 5;
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) v.merge(v.shfl_down(off));
  if (lane == 0) scratch[warp] = v;
  __syncthreads();
  if (warp == 0) {
    A w;
    if (lane < nwarps) w = scratch[lane];
    else w.zero();
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) w.merge(w.shfl_down(off));
    v = w;
  }
  __syncthreads();
  return v;
}

// The three sums of a Dots over a warp with six additions per lane instead of
// fifteen: lanes 16-31 take s3, lanes 0-15 s1 and s2 and then lanes 8-15 s2.
// Returns s1 in lanes 0-7, s2 in 8-15, s3 in 16-31 (all lanes of a range hold the
// same value).  An FP64 addition occupies the SM's FP64 lanes for 16 cycles per
// warp, so in the small FP64 steps these additions outweigh the stencil.
template <typename T>
__device__ __forceinline__ typename Dots<T>::S warp_sum3(const Dots<T>& v) {
  typedef typename Dots<T>::S S;
  const int lane = (threadIdx.x + blockDim.x * (threadIdx.y + blockDim.y * threadIdx.z)) & 31;
  const bool h16 = (lane & 16) != 0, h8 = (lane & 8) != 0;
  S k = h16 ? v.s3 : v.s1;
  k = sum_add(k, sum_xor(h16 ? v.s1 : v.s3, 16));
  const S k2 = sum_add(v.s2, sum_xor(v.s2, 16));
  const S give = (h16 || h8) ? k : k2;
  if (!h16 && h8) k = k2;
  k = sum_add(k, sum_xor(give, 8));
#pragma unroll
  for (int off = 4; off > 0; off >>= 1) k = sum_add(k, sum_xor(k, off));
  return k;
}

// The threads that run a sum or the end of a step together: the whole block, or
// the first N threads of a larger one.
struct BlockThreads {
  static __device__ __forceinline__ void sync() { __syncthreads(); }
  static __device__ __forceinline__ int count() { return (int)(blockDim.x * blockDim.y * blockDim.z); }
};
template <int N>
struct FirstThreads {
  static __device__ __forceinline__ void sync() { asm volatile("bar.sync 1, %0;" ::"n"(N) : "memory"); }
  static __device__ __forceinline__ int count() { return N; }
};

// Sum over the first nw warps of a group of warps, in a fixed order; the result is
// valid in every lane of the group's warp 0.  `warp` is the caller's place in its
// group.  Every thread of `Threads` calls it, and a barrier has to come before
// `scratch` is used again.
template <typename T, typename Threads = BlockThreads>
__device__ __forceinline__ Dots<T> reduce_group(const Dots<T>& v, Dots<T>* scratch, int nw, int warp) {
  typedef typename Dots<T>::S S;
  const int tid = threadIdx.x + blockDim.x * (threadIdx.y + blockDim.y * threadIdx.z);
  const int lane = tid & 31;
  S k = warp < nw ? warp_sum3(v) : S();
  if (nw > 1) {
    S* sc = reinterpret_cast<S*>(scratch);  // [warp][3]
    const int f = lane == 0 ? 0 : (lane == 8 ? 1 : 2);
    if (warp < nw && (lane == 0 || lane == 8 || lane == 16)) sc[warp * 3 + f] = k;
    Threads::sync();
    if (warp == 0) {
      // lane 8 f + i adds the warps i, i + 8, ...
      const int g = min(lane >> 3, 2), i = lane & 7;
      k = i < nw ? sc[i * 3 + g] : S();
      for (int w = i + 8; w < nw; w += 8) k = sum_add(k, sc[w * 3 + g]);
#pragma unroll
      for (int off = 4; off > 0; off >>= 1) k = sum_add(k, sum_xor(k, off));
    }
  }
  Dots<T> r;
  r.s1 = sum_from(k, 0);
  r.s2 = sum_from(k, 8);
  r.s3 = sum_from(k, 16);
  return r;
}
template <typename T, typename Threads = BlockThreads>
__device__ __forceinline__ Dots<T> reduce_warps(const Dots<T>& v, Dots<T>* scratch, int nw) {
  const int tid = threadIdx.x + blockDim.x * (threadIdx.y + blockDim.y * threadIdx.z);
  return reduce_group<T, Threads>(v, scratch, nw, tid >> 5);
}
template <typename T>
__device__ __forceinline__ Dots<T> block_sum(const Dots<T>& v, Dots<T>* scratch) {
  return reduce_warps(v, scratch, (int)(blockDim.x * blockDim.y * blockDim.z) >> 5);
}
template <typename T>
__device__ __forceinline__ Dots<T> block_reduce(const Dots<T>& v, Dots<T>* scratch) {
  const Dots<T> r = block_sum(v, scratch);
  __syncthreads();
  return r;
}

// ------------------------------------------------------------- iteration state
// One record per vector (sample z or probe v) of a Lanczos batch.
struct VecState {
  int status;     // VS_RUNNING, VS_DONE or a negative gmrf error code
  int m;          // completed steps = number of alpha values
  int m_min;      // the stopping rule may end the iteration only once m >= m_min (0: any m)
  int pad_;
  double znorm;   // ||z||
  double d_prev;  // 1 / d_{m-1}, the reciprocal of the LDL^T pivot d_{m-1} of T_m
  double u_prev;  // u_{m-1} = (L^{-1} e_1)_{m-1}
  double energy;  // e_1^T T_m^{-1} e_1 = sum_i u_i^2 / d_i
  double theta;   // smallest Ritz value theta_min (upper estimate)
  double err_est; // relative Theorem 1 estimate at m
  double amax;    // max |alpha_i|
  double bmax;    // max beta_i, i < m - 1
  double beta_last;  // beta_{m-1}
  double vscale;     // 1 / ||z|| at m = 0, then 1 / beta_{m-1}: the scale of v_m (one division per step)
};

// Loop-invariant parameters of the Lanczos steps.  The step index j (the
// basis vector v_j formed in the step, 0-based) is not a parameter: every
// step kernel reads it from its vector's state (VecState.m = completed
// steps), so one captured CUDA graph of c steps can be replayed.
struct StepParams {
  int m_max;      // largest subspace size
  int nslots;     // ring size of the stored basis (m_max + 1, or 2 when V_m is not kept)
  int solve;      // 1: the iteration solves A u = z (stopping rule on the CG residual), 0: sampling / quadrature
  double tol;     // stopping tolerance on the relative estimate
  double bd_tol;  // breakdown threshold relative to ||T_m||
  // bfloat16 copy of the basis for the assembly only ([nvec][m_max + 1][n]),
  // or null.  When set, the FP32 ring above holds just v_{j-1}, v_j (nslots 2),
  // so the recurrence itself is the same as with an FP32 basis.
  __nv_bfloat16* vb;
};

// Stores of v_j into the bfloat16 basis copy (round to nearest even).
__device__ __forceinline__ __nv_bfloat16* vb_at(const StepParams& P, int s, int j, size_t n, size_t i) {
  return P.vb + ((size_t)s * (size_t)(P.m_max + 1) + (size_t)j) * n + i;
}
__device__ __forceinline__ void vb_store1(__nv_bfloat16* p, float a) { *p = __float2bfloat16_rn(a); }
__device__ __forceinline__ void vb_store2(__nv_bfloat16* p, float a, float b) {
  *reinterpret_cast<__nv_bfloat162*>(p) = __floats2bfloat162_rn(a, b);
}
__device__ __forceinline__ void vb_store4(__nv_bfloat16* p, float a, float b, float c, float d) {
  const __nv_bfloat162 lo = __floats2bfloat162_rn(a, b), hi = __floats2bfloat162_rn(c, d);
  uint2 u;
  u.x = *reinterpret_cast<const unsigned*>(&lo);
  u.y = *reinterpret_cast<const unsigned*>(&hi);
  *reinterpret_cast<uint2*>(p) = u;
}

// Whether T_m has an eigenvalue at or below sigma: a leading determinant of
// T_m - sigma I that is not positive (Sturm sequence), in FP32 on float copies of alpha and
// beta^2.  The determinants' recurrence takes one dependent FMA per row where the
// pivots' takes a division; scale (a power of two near 1 / ||T_m||) and a power of two
// every fourth row keep it in range.
// Range: FP32 copies of T_m resolve eigenvalues down to about 1e-7 ||T_m||.  On spectra of
// condition up to 1e8 this and the pivots' form answer alike; beyond, both answer by their
// rounding, and pivots below about 10^-9.5 ||T_m|| in four consecutive rows underflow the
// determinants to 0, which counts as an eigenvalue below sigma.
__device__ __forceinline__ bool ritz_below(const float* __restrict__ af, const float* __restrict__ b2f, int m,
                                           float sigma, float scale) {
  float p1 = 1.f, p = (af[0] - sigma) * scale;
  bool bad = !(p > 0.f);
  int i = 1;
  auto row = [&](float a, float b2) {
    const float n = fmaf((a - sigma) * scale, p, -((b2 * scale) * scale) * p1);
    p1 = p;
    p = n;
    bad |= !(p > 0.f);
  };
  for (; i + 4 <= m; i += 4) {
    float a[4], b2[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      a[k] = af[i + k];
      b2[k] = b2f[i + k - 1];
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) row(a[k], b2[k]);
    // the power of two that brings the larger of the two near 1 (what follows a
    // determinant that is not positive does not matter)
    const int ex = (__float_as_int(fmaxf(p, p1)) >> 23) & 0xff;
    const float f = __int_as_float(min(max(254 - ex, 1), 254) << 23);
    p *= f;
    p1 *= f;
  }
  for (; i < m; ++i) row(af[i], b2f[i - 1]);
  return bad;
}

// Smallest eigenvalue of T_m by multisection over the block's threads on a
// geometric grid below `hi` (an upper bound).  All threads of the block call
// it; the result is returned to every thread.  Relative resolution 3e-4 or
// better, whatever the block's size, ample for the bound's lambda_min^{-1/2}.
// The first window is eight decades below hi, where 256 threads need two rounds, or
// two, where fewer do unless theta fell by more than that since it was last formed.
template <typename Threads>
__device__ __noinline__ static double smallest_ritz(const float* af, const float* b2f, int m, double hi_in, float scale,
                                                    int* s_int, float* s_flt) {
  const int tid = threadIdx.x + blockDim.x * (threadIdx.y + blockDim.y * threadIdx.z);
  const int nt = Threads::count();
  const float window = nt >= 256 ? 1e-8f : 1e-2f;
  float hi = (float)(hi_in * 1.0001) + 1e-30f;
  float lo = hi * window;
  for (int round = 0; round < 12; ++round) {
    // points p_t = lo * (hi/lo)^(t/(nt-1)), t = 0..nt-1
    const float lr = __logf(hi / lo) / (float)(nt - 1);
    float p = lo * __expf(lr * (float)tid);
    if (tid == 0) p = lo;
    if (tid == nt - 1) p = hi;
    const bool c = ritz_below(af, b2f, m, p, scale);
    if (tid == 0) s_int[0] = nt;  // first point with an eigenvalue below
    Threads::sync();
    if (c) atomicMin(&s_int[0], tid);
    Threads::sync();
    if (tid == 0) {
      const int t = s_int[0];
      float nlo = lo, nhi = hi;
      int again = 0;
      if (t == 0) {             // theta_min below lo: move the window down
        nhi = lo;
        nlo = lo * window;
        again = (nlo > 1e-35f) ? 2 : 3;
      } else if (t == nt) {     // hi was not an upper bound: widen up
        nlo = hi;
        nhi = hi * 1e4f;
        again = 2;
      } else {
        if (t < nt - 1) nhi = lo * __expf(lr * (float)t);
        if (t > 1) nlo = lo * __expf(lr * (float)(t - 1));
        again = (round == 0 || nhi > nlo * 1.0003f) ? 1 : 0;
      }
      s_flt[0] = nlo;
      s_flt[1] = nhi;
      s_int[1] = again;
    }
    Threads::sync();
    lo = s_flt[0];
    hi = s_flt[1];
    int again = s_int[1];
    Threads::sync();
    if (again == 0 || again == 3) break;
  }
  return (double)hi;
}

// Hands a block's partial sums to the block of vector s that comes last:
// publish() stores them and counts the block in, one acquire-release operation
// of thread 0 that orders this record alone (no fence of the whole block, which
// would wait for every store of q_j), and publish_wait() returns, in every
// thread, whether the block is the last of the nblk blocks of the vector (the
// counter is reset by it).  Stores that nobody reads before the kernel ends
// belong between the two.
__device__ __forceinline__ unsigned count_in(unsigned* counter) {
  unsigned t;
  asm volatile("atom.add.acq_rel.gpu.global.u32 %0, [%1], 1;" : "=r"(t) : "l"(counter) : "memory");
  return t;
}
template <typename T>
__device__ __forceinline__ unsigned publish(const Dots<T>& d, Dots<T>* partials, unsigned* counter, int s, int blk,
                                            int nblk) {
  const int tid = threadIdx.x + blockDim.x * (threadIdx.y + blockDim.y * threadIdx.z);
  unsigned t = 0;
  if (tid == 0) {
    partials[(size_t)s * nblk + blk] = d;
    if (nblk > 1) t = count_in(counter + s);
  }
  return t;
}
__device__ __forceinline__ bool publish_wait(unsigned t, unsigned* counter, int s, int nblk, int* s_flag) {
  const int tid = threadIdx.x + blockDim.x * (threadIdx.y + blockDim.y * threadIdx.z);
  if (tid == 0) {
    const int last = t == (unsigned)(nblk - 1);  // nblk 1: ticket 0
    if (last) counter[s] = 0u;
    *s_flag = last;
  }
  __syncthreads();
  return *s_flag != 0;
}
// a record another block published: from L2, whatever an L1 line holds
__device__ __forceinline__ Dots<float> load_partial(const Dots<float>* p) {
  const float2* q = reinterpret_cast<const float2*>(p);
  const float2 a = __ldcg(q), b = __ldcg(q + 1), c = __ldcg(q + 2);
  Dots<float> d;
  d.s1 = {a.x, a.y};
  d.s2 = {b.x, b.y};
  d.s3 = {c.x, c.y};
  return d;
}
__device__ __forceinline__ Dots<double> load_partial(const Dots<double>* p) {
  const double* q = reinterpret_cast<const double*>(p);
  Dots<double> d;
  d.s1 = __ldcg(q);
  d.s2 = __ldcg(q + 1);
  d.s3 = __ldcg(q + 2);
  return d;
}

// beta_j^2 from the three sums, or the caller's
__device__ __forceinline__ double step_b2(double a, double s2, double s3, double b2_direct) {
  return b2_direct >= 0.0 ? b2_direct : fma(a * a, s3 - 2.0, s2);
}

// Tests of doubles on their bits: a comparison takes the FP64 lanes as long as an addition.
__device__ __forceinline__ long long bits(double x) { return __double_as_longlong(x); }
__device__ __forceinline__ bool is_finite(double x) { return (__double2hiint(x) & 0x7ff00000) != 0x7ff00000; }
__device__ __forceinline__ bool is_positive(double x) { return bits(x) > 0; }  // of a finite x
// larger of two doubles that are not negative
__device__ __forceinline__ double larger(double x, double y) { return bits(x) > bits(y) ? x : y; }
__device__ __forceinline__ double one_sum(df v) { return df_to_double(v); }
__device__ __forceinline__ double one_sum(double v) { return v; }

// End of a Lanczos step for vector s, run by the last block of that vector
// (every thread of the block calls it).  Sums the per-block partial dot
// products in a fixed order, forms alpha_j and beta_j, advances the LDL^T
// recurrence of T_m and applies the stopping rule:
//   est = theta_min^{-1/2} ||r_m|| / ||x_m||,
//   ||r_m|| / ||z|| = beta_{m-1} |u_{m-1} / d_{m-1}|,  ||x_m|| / ||z|| = sqrt(e_1^T T_m^{-1} e_1).
// beta_j^2 comes from the three sums (one pass over the vectors), or, when
// b2_direct >= 0, is b2_direct = ||q_j - alpha_j v_j||^2 summed by a caller
// that holds both vectors (a second pass; exact also when beta_j << ||q_j||,
// where the one-pass form cancels to rounding noise).
//
// This runs between every two steps, so its latency counts in full.  GB300's
// dependent FP64 operations take about 64 cycles, a division or square root
// about 600: what the next step needs (alpha, beta, 1 / beta) is one warp's
// reciprocal square root, the recurrence of T_m (1 / d_j) and the stopping rule,
//   beta_j^2 u^2 / d^2 <= tol^2 (u-energy) theta,
// another's, both from beta_j^2; square roots of the estimate are taken only in a
// step that may stop.  The state's fields are loaded ahead, one per lane, and
// written one by one: a copy of the record costs the kernels this is inlined into
// registers (spills in the 3-D step's item loop, 4 % of a step at 256^3, 8 vectors).
// Only as many warps as there are partial sums take part in the sum.
// With warp_sum3 and publish(), before and now: FP64 64 x 64 step 17.2 -> 11.7 us
// (one vector; 12.7 with all of it in one warp), 93 -> 48 us (256 vectors); 512 x 512
// row-last pass, 320 vectors, 346 -> 317 us.  Comparisons on the bits, beta_j^2 in three
// operations, a lane per sum where pairs of floats become doubles, and smallest_ritz on
// determinants (26 us a call at m = 100 with a division per row and two counts in one
// thread): samples of 64 x 64 in FP64 849 -> 747 us, 61 x 75 x 90 1008 -> 982, 1024 x 1024
// 3904 -> 3768, 24 slots of 256 x 256 5489 -> 5313.
// The records come from rec(b), and rec's Threads run it; where the caller keeps the
// iteration in one kernel (Rec::kept), the state is in shared memory, alpha, beta, 1 / beta and the
// status also go to rec's shared copy, and the caller stores alpha_j and beta_j.
template <typename T, typename Rec>
__device__ __forceinline__ void finish_step_from(const StepParams& P, int j, int s, const Rec& rec, int nblk,
                            VecState* __restrict__ st, double* __restrict__ alpha, double* __restrict__ beta,
                            float* __restrict__ alpha_f, float* __restrict__ beta2_f, Dots<T>* red_scratch,
                            int* s_int, float* s_flt, double b2_direct) {
  typedef typename Rec::Threads Threads;
  const int tid = threadIdx.x + blockDim.x * (threadIdx.y + blockDim.y * threadIdx.z);
  const int nt = Threads::count();
  const int warp = tid >> 5, lane = tid & 31;
  const int nw = min(nt >> 5, (nblk + 31) >> 5);
  __shared__ int s_need_theta;
  __shared__ double s_theta_hi, s_pfac;
  __shared__ float s_scale;
  const size_t mo = (size_t)s * P.m_max;
  VecState* const v = st + s;
  // the state's fields d_prev .. beta_last, one per lane of warp 1 (the only warp
  // of a block of 32 threads: warp 0), in flight while the sums are formed
  const int wb = nt > 32 ? 1 : 0;
  const double field = warp == wb && lane < 8 ? (&v->d_prev)[lane] : 0.0;
  __shared__ double s_sum[3];
  Dots<T> acc;
  acc.zero();
  if (warp < nw)
    if (tid < nblk) {
      acc = rec(tid);
      for (int b = tid + 32 * nw; b < nblk; b += 32 * nw) acc.merge(rec(b));
    }
  acc = reduce_warps<T, Threads>(acc, red_scratch, nw);
  if (tid < 3) s_sum[tid] = one_sum(tid == 0 ? acc.s1 : (tid == 1 ? acc.s2 : acc.s3));  // a lane each
  Threads::sync();
  const double a = s_sum[0];
  // warp 0: alpha_j, beta_j and 1 / beta_j, which the next step waits for
  if (warp == 0) {
    const double b2 = step_b2(a, s_sum[1], s_sum[2], b2_direct);
    // a number, positive, and neither b2 nor 1 / sqrt(b2) near the ends of the range
    const bool plain = bits(b2) > bits(1e-290) && bits(b2) < bits(1e300);
    const double y = plain || b2 > 0.0 ? rsqrt(b2) : 0.0;
    // beta_j = sqrt(b2) from y by one Newton step on the residual b2 - b^2
    double b = b2 * y;
    b = fma(fma(-b, b, b2), 0.5 * y, b);
    if (!plain) b = b2 > 0.0 ? sqrt(b2) : 0.0;
    if (lane == 0) {
      if constexpr (Rec::kept) {
        rec.keep(a, b, y);
      } else {
        alpha[mo + j] = a;
        beta[mo + j] = b;
        alpha_f[mo + j] = (float)a;
        beta2_f[mo + j] = (float)(b * b);
      }
      v->beta_last = b;
      v->vscale = y;
    }
  }
  // warp 1: the recurrence of T_m and the stopping rule, on beta_j^2
  if (warp == wb) {
    const double b2 = step_b2(a, s_sum[1], s_sum[2], b2_direct);
    auto prev = [&](int k) { return __shfl_sync(0xffffffffu, field, k); };
    const double d_prev = prev(0), u_prev = prev(1), b_prev = prev(7);
    // LDL^T of T_m: d_0 = a_0, d_j = a_j - b_{j-1}^2 / d_{j-1}; u_0 = 1, u_j = -(b_{j-1}/d_{j-1}) u_{j-1}
    // (the state keeps 1 / d_{j-1})
    double d = a, u = 1.0, energy = prev(2), theta = prev(3), err = prev(4), amax = prev(5), bmax = prev(6);
    if (j > 0) {
      const double r = b_prev * d_prev;  // b_{j-1} / d_{j-1}
      d = a - b_prev * r;
      u = -r * u_prev;
    } else {
      energy = amax = bmax = 0.0;
      theta = a;
    }
    const double dinv = 1.0 / d;
    const bool finite = is_finite(a) && is_finite(b2) && is_finite(d);
    int need = 0, status = VS_RUNNING;
    double pfac = 0.0;
    amax = larger(amax, fabs(a));
    if (j > 0) bmax = larger(bmax, b_prev);
    if (!finite || !is_positive(d) || !is_positive(a)) {
      // the estimate of the last completed step stays on record
      status = finite ? GMRF_ERR_NOT_SPD : GMRF_ERR_NUMERIC;
      if (j > 0) {
        err = b_prev * fabs(u_prev) * d_prev;
        if (!P.solve) err *= rsqrt(energy) * rsqrt(theta);
      }
    } else {
      const double ud = u * dinv;
      energy += u * ud;
      // (||r_m|| / ||z||)^2, compared with tol^2 to save the square roots of a step that
      // does not stop.  Both underflow for tolerances below 1e-154, so a stop is decided on
      // the residual itself, formed from the factors where the square has lost digits
      const double rr2 = (is_positive(b2) ? b2 : 0.0) * (ud * ud);
      auto rres = [&]() {
        const bool tiny = bits(rr2) < bits(1e-280);
        const double r = sqrt(tiny ? (is_positive(b2) ? b2 : 0.0) : rr2);
        return tiny ? r * fabs(ud) : r;
      };
      const double bd = P.bd_tol * (amax + bmax);
      if (bits(b2) <= bits(bd * bd)) {  // bd is not negative; a negative b2 is the smaller one here too
        status = VS_DONE;  // invariant Krylov subspace: x_m is exact
        err = 0.0;
        need = !P.solve;   // theta still wanted for the T_m function of a sample
      } else if (P.solve) {
        // linear solve: x_m = ||z|| V_m T_m^{-1} e_1 is the CG iterate, with
        // relative residual ||r_m|| / ||z|| = beta_m |e_m^T T_m^{-1} e_1|
        if (bits(rr2) <= bits(P.tol * P.tol) || j + 1 >= P.m_max) {
          const double r = rres();
          if (r <= P.tol) status = VS_DONE;
          else if (j + 1 >= P.m_max) status = GMRF_ERR_NOT_CONVERGED;
          if (status != VS_RUNNING) err = r;
        }
      } else if (bits(rr2) <= bits(P.tol * P.tol * (energy * theta)) || j + 1 >= P.m_max) {
        // est_lb = ||r_m|| / (||x_m|| theta^{1/2}), theta >= theta_min(T_m), is a lower bound of est
        need = 1;
        pfac = rres() * rsqrt(energy);  // ||r_m|| / ||x_m||
        err = pfac * rsqrt(theta);
      }
    }
    if (lane == 0) {
      if (status != GMRF_ERR_NOT_SPD && status != GMRF_ERR_NUMERIC) {
        v->d_prev = dinv;
        v->u_prev = u;
      }
      v->m = j + 1;
      v->energy = energy;
      v->theta = theta;
      v->err_est = err;
      v->amax = amax;
      v->bmax = bmax;
      v->status = status;
      if constexpr (Rec::kept) *rec.status = status;
      s_pfac = pfac;
      s_need_theta = need;
      s_theta_hi = theta;
      // 1 over the power of two in max |alpha_i|, a scale of T_m
      s_scale = __int_as_float(min(max(254 - ((__float_as_int((float)amax) >> 23) & 0xff), 1), 253) << 23);
    }
  }
  Threads::sync();
  if (s_need_theta) {
    if constexpr (Rec::kept) {
      if (tid == 0) {
        alpha_f[mo + j] = (float)rec.scalars[0];
        beta2_f[mo + j] = (float)(rec.scalars[1] * rec.scalars[1]);
      }
      Threads::sync();
    }
    double th = smallest_ritz<Threads>(alpha_f + mo, beta2_f + mo, j + 1, s_theta_hi, s_scale, s_int, s_flt);
    if (tid == 0) {
      v->theta = th;
      if (v->status == VS_RUNNING) {
        const double est = s_pfac * rsqrt(th);
        v->err_est = est;
        if (est <= P.tol && j + 1 >= v->m_min) v->status = VS_DONE;
        else if (j + 1 >= P.m_max) v->status = GMRF_ERR_NOT_CONVERGED;
        if constexpr (Rec::kept) *rec.status = v->status;
      }
    }
  }
}

// the records that the blocks of a vector published
template <typename T>
struct PublishedRecords {
  static constexpr bool kept = false;
  typedef BlockThreads Threads;
  const Dots<T>* p;
  __device__ __forceinline__ Dots<T> operator()(int b) const { return load_partial(p + b); }
};
template <typename T>
__device__ static void finish_step(const StepParams& P, int j, int s, const Dots<T>* __restrict__ partials, int nblk,
                            VecState* __restrict__ st, double* __restrict__ alpha, double* __restrict__ beta,
                            float* __restrict__ alpha_f, float* __restrict__ beta2_f, Dots<T>* red_scratch,
                            int* s_int, float* s_flt, double b2_direct = -1.0) {
  finish_step_from<T>(P, j, s, PublishedRecords<T>{partials + (size_t)s * nblk}, nblk, st, alpha, beta, alpha_f,
                      beta2_f, red_scratch, s_int, s_flt, b2_direct);
}


// ------------------------------------------------------------------- Philox
__device__ __forceinline__ void philox4x32_10(uint32_t c[4], uint32_t k0, uint32_t k1) {
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    if (r) {
      k0 += 0x9E3779B9u;
      k1 += 0xBB67AE85u;
    }
    uint32_t lo0 = 0xD2511F53u * c[0];
    uint32_t hi0 = __umulhi(0xD2511F53u, c[0]);
    uint32_t lo1 = 0xCD9E8D57u * c[2];
    uint32_t hi1 = __umulhi(0xCD9E8D57u, c[2]);
    uint32_t n0 = hi1 ^ c[1] ^ k0;
    uint32_t n2 = hi0 ^ c[3] ^ k1;
    c[0] = n0;
    c[1] = lo1;
    c[2] = n2;
    c[3] = lo0;
  }
}

}  // namespace gmrf
