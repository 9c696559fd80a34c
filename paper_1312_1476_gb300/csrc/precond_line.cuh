// precond_line.cuh -- B_bar^{-1} by a transform along x and a recurrence along
// y, and the preconditioned Lanczos step built on it (squared operators, whose
// M^{-1/2} is B_bar^{-1}; see precond.cu for the operator).
//
// After the transform along x (DCT-II for MIRROR, real FFT for CIRCULANT)
// B_bar = kappa_bar^2 + L_x + L_y falls apart into one tridiagonal Toeplitz
// system per spectral column, (2 + s - shift - shift^-1) w = x with
// s = kappa_bar^2 + lambda_x.  Its Green's function is the two-sided
// exponential rho^|i| / (1/rho - rho), rho + 1/rho = 2 + s, so
//   w_i = gain (rho f_{i-1} + b_i),  f_i = x_i + rho f_{i-1},  b_i = x_i + rho b_{i+1},
// and the ends only set what enters the two recurrences: the reflected (or
// wrapped) sequence, f_{-1} = (b_0 + rho^N f_{N-1}) / (1 - rho^2N) with zero
// start values on the right (CIRCULANT f_{-1} = f_{N-1} / (1 - rho^N)).  About
// ten operations per value instead of a forward and an inverse transform, and
// nothing is transposed: the spectrum stays in rows.  rho enters as 1 - delta
// with delta rounded from FP64, so the gain 1/s of the smooth modes keeps full
// relative accuracy for any kappa_bar^2.
//
// The order of a spectrum row is free (a column only needs its own rho), so a
// row is stored the way the half-length FFT ends: pairs k = 0 .. L/2 - 1
// (L = nx/2), four reals each, {C_k, C_{N-k}, C_{L-k}, C_{L+k}} for MIRROR and
// {X_k, X_{L-k}} for CIRCULANT; pair 0 holds k = 0, L and L/2.
//
// Rows: T = L/8 threads per line, eight complex values each, Stockham radix-8
// passes (a last pass of 2 or 4) with padded shared-memory exchanges.  A line of
// up to 512 points lives inside a warp, so its exchanges need no block barrier;
// longer ones use a named barrier of their own threads.  The passes are bound by
// latency at one vector (each runs for a few microseconds on data in L2) and by
// instruction issue in a block of vectors; eight values per thread give a 1024-wide
// row two warps and 27 instructions per value and transform.
//
// Measured on GB300 against the kernels this replaces (transforms both ways
// along y on a transposed spectrum, one line per warp), FP32 MIRROR 1024 x 1024,
// one vector, profiler times with a warm cache: row-forward 9.3 -> 6.0 us, columns 11.2 ->
// 5.0, row-mid 14.2 -> 6.7, row-last with the step's scalar tail 16.7 -> 11.0; a step of an
// untraced call 57 -> 30.3.  320 vectors of 512 x 512, about 58 steps: 108 -> 67 ms a call,
// the passes of a step at 6.6 (row-forward), 5.3, 5.1 and 4.8 TB/s of their 17 arrays.  FP64
// CIRCULANT 512 x 512 step 81 -> 42 us.  Error of M^{-1/2} v against 64 bits at 128 x 128:
// 2.6e-7 -> 1.6e-7.
#pragma once

#include <cuda_runtime.h>

#include <utility>

#include "per_device.h"
#include "precond_line.h"
#include "trace.h"

namespace gmrf {
namespace line {

enum { L_FWD = 0, L_INV = 1, L_MID = 2, L_MIDW = 3, L_MIDG = 4, L_LAST = 5 };

// ------------------------------------------------------------ complex helpers
template <typename C>
struct RealOf;
template <>
struct RealOf<float2> { typedef float T; };
template <>
struct RealOf<double2> { typedef double T; };

template <typename C>
__device__ __forceinline__ C mk(typename RealOf<C>::T x, typename RealOf<C>::T y) {
  C r;
  r.x = x;
  r.y = y;
  return r;
}
template <typename C>
__device__ __forceinline__ C cadd(C a, C b) { return mk<C>(a.x + b.x, a.y + b.y); }
template <typename C>
__device__ __forceinline__ C csub(C a, C b) { return mk<C>(a.x - b.x, a.y - b.y); }
template <typename C>
__device__ __forceinline__ C cmul(C a, C b) { return mk<C>(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x); }
template <typename C>  // a * conj(b)
__device__ __forceinline__ C cmulc(C a, C b) { return mk<C>(a.x * b.x + a.y * b.y, a.y * b.x - a.x * b.y); }
// multiplication by -i (forward) or +i (inverse)
template <bool INV, typename C>
__device__ __forceinline__ C rot(C a) { return INV ? mk<C>(-a.y, a.x) : mk<C>(a.y, -a.x); }

template <bool INV, typename C>
__device__ __forceinline__ void dft2(C& a, C& b) {
  const C t = csub(a, b);
  a = cadd(a, b);
  b = t;
}
template <bool INV, typename C>
__device__ __forceinline__ void dft4(C& v0, C& v1, C& v2, C& v3) {
  const C s0 = cadd(v0, v2), d0 = csub(v0, v2), s1 = cadd(v1, v3), d1 = rot<INV>(csub(v1, v3));
  v0 = cadd(s0, s1);
  v2 = csub(s0, s1);
  v1 = cadd(d0, d1);
  v3 = csub(d0, d1);
}
template <bool INV, typename C>
__device__ __forceinline__ void dft8(C (&v)[8]) {
  typedef typename RealOf<C>::T R;
  const R h = (R)0.70710678118654752440;
  const C a0 = cadd(v[0], v[4]), a4 = csub(v[0], v[4]), a2 = cadd(v[2], v[6]), a6 = rot<INV>(csub(v[2], v[6]));
  const C a1 = cadd(v[1], v[5]), a5 = csub(v[1], v[5]), a3 = cadd(v[3], v[7]), a7 = rot<INV>(csub(v[3], v[7]));
  const C b0 = cadd(a0, a2), b2 = csub(a0, a2), b4 = cadd(a4, a6), b6 = csub(a4, a6);
  const C b1 = cadd(a1, a3), b3 = rot<INV>(csub(a1, a3)), b5 = cadd(a5, a7), b7 = csub(a5, a7);
  // e^{-+ i pi/4} b5 and e^{-+ 3 i pi/4} b7
  const C c5 = INV ? mk<C>(h * (b5.x - b5.y), h * (b5.x + b5.y)) : mk<C>(h * (b5.x + b5.y), h * (b5.y - b5.x));
  const C c7 = INV ? mk<C>(-h * (b7.x + b7.y), h * (b7.x - b7.y)) : mk<C>(h * (b7.y - b7.x), -h * (b7.x + b7.y));
  v[0] = cadd(b0, b1);
  v[4] = csub(b0, b1);
  v[2] = cadd(b2, b3);
  v[6] = csub(b2, b3);
  v[1] = cadd(b4, c5);
  v[5] = csub(b4, c5);
  v[3] = cadd(b6, c7);
  v[7] = csub(b6, c7);
}

// Programmatic dependent launch: a kernel of a chain may be placed while its
// predecessor drains; after_previous() returns once the predecessor has ended and
// its writes are visible, and every block calls it before anything else, also one
// that has nothing to do.  let_next() allows the successor to be placed.
__device__ __forceinline__ void after_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void let_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// ------------------------------------------------------------ lines of a block
__host__ __device__ constexpr int line_threads(int nx) { return nx / 16; }
__host__ __device__ constexpr int block_threads(int nx) { return line_threads(nx) > 128 ? line_threads(nx) : 128; }
__host__ __device__ constexpr int block_rows(int nx) { return block_threads(nx) / line_threads(nx); }
// shared-memory slot of element i of a line: one slot of padding per eight
__host__ __device__ constexpr int slot_of(int i) { return i + (i >> 3); }

// The threads of one line and its two exchange buffers.  Exchanges alternate
// between the buffers, so one synchronisation per exchange is enough: a
// buffer is rewritten only after the synchronisation of the exchange between.
template <typename R, int NX>
struct Line {
  typedef typename C2<R>::T C;
  static constexpr int L = NX / 2, T = L / 8;
  C* b;   // this line's buffers
  int t;  // thread of the line
  int id; // line of the block
  __device__ __forceinline__ C* buf(int which) const { return b + which * (slot_of(L)); }
  __device__ __forceinline__ void sync() const {
    if constexpr (T <= 32) __syncwarp();
    else asm volatile("bar.sync %0, %1;" ::"r"(1 + id), "n"(T) : "memory");
  }
};
template <typename R, int NX>
constexpr size_t row_smem() {
  return (size_t)block_rows(NX) * 2 * slot_of(NX / 2) * sizeof(typename C2<R>::T);
}

// Twiddles of the pass at stride NS > 1 of a length-L transform start at
// tw_off; entry (r, j) = exp(-2 pi i j r / (NS RAD)) at (r - 1) NS + j.
__host__ __device__ constexpr int pass_radix(int L, int NS) { return L / NS >= 8 ? 8 : L / NS; }
__host__ __device__ constexpr int tw_off(int L, int NS) {
  int off = 0;
  for (int ns = 8; ns < NS; ns *= 8) off += (pass_radix(L, ns) - 1) * ns;
  return off;
}

// Stockham passes from stride NS on.  v[r] holds element t + T r of the line
// before the first pass and after the last one.
template <typename R, int NX, int NS, bool INV>
__device__ __forceinline__ void fft_pass(typename C2<R>::T (&v)[8], const Line<R, NX>& ln,
                                         const typename C2<R>::T* __restrict__ tw, int& ph) {
  typedef typename C2<R>::T C;
  constexpr int L = NX / 2, T = L / 8, RAD = pass_radix(L, NS), Q = 8 / RAD;
  const int t = ln.t;
  if constexpr (NS > 1) {
    const C* w = tw + tw_off(L, NS);
#pragma unroll
    for (int q = 0; q < Q; ++q) {
      const int j = (t + T * q) & (NS - 1);
#pragma unroll
      for (int r = 1; r < RAD; ++r) {
        const C f = __ldg(w + (r - 1) * NS + j);
        v[q + r * Q] = INV ? cmulc(v[q + r * Q], f) : cmul(v[q + r * Q], f);
      }
    }
  }
  if constexpr (RAD == 8) dft8<INV>(v);
  else if constexpr (RAD == 4) {
    dft4<INV>(v[0], v[2], v[4], v[6]);
    dft4<INV>(v[1], v[3], v[5], v[7]);
  } else {
#pragma unroll
    for (int q = 0; q < 4; ++q) dft2<INV>(v[q], v[q + 4]);
  }
  if constexpr (NS * RAD < L) {
    C* sm = ln.buf(ph);
    ph ^= 1;
    const int base = (t / NS) * (NS * 8) + (t & (NS - 1));
#pragma unroll
    for (int r = 0; r < 8; ++r) sm[slot_of(base + r * NS)] = v[r];
    ln.sync();
#pragma unroll
    for (int r = 0; r < 8; ++r) v[r] = sm[slot_of(t + T * r)];
    fft_pass<R, NX, NS * 8, INV>(v, ln, tw, ph);
  }
}

template <int T>
__device__ __forceinline__ float shfl_t(float v, int src) { return __shfl_sync(0xffffffffu, v, src, T); }
template <int T>
__device__ __forceinline__ double shfl_t(double v, int src) { return __shfl_sync(0xffffffffu, v, src, T); }
template <int T, typename C>
__device__ __forceinline__ C shfl_c(C v, int src) { return mk<C>(shfl_t<T>(v.x, src), shfl_t<T>(v.y, src)); }

// Exchange of the upper half of a line with its mirror image, element i with
// OFF - i (OFF = L - 1: packing of the DCT; OFF = L: conjugate pairs).  up[r],
// r < 4, stands for element OFF - (t + T r) on one side and for element
// t + T (7 - r), which is v[7 - r], on the other: scatter goes from the first
// to the second, gather back.  With OFF = L, thread 0's up[0] stands for
// element L/2 (element 0 has no image).
template <typename R, int NX, int OFF, bool GATHER>
__device__ __forceinline__ void mirror_exchange(typename C2<R>::T (&up)[4], const Line<R, NX>& ln, int& ph) {
  typedef typename C2<R>::T C;
  constexpr int L = NX / 2, T = L / 8;
  const int t = ln.t;
  if constexpr (T <= 32) {
    const int src = OFF == L ? (T - t) & (T - 1) : T - 1 - t;
    C g[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) g[r] = shfl_c<T>(up[r], src);
    if (OFF == L && t == 0) {
      // thread 0 is its own image, one register further on: L - T r = T (8 - r)
      C o[4];
#pragma unroll
      for (int r = 0; r < 4; ++r) o[r] = up[r];
#pragma unroll
      for (int r = 0; r < 4; ++r) g[r] = GATHER ? o[(r + 3) & 3] : o[(r + 1) & 3];
    }
#pragma unroll
    for (int r = 0; r < 4; ++r) up[r] = g[r];
  } else {
    C* sm = ln.buf(ph);
    ph ^= 1;
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      int i = OFF - (t + T * r);
      if (OFF == L && i == L) i = L / 2;
      sm[slot_of(GATHER ? t + T * (7 - r) : i)] = up[r];
    }
    ln.sync();
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      int i = OFF - (t + T * r);
      if (OFF == L && i == L) i = L / 2;
      up[r] = sm[slot_of(GATHER ? i : t + T * (7 - r))];
    }
  }
}

// ------------------------------------------------------------ vector accesses
__device__ __forceinline__ void ld4(const float* p, float (&o)[4]) {
  const float4 v = *reinterpret_cast<const float4*>(p);
  o[0] = v.x; o[1] = v.y; o[2] = v.z; o[3] = v.w;
}
__device__ __forceinline__ void ld4(const double* p, double (&o)[4]) {
  const double2 a = *reinterpret_cast<const double2*>(p), b = *reinterpret_cast<const double2*>(p + 2);
  o[0] = a.x; o[1] = a.y; o[2] = b.x; o[3] = b.y;
}
__device__ __forceinline__ void st4(float* p, float a, float b, float c, float d) {
  *reinterpret_cast<float4*>(p) = make_float4(a, b, c, d);
}
__device__ __forceinline__ void st4(double* p, double a, double b, double c, double d) {
  *reinterpret_cast<double2*>(p) = make_double2(a, b);
  *reinterpret_cast<double2*>(p + 2) = make_double2(c, d);
}
__device__ __forceinline__ float2 ldpair(const float* p) { return *reinterpret_cast<const float2*>(p); }
__device__ __forceinline__ double2 ldpair(const double* p) { return *reinterpret_cast<const double2*>(p); }

// A real row as the 8 pairs of a thread: CIRCULANT pair r = x[2m, 2m+1] with
// m = t + T r; MIRROR pairs 2r, 2r+1 = x[4m .. 4m+3], r < 4.
template <int KIND, int T>
__device__ __forceinline__ int pair_at(int t, int r) {
  return KIND == GMRF_PREC_CIRCULANT ? 2 * (t + T * r) : 4 * (t + T * (r >> 1)) + 2 * (r & 1);
}
template <typename R, int KIND, int T>
__device__ __forceinline__ void load_row(typename C2<R>::T (&p)[8], const R* __restrict__ src, int t) {
  typedef typename C2<R>::T C;
  if constexpr (KIND == GMRF_PREC_CIRCULANT) {
#pragma unroll
    for (int r = 0; r < 8; ++r) p[r] = ldpair(src + 2 * (t + T * r));
  } else {
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      R q[4];
      ld4(src + 4 * (t + T * r), q);
      p[2 * r] = mk<C>(q[0], q[1]);
      p[2 * r + 1] = mk<C>(q[2], q[3]);
    }
  }
}
template <typename R, int KIND, int T>
__device__ __forceinline__ void store_row(const typename C2<R>::T (&p)[8], R* __restrict__ dst, int t) {
  typedef typename C2<R>::T C;
  if constexpr (KIND == GMRF_PREC_CIRCULANT) {
#pragma unroll
    for (int r = 0; r < 8; ++r) *reinterpret_cast<C*>(dst + 2 * (t + T * r)) = p[r];
  } else {
#pragma unroll
    for (int r = 0; r < 4; ++r)
      st4(dst + 4 * (t + T * r), p[2 * r].x, p[2 * r].y, p[2 * r + 1].x, p[2 * r + 1].y);
  }
}
// The same by element, for a caller's array that is not aligned for the vector accesses.
template <typename R, int KIND, int T>
__device__ __forceinline__ void load_row_elem(typename C2<R>::T (&p)[8], const R* __restrict__ src, int t) {
#pragma unroll
  for (int r = 0; r < 8; ++r) {
    const R* q = src + pair_at<KIND, T>(t, r);
    p[r] = mk<typename C2<R>::T>(q[0], q[1]);
  }
}
template <typename R, int KIND, int T>
__device__ __forceinline__ void store_row_elem(const typename C2<R>::T (&p)[8], R* __restrict__ dst, int t) {
#pragma unroll
  for (int r = 0; r < 8; ++r) {
    R* q = dst + pair_at<KIND, T>(t, r);
    q[0] = p[r].x;
    q[1] = p[r].y;
  }
}
template <typename R, int KIND, int T>
__device__ __forceinline__ void store_row_bf16(const typename C2<R>::T (&p)[8], __nv_bfloat16* dst, int t) {
  if constexpr (KIND == GMRF_PREC_CIRCULANT) {
#pragma unroll
    for (int r = 0; r < 8; ++r) vb_store2(dst + 2 * (t + T * r), (float)p[r].x, (float)p[r].y);
  } else {
#pragma unroll
    for (int r = 0; r < 4; ++r)
      vb_store4(dst + 4 * (t + T * r), (float)p[2 * r].x, (float)p[2 * r].y, (float)p[2 * r + 1].x,
                (float)p[2 * r + 1].y);
  }
}
// kappa^2 (always FP32 in memory) at the thread's pairs of a row
template <typename R, int KIND, int T>
__device__ __forceinline__ void load_kap(const Args<R>& a, size_t ro, typename C2<R>::T (&p)[8], int t) {
  typedef typename C2<R>::T C;
  if (!a.kappa2) {
#pragma unroll
    for (int r = 0; r < 8; ++r) p[r] = mk<C>(a.kappa2_const, a.kappa2_const);
    return;
  }
  float2 q[8];
  load_row<float, KIND, T>(q, a.kappa2 + ro, t);
#pragma unroll
  for (int r = 0; r < 8; ++r) p[r] = mk<C>((R)q[r].x, (R)q[r].y);
}

// ------------------------------------------------------------ row transforms
// {tw_k, d_k} of pair k (MIRROR) or {tw_k, -} (CIRCULANT)
__device__ __forceinline__ void ldpf(const float* p, float (&o)[4]) {
  const float4 v = __ldg(reinterpret_cast<const float4*>(p));
  o[0] = v.x; o[1] = v.y; o[2] = v.z; o[3] = v.w;
}
__device__ __forceinline__ void ldpf(const double* p, double (&o)[4]) {
  const double2 a = __ldg(reinterpret_cast<const double2*>(p)), b = __ldg(reinterpret_cast<const double2*>(p + 2));
  o[0] = a.x; o[1] = a.y; o[2] = b.x; o[3] = b.y;
}

// real row pairs p -> spectrum row S (packed pairs)
template <typename R, int KIND, int NX>
__device__ __forceinline__ void row_forward(const Args<R>& a, const typename C2<R>::T (&p)[8], R* __restrict__ S,
                                            const Line<R, NX>& ln, int& ph, bool live) {
  typedef typename C2<R>::T C;
  constexpr int L = NX / 2, T = L / 8;
  constexpr bool MIR = KIND == GMRF_PREC_MIRROR;
  const int t = ln.t;
  const R h = (R)0.70710678118654752440;
  C v[8], up[4];
  if constexpr (MIR) {
    // z[m] = (x[4m], x[4m+2]), z[L-1-m] = (x[4m+3], x[4m+1])
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      v[r] = mk<C>(p[2 * r].x, p[2 * r + 1].x);
      up[r] = mk<C>(p[2 * r + 1].y, p[2 * r].y);
    }
    mirror_exchange<R, NX, L - 1, false>(up, ln, ph);
#pragma unroll
    for (int r = 0; r < 4; ++r) v[7 - r] = up[r];
  } else {
#pragma unroll
    for (int r = 0; r < 8; ++r) v[r] = p[r];
  }
  fft_pass<R, NX, 1, false>(v, ln, a.tw, ph);
#pragma unroll
  for (int r = 0; r < 4; ++r) up[r] = v[7 - r];
  mirror_exchange<R, NX, L, true>(up, ln, ph);  // up[r] = Z[L - k], k = t + T r (thread 0: up[0] = Z[L/2])
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const int k = t + T * r;
    const C zk = v[r], zr = up[r];
    R f[4] = {0, 0, 0, 0};
    if constexpr (MIR) ldpf(a.pair + 4 * k, f);
    else {
      const C w = __ldg(reinterpret_cast<const C*>(a.pair) + k);
      f[0] = w.x;
      f[1] = w.y;
    }
    // X_k = (s - i d) / 2, X_{L-k} = (conj(s) - i conj(d)) / 2 with s = z_k + conj(z_{L-k}),
    // d = tw_k (z_k - conj(z_{L-k})); the halves are taken with d_k
    const C sk = mk<C>(zk.x + zr.x, zk.y - zr.y);
    const C dk = cmul(mk<C>(f[0], f[1]), mk<C>(zk.x - zr.x, zk.y + zr.y));
    const C Xk = mk<C>((R)0.5 * (sk.x + dk.y), (R)0.5 * (sk.y - dk.x));
    const C Xp = mk<C>((R)0.5 * (sk.x - dk.y), (R)-0.5 * (sk.y + dk.x));
    R o[4];
    if constexpr (MIR) {
      const C e = cmul(Xk, mk<C>(f[2], f[3]));    // d_k X_k
      const C g = cmulc(Xp, mk<C>(f[2], f[3]));   // d_{L-k} X_{L-k} = e^{-i pi/4} conj(d_k) X_{L-k}
      o[0] = e.x;
      o[1] = -e.y;
      o[2] = h * (g.x + g.y);
      o[3] = h * (g.x - g.y);
    } else {
      o[0] = Xk.x;
      o[1] = Xk.y;
      o[2] = Xp.x;
      o[3] = Xp.y;
    }
    if (r == 0 && t == 0) {
      // k = 0 and L from z_0, k = L/2 from z_{L/2} (X_{L/2} = conj z_{L/2})
      o[0] = zk.x + zk.y;
      if constexpr (MIR) {
        const C c8 = mk<C>((R)0.92387953251128675613, (R)-0.38268343236508977173);  // e^{-i pi/8}
        const C e = cmulc(c8, zr);
        o[1] = h * (zk.x - zk.y);
        o[2] = e.x;
        o[3] = -e.y;
      } else {
        o[1] = zk.x - zk.y;
        o[2] = zr.x;
        o[3] = -zr.y;
      }
    }
    if (live) st4(S + 4 * k, o[0], o[1], o[2], o[3]);
  }
}

// spectrum row q (load_spectrum) -> real row pairs p (times L)
template <typename R, int NX>
__device__ __forceinline__ void load_spectrum(R (&q)[4][4], const R* __restrict__ S, int t) {
  constexpr int T = line_threads(NX);
#pragma unroll
  for (int r = 0; r < 4; ++r) ld4(S + 4 * (t + T * r), q[r]);
}
template <typename R, int KIND, int NX>
__device__ __forceinline__ void row_inverse(const Args<R>& a, typename C2<R>::T (&p)[8], const R (&q)[4][4],
                                            const Line<R, NX>& ln, int& ph) {
  typedef typename C2<R>::T C;
  constexpr int L = NX / 2, T = L / 8;
  constexpr bool MIR = KIND == GMRF_PREC_MIRROR;
  const int t = ln.t;
  const R h = (R)0.70710678118654752440;
  C v[8], up[4];
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const int k = t + T * r;
    R f[4] = {0, 0, 0, 0};
    if constexpr (MIR) ldpf(a.pair + 4 * k, f);
    else {
      const C w = __ldg(reinterpret_cast<const C*>(a.pair) + k);
      f[0] = w.x;
      f[1] = w.y;
    }
    C Vk, Vp;
    if constexpr (MIR) {
      const C d = mk<C>(f[2], f[3]);
      Vk = cmulc(mk<C>(q[r][0], -q[r][1]), d);              // conj(d_k) (C_k - i C_{N-k})
      const C g = cmul(mk<C>(q[r][2], -q[r][3]), d);        // conj(d_{L-k}) = e^{i pi/4} d_k
      Vp = mk<C>(h * (g.x - g.y), h * (g.x + g.y));
    } else {
      Vk = mk<C>(q[r][0], q[r][1]);
      Vp = mk<C>(q[r][2], q[r][3]);
    }
    // E = (V_k + conj V_{L-k}) / 2, O = (V_k - conj V_{L-k}) conj(tw_k) / 2:
    // z_k = E + i O, z_{L-k} = conj(E) + i conj(O)
    const C E = mk<C>((R)0.5 * (Vk.x + Vp.x), (R)0.5 * (Vk.y - Vp.y));
    const C O = cmulc(mk<C>((R)0.5 * (Vk.x - Vp.x), (R)0.5 * (Vk.y + Vp.y)), mk<C>(f[0], f[1]));
    v[r] = mk<C>(E.x - O.y, E.y + O.x);
    up[r] = mk<C>(E.x + O.y, O.x - E.y);
    if (r == 0 && t == 0) {
      const R r2 = MIR ? (R)1.41421356237309504880 : (R)1;
      const R x0 = q[0][0], xl = r2 * q[0][1];
      v[0] = mk<C>((R)0.5 * (x0 + xl), (R)0.5 * (x0 - xl));
      if constexpr (MIR) {
        const C c8 = mk<C>((R)0.92387953251128675613, (R)-0.38268343236508977173);
        const C g = cmulc(mk<C>(q[0][2], -q[0][3]), c8);
        up[0] = mk<C>(g.x, -g.y);
      } else {
        up[0] = mk<C>(q[0][2], -q[0][3]);
      }
    }
  }
  mirror_exchange<R, NX, L, false>(up, ln, ph);
#pragma unroll
  for (int r = 0; r < 4; ++r) v[7 - r] = up[r];
  fft_pass<R, NX, 1, true>(v, ln, a.tw, ph);
  if constexpr (MIR) {
#pragma unroll
    for (int r = 0; r < 4; ++r) up[r] = v[7 - r];
    mirror_exchange<R, NX, L - 1, true>(up, ln, ph);  // up[r] = z[L - 1 - m], m = t + T r
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      p[2 * r] = mk<C>(v[r].x, up[r].y);
      p[2 * r + 1] = mk<C>(v[r].y, up[r].x);
    }
  } else {
#pragma unroll
    for (int r = 0; r < 8; ++r) p[r] = v[r];
  }
}

// boundary terms of R = B - B_bar: (L_bc - L_prec) for one missing or extra edge
template <int KIND>
__device__ __forceinline__ bool edge_terms(int bc) {
  return KIND == GMRF_PREC_CIRCULANT ? bc != GMRF_BC_PERIODIC : bc != GMRF_BC_NEUMANN;
}
template <int KIND, typename R>
__device__ __forceinline__ R edge_val(int bc, R wi, R wp) {
  const R b = bc == GMRF_BC_PERIODIC ? (wi - wp) : (bc == GMRF_BC_DIRICHLET ? wi : (R)0);
  const R pr = KIND == GMRF_PREC_CIRCULANT ? (wi - wp) : (R)0;
  return b - pr;
}

__device__ __forceinline__ void dot_add(Dots<float>& d, float v, float q) { d.add_dot2(v, q); }
__device__ __forceinline__ void dot_add(Dots<double>& d, double v, double q) { d.add(v, q); }

template <typename R, int KIND, int NX, int MODE>
__global__ void __launch_bounds__(block_threads(NX)) k_line_row(Args<R> a) {
  typedef typename C2<R>::T C;
  constexpr int T = line_threads(NX), RB = block_rows(NX);
  extern __shared__ __align__(16) unsigned char smraw[];
  __shared__ Dots<R> red[MODE == L_LAST ? block_threads(NX) / 32 : 1];
  __shared__ int s_int[4];
  __shared__ float s_flt[4];
  __shared__ R s_edge[MODE == L_MIDG ? RB : 1][2];
  after_previous();
  let_next();
  const int s = blockIdx.y;
  const bool step = a.in == nullptr;
  Line<R, NX> ln;
  ln.t = threadIdx.x % T;
  ln.id = threadIdx.x / T;
  ln.b = reinterpret_cast<C*>(smraw) + ln.id * 2 * slot_of(NX / 2);
  const int t = ln.t;
  int ph = 0;
  const bool live = blockIdx.x * RB + ln.id < a.ny;  // short grids of narrow rows: the block's last rows may be none
  const int y = live ? blockIdx.x * RB + ln.id : a.ny - 1;
  const size_t n = a.n, ro = (size_t)y * NX;
  R* S = a.T + (size_t)s * a.tstride + ro;
  const size_t slot = (size_t)s * a.P.nslots;
  C p[8], pa[8], pb[8], pc[8];
  // what does not depend on the step index is loaded ahead of the state
  R q[4][4];
  if constexpr (MODE != L_FWD && MODE != L_MIDG) load_spectrum<R, NX>(q, S, t);
  // FP32: so is what the elementwise part reads after the inverse transform
  // (FP64 has no registers to spare)
  constexpr bool PF = sizeof(R) == 4;
  if constexpr (PF && MODE == L_MID) load_kap<R, KIND, T>(a, ro, pa, t);
  if constexpr (PF && MODE == L_LAST)
    if (a.form == FORM_CTC) load_row<R, KIND, T>(pa, a.G + (size_t)s * n + ro, t);
  int j = 0;
  if (step) {
    if (a.st[s].status != VS_RUNNING) return;
    j = a.st[s].m;
  }

  if constexpr (MODE == L_FWD) {
    if (!step) {
      const R* src = a.in + (size_t)s * n + ro;
      if (a.in_elem) load_row_elem<R, KIND, T>(p, src, t);
      else load_row<R, KIND, T>(p, src, t);
    } else {
      load_row<R, KIND, T>(p, ((j & 1) ? a.W1 : a.W0) + (size_t)s * n + ro, t);
      const R inv_b = (R)a.st[s].vscale;
      if (j > 0) {
        C o[8];
        load_row<R, KIND, T>(o, a.V + (slot + (size_t)((j - 1) % a.P.nslots)) * n + ro, t);
        const R coef = (R)a.alpha[(size_t)s * a.P.m_max + (j - 1)];
#pragma unroll
        for (int r = 0; r < 8; ++r)
          p[r] = mk<C>((p[r].x - coef * o[r].x) * inv_b, (p[r].y - coef * o[r].y) * inv_b);
      } else {
#pragma unroll
        for (int r = 0; r < 8; ++r) p[r] = mk<C>(p[r].x * inv_b, p[r].y * inv_b);
      }
      if (live) {
        store_row<R, KIND, T>(p, a.V + (slot + (size_t)(j % a.P.nslots)) * n + ro, t);
        if (a.P.vb) store_row_bf16<R, KIND, T>(p, vb_at(a.P, s, j, n, ro), t);
      }
    }
    row_forward<R, KIND, NX>(a, p, S, ln, ph, live);
    return;
  }

  const R* vsrc = step ? a.V + (slot + (size_t)(j % a.P.nslots)) * n : a.in + (size_t)s * n;
  auto load_mid = [&]() {
    if (!PF) load_kap<R, KIND, T>(a, ro, pa, t);
    if (a.form == FORM_CTC) load_row<R, KIND, T>(pb, vsrc + ro, t);
  };
  auto load_last = [&]() {
    if (a.form != FORM_CTC) load_row<R, KIND, T>(pa, vsrc + ro, t);
    else if (!PF) load_row<R, KIND, T>(pa, a.G + (size_t)s * n + ro, t);
    if (step) {
      load_row<R, KIND, T>(pb, vsrc + ro, t);
      if (j > 0) load_row<R, KIND, T>(pc, a.V + (slot + (size_t)((j - 1) % a.P.nslots)) * n + ro, t);
    }
  };
  if constexpr (PF && MODE == L_MID) load_mid();
  if constexpr (PF && MODE == L_LAST) load_last();
  if constexpr (MODE == L_MIDG) load_row<R, KIND, T>(p, a.Wg + (size_t)s * n + ro, t);
  else row_inverse<R, KIND, NX>(a, p, q, ln, ph);
  if constexpr (MODE == L_INV) {
#pragma unroll
    for (int r = 0; r < 8; ++r) p[r] = mk<C>(p[r].x * a.scale, p[r].y * a.scale);
    if (live) {
      R* dst = a.out + (size_t)s * n + ro;
      if (a.out_elem) store_row_elem<R, KIND, T>(p, dst, t);
      else store_row<R, KIND, T>(p, dst, t);
    }
    return;
  }
  if constexpr (MODE == L_MIDW) {
    if (live) store_row<R, KIND, T>(p, a.Wg + (size_t)s * n + ro, t);
    return;
  }
  if constexpr (MODE == L_MID) {
    // p = w = B_bar^{-1} v (matched boundaries: R is diagonal): g = v + R w, then R g; or R w
    if constexpr (!PF) load_mid();
#pragma unroll
    for (int r = 0; r < 8; ++r) p[r] = mk<C>((pa[r].x - a.roff) * p[r].x, (pa[r].y - a.roff) * p[r].y);
    if (a.form == FORM_CTC) {
#pragma unroll
      for (int r = 0; r < 8; ++r) p[r] = cadd(pb[r], p[r]);
      if (live) store_row<R, KIND, T>(p, a.G + (size_t)s * n + ro, t);
#pragma unroll
      for (int r = 0; r < 8; ++r) p[r] = mk<C>((pa[r].x - a.roff) * p[r].x, (pa[r].y - a.roff) * p[r].y);
    }
    row_forward<R, KIND, NX>(a, p, S, ln, ph, live);
    return;
  }
  if constexpr (MODE == L_MIDG) {
    // the same with the boundary terms of R, whose y-partners are rows of other
    // blocks: w comes from the global buffer L_MIDW wrote
    const R* wg = a.Wg + (size_t)s * n;
    const bool hy = y == 0 || y == a.ny - 1;
    const size_t rp = (size_t)(y == 0 ? a.ny - 1 : 0) * NX;
    auto kap = [&](size_t o) -> R { return a.kappa2 ? (R)__ldg(a.kappa2 + o) : a.kappa2_const; };
    // (R w) at column x of row r0 (opposite boundary row r1)
    auto Rw = [&](size_t r0, size_t r1, int x, R wi) -> R {
      R e = (kap(r0 + x) - a.roff) * wi;
      if (x == 0) e += edge_val<KIND, R>(a.bc, wi, wg[r0 + NX - 1]);
      if (x == NX - 1) e += edge_val<KIND, R>(a.bc, wi, wg[r0]);
      if (hy) e += edge_val<KIND, R>(a.bc, wi, wg[r1 + x]);
      return e;
    };
    C w[8];
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      const int x = pair_at<KIND, T>(t, r);
      w[r] = mk<C>(Rw(ro, rp, x, p[r].x), Rw(ro, rp, x + 1, p[r].y));
    }
    if (a.form == FORM_CTC) {
      C gp[8];  // g of the opposite boundary row
#pragma unroll
      for (int r = 0; r < 8; ++r) gp[r] = mk<C>((R)0, (R)0);
      if (hy) {
#pragma unroll
        for (int r = 0; r < 8; ++r) {
          const int x = pair_at<KIND, T>(t, r);
          gp[r] = mk<C>(vsrc[rp + x] + Rw(rp, ro, x, wg[rp + x]), vsrc[rp + x + 1] + Rw(rp, ro, x + 1, wg[rp + x + 1]));
        }
      }
#pragma unroll
      for (int r = 0; r < 8; ++r) {
        const int x = pair_at<KIND, T>(t, r);
        const C vv = ldpair(vsrc + ro + x);
        w[r] = cadd(vv, w[r]);
      }
      if (live) store_row<R, KIND, T>(w, a.G + (size_t)s * n + ro, t);
      if (t == 0) s_edge[ln.id][0] = w[0].x;
      if (t == T - 1) s_edge[ln.id][1] = w[7].y;
      ln.sync();
      const R gf = s_edge[ln.id][0], gl = s_edge[ln.id][1];
#pragma unroll
      for (int r = 0; r < 8; ++r) {
        const int x = pair_at<KIND, T>(t, r);
        C e = mk<C>((kap(ro + x) - a.roff) * w[r].x, (kap(ro + x + 1) - a.roff) * w[r].y);
        if (x == 0) e.x += edge_val<KIND, R>(a.bc, w[r].x, gl);
        if (x + 1 == NX - 1) e.y += edge_val<KIND, R>(a.bc, w[r].y, gf);
        if (hy) {
          e.x += edge_val<KIND, R>(a.bc, w[r].x, gp[r].x);
          e.y += edge_val<KIND, R>(a.bc, w[r].y, gp[r].y);
        }
        w[r] = e;
      }
    }
    row_forward<R, KIND, NX>(a, w, S, ln, ph, live);
    return;
  }
  if constexpr (MODE == L_LAST) {
    // A v = g + h
    if constexpr (!PF) load_last();
#pragma unroll
    for (int r = 0; r < 8; ++r) p[r] = cadd(pa[r], p[r]);
    if (!step) {
      if (live) store_row<R, KIND, T>(p, a.out + (size_t)s * n + ro, t);
      return;
    }
    if (j > 0) {
      const R bprev = (R)a.beta[(size_t)s * a.P.m_max + (j - 1)];
#pragma unroll
      for (int r = 0; r < 8; ++r) p[r] = mk<C>(p[r].x - bprev * pc[r].x, p[r].y - bprev * pc[r].y);
    }
    Dots<R> d;
    d.zero();
    if (live) {
#pragma unroll
      for (int r = 0; r < 8; ++r) {
        dot_add(d, pb[r].x, p[r].x);
        dot_add(d, pb[r].y, p[r].y);
      }
    }
    d = block_sum(d, red);
    const int nblk = gridDim.x;
    const unsigned ticket = publish(d, a.partials, a.counters, s, blockIdx.x, nblk);
    if (live) store_row<R, KIND, T>(p, ((j & 1) ? a.W0 : a.W1) + (size_t)s * n + ro, t);
    if (publish_wait(ticket, a.counters, s, nblk, &s_int[3]))
      finish_step<R>(a.P, j, s, a.partials, nblk, a.st, a.alpha, a.beta, a.alpha_f, a.beta2_f, red, s_int, s_flt);
  }
}

// ------------------------------------------------------------ columns
__device__ __forceinline__ float fnma(float a, float b, float c) { return __fmaf_rn(-a, b, c); }
__device__ __forceinline__ double fnma(double a, double b, double c) { return __fma_rn(-a, b, c); }

// w = B_bar^{-1} along y on every column of the spectrum, in place.  A thread
// holds RY rows of VW = 16 bytes of columns (one chunk); chunk sums go to shared
// memory, SEG consecutive ones are summed by one lane, lanes by a shuffle scan
// weighted with powers of rho, and the second sweep over the thread's rows
// starts from the values that enter its chunk.
template <typename R, bool PER, int RY, int SEG>
__global__ void __launch_bounds__(512) k_line_col(Args<R> a, int nch, int cx, int step_mode) {
  constexpr int VW = 16 / (int)sizeof(R);
  extern __shared__ __align__(16) unsigned char smraw[];
  after_previous();
  let_next();
  const int s = blockIdx.y;
  if (step_mode && a.st[s].status != VS_RUNNING) return;
  const int ls = nch / SEG;  // scan lanes per column and direction, a power of two <= 32
  const int cols = cx * VW, pitch = ls * (SEG + 1) + 1;
  R* sF = reinterpret_cast<R*>(smraw);
  R* sB = sF + cols * pitch;
  R* sT = sB + cols * pitch;  // [cols][2] sums over the whole column
  const int tid = threadIdx.x, c = tid % cx, ch = tid / cx;
  const int col0 = blockIdx.x * cols + c * VW;
  const size_t nx = (size_t)a.nx;
  R* Tv = a.T + (size_t)s * a.tstride + (size_t)ch * RY * nx + col0;
  R x[RY][VW], y[RY][VW], delta[VW], gain[VW];
#pragma unroll
  for (int i = 0; i < RY; ++i) {
    if constexpr (VW == 4) {
      const float4 q = *reinterpret_cast<const float4*>(Tv + i * nx);
      x[i][0] = q.x; x[i][1] = q.y; x[i][2 % VW] = q.z; x[i][3 % VW] = q.w;
    } else {
      const double2 q = *reinterpret_cast<const double2*>(Tv + i * nx);
      x[i][0] = q.x; x[i][1] = q.y;
    }
  }
#pragma unroll
  for (int e = 0; e < VW; ++e) {
    delta[e] = __ldg(&a.col[col0 + e].delta);
    gain[e] = __ldg(&a.col[col0 + e].gain);
  }
  const int pf = ch + ch / SEG, pb = (nch - 1 - ch) + (nch - 1 - ch) / SEG;
#pragma unroll
  for (int e = 0; e < VW; ++e) {
    R f = x[0][e], b = x[RY - 1][e];
#pragma unroll
    for (int i = 1; i < RY; ++i) {
      f = fnma(delta[e], f, f) + x[i][e];
      b = fnma(delta[e], b, b) + x[RY - 1 - i][e];
    }
    sF[(c * VW + e) * pitch + pf] = f;
    sB[(c * VW + e) * pitch + pb] = b;
  }
  __syncthreads();
  // one lane per SEG chunks of a column and direction (the right-to-left
  // direction is stored reversed, so both run the same way)
  const int total = 2 * cols * ls;
  const int l = tid & (ls - 1);
  R excl = (R)0;
  for (int id = tid; id < total || ls > 1; id += blockDim.x) {
    const bool on = id < total;
    const int cd = on ? id / ls : 0, cc = cd >> 1;
    const R* base = ((cd & 1) ? sB : sF) + cc * pitch + l * (SEG + 1);
    const ColCoef<R>* k = a.col + blockIdx.x * cols + cc;
    const R dch = __ldg(&k->dchunk);
    R acc = base[0];
#pragma unroll
    for (int i = 1; i < SEG; ++i) acc = fnma(dch, acc, acc) + base[i];
    if (ls > 1) {
      R m = __ldg(&k->pseg);
      for (int off = 1; off < ls; off <<= 1) {
        const R u = __shfl_up_sync(0xffffffffu, acc, off, ls);
        if (l >= off) acc += m * u;
        m *= m;
      }
      const R u = __shfl_up_sync(0xffffffffu, acc, 1, ls);
      excl = l > 0 ? u : (R)0;
    }
    if (on && l == ls - 1) sT[cc * 2 + (cd & 1)] = acc;
    if (ls > 1) break;  // every lane has one item
  }
  __syncthreads();
  for (int id = tid; id < total; id += blockDim.x) {
    const int cd = id / ls, cc = cd >> 1, dir = cd & 1;
    R* base = (dir ? sB : sF) + cc * pitch + l * (SEG + 1);
    const ColCoef<R>* k = a.col + blockIdx.x * cols + cc;
    const R dch = __ldg(&k->dchunk), close = __ldg(&k->close);
    const R own = sT[cc * 2 + dir], oth = sT[cc * 2 + (dir ^ 1)];
    // what enters the column's first chunk: the wrapped or the reflected sequence
    R cin = PER ? own * close : (oth + __ldg(&k->pn) * own) * close;
    R m = __ldg(&k->pseg);
    for (int q = l; q; q >>= 1) {
      if (q & 1) cin *= m;
      m *= m;
    }
    R e = excl + cin;
#pragma unroll
    for (int i = 0; i < SEG; ++i) {
      const R u = base[i];
      base[i] = e;
      e = fnma(dch, e, e) + u;
    }
  }
  __syncthreads();
#pragma unroll
  for (int e = 0; e < VW; ++e) {
    R f = sF[(c * VW + e) * pitch + pf], b = sB[(c * VW + e) * pitch + pb];
#pragma unroll
    for (int i = 0; i < RY; ++i) {
      y[i][e] = fnma(delta[e], f, f);
      f = y[i][e] + x[i][e];
    }
#pragma unroll
    for (int i = RY - 1; i >= 0; --i) {
      b = fnma(delta[e], b, b) + x[i][e];
      y[i][e] = gain[e] * (y[i][e] + b);
    }
  }
#pragma unroll
  for (int i = 0; i < RY; ++i) {
    if constexpr (VW == 4)
      *reinterpret_cast<float4*>(Tv + i * nx) = make_float4(y[i][0], y[i][1], y[i][2 % VW], y[i][3 % VW]);
    else *reinterpret_cast<double2*>(Tv + i * nx) = make_double2(y[i][0], y[i][1]);
  }
}

// ------------------------------------------------------------ launchers
#define LINE_CK(x)                     \
  do {                                 \
    cudaError_t e_ = (x);              \
    if (e_ != cudaSuccess) return e_;  \
  } while (0)

// Launch, with the programmatic dependency on the stream's previous kernel where
// `early`: plain applies, which are launched one by one (M^{-1/2} v at 128 x 128
// 28.3 -> 24.4 us a call).  In the step graphs such edges cost more than they hide
// (1024 x 1024 sample 3.31 -> 3.76 ms, FP64 proposal at 512 x 512 1.79 -> 2.30 ms).
template <typename... A, typename... V>
cudaError_t launch_after(bool early, void (*k)(A...), dim3 grd, int threads, size_t sm, cudaStream_t s, V&&... v) {
  cudaLaunchConfig_t c = {};
  c.gridDim = grd;
  c.blockDim = dim3(threads);
  c.dynamicSmemBytes = sm;
  c.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  c.attrs = at;
  c.numAttrs = early ? 1 : 0;
  return cudaLaunchKernelEx(&c, k, std::forward<V>(v)...);
}

template <typename R, int KIND, int NX, int MODE>
cudaError_t row_launch_t(const Args<R>& a, int nvec, cudaStream_t s, int kc) {
  constexpr size_t sm = row_smem<R, NX>();
  if constexpr (sm > 40 * 1024) {
    static PerDevice attr;
    LINE_CK(set_attribute(attr, k_line_row<R, KIND, NX, MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
  }
  dim3 grd((a.ny + block_rows(NX) - 1) / block_rows(NX), nvec);
  trace_begin(kc, s);
  const cudaError_t e = launch_after(a.in != nullptr, k_line_row<R, KIND, NX, MODE>, grd, block_threads(NX), sm, s, a);
  trace_end(kc, s);
  return e;
}

template <typename R, int KIND, int MODE>
cudaError_t row_launch(const Args<R>& a, int nvec, cudaStream_t s, int kc) {
  switch (a.nx) {
    case 64: return row_launch_t<R, KIND, 64, MODE>(a, nvec, s, kc);
    case 128: return row_launch_t<R, KIND, 128, MODE>(a, nvec, s, kc);
    case 256: return row_launch_t<R, KIND, 256, MODE>(a, nvec, s, kc);
    case 512: return row_launch_t<R, KIND, 512, MODE>(a, nvec, s, kc);
    case 1024: return row_launch_t<R, KIND, 1024, MODE>(a, nvec, s, kc);
    case 2048: return row_launch_t<R, KIND, 2048, MODE>(a, nvec, s, kc);
    case 4096: return row_launch_t<R, KIND, 4096, MODE>(a, nvec, s, kc);
    default: return cudaErrorInvalidValue;
  }
}

template <typename R, bool PER, int RY, int SEG>
cudaError_t col_launch_t(const Args<R>& a, int nvec, int step_mode, cudaStream_t s, int kc) {
  constexpr int VW = 16 / (int)sizeof(R);
  const int nch = a.ny / RY, tc = a.nx / VW;
  // thread columns of a block: 32 bytes of a row at least (a whole sector), more
  // while that leaves a block of at most 256 threads and enough blocks
  int cx = 32 / 16;
  while (2 * cx * nch <= 256 && 2 * cx <= tc && (int64_t)(tc / (2 * cx)) * nvec >= 2 * 152) cx *= 2;
  while (cx * nch < 32 && 2 * cx <= tc) cx *= 2;
  const int ls = nch / SEG, cols = cx * VW;
  const size_t sm = ((size_t)2 * cols * (ls * (SEG + 1) + 1) + 2 * cols) * sizeof(R);
  dim3 grd(tc / cx, nvec);
  trace_begin(kc, s);
  const cudaError_t e = launch_after(!step_mode, k_line_col<R, PER, RY, SEG>, grd, cx * nch, sm, s, a, nch, cx,
                                     step_mode);
  trace_end(kc, s);
  return e;
}

// Rows per chunk and chunks per scan lane depend on ny alone (col_plan).
template <typename R, int KIND>
cudaError_t col_launch(const Args<R>& a, int nvec, int step_mode, cudaStream_t s, int kc) {
  constexpr bool PER = KIND == GMRF_PREC_CIRCULANT;
  switch (a.ny) {
    case 8: return col_launch_t<R, PER, 8, 1>(a, nvec, step_mode, s, kc);
    case 16: return col_launch_t<R, PER, 8, 2>(a, nvec, step_mode, s, kc);
    case 32: return col_launch_t<R, PER, 8, 4>(a, nvec, step_mode, s, kc);
    case 64:
    case 128:
    case 256:
    case 512:
    case 1024: return col_launch_t<R, PER, 8, 8>(a, nvec, step_mode, s, kc);
    case 2048: return col_launch_t<R, PER, 8, 16>(a, nvec, step_mode, s, kc);
    case 4096: return col_launch_t<R, PER, 16, 16>(a, nvec, step_mode, s, kc);
    default: return cudaErrorInvalidValue;
  }
}

inline bool host_edge_terms(int kind, int bc) {
  return kind == GMRF_PREC_CIRCULANT ? bc != GMRF_BC_PERIODIC : bc != GMRF_BC_NEUMANN;
}

// row-forward, columns, the middle rows, columns: everything of A before the last rows
template <typename R, int KIND>
cudaError_t first_passes(const Args<R>& a, int nvec, int step_mode, cudaStream_t s, bool apply) {
  LINE_CK((row_launch<R, KIND, L_FWD>(a, nvec, s, apply ? KC_PRE_APPLY : KC_PRE_ROW_FWD)));
  LINE_CK((col_launch<R, KIND>(a, nvec, step_mode, s, apply ? KC_PRE_APPLY : KC_PRE_COL)));
  const int km = apply ? KC_PRE_APPLY : KC_PRE_ROW_MID;
  if (host_edge_terms(KIND, a.bc)) {
    LINE_CK((row_launch<R, KIND, L_MIDW>(a, nvec, s, km)));
    LINE_CK((row_launch<R, KIND, L_MIDG>(a, nvec, s, km)));
  } else {
    LINE_CK((row_launch<R, KIND, L_MID>(a, nvec, s, km)));
  }
  return col_launch<R, KIND>(a, nvec, step_mode, s, apply ? KC_PRE_APPLY : KC_PRE_COL);
}

// one preconditioned Lanczos step
template <typename R, int KIND>
cudaError_t step_k(const Args<R>& a, int nvec, cudaStream_t s) {
  LINE_CK((first_passes<R, KIND>(a, nvec, 1, s, false)));
  return row_launch<R, KIND, L_LAST>(a, nvec, s, KC_PRE_ROW_LAST);
}

// out = scale B_bar^{-1} in; in and out are the caller's own arrays and may lie at any element
template <typename R, int KIND>
cudaError_t apply_k(Args<R> a, int nvec, cudaStream_t s) {
  a.in_elem = !row_aligned(KIND, sizeof(R), a.in);
  a.out_elem = !row_aligned(KIND, sizeof(R), a.out);
  LINE_CK((row_launch<R, KIND, L_FWD>(a, nvec, s, KC_PRE_APPLY)));
  LINE_CK((col_launch<R, KIND>(a, nvec, 0, s, KC_PRE_APPLY)));
  return row_launch<R, KIND, L_INV>(a, nvec, s, KC_PRE_APPLY);
}

// out = A in; in and out aligned for whole vectors (row_aligned)
template <typename R, int KIND>
cudaError_t operator_k(const Args<R>& a, int nvec, cudaStream_t s) {
  if (!row_aligned(KIND, sizeof(R), a.in) || !row_aligned(KIND, sizeof(R), a.out)) return cudaErrorMisalignedAddress;
  LINE_CK((first_passes<R, KIND>(a, nvec, 0, s, true)));
  return row_launch<R, KIND, L_LAST>(a, nvec, s, KC_PRE_APPLY);
}

}  // namespace line
}  // namespace gmrf
