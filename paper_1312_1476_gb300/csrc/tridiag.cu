// tridiag.cu -- functions of the small Lanczos matrix T_m, in FP64.
//
// Sample (Algorithm 1, last step): y = T_m^{-1/2} e_1.  The algorithm's
// caption notes that the square root of T_m may be replaced by a rational
// approximation; this library uses one.  From
//   t^{-1/2} = (2/pi) int_0^inf ds / (t + s^2) = (2/pi) int_R e^u / (t + e^{2u}) du,
// whose integrand is sech(u - log(t)/2) / (2 sqrt t), the trapezoid rule with
// step h on [u_lo, u_hi] gives
//   T^{-1/2} e_1 ~= sum_k (2h/pi) e^{u_k} (T + e^{2u_k} I)^{-1} e_1,
// a sum of shifted SPD tridiagonal solves (trailing_dets, one pole per
// thread).  Discretisation error ~ 4 exp(-pi^2 / h) and truncation error
// ~ (2/pi) exp(-pad) relative, with the window covering
// [log(theta_min)/2 - pad, log(theta_max)/2 + pad]; theta_min comes from the
// Sturm multisection of the stopping rule, theta_max from Gershgorin.
//
// Log det (Section 6, Gauss quadrature e_1^T log(T_m) e_1): from
//   log t = int_0^inf (1/(1+s) - 1/(t+s)) ds = int_R (e^u/(1+e^u) - e^u/(t+e^u)) du
// the trapezoid rule gives
//   e_1^T log(T) e_1 ~= sum_k h e^{u_k} (1/(1+e^{u_k}) - [(T + e^{u_k} I)^{-1}]_{11}),
// with [(T + sI)^{-1}]_{11} the ratio of the two largest trailing determinants.  Error ~ exp(-2 pi^2 / h).
#include <cuda_runtime.h>
#include <math.h>

#include <cmath>

#include "internal.h"

namespace gmrf {
namespace {

constexpr double kPi = 3.14159265358979323846;

struct DMax {
  double v;
  __device__ void zero() { v = 0.0; }
  __device__ void merge(const DMax& o) { v = fmax(v, o.v); }
  __device__ DMax shfl_down(int off) const { return {__shfl_down_sync(0xffffffffu, v, off)}; }
};
struct DSum {
  double v;
  __device__ void zero() { v = 0.0; }
  __device__ void merge(const DSum& o) { v += o.v; }
  __device__ DSum shfl_down(int off) const { return {__shfl_down_sync(0xffffffffu, v, off)}; }
};

__device__ __forceinline__ bool usable(const VecState& v) {
  return (v.status == VS_DONE || v.status == GMRF_ERR_NOT_CONVERGED) && v.m >= 1;
}

// Node window per vector.  kind 0: inverse square root; kind 1: log.
struct NodeRule {
  double h, pad;  // node spacing and what the window exceeds the spectrum by
};
// eps: the trapezoid rule's target accuracy
NodeRule node_rule(int kind, bool fp64) {
  const double eps = kind == 0 ? (fp64 ? 1e-15 : 1e-11) : (fp64 ? 1e-16 : 1e-12);
  if (kind == 0) return {kPi * kPi / std::log(4.0 / eps), std::log(2.0 / (kPi * eps))};
  return {2.0 * kPi * kPi / std::log(1.0 / eps), std::log(1.0 / eps) + 2.0};
}
__global__ void k_nodes(const VecState* st, const double* alpha, const double* beta, int m_max, int kind, NodeRule nd,
                        TmNodes* nodes) {
  __shared__ DMax red[8];
  const int s = blockIdx.x;
  const VecState v = st[s];
  TmNodes out = {0.0, 1.0, 0, 0};
  if (!usable(v)) {
    if (threadIdx.x == 0) nodes[s] = out;
    return;
  }
  const int m = v.m;
  const double* a = alpha + (size_t)s * m_max;
  const double* b = beta + (size_t)s * m_max;
  DMax g;
  g.zero();
  for (int i = threadIdx.x; i < m; i += blockDim.x) {
    double r = a[i];
    if (i > 0) r += fabs(b[i - 1]);
    if (i < m - 1) r += fabs(b[i]);
    g.v = fmax(g.v, r);
  }
  g = block_reduce(g, red);
  if (threadIdx.x < 2) {
    // the two logarithms side by side: an FP64 logarithm is a chain of some microseconds
    const double tmax = 2.0 * __shfl_sync(3u, g.v, 0);
    const double tmin = 0.5 * v.theta;
    const double lg = log(threadIdx.x == 0 ? tmin : tmax);
    const double lgmax = __shfl_sync(3u, lg, 1);
    if (threadIdx.x > 0) return;
    double h = nd.h, lo, hi;
    const double half = kind == 0 ? 0.5 : 1.0;
    lo = half * lg - nd.pad;
    hi = half * lgmax + nd.pad;
    if (!(tmin > 0.0) || !(tmax > 0.0) || !isfinite(lo) || !isfinite(hi)) {
      nodes[s] = out;  // L = 0: no usable window (reported through the vector's status)
      return;
    }
    int L = (int)ceil((hi - lo) / h) + 1;
    if (L > kMaxNodes) {
      L = kMaxNodes;
      h = (hi - lo) / (L - 1);
    }
    out.s_lo = lo;
    out.h = h;
    out.L = L;
    nodes[s] = out;
  }
}

// (T + sigma I)^{-1} e_1 by the determinants phi_i of the trailing blocks,
//   phi_m = 1, phi_i = (a_i + sigma) phi_{i+1} - b_i^2 phi_{i+2},
//   x_i = (-1)^i b_0 .. b_{i-1} phi_{i+1} / phi_0
// (the closed form of a tridiagonal inverse's first column).  phi_i / phi_{i+1} is
// the pivot of the backward LDL^T, so rounding acts as there (a relative
// perturbation of a_i and b_i), but the recurrence holds no division: one
// dependent FMA per row (64 cycles) where a pivot costs a division (580) and two
// more operations.  phi is kept as a mantissa and an exponent, rescaled by a power
// of two (exactly) when it leaves 2^+-128.  With the two logarithms of the window
// side by side and T_m^{-1} e_1 as one more pole: FP64 64 x 64 sample (102 rows) 133 ->
// 77 us for the three kernels, 1157 -> 1074 us a call.  Error against 80-bit sums as
// before (condition 1e6, 300 rows: 3.5e-13, LDL^T 6.6e-13).
struct Scaled {
  double v;
  int e;  // value v 2^e
  // back into range: v in [1, 2), or 0
  __device__ __forceinline__ void norm() {
    const int hi = __double2hiint(v), ex = ((hi >> 20) & 0x7ff) - 1023;
    if (v == 0.0 || ex == 1024) return;
    v = __hiloint2double((hi & 0x800fffff) | (1023 << 20), __double2loint(v));
    e += ex;
  }
};
__device__ __forceinline__ double pow2(int e) {  // 2^e, 0 below the normal range
  return e < -1022 ? 0.0 : __hiloint2double((min(e, 1023) + 1023) << 20, 0);
}

// phi_{i+1} of row i = m - 1 .. 0 through put(i, phi); returns phi_0
template <typename Put>
__device__ __forceinline__ Scaled trailing_dets(const double* __restrict__ a, const double* __restrict__ b, int m,
                                                double sigma, Put&& put) {
  Scaled p = {1.0, 0};  // phi_{i+1}
  double q = 0.0;       // phi_{i+2}, same exponent
  for (int i = m - 1; i >= 0; --i) {
    put(i, p);
    const double bi = i < m - 1 ? b[i] : 0.0;
    const double next = fma(a[i] + sigma, p.v, -(bi * (bi * q)));
    q = p.v;
    p.v = next;
    const int ex = ((__double2hiint(next) >> 20) & 0x7ff) - 1023;
    if (abs(ex) > 128 && ex < 1024 && next != 0.0) {
      const double s = __hiloint2double((1023 - ex) << 20, 0);
      p.v *= s;
      q *= s;
      p.e += ex;
    }
  }
  return p;
}

// x_i (times w) from the stored phi_{i+1} (get) into set(i, x).
template <typename Get, typename Set>
__device__ __forceinline__ void first_column(const double* __restrict__ b, int m, double w, Scaled phi0, Get&& get,
                                             Set&& set) {
  phi0.norm();
  Scaled pi = {w / phi0.v, -phi0.e};  // w (-1)^i b_0 .. b_{i-1} / phi_0
  for (int i = 0; i < m; ++i) {
    const Scaled f = get(i);
    set(i, pi.v * f.v * pow2(pi.e + f.e));
    pi.v *= -b[i < m - 1 ? i : 0];
    pi.norm();
  }
}

// y = T_m^{-1} e_1, one thread; work [m] keeps the phi's, y their exponents until
// they are used
__device__ void inverse_e1(const double* __restrict__ a, const double* __restrict__ b, int m, double* work, double* y) {
  const Scaled phi0 = trailing_dets(a, b, m, 0.0, [&](int i, const Scaled& f) {
    work[i] = f.v;
    y[i] = (double)f.e;
  });
  first_column(b, m, 1.0, phi0, [&](int i) -> Scaled { return {work[i], (int)y[i]}; },
               [&](int i, double x) { y[i] = x; });
}

// One pole per thread: D[s][i][k] = w_k ((T + sigma_k I)^{-1} e_1)_i, the phi's
// exponents kept in C[s][i][k].  Layout k-fastest for coalescing.  Thread
// kMaxNodes: T^{-1} e_1 itself into ycg[s][i] (work: its phi's), the CG
// coefficients of the accuracy check.
__global__ void k_poles(const VecState* st, const double* alpha, const double* beta, int m_max, const TmNodes* nodes,
                        int* C, double* D, double* ycg, double* work) {
  const int s = blockIdx.y;
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  const VecState v = st[s];
  const TmNodes nd = nodes[s];
  if (!usable(v) || (k >= nd.L && (k != kMaxNodes || !ycg))) return;
  const int m = v.m;
  const double* a = alpha + (size_t)s * m_max;
  const double* b = beta + (size_t)s * m_max;
  if (k == kMaxNodes) {
    inverse_e1(a, b, m, work + (size_t)s * m_max, ycg + (size_t)s * m_max);
    return;
  }
  const double u = nd.s_lo + nd.h * k;
  const double eu = exp(u);
  const double sigma = eu * eu;  // e^{2u}, one exponential
  const double w = (2.0 * nd.h / kPi) * eu;
  const size_t base = (size_t)s * m_max * kMaxNodes + k;
  const Scaled phi0 = trailing_dets(a, b, m, sigma, [&](int i, const Scaled& f) {
    C[base + (size_t)i * kMaxNodes] = f.e;
    D[base + (size_t)i * kMaxNodes] = f.v;
  });
  first_column(b, m, w, phi0,
               [&](int i) -> Scaled {
                 return {D[base + (size_t)i * kMaxNodes], C[base + (size_t)i * kMaxNodes]};
               },
               [&](int i, double x) { D[base + (size_t)i * kMaxNodes] = x; });
}

// y[s][i] = sum_k D[s][i][k] in a fixed order; one warp per component i.
__global__ void k_pole_sum(const VecState* st, int m_max, const TmNodes* nodes, const double* D, double* y) {
  const int s = blockIdx.y;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int i = blockIdx.x * (blockDim.x >> 5) + warp;
  const VecState v = st[s];
  const TmNodes nd = nodes[s];
  if (i >= m_max) return;
  if (!usable(v) || i >= v.m) {
    if (lane == 0) y[(size_t)s * m_max + i] = 0.0;
    return;
  }
  const double* row = D + (size_t)s * m_max * kMaxNodes + (size_t)i * kMaxNodes;
  double acc = 0.0;
  for (int k = lane; k < nd.L; k += 32) acc += row[k];
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, off);
  if (lane == 0) y[(size_t)s * m_max + i] = acc;
}

// q[s] = ||v||^2 e_1^T log(T_m) e_1.
__global__ void k_log(const VecState* st, const double* alpha, const double* beta, int m_max, const TmNodes* nodes,
                      double* q) {
  __shared__ DSum red[8];
  const int s = blockIdx.x;
  const VecState v = st[s];
  const TmNodes nd = nodes[s];
  if (!usable(v)) {
    if (threadIdx.x == 0) q[s] = (v.status == VS_DONE) ? 0.0 : NAN;
    return;
  }
  const int m = v.m;
  const double* a = alpha + (size_t)s * m_max;
  const double* b = beta + (size_t)s * m_max;
  DSum acc;
  acc.zero();
  for (int k = threadIdx.x; k < nd.L; k += blockDim.x) {
    const double u = nd.s_lo + nd.h * k;
    const double t = exp(u);
    // [(T + t I)^{-1}]_{11} = phi_1 / phi_0
    Scaled phi1 = {1.0, 0};
    const Scaled phi0 = trailing_dets(a, b, m, t, [&](int, const Scaled& f) { phi1 = f; });
    acc.v += nd.h * t * (1.0 / (1.0 + t) - phi1.v / phi0.v * pow2(phi1.e - phi0.e));
  }
  acc = block_reduce(acc, red);
  if (threadIdx.x == 0) q[s] = v.znorm * v.znorm * acc.v;
}

// Estimate and standard error over ng = nq / group draws, draw d being the sum
// of q[d * group .. d * group + group - 1] (group > 1: the colour classes of
// the coloured estimator, Section 6.1).
__global__ void k_logdet_reduce(const double* q, int nq, int group, double shift, double* out) {
  __shared__ DSum red[8];
  const int ng = nq / group;
  DSum s1;
  s1.zero();
  for (int d = threadIdx.x; d < ng; d += blockDim.x) {
    double t = 0.0;
    for (int c = 0; c < group; ++c) t += q[(size_t)d * group + c];
    s1.v += t;
  }
  s1 = block_reduce(s1, red);
  __shared__ double mean;
  if (threadIdx.x == 0) mean = s1.v / ng;
  __syncthreads();
  DSum s2;
  s2.zero();
  for (int d = threadIdx.x; d < ng; d += blockDim.x) {
    double t = 0.0;
    for (int c = 0; c < group; ++c) t += q[(size_t)d * group + c];
    s2.v += (t - mean) * (t - mean);
  }
  s2 = block_reduce(s2, red);
  if (threadIdx.x == 0) {
    out[0] = mean + shift;
    out[1] = ng > 1 ? sqrt(s2.v / (ng - 1) / ng) : NAN;
  }
}

// y = T_m^{-1} e_1 (the CG coefficients of a linear solve).  One thread per vector.
__global__ void k_tm_inv(const VecState* st, const double* alpha, const double* beta, int m_max, int nvec,
                         double* dwork, double* y) {
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= nvec) return;
  const VecState v = st[s];
  if (!usable(v)) return;
  const size_t o = (size_t)s * m_max;
  inverse_e1(alpha + o, beta + o, v.m, dwork + o, y + o);
}

}  // namespace

cudaError_t launch_tm_inv(const LanczosBufs& b, double* dwork, double* y, cudaStream_t s) {
  k_tm_inv<<<(b.nvec + 31) / 32, 32, 0, s>>>(b.st, b.alpha, b.beta, b.m_max, b.nvec, dwork, y);
  return cudaGetLastError();
}

cudaError_t launch_tm_inv_sqrt(const LanczosBufs& b, bool fp64, TmNodes* nodes, double* scratch, double* y,
                               cudaStream_t s, double* ycg, double* work) {
  k_nodes<<<b.nvec, 256, 0, s>>>(b.st, b.alpha, b.beta, b.m_max, 0, node_rule(0, fp64), nodes);
  int* C = (int*)scratch;
  double* D = scratch + (size_t)b.nvec * b.m_max * kMaxNodes;
  dim3 g1((kMaxNodes + 1 + 63) / 64, b.nvec);
  k_poles<<<g1, 64, 0, s>>>(b.st, b.alpha, b.beta, b.m_max, nodes, C, D, ycg, work);
  dim3 g2((b.m_max + 7) / 8, b.nvec);
  k_pole_sum<<<g2, 256, 0, s>>>(b.st, b.m_max, nodes, D, y);
  return cudaGetLastError();
}

cudaError_t launch_tm_log(const LanczosBufs& b, bool fp64, TmNodes* nodes, double* q, cudaStream_t s) {
  k_nodes<<<b.nvec, 256, 0, s>>>(b.st, b.alpha, b.beta, b.m_max, 1, node_rule(1, fp64), nodes);
  k_log<<<b.nvec, 256, 0, s>>>(b.st, b.alpha, b.beta, b.m_max, nodes, q);
  return cudaGetLastError();
}

cudaError_t launch_logdet_reduce(const double* q, int nq, int group, double shift, double* out, cudaStream_t s) {
  k_logdet_reduce<<<1, 256, 0, s>>>(q, nq, group, shift, out);
  return cudaGetLastError();
}

}  // namespace gmrf
