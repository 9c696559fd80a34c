// stencil3d_flat.cu -- the fused 3-D Lanczos step of Algorithm 1 with the
// 7-point lattice apply of Q (Section 2) on planes taken as flat ranges of cells,
// for the grids the TMA-staged kernel does not take: any width up to 512,
// periodic boundaries, FP64, unaligned pointers.
//
// A block owns 512 (FP64 on small grids 256) consecutive cells of a plane, whatever rows they belong
// to, and marches over a chunk of z planes.  Odd widths cost nothing (no tile is
// partly empty but the plane's last one), and every access is in order of the
// cells.  The neighbours of a cell lie 1 and nx cells before and after it; where
// the grid ends its place is taken by another cell of the same stage: the
// wrapped one (x: nx - 1 cells further, within the halo; y: the halo is loaded
// from the wrapped row), the cell itself (Neumann: the term c - c is exactly 0), or a
// slot that holds 0 (Dirichlet).  These four places per cell do not change from
// plane to plane.
//
// Planes (the range and nx cells on either side) are copied by element
// (cp.async) into a ring of four stages, three planes ahead.  A thread forms v_j
// from the elements it copied as soon as they have landed, keeps v_j and v_{j-1}
// of its own cells in registers (the z neighbours among them) and writes v_j to
// the stage for the others: one barrier per plane, and q_j and v_j go out
// straight from registers.  The z chunk depends on the grid alone, so a vector's
// sums do not depend on its batch.
//
// Bound: instruction issue (61 x 75 x 90, 4 vectors: 59 % of the slots, 200 instructions per
// cell with the chunks' halo planes, barriers next; 18.7 us a step), on smaller grids the
// latency of the planes one after another.  Measured against the register kernel this
// replaces, whole sample calls to 1e-6: 61 x 75 x 90, 4 vectors, FP32 1208 -> 1028 us
// (periodic 1946 -> 940), FP64 4725 -> 3410; 128 x 128 x 130, one vector, FP32 5286 -> 1268
// (periodic 9781 -> 1200), FP64 35.5 -> 4.5 ms; 33 x 40 x 37, one vector, FP32 636 -> 585, FP64
// 1197 -> 790.
#include <cuda_runtime.h>

#include <algorithm>

#include "internal.h"
#include "per_device.h"
#include "stencil_args.h"

namespace gmrf {
namespace {

constexpr int FNT = 256;      // threads
constexpr int FSTAGES = 4;
constexpr int FH = 4;         // halo elements of a thread at most: 2 nx <= FH FNT

// elements of a stage's q and v_{j-1} ranges: the halo on either side and a 0
__host__ __device__ inline int flat_pitch(int cells, int nx) { return cells + 2 * nx + 1; }
// bytes of a stage: q (then v), v_{j-1}, kappa^2
template <typename T>
__host__ __device__ inline size_t flat_stage(int cells, int nx) {
  return ((size_t)2 * flat_pitch(cells, nx) * sizeof(T) + (size_t)cells * sizeof(float) + 15) / 16 * 16;
}

template <int BYTES>
__device__ __forceinline__ void copy_elem(unsigned dst, const void* src, bool valid) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;\n" ::"r"(dst), "l"(src), "n"(BYTES), "r"(valid ? BYTES : 0)
               : "memory");
}
template <int N>
__device__ __forceinline__ void copies_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory"); }
__device__ __forceinline__ void copies_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }

__device__ __forceinline__ float form_v(float w, float vp, float coef, float inv_b) {
  return __fmul_rn(__fmaf_rn(-coef, vp, w), inv_b);
}
__device__ __forceinline__ double form_v(double w, double vp, double coef, double inv_b) {
  return fma(-coef, vp, w) * inv_b;
}

// FE: cells of a thread
template <typename T, int BC, bool STEP, int FE>
__global__ void __launch_bounds__(FNT, 3) k_stencil3d_flat(StencilArgs<T> a, int nrange, int zper) {
  constexpr int FC = FNT * FE;  // cells of a block
  extern __shared__ __align__(16) unsigned char smraw[];
  __shared__ Dots<T> red[FNT / 32];
  __shared__ int s_int[4];
  __shared__ float s_flt[4];
  const int s = blockIdx.y, li = blockIdx.x;
  int j = 0;
  if (STEP) {
    if (a.st[s].status != VS_RUNNING) return;
    j = a.st[s].m;
  }
  const int tid = threadIdx.x;
  const int nx = a.nx, nz = a.nz, plane = a.nx * a.ny;
  const size_t n = a.n;
  const int i0 = (li % nrange) * FC, zc = li / nrange;
  const int z0 = zc * zper, z1 = min(nz, z0 + zper);
  const int P = z1 - z0 + 2;  // planes z0 - 1 .. z1 (every chunk holds a plane)
  const T* Win = (STEP ? ((j & 1) ? a.W1 : a.W0) : a.Win) + (size_t)s * n;
  T* Wout = (STEP ? ((j & 1) ? a.W0 : a.W1) : a.Wout) + (size_t)s * n;
  const T* Vp = nullptr;
  T* Vc = nullptr;
  T coef = 0, inv_b = 1, bprev = 0;
  if (STEP) {
    const size_t base = (size_t)s * a.P.nslots;
    Vc = a.V + (base + (size_t)(j % a.P.nslots)) * n;
    inv_b = (T)a.st[s].vscale;
    if (j > 0) {
      Vp = a.V + (base + (size_t)((j - 1) % a.P.nslots)) * n;
      const size_t mo = (size_t)s * a.P.m_max + (j - 1);
      coef = (T)a.alpha[mo];
      bprev = (T)a.beta[mo];
    }
  }
  const bool use_vp = STEP && j > 0, kfield = a.kappa2 != nullptr;
  const int pitch = flat_pitch(FC, nx), zero = pitch - 1;
  const size_t stage_bytes = flat_stage<T>(FC, nx);
  auto stage_q = [&](int t) { return reinterpret_cast<T*>(smraw + (size_t)(t % FSTAGES) * stage_bytes); };

  // own cell e is cell i0 + tid + FNT e of the plane, at place nx + tid + FNT e of a stage
  int l[FE], r[FE], u[FE], d[FE];  // places of its neighbours
  int nin = 0;                     // own cells inside the plane
#pragma unroll
  for (int e = 0; e < FE; ++e) {
    const int c = tid + FNT * e, i = i0 + c, p = nx + c;
    const int y = i / nx, x = i - y * nx;
    if (i < plane) nin = e + 1;
    const int gone = BC == GMRF_BC_NEUMANN ? p : zero;  // Dirichlet: 0
    l[e] = x > 0 ? p - 1 : (BC == GMRF_BC_PERIODIC ? p + nx - 1 : gone);
    r[e] = x < nx - 1 ? p + 1 : (BC == GMRF_BC_PERIODIC ? p - nx + 1 : gone);
    u[e] = BC == GMRF_BC_PERIODIC || y > 0 ? p - nx : gone;
    d[e] = BC == GMRF_BC_PERIODIC || y < a.ny - 1 ? p + nx : gone;
  }
  // halo elements: nx before the range, then nx after it; cell of the plane, or -1
  int hat[FH], hcell[FH];
#pragma unroll
  for (int h = 0; h < FH; ++h) {
    const int k = tid + FNT * h;
    hat[h] = k < nx ? k : FC + k;  // place in a stage
    int i = k < nx ? i0 - nx + k : i0 + FC + (k - nx);
    if (BC == GMRF_BC_PERIODIC) {
      // one row beyond the plane wraps; what lies further out is never read
      if (i < 0) i += plane;
      else if (i >= plane) i -= plane;
    }
    if (k >= 2 * nx) hat[h] = -1;
    hcell[h] = i >= 0 && i < plane ? i : -1;
  }
  // a range that ends with the plane: in a periodic grid the rows after its last
  // cells are the wrapped first ones, at their places among the own cells
  auto own_cell = [&](int e) -> int {
    const int i = i0 + tid + FNT * e;
    if (i < plane) return i;
    return BC == GMRF_BC_PERIODIC && i - plane < nx ? i - plane : -1;
  };
  if (tid < FSTAGES) stage_q(tid)[zero] = (T)0;

  const unsigned sm0 = (unsigned)__cvta_generic_to_shared(smraw);
  auto copy_plane = [&](int t) {
    if (t < P) {
      int gz = z0 - 1 + t;
      bool zin = gz >= 0 && gz < nz;
      if (!zin && BC == GMRF_BC_PERIODIC) {
        gz = gz < 0 ? gz + nz : gz - nz;
        zin = true;
      }
      const unsigned sq = sm0 + (unsigned)((t % FSTAGES) * stage_bytes), sv = sq + pitch * (unsigned)sizeof(T),
                     sk = sv + pitch * (unsigned)sizeof(T);
      const bool mid = t > 0 && t < P - 1;
      const size_t zo = (size_t)plane * (zin ? gz : 0);
#pragma unroll
      for (int e = 0; e < FE; ++e) {
        const int c = own_cell(e);
        const bool in = zin && c >= 0;
        const size_t i = zo + (in ? c : 0);
        const unsigned at = nx + tid + FNT * e;
        copy_elem<sizeof(T)>(sq + at * (unsigned)sizeof(T), Win + i, in);
        if (use_vp) copy_elem<sizeof(T)>(sv + at * (unsigned)sizeof(T), Vp + i, in);
        if (kfield && mid) copy_elem<4>(sk + (unsigned)(tid + FNT * e) * 4u, a.kappa2 + i, in);
      }
      if (mid) {
#pragma unroll
        for (int h = 0; h < FH; ++h) {
          if (FNT * h >= 2 * nx) break;
          if (hat[h] < 0) continue;
          const bool in = zin && hcell[h] >= 0;
          const size_t i = zo + (in ? hcell[h] : 0);
          copy_elem<sizeof(T)>(sq + (unsigned)hat[h] * (unsigned)sizeof(T), Win + i, in);
          if (use_vp) copy_elem<sizeof(T)>(sv + (unsigned)hat[h] * (unsigned)sizeof(T), Vp + i, in);
        }
      }
    }
    copies_commit();
  };
  // forms v_j of the elements this thread copied; its own cells' v_j and v_{j-1} in v, vp
  auto form_plane = [&](int t, T (&v)[FE], T (&vp)[FE]) {
    T* q = stage_q(t);
#pragma unroll
    for (int e = 0; e < FE; ++e) {
      T* p = q + nx + tid + FNT * e;
      vp[e] = use_vp ? p[pitch] : (T)0;
      v[e] = *p;
      if (STEP) {
        v[e] = use_vp ? form_v(v[e], vp[e], coef, inv_b) : v[e] * inv_b;
        *p = v[e];
      }
    }
    if (STEP && t > 0 && t < P - 1) {
#pragma unroll
      for (int h = 0; h < FH; ++h) {
        if (FNT * h >= 2 * nx) break;
        if (hat[h] < 0) continue;
        T* p = q + hat[h];
        *p = use_vp ? form_v(*p, p[pitch], coef, inv_b) : *p * inv_b;
      }
    }
  };

  Dots<T> sum;
  sum.zero();
  Dot2x2 dd;  // FP32: the sums over pairs of cells on paired instructions
  dd.zero();
  T vdn[FE], vc[FE], vpc[FE], vup[FE], vpu[FE];
#pragma unroll
  for (int t = 0; t < FSTAGES; ++t) copy_plane(t);
  copies_wait<FSTAGES - 2>();
  form_plane(0, vdn, vpc);
  form_plane(1, vc, vpc);
  for (int t = 1; t <= P - 2; ++t) {
    copies_wait<FSTAGES - 3>();
    form_plane(t + 1, vup, vpu);
    __syncthreads();  // plane t is formed, plane t - 1 is done with
    copy_plane(t + FSTAGES - 1);
    const T* q = stage_q(t);
    const float* k = reinterpret_cast<const float*>(q + 2 * pitch) + tid;
    const int z = z0 - 1 + t;
    const size_t o = (size_t)plane * z + i0 + tid;
    if (BC == GMRF_BC_NEUMANN) {
      // an edge that leaves the grid takes the centre value: its term is exactly 0
#pragma unroll
      for (int e = 0; e < FE; ++e) {
        if (z == 0) vdn[e] = vc[e];
      }
    }
    T res[FE];
    if constexpr (sizeof(T) == 4) {
#pragma unroll
      for (int e = 0; e < FE; e += 2) {
        const float2 c = make_float2(vc[e], vc[e + 1]);
        const float2 zu = BC == GMRF_BC_NEUMANN && z == nz - 1 ? c : make_float2(vup[e], vup[e + 1]);
        const float2 kk = kfield ? make_float2(k[FNT * e], k[FNT * (e + 1)]) : make_float2(a.kappa2_const, a.kappa2_const);
        float2 g = x2_fma(kk, c, x2_sub(c, make_float2(q[l[e]], q[l[e + 1]])));
        g = x2_add(g, x2_sub(c, make_float2(q[r[e]], q[r[e + 1]])));
        g = x2_add(g, x2_sub(c, make_float2(q[u[e]], q[u[e + 1]])));
        g = x2_add(g, x2_sub(c, make_float2(q[d[e]], q[d[e + 1]])));
        g = x2_add(g, x2_sub(c, make_float2(vdn[e], vdn[e + 1])));
        g = x2_add(g, x2_sub(c, zu));
        if (use_vp) g = x2_fma(make_float2(-bprev, -bprev), make_float2(vpc[e], vpc[e + 1]), g);
        res[e] = g.x;
        res[e + 1] = g.y;
      }
    } else {
#pragma unroll
      for (int e = 0; e < FE; ++e) {
        const T c = vc[e], zu = BC == GMRF_BC_NEUMANN && z == nz - 1 ? c : vup[e];
        const T kk = kfield ? (T)k[FNT * e] : a.kappa2_const;
        T g = fma(kk, c, c - q[l[e]]) + (c - q[r[e]]) + ((c - q[u[e]]) + (c - q[d[e]])) + ((c - vdn[e]) + (c - zu));
        if (use_vp) g = fma(-bprev, vpc[e], g);
        res[e] = g;
      }
    }
#pragma unroll
    for (int e = 0; e < FE; ++e) {
      if (e >= nin) {
        res[e] = (T)0;  // no part of the sums
        continue;
      }
      Wout[o + FNT * e] = STEP ? res[e] : res[e] * a.scale;
      if (STEP) {
        Vc[o + FNT * e] = vc[e];
        if (a.P.vb) vb_store1(vb_at(a.P, s, j, n, o + FNT * e), (float)vc[e]);
      }
    }
    if (STEP) {
      if constexpr (sizeof(T) == 4) {
#pragma unroll
        for (int e = 0; e < FE; e += 2)
          dd.add(make_float2(e < nin ? vc[e] : 0.f, e + 1 < nin ? vc[e + 1] : 0.f), make_float2(res[e], res[e + 1]));
      } else {
#pragma unroll
        for (int e = 0; e < FE; ++e)
          if (e < nin) sum.add(vc[e], res[e]);
      }
    }
#pragma unroll
    for (int e = 0; e < FE; ++e) {
      vdn[e] = vc[e];
      vc[e] = vup[e];
      vpc[e] = vpu[e];
    }
  }
  copies_wait<0>();
  if (!STEP) return;
  if constexpr (sizeof(T) == 4) sum = dd.merged();
  sum = block_sum(sum, red);
  const int nblk = gridDim.x;
  const unsigned ticket = publish(sum, a.partials, a.counters, s, li, nblk);
  if (publish_wait(ticket, a.counters, s, nblk, &s_int[3]))
    finish_step<T>(a.P, j, s, a.partials, nblk, a.st, a.alpha, a.beta, a.alpha_f, a.beta2_f, red, s_int, s_flt);
}

// Cells of a thread, ranges of a plane and planes of a chunk, from the grid (and
// the precision) alone.  Two cells a thread (four were 3 to 20 % slower; one only
// pays in FP64, where a plane of a range takes the SM's FP64 lanes a microsecond
// per 200 cells, and while the grid leaves SMs idle).  Chunks of at least eight
// planes, of at least four while a vector has less than a block for every second
// SM: the two halo planes of a chunk are copied besides (61 x 75 x 90, FP32: 4
// vectors 1035 us a call with 8 planes, 1148 with 4; one vector 736 and 701).
struct Flat {
  int fe, nrange, zper, blocks;
};
template <typename T>
Flat flat_plan(const Grid& g) {
  Flat f;
  const int plane = g.nx * g.ny;
  auto ranges = [&](int fe) { return (plane + FNT * fe - 1) / (FNT * fe); };
  f.fe = sizeof(T) == 8 && (int64_t)ranges(2) * ((g.nz + 7) / 8) < 152 ? 1 : 2;
  f.nrange = ranges(f.fe);
  int c = 1;
  for (;;) {
    const int64_t blocks = (int64_t)f.nrange * c;
    const int next = (g.nz + 2 * c - 1) / (2 * c);  // planes of a chunk, halved again
    if (blocks >= 2 * 152 || next < (blocks < 76 ? 4 : 8)) break;
    c *= 2;
  }
  f.zper = (g.nz + c - 1) / c;
  f.blocks = f.nrange * ((g.nz + f.zper - 1) / f.zper);
  return f;
}

template <typename T, int BC, bool STEP, int FE>
cudaError_t flat_launch_e(const Grid& g, const Flat& f, const StencilArgs<T>& a, int nvec, cudaStream_t s) {
  static PerDevice attr;
  const cudaError_t e = set_attribute(attr, k_stencil3d_flat<T, BC, STEP, FE>,
                                      cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)(FSTAGES * flat_stage<T>(FNT * FE, FH * FNT / 2)));
  if (e != cudaSuccess) return e;
  k_stencil3d_flat<T, BC, STEP, FE><<<dim3(f.blocks, nvec), FNT, FSTAGES * flat_stage<T>(FNT * FE, g.nx), s>>>(
      a, f.nrange, f.zper);
  return cudaGetLastError();
}
template <typename T, int BC, bool STEP>
cudaError_t flat_launch(const Grid& g, const StencilArgs<T>& a, int nvec, cudaStream_t s) {
  const Flat f = flat_plan<T>(g);
  if constexpr (sizeof(T) == 8)
    if (f.fe == 1) return flat_launch_e<T, BC, STEP, 1>(g, f, a, nvec, s);
  return flat_launch_e<T, BC, STEP, 2>(g, f, a, nvec, s);
}

}  // namespace

// The halo is nx cells on either side of a range: wider than this the tiles of the
// register kernel read less.
bool stencil3d_flat_eligible(const Grid& g) {
  return g.dim == 3 && 2 * g.nx <= FH * FNT && (int64_t)g.nx * g.ny < ((int64_t)1 << 30);
}
int stencil3d_flat_blocks_per_vector(const Grid& g) {
  return std::max(flat_plan<float>(g).blocks, flat_plan<double>(g).blocks);
}

template <typename T>
cudaError_t launch_stencil3d_flat(const Grid& g, const StencilArgs<T>& a, int nvec, bool step, cudaStream_t s) {
  switch (g.bc) {
    case GMRF_BC_PERIODIC:
      return step ? flat_launch<T, GMRF_BC_PERIODIC, true>(g, a, nvec, s)
                  : flat_launch<T, GMRF_BC_PERIODIC, false>(g, a, nvec, s);
    case GMRF_BC_NEUMANN:
      return step ? flat_launch<T, GMRF_BC_NEUMANN, true>(g, a, nvec, s)
                  : flat_launch<T, GMRF_BC_NEUMANN, false>(g, a, nvec, s);
    default:
      return step ? flat_launch<T, GMRF_BC_DIRICHLET, true>(g, a, nvec, s)
                  : flat_launch<T, GMRF_BC_DIRICHLET, false>(g, a, nvec, s);
  }
}
template cudaError_t launch_stencil3d_flat<float>(const Grid&, const StencilArgs<float>&, int, bool, cudaStream_t);
template cudaError_t launch_stencil3d_flat<double>(const Grid&, const StencilArgs<double>&, int, bool, cudaStream_t);

}  // namespace gmrf
