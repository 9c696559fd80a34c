// stencil2d_resident.cu -- Lanczos steps of Algorithm 1 with the 5-point lattice
// apply of Q (Section 2) on small 2-D grids, many steps in one launch.
//
// On a grid of a few thousand cells a step of its own launch is latency: the
// launch, the state and the vectors from L2, the blocks' sums through global
// memory, and the counter that finds the last block.  Here a thread-block cluster of up
// to 16 blocks keeps one vector for all its steps: q_{j-1}, v_{j-1} and kappa^2 of a
// thread's two cells stay in registers, v_j goes to the blocks' shared memory, where
// the neighbours read it (distributed shared memory), the state of the iteration is
// block 0's, and only v_j, alpha_j and beta_j are written out.  A step has three
// cluster barriers: v_j formed; the sums with block 0, which runs the end of the step
// (common.cuh); its alpha, beta and status with all blocks.  The status ends the loop,
// so a launch of any number of steps does no more than the iteration needs.
//
// The cells are dealt out in the tiles of the one-step kernel (lanczos_stencil.cu), a
// group of threads per tile as its blocks there, with the same arithmetic and the same
// order of every sum: the results are the same bits, so the number of vectors may decide
// between the two.  The places of a cell's neighbours do not change and absorb the
// boundary conditions: the wrapped cell, the cell itself (Neumann: the term c - c is
// exactly 0), or a slot that holds 0 (Dirichlet).
//
// Bound: the chain of a step's dependent operations.  FP64 64 x 64 (one vector, 102
// steps, cycles a step): v_j 670, the cells and their sums 3900 (an FP64 operation of a
// warp takes its quarter of the SM 64 cycles), the end of the step 5400 (about 3400
// since its comparisons left the FP64 lanes), the barriers 500 to 700 each.  Two cells a thread: with four or eight in fewer warps the call took 973 and
// 1260 us against 808, since an SM's quarters have their own FP64 lanes.  Measured,
// sample calls with one vector against the one-step kernel: FP64 to 1e-10 64 x 64
// 1131 -> 859 us, 24 x 24 671 -> 542, 91 x 77 1239 -> 1154; FP32 to 1e-6 731 -> 557,
// 563 -> 450, 784 -> 581, 190 x 150 807 -> 664.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstring>

#include "internal.h"
#include "per_device.h"
#include "stencil_args.h"

namespace gmrf {
namespace {

constexpr int kMaxCluster = 16;
constexpr int kMaxTiles = 4 * kMaxCluster;  // four groups of threads a block

__device__ __forceinline__ unsigned cluster_addr(unsigned local, unsigned rank) {
  unsigned r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(local), "r"(rank));
  return r;
}
__device__ __forceinline__ void cluster_ld(float& v, unsigned at) {
  asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(at) : "memory");
}
__device__ __forceinline__ void cluster_ld(double& v, unsigned at) {
  asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(at) : "memory");
}
__device__ __forceinline__ void cluster_st(unsigned at, unsigned long long v) {
  asm volatile("st.shared::cluster.b64 [%0], %1;" ::"r"(at), "l"(v) : "memory");
}
__device__ __forceinline__ void cluster_barrier() {
  asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}

// the tiles' records in block 0, and what block 0 hands back; its first group of
// threads runs the end of the step, as a block of the one-step kernel does
template <typename T>
struct ClusterRecords {
  static constexpr bool kept = true;
  typedef FirstThreads<tile2d_threads<T>()> Threads;
  const unsigned long long* p;  // [tile][3]
  double* scalars;
  int* status;
  __device__ __forceinline__ Dots<T> operator()(int b) const {
    static_assert(sizeof(Dots<T>) == 24, "a record is three 8-byte words");
    const unsigned long long w[3] = {p[3 * b], p[3 * b + 1], p[3 * b + 2]};
    Dots<T> d;
    memcpy(&d, w, sizeof(d));
    return d;
  }
  __device__ __forceinline__ void keep(double a, double b, double y) const {
    scalars[0] = a;
    scalars[1] = b;
    scalars[2] = y;
  }
};

// tpb: tiles of a block
template <typename T, int BC>
__global__ void __launch_bounds__(4 * tile2d_threads<T>()) k_resident2d(StencilArgs<T> a, int nsteps, int tpb) {
  constexpr int TX = kTileX, TY = tile2d_y<T>(), NT = tile2d_threads<T>(), E = kTileCells;
  extern __shared__ __align__(16) unsigned char smraw[];
  T* vs = reinterpret_cast<T*>(smraw);  // v_j of the block's tiles, then a 0
  __shared__ Dots<T> red[4][NT / 32];
  __shared__ unsigned long long rec[3 * kMaxTiles];
  __shared__ unsigned long long s_step[4];  // every block: alpha, beta, 1 / beta, status
  __shared__ VecState s_st;                 // block 0: the state, and what it hands out
  __shared__ double s_out[3];
  __shared__ int s_status;
  __shared__ int s_int[4];
  __shared__ float s_flt[4];
  const int s = blockIdx.y, rank = blockIdx.x, ncl = gridDim.x;  // a vector's blocks are one cluster
  if (a.st[s].status != VS_RUNNING) return;  // the same for all of them: block 0 writes it at the end
  int j = a.st[s].m;
  const int nx = a.nx, ny = a.ny, tgx = (nx + TX - 1) / TX, ntiles = tgx * ((ny + TY - 1) / TY);
  const int tid = threadIdx.x, group = tid / NT, w = tid % NT;
  const int tile = rank * tpb + group;
  const size_t n = a.n, so = (size_t)s * n, base = (size_t)s * a.P.nslots, mo = (size_t)s * a.P.m_max;
  T coef = 0, bprev = 0, inv_b = (T)a.st[s].vscale;
  const T* Win = ((j & 1) ? a.W1 : a.W0) + so;
  const T* Vp = nullptr;
  if (j > 0) {
    Vp = a.V + (base + (size_t)((j - 1) % a.P.nslots)) * n;
    coef = (T)a.alpha[mo + j - 1];
    bprev = (T)a.beta[mo + j - 1];
  }
  const unsigned vs0 = (unsigned)__cvta_generic_to_shared(vs);
  auto at = [&](int x, int y) -> unsigned {  // v_j of a cell
    const int t = (y / TY) * tgx + x / TX, b = t / tpb;
    return cluster_addr(vs0, (unsigned)b) +
           (unsigned)((t - b * tpb) * TX * TY + (y % TY) * TX + x % TX) * (unsigned)sizeof(T);
  };
  const int gx = (tile % tgx) * TX + (w & 31), gy = (tile / tgx) * TY + (w >> 5);
  const size_t cell = (size_t)gx + (size_t)nx * gy, next = (size_t)nx * (TY / E);  // own cells: cell + next e, e < nin
  int nin = 0;
  unsigned nb[E][4];
  T q[E], v[E], kap[E];
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const int x = gx, y = gy + e * (TY / E);
    q[e] = v[e] = (T)0;
    kap[e] = a.kappa2_const;
    nb[e][0] = nb[e][1] = nb[e][2] = nb[e][3] = vs0;
    if (tile >= ntiles || x >= nx || y >= ny) continue;
    nin = e + 1;
    const size_t i = cell + next * e;
    q[e] = Win[i];
    if (Vp) v[e] = Vp[i];
    if (a.kappa2) kap[e] = (T)__ldg(a.kappa2 + i);
    constexpr bool PER = BC == GMRF_BC_PERIODIC;
    // where the grid ends: the cell itself, or the slot behind the block's cells
    const unsigned gone = BC == GMRF_BC_NEUMANN ? at(x, y)
                                                : cluster_addr(vs0, (unsigned)rank) +
                                                      (unsigned)(tpb * TX * TY) * (unsigned)sizeof(T);
    nb[e][0] = x > 0 || PER ? at(x > 0 ? x - 1 : nx - 1, y) : gone;
    nb[e][1] = x < nx - 1 || PER ? at(x < nx - 1 ? x + 1 : 0, y) : gone;
    nb[e][2] = y > 0 || PER ? at(x, y > 0 ? y - 1 : ny - 1) : gone;
    nb[e][3] = y < ny - 1 || PER ? at(x, y < ny - 1 ? y + 1 : 0) : gone;
  }
  T* own = vs + group * TX * TY + w;
  if (tid == 0) {
    vs[tpb * TX * TY] = (T)0;
    if (rank == 0) s_st = a.st[s];
  }
  auto store_ab = [&]() {  // of step j - 1, by one thread of block 0
    a.alpha[mo + j - 1] = s_out[0];
    a.beta[mo + j - 1] = s_out[1];
    a.alpha_f[mo + j - 1] = (float)s_out[0];
    a.beta2_f[mo + j - 1] = (float)(s_out[1] * s_out[1]);
  };

  for (int k = 0;; ++k) {
    // v_j = (q_{j-1} - alpha_{j-1} v_{j-1}) / beta_{j-1}   (v_0 = z / ||z||)
    T* Vc = a.V + (base + (size_t)(j % a.P.nslots)) * n;
    T vp[E];
#pragma unroll
    for (int e = 0; e < E; ++e) {
      vp[e] = v[e];
      if (e >= nin) continue;
      v[e] = next_v(q[e], vp[e], coef, inv_b, j > 0);
      own[e * NT] = v[e];
    }
    cluster_barrier();
    // stores to global memory follow the barrier, which would wait for them
    if (rank == 0 && tid == 0 && k > 0) store_ab();
#pragma unroll
    for (int e = 0; e < E; ++e) {
      if (e >= nin) continue;
      const size_t i = cell + next * e;
      Vc[i] = v[e];
      if (a.P.vb) vb_store1(vb_at(a.P, s, j, n, i), (float)v[e]);
    }
    Dots<T> d;
    d.zero();
#pragma unroll
    for (int e = 0; e < E; ++e) {
      if (e >= nin) continue;
      T l, r, u, b;
      cluster_ld(l, nb[e][0]);
      cluster_ld(r, nb[e][1]);
      cluster_ld(u, nb[e][2]);
      cluster_ld(b, nb[e][3]);
      const T c = v[e];
      q[e] = b_cell(kap[e], c, edge(c, l), edge(c, r), edge(c, u), edge(c, b));
      if (j > 0) q[e] = less(q[e], bprev, vp[e]);
      d.add(c, q[e]);
    }
    d = reduce_group(d, red[group], NT / 32, w >> 5);
    if (w == 0 && tile < ntiles) {
      unsigned long long r[3];
      memcpy(r, &d, sizeof(d));
      const unsigned to = cluster_addr((unsigned)__cvta_generic_to_shared(rec), 0u) + (unsigned)tile * 24u;
#pragma unroll
      for (int i = 0; i < 3; ++i) cluster_st(to + 8u * i, r[i]);
    }
    cluster_barrier();
    if (rank == 0 && tid < NT) {
      finish_step_from<T>(a.P, j, 0, ClusterRecords<T>{rec, s_out, &s_status}, ntiles, &s_st, a.alpha + mo,
                          a.beta + mo, a.alpha_f + mo, a.beta2_f + mo, red[0], s_int, s_flt, -1.0);
      FirstThreads<NT>::sync();
      if (tid < ncl) {
        const unsigned to = cluster_addr((unsigned)__cvta_generic_to_shared(s_step), (unsigned)tid);
#pragma unroll
        for (int i = 0; i < 3; ++i) cluster_st(to + 8u * i, (unsigned long long)__double_as_longlong(s_out[i]));
        cluster_st(to + 24u, (unsigned long long)(long long)s_status);
      }
    }
    cluster_barrier();
    coef = (T)__longlong_as_double((long long)s_step[0]);
    bprev = (T)__longlong_as_double((long long)s_step[1]);
    inv_b = (T)__longlong_as_double((long long)s_step[2]);
    const int status = (int)(long long)s_step[3];
    ++j;
    if (status != VS_RUNNING || k + 1 >= nsteps) break;
  }
  if (rank == 0 && tid == 0) {
    store_ab();
    a.st[s] = s_st;
  }
  // q_{j-1}, where the next launch, or a continued iteration, looks for it
  T* Wout = ((j & 1) ? a.W1 : a.W0) + so;
#pragma unroll
  for (int e = 0; e < E; ++e)
    if (e < nin) Wout[cell + next * e] = q[e];
}

template <typename T>
int tiles_of(const Grid& g) {
  return ((g.nx + kTileX - 1) / kTileX) * ((g.ny + tile2d_y<T>() - 1) / tile2d_y<T>());
}

// the launch of nvec vectors; returns the tiles of a block
template <typename T, int BC>
cudaError_t config(const Grid& g, int nvec, cudaLaunchConfig_t& c, cudaLaunchAttribute& at, int& tpb) {
  static PerDevice attr;
  const cudaError_t e = set_attribute(attr, k_resident2d<T, BC>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (e != cudaSuccess) return e;
  const int tiles = tiles_of<T>(g);
  int ncl = 1;
  while (ncl < kMaxCluster && ncl < tiles) ncl *= 2;
  tpb = (tiles + ncl - 1) / ncl;
  c = {};
  c.gridDim = dim3(ncl, nvec);
  c.blockDim = dim3(tpb * tile2d_threads<T>());
  c.dynamicSmemBytes = ((size_t)tpb * kTileX * tile2d_y<T>() + 1) * sizeof(T);
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = ncl;
  at.val.clusterDim.y = 1;
  at.val.clusterDim.z = 1;
  c.attrs = &at;
  c.numAttrs = 1;
  return cudaSuccess;
}

template <typename T, int BC>
cudaError_t launch(const Grid& g, const StencilArgs<T>& a, int nvec, int nsteps, cudaStream_t s) {
  cudaLaunchConfig_t c;
  cudaLaunchAttribute at;
  int tpb = 0;
  const cudaError_t e = config<T, BC>(g, nvec, c, at, tpb);
  if (e != cudaSuccess) return e;
  c.stream = s;
  return cudaLaunchKernelEx(&c, k_resident2d<T, BC>, a, nsteps, tpb);
}

template <typename T, int BC>
bool fits(const Grid& g) {
  cudaLaunchConfig_t c;
  cudaLaunchAttribute at;
  int tpb = 0, n = 0;
  if (config<T, BC>(g, 1, c, at, tpb) == cudaSuccess &&
      cudaOccupancyMaxActiveClusters(&n, k_resident2d<T, BC>, &c) == cudaSuccess)
    return n > 0;
  cudaGetLastError();
  return false;
}
template <typename T>
bool fits(const Grid& g) {
  switch (g.bc) {
    case GMRF_BC_PERIODIC: return fits<T, GMRF_BC_PERIODIC>(g);
    case GMRF_BC_NEUMANN: return fits<T, GMRF_BC_NEUMANN>(g);
    default: return fits<T, GMRF_BC_DIRICHLET>(g);
  }
}

}  // namespace

// Up to four tiles a block (FP64 three: its lanes bound them), and not more tiles of all
// vectors than this: beyond, the launches of the one-step kernel are hidden by its
// work, and its many blocks fill the SMs better than clusters do.
// 64 x 64, calls with 8, 32 and 64 vectors, clusters against one-step: FP64 1011 and
// 1143 us, 1342 and 1670, 2280 and 2204; FP32 581 and 843, 648 and 960, 1330 and 1175.
// More than a tile a block: FP64 91 x 77 (36 tiles) 4 vectors 1176 and 1245, 8 1552 and
// 1440, 100 x 100 (52) one vector 1311 and 1221; FP32 91 x 77 (18) 8 vectors 647 and
// 833, 16 1360 and 1275, 190 x 150 (60) 4 vectors 677 and 860.
static bool takes(const Grid& g, bool fp64, int nvec) {
  if (g.dim != 2 || g.op != GMRF_OP_SHIFTED_LAPLACIAN || stencil2d_strip_eligible(g, fp64)) return false;
  if (g.n > (size_t)kMaxTiles * 512) return false;
  const int tiles = fp64 ? tiles_of<double>(g) : tiles_of<float>(g);
  const int64_t all = (int64_t)tiles * nvec;
  if (tiles <= kMaxCluster) return all <= (fp64 ? 5 : 2) * 152;
  return tiles <= (fp64 ? 3 * kMaxCluster : kMaxTiles) && all <= (fp64 ? 152 : 256);
}
void stencil2d_resident_ask(Grid& g, bool fp64, int nvec) {
  if (g.clusters < 0 && takes(g, fp64, nvec)) g.clusters = (fp64 ? fits<double>(g) : fits<float>(g)) ? 1 : 0;
}
bool stencil2d_resident_eligible(const Grid& g, bool fp64, int nvec) { return g.clusters > 0 && takes(g, fp64, nvec); }

template <typename T>
cudaError_t launch_stencil2d_resident(const Grid& g, const StencilArgs<T>& a, int nvec, int nsteps, cudaStream_t s) {
  switch (g.bc) {
    case GMRF_BC_PERIODIC: return launch<T, GMRF_BC_PERIODIC>(g, a, nvec, nsteps, s);
    case GMRF_BC_NEUMANN: return launch<T, GMRF_BC_NEUMANN>(g, a, nvec, nsteps, s);
    default: return launch<T, GMRF_BC_DIRICHLET>(g, a, nvec, nsteps, s);
  }
}
template cudaError_t launch_stencil2d_resident<float>(const Grid&, const StencilArgs<float>&, int, int, cudaStream_t);
template cudaError_t launch_stencil2d_resident<double>(const Grid&, const StencilArgs<double>&, int, int, cudaStream_t);

}  // namespace gmrf
