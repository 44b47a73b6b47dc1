// pt_common.cuh — device-side definitions shared by the solver's kernels.
//
// Padded box layout: every staggered field of an nx x ny x nz grid lives in a box of
// px x py x (nz + 1) elements, px = roundup(nx + 1, 16), py = ny + 1, element (i, j, k) at
// i + px * (j + py * k). A cell (i, j, k) and its lower x-, y-, z-faces and lower xy-, xz-,
// yz-edges share one index, so every stencil offset is one of +-1, +-px, +-pxy.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <cmath>

namespace pt {

struct Box {
  int nx, ny, nz;
  int px;             // x pitch (elements)
  long long pxy;      // px * py
  long long n;        // elements per field
};

// Scalars of one physical step, in FP64 (the FP32 path converts what it needs).
struct Coef {
  double rdx, rdy, rdz;        // 1 / dx, ...
  double h2;                   // min(dx, dy, dz)^2
  double phi0, rphi0, k0, mu0, eta0, R_weak, n_pow, tau0;
  double alpha, B, beta_d, beta_phi, G;
  double rhof_g, rhos_g, rho_bg_g;  // densities times gravity, background phi0 rho_f + (1-phi0) rho_s
  int powerlaw_on, compaction_on;
  double dt, rdt;
  double damp_x, damp_y, damp_z, rho_i, rrho_i, beta_n, rel_mu, rel_eta;
  double dtauv_fac;            // cfl_v h^2 rho_i / (1 + beta_n):   dtau_V = dtauv_fac / mu
  double dtaupt_fac;           // dtpt_scale (1 + beta_n) / nz:     dtau_Pt = dtaupt_fac * mu
  double dtaupf_fac;           // cfl_pf h^2 (1 + beta_d B / alpha): dtau_Pf = dtaupf_fac / kmax
  double rGdtS;                // 1 / (G dtS): xi = mu / (G dtS)
  double ebg;                  // background xy strain rate tau_bg / (2 mu0) (Eqs. 32-33)
  int bg_on;                   // tau_bg != 0: wall xy-edges carry the background stress
};

// Mean shear viscosity over the centres next to the xy-edge with box index q = (i, j, .)
// that lie inside the grid (four inside, two on a wall, one in a corner), in a fixed order.
template <class T>
__device__ inline double edge_mean_mu_xy(const Box& b, const T* mu, long long q, int i, int j) {
  double s = 0.0;
  int n = 0;
  if (i > 0 && j > 0) { s += (double)mu[q - 1 - b.px]; ++n; }
  if (i < b.nx && j > 0) { s += (double)mu[q - b.px]; ++n; }
  if (i > 0 && j < b.ny) { s += (double)mu[q - 1]; ++n; }
  if (i < b.nx && j < b.ny) { s += (double)mu[q]; ++n; }
  return s / n;
}

__host__ __device__ inline long long cidx(const Box& b, int i, int j, int k) {
  return (long long)i + (long long)b.px * j + b.pxy * k;
}

// Levels per block of a kernel whose blocks march up z-columns of the box (`cols` of them, `levels`
// levels each). A chunk of zc levels costs zc + fill steps (its pipeline fill and, where halo levels
// are recomputed, those); the steps of an SM's blocks share its issue slots or pipes, and every wave adds
// base of a step's latency that they do not hide: the chunk with the least (zc + fill) *
// (ceil(blocks / SMs) + base * waves), without the rounding beyond four waves, where blocks end at
// different times. A grid whose columns alone do not fill the chip (96^3: 48 columns of the FP32
// correction pass for 304 block slots) gets shorter chunks, a large one the longest, which recompute and
// refill least.
inline int march_chunk(long long cols, int levels, int max_chunk, int blocks_per_sm, int sms, double fill,
                       double base) {
  const double slots = (double)blocks_per_sm * sms;
  int best = 1;
  double best_cost = 1e300;
  for (int zc = 1; zc <= std::min(max_chunk, levels); ++zc) {
    const double blocks = (double)(cols * ((levels + zc - 1) / zc));
    const bool few = blocks <= 4 * slots;
    const double share = few ? std::ceil(blocks / sms) : blocks / sms + 0.5 * blocks_per_sm;
    const double waves = few ? std::ceil(blocks / slots) : blocks / slots;
    const double cost = (zc + fill) * (share + base * waves);
    if (cost < best_cost) {
      best_cost = cost;
      best = zc;
    }
  }
  return best;
}

inline int sm_count() {
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1)
    return 152;
  return sms;
}

// The kernels of an iteration are chained: launch_chained lets the next kernel's blocks be set up while the
// last blocks of the stream's previous kernel finish, and its first statement, chain_begin, waits until
// everything before it is complete and visible. On a small grid the gap between two kernels costs as much as
// a kernel's work: an iteration takes 16.5 us instead of 21.2 at 32^3 cells in FP64, 12.1 instead of 16.8 in
// double-float and 7.6 instead of 10.6 (its share of the outer phases included) in FP32; from 127^3 cells on
// the gain is 3 % and less. The previous kernel does not release its successor early: the waiting blocks
// then land on the SMs in the uneven order in which these have room, which cost the FP64 kernels up to 27 %
// at 32^3 to 48^3 and double-float 7 % at 383^3. The pointers of a chained kernel and of the functions
// it inlines are not __restrict__, so that no load moves above the wait.
__device__ __forceinline__ void chain_begin() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
template <class... P, class... A>
inline void launch_chained(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, A... args) {
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

// Point kernels of the FP64 pipe run 128 threads per block, which spreads a small grid over the SMs, on a
// tile of 32 x 4 points of a plane or, where rows leave much of their last tile empty, on 128 points of
// the plane in linear order (x fastest): a warp instruction with one lane costs the FP64 pipe the same 16
// cycles as a full one (33 x 33 points fill 52 % of their tiles), but a warp that straddles rows reads two
// lines per load. Extents: the cells, or the
// box where wall indices carry values.
constexpr int kPlaneThreads = 128;
struct Plane {
  int nxe, n;
  int tiles_x;   // tiles per row of tiles, 0: linear order
};
__device__ __forceinline__ bool plane_point(const Plane& p, int& i, int& j) {
  if (p.tiles_x) {
    const int by = (int)(blockIdx.x / (unsigned)p.tiles_x), bx = (int)blockIdx.x - by * p.tiles_x;
    i = bx * 32 + (int)(threadIdx.x & 31);
    j = by * 4 + (int)(threadIdx.x >> 5);
    return i < p.nxe && j * p.nxe < p.n;
  }
  const unsigned t = blockIdx.x * kPlaneThreads + threadIdx.x;
  j = (int)(t / (unsigned)p.nxe);
  i = (int)(t - (unsigned)j * (unsigned)p.nxe);
  return t < (unsigned)p.n;
}
inline Plane plane_of(const Box& b, int wall) {
  const int nx = b.nx + wall, ny = b.ny + wall, tiles_x = (nx + 31) / 32;
  const bool tiles = (long long)nx * ny >= 9LL * (tiles_x * 32) * ((ny + 3) / 4 * 4) / 10;   // at least 90 % full
  return Plane{nx, nx * ny, tiles ? tiles_x : 0};
}
inline dim3 plane_grid(const Plane& p, int levels) {
  const int rows = p.n / p.nxe;
  return dim3((unsigned)(p.tiles_x ? p.tiles_x * ((rows + 3) / 4) : (p.n + kPlaneThreads - 1) / kPlaneThreads),
              (unsigned)levels, 1);
}

// Indices of the residual max-norm slots in the device reduction block.
enum { RED_V = 0, RED_PT = 1, RED_PF = 2, RED_PIC = 3, RED_MUMAX = 4, RED_GMAX = 5, RED_N = 8 };

// Max-reduction of non-negative doubles through their bit patterns (monotone for x >= 0; a
// NaN from fabs has the largest pattern and therefore surfaces in the norm). Every thread of
// the block must call it (it synchronises the block).
template <bool LOG>
__device__ inline void block_max_atomic_impl(double v, unsigned long long* slot) {
  unsigned long long u = (unsigned long long)__double_as_longlong(v);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    unsigned long long w = __shfl_xor_sync(0xffffffffu, u, o);
    u = w > u ? w : u;
  }
  __shared__ unsigned long long warp_max[32];
  const int lane = (threadIdx.x + blockDim.x * (threadIdx.y + blockDim.y * threadIdx.z)) & 31;
  const int warp = (threadIdx.x + blockDim.x * (threadIdx.y + blockDim.y * threadIdx.z)) >> 5;
  const int nwarps = (blockDim.x * blockDim.y * blockDim.z + 31) >> 5;
  if (lane == 0) warp_max[warp] = u;
  __syncthreads();
  if (warp == 0) {
    u = lane < nwarps ? warp_max[lane] : 0ull;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      unsigned long long w = __shfl_xor_sync(0xffffffffu, u, o);
      u = w > u ? w : u;
    }
    if (LOG) {
      if (lane == 0) {
        const double l = log(__longlong_as_double((long long)u));
        if (!(l <= 0.0)) atomicMax(slot, (unsigned long long)__double_as_longlong(l));   // > 0 or NaN
      }
    } else if (lane == 0 && u != 0ull) {
      atomicMax(slot, u);
    }
  }
  __syncthreads();  // warp_max may be reused by the next call in the same kernel
}

__device__ inline void block_max_atomic(double v, unsigned long long* slot) { block_max_atomic_impl<false>(v, slot); }

// The same for values >= 1 whose log goes into the slot: log is monotone, so the block takes the
// max of the values and one thread the log (a NaN still has the largest pattern). Every thread of
// the block calls it; a thread with nothing to contribute passes 1.
__device__ inline void block_max_log_atomic(double v, unsigned long long* slot) { block_max_atomic_impl<true>(v, slot); }

}  // namespace pt
