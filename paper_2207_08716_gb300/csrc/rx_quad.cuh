// rx_quad.cuh — four cells per thread in the FP32 kernels of the reactive solver (rx_kernels.cu,
// rx_mg_kernels.cu).
//
// These kernels read two arrays with their six neighbours and four to seven at the own index, and with one
// cell per thread issue some 20 loads and 21 products for k per cell: instruction issue bounds them before
// HBM does. A thread takes four consecutive cells of a row (one 16-byte load per array and row) and marches
// a chunk of levels: an x face's flux is formed once for both its cells, k once per cell instead of once
// per neighbour in x and z, the next level's values are loaded once, serving this level as z-neighbours
// and the next as own values, and the flux through a z face is carried up. Rows start on 16 floats and
// are padded beyond nx, so the last four of a row may take in padding: it is read, never used by a cell
// (the x-face tests) and written with values that nothing reads.
#pragma once

#include "rx.cuh"

namespace pt {

constexpr int kQuadThreads = 128;
constexpr int kQuadChunk = 16;   // levels per thread at most
struct Quads {
  int per_row, n;   // quads per row and per plane, in linear order over the threads
};
__device__ __forceinline__ bool quad_point(const Quads& p, int& i, int& j) {
  const unsigned t = blockIdx.x * kQuadThreads + threadIdx.x;
  j = (int)(t / (unsigned)p.per_row);
  i = 4 * (int)(t - (unsigned)j * (unsigned)p.per_row);
  return t < (unsigned)p.n;
}
inline Quads quads_of(const Box& b) {
  const int r = (b.nx + 3) / 4;
  return Quads{r, r * b.ny};
}
inline dim3 quad_grid(const Quads& p, int levels, int blocks_per_sm, int* zchunk) {
  const unsigned gx = (unsigned)((p.n + kQuadThreads - 1) / kQuadThreads);
  // a chunk's start loads the level below and its own level: about one and a half level's loads
  *zchunk = march_chunk(gx, levels, kQuadChunk, blocks_per_sm, sm_count(), 1.0, 1.5);
  return dim3(gx, (unsigned)((levels + *zchunk - 1) / *zchunk), 1);
}

// Grids that take the quads. Below some 300 k cells they leave the chip idle (a block has 512 cells of a
// level, and a chunk starts with two dependent loads) and one cell per thread is faster: a V-cycle of one
// level (30 sweeps) takes 64 us at 32^3 cells, 115 at 262 k, 150 at 393 k and 200 at 80^3 so, and 89, 127,
// 142 and 165 with quads.
constexpr long long kQuadCells = 300000;
inline bool quads_pay(const Box& b) { return (long long)b.nx * b.ny * b.nz >= kQuadCells; }

__device__ __forceinline__ float4 quad_load(const float* a, long long q) {
  return *reinterpret_cast<const float4*>(a + q);
}
__device__ __forceinline__ void quad_store(float* a, long long q, const float4& v) {
  *reinterpret_cast<float4*>(a + q) = v;
}
__device__ __forceinline__ float quad_get(const float4& v, int n) {
  return n == 0 ? v.x : n == 1 ? v.y : n == 2 ? v.z : v.w;
}
__device__ __forceinline__ void quad_set(float4& v, int n, float x) {
  if (n == 0) v.x = x;
  else if (n == 1) v.y = x;
  else if (n == 2) v.z = x;
  else v.w = x;
}
// Largest changes of a thread's cells, as bit patterns of |x| (a NaN is the largest): in FP64 per cell the
// change norm took as long on the FP64 pipe as two sweeps.
struct QuadChange {
  unsigned phi, Pf, Xs;
};
__device__ __forceinline__ void quad_max(unsigned& m, float x) { m = max(m, __float_as_uint(fabsf(x))); }
__device__ __forceinline__ double quad_change(const QuadChange& m, float pf_iscale) {
  return rx_change((double)__uint_as_float(m.phi), (double)__uint_as_float(m.Pf) * (double)pf_iscale,
                   (double)__uint_as_float(m.Xs));
}

// Own values at the current level and the z-face terms below it.
struct QuadColumn {
  float4 Pf, phi;
  float k[4];                    // k of the own values
  float fz[4], kz[4];            // (k_d + k) (Pf - Pf_d - rho_f g dz) and k_d + k of the lower faces
};

__device__ __forceinline__ QuadColumn quad_column(const Box& b, const RxCoef<float>& c, const float* Pf,
                                                  const float* phi, int i, int j, int k) {
  const long long q = cidx(b, i, j, k);
  QuadColumn s;
  s.Pf = quad_load(Pf, q);
  s.phi = quad_load(phi, q);
#pragma unroll
  for (int v = 0; v < 4; ++v) {
    s.k[v] = rx_perm(c, quad_get(s.phi, v));
    s.fz[v] = 0.0f;
    s.kz[v] = 0.0f;
  }
  if (k > 0) {
    const float4 Pd = quad_load(Pf, q - b.pxy), hd = quad_load(phi, q - b.pxy);
#pragma unroll
    for (int v = 0; v < 4; ++v) {
      s.kz[v] = rx_perm(c, quad_get(hd, v)) + s.k[v];
      s.fz[v] = s.kz[v] * ((quad_get(s.Pf, v) - quad_get(Pd, v)) - c.rhofg_dz);
    }
  }
  return s;
}

// Level k: own values, div[v] = sum over the faces of (k + k_nb)(Pf_nb - Pf) / d^2 (z with the buoyancy;
// twice minus the divergence of the Darcy flux) and, with KD, kd[v] = sum of (k + k_nb) / d^2. Leaves the
// column at level k + 1.
template <bool KD>
__device__ __forceinline__ void quad_level(const Box& b, const RxCoef<float>& c, const float* gPf,
                                           const float* gphi, int i, int j, int k, QuadColumn& col,
                                           float (&Pf)[4], float (&ph)[4], float (&div)[4], float (&kd)[4]) {
  const long long q = cidx(b, i, j, k);
  const long long px = b.px, pxy = b.pxy;
  const bool has_d = j > 0, has_u = j < b.ny - 1, up = k < b.nz - 1;
  const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
  // loads
  float4 Pn = zero, hn = zero, Pd = zero, hd = zero, Pu = zero, hu = zero;
  float Pl = 0.f, hl = 0.f, Pr = 0.f, hr = 0.f;
  if (up) { Pn = quad_load(gPf, q + pxy); hn = quad_load(gphi, q + pxy); }
  if (has_d) { Pd = quad_load(gPf, q - px); hd = quad_load(gphi, q - px); }
  if (has_u) { Pu = quad_load(gPf, q + px); hu = quad_load(gphi, q + px); }
  if (i > 0) { Pl = gPf[q - 1]; hl = gphi[q - 1]; }
  if (i + 4 < b.nx) { Pr = gPf[q + 4]; hr = gphi[q + 4]; }
#pragma unroll
  for (int v = 0; v < 4; ++v) {
    Pf[v] = quad_get(col.Pf, v);
    ph[v] = quad_get(col.phi, v);
  }
  // x faces i .. i + 4 (zero through the walls)
  float fx[5], kx[5];
  kx[0] = i > 0 ? rx_perm(c, hl) + col.k[0] : 0.f;
  fx[0] = kx[0] * (Pf[0] - Pl);
#pragma unroll
  for (int v = 1; v < 4; ++v) {
    kx[v] = i + v < b.nx ? col.k[v - 1] + col.k[v] : 0.f;
    fx[v] = i + v < b.nx ? kx[v] * (Pf[v] - Pf[v - 1]) : 0.f;
  }
  kx[4] = i + 4 < b.nx ? col.k[3] + rx_perm(c, hr) : 0.f;
  fx[4] = i + 4 < b.nx ? kx[4] * (Pr - Pf[3]) : 0.f;
#pragma unroll
  for (int v = 0; v < 4; ++v) {
    const float kc = col.k[v];
    const float kyd = has_d ? rx_perm(c, quad_get(hd, v)) + kc : 0.f, kyu = has_u ? kc + rx_perm(c, quad_get(hu, v)) : 0.f;
    const float sy = fmaf(kyd, quad_get(Pd, v) - Pf[v], kyu * (quad_get(Pu, v) - Pf[v]));
    const float kn = rx_perm(c, quad_get(hn, v));
    const float kzu = up ? kc + kn : 0.f;
    const float fzu = kzu * ((quad_get(Pn, v) - Pf[v]) - c.rhofg_dz);
    div[v] = fmaf(fx[v + 1] - fx[v], c.rdx2, fmaf(sy, c.rdy2, (fzu - col.fz[v]) * c.rdz2));
    if (KD) kd[v] = fmaf(kx[v] + kx[v + 1], c.rdx2, fmaf(kyd + kyu, c.rdy2, (kzu + col.kz[v]) * c.rdz2));
    col.fz[v] = fzu;
    col.kz[v] = kzu;
    col.k[v] = kn;
  }
  col.Pf = Pn;
  col.phi = hn;
}

}  // namespace pt
