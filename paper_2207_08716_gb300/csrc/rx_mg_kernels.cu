// rx_mg_kernels.cu — geometric multigrid (FAS V-cycle) of the reactive porosity-wave step (thesis
// Art. 3, Eqs. 8-10; the thesis's future-work section on multigrid-accelerated PT iterations).
//
// The smoother is the reactive PT iteration with a local pseudo step: per cell
//   gP   = R - (Pf - Pf_o) / dt + fP
//   Pf'  = Pf + gP / (Dk / (omega BP) + 1/dt + a)        (Dk: Jacobi diagonal of the Darcy operator)
//   phi' = clamp(phi_o + dt dphi, 1e-4, 1) + fphi,   Xs' = (Xs_o + (dt/tau) Xs_eq) / (1 + dt/tau) + fX
// with every right-hand side at the sweep's input and f = 0 on the finest grid. Coarse grids are
// 2 x 2 x 2 agglomerations; the restriction takes 8-child means of the iterate and of the
// residual (g = target - current), the FAS source is f_c = mean(r) - g_c(u0_c), and the
// correction u_c - u0_c (written by the coarse level's last sweep) comes back by trilinear
// interpolation (3/4, 1/4 per direction, the neighbour held at the wall). In FP64 and on small
// FP32 grids the sweeps, the restriction and the right-hand side run one thread per cell, on FP32 grids
// from kQuadCells four cells per thread (rx_quad.cuh); the prolongation has one thread per pair of coarse
// cells, and a small coarsest grid is swept in one block.
#include "rx_quad.cuh"

namespace pt {

namespace {

// Step equations at cell (i, j, k) of a grid: the rate R, gP, the Jacobi denominator (DEN) and
// the porosity and Xs targets (with the FAS sources when FAS).
template <class T>
struct MgEq {
  T R, gP, den, phi1, Xs1;
};

// The cell's own part of the step equations, given the Darcy divergence divq and (DEN) the Jacobi
// diagonal Dk of the Darcy operator; no FAS sources.
template <class T, bool DEN>
__device__ __forceinline__ MgEq<T> mg_cell(const RxCoef<T>& c, T romega, T divq, T Dk, T Pf, T ph, T Xs, T Pf_o,
                                           T phi_o, T Xs_o) {
  const T w = rx_rcp(T(1) - ph), ixs = rx_rcp(T(1) - Xs);
  const T xr = c.beta_x * Pf + c.half_xs;
  const bool pos = xr > T(0), below = xr < c.xs_max;     // Xs_eq is xr clamped to [0, xs_max]
  const T xseq = pos ? (below ? xr : c.xs_max) : T(0);
  const T dXs = (xseq - Xs) * c.rtau;
  const T rbp = rx_rcp(rx_bp(c, ph));
  const T src = c.sr_opdx * (T(1) - ph) * ixs;
  const T comp = Pf * w * c.reta;                        // -Pe / (eta (1 - phi)), Pe = -Pf
  MgEq<T> e;
  e.R = (-divq - comp + src * dXs) * rbp;
  e.gP = e.R - (Pf - Pf_o) * c.rdt;
  if (DEN) {
    const T dxs_dpf = pos && below ? c.beta_x : T(0);
    const T a = (w * c.reta - src * dxs_dpf * c.rtau) * rbp;
    e.den = Dk * rbp * romega + c.rdt + a;
  } else {
    e.den = T(1);
  }
  const T bphi = c.beta_d - c.beta_s * w;
  const T dphi = (T(1) - ph) * (bphi * e.R + comp - c.opdx * ixs * dXs);
  e.phi1 = rx_clamp(phi_o + c.dt * dphi, T(1e-4), T(1));
  e.Xs1 = (Xs_o + c.dt_tau * xseq) * c.r1dt_tau;
  return e;
}

template <class T, bool FAS, bool DEN>
__device__ __forceinline__ MgEq<T> mg_eq(const Box& b, const RxCoef<T>& c, T romega, const RxIn<T>& in,
                                         const MgSrc<T>& f, long long q, int i, int j, int k) {
  const long long px = b.px, pxy = b.pxy;
  const T Pf = in.Pf[q], ph = in.phi[q];
  const T kc = rx_perm(c, ph);
  // Darcy flux through the six faces (zero through the walls): s_d = sum over the d-faces of the
  // face permeability (k + k_nb, twice the mean) times the pressure difference (z: minus the
  // buoyancy rho_f g dz across the face); k_d = the sum of those face permeabilities
  T sx = T(0), sy = T(0), sz = T(0), kx = T(0), ky = T(0), kz = T(0);
  if (i > 0) {
    const T kf = rx_perm(c, in.phi[q - 1]) + kc;
    sx = fma(kf, in.Pf[q - 1] - Pf, sx);
    kx += kf;
  }
  if (i < b.nx - 1) {
    const T kf = kc + rx_perm(c, in.phi[q + 1]);
    sx = fma(kf, in.Pf[q + 1] - Pf, sx);
    kx += kf;
  }
  if (j > 0) {
    const T kf = rx_perm(c, in.phi[q - px]) + kc;
    sy = fma(kf, in.Pf[q - px] - Pf, sy);
    ky += kf;
  }
  if (j < b.ny - 1) {
    const T kf = kc + rx_perm(c, in.phi[q + px]);
    sy = fma(kf, in.Pf[q + px] - Pf, sy);
    ky += kf;
  }
  if (k > 0) {
    const T kf = rx_perm(c, in.phi[q - pxy]) + kc;
    sz = fma(kf, (in.Pf[q - pxy] - Pf) + c.rhofg_dz, sz);
    kz += kf;
  }
  if (k < b.nz - 1) {
    const T kf = kc + rx_perm(c, in.phi[q + pxy]);
    sz = fma(kf, (in.Pf[q + pxy] - Pf) - c.rhofg_dz, sz);
    kz += kf;
  }
  // div qD = -(1/2) sum_d s_d / d^2
  const T divq = T(-0.5) * fma(sx, c.rdx2, fma(sy, c.rdy2, sz * c.rdz2));
  const T Dk = DEN ? T(0.5) * fma(kx, c.rdx2, fma(ky, c.rdy2, kz * c.rdz2)) : T(0);
  MgEq<T> e = mg_cell<T, DEN>(c, romega, divq, Dk, Pf, ph, in.Xs[q], in.Pf_o[q], in.phi_o[q], in.Xs_o[q]);
  if (FAS) {
    e.gP += f.fP[q];
    e.phi1 += f.fphi[q];
    e.Xs1 += f.fX[q];
  }
  return e;
}

dim3 grid_of(const Box& b) { return dim3((unsigned)((b.nx + 31) / 32), (unsigned)((b.ny + 7) / 8), (unsigned)b.nz); }

}  // namespace

// LASTE: the last sweep of a coarse level's visit writes the correction e = u' - u0 into the u0
// slots (read and written by the same thread) instead of u', which nothing reads afterwards.
template <class T, bool FAS, bool LASTE>
__global__ void __launch_bounds__(256, sizeof(T) == 4 ? 8 : 5) k_mg_smooth(
    Box b, RxCoef<T> c, T romega, RxIn<T> in, MgSrc<T> f, RxOut<T> out, MgE<T> e0, unsigned long long* red, int check) {
  chain_begin();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int j = blockIdx.y * blockDim.y + threadIdx.y;
  const int k = blockIdx.z;
  double chg = 0.0;
  if (i < b.nx && j < b.ny && k < b.nz) {
    const long long q = cidx(b, i, j, k);
    const MgEq<T> e = mg_eq<T, FAS, true>(b, c, romega, in, f, q, i, j, k);
    const T Pf = in.Pf[q], ph = in.phi[q], Xs = in.Xs[q];
    const T Pf1 = Pf + e.gP * rx_rcp(e.den);
    if (LASTE) {
      e0.Pf[q] = Pf1 - e0.Pf[q];
      e0.phi[q] = e.phi1 - e0.phi[q];
      e0.Xs[q] = e.Xs1 - e0.Xs[q];
    } else {
      out.Pf[q] = Pf1;
      out.phi[q] = e.phi1;
      out.Xs[q] = e.Xs1;
      if (out.R) out.R[q] = e.R;
    }
    if (check)
      chg = rx_change((double)rx_abs(e.phi1 - ph), (double)rx_abs(Pf1 - Pf) * (double)c.pf_iscale,
                      (double)rx_abs(e.Xs1 - Xs));
  }
  if (check) block_max_atomic(chg, red + RED_V);
}

// The same sweep in FP32 with four cells per thread, marching z (rx_quad.cuh). FAS and LASTE as above. At
// 128 x 128 x 512 it takes 57 us cold (one cell per thread: 90; 36 B per cell at the copy peak: 45). Five
// blocks of 96 registers: the V-cycle measured 6 % faster than with four or with an uncapped count, 8 %
// faster than with six.
constexpr int kSmoothBlocks = 5;
template <bool FAS, bool LASTE>
__global__ void __launch_bounds__(kQuadThreads, kSmoothBlocks) k_mg_smooth4(Box b, RxCoef<float> c, float romega,
                                                                            RxIn<float> in, MgSrc<float> f,
                                                                            RxOut<float> out, MgE<float> e0,
                                                                            unsigned long long* red, int check,
                                                                            Quads qd, int zchunk) {
  chain_begin();
  int i, j;
  QuadChange chg{0u, 0u, 0u};
  if (quad_point(qd, i, j)) {
    const int k0 = blockIdx.y * zchunk, k1 = min(k0 + zchunk, b.nz);
    QuadColumn col = quad_column(b, c, in.Pf, in.phi, i, j, k0);
    for (int k = k0; k < k1; ++k) {
      const long long q = cidx(b, i, j, k);
      const float4 Xs = quad_load(in.Xs, q), Pfo = quad_load(in.Pf_o, q), pho = quad_load(in.phi_o, q),
                   Xso = quad_load(in.Xs_o, q);
      float4 fP, fh, fX, uP, uh, uX;
      if (FAS) { fP = quad_load(f.fP, q); fh = quad_load(f.fphi, q); fX = quad_load(f.fX, q); }
      if (LASTE) { uP = quad_load(e0.Pf, q); uh = quad_load(e0.phi, q); uX = quad_load(e0.Xs, q); }
      float Pf[4], ph[4], div[4], kd[4];
      quad_level<true>(b, c, in.Pf, in.phi, i, j, k, col, Pf, ph, div, kd);
      float4 oP, oh, oX, oR;
#pragma unroll
      for (int v = 0; v < 4; ++v) {
        const float X = quad_get(Xs, v);
        const MgEq<float> e = mg_cell<float, true>(c, romega, -0.5f * div[v], 0.5f * kd[v], Pf[v], ph[v], X,
                                                   quad_get(Pfo, v), quad_get(pho, v), quad_get(Xso, v));
        const float gP = FAS ? e.gP + quad_get(fP, v) : e.gP;
        const float P1 = Pf[v] + gP * rx_rcp(e.den);
        const float h1 = FAS ? e.phi1 + quad_get(fh, v) : e.phi1, X1 = FAS ? e.Xs1 + quad_get(fX, v) : e.Xs1;
        quad_set(oP, v, LASTE ? P1 - quad_get(uP, v) : P1);
        quad_set(oh, v, LASTE ? h1 - quad_get(uh, v) : h1);
        quad_set(oX, v, LASTE ? X1 - quad_get(uX, v) : X1);
        quad_set(oR, v, e.R);
        if (check && i + v < b.nx) {
          quad_max(chg.phi, h1 - ph[v]);
          quad_max(chg.Pf, P1 - Pf[v]);
          quad_max(chg.Xs, X1 - X);
        }
      }
      quad_store(LASTE ? e0.Pf : out.Pf, q, oP);
      quad_store(LASTE ? e0.phi : out.phi, q, oh);
      quad_store(LASTE ? e0.Xs : out.Xs, q, oX);
      if (!LASTE && out.R) quad_store(out.R, q, oR);
    }
  }
  if (check) block_max_atomic(quad_change(chg, c.pf_iscale), red + RED_V);
}

// One fine cell per thread: its residual (the step equations, without the Jacobi denominator) and
// iterate; the 8 children of a coarse cell sit in one block of 32 x 4 x 2 threads (x pairs
// summed by a warp shuffle, y and z pairs through shared memory), whose 16 x 2 x 1 coarse cells
// receive the 8-child means.
constexpr int kRbx = 32, kRby = 4, kRbz = 2;

template <class T, bool FAS>
__global__ void __launch_bounds__(kRbx * kRby * kRbz) k_mg_restrict(Box fb, Box cb, RxCoef<T> c, RxIn<T> in,
                                                                    MgSrc<T> f, MgCoarse<T> out) {
  chain_begin();
  const int tx = threadIdx.x, ty = threadIdx.y, tz = threadIdx.z;
  const int i = blockIdx.x * kRbx + tx, j = blockIdx.y * kRby + ty, k = blockIdx.z * kRbz + tz;
  T v[6] = {T(0), T(0), T(0), T(0), T(0), T(0)};        // Pf, phi, Xs, gP, gphi, gX
  if (i < fb.nx && j < fb.ny && k < fb.nz) {
    const long long q = cidx(fb, i, j, k);
    const MgEq<T> e = mg_eq<T, FAS, false>(fb, c, T(1), in, f, q, i, j, k);
    const T ph = in.phi[q], Xs = in.Xs[q];
    v[0] = in.Pf[q];
    v[1] = ph;
    v[2] = Xs;
    v[3] = e.gP;
    v[4] = e.phi1 - ph;
    v[5] = e.Xs1 - Xs;
  }
  __shared__ T part[kRbz][kRby][kRbx / 2][6];
#pragma unroll
  for (int n = 0; n < 6; ++n) {
    const T o = __shfl_down_sync(0xffffffffu, v[n], 1);
    if ((tx & 1) == 0) part[tz][ty][tx >> 1][n] = v[n] + o;
  }
  __syncthreads();
  if (tz == 0 && (ty & 1) == 0 && tx < kRbx / 2) {
    const int I = blockIdx.x * (kRbx / 2) + tx, J = blockIdx.y * (kRby / 2) + (ty >> 1), K = blockIdx.z;
    if (I < cb.nx && J < cb.ny && K < cb.nz) {
      T s[6];
#pragma unroll
      for (int n = 0; n < 6; ++n)
        s[n] = T(0.125) * ((part[0][ty][tx][n] + part[0][ty + 1][tx][n]) + (part[1][ty][tx][n] + part[1][ty + 1][tx][n]));
      const long long Q = cidx(cb, I, J, K);
      out.Pf[Q] = s[0];
      out.phi[Q] = s[1];
      out.Xs[Q] = s[2];
      out.Pf0[Q] = s[0];
      out.phi0[Q] = s[1];
      out.Xs0[Q] = s[2];
      out.fP[Q] = s[3];
      out.fphi[Q] = s[4];
      out.fX[Q] = s[5];
    }
  }
}

// The restriction in FP32: four fine cells per thread, marching z (rx_quad.cuh), the two rows of a coarse
// row in neighbouring lanes: x pairs and z pairs are summed in the thread, y pairs by a shuffle after which
// the even row's lane holds the iterate's sums and the odd row's the residual's. One cell per thread took
// 75 us cold at 128 x 128 x 512, this takes 53; with the right-hand side and the prolongation below (65 us,
// now 42) the whole V-cycle is 7 % shorter.
constexpr int kRestrictBlocks = 4;
struct QuadRows {
  int per_row, n;   // quads per row; threads: two per quad of a coarse row
};
template <bool FAS>
__global__ void __launch_bounds__(kQuadThreads, kRestrictBlocks) k_mg_restrict4(Box fb, Box cb, RxCoef<float> c,
                                                                                RxIn<float> in, MgSrc<float> f,
                                                                                MgCoarse<float> out, QuadRows qr,
                                                                                int zchunk) {
  chain_begin();
  const int t = min((int)(blockIdx.x * kQuadThreads + threadIdx.x), qr.n - 2 + (int)(threadIdx.x & 1));
  const bool own = (int)(blockIdx.x * kQuadThreads + threadIdx.x) < qr.n;
  const int odd = t & 1, J = (t >> 1) / qr.per_row, P = (t >> 1) - J * qr.per_row;
  const int i = 4 * P, j = 2 * J + odd;
  const int K0 = blockIdx.y * zchunk, K1 = min(K0 + zchunk, cb.nz);
  QuadColumn col = quad_column(fb, c, in.Pf, in.phi, i, j, 2 * K0);
  for (int K = K0; K < K1; ++K) {
    float acc[6][2] = {};                                  // Pf, phi, Xs, gP, gphi, gX of the two coarse cells
#pragma unroll 1
    for (int k = 2 * K; k < 2 * K + 2; ++k) {
      const long long q = cidx(fb, i, j, k);
      const float4 Xs = quad_load(in.Xs, q), Pfo = quad_load(in.Pf_o, q), pho = quad_load(in.phi_o, q),
                   Xso = quad_load(in.Xs_o, q);
      float4 fP, fh, fX;
      if (FAS) { fP = quad_load(f.fP, q); fh = quad_load(f.fphi, q); fX = quad_load(f.fX, q); }
      float Pf[4], ph[4], div[4], kd[4];
      quad_level<false>(fb, c, in.Pf, in.phi, i, j, k, col, Pf, ph, div, kd);
#pragma unroll
      for (int v = 0; v < 4; ++v) {
        const float X = quad_get(Xs, v);
        const MgEq<float> e = mg_cell<float, false>(c, 1.0f, -0.5f * div[v], 0.0f, Pf[v], ph[v], X, quad_get(Pfo, v),
                                                    quad_get(pho, v), quad_get(Xso, v));
        acc[0][v >> 1] += Pf[v];
        acc[1][v >> 1] += ph[v];
        acc[2][v >> 1] += X;
        acc[3][v >> 1] += FAS ? e.gP + quad_get(fP, v) : e.gP;
        acc[4][v >> 1] += (FAS ? e.phi1 + quad_get(fh, v) : e.phi1) - ph[v];
        acc[5][v >> 1] += (FAS ? e.Xs1 + quad_get(fX, v) : e.Xs1) - X;
      }
    }
    float2 r[3];
#pragma unroll
    for (int n = 0; n < 3; ++n) {
      const float gx = __shfl_xor_sync(0xffffffffu, odd ? acc[n][0] : acc[n + 3][0], 1);
      const float gy = __shfl_xor_sync(0xffffffffu, odd ? acc[n][1] : acc[n + 3][1], 1);
      r[n] = make_float2(0.125f * ((odd ? acc[n + 3][0] : acc[n][0]) + gx),
                         0.125f * ((odd ? acc[n + 3][1] : acc[n][1]) + gy));
    }
    if (own) {
      const long long Q = cidx(cb, 2 * P, J, K);          // 8-byte aligned; the second cell may be padding
      auto put = [&](float* a, const float2& x) { *reinterpret_cast<float2*>(a + Q) = x; };
      if (odd) {
        put(out.fP, r[0]);
        put(out.fphi, r[1]);
        put(out.fX, r[2]);
      } else {
        put(out.Pf, r[0]);
        put(out.phi, r[1]);
        put(out.Xs, r[2]);
        put(out.Pf0, r[0]);
        put(out.phi0, r[1]);
        put(out.Xs0, r[2]);
      }
    }
  }
}

template <class T>
__global__ void __launch_bounds__(256) k_mg_coarse_rhs(Box b, RxCoef<T> c, RxIn<T> u0, MgCoarse<T> out) {
  chain_begin();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int j = blockIdx.y * blockDim.y + threadIdx.y;
  const int k = blockIdx.z;
  if (i >= b.nx || j >= b.ny || k >= b.nz) return;
  const long long q = cidx(b, i, j, k);
  const MgEq<T> e = mg_eq<T, false, false>(b, c, T(1), u0, MgSrc<T>{nullptr, nullptr, nullptr}, q, i, j, k);
  out.fP[q] -= e.gP;
  out.fphi[q] -= e.phi1 - u0.phi[q];
  out.fX[q] -= e.Xs1 - u0.Xs[q];
}

__global__ void __launch_bounds__(kQuadThreads, kRestrictBlocks) k_mg_coarse_rhs4(Box b, RxCoef<float> c,
                                                                                  RxIn<float> u0, MgCoarse<float> out,
                                                                                  Quads qd, int zchunk) {
  chain_begin();
  int i, j;
  if (!quad_point(qd, i, j)) return;
  const int k0 = blockIdx.y * zchunk, k1 = min(k0 + zchunk, b.nz);
  QuadColumn col = quad_column(b, c, u0.Pf, u0.phi, i, j, k0);
  for (int k = k0; k < k1; ++k) {
    const long long q = cidx(b, i, j, k);
    const float4 Xs = quad_load(u0.Xs, q), Pfo = quad_load(u0.Pf_o, q), pho = quad_load(u0.phi_o, q),
                 Xso = quad_load(u0.Xs_o, q);
    float4 fP = quad_load(out.fP, q), fh = quad_load(out.fphi, q), fX = quad_load(out.fX, q);
    float Pf[4], ph[4], div[4], kd[4];
    quad_level<false>(b, c, u0.Pf, u0.phi, i, j, k, col, Pf, ph, div, kd);
#pragma unroll
    for (int v = 0; v < 4; ++v) {
      const float X = quad_get(Xs, v);
      const MgEq<float> e = mg_cell<float, false>(c, 1.0f, -0.5f * div[v], 0.0f, Pf[v], ph[v], X, quad_get(Pfo, v),
                                                  quad_get(pho, v), quad_get(Xso, v));
      quad_set(fP, v, quad_get(fP, v) - e.gP);
      quad_set(fh, v, quad_get(fh, v) - (e.phi1 - ph[v]));
      quad_set(fX, v, quad_get(fX, v) - (e.Xs1 - X));
    }
    quad_store(out.fP, q, fP);
    quad_store(out.fphi, q, fh);
    quad_store(out.fX, q, fX);
  }
}

// One thread per pair of coarse cells (2P, 2P + 1; J, K) and field: its 4 x 2 x 2 fine cells (the last pair
// of an odd row has its second half in the padding). The 3 x 3 coarse rows around are read once each (one
// thread per fine x-pair read 4 rows per pair, 6 loads per fine cell instead of 2) and folded into the four
// fine rows with 9/16, 3/16 and 1/16, then x: the low child takes 3/4 of its column and 1/4 of the one
// below, the high child 1/4 of the one above; columns and rows are held inside the grid.
template <class T>
struct __align__(16) MgQuad {
  T v[4];
};
template <class T>
struct __align__(2 * sizeof(T)) MgPair {
  T v[2];
};
constexpr int kProlongThreads = 128;
template <class T>
__global__ void __launch_bounds__(kProlongThreads) k_mg_prolong(Box fb, Box cb, MgCorr<T> corr, T* Pf, T* phi, T* Xs,
                                                                int per_row) {
  chain_begin();
  const int t = blockIdx.x * kProlongThreads + threadIdx.x, J = t / per_row, P = t - J * per_row, K = blockIdx.y;
  if (J >= cb.ny) return;
  const int field = blockIdx.z;
  const T* e = field == 0 ? corr.Pf : field == 1 ? corr.phi : corr.Xs;
  T* u = field == 0 ? Pf : field == 1 ? phi : Xs;
  const int lo = max(2 * P - 1, 0), hi = min(2 * P + 2, cb.nx - 1);
  const bool lone = 2 * P + 1 >= cb.nx;
  const T one = T(0.75), side = T(0.25);
  T r[2][2][4];                                            // fine rows (z, y) at the columns 2P - 1 .. 2P + 2
#pragma unroll
  for (int n = 0; n < 16; ++n) r[n >> 3][(n >> 2) & 1][n & 3] = T(0);
#pragma unroll
  for (int dz = -1; dz <= 1; ++dz) {
    const int Kc = min(max(K + dz, 0), cb.nz - 1);
    T y[2][4];
#pragma unroll
    for (int d = 0; d < 4; ++d) y[0][d] = y[1][d] = T(0);
#pragma unroll
    for (int dy = -1; dy <= 1; ++dy) {
      const int Jc = min(max(J + dy, 0), cb.ny - 1);
      const T* row = e + cidx(cb, 0, Jc, Kc);
      const MgPair<T> m = *reinterpret_cast<const MgPair<T>*>(row + 2 * P);
      const T x[4] = {row[lo], m.v[0], lone ? m.v[0] : m.v[1], row[hi]};
#pragma unroll
      for (int d = 0; d < 4; ++d) {
        if (dy <= 0) y[0][d] = fma(dy < 0 ? side : one, x[d], y[0][d]);
        if (dy >= 0) y[1][d] = fma(dy > 0 ? side : one, x[d], y[1][d]);
      }
    }
#pragma unroll
    for (int n = 0; n < 8; ++n) {
      const int h = n >> 2, d = n & 3;
      if (dz <= 0) r[0][h][d] = fma(dz < 0 ? side : one, y[h][d], r[0][h][d]);
      if (dz >= 0) r[1][h][d] = fma(dz > 0 ? side : one, y[h][d], r[1][h][d]);
    }
  }
#pragma unroll
  for (int n = 0; n < 4; ++n) {
    const T* c = r[n >> 1][n & 1];
    MgQuad<T>* at = reinterpret_cast<MgQuad<T>*>(u + cidx(fb, 4 * P, 2 * J + (n & 1), 2 * K + (n >> 1)));
    MgQuad<T> w = *at;
    w.v[0] += fma(one, c[1], side * c[0]);
    w.v[1] += fma(one, c[1], side * c[2]);
    w.v[2] += fma(one, c[2], side * c[1]);
    w.v[3] += fma(one, c[2], side * c[3]);
    if (field == 1)
#pragma unroll
      for (int m = 0; m < 4; ++m) w.v[m] = rx_clamp(w.v[m], T(1e-4), T(1));
    *at = w;
  }
}

template <class T>
__global__ void __launch_bounds__(256) k_mg_restrict_old(Box fb, Box cb, const T* __restrict__ a,
                                                         const T* __restrict__ b, const T* __restrict__ d, T* A, T* B,
                                                         T* D) {
  const int I = blockIdx.x * blockDim.x + threadIdx.x;
  const int J = blockIdx.y * blockDim.y + threadIdx.y;
  const int K = blockIdx.z;
  if (I >= cb.nx || J >= cb.ny || K >= cb.nz) return;
  T sa = T(0), sb = T(0), sd = T(0);
#pragma unroll
  for (int n = 0; n < 8; ++n) {
    const long long q = cidx(fb, 2 * I + (n & 1), 2 * J + ((n >> 1) & 1), 2 * K + (n >> 2));
    sa += a[q];
    sb += b[q];
    sd += d[q];
  }
  const long long Q = cidx(cb, I, J, K);
  A[Q] = sa * T(0.125);
  B[Q] = sb * T(0.125);
  D[Q] = sd * T(0.125);
}

// All sweeps of a visit of the coarsest grid in one block: a few hundred cells take longer to launch than
// to sweep (30 launches a V-cycle). The iterate ping-pongs between the two buffers, a barrier between
// sweeps; the last one writes e = u' - u0 over u0. Measured for a three-level cycle with 30 sweeps, in one
// block and with a launch each: FP32 78 and 139 us at 64 cells, 101 and 126 at 512, 126 and 127 at 1024;
// FP64, bound by the one SM's FP64 pipe, 251 and 284 at 64, 262 and 284 at 128, 370 and 284 at 256.
constexpr int kCoarsestThreads = 512;
template <class T>
__global__ void __launch_bounds__(kCoarsestThreads) k_mg_coarsest(Box b, RxCoef<T> c, T romega, RxIn<T> in0,
                                                                  RxIn<T> in1, MgSrc<T> f, RxOut<T> out0,
                                                                  RxOut<T> out1, MgE<T> e0, int sweeps) {
  chain_begin();
  const int plane = b.nx * b.ny, n = plane * b.nz;
  for (int s = 0; s < sweeps; ++s) {
    const RxIn<T> in = (s & 1) ? in1 : in0;
    const RxOut<T> out = (s & 1) ? out0 : out1;
    const bool last = s == sweeps - 1;
    for (int t = threadIdx.x; t < n; t += kCoarsestThreads) {
      const int k = t / plane, r = t - k * plane, j = r / b.nx, i = r - j * b.nx;
      const long long q = cidx(b, i, j, k);
      const MgEq<T> e = mg_eq<T, true, true>(b, c, romega, in, f, q, i, j, k);
      const T Pf1 = in.Pf[q] + e.gP * rx_rcp(e.den);
      if (last) {
        e0.Pf[q] = Pf1 - e0.Pf[q];
        e0.phi[q] = e.phi1 - e0.phi[q];
        e0.Xs[q] = e.Xs1 - e0.Xs[q];
      } else {
        out.Pf[q] = Pf1;
        out.phi[q] = e.phi1;
        out.Xs[q] = e.Xs1;
      }
    }
    __syncthreads();
  }
}

template <class T>
bool mg_coarsest_fits(const Box& b) {
  return (long long)b.nx * b.ny * b.nz <= (sizeof(T) == 4 ? 512 : 128);
}

template <class T>
void mg_coarsest(cudaStream_t s, Box b, const RxCoef<T>& c, double omega, const RxIn<T>& in0, const RxIn<T>& in1,
                 const MgSrc<T>& fas, const RxOut<T>& out0, const RxOut<T>& out1, const MgE<T>& e0, int sweeps) {
  launch_chained(k_mg_coarsest<T>, 1, kCoarsestThreads, 0, s, b, c, (T)(1.0 / omega), in0, in1, fas, out0, out1, e0,
                 sweeps);
}

template <class T>
void mg_smooth(cudaStream_t s, Box b, const RxCoef<T>& c, double omega, const RxIn<T>& in, const MgSrc<T>* fas,
               const RxOut<T>& out, const MgE<T>* laste, unsigned long long* red, int check) {
  const T romega = (T)(1.0 / omega);
  const MgSrc<T> none{nullptr, nullptr, nullptr};
  const MgE<T> noe{nullptr, nullptr, nullptr};
  if constexpr (sizeof(T) == 4) {
    if (quads_pay(b)) {
      const Quads qd = quads_of(b);
      int zc;
      const dim3 g = quad_grid(qd, b.nz, kSmoothBlocks, &zc);
      if (!fas)
        launch_chained(k_mg_smooth4<false, false>, g, kQuadThreads, 0, s, b, c, romega, in, none, out, noe, red,
                       check, qd, zc);
      else if (!laste)
        launch_chained(k_mg_smooth4<true, false>, g, kQuadThreads, 0, s, b, c, romega, in, *fas, out, noe, red,
                       check, qd, zc);
      else
        launch_chained(k_mg_smooth4<true, true>, g, kQuadThreads, 0, s, b, c, romega, in, *fas, out, *laste, red,
                       check, qd, zc);
      return;
    }
  }
  const dim3 g = grid_of(b), blk(32, 8, 1);
  if (!fas)
    launch_chained(k_mg_smooth<T, false, false>, g, blk, 0, s, b, c, romega, in, none, out, noe, red, check);
  else if (!laste)
    launch_chained(k_mg_smooth<T, true, false>, g, blk, 0, s, b, c, romega, in, *fas, out, noe, red, check);
  else
    launch_chained(k_mg_smooth<T, true, true>, g, blk, 0, s, b, c, romega, in, *fas, out, *laste, red, check);
}

template <class T>
void mg_restrict(cudaStream_t s, Box fine, Box coarse, const RxCoef<T>& c, const RxIn<T>& in, const MgSrc<T>* fas,
                 const MgCoarse<T>& out) {
  const MgSrc<T> none{nullptr, nullptr, nullptr};
  if constexpr (sizeof(T) == 4) {
    if (quads_pay(fine)) {
      const int per_row = (fine.nx + 3) / 4;
      const QuadRows qr{per_row, 2 * per_row * coarse.ny};
      const unsigned gx = (unsigned)((qr.n + kQuadThreads - 1) / kQuadThreads);
      const int zc = march_chunk(gx, coarse.nz, kQuadChunk / 2, kRestrictBlocks, sm_count(), 1.0, 0.75);
      const dim3 g(gx, (unsigned)((coarse.nz + zc - 1) / zc), 1);
      if (fas)
        launch_chained(k_mg_restrict4<true>, g, kQuadThreads, 0, s, fine, coarse, c, in, *fas, out, qr, zc);
      else
        launch_chained(k_mg_restrict4<false>, g, kQuadThreads, 0, s, fine, coarse, c, in, none, out, qr, zc);
      return;
    }
  }
  const dim3 g((unsigned)((fine.nx + kRbx - 1) / kRbx), (unsigned)((fine.ny + kRby - 1) / kRby),
               (unsigned)((fine.nz + kRbz - 1) / kRbz));
  const dim3 blk(kRbx, kRby, kRbz);
  if (fas)
    launch_chained(k_mg_restrict<T, true>, g, blk, 0, s, fine, coarse, c, in, *fas, out);
  else
    launch_chained(k_mg_restrict<T, false>, g, blk, 0, s, fine, coarse, c, in, none, out);
}

template <class T>
void mg_coarse_rhs(cudaStream_t s, Box coarse, const RxCoef<T>& c, const RxIn<T>& u0, const MgCoarse<T>& out) {
  if constexpr (sizeof(T) == 4) {
    if (quads_pay(coarse)) {
      const Quads qd = quads_of(coarse);
      int zc;
      const dim3 g = quad_grid(qd, coarse.nz, kRestrictBlocks, &zc);
      launch_chained(k_mg_coarse_rhs4, g, kQuadThreads, 0, s, coarse, c, u0, out, qd, zc);
      return;
    }
  }
  launch_chained(k_mg_coarse_rhs<T>, grid_of(coarse), dim3(32, 8, 1), 0, s, coarse, c, u0, out);
}

template <class T>
void mg_prolong(cudaStream_t s, Box fine, Box coarse, const MgCorr<T>& e, T* Pf, T* phi, T* Xs) {
  const int per_row = (coarse.nx + 1) / 2;
  const dim3 g((unsigned)((per_row * coarse.ny + kProlongThreads - 1) / kProlongThreads), (unsigned)coarse.nz, 3);
  launch_chained(k_mg_prolong<T>, g, kProlongThreads, 0, s, fine, coarse, e, Pf, phi, Xs, per_row);
}

template <class T>
void mg_restrict_old(cudaStream_t s, Box fine, Box coarse, const T* Pf_o, const T* phi_o, const T* Xs_o, T* cPf_o,
                     T* cphi_o, T* cXs_o) {
  k_mg_restrict_old<T><<<grid_of(coarse), dim3(32, 8, 1), 0, s>>>(fine, coarse, Pf_o, phi_o, Xs_o, cPf_o, cphi_o,
                                                                  cXs_o);
}

#define MG_INSTANTIATE(T)                                                                                          \
  template void mg_smooth<T>(cudaStream_t, Box, const RxCoef<T>&, double, const RxIn<T>&, const MgSrc<T>*,        \
                             const RxOut<T>&, const MgE<T>*, unsigned long long*, int);                           \
  template void mg_restrict<T>(cudaStream_t, Box, Box, const RxCoef<T>&, const RxIn<T>&, const MgSrc<T>*,         \
                               const MgCoarse<T>&);                                                               \
  template void mg_coarse_rhs<T>(cudaStream_t, Box, const RxCoef<T>&, const RxIn<T>&, const MgCoarse<T>&);        \
  template bool mg_coarsest_fits<T>(const Box&);                                                                 \
  template void mg_coarsest<T>(cudaStream_t, Box, const RxCoef<T>&, double, const RxIn<T>&, const RxIn<T>&,       \
                               const MgSrc<T>&, const RxOut<T>&, const RxOut<T>&, const MgE<T>&, int);            \
  template void mg_prolong<T>(cudaStream_t, Box, Box, const MgCorr<T>&, T*, T*, T*);                             \
  template void mg_restrict_old<T>(cudaStream_t, Box, Box, const T*, const T*, const T*, T*, T*, T*);
MG_INSTANTIATE(double)
MG_INSTANTIATE(float)

}  // namespace pt
