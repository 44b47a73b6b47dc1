// rx_kernels.cu — reactive porosity-wave solver (thesis Art. 3, Eqs. 8-10; appendix A.6 form):
// one fused pseudo-transient iteration per launch. Per cell it reads Pf and k = k0 (phi/phi0)^3
// (FP64: stored with phi; FP32: from phi) with their six neighbours (Darcy flux, k averaged to the
// faces), phi, Xs and the old step, and writes the next Pf, phi, Xs (FP64: and k(phi')): 6 arrays read
// and 3 written in FP32, 7 and 4 in FP64 (the rate dPf/dt only on check and final iterations). Divisions
// are refined hardware reciprocals (rx_rcp).
#include "rx_quad.cuh"
#include "rx.cuh"

namespace pt {

// The cell's own part of the iteration, given the Darcy divergence divq at the iterate. FP64 is bound by its
// pipe: three-instruction reciprocals and comparisons and products shared between the clamp, its slope, R
// and dphi took 128 x 125 x 512 from 1279 to 1202 us an iteration.
template <class T>
struct RxNew {
  T Pf, phi, Xs, R;
};
template <class T>
__device__ __forceinline__ RxNew<T> rx_cell(const RxCoef<T>& c, T dtau, T divq, T Pf, T ph, T Xs, T Pf_o, T phi_o,
                                            T Xs_o) {
  const T om = T(1) - ph, w = rx_rcp(om), ixs = rx_rcp(T(1) - Xs);
  const T xr = c.beta_x * Pf + c.half_xs;
  const bool pos = xr > T(0), below = xr < c.xs_max;    // Xs_eq is xr clamped to [0, xs_max]
  const T xseq = pos ? (below ? xr : c.xs_max) : T(0);
  const T dXs = (xseq - Xs) * c.rtau, t = ixs * dXs;
  const T rbp = rx_rcp(rx_bp(c, ph));
  const T so = c.sr_opdx * om, wr = w * c.reta;
  const T comp = Pf * wr;                               // -Pe / (eta (1 - phi)), Pe = -Pf
  RxNew<T> n;
  n.R = fma(so, t, -divq - comp) * rbp;
  const T dxs_dpf = pos && below ? c.beta_x : T(0);
  const T a = (wr - so * ixs * dxs_dpf * c.rtau) * rbp; // -dR/dPf of the cell's own terms
  n.Xs = (Xs_o + c.dt_tau * xseq) * c.r1dt_tau;
  n.Pf = Pf + dtau * (n.R - (Pf - Pf_o) * c.rdt) * rx_rcp(T(1) + dtau * (c.rdt + a));
  const T bphi = c.beta_d - c.beta_s * w;
  const T dphi = om * fma(bphi, n.R, fma(-c.opdx, t, comp));
  n.phi = rx_clamp(phi_o + c.dt * dphi, T(1e-4), T(1));
  return n;
}

// One cell per thread. FP64, bound by the FP64 pipe: k travels with phi, each cell writing k(phi') for the
// next iteration. FP32 recomputes k from phi and takes this form on small grids only (quads_pay).
template <class T>
__global__ void __launch_bounds__(kPlaneThreads) k_rx_iter(Box b, RxCoef<T> c, T dtau, RxIn<T> in, RxOut<T> out,
                                                           unsigned long long* red, int check, Plane pl) {
  chain_begin();
  int i, j;
  const int k = blockIdx.y;
  double chg = 0.0, kb = 0.0;
  if (plane_point(pl, i, j)) {
    const long long q = cidx(b, i, j, k);
    const long long px = b.px, pxy = b.pxy;
    constexpr bool kstored = sizeof(T) == 8;
    auto perm = [&](long long o) { return kstored ? in.k[o] : rx_perm(c, in.phi[o]); };
    const T Pf = in.Pf[q], ph = in.phi[q], Xs = in.Xs[q], kc = perm(q);
    // Darcy flux through the six faces, zero through the walls; z faces carry rho_f g
    T sx = T(0), sy = T(0), sz = T(0);
    if (i > 0) sx = (perm(q - 1) + kc) * (in.Pf[q - 1] - Pf);
    if (i < b.nx - 1) sx = fma(kc + perm(q + 1), in.Pf[q + 1] - Pf, sx);
    if (j > 0) sy = (perm(q - px) + kc) * (in.Pf[q - px] - Pf);
    if (j < b.ny - 1) sy = fma(kc + perm(q + px), in.Pf[q + px] - Pf, sy);
    if (k > 0) sz = (perm(q - pxy) + kc) * ((in.Pf[q - pxy] - Pf) + c.rhofg_dz);
    if (k < b.nz - 1) sz = fma(kc + perm(q + pxy), (in.Pf[q + pxy] - Pf) - c.rhofg_dz, sz);
    // div qD = -(1/2) sum_d [(k + k_r)(dPf_r) - (k_l + k)(dPf_l)] / d^2
    const T divq = T(-0.5) * fma(sx, c.rdx2, fma(sy, c.rdy2, sz * c.rdz2));
    const RxNew<T> n = rx_cell(c, dtau, divq, Pf, ph, Xs, in.Pf_o[q], in.phi_o[q], in.Xs_o[q]);
    const T k1 = rx_perm(c, n.phi);
    out.Pf[q] = n.Pf;
    out.phi[q] = n.phi;
    out.Xs[q] = n.Xs;
    if (kstored) out.k[q] = k1;
    if (out.R) out.R[q] = n.R;
    if (check) {
      chg = rx_change((double)rx_abs(n.phi - ph), (double)rx_abs(n.Pf - Pf) * (double)c.pf_iscale,
                      (double)rx_abs(n.Xs - Xs));
      kb = (double)(k1 * rx_rcp(rx_bp(c, n.phi)));
    }
  }
  if (check) {
    block_max_atomic(chg, red + RED_V);
    block_max_atomic(kb, red + RED_MUMAX);
  }
}

// FP32, bound by HBM: four cells per thread, marching z (rx_quad.cuh). At 255 x 255 x 1020 and 36 B per cell
// one cell per thread took 590 us an iteration (0.60 of the copy peak, checks included) and this takes 435
// (0.81); 75 of the difference is the change norm, which was FP64 arithmetic per cell. Four blocks of 128
// registers measured 4 % faster than five of 96; chunks of 32 levels 1 % faster than 16 here, and 2 % slower
// in the V-cycle.
constexpr int kIterBlocks = 4;
__global__ void __launch_bounds__(kQuadThreads, kIterBlocks) k_rx_iter4(Box b, RxCoef<float> c, float dtau,
                                                                        RxIn<float> in, RxOut<float> out,
                                                                        unsigned long long* red, int check, Quads qd,
                                                                        int zchunk) {
  chain_begin();
  int i, j;
  QuadChange chg{0u, 0u, 0u};
  int kb = 0;   // largest k / beta_P (not negative) as its bits; a NaN is the largest
  if (quad_point(qd, i, j)) {
    const int k0 = blockIdx.y * zchunk, k1 = min(k0 + zchunk, b.nz);
    QuadColumn col = quad_column(b, c, in.Pf, in.phi, i, j, k0);
    for (int k = k0; k < k1; ++k) {
      const long long q = cidx(b, i, j, k);
      const float4 Xs = quad_load(in.Xs, q), Pfo = quad_load(in.Pf_o, q), pho = quad_load(in.phi_o, q),
                   Xso = quad_load(in.Xs_o, q);
      float Pf[4], ph[4], div[4], kd[4];
      quad_level<false>(b, c, in.Pf, in.phi, i, j, k, col, Pf, ph, div, kd);
      float4 oP, oh, oX, oR;
#pragma unroll
      for (int v = 0; v < 4; ++v) {
        const float X = quad_get(Xs, v);
        const RxNew<float> n = rx_cell(c, dtau, -0.5f * div[v], Pf[v], ph[v], X, quad_get(Pfo, v), quad_get(pho, v),
                                       quad_get(Xso, v));
        quad_set(oP, v, n.Pf);
        quad_set(oh, v, n.phi);
        quad_set(oX, v, n.Xs);
        quad_set(oR, v, n.R);
        if (check && i + v < b.nx) {
          quad_max(chg.phi, n.phi - ph[v]);
          quad_max(chg.Pf, n.Pf - Pf[v]);
          quad_max(chg.Xs, n.Xs - X);
          kb = max(kb, __float_as_int(rx_perm(c, n.phi) * rx_rcp(rx_bp(c, n.phi))));
        }
      }
      quad_store(out.Pf, q, oP);
      quad_store(out.phi, q, oh);
      quad_store(out.Xs, q, oX);
      if (out.R) quad_store(out.R, q, oR);
    }
  }
  if (check) {
    block_max_atomic(quad_change(chg, c.pf_iscale), red + RED_V);
    block_max_atomic((double)__int_as_float(kb), red + RED_MUMAX);
  }
}

template <class T>
__global__ void __launch_bounds__(256) k_rx_kbmax(Box b, RxCoef<T> c, const T* phi,
                                                  unsigned long long* red) {
  chain_begin();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int j = blockIdx.y * blockDim.y + threadIdx.y;
  const int k = blockIdx.z;
  double kb = 0.0;
  if (i < b.nx && j < b.ny && k < b.nz) {
    const T ph = phi[cidx(b, i, j, k)];
    kb = (double)(rx_perm(c, ph) / rx_bp(c, ph));
  }
  block_max_atomic(kb, red + RED_MUMAX);
}

template <class T>
__global__ void __launch_bounds__(256) k_rx_begin(Box b, RxCoef<T> c, const double* __restrict__ Pf,
                                                  const double* __restrict__ phi, const double* __restrict__ Xs,
                                                  T* Pf1, T* phi1, T* Xs1, T* Pf_o, T* phi_o, T* Xs_o, T* k1) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int j = blockIdx.y * blockDim.y + threadIdx.y;
  const int k = blockIdx.z;
  if (i >= b.nx || j >= b.ny || k >= b.nz) return;
  const long long q = cidx(b, i, j, k);
  const T a = (T)Pf[q], p = (T)phi[q], x = (T)Xs[q];
  Pf1[q] = a; phi1[q] = p; Xs1[q] = x;
  Pf_o[q] = a; phi_o[q] = p; Xs_o[q] = x;
  if (k1) k1[q] = rx_perm(c, p);
}

template <class T>
__global__ void __launch_bounds__(256) k_rx_end(Box b, const T* __restrict__ Pf, const T* __restrict__ phi,
                                                const T* __restrict__ Xs, const T* __restrict__ R, double* Pf1,
                                                double* phi1, double* Xs1, double* R1) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int j = blockIdx.y * blockDim.y + threadIdx.y;
  const int k = blockIdx.z;
  if (i >= b.nx || j >= b.ny || k >= b.nz) return;
  const long long q = cidx(b, i, j, k);
  Pf1[q] = (double)Pf[q]; phi1[q] = (double)phi[q]; Xs1[q] = (double)Xs[q]; R1[q] = (double)R[q];
}

namespace {
dim3 rx_grid(const Box& b) {
  return dim3((unsigned)((b.nx + 31) / 32), (unsigned)((b.ny + 7) / 8), (unsigned)b.nz);
}
}  // namespace

template <class T>
void rx_iter(cudaStream_t s, Box b, const RxCoef<T>& c, double dtau, const RxIn<T>& in, const RxOut<T>& out,
             unsigned long long* red, int check) {
  if constexpr (sizeof(T) == 4) {
    if (quads_pay(b)) {
      const Quads qd = quads_of(b);
      int zc;
      const dim3 g = quad_grid(qd, b.nz, kIterBlocks, &zc);
      launch_chained(k_rx_iter4, g, kQuadThreads, 0, s, b, c, (float)dtau, in, out, red, check, qd, zc);
      return;
    }
  }
  const Plane pl = plane_of(b, 0);
  launch_chained(k_rx_iter<T>, plane_grid(pl, b.nz), kPlaneThreads, 0, s, b, c, (T)dtau, in, out, red, check, pl);
}
template <class T>
void rx_kbmax(cudaStream_t s, Box b, const RxCoef<T>& c, const T* phi, unsigned long long* red) {
  launch_chained(k_rx_kbmax<T>, rx_grid(b), dim3(32, 8, 1), 0, s, b, c, phi, red);
}
template <class T>
void rx_begin(cudaStream_t s, Box b, const RxCoef<T>& c, const double* Pf, const double* phi, const double* Xs,
              T* Pf1, T* phi1, T* Xs1, T* Pf_o, T* phi_o, T* Xs_o, T* k1) {
  k_rx_begin<T><<<rx_grid(b), dim3(32, 8, 1), 0, s>>>(b, c, Pf, phi, Xs, Pf1, phi1, Xs1, Pf_o, phi_o, Xs_o, k1);
}
template <class T>
void rx_end(cudaStream_t s, Box b, const T* Pf, const T* phi, const T* Xs, const T* R, double* Pf1, double* phi1,
            double* Xs1, double* R1) {
  k_rx_end<T><<<rx_grid(b), dim3(32, 8, 1), 0, s>>>(b, Pf, phi, Xs, R, Pf1, phi1, Xs1, R1);
}

#define RX_INSTANTIATE(T)                                                                                         \
  template void rx_iter<T>(cudaStream_t, Box, const RxCoef<T>&, double, const RxIn<T>&, const RxOut<T>&,         \
                           unsigned long long*, int);                                                            \
  template void rx_kbmax<T>(cudaStream_t, Box, const RxCoef<T>&, const T*, unsigned long long*);                \
  template void rx_begin<T>(cudaStream_t, Box, const RxCoef<T>&, const double*, const double*, const double*,   \
                            T*, T*, T*, T*, T*, T*, T*);                                                         \
  template void rx_end<T>(cudaStream_t, Box, const T*, const T*, const T*, const T*, double*, double*, double*,  \
                          double*);
RX_INSTANTIATE(double)
RX_INSTANTIATE(float)

}  // namespace pt
