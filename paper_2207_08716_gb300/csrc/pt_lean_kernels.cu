// pt_lean_kernels.cu — the FP64-lean form of one PT iteration (two kernels per iteration).
//
// GB300 issues 2 FP64 lanes per SM per clock (~1.26 TFLOP/s) against ~6.7 TB/s of HBM, so an
// FP64 PT iteration is bound by FP64 instructions, not bytes. This form therefore trades bytes
// for FP64 work wherever a quantity changes less often than every iteration:
//   * coefficients that depend only on mu, eta and the old stresses (which change at Picard
//     updates and step starts) are kept in arrays refreshed by k_lean_coef:
//       centres  cm2 = 2 mu / (1 + xi), toa_ii = tau_o_ii xi / (1 + xi), idtp = 1 / dtau_Pt,
//                ieta = 1 / eta
//       edges    em2 = 2 mu_e / (1 + xi_e), toa_e = tau_o_e xi_e / (1 + xi_e)
//       faces    dtv = dtau_V (mean of the two centres' values)
//     with xi = mu / (G dtS) (Eq. 21, backward-Euler Maxwell step);
//   * k = k0 e^logk (phi / phi0)^3 (Eq. 23) and w = 1 / (1 - phi) travel with phi: the
//     porosity update of iteration k writes them for iteration k+1;
//   * the log-space porosity update (Eq. 22) is L = Lo + delta, so
//       phi'  = phi_o - (1 - phi_o) expm1(delta),   1 / (1 - phi') = (1 / (1 - phi_o)) e^-delta,
//     with both exponentials from one Taylor polynomial of exp (|delta| is tiny; large |delta|
//     falls back to CUDA's expm1) — no exp, no division, no cancellation in 1 - e^L;
//   * the largest neighbour permeability (pseudo-time step of Pf) is found with 64-bit
//     integer compares of the positive doubles' bit patterns (exact, off the FP64 pipe).
// k_lean_cells: Darcy flux and divergence (Eq. 20), div V and numerical div V (Eq. 17),
// local-implicit Pt, Pf (Eqs. 17-18), stresses at centres and the cell's three lower edges
// (Eq. 21), porosity (Eq. 22). k_lean_faces: momentum residual (Eq. 19) with Pt^{k+1},
// damped R, V^{k+1}. k_lean_picard: Picard targets (Eqs. 24-26) with log-space relaxation.
#include "pt_df_body.cuh"
#include "pt_lean_body.cuh"

#include <algorithm>

namespace pt {

// ------------------------------------------------------------------------------ cells
// A thread takes a chunk of levels of its column (lean_cell_level's carried values). 94.5 FP64 instructions
// per cell at 191^3 (100.1 before the carried flux, the folded spacings and the shared difference of the
// new pressures), 1.22 ms a launch against 1.31; the pipe runs at 86 % either way.
constexpr int kLeanCellBlocks = 5;
__global__ void __launch_bounds__(kPlaneThreads, kLeanCellBlocks) k_lean_cells(Box b, LeanCoef<double> c,
                                                                               LeanCellIn<double> in,
                                                                               LeanCellOut<double> out,
                                                                               unsigned long long* red, int check,
                                                                               Plane pl, int zchunk) {
  chain_begin();
  int i, j;
  double r_pt = 0.0, r_pf = 0.0;
  if (plane_point(pl, i, j)) {
    const int k0 = blockIdx.y * zchunk, k1 = min(k0 + zchunk, b.nz);
    LeanColumn col = lean_column(b, c, in, i, j, k0);
    for (int k = k0; k < k1; ++k) lean_cell_level(b, c, in, out, i, j, k, check, col, r_pt, r_pf);
  }
  if (check) {
    block_max_atomic(r_pt, red + RED_PT);
    block_max_atomic(r_pf, red + RED_PF);
  }
}

// ------------------------------------------------- double-float cells, z-marching
// Each 32 x 8 block marches up a chunk of z-levels (march_chunk) of its column. Every array a level reads
// is copied by 16-byte cp.async into a shared-memory stage one level ahead (Pf, phi, k, Vz two, since
// level k reads them at k + 1), rows by warps: two arrays' 16 vectors of a row at a time, the row ends
// of all six neighbour arrays in one instruction, the halo rows above and below by six of the warps. So
// no load from global memory is waited for inside a level, neighbours come from shared memory by
// constant offsets, and one barrier per level separates a slot's readers from its refill. The Darcy
// flux through a z face is formed once and carried up. 111,616 B per block, 2 blocks per SM. At 239^3:
// 1.05 ms a launch when the neighbours were read from global memory (1929 instructions per cell, 55 % of
// the issue slots), 0.67 ms in this form (5.2 TB/s of its 256 B per cell, 0.77 of the copy peak).
constexpr int kLeanZChunk = 16;   // the longest chunk (32: the same at 383^3, 14.0 against 13.0 ms at 127^3)
constexpr int kZmarchBlocks = 2;

__device__ __forceinline__ void cp_async16(void* smem, const void* gmem) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(gmem) : "memory");
}

// The copies of one thread: pointers at level 0 (its row or halo row and column), places in the stage.
struct DfStager {
  const df64 *h3a, *h3b, *h2, *pw[kDfPoint / 2];   // pairs: the lower half-warp's array or the upper's
  const df64 *edge, *halo;
  int d_row, d_pw, d_edge, d_halo;                 // offsets into the stage
  bool ok_row, ok_edge, ok_halo, edge3, halo3;     // edge3, halo3: an array of three slots
};

__device__ __forceinline__ DfStager df_stager(const Box& b, const LeanCellIn<df64>& in, int i0, int j0) {
  const int lane = threadIdx.x, w = threadIdx.y, hi = lane >> 4, v = lane & 15;
  DfStager s;
  const int j = j0 + w, col = i0 + 2 * v;
  s.ok_row = j <= b.ny && col < b.px;
  const long long q = (long long)col + (long long)b.px * j;
  s.h3a = (hi ? in.phi : in.Pf) + q;
  s.h3b = (hi ? in.Vz : in.perm) + q;
  s.h2 = (hi ? in.Vy : in.Vx) + q;
  const df64* const p[kDfPoint] = {in.Pto, in.Pfo, in.phio, in.ieta, in.idtp, in.cm2, in.toa_xx, in.toa_yy,
                                   in.toa_zz, in.em2_xy, in.em2_xz, in.em2_yz, in.toa_xy, in.toa_xz, in.toa_yz,
                                   in.Pt};          // the order of the S_ slots
#pragma unroll
  for (int n = 0; n < kDfPoint / 2; ++n) s.pw[n] = (hi ? p[2 * n + 1] : p[2 * n]) + q;
  s.d_row = (w + 1) * kDfW + 2 + 2 * v;
  s.d_pw = kDfPW + hi * 256 + 32 * w + 2 * v;
  // row ends: lanes 0-11, array lane / 2, the vector left (even lanes) or right of the row
  const int a = lane >> 1, ec = (lane & 1) ? i0 + 32 : i0 - 2;
  s.edge3 = a < kDfHalo3;
  s.ok_edge = lane < 12 && j <= b.ny && ec >= 0 && ec < b.px;
  s.edge = (a == 0 ? in.Pf : a == 1 ? in.phi : a == 2 ? in.perm : a == 3 ? in.Vz : a == 4 ? in.Vx : in.Vy) + ec +
           (long long)b.px * j;
  s.d_edge = (s.edge3 ? a * 3 * kDfAR : kDfH2 + (a - kDfHalo3) * 2 * kDfAR) + (w + 1) * kDfW + ((lane & 1) ? 34 : 0);
  // halo rows: warps 0-5, one array each, the row below (lower half-warp) and above
  const int hj = hi ? j0 + 8 : j0 - 1;
  s.halo3 = w < kDfHalo3;
  s.ok_halo = w < 6 && hj >= 0 && hj <= b.ny && col < b.px;
  s.halo = (w == 0 ? in.Pf : w == 1 ? in.phi : w == 2 ? in.perm : w == 3 ? in.Vz : w == 4 ? in.Vx : in.Vy) + col +
           (long long)b.px * hj;
  s.d_halo = (s.halo3 ? w * 3 * kDfAR : kDfH2 + (w - kDfHalo3) * 2 * kDfAR) + (hi ? 9 * kDfW : 0) + 2 + 2 * v;
  return s;
}

// Level L of Pf, phi, k, Vz into slot m3 of three.
__device__ __forceinline__ void df_stage3(df64* st, const DfStager& s, long long pxy, int L, int m3) {
  const long long o = pxy * L;
  const int t = m3 * kDfAR, hi = threadIdx.x >> 4;
  if (s.ok_row) {
    cp_async16(st + t + hi * 3 * kDfAR + s.d_row, s.h3a + o);
    cp_async16(st + t + (2 + hi) * 3 * kDfAR + s.d_row, s.h3b + o);
  }
  if (s.ok_edge && s.edge3) cp_async16(st + t + s.d_edge, s.edge + o);
  if (s.ok_halo && s.halo3) cp_async16(st + t + s.d_halo, s.halo + o);
}
// Level L of Vx, Vy and the pointwise arrays into slot m2 of two.
__device__ __forceinline__ void df_stage2(df64* st, const DfStager& s, long long pxy, int L, int m2) {
  const long long o = pxy * L;
  const int t = m2 * kDfAR, hi = threadIdx.x >> 4;
  if (s.ok_row) {
    cp_async16(st + t + kDfH2 + hi * 2 * kDfAR + s.d_row, s.h2 + o);
#pragma unroll
    for (int n = 0; n < kDfPoint / 2; ++n) cp_async16(st + m2 * kDfPWSlot + n * 512 + s.d_pw, s.pw[n] + o);
  }
  if (s.ok_edge && !s.edge3) cp_async16(st + t + s.d_edge, s.edge + o);
  if (s.ok_halo && !s.halo3) cp_async16(st + t + s.d_halo, s.halo + o);
}

template <bool INNER>
__device__ __forceinline__ void df_cells_run(const Box& b, const LeanCoef<df64>& c, const LeanCellIn<df64>& in,
                                             const LeanCellOut<df64>& out, int i, int j, int k0, int k1, int check,
                                             df64* st, unsigned long long& m_pt, unsigned long long& m_pf) {
  const DfStager s = df_stager(b, in, i - (int)threadIdx.x, j - (int)threadIdx.y);
  df_stage3(st, s, b.pxy, k0, 0);
  df_stage3(st, s, b.pxy, k0 + 1, 1);
  df_stage2(st, s, b.pxy, k0, 0);
  asm volatile("cp.async.commit_group;\n" ::: "memory");
  DfColumn col;
  col.phi_d = col.k_d = col.vx_d = col.vy_d = col.fz = df64(0.0f, 0.0f);
  if (k0 > 0 && (INNER || (i <= b.nx && j <= b.ny))) {
    const long long q = cidx(b, i, j, k0), d = q - b.pxy;
    col.phi_d = in.phi[d];
    col.k_d = in.perm[d];
    col.vx_d = in.Vx[d];
    col.vy_d = in.Vy[d];
    // as df_cell_level forms it, so that both cells of a chunk's boundary take the same flux
    col.fz = (col.k_d + in.perm[q]) * (dfu::subn(in.Pf[q], in.Pf[d]) + c.buoy_dz);
  }
  const df64* const t3 = st + (threadIdx.y + 1) * kDfW + threadIdx.x + 2;
  const df64* const tp = st + kDfPW + 32 * threadIdx.y + threadIdx.x;
  int m3 = 0;                                       // slot of level k in the rings of three
  for (int k = k0; k < k1; ++k) {
    const int m2 = (k - k0) & 1, m3p = m3 == 2 ? 0 : m3 + 1, m3n = m3p == 2 ? 0 : m3p + 1;
    asm volatile("cp.async.wait_group 0;\n" ::: "memory");
    __syncthreads();   // level k's copies are visible, and every thread is done with level k - 1
    if (k + 1 < k1) {
      df_stage2(st, s, b.pxy, k + 1, m2 ^ 1);
      df_stage3(st, s, b.pxy, k + 2, m3n);          // k + 2 <= nz: a level of the box
    }
    asm volatile("cp.async.commit_group;\n" ::: "memory");
    df_cell_level<INNER>(b, c, in.K0, out, i, j, k, check, col, m_pt, m_pf, t3 + m3 * kDfAR, t3 + m3p * kDfAR,
                         t3 + kDfH2 + m2 * kDfAR, tp + m2 * kDfPWSlot);
    m3 = m3p;
  }
}

__global__ void __launch_bounds__(256, kZmarchBlocks) k_df_cells(Box b, LeanCoef<df64> c, LeanCellIn<df64> in,
                                                                 LeanCellOut<df64> out, unsigned long long* red,
                                                                 int check, int zchunk) {
  chain_begin();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  df64* const st = reinterpret_cast<df64*>(smem_raw);
  const int i = blockIdx.x * 32 + threadIdx.x;
  const int j = blockIdx.y * 8 + threadIdx.y;
  const int k0 = blockIdx.z * zchunk;
  const int k1 = min(k0 + zchunk, b.nz);
  const bool inner = blockIdx.x > 0 && blockIdx.y > 0 && (int)blockIdx.x * 32 + 32 < b.nx && (int)blockIdx.y * 8 + 8 < b.ny;
  unsigned long long m_pt = 0ull, m_pf = 0ull;     // norms as bit patterns: a NaN stays the largest
  if (inner) df_cells_run<true>(b, c, in, out, i, j, k0, k1, check, st, m_pt, m_pf);
  else df_cells_run<false>(b, c, in, out, i, j, k0, k1, check, st, m_pt, m_pf);
  if (check) {
    block_max_atomic(__longlong_as_double((long long)m_pt), red + RED_PT);
    block_max_atomic(__longlong_as_double((long long)m_pf), red + RED_PF);
  }
}

__global__ void __launch_bounds__(256) k_df_faces(Box b, LeanCoef<df64> c, LeanFaceIn<df64> in, df64* Vx,
                                                  df64* Vy, df64* Vz, df64* Rx, df64* Ry, df64* Rz,
                                                  unsigned long long* red, int check) {
  chain_begin();
  double r_v = 0.0;
  df_face_point(b, c, in, Vx, Vy, Vz, Rx, Ry, Rz, blockIdx.x * 32 + threadIdx.x, blockIdx.y * 8 + threadIdx.y,
                blockIdx.z, check, r_v);
  if (check) block_max_atomic(r_v, red + RED_V);
}

// ------------------------------------------------------------------------------ faces
__global__ void __launch_bounds__(kPlaneThreads) k_lean_faces(Box b, LeanCoef<double> c, LeanFaceIn<double> in,
                                                              double* Vx, double* Vy, double* Vz, double* Rx,
                                                              double* Ry, double* Rz, unsigned long long* red,
                                                              int check, Plane pl) {
  chain_begin();
  int i, j;
  double r_v = 0.0;
  if (plane_point(pl, i, j))
    lean_face_point(b, c, in, Vx, Vy, Vz, Rx, Ry, Rz, i, j, (int)blockIdx.y, check, r_v);
  if (check) block_max_atomic(r_v, red + RED_V);
}

// ------------------------------------------------------------------------------ Picard
template <class T>
__global__ void __launch_bounds__(kPlaneThreads) k_lean_picard(Box b, LeanCoef<T> c, LeanPicardIn<T> in,
                                                               T* mu, T* eta,
                                                               unsigned long long* red, Plane pl) {
  chain_begin();
  int i, j;
  double m = 1.0;
  if (plane_point(pl, i, j)) lean_picard_point(b, c, in, mu, eta, i, j, (int)blockIdx.y, m);
  block_max_log_atomic(m, red + RED_PIC);
}

// ---------------------------------------------------------------------- end-of-step stresses
// One pass over centres and edges with third-order reciprocals (the two step-by-step kernels divide
// by 1 + xi: 13.2 + 16.2 ms at 511^3).
__global__ void __launch_bounds__(256) k_lean_stresses(Box b, LeanCoef<double> c, StressCoef sc, StressIn in,
                                                       StressCentre ce, StressOut out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int j = blockIdx.y * blockDim.y + threadIdx.y;
  const int k = blockIdx.z;
  stress_edges_point(b, sc, in, out.txy, out.txz, out.tyz, i, j, k);
  if (i >= b.nx || j >= b.ny || k >= b.nz) return;
  const long long q = cidx(b, i, j, k);
  const double dvx = in.Vx[q + 1] - in.Vx[q], dvy = in.Vy[q + b.px] - in.Vy[q], dvz = in.Vz[q + b.pxy] - in.Vz[q];
  const double divV = fma(dvx, c.rdx, fma(dvy, c.rdy, dvz * c.rdz));
  double divVn = divV;
  if (c.beta_n != 0.0) {
    const double Pt = ce.Pt[q], Pf = ce.Pf[q];
    const double cc = c.compaction_on ? lean_detail::rcp_full(ce.eta[q] * (1.0 - ce.phi[q])) : 0.0;
    divVn = fma(Pt - Pf, cc, fma(-c.bd_rdt_a, Pf - ce.Pfo[q], fma(c.bd_rdt, Pt - ce.Pto[q], divV)));
  }
  double txx, tyy, tzz;
  centre_stresses(sc, in.mu[q], dvx, dvy, dvz, divV, divVn, in.txxo[q], in.tyyo[q], in.tzzo[q], txx, tyy, tzz);
  out.txx[q] = txx;
  out.tyy[q] = tyy;
  out.tzz[q] = tzz;
}
void lean_stresses(dim3 gr, dim3 bl, cudaStream_t st, Box b, const LeanCoef<double>& c, const StressCoef& sc,
                   const StressIn& in, const StressCentre& ce, const StressOut& out) {
  k_lean_stresses<<<gr, bl, 0, st>>>(b, c, sc, in, ce, out);
}

// --------------------------------------------------------------------- coefficient refresh
// From mu, eta and the raw old stresses (after a Picard update or a step start).
template <class T>
__global__ void __launch_bounds__(kPlaneThreads) k_lean_coef(Box b, LeanCoef<T> c, LeanCoefIn<T> in,
                                                             LeanCoefOut<T> out, Plane pl) {
  int i, j;
  if (plane_point(pl, i, j)) lean_coef_point(b, c, in, out, i, j, (int)blockIdx.y);
}

// ------------------------------------------------------------------------ step start
// phio = phi, Eo = 1 - phi, iEo = 1 / (1 - phi), w = iEo, k from phi; Pto, Pfo; max(mu).
template <class T>
__global__ void __launch_bounds__(256) k_lean_begin(Box b, LeanCoef<T> c, LeanBeginIn<T> in,
                                                    LeanBeginOut<T> out, unsigned long long* red) {
  using namespace lean_detail;
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int j = blockIdx.y * blockDim.y + threadIdx.y;
  const int k = blockIdx.z;
  double m = 0.0;
  if (i < b.nx && j < b.ny && k < b.nz) {
    const long long q = cidx(b, i, j, k);
    const T ph = in.phi[q];
    out.Pto[q] = in.Pt[q];
    out.Pfo[q] = in.Pf[q];
    out.phio[q] = ph;
    if constexpr (!LeanRecompute<T>::value) {   // the recomputing forms derive these from phi
      const T Eo = T(1.0) - ph;
      const T iEo = T(1.0) / Eo;
      out.Eo[q] = Eo;
      out.iEo[q] = iEo;
      out.w[q] = iEo;
    }
    out.perm[q] = (in.K0 ? in.K0[q] : c.k0r3) * ph * ph * ph;   // K0 = k0 e^logk / phi0^3
    m = to_d(in.mu[q]);
  }
  block_max_atomic(m, red + RED_MUMAX);
}

// K0 = k0r3 e^logk, k0r3 = k0 / phi0^3: k = K0 phi^3.
template <class T>
__global__ void k_lean_k0(Box b, double k0r3, const double* __restrict__ logk, T* __restrict__ K0) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int j = blockIdx.y * blockDim.y + threadIdx.y;
  const int k = blockIdx.z;
  if (i < b.nx && j < b.ny && k < b.nz) {
    const long long q = cidx(b, i, j, k);
    K0[q] = lean_detail::from_d<T>(k0r3 * exp(logk[q]));
  }
}

// ----------------------------------------------------------- FP64 <-> double-float copies
// Element-wise over whole padded boxes (padding included), one array per blockIdx.y.
__global__ void k_to_df64(DfCopy cp, long long n) {
  const double* __restrict__ src = cp.d[blockIdx.y];
  df64* __restrict__ dst = cp.f[blockIdx.y];
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x)
    dst[e] = df64(src[e]);
}
__global__ void k_from_df64(DfCopy cp, long long n) {
  double* __restrict__ dst = cp.d[blockIdx.y];
  const df64* __restrict__ src = cp.f[blockIdx.y];
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x)
    dst[e] = (double)src[e];
}

void df64_convert(cudaStream_t st, const DfCopy& cp, int narrays, long long n, bool to_df) {
  if (narrays <= 0) return;
  int sms = 152;
  int dev = 0;
  if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const long long want = (n + 255) / 256;
  const unsigned gx = (unsigned)std::max(1LL, std::min<long long>(want, 8LL * sms));
  const dim3 gr(gx, (unsigned)narrays, 1);
  if (to_df) k_to_df64<<<gr, 256, 0, st>>>(cp, n);
  else k_from_df64<<<gr, 256, 0, st>>>(cp, n);
}

// ---------------------------------------------------------------- math check (test aid)
// One of the hand-written device routines applied element-wise, so that each can be compared
// with CUDA's own functions and with its stated error bound (the kernels inline the same code).
__global__ void k_math_check(int fn, const double* __restrict__ a, const double* __restrict__ b,
                             double* __restrict__ out, long long n) {
  using namespace lean_detail;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x) {
    const double x = a[e], y = b ? b[e] : 0.0;
    double r = 0.0, p = 0.0, m = 0.0;
    switch (fn) {
      case MATH_RCP_PSEUDO: r = rcp_pseudo(x); break;
      case MATH_RCP_FULL: r = rcp_full(x); break;
      case MATH_EXPM1_POS: expm1_pair(x, p, m); r = p; break;
      case MATH_EXPM1_NEG: expm1_pair(x, p, m); r = m; break;
      case MATH_DF_ADD: r = (double)(df64(x) + df64(y)); break;
      case MATH_DF_SUB: r = (double)(df64(x) - df64(y)); break;
      case MATH_DF_MUL: r = (double)(df64(x) * df64(y)); break;
      case MATH_DF_FMA: r = (double)fma(df64(x), df64(y), df64(x)); break;
      case MATH_DF_RCP: r = (double)df_rcp(df64(x)); break;
      case MATH_DF_SQRT: r = (double)df_sqrt(df64(x)); break;
      case MATH_DF_ROOT: r = (double)df_root(df64(x), (int)y); break;
      case MATH_DF_EXPM1_POS: r = (double)df_expm1(df64(x)); break;
      case MATH_TO_FLOAT: r = (double)to_float(x); break;
      case MATH_HALF: r = half_of(x); break;
      case MATH_SQRT_FULL: r = sqrt_full(x); break;
      case MATH_ROOT_FULL: r = root_full(x, rcp_full(x), (int)y, root_series((int)y)); break;
      case MATH_DF_RCP_SUM: r = (double)dfu::rcp(dfu::add(df64(x), df64(y))); break;
      case MATH_DF_EXPM1_NEG: r = (double)df_expm1(-df64(x)); break;
      default: r = nan(""); break;
    }
    out[e] = r;
  }
}

void math_check(cudaStream_t st, int fn, const double* a, const double* b, double* out, long long n) {
  if (n <= 0) return;
  const unsigned g = (unsigned)std::min<long long>((n + 255) / 256, 4096);
  k_math_check<<<g, 256, 0, st>>>(fn, a, b, out, n);
}

// The wall indices i = nx, j = ny carry stress under a background shear only.
template <>
void lean_cells<double>(cudaStream_t st, Box b, const LeanCoef<double>& c, const LeanCellIn<double>& in,
                        const LeanCellOut<double>& out, unsigned long long* red, int check) {
  const Plane pl = plane_of(b, c.bg_on ? 1 : 0);
  const dim3 g = plane_grid(pl, 1);
  // the pipe is shared by an SM's blocks: a level takes as long as there are blocks on the SM. Up to some 30
  // waves of blocks even SMs count more than the carried level: chunks of 1 or 2 measured 5-7 % faster at
  // 63^3-80 x 90 x 100 and 1-3 % at 96^3 and 127^3 than up to 8, which are 0.5 % faster from 160^3 on
  const bool large = (long long)g.x * b.nz > 30LL * kLeanCellBlocks * sm_count();
  const int zc = large ? march_chunk(g.x, b.nz, 8, kLeanCellBlocks, sm_count(), 0.15, 0.3)
                       : march_chunk(g.x, b.nz, 2, kLeanCellBlocks, sm_count(), 0.05, 0.6);
  launch_chained(k_lean_cells, dim3(g.x, (unsigned)((b.nz + zc - 1) / zc)), kPlaneThreads, 0, st, b, c, in, out, red,
                 check, pl, zc);
}
// The double-float form: the wall indices i = nx, j = ny carry stress under a background shear only.
template <>
void lean_cells<df64>(cudaStream_t st, Box b, const LeanCoef<df64>& c, const LeanCellIn<df64>& in,
                      const LeanCellOut<df64>& out, unsigned long long* red, int check) {
  const int smem = kDfStageElems * (int)sizeof(df64), w = c.bg_on ? 1 : 0;
  cudaFuncSetAttribute(k_df_cells, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  const unsigned gx = (b.nx + w + 31) / 32, gy = (b.ny + w + 7) / 8;
  const int zc = march_chunk((long long)gx * gy, b.nz, kLeanZChunk, kZmarchBlocks, sm_count(), 1.0, 1.6);
  launch_chained(k_df_cells, dim3(gx, gy, (unsigned)((b.nz + zc - 1) / zc)), dim3(32, 8, 1), smem, st, b, c, in, out,
                 red, check, zc);
}
template <>
void lean_faces<df64>(cudaStream_t st, Box b, const LeanCoef<df64>& c, const LeanFaceIn<df64>& in, df64* Vx,
                      df64* Vy, df64* Vz, df64* Rx, df64* Ry, df64* Rz, unsigned long long* red, int check) {
  const dim3 g((unsigned)((b.nx + 31) / 32), (unsigned)((b.ny + 7) / 8), (unsigned)b.nz);
  launch_chained(k_df_faces, g, dim3(32, 8, 1), 0, st, b, c, in, Vx, Vy, Vz, Rx, Ry, Rz, red, check);
}
template <>
void lean_faces<double>(cudaStream_t st, Box b, const LeanCoef<double>& c, const LeanFaceIn<double>& in, double* Vx,
                        double* Vy, double* Vz, double* Rx, double* Ry, double* Rz, unsigned long long* red,
                        int check) {
  const Plane pl = plane_of(b, 0);
  launch_chained(k_lean_faces, plane_grid(pl, b.nz), kPlaneThreads, 0, st, b, c, in, Vx, Vy, Vz, Rx, Ry, Rz, red,
                 check, pl);
}
template <class T>
void lean_picard(cudaStream_t st, Box b, const LeanCoef<T>& c, const LeanPicardIn<T>& in, T* mu, T* eta,
                 unsigned long long* red) {
  const Plane pl = plane_of(b, 0);
  launch_chained(k_lean_picard<T>, plane_grid(pl, b.nz), kPlaneThreads, 0, st, b, c, in, mu, eta, red, pl);
}
template <class T>
void lean_coef(cudaStream_t st, Box b, const LeanCoef<T>& c, const LeanCoefIn<T>& in, const LeanCoefOut<T>& out) {
  const Plane pl = plane_of(b, c.bg_on ? 1 : 0);
  k_lean_coef<T><<<plane_grid(pl, b.nz), kPlaneThreads, 0, st>>>(b, c, in, out, pl);
}
template <class T>
void lean_begin(dim3 gr, dim3 bl, cudaStream_t st, Box b, const LeanCoef<T>& c, const LeanBeginIn<T>& in,
                const LeanBeginOut<T>& out, unsigned long long* red) {
  k_lean_begin<T><<<gr, bl, 0, st>>>(b, c, in, out, red);
}
template <class T>
void lean_k0(dim3 gr, dim3 bl, cudaStream_t st, Box b, double k0r3, const double* logk, T* K0) {
  k_lean_k0<T><<<gr, bl, 0, st>>>(b, k0r3, logk, K0);
}

template void lean_picard<double>(cudaStream_t, Box, const LeanCoef<double>&, const LeanPicardIn<double>&,
                                  double*, double*, unsigned long long*);
template void lean_coef<double>(cudaStream_t, Box, const LeanCoef<double>&, const LeanCoefIn<double>&,
                                const LeanCoefOut<double>&);
template void lean_begin<double>(dim3, dim3, cudaStream_t, Box, const LeanCoef<double>&, const LeanBeginIn<double>&,
                                 const LeanBeginOut<double>&, unsigned long long*);
template void lean_k0<double>(dim3, dim3, cudaStream_t, Box, double, const double*, double*);

template void lean_picard<df64>(cudaStream_t, Box, const LeanCoef<df64>&, const LeanPicardIn<df64>&,
                                  df64*, df64*, unsigned long long*);
template void lean_coef<df64>(cudaStream_t, Box, const LeanCoef<df64>&, const LeanCoefIn<df64>&,
                                const LeanCoefOut<df64>&);
template void lean_begin<df64>(dim3, dim3, cudaStream_t, Box, const LeanCoef<df64>&, const LeanBeginIn<df64>&,
                                 const LeanBeginOut<df64>&, unsigned long long*);
template void lean_k0<df64>(dim3, dim3, cudaStream_t, Box, double, const double*, df64*);

}  // namespace pt
