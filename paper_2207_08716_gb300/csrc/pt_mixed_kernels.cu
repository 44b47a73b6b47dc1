// pt_mixed_kernels.cu — mixed precision (PT_FP32): FP32 PT iterations on the correction of an
// FP64 defect-correction loop.
//
// One outer iteration at the FP64 state u = (V, Pt, Pf, phi; mu, eta):
//   (i)   FP64 residuals of Eqs. 17-19 at u: r_Pt (numerical div V), r_Pf (fluid pressure),
//         r_F (momentum) — stored in FP32 as the right-hand side of the correction problem —
//         and their max-norms (k_mix_perm, k_mix_prepare, k_mix_faces);
//   (ii)  FP64 Picard update of mu, eta (Eqs. 24-26) from the stresses at u (k_mix_faces);
//   (iii) FP32 PT on the correction delta = (dV, dPt, dPf) of the system linearised at u with
//         frozen coefficients (k, 1/(eta(1-phi)), mu, pseudo-time steps): the same damped,
//         local-implicit scheme as the FP64 iteration, iterating on the small correction so
//         that FP32 keeps its relative precision on it (k_corr_iteration, one pass per iteration);
//   (iv)  u <- u + delta in FP64 (k_mix_update), then the porosity time integration of
//         Eq. 22 in FP64 (log space) from the corrected pressures and velocities.
// Converged when the FP64 residual max-norms and the Picard change are below tol.
#include "pt_mixed.cuh"
#include "pt_lean_body.cuh"
#include "../../include/porowave_pt.h"

#include <type_traits>

namespace pt {

// The outer phases run on the FP64 pipe (2 lanes per SM and clock), so they are written to its
// instruction count: coefficients folded on the host (LeanCoef), fused multiply-adds, third-order
// reciprocals and no division, the porosity by expm1 of its small increment, norms through bit patterns.
// At 255^3 an outer iteration's phases took 13.0 ms (141 FP64 instructions per cell in k_mix_prepare
// alone, 137 in the Picard update, 67 at the edges); now 7.8 ms: 101 in k_mix_prepare with the edges, 83 in
// k_mix_faces with the Picard update, 36 in k_mix_porosity, the pipe at 82-84 %. Conversions on the integer
// units, powers of two folded into coefficients and fewer products gave the last 1.2 ms.

// k of the iterate (Eq. 23), read with its neighbours by mix_prepare_point.
__device__ __forceinline__ void mix_perm_point(const Box& b, const LeanCoef<double>& c, const double* phi,
                                               const double* logk, double* perm, int i, int j, int k) {
  if (i >= b.nx || j >= b.ny || k >= b.nz) return;
  const long long q = cidx(b, i, j, k);
  const double ph = phi[q], k3 = c.k0r3 * ph * ph * ph;
  perm[q] = logk ? k3 * exp(logk[q]) : k3;
}

// (i) FP64 residuals at cell centres, stresses at u (centres and lower edges), and the frozen
// coefficients of the correction problem (in FP32).
__device__ __forceinline__ void mix_prepare_point(const Box& b, const LeanCoef<double>& c, const StressCoef& sc,
                                                  const MixPrepIn& in, const MixPrepOut& out, int i, int j, int k,
                                                  double& r_pt, double& r_pf) {
  using namespace lean_detail;
  stress_edges_point(b, sc, in.s, out.txy, out.txz, out.tyz, i, j, k);
  if (i < b.nx && j < b.ny && k < b.nz) {
    const long long q = cidx(b, i, j, k);
    const long long px = b.px, pxy = b.pxy;
    const double Pt = in.Pt[q], Pf = in.Pf[q], ph = in.phi[q], mu = in.s.mu[q];
    const double dPt = Pt - in.Pto[q], dPf = Pf - in.Pfo[q], dpp = Pt - Pf;
    const double dvx = in.s.Vx[q + 1] - in.s.Vx[q], dvy = in.s.Vy[q + px] - in.s.Vy[q];
    const double dvz = in.s.Vz[q + pxy] - in.s.Vz[q];
    const double divV = fma(dvx, c.rdx, fma(dvy, c.rdy, dvz * c.rdz));
    const double cc = c.compaction_on ? rcp_full(in.eta[q] * (1.0 - ph)) : 0.0;
    const double divVn = fma(dpp, cc, fma(-c.bd_rdt_a, dPf, fma(c.bd_rdt, dPt, divV)));
    const double kc = in.perm[q];
    double sx = 0.0, sy = 0.0, sz = 0.0;
    if (i > 0) sx = -(in.perm[q - 1] + kc) * (Pf - in.Pf[q - 1]);
    if (i < b.nx - 1) sx = fma(kc + in.perm[q + 1], in.Pf[q + 1] - Pf, sx);
    if (j > 0) sy = -(in.perm[q - px] + kc) * (Pf - in.Pf[q - px]);
    if (j < b.ny - 1) sy = fma(kc + in.perm[q + px], in.Pf[q + px] - Pf, sy);
    if (k > 0) sz = -(in.perm[q - pxy] + kc) * ((Pf - in.Pf[q - pxy]) + c.buoy_dz);
    if (k < b.nz - 1) sz = fma(kc + in.perm[q + pxy], (in.Pf[q + pxy] - Pf) + c.buoy_dz, sz);
    const double divqD = -fma(sx, c.hrdx2, fma(sy, c.hrdy2, sz * c.hrdz2));
    const double rpf = fma(-dpp, cc, fma(-c.bd_rdt_a, dPt, fma(c.bda_B_rdt, dPf, divqD)));
    // stresses at u (Eq. 21) for the momentum residual and the Picard update
    double txx, tyy, tzz;
    centre_stresses(sc, mu, dvx, dvy, dvz, divV, divVn, in.s.txxo[q], in.s.tyyo[q], in.s.tzzo[q], txx, tyy, tzz);
    out.txx[q] = txx;
    out.tyy[q] = tyy;
    out.tzz[q] = tzz;
    // right-hand side and frozen coefficients of the correction problem (the iteration derives
    // 1/dtau_Pf from the largest neighbour k and the local-implicit denominators itself)
    out.r_pt[q] = to_float(divVn);
    out.r_pf[q] = to_float(rpf);
    out.cc[q] = to_float(cc);
    out.perm[q] = to_float(kc);
    out.idtp[q] = to_float(rcp_full(c.dtaupt_fac * mu));
    r_pt = divVn;
    r_pf = rpf;
  }
}

// (i) FP64 momentum residual at u (Eq. 19), stored in FP32; its max-norm. (ii) Picard update of mu and
// eta from the stresses at u, and the correction problem's mu and velocity pseudo-step dtau_V = fac / mu
// at centres in FP32 (the iteration forms 2 mu/(1+xi) at centres and edges and the face pseudo-steps
// from them).
__device__ __forceinline__ void mix_faces_point(const Box& b, const LeanCoef<double>& c, const MixFaceIn& in,
                                                const MixFaceOut& out, int i, int j, int k, double& r_v,
                                                double& pic) {
  using namespace lean_detail;
  if (i >= b.nx || j >= b.ny || k >= b.nz) return;   // the faces i = nx, j = ny, k = nz are walls
  const long long q = cidx(b, i, j, k);
  const long long px = b.px, pxy = b.pxy;
  const LeanPicardIn<double>& t = in.s;
  const double txx = t.txx[q], tyy = t.tyy[q], tzz = t.tzz[q], txy = t.txy[q], txz = t.txz[q], tyz = t.tyz[q];
  const double Pt = t.Pt1[q];
  if (i > 0) {
    const double F = fma(txx - t.txx[q - 1], c.rdx,
                         fma(t.txy[q + px] - txy, c.rdy, fma(t.txz[q + pxy] - txz, c.rdz, -((Pt - t.Pt1[q - 1]) * c.rdx))));
    out.rfx[q] = to_float(F);
    r_v = F;
  }
  if (j > 0) {
    const double F = fma(t.txy[q + 1] - txy, c.rdx,
                         fma(tyy - t.tyy[q - px], c.rdy, fma(t.tyz[q + pxy] - tyz, c.rdz, -((Pt - t.Pt1[q - px]) * c.rdy))));
    out.rfy[q] = to_float(F);
    r_v = abs_max(r_v, F);
  }
  if (k > 0) {
    const double rog = (0.5 * (t.phi1[q - pxy] + t.phi1[q]) - c.phi0) * c.drho_g;
    const double F = fma(t.txz[q + 1] - txz, c.rdx, fma(t.tyz[q + px] - tyz, c.rdy,
                         fma(tzz - t.tzz[q - pxy], c.rdz, fma(-(Pt - t.Pt1[q - pxy]), c.rdz, -rog))));
    out.rfz[q] = to_float(F);
    r_v = abs_max(r_v, F);
  }
  lean_picard_point(b, c, t, in.mu, in.eta, i, j, k, pic);
  const double mu = in.mu[q];
  out.mu[q] = to_float(mu);
  out.dtvc[q] = to_float(c.dtauv_fac * rcp_full(mu));
}

// phi^{k+1} = 1 - (1 - phi_o) exp(delta) at the corrected state, delta = -[beta_phi ((Pf1 - Pfo) -
// (Pt1 - Pto)) + dt ((Pf1 - Pt1) / eta + V . grad(1 - phi) / (1 - phi))] (Eq. 22 in log space).
__device__ __forceinline__ void mix_porosity_point(const Box& b, const LeanCoef<double>& c, const MixPorosity& p,
                                                   int i, int j, int k) {
  using namespace lean_detail;
  if (i >= b.nx || j >= b.ny || k >= b.nz) return;
  const long long q = cidx(b, i, j, k);
  const long long px = b.px, pxy = b.pxy;
  const double ph = p.phi[q], om = 1.0 - ph;
  double ax = 0.0, ay = 0.0, az = 0.0;
  if (i > 0) ax = p.Vx[q] * (ph - p.phi[q - 1]);
  if (i < b.nx - 1) ax = fma(p.Vx[q + 1], p.phi[q + 1] - ph, ax);
  if (j > 0) ay = p.Vy[q] * (ph - p.phi[q - px]);
  if (j < b.ny - 1) ay = fma(p.Vy[q + px], p.phi[q + px] - ph, ay);
  if (k > 0) az = p.Vz[q] * (ph - p.phi[q - pxy]);
  if (k < b.nz - 1) az = fma(p.Vz[q + pxy], p.phi[q + pxy] - ph, az);
  const double adv = -fma(ax, c.hrdx, fma(ay, c.hrdy, az * c.hrdz));   // times 1 / (1 - phi)
  const double pt1 = p.Pt1[q], pf1 = p.Pf1[q], eta = p.eta[q];
  const double r = rcp_full(om * eta);                                 // both quotients from one reciprocal
  const double comp = c.compaction_on ? (pf1 - pt1) * om : 0.0;
  const double rate = fma(adv, eta, comp) * r;
  const double dP = (pf1 - p.Pfo[q]) - (pt1 - p.Pto[q]);
  double em, unused;
  expm1_pair(-fma(c.beta_phi, dP, c.dt * rate), em, unused);
  const double phio = p.phio[q];
  p.phi1[q] = fma(phio - 1.0, em, phio);
}

__global__ void __launch_bounds__(kPlaneThreads) k_mix_begin(Box b, const double* __restrict__ Pt,
                                                             const double* __restrict__ Pf,
                                                             const double* __restrict__ phi,
                                                             const double* __restrict__ mu, double* __restrict__ Pto,
                                                             double* __restrict__ Pfo, double* __restrict__ phio,
                                                             unsigned long long* red, Plane pl) {
  int i, j;
  double m = 0.0;
  if (plane_point(pl, i, j)) {
    const long long q = cidx(b, i, j, (int)blockIdx.y);
    Pto[q] = Pt[q];
    Pfo[q] = Pf[q];
    phio[q] = phi[q];
    m = mu[q];
  }
  block_max_atomic(m, red + RED_MUMAX);
}

__global__ void __launch_bounds__(kPlaneThreads) k_mix_perm(Box b, LeanCoef<double> c, const double* phi,
                                                            const double* logk,
                                                            double* perm, Plane pl) {
  chain_begin();
  int i, j;
  if (plane_point(pl, i, j)) mix_perm_point(b, c, phi, logk, perm, i, j, (int)blockIdx.y);
}

__global__ void __launch_bounds__(kPlaneThreads) k_mix_porosity(Box b, LeanCoef<double> c, MixPorosity p, Plane pl) {
  chain_begin();
  int i, j;
  if (plane_point(pl, i, j)) mix_porosity_point(b, c, p, i, j, (int)blockIdx.y);
}

__global__ void __launch_bounds__(kPlaneThreads) k_mix_prepare(Box b, LeanCoef<double> c, StressCoef sc,
                                                               MixPrepIn in, MixPrepOut out, unsigned long long* red,
                                                               Plane pl) {
  chain_begin();
  int i, j;
  double r_pt = 0.0, r_pf = 0.0;
  if (plane_point(pl, i, j)) mix_prepare_point(b, c, sc, in, out, i, j, (int)blockIdx.y, r_pt, r_pf);
  block_max_atomic(lean_detail::abs_max(r_pt, 0.0), red + RED_PT);
  block_max_atomic(lean_detail::abs_max(r_pf, 0.0), red + RED_PF);
}

__global__ void __launch_bounds__(kPlaneThreads) k_mix_faces(Box b, LeanCoef<double> c, MixFaceIn in, MixFaceOut out,
                                                             unsigned long long* red, Plane pl) {
  chain_begin();
  int i, j;
  double r_v = 0.0, pic = 1.0;
  if (plane_point(pl, i, j)) mix_faces_point(b, c, in, out, i, j, (int)blockIdx.y, r_v, pic);
  block_max_atomic(lean_detail::abs_max(r_v, 0.0), red + RED_V);
  block_max_log_atomic(pic, red + RED_PIC);
}

// (iii) one FP32 PT iteration on the correction in a single pass.
//
// The iteration's two halves depend on each other across neighbours: the faces (momentum,
// damped R, dV) of level k read the cells' stresses and new dPt at k and k-1 (own cell, x- and
// y-neighbours below) and the edge stresses at k and k+1 (own edge, x- and y-neighbours above).
// A block of 32 x rows threads owns a tile of 30 x (rows - 2) faces and cells and marches up a column of face levels:
// at level L every thread computes the cell and the three lower edges at its index for the tile
// plus a one-cell halo on each side (the halo is recomputed by the neighbouring tiles' blocks from
// the same inputs, bit for bit). Stresses and the new dPt never go to global memory: per cell the
// pass reads dV, dPt, dPf, R, the right-hand sides and the frozen cc, k, 1/dtau_Pt, mu, dtau_V (18
// arrays) and writes dV', dPt', dPf', R (8 arrays): 104 B per cell. dV is read from one buffer and
// written to another (other blocks' halos still read the old dV). The pseudo-step of dPf (largest
// neighbour k), the local-implicit denominators, 2 mu/(1+xi) at centres and edges (mean of the
// four centres' mu) and the face pseudo-steps (mean of the two centres') are formed here.
//
// What bounds it is instruction issue and the latency between block barriers, not DRAM, so:
//   * one barrier per level: in the interval of level L a thread computes the faces of level L - 2
//     and then the cell and edges of level L, which no thread reads before the next barrier;
//   * a point's own values of the levels below (stresses, dV, the Darcy flux through the lower z
//     face) are carried in registers, x-neighbours of the stresses come by warp shuffle (a warp is a
//     row of the tile), so that only tyy, dPt' and the xy and yz edge stresses, which the row above
//     or below reads, go through shared memory (rings of three levels);
//   * the 12 arrays read at a point's own index and its x- and y-neighbours' are staged by 16-byte
//     cp.async one level ahead: a row of a tile is 9 aligned vectors, so that a level takes 4 copies of
//     27 lanes per warp instead of 12 of 32. dVz, dPf and k run one level further ahead (the cell of
//     level L reads them at L + 1), dtau_V two levels behind (the faces' level);
//   * the faces' own R and right-hand side are loaded an interval before their use;
//   * every ring has three slots and the loop takes three levels per turn, so that slots are constants
//     and the carried values change names instead of registers;
//   * tiles that touch no wall in x and y (INNER) take no wall tests; the z tests are uniform. A sweep
//     without damping neither reads nor keeps R (nothing reads it before an evaluation writes it).
// Measured at 511^3: 4.83 ms a sweep with two barriers a level, every neighbour from shared memory and
// 32 x 8 blocks; 3.08 ms in this form (4.5 TB/s of its 104 B per cell, 0.67 of the copy peak; at
// 239^3 546 thread instructions per cell against 791, issue slots 58 % busy).
constexpr int kCorrTX = 30;
constexpr int kCorrZChunk = 64; // the longest column of a block
constexpr int kCorrW = 36;      // floats of a staged row: 32 points and up to 3 in front (16-byte alignment)
// Staged arrays, in units of one level's tile (rows of kCorrW), three slots each: a level's
// slot is its distance from the column's first level modulo 3 (DTV: the slot of the level above).
enum { C_VX = 0, C_VY = 3, C_PT = 6, C_CC = 9, C_IDTP = 12, C_RPT = 15, C_RPF = 18, C_DTV = 21, C_MU = 24, C_VZ = 27,
       C_K = 30, C_PF = 33, kCorrStage = 36 };
enum { R_TYY, R_P, R_XY, R_YZ, kCorrRing };   // values the neighbouring rows read, three levels each
// ROWS: rows (warps) of a block, the tile's and a halo row on each side; BLOCKS per SM asked of the
// register allocator.
template <int ROWS, int BLOCKS>
struct CorrShape {
  static constexpr int rows = ROWS, blocks = BLOCKS, threads = 32 * ROWS, ty = ROWS - 2;
  static constexpr int smem = (kCorrStage * kCorrW + 3 * kCorrRing * 32) * ROWS * (int)sizeof(float);
};
// A step of 60 sweeps at 511^3 and one of 240 at 96^3: 10 rows, 2 blocks of 96 registers 340 and 12.2 ms;
// 8 rows, 3 blocks (80 registers) 343 and 13.8; 12 rows, 2 blocks 352 and 12.9; 10 rows, 3 blocks
// (64 registers, spilling) 460 and 18.1. The ensemble engine's tile is part of its interface (30 x 6).
using CorrSingle = CorrShape<10, 2>;
using CorrBatch = CorrShape<8, 3>;

__device__ __forceinline__ void corr_cp16(float* smem, const float* gmem) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(gmem) : "memory");
}

// a / b for b far inside the normal range: the hardware's approximate reciprocal (1 ulp) times a
__device__ __forceinline__ float corr_div(float a, float b) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(b));
  return a * r;
}
// 2 m / (1 + m / (G dtS)) of the viscosity m, and of the mean of four given their sum
__device__ __forceinline__ float corr_modulus(const CorrCoef<float>& c, float m) {
  return corr_div(2.0f * m, fmaf(m, c.rG, 1.0f));
}
__device__ __forceinline__ float corr_modulus4(const CorrCoef<float>& c, float sum) {
  return corr_div(0.5f * sum, fmaf(sum, 0.25f * c.rG, 1.0f));
}

// One tile of the iteration: faces and cells of columns [tbx kCorrTX, +kCorrTX) x [tby kCorrTY,
// +kCorrTY) and face levels [k0, ke), ke <= nz (the level nz holds walls only), by a 32 x SH::rows
// block whose dynamic shared memory (SH::smem) starts at corr_smem. Leaves no copy in flight:
// the block may start another tile after a barrier.
template <class SH, bool INNER>
__device__ __forceinline__ void corr_tile_run(const Box& b, const CorrCoef<float>& c, const CorrIn<float>& in,
                                              const CorrOut<float>& out, int tbx, int tby, int k0, int ke,
                                              unsigned long long* red, int check, float* corr_smem) {
  using T = float;
  constexpr int kCorrTY = SH::ty;
  constexpr int AR = SH::rows * kCorrW;
  const int tx = threadIdx.x, ty = threadIdx.y;
  const int i0 = tbx * kCorrTX - 1;
  const int i = i0 + tx;
  const int j = tby * kCorrTY - 1 + ty;
  const int ga = i0 & ~3;                       // first staged column (a multiple of 4; -4 for the first tile)
  const int ipx = b.px, ipxy = (int)b.pxy;      // the host keeps the box below 2^31 elements
  const bool row_own = ty >= 1 && ty <= kCorrTY;           // uniform over a warp
  const bool own = row_own && tx >= 1 && tx <= kCorrTX && (INNER || (i < b.nx && j < b.ny));
  // this thread's place in a staged tile and in a ring level
  const float* const st = corr_smem + ty * kCorrW + (i0 - ga) + tx;
  float* const ring = corr_smem + kCorrStage * AR + ty * 32 + tx;
  constexpr int RA = SH::rows * 32, RL = kCorrRing * RA;   // one ring array, one level of the rings

  // ---- staging: lanes 0-26 copy three arrays' rows of 9 vectors in each of four rounds
  const int sub = tx / 9, vec = tx - 9 * sub;
  const int col = ga + 4 * vec;
  const bool cp_ok = tx < 27 && j >= 0 && j <= b.ny && col >= 0 && col < b.px;
  const int cq = col + ipx * j;
  const float* const g0 = (sub == 0 ? in.Vx : sub == 1 ? in.Vy : in.Pt) + cq;
  const float* const g1 = (sub == 0 ? in.cc : sub == 1 ? in.idtp : in.r_pt) + cq;
  const float* const g2 = (sub == 0 ? in.r_pf : sub == 1 ? in.dtvc : in.mu) + cq;
  const float* const g3 = (sub == 0 ? in.Vz : sub == 1 ? in.perm : in.Pf) + cq;
  float* const sdst = corr_smem + 3 * sub * AR + ty * kCorrW + 4 * vec;
  static_assert(C_VY == 3 && C_PT == 6 && C_CC == 9 && C_RPF == 18 && C_VZ == 27, "a round's three arrays in order");
  const int lag2 = sub == 1 ? 2 : 0;            // DTV is staged two levels behind
  // level L of every array but VZ, K, PF (and DTV at L - 2) into slot s; level L of VZ, K, PF
  auto stage_a = [&](int s, int L) {
    if (!cp_ok) return;
    if (L >= 0 && L <= b.nz) {
      corr_cp16(sdst + (C_VX + s) * AR, g0 + ipxy * L);
      corr_cp16(sdst + (C_CC + s) * AR, g1 + ipxy * L);
    }
    const int M = L - lag2;
    if (M >= 0 && M <= b.nz) corr_cp16(sdst + (C_RPF + s) * AR, g2 + ipxy * M);
  };
  auto stage_b = [&](int s, int L) {
    if (cp_ok && L >= 0 && L <= b.nz) corr_cp16(sdst + (C_VZ + s) * AR, g3 + ipxy * L);
  };

  unsigned r_pt = 0u, r_pf = 0u, r_v = 0u;      // norms as bit patterns of |x|: a NaN stays the largest
  auto keep_max = [](unsigned& m, float x) { m = max(m, __float_as_uint(fabsf(x))); };

  // ---- carried up the column
  T vx1 = T(0), vy1 = T(0), vz1 = T(0), vx2 = T(0), vy2 = T(0), vz2 = T(0);   // dV at L - 1, L - 2
  T mux1 = T(0), muy1 = T(0);                   // mu of this cell plus its x- / y-neighbour's at L - 1
  T k1 = T(0), fz1 = T(0);                      // k at L - 1; Darcy flux term through the face L - 1/2
  T txx1 = T(0), tyy1 = T(0), tzz1 = T(0), P1 = T(0), exy1 = T(0), exz1 = T(0), eyz1 = T(0);   // level L - 1
  T txx2 = T(0), tyy2 = T(0), tzz2 = T(0), P2 = T(0), exy2 = T(0), exz2 = T(0), eyz2 = T(0);   // level L - 2
  T tzz3 = T(0), P3 = T(0), dtv_zm = T(0);      // level L - 3
  T rfx = T(0), rfy = T(0), rfz = T(0), Rx0 = T(0), Ry0 = T(0), Rz0 = T(0);   // the faces of level L - 2
  const bool own_fx = own && (INNER || i > 0), own_fy = own && (INNER || j > 0);
  const bool damped = c.damp_x != T(0) || c.damp_y != T(0) || c.damp_z != T(0);
  const bool keep_R = damped || out.eval;

  stage_a(0, k0 - 1);
  stage_b(0, k0 - 1);
  stage_b(1, k0);
  asm volatile("cp.async.commit_group;\n" ::: "memory");

  // the interval of level L, whose slot is s = (L - k0 + 1) mod 3
  auto level = [&](auto slot, int L) {
    constexpr int s = decltype(slot)::value, sp = (s + 1) % 3, sm = (s + 2) % 3;   // slots of L, L + 1, L + 2
    asm volatile("cp.async.wait_group 0;\n" ::: "memory");   // this thread's copies have landed
    // every thread's copies and ring values are visible, and every thread is done with the interval
    // before: the slots refilled below
    __syncthreads();
    if (L <= ke) stage_a(sp, L + 1);
    if (L + 2 <= ke) stage_b(sm, L + 2);
    asm volatile("cp.async.commit_group;\n" ::: "memory");

    // ---------------- faces of level F = L - 2
    const int F = L - 2;
    const float* const dv = st + (C_DTV + s) * AR;
    const T dtv_c = dv[0];
    if (F >= k0 && row_own) {
      const float* const rg = ring + sp * RL;       // ring level F
      const T txx_l = __shfl_up_sync(0xffffffffu, txx2, 1), P_l = __shfl_up_sync(0xffffffffu, P2, 1);
      const T exy_r = __shfl_down_sync(0xffffffffu, exy2, 1), exz_r = __shfl_down_sync(0xffffffffu, exz2, 1);
      const T exy_u = rg[R_XY * RA + 32], eyz_u = rg[R_YZ * RA + 32];
      const T tyy_d = rg[R_TYY * RA - 32], P_d = rg[R_P * RA - 32];
      const int q = i + ipx * j + ipxy * F;
      if (own_fx) {
        const T Fx = rfx + (txx2 - txx_l) * c.rdx + (exy_u - exy2) * c.rdy + (exz1 - exz2) * c.rdz - (P2 - P_l) * c.rdx;
        const T R1 = Fx * c.rrho_i + c.damp_x * Rx0;
        if (keep_R) out.Rx[q] = R1;
        if (!out.eval) out.Vx[q] = vx2 + T(0.5) * (dv[-1] + dtv_c) * R1;
        if (check) keep_max(r_v, Fx);
      }
      if (own_fy) {
        const T Fy = rfy + (exy_r - exy2) * c.rdx + (tyy2 - tyy_d) * c.rdy + (eyz1 - eyz2) * c.rdz - (P2 - P_d) * c.rdy;
        const T R1 = Fy * c.rrho_i + c.damp_y * Ry0;
        if (keep_R) out.Ry[q] = R1;
        if (!out.eval) out.Vy[q] = vy2 + T(0.5) * (dv[-kCorrW] + dtv_c) * R1;
        if (check) keep_max(r_v, Fy);
      }
      if (own && F > 0) {
        const T Fz = rfz + (exz_r - exz2) * c.rdx + (eyz_u - eyz2) * c.rdy + (tzz2 - tzz3) * c.rdz - (P2 - P3) * c.rdz;
        const T R1 = Fz * c.rrho_i + c.damp_z * Rz0;
        if (keep_R) out.Rz[q] = R1;
        if (!out.eval) out.Vz[q] = vz2 + T(0.5) * (dtv_zm + dtv_c) * R1;
        if (check) keep_max(r_v, Fz);
      }
    }
    dtv_zm = dtv_c;
    // the next interval's faces (level L - 1): their own R and right-hand side
    if (L - 1 >= k0 && L - 1 < ke) {
      const int q = i + ipx * j + ipxy * (L - 1);
      if (own_fx) rfx = in.rfx[q];
      if (own_fy) rfy = in.rfy[q];
      if (own && L - 1 > 0) rfz = in.rfz[q];
      if (damped) {
        if (own_fx) Rx0 = out.Rx[q];
        if (own_fy) Ry0 = out.Ry[q];
        if (own && L - 1 > 0) Rz0 = out.Rz[q];
      }
    }
    if (L > ke) return;                             // (uniform) nothing above is needed

    // ---------------- cell and lower edges at (i, j, L). The lowest row needs cells only, the highest
    // edges only; the lanes of the other side's halo compute values nobody reads.
    T txx = T(0), tyy = T(0), tzz = T(0), P = T(0), exy = T(0), exz = T(0), eyz = T(0);
    T vx_c = T(0), vy_c = T(0), vz_c = T(0), mux = T(0), muy = T(0), k_c = T(0), fz = T(0);
    if (L >= 0 && L < b.nz) {
      const float* const S = st + s * AR;
      const float* const Sp = st + sp * AR;
      vx_c = S[C_VX * AR];
      vy_c = S[C_VY * AR];
      vz_c = S[C_VZ * AR];
      const T mu_c = S[C_MU * AR];
      if (ty >= 1) {
        const T mu_l = S[C_MU * AR - 1], mu_d = S[C_MU * AR - kCorrW];
        mux = mu_l + mu_c;
        muy = mu_d + mu_c;
        if (L >= k0) {
          if (INNER || (i > 0 && i < b.nx && j > 0 && j < b.ny))
            exy = corr_modulus4(c, (S[C_MU * AR - kCorrW - 1] + mu_d) + mux) *
                  ((vx_c - S[C_VX * AR - kCorrW]) * c.hrdy + (vy_c - S[C_VY * AR - 1]) * c.hrdx);
          if (L > 0) {
            if (INNER || (i > 0 && i < b.nx && j < b.ny))
              exz = corr_modulus4(c, mux1 + mux) * ((vx_c - vx1) * c.hrdz + (vz_c - S[C_VZ * AR - 1]) * c.hrdx);
            if (INNER || (i < b.nx && j > 0 && j < b.ny))
              eyz = corr_modulus4(c, muy1 + muy) * ((vy_c - vy1) * c.hrdz + (vz_c - S[C_VZ * AR - kCorrW]) * c.hrdy);
          }
        }
      }
      if (L < ke && ty <= kCorrTY && (INNER || (i >= 0 && j >= 0 && i < b.nx && j < b.ny))) {
        const T dPt = S[C_PT * AR], dPf = S[C_PF * AR], cc = S[C_CC * AR];
        const T rpt = S[C_RPT * AR];
        const T gx = (S[C_VX * AR + 1] - vx_c) * c.rdx, gy = (S[C_VY * AR + kCorrW] - vy_c) * c.rdy;
        const T gz = (Sp[C_VZ * AR] - vz_c) * c.rdz;
        const T divV = gx + gy + gz;
        const T cpl = c.bd_rdt_a + cc;                 // beta_d alpha / dt + cc
        const T rho_pt = rpt + divV + (c.bd_rdt + cc) * dPt - cpl * dPf;
        // dP' = dP - dtau rho(dP', ...) solved for dP' (local terms implicit; the quotient only
        // scales the pseudo-step, so the fast reciprocal does)
        const T idtp = S[C_IDTP * AR];
        const T dPt1 = corr_div(dPt * idtp - (rpt + divV - cpl * dPf), idtp + c.bd_rdt + cc);
        const T third = divV * T(1.0 / 3.0);
        const T bn = c.beta_n * (rho_pt - rpt);
        const T cm2 = corr_modulus(c, mu_c);
        txx = cm2 * (gx - third + bn);
        tyy = cm2 * (gy - third + bn);
        tzz = cm2 * (gz - third + bn);
        P = out.eval ? dPt : dPt1;
        if (row_own) {
          // Darcy flux divergence, the largest neighbour k and dPf' (the tile's own cells; the flux
          // through the lower z face is the level below's upper one)
          k_c = S[C_K * AR];
          T kzp = T(0), sz = -fz1;
          if (L < b.nz - 1) {
            kzp = Sp[C_K * AR];
            const T kf = k_c + kzp, dn = Sp[C_PF * AR] - dPf;
            fz = kf * dn;
            sz = fmaf(kf, dn, -fz1);
          }
          if (L >= k0 && own) {
            const T rpf = S[C_RPF * AR];
            T kmax = fmaxf(k_c, fmaxf(k1, kzp)), sx = T(0), sy = T(0);
            if (INNER || i > 0) {
              const T kn = S[C_K * AR - 1];
              kmax = fmaxf(kmax, kn);
              sx -= (kn + k_c) * (dPf - S[C_PF * AR - 1]);
            }
            if (INNER || i < b.nx - 1) {
              const T kn = S[C_K * AR + 1];
              kmax = fmaxf(kmax, kn);
              sx += (k_c + kn) * (S[C_PF * AR + 1] - dPf);
            }
            if (INNER || j > 0) {
              const T kn = S[C_K * AR - kCorrW];
              kmax = fmaxf(kmax, kn);
              sy -= (kn + k_c) * (dPf - S[C_PF * AR - kCorrW]);
            }
            if (INNER || j < b.ny - 1) {
              const T kn = S[C_K * AR + kCorrW];
              kmax = fmaxf(kmax, kn);
              sy += (k_c + kn) * (S[C_PF * AR + kCorrW] - dPf);
            }
            const T divq = -(sx * c.hrdx2 + sy * c.hrdy2 + sz * c.hrdz2);
            const T rho_pf = rpf + divq + (c.bda_B_rdt + cc) * dPf - cpl * dPt;
            const T idtf = kmax * c.ifac_pf;
            const T dPf1 = corr_div(dPf * idtf - (rpf + divq - cpl * dPt), idtf + c.bda_B_rdt + cc);
            const int q = i + ipx * j + ipxy * L;
            if (!out.eval) {
              out.Pt[q] = dPt1;
              out.Pf[q] = dPf1;
            }
            if (out.res_pt) {
              out.res_pt[q] = rho_pt;
              out.res_pf[q] = rho_pf;
            }
            if (check) {
              keep_max(r_pt, rho_pt);
              keep_max(r_pf, rho_pf);
            }
          }
        }
      }
    }
    float* const rw = ring + s * RL;
    rw[R_TYY * RA] = tyy;
    rw[R_P * RA] = P;
    rw[R_XY * RA] = exy;
    rw[R_YZ * RA] = eyz;
    // one level up
    tzz3 = tzz2; P3 = P2;
    txx2 = txx1; tyy2 = tyy1; tzz2 = tzz1; P2 = P1; exy2 = exy1; exz2 = exz1; eyz2 = eyz1;
    txx1 = txx; tyy1 = tyy; tzz1 = tzz; P1 = P; exy1 = exy; exz1 = exz; eyz1 = eyz;
    vx2 = vx1; vy2 = vy1; vz2 = vz1;
    vx1 = vx_c; vy1 = vy_c; vz1 = vz_c;
    mux1 = mux; muy1 = muy; k1 = k_c; fz1 = fz;
  };
  for (int L = k0 - 1;; L += 3) {
    level(std::integral_constant<int, 0>{}, L);
    if (L + 1 > ke + 1) break;
    level(std::integral_constant<int, 1>{}, L + 1);
    if (L + 2 > ke + 1) break;
    level(std::integral_constant<int, 2>{}, L + 2);
    if (L + 3 > ke + 1) break;
  }
  asm volatile("cp.async.wait_group 0;\n" ::: "memory");   // the last look-ahead copies
  if (check) {
    block_max_atomic((double)__uint_as_float(r_pt), red + RED_PT);
    block_max_atomic((double)__uint_as_float(r_pf), red + RED_PF);
    block_max_atomic((double)__uint_as_float(r_v), red + RED_V);
  }
}

template <class SH>
__device__ __forceinline__ void corr_tile(const Box& b, const CorrCoef<float>& c, const CorrIn<float>& in,
                                          const CorrOut<float>& out, int tbx, int tby, int k0, int ke,
                                          unsigned long long* red, int check, float* corr_smem) {
  // every point the tile computes or stages has its x- and y-neighbours inside the grid
  const bool inner = tbx > 0 && tby > 0 && (tbx + 1) * kCorrTX + 1 < b.nx && (tby + 1) * SH::ty + 1 < b.ny;
  if (inner) corr_tile_run<SH, true>(b, c, in, out, tbx, tby, k0, ke, red, check, corr_smem);
  else corr_tile_run<SH, false>(b, c, in, out, tbx, tby, k0, ke, red, check, corr_smem);
}

__global__ void __launch_bounds__(CorrSingle::threads, CorrSingle::blocks) k_corr_iteration(Box b, CorrCoef<float> c, CorrIn<float> in,
                                                        CorrOut<float> out, unsigned long long* red, int check,
                                                        int zchunk) {
  chain_begin();
  extern __shared__ __align__(16) float corr_smem[];   // CorrSingle::smem, dynamic (above 48 KB)
  const int k0 = blockIdx.z * zchunk;
  corr_tile<CorrSingle>(b, c, in, out, blockIdx.x, blockIdx.y, k0, min(k0 + zchunk, b.nz), red, check, corr_smem);
}

// (iv) u <- u + delta (FP64 += FP32 correction).
__device__ __forceinline__ void mix_update_point(const Box& b, const MixUpdate& u, int i, int j, int k) {
  if (i > b.nx || j > b.ny || k > b.nz) return;
  const long long q = cidx(b, i, j, k);
  const double w = u.omega;
  if (i > 0 && i < b.nx && j < b.ny && k < b.nz) u.Vx[q] = fma(w, (double)u.dVx[q], u.Vx[q]);
  if (j > 0 && j < b.ny && i < b.nx && k < b.nz) u.Vy[q] = fma(w, (double)u.dVy[q], u.Vy[q]);
  if (k > 0 && k < b.nz && i < b.nx && j < b.ny) u.Vz[q] = fma(w, (double)u.dVz[q], u.Vz[q]);
  if (i < b.nx && j < b.ny && k < b.nz) {
    u.Pt1[q] = fma(w, (double)u.dPt[q], u.Pt[q]);
    u.Pf1[q] = fma(w, (double)u.dPf[q], u.Pf[q]);
  }
}

__global__ void __launch_bounds__(kPlaneThreads) k_mix_update(Box b, MixUpdate u, Plane pl) {
  chain_begin();
  int i, j;
  if (plane_point(pl, i, j)) mix_update_point(b, u, i, j, (int)blockIdx.y);
}

void mix_begin(cudaStream_t s, Box b, const double* Pt, const double* Pf, const double* phi, const double* mu,
               double* Pto, double* Pfo, double* phio, unsigned long long* red) {
  const Plane pl = plane_of(b, 0);
  k_mix_begin<<<plane_grid(pl, b.nz), kPlaneThreads, 0, s>>>(b, Pt, Pf, phi, mu, Pto, Pfo, phio, red, pl);
}
void mix_perm(cudaStream_t s, Box b, const LeanCoef<double>& c, const double* phi, const double* logk, double* perm) {
  const Plane pl = plane_of(b, 0);
  launch_chained(k_mix_perm, plane_grid(pl, b.nz), kPlaneThreads, 0, s, b, c, phi, logk, perm, pl);
}
void mix_prepare(cudaStream_t s, Box b, const LeanCoef<double>& c, const StressCoef& sc, const MixPrepIn& in,
                 const MixPrepOut& out, unsigned long long* red) {
  const Plane pl = plane_of(b, c.bg_on ? 1 : 0);   // wall edges carry stress under a background shear only
  launch_chained(k_mix_prepare, plane_grid(pl, b.nz), kPlaneThreads, 0, s, b, c, sc, in, out, red, pl);
}
void mix_faces(cudaStream_t s, Box b, const LeanCoef<double>& c, const MixFaceIn& in, const MixFaceOut& out,
               unsigned long long* red) {
  const Plane pl = plane_of(b, 0);
  launch_chained(k_mix_faces, plane_grid(pl, b.nz), kPlaneThreads, 0, s, b, c, in, out, red, pl);
}
void mix_porosity(cudaStream_t s, Box b, const LeanCoef<double>& c, const MixPorosity& p) {
  const Plane pl = plane_of(b, 0);
  launch_chained(k_mix_porosity, plane_grid(pl, b.nz), kPlaneThreads, 0, s, b, c, p, pl);
}
void mix_update(cudaStream_t s, Box b, const MixUpdate& u) {
  const Plane pl = plane_of(b, 0);
  launch_chained(k_mix_update, plane_grid(pl, b.nz), kPlaneThreads, 0, s, b, u, pl);
}
void corr_iteration(cudaStream_t s, Box b, const CorrCoef<float>& c, const CorrIn<float>& in,
                    const CorrOut<float>& out, unsigned long long* red, int check) {
  // the faces i = nx, j = ny, k = nz are walls: tiles cover the cells and their lower faces
  const unsigned gx = (b.nx + kCorrTX - 1) / kCorrTX, gy = (b.ny + CorrSingle::ty - 1) / CorrSingle::ty;
  // grids of a few levels per block slot (up to some 56^3) are latency: two blocks on an SM cost little more
  // than one (48^3: 1412 -> 1297 us per 120 sweeps with their outer phases)
  const long long cols = (long long)gx * gy;
  const double base = cols * b.nz < 4LL * CorrSingle::blocks * sm_count() ? 2.0 : 1.0;
  const int zc = march_chunk(cols, b.nz, kCorrZChunk, CorrSingle::blocks, sm_count(), 3.0, base);
  const dim3 g(gx, gy, (unsigned)((b.nz + zc - 1) / zc));
  cudaFuncSetAttribute(k_corr_iteration, cudaFuncAttributeMaxDynamicSharedMemorySize, CorrSingle::smem);
  launch_chained(k_corr_iteration, g, dim3(32, CorrSingle::rows, 1), CorrSingle::smem, s, b, c, in, out, red, check,
                 zc);
}


// ============================================================ multigrid transfers (FP32)
// Level f (fine, n cells per direction) and level c (coarse, ceil(n / 2)), through the weight
// tables of c.ax (MgAxis).
__global__ void __launch_bounds__(256) k_mg_coef(MgLevel f, MgLevel c, float dtaupt_fac, float dtauv_fac) {
  chain_begin();
  const int I = blockIdx.x * blockDim.x + threadIdx.x, J = blockIdx.y * blockDim.y + threadIdx.y;
  const int K = blockIdx.z;
  if (I >= c.b.nx || J >= c.b.ny || K >= c.b.nz) return;
  const int i0 = c.ax[0].box_i0[I], j0 = c.ax[1].box_i0[J], k0 = c.ax[2].box_i0[K];
  const float* wx = c.ax[0].box_w + 3 * I;
  const float* wy = c.ax[1].box_w + 3 * J;
  const float* wz = c.ax[2].box_w + 3 * K;
  float m = 0.f, k = 0.f, cc = 0.f;
  for (int dz = 0; dz < 3; ++dz)
    for (int dy = 0; dy < 3; ++dy)
      for (int dx = 0; dx < 3; ++dx) {
        const float w = wx[dx] * wy[dy] * wz[dz];
        if (w == 0.f) continue;
        const long long q = cidx(f.b, i0 + dx, j0 + dy, k0 + dz);
        m += w * f.mu[q];
        k += w * f.perm[q];
        cc += w * f.cc[q];
      }
  const long long qc = cidx(c.b, I, J, K);
  c.mu[qc] = m;
  c.perm[qc] = k;
  c.cc[qc] = cc;
  c.idtp[qc] = 1.0f / (dtaupt_fac * m);
  c.dtvc[qc] = dtauv_fac / m;
}

__global__ void __launch_bounds__(256) k_mg_restrict(MgLevel f, MgLevel c, float rho_i) {
  chain_begin();
  const int I = blockIdx.x * blockDim.x + threadIdx.x, J = blockIdx.y * blockDim.y + threadIdx.y;
  const int K = blockIdx.z;
  const Box& B = c.b;
  if (I > B.nx || J > B.ny || K > B.nz) return;
  const long long qc = cidx(B, I, J, K);
  // a zero correction and damped residual on the coarse grid (walls included)
  c.dVx[0][qc] = 0.f; c.dVx[1][qc] = 0.f; c.dVy[0][qc] = 0.f; c.dVy[1][qc] = 0.f;
  c.dVz[0][qc] = 0.f; c.dVz[1][qc] = 0.f; c.dPt[0][qc] = 0.f; c.dPf[0][qc] = 0.f;
  c.Rx[qc] = 0.f; c.Ry[qc] = 0.f; c.Rz[qc] = 0.f;
  const Box& F = f.b;
  const MgAxis &X = c.ax[0], &Y = c.ax[1], &Z = c.ax[2];
  if (I < B.nx && J < B.ny && K < B.nz) {
    const int i0 = X.box_i0[I], j0 = Y.box_i0[J], k0 = Z.box_i0[K];
    const float *bx = X.box_w + 3 * I, *by = Y.box_w + 3 * J, *bz = Z.box_w + 3 * K;
    float a = 0.f, b = 0.f;
    for (int dz = 0; dz < 3; ++dz)
      for (int dy = 0; dy < 3; ++dy)
        for (int dx = 0; dx < 3; ++dx) {
          const float w = bx[dx] * by[dy] * bz[dz];
          if (w == 0.f) continue;
          const long long q = cidx(F, i0 + dx, j0 + dy, k0 + dz);
          a += w * f.res_pt[q];
          b += w * f.res_pf[q];
        }
    c.rpt[qc] = a;
    c.rpf[qc] = b;
  }
  // faces: hat weights along the normal, box weights across it
  if (I > 0 && I < B.nx && J < B.ny && K < B.nz) {
    const int i0 = X.hat_i0[I], j0 = Y.box_i0[J], k0 = Z.box_i0[K];
    const float *h = X.hat_w + 4 * I, *by = Y.box_w + 3 * J, *bz = Z.box_w + 3 * K;
    float s = 0.f;
    for (int dz = 0; dz < 3; ++dz)
      for (int dy = 0; dy < 3; ++dy)
        for (int dx = 0; dx < 4; ++dx) {
          const float w = h[dx] * by[dy] * bz[dz];
          if (w == 0.f) continue;
          s += w * f.Rx[cidx(F, i0 + dx, j0 + dy, k0 + dz)];
        }
    c.rfx[qc] = rho_i * s;
  }
  if (J > 0 && J < B.ny && I < B.nx && K < B.nz) {
    const int i0 = X.box_i0[I], j0 = Y.hat_i0[J], k0 = Z.box_i0[K];
    const float *bx = X.box_w + 3 * I, *h = Y.hat_w + 4 * J, *bz = Z.box_w + 3 * K;
    float s = 0.f;
    for (int dz = 0; dz < 3; ++dz)
      for (int dy = 0; dy < 4; ++dy)
        for (int dx = 0; dx < 3; ++dx) {
          const float w = bx[dx] * h[dy] * bz[dz];
          if (w == 0.f) continue;
          s += w * f.Ry[cidx(F, i0 + dx, j0 + dy, k0 + dz)];
        }
    c.rfy[qc] = rho_i * s;
  }
  if (K > 0 && K < B.nz && I < B.nx && J < B.ny) {
    const int i0 = X.box_i0[I], j0 = Y.box_i0[J], k0 = Z.hat_i0[K];
    const float *bx = X.box_w + 3 * I, *by = Y.box_w + 3 * J, *h = Z.hat_w + 4 * K;
    float s = 0.f;
    for (int dz = 0; dz < 4; ++dz)
      for (int dy = 0; dy < 3; ++dy)
        for (int dx = 0; dx < 3; ++dx) {
          const float w = bx[dx] * by[dy] * h[dz];
          if (w == 0.f) continue;
          s += w * f.Rz[cidx(F, i0 + dx, j0 + dy, k0 + dz)];
        }
    c.rfz[qc] = rho_i * s;
  }
}

__global__ void __launch_bounds__(256) k_mg_prolong(MgLevel c, int dc, MgLevel f, int df) {
  chain_begin();
  const int i = blockIdx.x * blockDim.x + threadIdx.x, j = blockIdx.y * blockDim.y + threadIdx.y;
  const int k = blockIdx.z;
  const Box& B = f.b;
  if (i > B.nx || j > B.ny || k > B.nz) return;
  const long long q = cidx(B, i, j, k);
  const MgAxis &X = c.ax[0], &Y = c.ax[1], &Z = c.ax[2];
  if (i < B.nx && j < B.ny && k < B.nz) {   // cells: trilinear between coarse centres
    float pt = 0.f, pf = 0.f;
    for (int a = 0; a < 2; ++a)
      for (int bb = 0; bb < 2; ++bb)
        for (int cc = 0; cc < 2; ++cc) {
          const float w = Z.lin_w[2 * k + a] * Y.lin_w[2 * j + bb] * X.lin_w[2 * i + cc];
          const long long qc = cidx(c.b, X.lin_ab[2 * i + cc], Y.lin_ab[2 * j + bb], Z.lin_ab[2 * k + a]);
          pt += w * c.dPt[dc][qc];
          pf += w * c.dPf[dc][qc];
        }
    f.dPt[df][q] += pt;
    f.dPf[df][q] += pf;
  }
  // faces: linear between coarse faces along the normal (coarse wall faces are zero), between
  // coarse centres across it
  if (i > 0 && i < B.nx && j < B.ny && k < B.nz) {
    const int n0 = X.fl_n0[i];
    const float t = X.fl_t[i];
    float v = 0.f;
    for (int a = 0; a < 2; ++a)
      for (int bb = 0; bb < 2; ++bb) {
        const int y = Y.lin_ab[2 * j + bb], z = Z.lin_ab[2 * k + a];
        v += Z.lin_w[2 * k + a] * Y.lin_w[2 * j + bb] *
             ((1.f - t) * c.dVx[dc][cidx(c.b, n0, y, z)] + t * c.dVx[dc][cidx(c.b, n0 + 1, y, z)]);
      }
    f.dVx[df][q] += v;
  }
  if (j > 0 && j < B.ny && i < B.nx && k < B.nz) {
    const int n0 = Y.fl_n0[j];
    const float t = Y.fl_t[j];
    float v = 0.f;
    for (int a = 0; a < 2; ++a)
      for (int cc = 0; cc < 2; ++cc) {
        const int x = X.lin_ab[2 * i + cc], z = Z.lin_ab[2 * k + a];
        v += Z.lin_w[2 * k + a] * X.lin_w[2 * i + cc] *
             ((1.f - t) * c.dVy[dc][cidx(c.b, x, n0, z)] + t * c.dVy[dc][cidx(c.b, x, n0 + 1, z)]);
      }
    f.dVy[df][q] += v;
  }
  if (k > 0 && k < B.nz && i < B.nx && j < B.ny) {
    const int n0 = Z.fl_n0[k];
    const float t = Z.fl_t[k];
    float v = 0.f;
    for (int bb = 0; bb < 2; ++bb)
      for (int cc = 0; cc < 2; ++cc) {
        const int x = X.lin_ab[2 * i + cc], y = Y.lin_ab[2 * j + bb];
        v += Y.lin_w[2 * j + bb] * X.lin_w[2 * i + cc] *
             ((1.f - t) * c.dVz[dc][cidx(c.b, x, y, n0)] + t * c.dVz[dc][cidx(c.b, x, y, n0 + 1)]);
      }
    f.dVz[df][q] += v;
  }
}

void mg_coef(cudaStream_t s, const MgLevel& f, const MgLevel& c, float dtaupt_fac, float dtauv_fac) {
  const dim3 bl(32, 8, 1), g((c.b.nx + 31) / 32, (c.b.ny + 7) / 8, c.b.nz);
  launch_chained(k_mg_coef, g, bl, 0, s, f, c, dtaupt_fac, dtauv_fac);
}
void mg_restrict(cudaStream_t s, const MgLevel& f, const MgLevel& c, float rho_i) {
  const dim3 bl(32, 8, 1), g((c.b.nx + 1 + 31) / 32, (c.b.ny + 1 + 7) / 8, c.b.nz + 1);
  launch_chained(k_mg_restrict, g, bl, 0, s, f, c, rho_i);
}
void mg_prolong(cudaStream_t s, const MgLevel& c, int dc, const MgLevel& f, int df) {
  const dim3 bl(32, 8, 1), g((f.b.nx + 1 + 31) / 32, (f.b.ny + 1 + 7) / 8, f.b.nz + 1);
  launch_chained(k_mg_prolong, g, bl, 0, s, c, dc, f, df);
}

// ============================================================ batched FP32 ensembles (engine)
namespace {

__device__ inline unsigned long long mb_global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// Last member whose first work item (tile_base or ctile_base) is <= t.
template <long long MixBatchInst::*BASE>
__device__ inline int mb_find(const MixBatchInst* inst, int ninst, long long t) {
  int lo = 0, hi = ninst - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (inst[mid].*BASE <= t) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

// The first work item >= `next` that this CTA visits in a grid stride starting at blockIdx.x:
// a CTA skips a member that has no work in a launch in one step instead of tile by tile.
__device__ inline long long mb_skip_to(long long next, long long t0) {
  const long long g = gridDim.x;
  return next + ((t0 + (long long)blockIdx.x - next) % g + g) % g;
}

__device__ inline bool mb_runs(int phase, const MixBatchStatus& s) {
  switch (phase) {
    case MB_PH_PERM: case MB_PH_PREP: case MB_PH_FACES: return s.phase == MB_PREP;
    case MB_PH_INIT: return s.phase == MB_INNER && s.fresh;
    default: return s.phase == MB_UPDATE;
  }
}

constexpr int kMbBX = 32, kMbBY = 8;   // point tiles: 32 x 8 cells of one z-level

}  // namespace

// The point phases over every member's tiles (grid-stride over the flat work list; a member not
// in the phase skips its tiles, uniformly per CTA, so the block-wide reductions stay collective).
template <int PHASE>
__global__ void __launch_bounds__(kMbBX * kMbBY) k_mb_points(const MixBatchInst* __restrict__ inst,
                                                            const MixBatchStatus* __restrict__ st, int ninst,
                                                            long long t0, long long t1) {
  for (long long t = t0 + blockIdx.x; t < t1; t += gridDim.x) {
    const int m = mb_find<&MixBatchInst::tile_base>(inst, ninst, t);
    const MixBatchStatus& S = st[m];
    if (!mb_runs(PHASE, S)) {   // uniform over the CTA: on to the next member's tiles
      t = mb_skip_to(m + 1 < ninst ? inst[m + 1].tile_base : t1, t0) - gridDim.x;
      continue;
    }
    const MixBatchInst& I = inst[m];
    const long long local = t - I.tile_base;
    const long long per_z = (long long)I.gx * I.gy;
    const int kz = (int)(local / per_z);
    const int r = (int)(local - (long long)kz * per_z);
    const int ty = r / I.gx, tx = r - ty * I.gx;
    const int i = tx * kMbBX + threadIdx.x, j = ty * kMbBY + threadIdx.y;
    const Box& b = I.b;
    const int a = S.cur;
    if (PHASE == MB_PH_PERM) {
      mix_perm_point(b, I.lc, I.phi[a], I.logk, I.perm, i, j, kz);
    } else if (PHASE == MB_PH_PREP) {
      const MixPrepIn pin{StressIn{I.Vx, I.Vy, I.Vz, I.mu, I.txxo, I.tyyo, I.tzzo, I.txyo, I.txzo, I.tyzo},
                          I.Pt[a], I.Pf[a], I.phi[a], I.eta, I.perm, I.Pto, I.Pfo};
      const MixPrepOut pout{I.s_txx, I.s_tyy, I.s_tzz, I.s_txy, I.s_txz, I.s_tyz, I.rpt, I.rpf, I.ccf, I.kf, I.idtp};
      double r_pt = 0.0, r_pf = 0.0;
      mix_prepare_point(b, I.lc, I.sc, pin, pout, i, j, kz, r_pt, r_pf);
      block_max_atomic(lean_detail::abs_max(r_pt, 0.0), I.red + RED_PT);
      block_max_atomic(lean_detail::abs_max(r_pf, 0.0), I.red + RED_PF);
    } else if (PHASE == MB_PH_FACES) {
      double r_v = 0.0, pic = 1.0;
      mix_faces_point(b, I.lc,
                      MixFaceIn{LeanPicardIn<double>{I.s_txx, I.s_tyy, I.s_tzz, I.s_txy, I.s_txz, I.s_tyz, I.phi[a],
                                                     I.Pt[a], I.Pf[a]},
                                I.mu, I.eta},
                      MixFaceOut{I.rfx, I.rfy, I.rfz, I.muf, I.dtvc}, i, j, kz, r_v, pic);
      block_max_atomic(lean_detail::abs_max(r_v, 0.0), I.red + RED_V);
      block_max_log_atomic(pic, I.red + RED_PIC);
    } else if (PHASE == MB_PH_INIT) {
      if (i <= b.nx && j <= b.ny && kz <= b.nz) {   // a zero correction and damped residual
        const long long q = cidx(b, i, j, kz);
        I.dVx[0][q] = 0.f; I.dVy[0][q] = 0.f; I.dVz[0][q] = 0.f; I.dPt[0][q] = 0.f; I.dPf[0][q] = 0.f;
        I.Rx[q] = 0.f; I.Ry[q] = 0.f; I.Rz[q] = 0.f;
      }
    } else if (PHASE == MB_PH_UPDATE) {   // the new pressures go to the other buffer, phi follows them
      const int d = S.inner & 1;   // the last correction's buffer
      mix_update_point(b, MixUpdate{I.Vx, I.Vy, I.Vz, I.Pt[a], I.Pf[a], I.Pt[1 - a], I.Pf[1 - a], I.dVx[d], I.dVy[d],
                                    I.dVz[d], I.dPt[d], I.dPf[d], S.omega}, i, j, kz);
    } else {   // MB_PH_POROSITY
      mix_porosity_point(b, I.lc, MixPorosity{I.Vx, I.Vy, I.Vz, I.phi[a], I.Pt[1 - a], I.Pf[1 - a], I.Pto, I.Pfo, I.Lo,
                                              I.eta, I.phi[1 - a]}, i, j, kz);
    }
  }
}

// Correction iteration number inner + step of the members in MB_INNER (within their budget),
// one corr_tile per work item; the block's shared memory is reused from tile to tile.
__global__ void __launch_bounds__(CorrBatch::threads, CorrBatch::blocks) k_mb_corr(const MixBatchInst* __restrict__ inst,
                                                       const MixBatchStatus* __restrict__ st, int ninst,
                                                       long long t0, long long t1, int step, int nup,
                                                       int zchunk) {
  extern __shared__ __align__(16) float corr_smem[];
  __shared__ CorrCoef<float> s_cc;   // the member's coefficients, read from shared memory by the tile
  for (long long t = t0 + blockIdx.x; t < t1; t += gridDim.x) {
    const int m = mb_find<&MixBatchInst::ctile_base>(inst, ninst, t);
    const MixBatchStatus& S = st[m];
    const MixBatchInst& I = inst[m];
    const int it = S.inner + step;
    if (S.phase != MB_INNER || it > I.max_iter - S.iters) {   // uniform over the CTA
      t = mb_skip_to(m + 1 < ninst ? inst[m + 1].ctile_base : t1, t0) - gridDim.x;
      continue;
    }
    const int d = (it - 1) & 1;
    if (threadIdx.x == 0 && threadIdx.y == 0) s_cc = I.cc;
    // the argument pointers as offsets of one base (cheap to recompute, unlike pointers loaded
    // from the descriptor): slots rpt, rpf, rfx, rfy, rfz, cc, k, idtp, mu, dtvc, dVx[2], dVy[2],
    // dVz[2], dPt[2], dPf[2], Rx, Ry, Rz
    float* const B = const_cast<float*>(I.fbase);
    const long long fs = I.fstride;
    auto P = [B, fs](int slot) { return B + slot * fs; };
    const CorrIn<float> ci{P(10 + d), P(12 + d), P(14 + d), P(16 + d), P(18 + d), P(5), P(6), P(7), P(0), P(1),
                           P(8), P(9), P(2), P(3), P(4)};
    const CorrOut<float> co{P(11 - d), P(13 - d), P(15 - d), P(17 - d), P(19 - d), P(20), P(21), P(22)};
    const long long local = t - I.ctile_base;
    const long long per_z = (long long)I.cgx * I.cgy;
    const int bz = (int)(local / per_z);
    const int r = (int)(local - (long long)bz * per_z);
    const int tby = r / I.cgx, tbx = r - tby * I.cgx;
    const int k0 = bz * zchunk;
    const Box b = I.b;
    unsigned long long* const ired = I.ired;
    __syncthreads();   // s_cc written
    corr_tile<CorrBatch>(b, s_cc, ci, co, tbx, tby, k0, min(k0 + zchunk, b.nz), ired, step == nup, corr_smem);
    __syncthreads();   // the next tile's stage and rings overwrite this one's
  }
}

// Outer decision of the members in MB_PREP (the host loop's, in the same order): non-finite
// norms stop the member (PT_ENAN), norms below tol end its step (PT_OK); otherwise the outer
// weight adapts (halved down to 1/16 when the residual more than doubled, grown by 1.25 up to 1
// while it falls), the inner target is rtol times the residual, and a correction solve starts.
__global__ void k_mb_decide_outer(const MixBatchInst* __restrict__ inst, MixBatchStatus* __restrict__ st,
                                  int ninst) {
  const int m = blockIdx.x * blockDim.x + threadIdx.x;
  if (m >= ninst || st[m].phase != MB_PREP) return;
  MixBatchStatus& S = st[m];
  unsigned long long* red = inst[m].red;
  const int slot[4] = {RED_V, RED_PT, RED_PF, RED_PIC};
  bool finite = true;
  double r = 0.0;
  for (int s = 0; s < 4; ++s) {
    const double v = __longlong_as_double((long long)red[slot[s]]);
    S.res[s] = v;
    finite = finite && isfinite(v);
    r = fmax(r, v);
    red[slot[s]] = 0ull;
  }
  if (!finite) {
    S.phase = MB_DONE;
    S.status = PT_ENAN;
    S.t_stop = mb_global_ns();
    return;
  }
  if (r < inst[m].tol) {
    S.phase = MB_DONE;
    S.status = PT_OK;
    S.t_stop = mb_global_ns();
    return;
  }
  if (S.prev > 0.0) {
    if (r > 2.0 * S.prev) S.omega = fmax(S.omega * 0.5, 0.0625);
    else if (r < S.prev) S.omega = fmin(S.omega * 1.25, 1.0);
  }
  S.prev = r;
  S.target = inst[m].rtol * r;
  S.phase = MB_INNER;
  S.fresh = 1;
  S.inner = 0;
}

// Inner decision after `nup` correction launches: the iterations that ran are counted; after a
// check iteration a non-finite norm stops the member (PT_ENAN) and a drop below the target ends
// the solve; so does a spent budget (max_iter - iters).
__global__ void k_mb_decide_inner(const MixBatchInst* __restrict__ inst, MixBatchStatus* __restrict__ st,
                                  int ninst, int nup) {
  const int m = blockIdx.x * blockDim.x + threadIdx.x;
  if (m >= ninst || st[m].phase != MB_INNER) return;
  MixBatchStatus& S = st[m];
  S.fresh = 0;
  const int budget = inst[m].max_iter - S.iters;
  const int ran = min(nup, budget - S.inner);
  S.inner += ran;
  bool stop = S.inner >= budget;
  if (ran == nup) {   // the last launch was a check iteration
    unsigned long long* red = inst[m].ired;
    const double v = __longlong_as_double((long long)red[RED_V]);
    const double pt = __longlong_as_double((long long)red[RED_PT]);
    const double pf = __longlong_as_double((long long)red[RED_PF]);
    red[RED_V] = 0ull;
    red[RED_PT] = 0ull;
    red[RED_PF] = 0ull;
    if (!(isfinite(v) && isfinite(pt) && isfinite(pf))) {
      S.iters += S.inner;
      S.phase = MB_DONE;
      S.status = PT_ENAN;
      S.t_stop = mb_global_ns();
      return;
    }
    if (fmax(fmax(v, pt), pf) < S.target) stop = true;
  }
  if (stop) S.phase = MB_UPDATE;
}

// End of an outer iteration: the iterate moved to the other buffers; the solve's iterations are
// counted; a member whose budget is spent stops unconverged (PT_ENOTCONV), the others go on.
__global__ void k_mb_finish(const MixBatchInst* __restrict__ inst, MixBatchStatus* __restrict__ st, int ninst) {
  const int m = blockIdx.x * blockDim.x + threadIdx.x;
  if (m >= ninst || st[m].phase != MB_UPDATE) return;
  MixBatchStatus& S = st[m];
  S.cur = 1 - S.cur;
  S.iters += S.inner;
  S.inner = 0;
  S.outer += 1;
  if (S.iters >= inst[m].max_iter) {
    S.phase = MB_DONE;
    S.status = PT_ENOTCONV;
    S.t_stop = mb_global_ns();
  } else {
    S.phase = MB_PREP;
  }
}

__global__ void k_mb_start(const MixBatchInst* __restrict__ inst, MixBatchStatus* __restrict__ st, int ninst) {
  const int m = blockIdx.x * blockDim.x + threadIdx.x;
  if (m >= ninst) return;
  MixBatchStatus& S = st[m];
  S.phase = MB_PREP;
  S.cur = 0;
  S.inner = 0;
  S.iters = 0;
  S.outer = 0;
  S.status = PT_ENOTCONV;
  S.fresh = 0;
  S.omega = 1.0;
  S.prev = 0.0;
  S.target = 0.0;
  for (int s = 0; s < 4; ++s) S.res[s] = 0.0;
  for (int s = 0; s < RED_N; ++s) {
    inst[m].red[s] = 0ull;
    inst[m].ired[s] = 0ull;
  }
  S.t_start = mb_global_ns();
  S.t_stop = 0ull;
}

void mb_points(int grid, cudaStream_t s, int phase, const MixBatchInst* inst, const MixBatchStatus* st, int ninst,
               long long t0, long long t1) {
  const dim3 bl(kMbBX, kMbBY, 1);
  switch (phase) {
    case MB_PH_PERM: k_mb_points<MB_PH_PERM><<<grid, bl, 0, s>>>(inst, st, ninst, t0, t1); break;
    case MB_PH_PREP: k_mb_points<MB_PH_PREP><<<grid, bl, 0, s>>>(inst, st, ninst, t0, t1); break;
    case MB_PH_FACES: k_mb_points<MB_PH_FACES><<<grid, bl, 0, s>>>(inst, st, ninst, t0, t1); break;
    case MB_PH_INIT: k_mb_points<MB_PH_INIT><<<grid, bl, 0, s>>>(inst, st, ninst, t0, t1); break;
    case MB_PH_UPDATE: k_mb_points<MB_PH_UPDATE><<<grid, bl, 0, s>>>(inst, st, ninst, t0, t1); break;
    default: k_mb_points<MB_PH_POROSITY><<<grid, bl, 0, s>>>(inst, st, ninst, t0, t1); break;
  }
}

void mb_corr(int grid, cudaStream_t s, const MixBatchInst* inst, const MixBatchStatus* st, int ninst,
             long long t0, long long t1, int step, int nup, int zchunk) {
  k_mb_corr<<<grid, dim3(32, CorrBatch::rows, 1), CorrBatch::smem, s>>>(inst, st, ninst, t0, t1, step, nup, zchunk);
}

void mb_decide_outer(cudaStream_t s, const MixBatchInst* inst, MixBatchStatus* st, int ninst) {
  k_mb_decide_outer<<<(ninst + 127) / 128, 128, 0, s>>>(inst, st, ninst);
}
void mb_decide_inner(cudaStream_t s, const MixBatchInst* inst, MixBatchStatus* st, int ninst, int nup) {
  k_mb_decide_inner<<<(ninst + 127) / 128, 128, 0, s>>>(inst, st, ninst, nup);
}
void mb_finish(cudaStream_t s, const MixBatchInst* inst, MixBatchStatus* st, int ninst) {
  k_mb_finish<<<(ninst + 127) / 128, 128, 0, s>>>(inst, st, ninst);
}
void mb_start(cudaStream_t s, const MixBatchInst* inst, MixBatchStatus* st, int ninst) {
  k_mb_start<<<(ninst + 127) / 128, 128, 0, s>>>(inst, st, ninst);
}

int mb_points_blocks_per_sm() {
  int n = 0;
  const cudaError_t e =
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_mb_points<MB_PH_PREP>, kMbBX * kMbBY, 0);
  return (e == cudaSuccess && n > 0) ? n : 1;
}

int mb_corr_blocks_per_sm() {
  int n = 0;
  cudaFuncSetAttribute(k_mb_corr, cudaFuncAttributeMaxDynamicSharedMemorySize, CorrBatch::smem);
  const cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_mb_corr, CorrBatch::threads, CorrBatch::smem);
  return (e == cudaSuccess && n > 0) ? n : 1;
}

int corr_tile_x() { return kCorrTX; }
int corr_tile_y() { return CorrBatch::ty; }

}  // namespace pt
