// pt_df_body.cuh — the double-float PT iteration (PT_DF64): cells and faces at one box index.
//
// The form is bound by instruction issue as much as by HBM, so some of its sums and products stay
// unnormalised: a pair (s, e) straight from a two-sum or an exact product holds the value to 2^-48 of its
// operands whether or not |e| <= ulp(s) / 2, and the next sum takes both parts anyway (8 instructions
// where the normalising one takes 11, 12 for a term of a sum of products where it takes 15). Differences
// of neighbour values, the Darcy sums, the two residuals and k keep the normal form: unnormalised, the low
// parts of cancelled high ones are rounded twice, and the errors against 64 bits grew by 1.3x (Vx at
// 191 x 180 x 200, 30 iterations: 4.8e-14 against 3.7e-14); with them normal every field's error is at
// or below that of all-normal arithmetic (3.6e-14), for 147 ms a step at 383^3 against 144 without and
// 154 with everything normal.
#pragma once

#include "pt_lean_body.cuh"

namespace pt {
namespace dfu {

// x + y, x - y, x y, a b + c with no final normalisation
__device__ __forceinline__ df64 add(df64 x, df64 y) {
  float s, e;
  dfd::two_sum(x.hi, y.hi, s, e);
  return df64(s, __fadd_rn(e, __fadd_rn(x.lo, y.lo)));
}
__device__ __forceinline__ df64 sub(df64 x, df64 y) { return add(x, -y); }
__device__ __forceinline__ df64 subn(df64 x, df64 y) { return x - y; }   // normalised
__device__ __forceinline__ df64 mul(df64 x, df64 y) {
  const float p = __fmul_rn(x.hi, y.hi);
  float e = __fmaf_rn(x.hi, y.hi, -p);
  e = __fmaf_rn(x.hi, y.lo, e);
  return df64(p, __fmaf_rn(x.lo, y.hi, e));
}
__device__ __forceinline__ df64 mad(df64 a, df64 b, df64 c) {
  const df64 p = mul(a, b);
  float s, t;
  dfd::two_sum(p.hi, c.hi, s, t);
  return df64(s, __fadd_rn(t, __fadd_rn(p.lo, c.lo)));
}
__device__ __forceinline__ df64 norm(df64 x) { return dfd::renorm(x.hi, x.lo); }
__device__ __forceinline__ df64 half(df64 x) { return df64(0.5f * x.hi, 0.5f * x.lo); }

// 1 / x (x > 0, far inside the normal range): the hardware's approximate reciprocal (1 ulp) and one
// third-order step r (1 + d + d^2), d = 1 - x r from the exact product: rounding-limited.
__device__ __forceinline__ df64 rcp(df64 x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x.hi));
  const float p = __fmul_rn(x.hi, r);
  float q = __fmaf_rn(x.hi, r, -p);
  q = __fmaf_rn(x.lo, r, q);
  const float d = __fsub_rn(__fsub_rn(1.0f, p), q);   // 1 - p is exact (p within an ulp or two of 1)
  return dfd::renorm(r, __fmul_rn(r, __fmaf_rn(d, d, d)));
}

}  // namespace dfu

// One level of a column of cells from a staged tile: pressures, porosity, k, stresses of the centre and
// of its three lower edges.
// The stage (units of df64): per level a tile of (8 + 2) rows x kDfW columns, the 32 x 8 points of the
// block at column 2 and row 1, of the six arrays whose neighbours are read -- Pf, phi, k, Vz in three
// slots (levels k, k + 1, and k + 2 in flight), Vx, Vy in two -- and the 16 arrays read at the own index
// only, 256 values each, in two slots.
constexpr int kDfW = 36, kDfAR = 10 * kDfW;
enum { H_PF, H_PHI, H_K, H_VZ, kDfHalo3 };                 // three slots each
enum { H_VX, H_VY, kDfHalo2 };                             // two slots each
enum { S_PT = kStageSlots, kDfPoint };                     // the stage's pointwise slots and Pt
constexpr int kDfH2 = kDfHalo3 * 3 * kDfAR, kDfPW = kDfH2 + kDfHalo2 * 2 * kDfAR, kDfPWSlot = kDfPoint * 256;
constexpr int kDfStageElems = kDfPW + 2 * kDfPWSlot;
static_assert(kDfPoint % 2 == 0, "the pointwise arrays are copied in pairs");

struct DfColumn {                // carried from level k - 1
  df64 phi_d, k_d, vx_d, vy_d;
  df64 fz;                       // Darcy term (k + k_below) (Pf - Pf_below + buoyancy) through the lower face
};

// s3, s3p: this thread's place in the three-slot tiles of level k and k + 1; s2: in the two-slot tiles;
// pw: in the pointwise slots. INNER: the block's columns touch no wall in x and y.
template <bool INNER>
__device__ __forceinline__ void df_cell_level(const Box& b, const LeanCoef<df64>& c, const df64* K0,
                                              const LeanCellOut<df64>& out, int i, int j, int k, int check,
                                              DfColumn& col, unsigned long long& m_pt, unsigned long long& m_pf,
                                              const df64* s3, const df64* s3p, const df64* s2, const df64* pw) {
  using namespace dfu;
  const long long q = cidx(b, i, j, k);
  const df64 zero(0.0f, 0.0f);
  const bool up = k < b.nz - 1;            // levels [0, nz): the level nz holds walls only
  const bool ci = INNER || i < b.nx, cj = INNER || j < b.ny;
  auto A3 = [&](int a, int o) { return s3[a * 3 * kDfAR + o]; };
  auto A3p = [&](int a) { return s3p[a * 3 * kDfAR]; };
  auto A2 = [&](int a, int o) { return s2[a * 2 * kDfAR + o]; };
  auto PW = [&](int a) { return pw[a * 256]; };
  const df64 vx = A2(H_VX, 0), vy = A2(H_VY, 0), vz = A3(H_VZ, 0);
  // ---- the three lower edges
  df64 t_xy = zero, t_xz = zero, t_yz = zero;
  const bool li = INNER || (i > 0 && ci), lj = INNER || (j > 0 && cj);   // inner faces below in x, y
  if (li && lj) {
    t_xy = fma(PW(S_EXY), mad(subn(vy, A2(H_VY, -1)), c.hrdx, mul(subn(vx, A2(H_VX, -kDfW)), c.hrdy)), PW(S_TXY));
  } else if (c.bg_on) {   // wall xy-edge under background shear (Eqs. 32-33)
    t_xy = PW(S_TXY);
  }
  if (k > 0) {
    if (li && cj)
      t_xz = fma(PW(S_EXZ), mad(subn(vz, A3(H_VZ, -1)), c.hrdx, mul(subn(vx, col.vx_d), c.hrdz)), PW(S_TXZ));
    if (ci && lj)
      t_yz = fma(PW(S_EYZ), mad(subn(vz, A3(H_VZ, -kDfW)), c.hrdy, mul(subn(vy, col.vy_d), c.hrdz)), PW(S_TYZ));
  }
  col.vx_d = vx;
  col.vy_d = vy;
  const df64 Pf = A3(H_PF, 0), ph = A3(H_PHI, 0), kc = A3(H_K, 0);
  if (ci && cj) {
    const df64 Pt = PW(S_PT);
    const df64 vxr = A2(H_VX, 1), vyr = A2(H_VY, kDfW), vz_u = A3p(H_VZ);
    const df64 gx = mul(subn(vxr, vx), c.rdx), gy = mul(subn(vyr, vy), c.rdy), gz = mul(subn(vz_u, vz), c.rdz);
    const df64 divV = norm(add(add(gx, gy), gz));
    const df64 w = rcp(sub(df64(1.0f, 0.0f), ph)), ieta = PW(S_IETA);
    const df64 cc = c.compaction_on ? ieta * w : zero;
    const df64 Pto = PW(S_PTO), Pfo = PW(S_PFO);
    const df64 dPt = subn(Pt, Pto), dPf = subn(Pf, Pfo), dpp = subn(Pt, Pf);
    const df64 divVn = fma(dpp, cc, fma(-c.bd_rdt_a, dPf, fma(c.bd_rdt, dPt, divV)));
    // Darcy flux through the six faces (zero on the boundary) and the largest neighbour k; the advection
    // sums v_r phi_r - v_l phi_l over the same faces (wall velocities are zero)
    df64 kmax = kc, sx = zero, sy = zero, ax = zero, ay = zero;
    if (INNER || i > 0) {
      const df64 kn = A3(H_K, -1);
      kmax = lean_detail::pos_max(kmax, kn);
      sx = (kn + kc) * subn(A3(H_PF, -1), Pf);
      ax = mul(-vx, A3(H_PHI, -1));
    }
    if (INNER || i < b.nx - 1) {
      const df64 kn = A3(H_K, 1);
      kmax = lean_detail::pos_max(kmax, kn);
      sx = fma(kc + kn, subn(A3(H_PF, 1), Pf), sx);
      ax = mad(vxr, A3(H_PHI, 1), ax);
    }
    if (INNER || j > 0) {
      const df64 kn = A3(H_K, -kDfW);
      kmax = lean_detail::pos_max(kmax, kn);
      sy = (kn + kc) * subn(A3(H_PF, -kDfW), Pf);
      ay = mul(-vy, A3(H_PHI, -kDfW));
    }
    if (INNER || j < b.ny - 1) {
      const df64 kn = A3(H_K, kDfW);
      kmax = lean_detail::pos_max(kmax, kn);
      sy = fma(kc + kn, subn(A3(H_PF, kDfW), Pf), sy);
      ay = mad(vyr, A3(H_PHI, kDfW), ay);
    }
    df64 fz_u = zero, az = zero;
    if (k > 0) {
      kmax = lean_detail::pos_max(kmax, col.k_d);
      az = mul(-vz, col.phi_d);
    }
    if (up) {
      const df64 k_u = A3p(H_K);
      kmax = lean_detail::pos_max(kmax, k_u);
      fz_u = (kc + k_u) * (subn(A3p(H_PF), Pf) + c.buoy_dz);
      az = mad(vz_u, A3p(H_PHI), az);
    }
    const df64 sz = subn(fz_u, col.fz);
    col.fz = fz_u;
    // div qD = -1/2 sum_d rd^2 [(k + k_r)(Pf_r - Pf) - (k_l + k)(Pf - Pf_l)]
    const df64 divqD = -fma(sx, c.hrdx2, fma(sy, c.hrdy2, sz * c.hrdz2));
    const df64 resF = fma(-dpp, cc, fma(-c.bd_rdt_a, dPt, fma(c.bda_B_rdt, dPf, divqD)));
    // local-implicit pressure updates, Eqs. 17-18: P1 = P - res / (1/dtau + d res/dP)
    const df64 Pt1 = norm(mad(-rcp(add(PW(S_IDTP), cc)), divVn, Pt));
    const df64 Pf1 = norm(mad(-rcp(add(mad(kmax, c.ifac_pf, c.bda_B_rdt), cc)), resF, Pf));
    // normal deviatoric stresses (Eq. 21): tau = tau_o xi/(1+xi) + 2 mu/(1+xi) (edot + beta_n divVn)
    df64 s3n = mul(divV, df64(-1.0 / 3.0));
    if (c.beta_n.hi != 0.0f) s3n = mad(c.beta_n, divVn, s3n);
    const df64 cm2 = PW(S_CM2);
    const df64 sxx = fma(cm2, norm(add(gx, s3n)), PW(S_TXX));
    const df64 syy = fma(cm2, norm(add(gy, s3n)), PW(S_TYY));
    const df64 szz = fma(cm2, norm(add(gz, s3n)), PW(S_TZZ));
    // porosity in log space (Eq. 22): L = Lo + delta (see lean_cell_level)
    const df64 adv = mul(-w, mad(half(-ph), divV, mad(ax, c.hrdx, mad(ay, c.hrdy, mul(az, c.hrdz)))));
    const df64 dp1 = sub(Pf1, Pt1);
    const df64 rate = c.compaction_on ? mad(dp1, ieta, adv) : adv;
    const df64 delta = -norm(mad(c.beta_phi, sub(dp1, sub(Pfo, Pto)), mul(c.dt, rate)));
    const df64 em = lean_detail::df_expm1(delta);
    const df64 phio = PW(S_PHIO);
    const df64 ph1 = norm(mad(sub(phio, df64(1.0f, 0.0f)), em, phio));
    const df64 K = K0 ? K0[q] : c.k0r3;
    out.Pt[q] = Pt1;
    out.Pf[q] = Pf1;
    out.txx[q] = sxx;
    out.tyy[q] = syy;
    out.tzz[q] = szz;
    out.phi[q] = ph1;
    out.perm[q] = K * ph1 * ph1 * ph1;
    if (check) {
      const unsigned long long a = (unsigned long long)__double_as_longlong(fabs((double)divVn));
      const unsigned long long f = (unsigned long long)__double_as_longlong(fabs((double)resF));
      m_pt = a > m_pt ? a : m_pt;                    // bit patterns: a NaN stays the largest
      m_pf = f > m_pf ? f : m_pf;
    }
  }
  if (INNER || (i <= b.nx && j <= b.ny)) {
    out.txy[q] = t_xy;
    if (cj) out.txz[q] = t_xz;
    if (ci) out.tyz[q] = t_yz;
  }
  col.phi_d = ph;
  col.k_d = kc;
}

// Momentum residual, damped R and velocity update of the three lower faces of the cell (i, j, k).
__device__ __forceinline__ void df_face_point(const Box& b, const LeanCoef<df64>& c, const LeanFaceIn<df64>& in,
                                              df64* Vx, df64* Vy, df64* Vz, df64* Rx, df64* Ry, df64* Rz, int i, int j, int k, int check, double& r_v) {
  using namespace dfu;
  if (i >= b.nx || j >= b.ny || k >= b.nz) return;   // the faces i = nx, j = ny, k = nz are walls
  const long long q = cidx(b, i, j, k);
  const long long px = b.px, pxy = b.pxy;
  const bool fx = i > 0, fy = j > 0, fz = k > 0;
  // all loads before the first store (the arrays are not declared non-aliasing)
  const df64 zero(0.0f, 0.0f);
  df64 Fx = zero, Fy = zero, Fz = zero, Rx1 = zero, Ry1 = zero, Rz1 = zero, Vx1 = zero, Vy1 = zero, Vz1 = zero;
  const df64 P = in.Pt1[q], dtv = in.dtv_x[q];       // dtv: half the centre's dtau_V
  const df64 txy = in.txy[q], txz = in.txz[q], tyz = in.tyz[q];
  // F / rho_i directly (the spacings carry 1/rho_i); the norm takes |F| = rho_i |F / rho_i|
  if (fx) {
    Fx = mad(subn(subn(in.txx[q], in.txx[q - 1]), subn(P, in.Pt1[q - 1])), c.rdx_r,
             mad(subn(in.txy[q + px], txy), c.rdy_r, mul(subn(in.txz[q + pxy], txz), c.rdz_r)));
    Rx1 = norm(mad(c.damp_x, Rx[q], Fx));
    Vx1 = norm(mad(add(in.dtv_x[q - 1], dtv), Rx1, Vx[q]));
  }
  if (fy) {
    Fy = mad(subn(subn(in.tyy[q], in.tyy[q - px]), subn(P, in.Pt1[q - px])), c.rdy_r,
             mad(subn(in.txy[q + 1], txy), c.rdx_r, mul(subn(in.tyz[q + pxy], tyz), c.rdz_r)));
    Ry1 = norm(mad(c.damp_y, Ry[q], Fy));
    Vy1 = norm(mad(add(in.dtv_x[q - px], dtv), Ry1, Vy[q]));
  }
  if (fz) {
    // buoyancy -(rho g - rho_BG g) averaged to the face: -((phi_d + phi) / 2 - phi0) drho_g
    Fz = mad(subn(subn(in.tzz[q], in.tzz[q - pxy]), subn(P, in.Pt1[q - pxy])), c.rdz_r,
             mad(subn(in.txz[q + 1], txz), c.rdx_r,
                 mad(subn(in.tyz[q + px], tyz), c.rdy_r,
                     mul(subn(half(add(in.phi[q - pxy], in.phi[q])), c.phi0), -c.drho_g_r))));
    Rz1 = norm(mad(c.damp_z, Rz[q], Fz));
    Vz1 = norm(mad(add(in.dtv_x[q - pxy], dtv), Rz1, Vz[q]));
  }
  if (fx) { Rx[q] = Rx1; Vx[q] = Vx1; }
  if (fy) { Ry[q] = Ry1; Vy[q] = Vy1; }
  if (fz) { Rz[q] = Rz1; Vz[q] = Vz1; }
  if (check) {
    const double m = lean_detail::abs_max(lean_detail::abs_max((double)Fx, (double)Fy), (double)Fz);
    r_v = m * (double)c.rho_i;
  }
}

}  // namespace pt
