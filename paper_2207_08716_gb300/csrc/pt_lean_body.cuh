// pt_lean_body.cuh — per-point bodies of the FP64-lean PT kernels (see pt_lean_kernels.cu for
// the method), shared by the single-instance kernels and the batched (ensemble) kernels.
#pragma once

#include "df64.cuh"
#include "pt_lean.cuh"

namespace pt {
namespace lean_detail {

// exp(d) - 1 and exp(-d) - 1 from the Taylor series of exp split into its odd part
// O = d + d^3/3! + ... and even part E = d^2/2! + d^4/4! + ... (truncated after d^3 / d^2 for
// |d| <= 2^-20 and after d^9 / d^8 for |d| <= 2^-6: in both cases the first dropped term is
// below 2^-60 |d|). expm1(d) = E + O, expm1(-d) = E - O.
__device__ inline void expm1_pair(double d, double& em_pos, double& em_neg) {
  const int ad = __double2hiint(d) & 0x7fffffff;      // |d|'s upper word: the tiers off the FP64 pipe
  if (ad < 0x3eb00000) {                              // |d| < 2^-20
    const double d2 = d * d;
    const double O = d * fma(d2, 1.0 / 6.0, 1.0);
    em_pos = fma(0.5, d2, O);
    em_neg = fma(0.5, d2, -O);
  } else if (ad < 0x3f900000) {                       // |d| < 2^-6
    const double d2 = d * d;
    const double E = d2 * fma(d2, fma(d2, fma(d2, 1.0 / 40320.0, 1.0 / 720.0), 1.0 / 24.0), 0.5);
    const double O = d * fma(d2, fma(d2, fma(d2, fma(d2, 1.0 / 362880.0, 1.0 / 5040.0), 1.0 / 120.0), 1.0 / 6.0), 1.0);
    em_pos = E + O;
    em_neg = E - O;
  } else {
    em_pos = expm1(d);
    em_neg = expm1(-d);
  }
}

// The FP64 pipe takes a warp instruction every 16 cycles, in which an SM issues 64 others: conversions
// between FP64 and FP32 and one halving, which run on it, are done on the integers. (Other powers of two
// are folded into the coefficients they meet: nothing changes the exponent of a value that may be
// anything.)
// x / 2 for |x| >= 2^-1021, infinities and NaN staying what they are
__device__ inline double half_of(double x) {
  const int hi = __double2hiint(x);
  return __hiloint2double((hi & 0x7ff00000) == 0x7ff00000 ? hi : hi - 0x00100000, __double2loint(x));
}
// x to FP32, to nearest even as the conversion rounds; values outside FP32's normal range take that
__device__ inline float to_float(double x) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x), a = hi & 0x7fffffffu;
  if (a - 0x38100000u >= 0x47f00000u - 0x38100000u) return (float)x;
  const unsigned t = __funnelshift_l(lo, a - 0x38000000u, 3);     // |x| >> 29, exponent rebased
  return __uint_as_float((t + (((lo & 0x1fffffffu) + 0x0fffffffu + (t & 1u)) >> 29)) | (hi & 0x80000000u));
}

// max of positive values through their bit patterns (monotone for x > 0)
__device__ inline double pos_max(double a, double b) {
  const long long ia = __double_as_longlong(a), ib = __double_as_longlong(b);
  return __longlong_as_double(ia > ib ? ia : ib);
}

// 1 / x for the local-implicit pseudo-step denominators (x > 0, far inside the normal range):
// the hardware's approximate reciprocal refined by one Newton step, r' = r + r (1 - x r), whose
// relative error is the square of the seed's (the approximate FP64 reciprocal is good to about
// 2^-20, so ~2^-40 after the step; measured below 1e-12). It only scales the pseudo-time step of
// the update P - res / x, so the fixed point of the iteration does not depend on it.
__device__ inline double rcp_pseudo(double x) {
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
  return fma(r, fma(-x, r, 1.0), r);
}

// 1 / x to rounding accuracy for the coefficients that set the fixed point (x > 0, normal): one
// third-order step r (1 + e + e^2), e = 1 - x r, on the hardware's approximate reciprocal r (good to
// about 2^-20, so e^3 is below the rounding): three FP64 instructions, where two Newton steps take four.
__device__ inline double rcp_full(double x) {
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
  const double e = fma(-x, r, 1.0);
  return fma(r, fma(e, e, e), r);
}

// sqrt(x), x > 0 and normal, from the hardware's approximate reciprocal root r: s = x r,
// e = 1 - x r^2, sqrt(x) = s (1 - e)^(-1/2) = s (1 + e/2 + 3 e^2 / 8 + ...): five FP64 instructions.
__device__ inline double sqrt_full(double x) {
  double r;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
  const double s = x * r, e = fma(-s, r, 1.0);
  return fma(s * e, fma(0.375, e, 0.5), s);
}

// x^(1/m) for 3 <= m <= 64 with rx = 1/x: from the FP32 root y (|t| <= 64 2^-20 for
// t = (x - y^m) / x) by the series above; the first dropped term is below 2^-57. y^m by square and
// multiply, m is uniform. For m = 10 10 FP64 instructions, where exp(log x / 10) takes some 45.
// x far from 1 (never near a solution) falls back to the library functions, a NaN stays one.
__device__ inline double root_full(double x, double rx, int m, const RootSeries& k) {
  const int e2 = (__double2hiint(x) >> 20) - 1023;      // a negative x falls outside too
  if (e2 < -60 || e2 > 60) return exp(k.a * log(x));
  float lg, y0;
  // the seed from x cut to 24 bits
  const float xf = __uint_as_float(__funnelshift_l((unsigned)__double2loint(x),
                                                   (unsigned)__double2hiint(x) - 0x38000000u, 3));
  asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(lg) : "f"(xf));
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y0) : "f"(lg * k.af));
  const unsigned yb = __float_as_uint(y0);              // to FP64 exactly, normal in FP32
  const double y = __hiloint2double((int)((yb >> 3) + 0x38000000u), (int)(yb << 29));
  int e = m;
  double b = y;
  while (!(e & 1)) {
    b *= b;
    e >>= 1;
  }
  double ym = b;
  for (e >>= 1; e; e >>= 1) {
    b *= b;
    if (e & 1) ym *= b;
  }
  const double t = (x - ym) * rx;
  return fma(y, t * fma(t, fma(t, k.c, k.b), k.a), y);
}

// ---- the same operations in double-float (PT_DF64): one Newton step from the FP32 seed
// reaches the format's own rounding (~2^-46)
__device__ inline df64 rcp_full(df64 x) { return df_rcp(x); }

__device__ inline df64 pos_max(df64 a, df64 b) { return a < b ? b : a; }

// exp(d) - 1 with the tiers of the FP64 pair: for |d| <= 2^-20 d + d^2/2 + d^3/6 with d^2 exact to the
// pair and the cubic term (below 2^-42 |d|) in FP32; up to 2^-6 the split series; outside them the library
// expm1 in FP64.
__device__ inline df64 df_expm1(df64 d) {
  const float ad = fabsf(d.hi);
  if (ad <= 0x1p-20f) {
    const float p = __fmul_rn(d.hi, d.hi);
    const float e = __fmaf_rn(2.0f * d.hi, d.lo, __fmaf_rn(d.hi, d.hi, -p));   // d^2 = p + e
    float s, t;
    dfd::fast_two_sum(d.hi, 0.5f * p, s, t);
    return dfd::renorm(s, __fadd_rn(t, __fmaf_rn(p * d.hi, 1.0f / 6.0f, __fmaf_rn(0.5f, e, d.lo))));
  }
  if (ad <= 0.015625f) {
    const df64 d2 = d * d;
    const df64 E = d2 * fma(d2, fma(d2, fma(d2, df64(1.0 / 40320.0), df64(1.0 / 720.0)), df64(1.0 / 24.0)),
                            df64(0.5));
    const df64 O = d * fma(d2, fma(d2, fma(d2, fma(d2, df64(1.0 / 362880.0), df64(1.0 / 5040.0)),
                                           df64(1.0 / 120.0)), df64(1.0 / 6.0)), df64(1.0));
    return E + O;
  }
  return df64(expm1((double)d));
}

// conversions between the field type and FP64 (identity for FP64)
__device__ inline double to_d(double x) { return x; }
__device__ inline double to_d(df64 x) { return (double)x; }
template <class T>
__device__ inline T from_d(double x) { return T(x); }

// x^rel of the log-space Picard relaxation (x > 0, rx = 1/x): the square root for rel = 1/2, the
// m-th root for rel = 1/m (root = m, set on the host), else exp(rel log x) in FP64.
__device__ inline double relax_pow(double x, double rx, double rel, int root, const RootSeries& k) {
  if (root == 2) return sqrt_full(x);
  if (root > 2) return root_full(x, rx, root, k);
  return exp(rel * log(x));
}
__device__ inline df64 relax_pow(df64 x, df64 /*rx*/, double rel, int root, const RootSeries& /*k*/) {
  if (root == 2) return df_sqrt(x);
  if (root > 2) return df_root(x, root);
  return df64(exp(rel * log((double)x)));
}

// max of |values| whose NaN is the largest, through bit patterns. The sign is cleared in assembly: the
// compiler takes a mask of it for fabs, an addition on the FP64 pipe.
__device__ inline unsigned long long abs_bits(double x) {
  unsigned long long u;
  asm("and.b64 %0, %1, 0x7fffffffffffffff;" : "=l"(u) : "l"(__double_as_longlong(x)));
  return u;
}
__device__ inline double abs_max(double a, double b) {
  const unsigned long long ia = abs_bits(a), ib = abs_bits(b);
  return __longlong_as_double((long long)(ia > ib ? ia : ib));
}
__device__ inline df64 abs_max(df64 a, df64 b) { return a < b ? b : a; }   // positive values; drops a NaN

}  // namespace lean_detail

// Which arrays a form stores. The FP64 form is bound by the FP64 pipe and stores everything that
// changes less often than every iteration (1/(1-phi) and k travelling with phi, 1 - phi_o and its
// reciprocal, edge moduli pre-multiplied by both spacings, three face pseudo-steps). The double-float
// form is bound by HBM and instruction issue, so it recomputes 1/(1-phi), 1 - phi_o and its reciprocal,
// keeps one modulus per edge (em2_* hold 2 mu/(1+xi); eb_* unused) and one velocity pseudo-step per
// centre (dtv_x = dtv_y = dtv_z hold half of fac / mu; a face adds its two): 56 fewer bytes per cell and
// iteration. k(phi) travels with phi in both (recomputing it for the cell and its six neighbours costs
// more issue slots than its 16 bytes).
template <class T>
struct LeanRecompute { static constexpr bool value = false; };
template <>
struct LeanRecompute<df64> { static constexpr bool value = true; };

// Shared-memory stage of the double-float cells kernel (pointwise arrays, slot order).
enum { S_PTO, S_PFO, S_PHIO, S_IETA, S_IDTP, S_CM2, S_TXX, S_TYY, S_TZZ, S_EXY, S_EXZ, S_EYZ, S_TXY, S_TXZ,
       S_TYZ, kStageSlots };

// Cells of a column in FP64, level by level: pressures, porosity, k, 1/(1-phi), stresses of the centre and
// of its three lower edges. The form is bound by the FP64 pipe, so what the level below has formed or
// loaded is carried: the Darcy term through the lower z face, and the z-neighbours' values.
struct LeanColumn {
  double Pf, kk, phi, vz;          // own values at the current level
  double k_d, phi_d, vx_d, vy_d;   // one level below
  double fz;                       // (k_d + k) (Pf - Pf_d + buoyancy), 0 at the floor
};

__device__ __forceinline__ LeanColumn lean_column(const Box& b, const LeanCoef<double>& c,
                                                  const LeanCellIn<double>& in, int i, int j, int k) {
  const long long q = cidx(b, i, j, k);
  LeanColumn s;
  s.Pf = in.Pf[q];
  s.kk = in.perm[q];
  s.phi = in.phi[q];
  s.vz = in.Vz[q];
  s.k_d = s.phi_d = s.vx_d = s.vy_d = s.fz = 0.0;
  if (k > 0) {
    const long long d = q - b.pxy;
    s.k_d = in.perm[d];
    s.phi_d = in.phi[d];
    s.vx_d = in.Vx[d];
    s.vy_d = in.Vy[d];
    s.fz = (s.k_d + s.kk) * ((s.Pf - in.Pf[d]) + c.buoy_dz);
  }
  return s;
}

// Level k in [0, nz) (the level nz holds walls only) at i <= nx, j <= ny; leaves the column at k + 1.
__device__ __forceinline__ void lean_cell_level(const Box& b, const LeanCoef<double>& c,
                                                const LeanCellIn<double>& in, const LeanCellOut<double>& out, int i,
                                                int j, int k, int check, LeanColumn& col, double& r_pt, double& r_pf) {
  using namespace lean_detail;
  const long long q = cidx(b, i, j, k);
  const long long px = b.px, pxy = b.pxy;
  const double vx = in.Vx[q], vy = in.Vy[q], vz = col.vz, vz_u = in.Vz[q + pxy];
  const bool up = k < b.nz - 1;
  double Pf_u = 0.0, k_u = 0.0, phi_u = 0.0;
  if (up) {
    Pf_u = in.Pf[q + pxy];
    k_u = in.perm[q + pxy];
    phi_u = in.phi[q + pxy];
  }
  // ---- edges owned by this index, stored at the end with the cell's outputs, after every load (the
  // arrays are not declared non-aliasing); toa_xy holds the background part too
  double t_xy = 0.0, t_xz = 0.0, t_yz = 0.0;
  const bool ix = i > 0 && i < b.nx, jy = j > 0 && j < b.ny;
  if (ix && jy) {
    t_xy = fma(in.eb_xy[q], vy - in.Vy[q - 1], fma(in.em2_xy[q], vx - in.Vx[q - px], in.toa_xy[q]));
  } else if (c.bg_on) {   // wall xy-edge under background shear (Eqs. 32-33)
    t_xy = in.toa_xy[q];
  }
  if (k > 0) {
    if (ix && j < b.ny)
      t_xz = fma(in.eb_xz[q], vz - in.Vz[q - 1], fma(in.em2_xz[q], vx - col.vx_d, in.toa_xz[q]));
    if (i < b.nx && jy)
      t_yz = fma(in.eb_yz[q], vz - in.Vz[q - px], fma(in.em2_yz[q], vy - col.vy_d, in.toa_yz[q]));
  }
  double fz_u = 0.0;
  if (i < b.nx && j < b.ny) {
    const double Pt = in.Pt[q], Pf = col.Pf, Pto = in.Pto[q], Pfo = in.Pfo[q], ph = col.phi, kc = col.kk;
    const double ieta = in.ieta[q], w = in.w[q];
    const double vxr = in.Vx[q + 1], vyr = in.Vy[q + px];
    const double dvx = vxr - vx, dvy = vyr - vy, dvz = vz_u - vz;
    const double divV = fma(dvx, c.rdx, fma(dvy, c.rdy, dvz * c.rdz));
    const double cc = c.compaction_on ? ieta * w : 0.0;
    const double dPt = Pt - Pto, dPf = Pf - Pfo, dpp = Pt - Pf;
    // explicit fused multiply-adds: the same rounding in every kernel that inlines this body
    const double divVn = fma(dpp, cc, fma(-c.bd_rdt_a, dPf, fma(c.bd_rdt, dPt, divV)));
    // Darcy flux through the six faces (zero on the boundary), the largest neighbour k, and the
    // advection sums v_r phi_r - v_l phi_l over the same faces (wall velocities are zero)
    double kmax = pos_max(kc, col.k_d), sx = 0.0, sy = 0.0, ax = 0.0, ay = 0.0, az = -vz * col.phi_d;
    if (i > 0) {
      const double kn = in.perm[q - 1];
      kmax = pos_max(kmax, kn);
      sx = (kn + kc) * (in.Pf[q - 1] - Pf);
      ax = -vx * in.phi[q - 1];
    }
    if (i < b.nx - 1) {
      const double kn = in.perm[q + 1];
      kmax = pos_max(kmax, kn);
      sx = fma(kc + kn, in.Pf[q + 1] - Pf, sx);
      ax = fma(vxr, in.phi[q + 1], ax);
    }
    if (j > 0) {
      const double kn = in.perm[q - px];
      kmax = pos_max(kmax, kn);
      sy = (kn + kc) * (in.Pf[q - px] - Pf);
      ay = -vy * in.phi[q - px];
    }
    if (j < b.ny - 1) {
      const double kn = in.perm[q + px];
      kmax = pos_max(kmax, kn);
      sy = fma(kc + kn, in.Pf[q + px] - Pf, sy);
      ay = fma(vyr, in.phi[q + px], ay);
    }
    if (up) {
      kmax = pos_max(kmax, k_u);
      fz_u = (kc + k_u) * ((Pf_u - Pf) + c.buoy_dz);
      az = fma(vz_u, phi_u, az);
    }
    // div qD = -1/2 sum_d rd^2 [(k + k_r)(Pf_r - Pf) - (k_l + k)(Pf - Pf_l)]
    const double divqD = -fma(sx, c.hrdx2, fma(sy, c.hrdy2, (fz_u - col.fz) * c.hrdz2));
    // local-implicit pressure updates, Eqs. 17-18: P1 = P - res / (1/dtau + d res/dP), the
    // residuals being divVn (row Pt) and resF (row Pf)
    const double resF = fma(-dpp, cc, fma(-c.bd_rdt_a, dPt, fma(c.bda_B_rdt, dPf, divqD)));
    const double Pt1 = fma(-rcp_pseudo(in.idtp[q] + cc), divVn, Pt);   // idtp holds 1/dtau_Pt + beta_d/dt
    const double Pf1 = fma(-rcp_pseudo(fma(kmax, c.ifac_pf, c.bda_B_rdt) + cc), resF, Pf);
    // normal deviatoric stresses (Eq. 21): tau = tau_o xi/(1+xi) + 2 mu/(1+xi) (edot + beta_n divVn)
    const double s3 = fma(c.beta_n, divVn, divV * (-1.0 / 3.0));
    const double cm2 = in.cm2[q];
    const double sxx = fma(cm2, fma(dvx, c.rdx, s3), in.toa_xx[q]);
    const double syy = fma(cm2, fma(dvy, c.rdy, s3), in.toa_yy[q]);
    const double szz = fma(cm2, fma(dvz, c.rdz, s3), in.toa_zz[q]);
    // porosity in log space (Eq. 22): L = Lo + delta,
    // delta = -[beta_phi ((Pf1 - Pfo) - (Pt1 - Pto)) + dt (Pf1 - Pt1) / eta + dt V.grad(1-phi)/(1-phi)]
    // V.grad(1-phi)/(1-phi) = -(w/2) sum_d rd [v_r (phi_r - phi) + v_l (phi - phi_l)]
    //                      = -(w/2) [sum_d rd (v_r phi_r - v_l phi_l) - phi divV]
    const double adv = -half_of(w) * fma(ph, -divV, fma(ax, c.rdx, fma(ay, c.rdy, az * c.rdz)));
    const double dp1 = Pf1 - Pt1;
    const double rate = c.compaction_on ? fma(dp1, ieta, adv) : adv;
    const double delta = -fma(c.beta_phi, dp1 - (Pfo - Pto), c.dt * rate);
    double em_p, em_n;
    expm1_pair(delta, em_p, em_n);
    const double phio = in.phio[q], Eo = in.Eo[q], iEo = in.iEo[q];
    const double K = in.K0 ? in.K0[q] : c.k0r3;
    const double ph1 = fma(-Eo, em_p, phio);
    // every load above precedes the stores (the arrays are not declared non-aliasing)
    out.Pt[q] = Pt1;
    out.Pf[q] = Pf1;
    out.txx[q] = sxx;
    out.tyy[q] = syy;
    out.tzz[q] = szz;
    out.phi[q] = ph1;
    out.w[q] = fma(iEo, em_n, iEo);
    out.perm[q] = K * ph1 * ph1 * ph1;
    if (check) {   // of the column: a NaN stays the largest
      r_pt = abs_max(r_pt, divVn);
      r_pf = abs_max(r_pf, resF);
    }
  }
  out.txy[q] = t_xy;
  if (j < b.ny) out.txz[q] = t_xz;
  if (i < b.nx) out.tyz[q] = t_yz;
  col.k_d = col.kk; col.phi_d = col.phi; col.vx_d = vx; col.vy_d = vy; col.fz = fz_u;
  col.Pf = Pf_u; col.kk = k_u; col.phi = phi_u; col.vz = vz_u;
}

// Momentum residual, damped R and velocity update of the three lower faces of (i, j, k) in FP64; bit d
// of `mask` includes the face normal to direction d in the residual norm r_v.
__device__ __forceinline__ void lean_face_point(const Box& b, const LeanCoef<double>& c, const LeanFaceIn<double>& in,
                                                double* Vx, double* Vy, double* Vz, double* Rx, double* Ry, double* Rz,
                                                int i, int j, int k, int check, double& r_v, int mask = 7) {
  if (i < b.nx && j < b.ny && k < b.nz) {   // the faces i = nx, j = ny, k = nz are walls
    const long long q = cidx(b, i, j, k);
    const long long px = b.px, pxy = b.pxy;
    const bool fx = i > 0, fy = j > 0, fz = k > 0;
    // all loads before the first store (the arrays are not declared non-aliasing)
    double Fx = 0.0, Fy = 0.0, Fz = 0.0, Rx1 = 0.0, Ry1 = 0.0, Rz1 = 0.0, Vx1 = 0.0, Vy1 = 0.0, Vz1 = 0.0;
    // F / rho_i directly (the spacings carry 1/rho_i); the norm takes |F| = rho_i |F / rho_i|
    if (fx) {
      Fx = (in.txx[q] - in.txx[q - 1]) * c.rdx_r + (in.txy[q + px] - in.txy[q]) * c.rdy_r +
           (in.txz[q + pxy] - in.txz[q]) * c.rdz_r - (in.Pt1[q] - in.Pt1[q - 1]) * c.rdx_r;
      Rx1 = fma(c.damp_x, Rx[q], Fx);
      Vx1 = fma(in.dtv_x[q], Rx1, Vx[q]);
    }
    if (fy) {
      Fy = (in.txy[q + 1] - in.txy[q]) * c.rdx_r + (in.tyy[q] - in.tyy[q - px]) * c.rdy_r +
           (in.tyz[q + pxy] - in.tyz[q]) * c.rdz_r - (in.Pt1[q] - in.Pt1[q - px]) * c.rdy_r;
      Ry1 = fma(c.damp_y, Ry[q], Fy);
      Vy1 = fma(in.dtv_y[q], Ry1, Vy[q]);
    }
    if (fz) {
      // buoyancy -(rho g - rho_BG g) averaged to the face, rho g - rho_BG g = (phi - phi0) drho_g
      const double rog = (0.5 * (in.phi[q - pxy] + in.phi[q]) - c.phi0) * c.drho_g_r;
      Fz = (in.txz[q + 1] - in.txz[q]) * c.rdx_r + (in.tyz[q + px] - in.tyz[q]) * c.rdy_r +
           (in.tzz[q] - in.tzz[q - pxy]) * c.rdz_r - (in.Pt1[q] - in.Pt1[q - pxy]) * c.rdz_r - rog;
      Rz1 = fma(c.damp_z, Rz[q], Fz);
      Vz1 = fma(in.dtv_z[q], Rz1, Vz[q]);
    }
    if (fx) { Rx[q] = Rx1; Vx[q] = Vx1; }
    if (fy) { Ry[q] = Ry1; Vy[q] = Vy1; }
    if (fz) { Rz[q] = Rz1; Vz[q] = Vz1; }
    if (check) {
      double m = 0.0;
      if (mask & 1) m = Fx;
      if (mask & 2) m = lean_detail::abs_max(m, Fy);
      if (mask & 4) m = lean_detail::abs_max(m, Fz);
      r_v = lean_detail::abs_max(m, 0.0) * c.rho_i;
    }
  }
}

// Picard targets and relaxation at cell (i, j, k). m = max(x, 1/x) over the ratios x = mu*/mu
// and eta*/eta (>= 1): its log is the Picard change max(|log mu* - log mu|, |log eta* - log eta|),
// taken once per block by the caller (log is monotone).
template <class T>
__device__ __forceinline__ void lean_picard_point(const Box& b, const LeanCoef<T>& c, const LeanPicardIn<T>& in,
                                                  T* mu, T* eta, int i, int j, int k,
                                                  double& m) {
  using namespace lean_detail;
  if (i < b.nx && j < b.ny && k < b.nz) {
    const long long q = cidx(b, i, j, k);
    const long long px = b.px, pxy = b.pxy;
    const T axy = in.txy[q] + in.txy[q + 1] + in.txy[q + px] + in.txy[q + 1 + px];
    const T axz = in.txz[q] + in.txz[q + 1] + in.txz[q + pxy] + in.txz[q + 1 + pxy];
    const T ayz = in.tyz[q] + in.tyz[q + px] + in.tyz[q + pxy] + in.tyz[q + px + pxy];
    const T sxx = in.txx[q], syy = in.tyy[q], szz = in.tzz[q];
    // (tau_II / tau0)^2 = N / (2 tau0^2) + A / (16 tau0^2) with N = sxx^2 + syy^2 + szz^2 and A the sum of
    // the squares of the edges' sums (explicit FMAs: every form that inlines this body rounds it alike)
    const T N = fma(sxx, sxx, fma(syy, syy, szz * szz)), A = fma(axy, axy, fma(axz, axz, ayz * ayz));
    // Eq. 24: mu* = mu0 / (1 + (tau_II / tau0)^(n-1)); the log-space relaxation
    // exp(rel log mu* + (1 - rel) log mu) is written mu (mu* / mu)^rel (a square root for rel = 1/2)
    T den = T(1.0);
    if (c.powerlaw_on) {
      const T x2 = fma(N, c.rtau0_2h, A * c.rtau0_2s);
      const double p = c.n_pow - 1.0;
      den = p == 2.0 ? T(1.0) + x2 : from_d<T>(1.0 + exp(0.5 * p * log(to_d(x2))));
    }
    const T mu_old = mu[q], eta_old = eta[q];
    const T D = den * mu_old;
    const T x_mu = c.mu0 * rcp_full(D), rx_mu = D * c.rmu0;          // mu* / mu and its inverse
    const T mu_new = mu_old * relax_pow(x_mu, rx_mu, c.rel_mu, c.root_mu, c.series_mu);
    const T eta0R = (in.Pf1[q] > in.Pt1[q]) ? c.eta0_weak : c.eta0;
    // Eq. 26: eta* = eta0 mu / phi R (with the relaxed mu), relaxed the same way
    const T x_eta = eta0R * mu_new * rcp_full(in.phi1[q] * eta_old), rx_eta = rcp_full(x_eta);
    m = to_d(abs_max(abs_max(x_mu, rx_mu), abs_max(x_eta, rx_eta)));
    if constexpr (LeanRecompute<T>::value) {
      if (!(x_mu == x_mu && x_eta == x_eta)) m = to_d(x_mu) + to_d(x_eta);   // NaN stays NaN
    }
    mu[q] = mu_new;
    eta[q] = eta_old * relax_pow(x_eta, rx_eta, c.rel_eta, c.root_eta, c.series_eta);
  }
}

// Mean shear viscosity over the centres next to the xy-edge q = (i, j, .) that lie inside the
// grid (four inside, two on a wall, one in a corner), in a fixed order (1/n exact: n = 1, 2, 4).
template <class T>
__device__ inline T lean_edge_mean_mu_xy(const Box& b, const T* mu, long long q, int i, int j) {
  T s = T(0.0);
  int n = 0;
  if (i > 0 && j > 0) { s += mu[q - 1 - b.px]; ++n; }
  if (i < b.nx && j > 0) { s += mu[q - b.px]; ++n; }
  if (i > 0 && j < b.ny) { s += mu[q - 1]; ++n; }
  if (i < b.nx && j < b.ny) { s += mu[q]; ++n; }
  return s * T(n == 4 ? 0.25 : (n == 2 ? 0.5 : 1.0));
}

// Maxwell stress (Eq. 21) of viscosity m, xi = m rG: tau = (tau_o xi + 2 m edot) / (1 + xi), as
// tau_o + s (2 m edot - tau_o) with s = 1 / (1 + xi).
__device__ __forceinline__ double maxwell_s(double m, double rG) { return lean_detail::rcp_full(fma(m, rG, 1.0)); }
__device__ __forceinline__ double maxwell(double s, double m, double e2, double to) {   // e2 = 2 edot
  return fma(s, fma(m, e2, -to), to);
}
// An edge's stress from the sum of its four centres' viscosities and half its strain rate:
// xi = (m4 / 4) rG, 2 m edot = m4 (edot / 2)
__device__ __forceinline__ double edge_stress(const StressCoef& sc, double m4, double he, double to) {
  return maxwell(maxwell_s(m4, sc.rG4), m4, he, to);
}
// The three normal stresses of a centre of viscosity m (Eq. 21): twice the deviatoric strain rate and
// beta_n times the numerical divergence divVn.
__device__ __forceinline__ void centre_stresses(const StressCoef& sc, double m, double dvx, double dvy, double dvz,
                                                double divV, double divVn, double to_xx, double to_yy, double to_zz,
                                                double& txx, double& tyy, double& tzz) {
  const double s = maxwell_s(m, sc.rG), s3 = fma(sc.tbeta_n, divVn, divV * (-2.0 / 3.0));
  txx = maxwell(s, m, fma(dvx, sc.trdx, s3), to_xx);
  tyy = maxwell(s, m, fma(dvy, sc.trdy, s3), to_yy);
  tzz = maxwell(s, m, fma(dvz, sc.trdz, s3), to_zz);
}

// Shear stresses on the three lower edges of (i, j, k), zero on boundary edges unless a background
// shear is applied (Eqs. 32-33). An edge's viscosity is the mean of its four centres'.
__device__ __forceinline__ void stress_edges_point(const Box& b, const StressCoef& sc, const StressIn& in,
                                                   double* txy, double* txz, double* tyz, int i, int j, int k) {
  if (i > b.nx || j > b.ny || k > b.nz) return;
  const long long q = cidx(b, i, j, k);
  const long long px = b.px, pxy = b.pxy;
  if (k < b.nz) {
    double t = 0.0;
    if (i > 0 && i < b.nx && j > 0 && j < b.ny) {
      const double m4 = (in.mu[q - 1 - px] + in.mu[q - px]) + (in.mu[q - 1] + in.mu[q]);
      const double he = fma(in.Vx[q] - in.Vx[q - px], sc.qrdy, fma(in.Vy[q] - in.Vy[q - 1], sc.qrdx, sc.hebg));
      t = edge_stress(sc, m4, he, in.txyo[q]);
    } else if (sc.bg_on) {   // wall edge: background part only
      const double m = lean_edge_mean_mu_xy(b, in.mu, q, i, j);
      t = maxwell(maxwell_s(m, sc.rG), m, sc.tebg, in.txyo[q]);
    }
    txy[q] = t;
  }
  if (j < b.ny) {
    double t = 0.0;
    if (i > 0 && i < b.nx && k > 0 && k < b.nz) {
      const double m4 = (in.mu[q - 1 - pxy] + in.mu[q - pxy]) + (in.mu[q - 1] + in.mu[q]);
      const double he = fma(in.Vx[q] - in.Vx[q - pxy], sc.qrdz, (in.Vz[q] - in.Vz[q - 1]) * sc.qrdx);
      t = edge_stress(sc, m4, he, in.txzo[q]);
    }
    txz[q] = t;
  }
  if (i < b.nx) {
    double t = 0.0;
    if (j > 0 && j < b.ny && k > 0 && k < b.nz) {
      const double m4 = (in.mu[q - px - pxy] + in.mu[q - pxy]) + (in.mu[q - px] + in.mu[q]);
      const double he = fma(in.Vy[q] - in.Vy[q - pxy], sc.qrdz, (in.Vz[q] - in.Vz[q - px]) * sc.qrdy);
      t = edge_stress(sc, m4, he, in.tyzo[q]);
    }
    tyz[q] = t;
  }
}

// Coefficient refresh at box index (i, j, k).
template <class T>
__device__ __forceinline__ void lean_coef_point(const Box& b, const LeanCoef<T>& c, const LeanCoefIn<T>& in,
                                                const LeanCoefOut<T>& out, int i, int j, int k) {
  using namespace lean_detail;
  if (i > b.nx || j > b.ny || k > b.nz) return;
  const long long q = cidx(b, i, j, k);
  const long long px = b.px, pxy = b.pxy;
  constexpr bool RC = LeanRecompute<T>::value;
  const T rG = c.rGdtS;
  const T one = T(1.0), two = T(2.0);
  if (i < b.nx && j < b.ny && k < b.nz) {
    const T m = in.mu[q];
    const T s = rcp_full(fma(m, rG, one));
    const T a = one - s;                              // xi / (1 + xi)
    out.cm2[q] = two * m * s;
    out.toa_xx[q] = in.txxo[q] * a;
    out.toa_yy[q] = in.tyyo[q] * a;
    out.toa_zz[q] = in.tzzo[q] * a;
    out.idtp[q] = rcp_full(c.dtaupt_fac * m) + c.bd_rdt;   // 1/dtau_Pt + beta_d/dt
    out.ieta[q] = rcp_full(in.eta[q]);
  }
  if (k < b.nz && i > 0 && i < b.nx && j > 0 && j < b.ny) {
    const T m = T(0.25) * (in.mu[q - 1 - px] + in.mu[q - px] + in.mu[q - 1] + in.mu[q]);
    const T s = rcp_full(fma(m, rG, one));
    if constexpr (RC) {
      out.em2_xy[q] = two * m * s;
    } else {
      out.em2_xy[q] = two * m * s * c.hrdy;
      out.eb_xy[q] = two * m * s * c.hrdx;
    }
    // the background shear's stress 2 mu/(1+xi) tau_bg/(2 mu0) (Eqs. 32-33) joins the old-stress part
    out.toa_xy[q] = in.txyo[q] * (one - s) + two * m * s * c.ebg;
  } else if (k < b.nz && c.bg_on) {   // wall xy-edges carry the background stress
    const T m = lean_edge_mean_mu_xy(b, in.mu, q, i, j);
    const T s = rcp_full(fma(m, rG, one));
    out.toa_xy[q] = in.txyo[q] * (one - s) + two * m * s * c.ebg;
  }
  if (j < b.ny && i > 0 && i < b.nx && k > 0 && k < b.nz) {
    const T m = T(0.25) * (in.mu[q - 1 - pxy] + in.mu[q - pxy] + in.mu[q - 1] + in.mu[q]);
    const T s = rcp_full(fma(m, rG, one));
    if constexpr (RC) {
      out.em2_xz[q] = two * m * s;
    } else {
      out.em2_xz[q] = two * m * s * c.hrdz;
      out.eb_xz[q] = two * m * s * c.hrdx;
    }
    out.toa_xz[q] = in.txzo[q] * (one - s);
  }
  if (i < b.nx && j > 0 && j < b.ny && k > 0 && k < b.nz) {
    const T m = T(0.25) * (in.mu[q - px - pxy] + in.mu[q - pxy] + in.mu[q - px] + in.mu[q]);
    const T s = rcp_full(fma(m, rG, one));
    if constexpr (RC) {
      out.em2_yz[q] = two * m * s;
    } else {
      out.em2_yz[q] = two * m * s * c.hrdz;
      out.eb_yz[q] = two * m * s * c.hrdy;
    }
    out.toa_yz[q] = in.tyzo[q] * (one - s);
  }
  // pseudo-time steps of the velocities, mean of the two centres' dtau_V = fac / mu (the
  // recomputing forms store half the centre values and add two in the faces kernel)
  if constexpr (RC) {
    if (i < b.nx && j < b.ny && k < b.nz) out.dtv_x[q] = T(0.5) * c.dtauv_fac * rcp_full(in.mu[q]);
    return;
  }
  const T imu = (i < b.nx && j < b.ny && k < b.nz) ? rcp_full(in.mu[q]) : T(0.0);
  if (i > 0 && i < b.nx && j < b.ny && k < b.nz)
    out.dtv_x[q] = T(0.5) * c.dtauv_fac * (rcp_full(in.mu[q - 1]) + imu);
  if (j > 0 && j < b.ny && i < b.nx && k < b.nz)
    out.dtv_y[q] = T(0.5) * c.dtauv_fac * (rcp_full(in.mu[q - px]) + imu);
  if (k > 0 && k < b.nz && i < b.nx && j < b.ny)
    out.dtv_z[q] = T(0.5) * c.dtauv_fac * (rcp_full(in.mu[q - pxy]) + imu);
}

}  // namespace pt
