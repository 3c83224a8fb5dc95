// rb_setup.cu -- per-walker set-up (steps a1/a2): theta -> phase-basis
// coefficients, constant phase, detector delays and complex prefactors, and
// (for the gradient) their tangents.
//
// Waveform (Sec. II.B; TaylorF2 from the PN literature cited there):
//   h+ = A f^-7/6 (1+cos^2 i)/2 e^{-i Psi},  hx = -i A f^-7/6 cos i e^{-i Psi},
//   A = sqrt(5/24) pi^-2/3 Mc^5/6 / d_L,
//   Psi = 2 pi f t_c - phi_c - pi/4 + 3/(128 eta v^5) sum_k phi_k v^k, v = (pi M f)^1/3,
// point-particle phi_k to 3.5PN, aligned-spin 1.5PN (beta) and 2PN (sigma,
// kappa = 1) terms, and 5PN/6PN tidal terms written per body (equivalent to
// the Lambda-tilde / delta-Lambda-tilde form of the paper's appendix).
// Detector response: h_d = (F+ h+ + Fx hx) e^{-2 pi i f dt_d}, dt_d = -n.r_d/c.
//
// On sm_103a an FP64 warp instruction occupies its SM sub-partition's FP64
// unit for ~65 cycles whatever the number of active lanes, so what limits
// this step is the number of FP64 instructions each warp issues.  A block
// handles 32 walkers (one per lane) and splits each walker's FP64 work into
// roles run by different warps, exchanging results through shared memory:
//   phase 1  warp 0: ln(pi Mc), (pi Mc)^-5/3, (pi Mc)^1/3, Mc^5/6 / d_L
//            warp 1: eta, ln eta, eta^-1/5
//            warp 2: PN coefficients phi_k (polynomials in eta, X_i, chi_i, Lambda_i)
//            warp 3: sky direction, detector delays tau_d = t_c + dt_d
//            warp 4: polarisation and inclination sines/cosines
//   phase 2  warp 0: basis coefficients c_k, constant phase Phi0, their
//                    differences to the fiducial values, exp(-i dPhi0) - 1
//            warps 1-3: antenna factor P_d = F+ (1+cos^2 i)/2 - i Fx cos i (FP64,
//                    since F+ = D:(XX - YY) cancels)
//            warp 4: delay differences
//   phase 3  warps 1-3: prefactor ratio rho_d and rho_d - 1
//   (gradient) the warps after these: tangents, FP32 dual numbers (mixed modes)
//            or written out in FP64 from the phase-1 results.
// Every role is a noinline function, so a walker at theta_ref reproduces the
// fiducial values bit for bit (the reference kernel runs the same roles).
#include <type_traits>

#include "rb.h"
#include "rb_api_internal.h"
#include "rb_dd.cuh"
#include "rb_internal.cuh"
#include "rb_setup_dd.cuh"

namespace rb {

constexpr int kRoleThreads = 5 * 32;  // warps 0-4 take part in the FP64 phases

// Barrier over the FP64-phase warps only (the tangent warps run on their own).
__device__ __forceinline__ void roles_sync() { asm volatile("bar.sync 1, %0;" ::"n"(kRoleThreads) : "memory"); }

// ---------------------------------------------------------------------------
// Roles (FP64).  noinline: one instruction sequence for every caller.
// ---------------------------------------------------------------------------
__device__ __noinline__ void role_mass(double Mc, double dL, double* lnMc, double* N0, double* a1, double* amp) {
  const double l = log(kPi * Mc * kMsunS);
  *lnMc = l;
  *N0 = (3.0 / 128.0) * exp(-(5.0 / 3.0) * l);
  *a1 = exp(l * (1.0 / 3.0));
  // Mc^5/6 / d_L  (Msun^5/6 / Mpc):  Mc^5/6 = exp(5/6 l) / (pi G Msun / c^3)^5/6
  *amp = exp((5.0 / 6.0) * l) * (1.0 / 9.802409278970853e-05) / dL;
}

__device__ __noinline__ void role_eta(double q, double* eta, double* lneta, double* a2) {
  const double opq = 1.0 + q;
  const double e = q / (opq * opq);
  const double le = log(e);
  *eta = e;
  *lneta = le;
  *a2 = exp(-0.2 * le);  // eta^-1/5
}

// phi: phi2, phi3, phi4, phi5p, phi6c, phi7, phi10, phi12
__device__ __noinline__ void role_pn(double q, double chi1, double chi2, double L1, double L2, double* phi) {
  const double opq = 1.0 + q;
  const double eta = q / (opq * opq);
  const double X1 = 1.0 / opq, X2 = q / opq;
  const double X1_2 = X1 * X1, X2_2 = X2 * X2;
  const double X1_4 = X1_2 * X1_2, X2_4 = X2_2 * X2_2;
  const double beta = (chi1 * (113.0 * X1_2 + 75.0 * eta) + chi2 * (113.0 * X2_2 + 75.0 * eta)) / 12.0;
  const double sigma = eta * (474.0 / 48.0) * chi1 * chi2 + (486.0 / 96.0) * (X1_2 * chi1 * chi1 + X2_2 * chi2 * chi2);
  phi[0] = 3715.0 / 756.0 + (55.0 / 9.0) * eta;
  phi[1] = -16.0 * kPi + 4.0 * beta;
  phi[2] = 15293365.0 / 508032.0 + (27145.0 / 504.0) * eta + (3085.0 / 72.0) * eta * eta - 10.0 * sigma;
  phi[3] = kPi * (38645.0 / 756.0 - (65.0 / 9.0) * eta);
  phi[4] = 11583231236531.0 / 4694215680.0 - (640.0 / 3.0) * kPi * kPi - (6848.0 / 21.0) * kEulerGamma +
           eta * (-15737765635.0 / 3048192.0 + (2255.0 / 12.0) * kPi * kPi) + (76055.0 / 1728.0) * eta * eta -
           (127825.0 / 1296.0) * eta * eta * eta;
  phi[5] = kPi * (77096675.0 / 254016.0 + (378515.0 / 1512.0) * eta - (74045.0 / 756.0) * eta * eta);
  phi[6] = (-288.0 + 264.0 * X1) * X1_4 * L1 + (-288.0 + 264.0 * X2) * X2_4 * L2;
  phi[7] = X1_4 * L1 * (-15895.0 / 28.0 + 4595.0 / 28.0 * X1 + 5715.0 / 14.0 * X1_2 - 325.0 / 7.0 * X1_2 * X1) +
           X2_4 * L2 * (-15895.0 / 28.0 + 4595.0 / 28.0 * X2 + 5715.0 / 14.0 * X2_2 - 325.0 / 7.0 * X2_2 * X2);
}

// sky: sin/cos dec, sin/cos (ra - gmst); tau_d = t_c - n.r_d / c
__device__ __noinline__ void role_sky(double ra, double dec, double tc, const EventConst& ec, double* sky,
                                      double* tau) {
  double sd, cd, sa, ca;
  sincos(dec, &sd, &cd);
  sincos(ra - ec.gmst, &sa, &ca);
  sky[0] = sd;
  sky[1] = cd;
  sky[2] = sa;
  sky[3] = ca;
  const double n0 = cd * ca, n1 = cd * sa, n2 = sd;
  for (int d = 0; d < kMaxDet; ++d) {
    const DetGeom& g = ec.det[d];
    tau[d] = (d < ec.n_det) ? tc - (n0 * g.r[0] + n1 * g.r[1] + n2 * g.r[2]) / kClight : 0.0;
  }
}

__device__ __noinline__ void role_orient(double psi, double iota, double* o) {
  double sp, cp;
  sincos(psi, &sp, &cp);
  o[0] = sp;
  o[1] = cp;
  o[2] = cos(iota);
}

// c_k and Phi0 from the phase-1 results (see walker layout in rb_internal.cuh)
__device__ __noinline__ void role_coef(double lnMc, double N0, double a1, double a2, double lneta, const double* phi,
                                       double phic, double* c, double* phi0) {
  const double u = lnMc - 0.6 * lneta;  // ln(pi M)
  const double a = a1 * a2;             // (pi M)^1/3
  const double a2p = a * a, a3 = a2p * a, a4 = a2p * a2p, a5 = a4 * a, a6 = a3 * a3, a7 = a6 * a;
  const double a10 = a5 * a5, a12 = a6 * a6;
  c[0] = N0;
  c[1] = N0 * a2p * phi[0];
  c[2] = N0 * a3 * phi[1];
  c[3] = N0 * a4 * phi[2];
  c[4] = N0 * a5 * phi[3];                                                    // ln f
  c[5] = N0 * a6 * (phi[4] - (6848.0 / 21.0) * (1.3862943611198906 + u / 3.0));  // f^1/3 (ln 4 = 1.386...)
  c[6] = N0 * a6 * (-6848.0 / 63.0);                                          // f^1/3 ln f
  c[7] = N0 * a7 * phi[5];
  c[8] = N0 * a10 * phi[6];
  c[9] = N0 * a12 * phi[7];
  // -phi_c - pi/4 + the v^0 part of the 2.5PN term, 1 - 3 ln v_lso + ln(pi M), v_lso = 6^-1/2
  *phi0 = -phic - 0.25 * kPi + N0 * a5 * phi[3] * (1.0 + 1.5 * 1.791759469228055 + u);
}

// P_d = F+ (1 + cos^2 i)/2 - i Fx cos i,  F+ = X.DX - Y.DY,  Fx = X.DY + Y.DX
__device__ __noinline__ void role_antenna(const DetGeom& g, const double* sky, const double* ori, double* P) {
  const double sd = sky[0], cd = sky[1], sg = -sky[2], cg = sky[3];  // g = gmst - ra
  const double sp = ori[0], cp = ori[1], ci = ori[2];
  const double X[3] = {-cp * sg - sp * cg * sd, -cp * cg + sp * sg * sd, sp * cd};
  const double Y[3] = {sp * sg - cp * cg * sd, sp * cg + cp * sg * sd, cp * cd};
  double DX[3], DY[3];
  for (int i = 0; i < 3; ++i) {
    DX[i] = g.D[i][0] * X[0] + g.D[i][1] * X[1] + g.D[i][2] * X[2];
    DY[i] = g.D[i][0] * Y[0] + g.D[i][1] * Y[1] + g.D[i][2] * Y[2];
  }
  const double fp = (X[0] * DX[0] + X[1] * DX[1] + X[2] * DX[2]) - (Y[0] * DY[0] + Y[1] * DY[1] + Y[2] * DY[2]);
  const double fx = (X[0] * DY[0] + X[1] * DY[1] + X[2] * DY[2]) + (Y[0] * DX[0] + Y[1] * DX[1] + Y[2] * DX[2]);
  P[0] = fp * (1.0 + ci * ci) * 0.5;
  P[1] = -fx * ci;
}

__device__ __forceinline__ double wrap_pi(double x) { return x - kTwoPi * rint(x * (1.0 / kTwoPi)); }

// ---------------------------------------------------------------------------
// The block-level set-up: 32 walkers, phases 1-3 over warps 0-4 (+ tangents).
// ---------------------------------------------------------------------------
struct SetupSmem {
  double th[kNPar][kSetupWalkers];
  double lnMc[kSetupWalkers], N0[kSetupWalkers], a1[kSetupWalkers], amp[kSetupWalkers];
  double eta[kSetupWalkers], lneta[kSetupWalkers], a2[kSetupWalkers];
  double phi[8][kSetupWalkers];
  double sky[4][kSetupWalkers], tau[kMaxDet][kSetupWalkers];
  double ori[3][kSetupWalkers];
  double c[kNBasis][kSetupWalkers], phi0[kSetupWalkers];
  double P[kMaxDet][2][kSetupWalkers];
  double e64[2][kSetupWalkers];   // exp(-i dPhi0)
  int valid[kSetupWalkers];
};

// ---------------------------------------------------------------------------
// FP64 tangents, written out (the FP64 set-up's warps 5-9): from the phase-1
// results in shared memory, without the structurally zero terms that dual
// numbers carry.  An FP64 warp instruction costs ~65 clocks, and the dual-number
// form took ~1750 of them per detector and ~575 per pair of intrinsic
// parameters; here ~130 per detector, ~130 for q and ~90 for the others.  1000
// walkers, 3 detectors: set-up with the gradient 40.3 -> 19.4 us.
// ---------------------------------------------------------------------------
constexpr int kTan64Warps = 2 + kMaxDet;
constexpr int kTan64Threads = kRoleThreads + kTan64Warps * 32;
__device__ __forceinline__ void tangents_go() { asm volatile("bar.arrive 2, %0;" ::"n"(kTan64Threads) : "memory"); }
__device__ __forceinline__ void tangents_wait() { asm volatile("bar.sync 2, %0;" ::"n"(kTan64Threads) : "memory"); }

// Powers of a = (pi M)^1/3 times N0, ln(pi M), and the parts of c_5.
struct Pow64 {
  double N2, N3, N4, N5, N6, N7, N10, N12, u;
};
__device__ __forceinline__ Pow64 pow64(const SetupSmem& S, int l) {
  Pow64 p;
  const double a = S.a1[l] * S.a2[l], a2 = a * a, a4 = a2 * a2, N0 = S.N0[l];
  p.N2 = N0 * a2;
  p.N3 = p.N2 * a;
  p.N4 = N0 * a4;
  p.N5 = p.N4 * a;
  p.N6 = p.N4 * a2;
  p.N7 = p.N6 * a;
  p.N10 = p.N6 * a4;
  p.N12 = p.N10 * a2;
  p.u = S.lnMc[l] - 0.6 * S.lneta[l];
  return p;
}
constexpr double kC5 = -6848.0 / 21.0, kC6 = -6848.0 / 63.0, kLn4 = 1.3862943611198906;
constexpr double kPhi0Const = 1.0 + 1.5 * 1.791759469228055;  // 1 + 3/2 ln 6

// d / d(Mc, chi1, chi2, Lambda1, Lambda2): c_k goes as Mc^(m/3 - 5/3) (m the power of a),
// and linearly with the spin and tidal terms.
__device__ void tangents64_mass(const SetupSmem& S, int l, WalkerTan<double>& o) {
  const Pow64 p = pow64(S, l);
  const double Mc = S.th[0][l], q = S.th[1][l], chi1 = S.th[2][l], chi2 = S.th[3][l], eta = S.eta[l];
  const double iM = 1.0 / Mc, iM3 = iM * (1.0 / 3.0);
  const double c5 = p.N6 * fma(kC5, fma(p.u, 1.0 / 3.0, kLn4), S.phi[4][l]), c6 = p.N6 * kC6;
  o.dc[0][0] = S.N0[l] * (-5.0 * iM3);
  o.dc[1][0] = p.N2 * S.phi[0][l] * (-3.0 * iM3);
  o.dc[2][0] = p.N3 * S.phi[1][l] * (-2.0 * iM3);
  o.dc[3][0] = p.N4 * S.phi[2][l] * -iM3;
  o.dc[4][0] = 0.0;
  o.dc[5][0] = (c5 + 3.0 * c6) * iM3;
  o.dc[6][0] = c6 * iM3;
  o.dc[7][0] = p.N7 * S.phi[5][l] * (2.0 * iM3);
  o.dc[8][0] = p.N10 * S.phi[6][l] * (5.0 * iM3);
  o.dc[9][0] = p.N12 * S.phi[7][l] * (7.0 * iM3);
  o.dphi0[0] = p.N5 * S.phi[3][l] * iM;
  o.lnamp_Mc = (5.0 / 6.0) * iM;
  o.lnamp_dL = -1.0 / S.th[6][l];
  const double X1 = 1.0 / (1.0 + q), X2 = q * X1;
  const double X1_2 = X1 * X1, X2_2 = X2 * X2, e75 = 75.0 * eta, es = eta * (474.0 / 48.0);
#pragma unroll
  for (int k = 0; k < kNBasis; ++k)
#pragma unroll
    for (int j = 2; j < kNTanIntr; ++j)
      if (!((k == 2 || k == 3) && j < 4) && !(k >= 8 && j >= 4)) o.dc[k][j] = 0.0;
  // phi3 = -16 pi + 4 beta, phi4 = ... - 10 sigma
  o.dc[2][2] = p.N3 * ((1.0 / 3.0) * fma(113.0, X1_2, e75));
  o.dc[2][3] = p.N3 * ((1.0 / 3.0) * fma(113.0, X2_2, e75));
  o.dc[3][2] = p.N4 * (-10.0 * fma(es, chi2, (486.0 / 48.0) * X1_2 * chi1));
  o.dc[3][3] = p.N4 * (-10.0 * fma(es, chi1, (486.0 / 48.0) * X2_2 * chi2));
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const double X = i ? X2 : X1, Xs = i ? X2_2 : X1_2, X4 = Xs * Xs;
    o.dc[8][4 + i] = p.N10 * (fma(264.0, X, -288.0) * X4);
    o.dc[9][4 + i] = p.N12 * (X4 * fma(fma(fma(-325.0 / 7.0, X, 5715.0 / 14.0), X, 4595.0 / 28.0), X, -15895.0 / 28.0));
  }
}

// d / dq: eta' = (1 - q) / (1 + q)^3, (ln eta)' = (1 - q) / (q (1 + q)), X1' = -X1^2 = -X2',
// (ln a)' = -(ln eta)' / 5, u' = -3/5 (ln eta)'.
__device__ void tangents64_q(const SetupSmem& S, int l, WalkerTan<double>& o) {
  const Pow64 p = pow64(S, l);
  const double q = S.th[1][l], chi1 = S.th[2][l], chi2 = S.th[3][l], L1 = S.th[4][l], L2 = S.th[5][l], eta = S.eta[l];
  const double X1 = 1.0 / (1.0 + q), X2 = q * X1, X1_2 = X1 * X1;
  const double dle = (1.0 - q) * X1 / q, de = eta * dle, dla = -0.2 * dle, du = -0.6 * dle;
  const double dX1 = -X1_2, dX2 = X1_2;
  const double d2 = (55.0 / 9.0) * de;
  const double d3 = (1.0 / 3.0) * fma(chi1, fma(226.0 * X1, dX1, 75.0 * de), chi2 * fma(226.0 * X2, dX2, 75.0 * de));
  const double ds = fma(de * (474.0 / 48.0), chi1 * chi2, (486.0 / 48.0) * fma(X1 * dX1, chi1 * chi1, X2 * dX2 * (chi2 * chi2)));
  const double d4 = fma(fma(3085.0 / 36.0, eta, 27145.0 / 504.0), de, -10.0 * ds);
  const double d5 = (-kPi * 65.0 / 9.0) * de;
  const double d6 = fma(fma(-127825.0 / 432.0, eta, 76055.0 / 864.0), eta,
                        -15737765635.0 / 3048192.0 + (2255.0 / 12.0) * kPi * kPi) * de;
  const double d7 = fma(-kPi * 74045.0 / 378.0, eta, kPi * 378515.0 / 1512.0) * de;
  double d10 = 0.0, d12 = 0.0;
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const double X = i ? X2 : X1, LX = (i ? L2 * dX2 : L1 * dX1) * (X * X * X);
    d10 = fma(fma(1320.0, X, -1152.0), LX, d10);
    d12 = fma(fma(fma(fma(-7.0 * 325.0 / 7.0, X, 6.0 * 5715.0 / 14.0), X, 5.0 * 4595.0 / 28.0), X, -4.0 * 15895.0 / 28.0), LX, d12);
  }
  const double c5 = fma(kC5, fma(p.u, 1.0 / 3.0, kLn4), S.phi[4][l]);  // c_5 / N6
  o.dc[0][1] = 0.0;
  o.dc[1][1] = p.N2 * fma(2.0 * dla, S.phi[0][l], d2);
  o.dc[2][1] = p.N3 * fma(3.0 * dla, S.phi[1][l], d3);
  o.dc[3][1] = p.N4 * fma(4.0 * dla, S.phi[2][l], d4);
  const double t5 = fma(5.0 * dla, S.phi[3][l], d5);
  o.dc[4][1] = p.N5 * t5;
  o.dc[5][1] = p.N6 * fma(6.0 * dla, c5, fma(kC6, du, d6));
  o.dc[6][1] = p.N6 * (6.0 * kC6 * dla);
  o.dc[7][1] = p.N7 * fma(7.0 * dla, S.phi[5][l], d7);
  o.dc[8][1] = p.N10 * fma(10.0 * dla, S.phi[6][l], d10);
  o.dc[9][1] = p.N12 * fma(12.0 * dla, S.phi[7][l], d12);
  o.dphi0[1] = p.N5 * fma(t5, kPhi0Const + p.u, S.phi[3][l] * du);
}

// One detector's ln P and delay with respect to (iota, psi, ra, dec).  With
// F+ = X.DX - Y.DY, Fx = 2 X.DY and the polarisation frame's derivatives
//   d(X, Y)/dpsi = (Y, -X),  d(X, Y)/dra = (z x X, z x Y),  d(X, Y)/ddec = (-sin psi n, -cos psi n):
//   dF+/dpsi = 2 Fx, dFx/dpsi = -2 F+,  dF+ = 2 (DX.dX - DY.dY),  dFx = 2 (DY.dX + DX.dY).
__device__ void tangents64_det(const DetGeom& g, const SetupSmem& S, int l, double si, int d, WalkerTan<double>& o) {
  const double sd = S.sky[0][l], cd = S.sky[1][l], sg = -S.sky[2][l], cg = S.sky[3][l];  // g = gmst - ra
  const double sp = S.ori[0][l], cp = S.ori[1][l], ci = S.ori[2][l];
  const double X[3] = {-cp * sg - sp * cg * sd, -cp * cg + sp * sg * sd, sp * cd};
  const double Y[3] = {sp * sg - cp * cg * sd, sp * cg + cp * sg * sd, cp * cd};
  const double n[3] = {cd * cg, -cd * sg, sd};
  double DX[3], DY[3];
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    DX[i] = g.D[i][0] * X[0] + g.D[i][1] * X[1] + g.D[i][2] * X[2];
    DY[i] = g.D[i][0] * Y[0] + g.D[i][1] * Y[1] + g.D[i][2] * Y[2];
  }
  const double fp = (X[0] * DX[0] + X[1] * DX[1] + X[2] * DX[2]) - (Y[0] * DY[0] + Y[1] * DY[1] + Y[2] * DY[2]);
  const double fx = 2.0 * (X[0] * DY[0] + X[1] * DY[1] + X[2] * DY[2]);
  const double nX = n[0] * DX[0] + n[1] * DX[1] + n[2] * DX[2], nY = n[0] * DY[0] + n[1] * DY[1] + n[2] * DY[2];
  // dra: z x X = (-X1, X0, 0)
  const double fp_r = 2.0 * ((DX[1] * X[0] - DX[0] * X[1]) - (DY[1] * Y[0] - DY[0] * Y[1]));
  const double fx_r = 2.0 * ((DY[1] * X[0] - DY[0] * X[1]) + (DX[1] * Y[0] - DX[0] * Y[1]));
  const double fp_d = 2.0 * (cp * nY - sp * nX), fx_d = -2.0 * (sp * nY + cp * nX);
  const double ip = 0.5 * fma(ci, ci, 1.0);  // (1 + cos^2 iota) / 2
  const double Pr = fp * ip, Pi = -fx * ci;
  const double iden = 1.0 / (Pr * Pr + Pi * Pi);
  const double dPr[4] = {-fp * ci * si, 2.0 * fx * ip, fp_r * ip, fp_d * ip};
  const double dPi[4] = {fx * si, 2.0 * fp * ci, -fx_r * ci, -fx_d * ci};
#pragma unroll
  for (int j = 0; j < 4; ++j) {  // d ln P = dP conj(P) / |P|^2
    o.dlnP[d][j][0] = (dPr[j] * Pr + dPi[j] * Pi) * iden;
    o.dlnP[d][j][1] = (dPi[j] * Pr - dPr[j] * Pi) * iden;
  }
  o.dtd[d][0] = (cd * sg * g.r[0] + cd * cg * g.r[1]) * (-1.0 / kClight);
  o.dtd[d][1] = (-sd * cg * g.r[0] + sd * sg * g.r[1] + cd * g.r[2]) * (-1.0 / kClight);
}

__device__ void tangent64_warp(const SetupSmem& S, const EventConst& ec, double iota, WalkerTan<double>& o, int which) {
  const int l = threadIdx.x & 31;
  const int d = which - 2;
  const double si = d >= 0 && d < ec.n_det ? sin(iota) : 0.0;  // alongside phase 1
  tangents_wait();
  if (which == 0) tangents64_mass(S, l, o);
  else if (which == 1) tangents64_q(S, l, o);
  else if (d < ec.n_det) tangents64_det(ec.det[d], S, l, si, d, o);  // entries of detectors beyond n_det are never read
}

// Runs phases 1 and 2 for the walkers of this block and leaves the absolute
// values in shared memory.  Warps 0-4 (and only they) must call it.
// signal: warps waiting in tangents_wait() are let go after phase 1.
__device__ void setup_absolute(const double* __restrict__ theta, int64_t w0, int64_t W, const EventConst& ec,
                               SetupSmem& S, bool signal = false) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int i = threadIdx.x; i < kNPar * kSetupWalkers; i += kRoleThreads) {
    const int l = i / kNPar, j = i % kNPar;
    const int64_t w = (w0 + l < W) ? w0 + l : W - 1;  // pad with the last walker
    S.th[j][l] = theta[w * kNPar + j];
  }
  roles_sync();
  const int l = lane;
  if (warp == 0) {
    double th[kNPar];
    for (int j = 0; j < kNPar; ++j) th[j] = S.th[j][l];
    S.valid[l] = theta_valid(th) ? 1 : 0;
    role_mass(th[0], th[6], &S.lnMc[l], &S.N0[l], &S.a1[l], &S.amp[l]);
  } else if (warp == 1) {
    role_eta(S.th[1][l], &S.eta[l], &S.lneta[l], &S.a2[l]);
  } else if (warp == 2) {
    double phi[8];
    role_pn(S.th[1][l], S.th[2][l], S.th[3][l], S.th[4][l], S.th[5][l], phi);
    for (int k = 0; k < 8; ++k) S.phi[k][l] = phi[k];
  } else if (warp == 3) {
    double sky[4], tau[kMaxDet];
    role_sky(S.th[11][l], S.th[12][l], S.th[7][l], ec, sky, tau);
    for (int k = 0; k < 4; ++k) S.sky[k][l] = sky[k];
    for (int d = 0; d < kMaxDet; ++d) S.tau[d][l] = tau[d];
  } else if (warp == 4) {
    double o[3];
    role_orient(S.th[10][l], S.th[9][l], o);
    for (int k = 0; k < 3; ++k) S.ori[k][l] = o[k];
  }
  roles_sync();
  if (signal) tangents_go();
  if (warp == 0) {
    double phi[8], c[kNBasis], phi0;
    for (int k = 0; k < 8; ++k) phi[k] = S.phi[k][l];
    role_coef(S.lnMc[l], S.N0[l], S.a1[l], S.a2[l], S.lneta[l], phi, S.th[8][l], c, &phi0);
    for (int k = 0; k < kNBasis; ++k) S.c[k][l] = c[k];
    S.phi0[l] = phi0;
  } else if (warp >= 1 && warp <= kMaxDet) {
    const int d = warp - 1;
    if (d < ec.n_det) {
      double sky[4], ori[3], P[2];
      for (int k = 0; k < 4; ++k) sky[k] = S.sky[k][l];
      for (int k = 0; k < 3; ++k) ori[k] = S.ori[k][l];
      role_antenna(ec.det[d], sky, ori, P);
      S.P[d][0][l] = P[0];
      S.P[d][1][l] = P[1];
    } else {
      S.P[d][0][l] = S.P[d][1][l] = 0.0;
    }
  }
  roles_sync();
}

// FP64 reference kernel (FP64 and FP64-phase paths): one block; every lane
// evaluates theta_ref.
__global__ void __launch_bounds__(7 * 32) k_ref_values(const double* theta, EventConst ec, RefValues* out) {
  __shared__ SetupSmem S;
  setup_absolute(theta, 0, 1, ec, S);
  if (threadIdx.x == 0) {
    Values v;
    for (int k = 0; k < kNBasis; ++k) v.c[k] = S.c[k][0];
    v.phi0 = S.phi0[0];
    for (int d = 0; d < kMaxDet; ++d) {
      v.tau[d] = S.tau[d][0];
      v.P64[d][0] = S.P[d][0][0];
      v.P64[d][1] = S.P[d][1][0];
      v.P32[d][0] = (float)v.P64[d][0];
      v.P32[d][1] = (float)v.P64[d][1];
    }
    v.amp = S.amp[0];
    v.valid = S.valid[0];
    v.pad = 0;
    out->v = v;
  }
}

// Batch set-up in FP64 for the FP64 paths: RB_FP64 writes WalkerF64 (+
// double tangents), RB_MIXED_F64PHASE writes WalkerF64 (+ float tangents).
// (RB_MIXED uses the float-float set-up, k_setup_dd.)
template <int MODE>
constexpr int setup_threads(bool grad) {
  return !grad ? kRoleThreads : MODE == RB_FP64 ? kTan64Threads : kRoleThreads + kTanWarps * 32;
}
template <int MODE, bool GRAD>
__global__ void __launch_bounds__(setup_threads<MODE>(GRAD)) k_setup(const double* __restrict__ theta, int64_t W, EventConst ec,
                                                  const RefValues* __restrict__ ref, void* __restrict__ ws_out,
                                                  void* __restrict__ tan_out) {
  static_assert(MODE == RB_FP64 || MODE == RB_MIXED_F64PHASE, "RB_MIXED uses the float-float set-up");
  __shared__ SetupSmem S;
  const int64_t w0 = (int64_t)blockIdx.x * kSetupWalkers;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t w = w0 + lane;
  const bool mine = w < W;
  if (warp >= 5) {
    // tangents (gradient only): these warps take no part in the role barriers
    // (the FP64 ones start from the phase-1 results)
    if constexpr (GRAD && MODE == RB_FP64) {
      const int64_t wc = mine ? w : W - 1;  // pad lanes repeat the last walker's record
      tangent64_warp(S, ec, theta[wc * kNPar + 9], static_cast<WalkerTan<double>*>(tan_out)[wc], warp - 5);
    } else if constexpr (GRAD) {
      tangent_warp<float>(theta, W, w0, ec, static_cast<WalkerTan<float>*>(tan_out) + w0, warp - 5);
    }
    return;
  }
  setup_absolute(theta, w0, W, ec, S, GRAD && MODE == RB_FP64);
  const Values& r = ref->v;
  const int l = lane;
  if (warp == 0) {
    // constant-phase factor exp(-i dPhi0) (FP64; from the half angle for the FP64-phase mode)
    const double dphi0 = wrap_pi(S.phi0[l] - r.phi0);
    if (MODE == RB_FP64) {
      double sp, cp;
      sincos(dphi0, &sp, &cp);
      S.e64[0][l] = cp;
      S.e64[1][l] = -sp;
    } else {
      // exp(-i dPhi0) - 1 = -2 sin^2(pi y) - 2i sin(pi y) cos(pi y), y = dPhi0 / 2pi as a float pair,
      // plus the first-order term of the low part: d/dy exp(-2 pi i y) = -2 pi i exp(-2 pi i y)
      const double y64 = dphi0 * (1.0 / kTwoPi);
      const float yh = (float)y64, yl = (float)(y64 - (double)yh);
      float sn, cs;
      sincos_pi_half(yh, sn, cs);
      const float er = -2.f * sn * sn, ei = -2.f * sn * cs;
      const float t = 6.28318530717958648f * yl;
      S.e64[0][l] = 1.0 + ((double)er + (double)(ei * t));
      S.e64[1][l] = (double)ei - (double)((1.f + er) * t);
    }
  } else if (warp == 4 && mine) {
    for (int d = 0; d < kMaxDet; ++d) {
      const double dt = (d < ec.n_det) ? S.tau[d][l] - r.tau[d] : 0.0;
      static_cast<WalkerF64*>(ws_out)[w].tau[d] = dt;
    }
  }
  roles_sync();
  // phase 3: coefficient differences (warp 0) and prefactor ratios per detector (warps 1-3), FP64
  if (warp == 0 && mine) {
    WalkerF64* o = static_cast<WalkerF64*>(ws_out) + w;
    for (int k = 0; k < kNBasis; ++k) o->dc[k] = S.c[k][l] - r.c[k];
    o->valid = S.valid[l];
    o->pad = 0;
  } else if (warp >= 1 && warp <= kMaxDet && mine) {
    const int d = warp - 1;
    double rho_r = 0.0, rho_i = 0.0, sig_r = 0.0, sig_i = 0.0;
    if (d < ec.n_det) {
      // Q = ampr P exp(-i dPhi0);  rho = Q / P_ref;  sig = (Q - P_ref) / P_ref
      const double ampr = S.amp[l] / r.amp;
      const double er = S.e64[0][l], ei = S.e64[1][l];
      const double pr = S.P[d][0][l], pi = S.P[d][1][l];
      const double qr = ampr * (pr * er - pi * ei), qi = ampr * (pr * ei + pi * er);
      const double rr = r.P64[d][0], ri = r.P64[d][1];
      const double den = rr * rr + ri * ri;
      rho_r = (qr * rr + qi * ri) / den;
      rho_i = (qi * rr - qr * ri) / den;
      const double xr = qr - rr, xi = qi - ri;
      sig_r = (xr * rr + xi * ri) / den;
      sig_i = (xi * rr - xr * ri) / den;
    }
    WalkerF64* o = static_cast<WalkerF64*>(ws_out) + w;
    o->rho[d][0] = rho_r;
    o->rho[d][1] = rho_i;
    o->sig[d][0] = sig_r;
    o->sig[d][1] = sig_i;
  }
}


// Float-float reference kernel (mixed path and the fast summary build): one
// block, every lane evaluates theta_ref; also writes the reference copies
// used by the summary build (c/2pi, Phi0/2pi, tau as float pairs and the
// complex h0 prefactor K_d = A_ref P_d in FP64).
__global__ void __launch_bounds__(kDdRoleThreads) k_ref_dd(const double* theta, EventConst ec, RefValues* out,
                                                          SummarySync* base_reset) {
  __shared__ DdSmem S;
  // a fast summary build follows on the same stream: it leaves log L(theta_ref)
  // in the fixed-point accumulator, zeroed here
  if (base_reset && threadIdx.x == 0) {
    base_reset->base_acc = 0ull;
    base_reset->overflow = 0u;
    base_reset->base_in_acc = 1u;
  }
  // a kernel launched programmatically after this one (the chunk records of
  // the rebuild + batch step) may start and load its own inputs now; it waits
  // for this grid's completion before it reads the reference values
  asm volatile("griddepcontrol.launch_dependents;");
  setup_load_dd<true>(theta, 0, 1, S);
  setup_absolute_dd(ec, S);
  const int j = threadIdx.x;
  RefDD& R = out->dd;
  auto put = [](float* p, dd v) { p[0] = v.h; p[1] = v.l; };
  if (j < kNBasis) {
    const dd c = ld2(S.c[j][0]);
    put(R.c[j], c);
    put(out->chat[j], fx::mul(c, inv2pi()));
  } else if (j == kNBasis) {
    const dd p = ld2(S.phi0[0]);
    put(R.phi0, p);
    put(out->phi0t, fx::mul(p, inv2pi()));
  } else if (j == kNBasis + 1) {
    put(R.amp, ld2(S.amp[0]));
  } else if (j >= 32 && j < 32 + kMaxDet) {
    const int d = j - 32;
    const bool on = d < ec.n_det;
    const dd t = on ? ld2(S.tau[d][0]) : dd{0.f, 0.f};
    put(R.tau[d], t);
    put(out->taut[d], t);
    const dd pr = on ? ld2(S.P[d][0][0]) : dd{0.f, 0.f}, pi = on ? ld2(S.P[d][1][0]) : dd{0.f, 0.f};
    put(R.P[d][0], pr);
    put(R.P[d][1], pi);
    // sqrt(5/24) pi^{-2/3} (G Msun/c^3)^{5/6} / (1 Mpc / c): h0 amplitude per Msun^{5/6}/Mpc
    constexpr fx::cdd kAmpH(8.035028173395984e-06 / kMpcS);
    const dd a = fx::mul(fx::K(kAmpH), ld2(S.amp[0]));
    out->K[d][0] = fx::to_double(fx::mul(a, pr));
    out->K[d][1] = fx::to_double(fx::mul(a, pi));
  }
}

// Mixed batch set-up: WalkerMixed (+ float tangents on the warps after the
// role warps).
template <bool GRAD>
__device__ __forceinline__ void setup_dd_block(const double* __restrict__ theta, int64_t W, const EventConst& ec,
                                               const RefValues* __restrict__ ref, void* __restrict__ ws_out,
                                               void* __restrict__ tan_out) {
  __shared__ DdSmem S;
  const int64_t w0 = (int64_t)blockIdx.x * kSetupWalkers;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const bool mine = w0 + lane < W;
  if (warp >= kDdRoleWarps) {
    if (GRAD) tangent_warp<float>(theta, W, w0, ec, static_cast<WalkerTan<float>*>(tan_out) + w0, warp - kDdRoleWarps);
    return;
  }
  setup_load_dd<!GRAD>(theta, w0, W, S);
  setup_absolute_dd(ec, S);
  setup_record_dd(ref->dd, ec, S, static_cast<WalkerMixed*>(ws_out) + w0 + lane, mine);
}
template <bool GRAD>
__global__ void __launch_bounds__(kDdRoleThreads + kTanWarps * 32) k_setup_dd(const double* __restrict__ theta, int64_t W,
                                                                 EventConst ec, const RefValues* __restrict__ ref,
                                                                 void* __restrict__ ws_out,
                                                                 void* __restrict__ tan_out) {
  setup_dd_block<GRAD>(theta, W, ec, ref, ws_out, tan_out);
}
// With the gradient, held to the registers of three blocks per SM instead of two (40
// instead of 72, with spills: a full wave takes about a quarter longer), for
// batches it spares a wave.
__global__ void __launch_bounds__(kDdRoleThreads + kTanWarps * 32, 3) k_setup_dd_dense(const double* __restrict__ theta, int64_t W,
                                                                 EventConst ec, const RefValues* __restrict__ ref,
                                                                 void* __restrict__ ws_out,
                                                                 void* __restrict__ tan_out) {
  setup_dd_block<true>(theta, W, ec, ref, ws_out, tan_out);
}

// Host-side launchers.
cudaError_t launch_ref_values(const double* theta_ref_dev, const EventConst& ec, RefValues* out, cudaStream_t s) {
  k_ref_values<<<1, 5 * 32, 0, s>>>(theta_ref_dev, ec, out);
  return cudaGetLastError();
}

template <int MODE>
static cudaError_t launch_setup_t(const double* theta, int64_t W, const EventConst& ec, const RefValues* ref, void* ws,
                                  void* tan, bool grad, cudaStream_t s) {
  const unsigned grid = (unsigned)((W + kSetupWalkers - 1) / kSetupWalkers);
  if (grad)
    k_setup<MODE, true><<<grid, setup_threads<MODE>(true), 0, s>>>(theta, W, ec, ref, ws, tan);
  else
    k_setup<MODE, false><<<grid, 5 * 32, 0, s>>>(theta, W, ec, ref, ws, tan);
  return cudaGetLastError();
}

// Absolute values of W walkers for the full-grid likelihood (32 walkers per
// block, the float-float set-up of the mixed path; lane l writes walker w0 + l).
__global__ void __launch_bounds__(kDdRoleThreads) k_setup_abs(const double* __restrict__ theta, int64_t W,
                                                             EventConst ec, WalkerAbs* __restrict__ out) {
  __shared__ DdSmem S;
  const int64_t w0 = (int64_t)blockIdx.x * kSetupWalkers;
  setup_load_dd<true>(theta, w0, W, S);
  setup_absolute_dd(ec, S);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t w = w0 + lane;
  if (w >= W) return;
  WalkerAbs& o = out[w];
  auto put = [](float* p, dd v) { p[0] = v.h; p[1] = v.l; };
  if (warp == 0) {
    for (int k = 0; k < kNBasis; ++k) put(o.chat[k], fx::mul(ld2(S.c[k][lane]), inv2pi()));
    put(o.phi0t, fx::mul(ld2(S.phi0[lane]), inv2pi()));
    o.valid = S.valid[lane];
    o.pad[0] = o.pad[1] = o.pad[2] = 0;
  } else if (warp >= 1 && warp <= kMaxDet) {
    const int d = warp - 1;
    const bool on = d < ec.n_det;
    put(o.taut[d], on ? ld2(S.tau[d][lane]) : dd{0.f, 0.f});
    constexpr fx::cdd kAmpH(8.035028173395984e-06 / kMpcS);
    const dd a = fx::mul(fx::K(kAmpH), ld2(S.amp[lane]));
    o.K[d][0] = on ? fx::to_double(fx::mul(a, ld2(S.P[d][0][lane]))) : 0.0;
    o.K[d][1] = on ? fx::to_double(fx::mul(a, ld2(S.P[d][1][lane]))) : 0.0;
  }
}

cudaError_t launch_setup_abs(const double* theta, int64_t W, const EventConst& ec, WalkerAbs* out, cudaStream_t s) {
  const unsigned grid = (unsigned)((W + kSetupWalkers - 1) / kSetupWalkers);
  k_setup_abs<<<grid, kDdRoleThreads, 0, s>>>(theta, W, ec, out);
  return cudaGetLastError();
}

// The FP32 tangents alone, one warp per tangent group and 32 walkers per
// block: they depend on theta only, so the combined rebuild + batch runs them
// on a stream of their own from the start of the call.
__global__ void __launch_bounds__(kTanWarps * 32) k_tangents(const double* __restrict__ theta, int64_t W, EventConst ec,
                                                             void* __restrict__ tan_out) {
  const int64_t w0 = (int64_t)blockIdx.x * kSetupWalkers;
  tangent_warp<float>(theta, W, w0, ec, static_cast<WalkerTan<float>*>(tan_out) + w0, threadIdx.x >> 5);
}

cudaError_t launch_tangents(const double* theta, int64_t W, const EventConst& ec, void* tan, cudaStream_t s) {
  const unsigned grid = (unsigned)((W + kSetupWalkers - 1) / kSetupWalkers);
  k_tangents<<<grid, kTanWarps * 32, 0, s>>>(theta, W, ec, tan);
  return cudaGetLastError();
}

// Phase directions of the fiducial waveform for the bin placement without the
// PN ansatz: dc_k / dtheta_j at theta_ref (the mixed tangents' dual numbers in
// FP64), out[k][j] for j = Mc, q, chi1, chi2, Lambda1, Lambda2.
// With the basis functions g_k they give dPsi(f) / dtheta_j = sum_k out[k][j] g_k(f);
// the constant phase does not vary with f and is not needed.
__global__ void k_ref_phase_tangents(const double* __restrict__ theta_ref, double* __restrict__ out) {
  const int part = threadIdx.x;
  if (part >= 3) return;
  WalkerTan<double> t;
  tangents_intrinsic<double>(theta_ref, part, t);
  for (int k = 0; k < kNBasis; ++k)
    for (int j = 2 * part; j < 2 * part + 2; ++j) out[k * kNTanIntr + j] = t.dc[k][j];
}

cudaError_t launch_ref_phase_tangents(const double* theta_ref_dev, double* out, cudaStream_t s) {
  k_ref_phase_tangents<<<1, 32, 0, s>>>(theta_ref_dev, out);
  return cudaGetLastError();
}

cudaError_t launch_ref_dd(const double* theta_ref_dev, const EventConst& ec, RefValues* out, SummarySync* base_reset,
                          cudaStream_t s) {
  k_ref_dd<<<1, kDdRoleThreads, 0, s>>>(theta_ref_dev, ec, out, base_reset);
  return cudaGetLastError();
}

cudaError_t launch_setup(int mode, const double* theta, int64_t W, const EventConst& ec, const RefValues* ref,
                         void* ws, void* tan, bool grad, cudaStream_t s) {
  if (mode == RB_MIXED) {
    const unsigned grid = (unsigned)((W + kSetupWalkers - 1) / kSetupWalkers);
    // the denser form where it takes fewer waves: 12000 walkers are 375 blocks, two
    // waves of 304 or one of 456 (152 SMs); call with 1 detector, 100 bins 38.4 -> 34.1 us, with 3
    // detectors, 500 bins 85.4 -> 80.6; at 16384, two waves in either form, it loses 2.7
    const unsigned n_sm = (unsigned)sm_count(), sparse = (grid + 2 * n_sm - 1) / (2 * n_sm), dense = (grid + 3 * n_sm - 1) / (3 * n_sm);
    if (grad && dense < sparse)
      k_setup_dd_dense<<<grid, kDdRoleThreads + kTanWarps * 32, 0, s>>>(theta, W, ec, ref, ws, tan);
    else if (grad)
      k_setup_dd<true><<<grid, kDdRoleThreads + kTanWarps * 32, 0, s>>>(theta, W, ec, ref, ws, tan);
    else
      k_setup_dd<false><<<grid, kDdRoleThreads, 0, s>>>(theta, W, ec, ref, ws, tan);
    return cudaGetLastError();
  }
  if (mode == RB_FP64) return launch_setup_t<RB_FP64>(theta, W, ec, ref, ws, tan, grad, s);
  return launch_setup_t<RB_MIXED_F64PHASE>(theta, W, ec, ref, ws, tan, grad, s);
}

}  // namespace rb
