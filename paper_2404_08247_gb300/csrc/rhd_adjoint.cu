// rhd_adjoint.cu -- reverse-mode derivative of the IMEX PD-ARS step.
//
// One step (Sec. 3.2, eq. imex1/imex2, epsilon = 0) written with the stage-2
// explicit state y2 = (y(n) + yh)/2 + (dt/2) s(yh), which equals eq. (imex2)'s
// explicit part because dt f(yh) = yh - y*:
//   y*  = y(n) + dt s(y(n)),  yh = LS_1(y*),  y2 = ...,  y1 = LS_(1/2)(y2).
// Given ybar1 = dL/dy1 the adjoint is
//   q    = LS_(1/2)^T ybar1                                  (kernel A)
//   gh   = q/2 + (dt/2) s'(yh)^T q                           (faces B, cell C)
//   q'   = LS_1^T gh,   ybar(n) = q/2 + q' + dt s'(y(n))^T q'  (cell C, faces D, gather)
// LS^T is the implicit-function theorem on the converged local solve
// (Sec. 3.3, eq. egupdate-fupdate): with x = (Egas, E, F) and the momentum
// eliminated by m = p - F/(c chat), p = m(t) + F(t)/(c chat), the solution
// satisfies r(x; Egas(t), E(t), F(t), p, chi) = 0 with
//   r_G = Egas - Egas(t) + (c/chat) R,  r_E = E - E(t) - R,
//   r_F = F (1 + k g) - F(t) - k (a T^4 v + v.P),  R = k [(a T^4 - E) g + v.F/c^2],
// k = chat chi theta dt, so (dr/dx)^T lambda = xbar gives every input cotangent.
// s'^T is the transpose of the PLM/HLL transport (Sec. 3.3 Godunov step, Sec.
// 4.3 speeds and optical-depth factor) on the active branch of every limiter,
// max and clip.  It is done per face: kernel B/D differentiates each face flux
// once and writes its 16 stencil partials (and the two opacity partials of its
// optical-depth factor) to scratch; the next per-cell kernel gathers the four
// faces per axis that touch its cell.  No atomics: every sum has a fixed order.
#include "rhd_adjoint.cuh"

namespace rhd {

// ------------------------------------------------------------ face partials

// Face grid of axis d: n[d] faces per line (periodic; face n == face 0) or
// n[d] + 1 (reflecting; faces 0..n, face 0 and face n on the walls).  Face f
// lies between cells f-1 and f of its line.
__host__ __device__ inline int faces_along(const Geometry& g, int d) {
  return g.n[d] + (g.bc[d][0] != RHD_BC_PERIODIC ? 1 : 0);
}

__host__ __device__ inline long long face_count(const Geometry& g, int d) {
  return (long long)g.ncell / g.n[d] * faces_along(g, d);
}

__device__ __forceinline__ long long face_index(const Geometry& g, int d, int x, int y, int z) {
  int n0 = d == 0 ? faces_along(g, 0) : g.n[0];
  int n1 = d == 1 ? faces_along(g, 1) : g.n[1];
  return x + (long long)n0 * (y + (long long)n1 * z);
}

// Half PLM slope (monotonised-central limiter) and the candidate it selects:
// 0 none (extremum), 1 u_0 - u_-, 2 u_+ - u_0, 3 (u_+ - u_-)/4.  Signs and the
// minimum are taken on the integer pipe, as in the forward half_slope.
__device__ __forceinline__ double half_slope_branch(double um, double u0, double up, int& br) {
  double dm = u0 - um, dp = up - u0;
  long long bm = dbits(dm), bp = dbits(dp);
  long long am = bm & kMag, ap = bp & kMag, aq = quarter_mag(abs_bits(dm + dp));
  br = 0;
  if (!(((bm ^ bp) >= 0) & (am != 0) & (ap != 0))) return 0.0;
  long long m = min(min(am, ap), aq);
  br = m == am ? 1 : m == ap ? 2 : 3;
  return __longlong_as_double(m | (bm & ~kMag));
}

// Reverse of it: the slope's cotangent s onto (u_-, u_0, u_+), whose partials
// are 0, +-1 or +-1/4 by the branch, so that nothing is multiplied.
__device__ __forceinline__ void half_slope_vjp(int br, double s, double& gm, double& g0,
                                               double& gp) {
  const double q = 0.25 * s;
  gm = br == 1 ? -s : br == 3 ? -q : 0.0;
  g0 = br == 1 ? s : br == 2 ? -s : 0.0;
  gp = br == 2 ? s : br == 3 ? q : 0.0;
}

// One face state after the free-streaming rescale, with the closure
// coefficients P = ha I + hb Ft Ft^T and their partials in (E, |Ft|^2).
struct FaceState {
  double E, F[3];
  double Fin[3], n2;  // the reconstructed flux before the rescale
  bool resc;
  double ha, hb, ha_E, ha_F2, hb_E, hb_F2;
  double P[3];  // row d of P
};

// (with h = s/2 = sqrt(E^2 - 3/4 |Ft|^2) as in the forward face_side; a flux
// scaled back has |Ft| = E)
__device__ __forceinline__ void face_state(int d, int closure, double E, const double Fin[3],
                                           FaceState& s) {
  s.E = E;
  s.n2 = dot3(Fin, Fin);
  const double E2 = E * E;
  s.resc = lt_nn(E2, s.n2);
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    s.Fin[j] = Fin[j];
    s.F[j] = Fin[j];
  }
  double F2 = s.n2;
  if (s.resc) {
    const double sc = E * rsqrt_pos(s.n2);
#pragma unroll
    for (int j = 0; j < 3; ++j) s.F[j] = Fin[j] * sc;
    F2 = E2;
  }
  if (closure == RHD_CLOSURE_EDDINGTON) {
    s.ha = E * (1.0 / 3.0);
    s.hb = 0.0;
    s.ha_E = 1.0 / 3.0;
    s.ha_F2 = s.hb_E = s.hb_F2 = 0.0;
  } else {
    // ha = (2h - E)/3, hb = 3/2/(E + h)
    const double x = fma(-0.75, F2, E2);
    const double ih = rsqrt_pos(x), h = x * ih;
    const double w = rcp_pos(E + h), hb2 = 0.75 * w * w;
    const double h2E = 2.0 * E * ih;  // d(2h)/dE
    s.ha = fma(2.0, h, -E) * (1.0 / 3.0);
    s.hb = 1.5 * w;
    s.ha_E = (h2E - 1.0) * (1.0 / 3.0);
    s.ha_F2 = -0.25 * ih;
    s.hb_E = -hb2 * (2.0 + h2E);
    s.hb_F2 = hb2 * 0.75 * ih;
  }
  double t = s.hb * s.F[d];
#pragma unroll
  for (int j = 0; j < 3; ++j) s.P[j] = t * s.F[j];
  s.P[d] += s.ha;
}

// Reverse of face_state: (gE, gF) hold the cotangents of E and of the rescaled
// Ft on entry (gP that of row d of P); on exit (gE, gF) are those of E and of
// the reconstructed Ft.
__device__ __forceinline__ void face_state_vjp(int d, const FaceState& s, const double gP[3],
                                               double& gE, double gF[3]) {
  double gPF = gP[0] * s.F[0] + gP[1] * s.F[1] + gP[2] * s.F[2];
  double gha = gP[d];
  double ghb = s.F[d] * gPF;
#pragma unroll
  for (int j = 0; j < 3; ++j) gF[j] += s.hb * s.F[d] * gP[j];
  gF[d] += s.hb * gPF;
  gE += gha * s.ha_E + ghb * s.hb_E;
  double gF2 = 2.0 * (gha * s.ha_F2 + ghb * s.hb_F2);
#pragma unroll
  for (int j = 0; j < 3; ++j) gF[j] += gF2 * s.F[j];
  if (s.resc) {
    // F = Fin E / |Fin|
    double in = rsqrt_pos(s.n2);
    double fg = s.Fin[0] * gF[0] + s.Fin[1] * gF[1] + s.Fin[2] * gF[2];
    gE += fg * in;
    double a = s.E * in, b = fg * in * in;
#pragma unroll
    for (int j = 0; j < 3; ++j) gF[j] = a * (gF[j] - s.Fin[j] * b);
  }
}

// d/dtau of the optical-depth factor eps = (1 - exp(-tau))/tau: (1 - eps)/tau -
// eps.  Below tau = 0.05 the difference cancels; there its Taylor series
// sum_k (-1)^k k tau^(k-1)/(k+1)! is used through tau^5 (truncation < 1e-14
// relative).
__device__ __forceinline__ double tau_factor_deriv(double tau, double eps) {
  if (tau < 0.05) {
    return -0.5 + tau * (1.0 / 3.0 + tau * (-0.125 + tau * (1.0 / 30.0 +
           tau * (-1.0 / 144.0 + tau * (1.0 / 840.0 - tau * (1.0 / 5760.0))))));
  }
  return fma(1.0 - eps, rcp_pos(tau), -eps);
}

struct FaceArgs {
  Geometry g;
  Physics ph;
  const double* rho;
  const double* kappa;
  const double* y[4];    // state whose transport is differentiated: E, Fx, Fy, Fz
  const double* cot[4];  // cotangent of the stage target: E, Fx, Fy, Fz
  const double* eps[3];  // TAU mode: the forward's factors of the +d faces
  double wE[3], wF[3];   // cotangent weights: chat/2 theta dt/dx_d, times c for F
  double* fp;            // face partials, FP_SLOTS per face, slot-major per axis
  long long off[3];      // start of axis d in fp
  long long nface[3];
  long long total;
};

// The face along axis D (a template parameter, so that every index into the
// per-axis arrays below is a compile-time constant and stays in registers).
template <int D>
__device__ __forceinline__ void face_vjp(const FaceArgs& A, long long fidx) {
  constexpr int d = D;
  const Geometry& g = A.g;
  int nf = faces_along(g, d);
  int fc[3];
  {
    int n0 = d == 0 ? nf : g.n[0];
    int n1 = d == 1 ? nf : g.n[1];
    fc[0] = (int)(fidx % n0);
    long long r = fidx / n0;
    fc[1] = (int)(r % n1);
    fc[2] = (int)(r / n1);
  }
  const int f = fc[d];
  const double inv_c = A.ph.inv_c;
  // stencil cells f-2, f-1 | f, f+1 along d (folded), as (E, Ft)
  double u[4][4];
  int idx[4];
  bool ghost[4];
  const int base = fc[0] * g.stride[0] + fc[1] * g.stride[1] + fc[2] * g.stride[2] -
                   f * g.stride[d];
#pragma unroll
  for (int p = 0; p < 4; ++p) {
    bool flip;
    int x = fold(f + p - 2, g.n[d], g.bc[d][0], g.bc[d][1], flip);
    idx[p] = base + x * g.stride[d];
    ghost[p] = (f + p - 2 < 0 || f + p - 2 >= g.n[d]) && flip;
    u[p][0] = __ldg(A.y[0] + idx[p]);
#pragma unroll
    for (int j = 0; j < 3; ++j) u[p][1 + j] = __ldg(A.y[1 + j] + idx[p]) * inv_c;
    if (flip) u[p][1 + d] = -u[p][1 + d];
  }
  // face cotangent (of the flux in units of chat/2): the face flux enters the
  // update of b with the weight and that of a with its negative; ghost cells
  // carry no update
  double ob[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    double ub = ghost[2] ? 0.0 : __ldg(A.cot[q] + idx[2]);
    double ua = ghost[1] ? 0.0 : __ldg(A.cot[q] + idx[1]);
    ob[q] = (ub - ua) * (q == 0 ? A.wE[d] : A.wF[d]);
  }
  // ---- forward: reconstruction, closure, speeds ----
  double L[4], R[4];
  int bl[4], br[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    L[q] = u[1][q] + half_slope_branch(u[0][q], u[1][q], u[2][q], bl[q]);
    R[q] = u[2][q] - half_slope_branch(u[1][q], u[2][q], u[3][q], br[q]);
  }
  FaceState sl, sr;
  face_state(d, A.ph.closure, L[0], &L[1], sl);
  face_state(d, A.ph.closure, R[0], &R[1], sr);
  double num = sl.P[d], den = sl.E;
  int side = 0;
  if (lt_nn(sl.P[d] * sr.E, sr.P[d] * sl.E)) {
    num = sr.P[d];
    den = sr.E;
    side = 1;
  }
  if (lt_nn(3.0 * num, den)) {
    num = 1.0;
    den = 3.0;
    side = -1;
  }
  // S/chat = sqrt(num/den) = num/sqrt(num den)
  const double rq = rsqrt_pos(num * den);
  const double S = num * rq;
  double eps = 1.0, tau = 0.0;
  const bool tau_mode = A.ph.hll_mode == RHD_HLL_TAU;
  if (tau_mode) {
    tau = 0.5 * (__ldg(A.kappa + idx[1]) * __ldg(A.rho + idx[1]) +
                 __ldg(A.kappa + idx[2]) * __ldg(A.rho + idx[2])) * g.dx[d];
    eps = ghost[1] ? tau_factor(tau) : __ldg(A.eps[d] + idx[1]);
  }
  // ---- reverse: HLL ----
  const double dE = sr.E - sl.E;
  double gEL = eps * S * ob[0], gER = -gEL;
  double gFL[3] = {0.0, 0.0, 0.0}, gFR[3] = {0.0, 0.0, 0.0};
  double gPL[3], gPR[3];
  gFL[d] = ob[0];
  gFR[d] = ob[0];
  const double geps = -S * dE * ob[0];
  double gS = -eps * dE * ob[0];
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    gPL[j] = ob[1 + j];
    gPR[j] = ob[1 + j];
    gFR[j] -= S * ob[1 + j];
    gFL[j] += S * ob[1 + j];
    gS -= (sr.F[j] - sl.F[j]) * ob[1 + j];
  }
  if (side >= 0) {
    // dS/dnum = 1/(2 sqrt(num den)), dS/dden = -S^2 of that
    const double gnum = 0.5 * gS * rq, gden = -gnum * S * S;
    if (side == 0) {
      gPL[d] += gnum;
      gEL += gden;
    } else {
      gPR[d] += gnum;
      gER += gden;
    }
  }
  face_state_vjp(d, sl, gPL, gEL, gFL);
  face_state_vjp(d, sr, gPR, gER, gFR);
  // ---- reverse: reconstruction, for E and the physical F (Ft = F/c) ----
  double gq[4][4];
  {
    const double gLq[4] = {gEL, gFL[0] * inv_c, gFL[1] * inv_c, gFL[2] * inv_c};
    const double gRq[4] = {gER, gFR[0] * inv_c, gFR[1] * inv_c, gFR[2] * inv_c};
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      double lm, l0, lp, rm, r0, rp;
      half_slope_vjp(bl[q], gLq[q], lm, l0, lp);
      half_slope_vjp(br[q], -gRq[q], rm, r0, rp);
      gq[0][q] = lm;
      gq[1][q] = (gLq[q] + l0) + rm;
      gq[2][q] = (gRq[q] + r0) + lp;
      gq[3][q] = rp;
    }
  }
  // store, not yet mirrored
  double* out = A.fp + A.off[d] + fidx;
  const long long NF = A.nface[d];
#pragma unroll
  for (int p = 0; p < 4; ++p) {
    out[(4 * p) * NF] = gq[p][0];
#pragma unroll
    for (int j = 0; j < 3; ++j) out[(4 * p + 1 + j) * NF] = gq[p][1 + j];
  }
  double ka = 0.0, kb = 0.0;
  if (tau_mode) {
    // tau = (chi_a + chi_b) dx/2, chi = kappa rho
    double gt = geps * tau_factor_deriv(tau, eps) * 0.5 * g.dx[d];
    ka = gt * __ldg(A.rho + idx[1]);
    kb = gt * __ldg(A.rho + idx[2]);
  }
  out[16 * NF] = ka;
  out[17 * NF] = kb;
}

__global__ void __launch_bounds__(256) face_vjp_kernel(const FaceArgs A) {
  long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= A.total) return;
  int d = 0;
  while (d + 1 < A.g.ndim && t >= A.off[d + 1] / FP_SLOTS) ++d;
  long long fidx = t - A.off[d] / FP_SLOTS;
  if (d == 0) face_vjp<0>(A, fidx);
  else if (d == 1) face_vjp<1>(A, fidx);
  else face_vjp<2>(A, fidx);
}

// Sum of the face partials of axis d that belong to cell (c), with the mirror
// images of reflecting walls folded back: acc (E, Fx, Fy, Fz) and kacc.
__device__ __forceinline__ void gather_axis(const Geometry& g, const double* fp,
                                            const long long off[3], const long long nface[3],
                                            int d, const int c[3], double acc[4],
                                            double& kacc) {
  const int n = g.n[d];
  const bool refl = g.bc[d][0] != RHD_BC_PERIODIC;
  const double* F = fp + off[d];
  const long long NF = nface[d];
  int cc[3] = {c[0], c[1], c[2]};
  const int j = c[d];
  auto add = [&](int f, int p, bool flip) {
    cc[d] = f;
    long long fi = face_index(g, d, cc[0], cc[1], cc[2]);
    acc[0] += F[(4 * p) * NF + fi];
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      double v = F[(4 * p + 1 + q) * NF + fi];
      acc[1 + q] += (flip && q == d) ? -v : v;
    }
  };
  auto addk = [&](int f, int slot) {
    cc[d] = f;
    kacc += F[slot * NF + face_index(g, d, cc[0], cc[1], cc[2])];
  };
#pragma unroll
  for (int p = 0; p < 4; ++p) {
    int f = j + 2 - p;  // the face whose stencil position p is this cell
    if (!refl) {
      add((f + n) % n, p, false);
    } else {
      if (f >= 0 && f <= n) add(f, p, false);
      if (j <= 1 && 1 - j - p >= 0) add(1 - j - p, p, true);            // ghost -1-j
      if (j >= n - 2 && 2 * n + 1 - j - p <= n) add(2 * n + 1 - j - p, p, true);  // ghost 2n-1-j
    }
  }
  if (!refl) {
    addk(j, 17);
    addk((j + 1) % n, 16);
  } else {
    addk(j, 17);
    addk(j + 1, 16);
    if (j == 0) addk(0, 16);
    if (j == n - 1) addk(n, 17);
  }
}

// ---------------------------------------------------------- local solve

// Adjoint of one converged local solve with output y (Egas, m, E, F) and
// stage weight theta (tdt = theta dt).  ybar: cotangent of the output; on exit
// yin: cotangent of the input state; chibar: dL/dchi.  Returns false if the
// Jacobian of the converged system is singular.
//
// (dr/dx)^T lambda = xbar is solved by its structure instead of a 5 x 5
// elimination.  The rows r_G + (c/chat) r_E = Egas - Egas(t) + (c/chat)(E -
// E(t)) and r_E leave mu0 and mu1 (lambda_G = mu0, lambda_E = (c/chat) mu0 +
// mu1) explicit in V = v.mu and U = Ft.mu, mu the flux rows' multipliers, whose
// own block is al I plus products of v and Ft:
//   d mu1 = x1 - (c/chat) x0 - (bv - (c/chat) a0) V - bu U,
//   al mu = x - v (vv V + uv U - ev mu1) - Ft (vu V + uu U - eu mu1),
// and its products with v and Ft are a 2 x 2 system for V and U.  The Jacobian's
// determinant is d al det(2 x 2), and d, al > 0 for |v| < c (d = 1 + k g + (c/chat)
// dR/dEgas; hb |Ft| <= 1, so al >= 1 + k (g - |v|/c)), so that the 2 x 2 system is
// singular where the Jacobian is; it is scaled by a power of two near 1/al, or its
// determinant, of order k^2, would overflow from k = 1e154 on.  All parts are
// linear in these coefficients: 200 FP64 operations a cell, where the matrix
// took 450; its m and F cotangents, in 64-bit terms, are the more accurate.
// With the faces' optical-depth factors from the forward's arrays a 512^2
// gradient over 20 steps takes 39.7 ms, before 49.2.
__device__ bool ls_adjoint(const Physics& ph, double tdt, double rho, double chi,
                           const double y[8], const double ybar[8], double yin[8],
                           double& chibar) {
  const double cr = ph.c_over_chat, icc = ph.inv_cchat, ic2 = ph.inv_c2, ic = ph.inv_c;
  const double irho = rcp_pos(rho);
  const double iCv = irho * ph.inv_cv_spec;
  const bool o2 = ph.vc_order == 2;
  const double Eg = y[0], E = y[4];
  double v[3], u[3];  // u: Ft
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    v[i] = y[1 + i] * irho;
    u[i] = y[5 + i] * ic;
  }
  const double svv = dot3(v, v), svu = dot3(v, u), suu = dot3(u, u);
  const double T = (Eg - 0.5 * rho * svv) * iCv;
  const double T3 = T * T * T;
  const double B = ph.a_rad * T3 * T, Bp = 4.0 * ph.a_rad * T3;
  const double g = o2 ? fma(0.5 * ic2, svv, 1.0) : 1.0;
  const double dk = ph.chat * tdt;  // dk/dchi
  const double k = dk * chi;
  // closure coefficients of P = ha I + hb Ft Ft^T and their partials
  double ha, hb, ha_E = 0.0, ha_F2 = 0.0, hb_E = 0.0, hb_F2 = 0.0;
  if (ph.closure == RHD_CLOSURE_EDDINGTON) {
    ha = E * (1.0 / 3.0);
    hb = 0.0;
    ha_E = 1.0 / 3.0;
  } else if (lt_nn(E * E, suu)) {
    const double iF2 = rcp_pos(suu);
    ha = 0.0;
    hb = E * iF2;
    hb_E = iF2;
    hb_F2 = -E * iF2 * iF2;
  } else {
    const double x = fma(-0.75, suu, E * E);
    const double ih = rsqrt_pos(x), h = x * ih;
    const double w = rcp_pos(E + h), hb2 = 0.75 * w * w;
    const double h2E = 2.0 * E * ih;
    ha = fma(2.0, h, -E) * (1.0 / 3.0);
    hb = 1.5 * w;
    ha_E = (h2E - 1.0) * (1.0 / 3.0);
    ha_F2 = -0.25 * ih;
    hb_E = -hb2 * (2.0 + h2E);
    hb_F2 = hb2 * 0.75 * ih;
  }
  // R = k[(B - E) g + v.F/c^2]: dR/dEgas; dR/dm = mv v + mu Ft per unit of m;
  // dR/dF with m = p - F/(c chat) folded in = ev v + eu Ft
  const double kB = k * Bp * iCv, kr = k * irho, kc = k * ic, q = B - E;
  const double R_Eg = g * kB;
  const double mv = o2 ? fma(kr * ic2, q, -R_Eg) : -R_Eg, mu = kr * ic;
  const double ev = fma(-icc, mv, k * ic2), eu = -icc * mu;
  // flux rows: d/dEgas = -kB v, d/dE = bv v + bu Ft, d/dF = al I + vv v v + ..
  const double Bh = B + ha, kg1 = fma(k, g, 1.0), kh = kr * hb;
  const double bv = -k * ha_E, bu = -k * hb_E * svu;
  const double o = o2 ? mu : 0.0;
  const double al = fma(-kc * hb, svu, fma(icc * kr, Bh, kg1));
  const double vv = -icc * kB, vu = -2.0 * kc * ha_F2, uv = -fma(kc, hb, icc * o);
  const double uu = fma(-2.0 * kc * hb_F2, svu, icc * kh);

  const double x0 = ybar[0], x1 = ybar[4];
  double x[3];
#pragma unroll
  for (int j = 0; j < 3; ++j) x[j] = fma(-icc, ybar[1 + j], ybar[5 + j]);
  const double id = rcp_pos(fma(cr, R_Eg, kg1));
  const double m0 = fma(-cr, x0, x1) * id, mV = -fma(cr, kB, bv) * id, mU = -bu * id;
  const double AV = fma(-ev, mV, vv), AU = fma(-ev, mU, uv), A0 = -ev * m0;
  const double BV = fma(-eu, mV, vu), BU = fma(-eu, mU, uu), B0 = -eu * m0;
  const long long ab = dbits(al) & kMag;
  const double sc = __longlong_as_double((2046ll << 52) - (ab & kInfBits));
  const double M11 = fma(svv, AV, fma(svu, BV, al)) * sc, M12 = fma(svv, AU, svu * BU) * sc;
  const double M21 = fma(svu, AV, suu * BV) * sc, M22 = fma(svu, AU, fma(suu, BU, al)) * sc;
  const double r1 = fma(-svv, A0, fma(-svu, B0, dot3(v, x)));
  const double r2 = fma(-svu, A0, fma(-suu, B0, dot3(u, x)));
  const double det = fma(M11, M22, -M12 * M21);
  const long long db = dbits(det) & kMag;
  if (db == 0 || db >= kInfBits || ab == 0 || ab >= kInfBits) return false;
  const double idet = copysign(rcp_pos(fabs(det)), det) * sc;
  const double V = fma(r1, M22, -M12 * r2) * idet, U = fma(M11, r2, -M21 * r1) * idet;
  const double m1 = fma(mV, V, fma(mU, U, m0));
  const double ca = fma(AV, V, fma(AU, U, A0)), cb = fma(BV, V, fma(BU, U, B0));
  const double ial = copysign(rcp_pos(fabs(al)), al);

  yin[0] = fma(R_Eg, m1, fma(kB, V, x0));
  yin[4] = fma(cr, yin[0], m1);
  chibar = dk * (fma(q, g, svu * ic) * m1 - fma(fma(ph.c, g, -hb * svu), U, -Bh * V));
  const double Pv = fma(mv, m1, -fma(o, U, kB * V)), Pu = fma(mu, m1, kh * U), Pm = kr * Bh;
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    const double l = fma(-v[j], ca, fma(-u[j], cb, x[j])) * ial;
    const double pbar = fma(Pv, v[j], fma(Pu, u[j], fma(Pm, l, ybar[1 + j])));
    yin[1 + j] = pbar;
    yin[5 + j] = fma(pbar, icc, l);
  }
  return true;
}

// ------------------------------------------------------------ cell kernels

struct CellArgs {
  Geometry g;
  Physics ph;
  double tdt;              // theta dt of the local solve (mode A, C)
  const double* rho;
  const double* kappa;
  const double* ys[NY];    // converged local-solve output (mode A: y1, C: yh)
  double* ybar[NY];        // the running adjoint dL/dy
  double* q[NY];           // stage cotangent scratch
  const double* fp;        // face partials to gather (null: none)
  long long off[3], nface[3];
  double* kbar;            // dL/dkappa (accumulated)
  DevStatus* st;
  int step;
};

// mode A: ybar += gather(fp); q = LS_(1/2)^T ybar                 (stage 2)
// mode C: gh = q/2 + gather(fp); q' = LS_1^T gh; ybar = q/2 + q'; q = q'  (stage 1)
// mode E: ybar += gather(fp)                                        (last)
template <int MODE>
__global__ void __launch_bounds__(256, 1) cell_adj_kernel(const CellArgs A) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  const Geometry& g = A.g;
  if (i >= g.ncell) return;
  double acc[4] = {0.0, 0.0, 0.0, 0.0}, kacc = 0.0;
  if (A.fp) {
    int c[3];
    c[0] = i % g.n[0];
    int r = i / g.n[0];
    c[1] = r % g.n[1];
    c[2] = r / g.n[1];
    for (int d = 0; d < g.ndim; ++d) gather_axis(g, A.fp, A.off, A.nface, d, c, acc, kacc);
  }
  double kb = kacc;
  if (MODE == 2) {
    A.ybar[Y_ERAD][i] += acc[0];
#pragma unroll
    for (int j = 0; j < 3; ++j) A.ybar[Y_FX + j][i] += acc[1 + j];
    A.kbar[i] += kb;
    return;
  }
  double cot[8];
  if (MODE == 0) {
#pragma unroll
    for (int s = 0; s < 8; ++s) cot[s] = A.ybar[s][i];
  } else {
#pragma unroll
    for (int s = 0; s < 8; ++s) cot[s] = 0.5 * A.q[s][i];
  }
  cot[Y_ERAD] += acc[0];
#pragma unroll
  for (int j = 0; j < 3; ++j) cot[Y_FX + j] += acc[1 + j];
  double y[8], yin[8], chibar = 0.0;
#pragma unroll
  for (int s = 0; s < 8; ++s) y[s] = __ldg(A.ys[s] + i);
  const double rho = __ldg(A.rho + i);
  const double chi = __ldg(A.kappa + i) * rho;
  bool ok = ls_adjoint(A.ph, A.tdt, rho, chi, y, cot, yin, chibar);
  if (!ok) {
    unsigned long long key = ((unsigned long long)i << 8) | (unsigned long long)RHD_ERR_NEWTON;
    unsigned long long old = atomicMin(&A.st->fail_key, key);
    if (key < old) {
      A.st->fail_step = A.step;
      A.st->fail_stage = MODE == 0 ? 2 : 1;
    }
#pragma unroll
    for (int s = 0; s < 8; ++s) yin[s] = 0.0;
    chibar = 0.0;
  }
  // the face terms first, then the solve's: the same order whether or not a
  // checkpoint boundary split the face terms off into the finishing gather
  double kv = A.kbar[i] + kb;
  A.kbar[i] = kv + chibar * rho;
  if (MODE == 0) {
#pragma unroll
    for (int s = 0; s < 8; ++s) A.q[s][i] = yin[s];
  } else {
#pragma unroll
    for (int s = 0; s < 8; ++s) {
      A.ybar[s][i] = 0.5 * A.q[s][i] + yin[s];
      A.q[s][i] = yin[s];
    }
  }
}

// ------------------------------------------------------------ launchers

long long adjoint_scratch_doubles(const Geometry& g) {
  long long s = 0;
  for (int d = 0; d < g.ndim; ++d) s += FP_SLOTS * face_count(g, d);
  return s;
}

static void face_layout(const Geometry& g, long long off[3], long long nface[3]) {
  long long o = 0;
  for (int d = 0; d < 3; ++d) {
    off[d] = o;
    nface[d] = d < g.ndim ? face_count(g, d) : 0;
    o += FP_SLOTS * nface[d];
  }
}

// One adjoint step: ybar holds dL/dy1 (plus, if pending_fp, the face partials
// of the previous adjoint step still to be gathered into it) and is left as
// the partial dL/dy(n) whose transport part is in fp (gathered by the next
// call with pending_fp = true, or by launch_adjoint_finish).
cudaError_t launch_adjoint_step(const AdjointStep& S, cudaStream_t s) {
  const Geometry& g = S.g;
  const int N = g.ncell;
  // one thread a cell or face: blocks of 64 spread a small grid over the SMs
  // (16 SMs' FP64 pipes did the work of a 64^2 grid in blocks of 256), blocks
  // of 256 where there are enough of them
  const int bs = N < 152 * 256 * 2 ? 64 : 256;
  const int nb = (N + bs - 1) / bs;
  CellArgs C;
  C.g = g;
  C.ph = S.ph;
  C.rho = S.rho;
  C.kappa = S.kappa;
  for (int q = 0; q < NY; ++q) {
    C.ybar[q] = S.ybar + (size_t)q * N;
    C.q[q] = S.q + (size_t)q * N;
  }
  face_layout(g, C.off, C.nface);
  C.kbar = S.kbar;
  C.st = S.st;
  C.step = S.step;

  FaceArgs F;
  F.g = g;
  F.ph = S.ph;
  F.rho = S.rho;
  F.kappa = S.kappa;
  F.fp = S.fp;
  face_layout(g, F.off, F.nface);
  F.total = 0;
  for (int d = 0; d < g.ndim; ++d) F.total += F.nface[d];
  const int fb = (int)((F.total + bs - 1) / bs);
  for (int d = 0; d < 3; ++d) F.eps[d] = S.eps[d];

  // A: stage-2 local solve at y1
  C.tdt = 0.5 * S.dt;
  for (int q = 0; q < NY; ++q) C.ys[q] = S.y1 + (size_t)q * N;
  C.fp = S.pending_fp ? S.fp : nullptr;
  cell_adj_kernel<0><<<nb, bs, 0, s>>>(C);
  // B: transport at yh, weight dt/2, cotangent q
  for (int q = 0; q < 4; ++q) {
    F.y[q] = S.yh + (size_t)(Y_ERAD + q) * N;
    F.cot[q] = S.q + (size_t)(Y_ERAD + q) * N;
  }
  flux_weights(g, S.ph, false, 0.5 * S.dt, F.wE, F.wF);
  face_vjp_kernel<<<fb, bs, 0, s>>>(F);
  // C: stage-1 local solve at yh
  C.tdt = S.dt;
  for (int q = 0; q < NY; ++q) C.ys[q] = S.yh + (size_t)q * N;
  C.fp = S.fp;
  cell_adj_kernel<1><<<nb, bs, 0, s>>>(C);
  // D: transport at y(n), weight dt, cotangent q'
  for (int q = 0; q < 4; ++q) F.y[q] = S.yn + (size_t)(Y_ERAD + q) * N;
  flux_weights(g, S.ph, false, S.dt, F.wE, F.wF);
  face_vjp_kernel<<<fb, bs, 0, s>>>(F);
  return cudaGetLastError();
}

cudaError_t launch_adjoint_finish(const AdjointStep& S, cudaStream_t s) {
  const Geometry& g = S.g;
  const int N = g.ncell;
  CellArgs C;
  C.g = g;
  C.ph = S.ph;
  C.tdt = 0.0;
  C.rho = S.rho;
  C.kappa = S.kappa;
  for (int q = 0; q < NY; ++q) {
    C.ys[q] = nullptr;
    C.ybar[q] = S.ybar + (size_t)q * N;
    C.q[q] = S.q + (size_t)q * N;
  }
  C.fp = S.fp;
  face_layout(g, C.off, C.nface);
  C.kbar = S.kbar;
  C.st = S.st;
  C.step = S.step;
  cell_adj_kernel<2><<<(N + 255) / 256, 256, 0, s>>>(C);
  return cudaGetLastError();
}

}  // namespace rhd
