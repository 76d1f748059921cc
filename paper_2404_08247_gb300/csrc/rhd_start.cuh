// rhd_start.cuh -- start of the implicit solve (Sec. 3.3): the outer iteration
// run to near convergence on pairs of floats.
#pragma once

#include <math.h>

#include "rhd_pair.cuh"

namespace rhd {

// A positive constant as a pair times a power of two.
struct PairScaled {
  Pair m;  // hi in [1, 2]
  int e;
};

// Constants of pair_start (fill_start); ok: every one is representable.
struct StartConsts {
  PairScaled inv_chat, chat, inv_c, chat_over_c, c_over_chat, c2, inv_c2;
  PairScaled q4;  // (c a/chat)^(1/4) (gamma - 1)/(kB/mu)
  // the solve's tolerances
  float newton_rtol, outer_rtol;
  int ok;
};

// emax: with it and the bound of 700 on E_tot's exponent the exponents that
// pair_start scales by stay within split_scaled's and widened's ranges (the host
// checks once what a test a cell would cost the mixed box 1.7 % for)
constexpr int kUnitMax = 190;  // of chat and c/chat; 400 of the others
inline PairScaled pair_scaled(double x, int& ok, int emax = 400) {
  PairScaled p = {{0.f, 0.f}, 0};
  if (!(x > 0.0) || !isfinite(x)) {
    ok = 0;
    return p;
  }
  const double m = 2.0 * frexp(x, &p.e);
  p.e -= 1;
  p.m.hi = (float)m;
  p.m.lo = (float)(m - (double)p.m.hi);
  if (p.e < -emax || p.e > emax) ok = 0;
  return p;
}

inline void fill_start(StartConsts& K, double c, double chat, double a_rad, double cv_spec,
                       double newton_rtol, double outer_rtol) {
  K.ok = 1;
  K.newton_rtol = (float)fmin(newton_rtol, 1e30);
  K.outer_rtol = (float)fmin(outer_rtol, 1e30);
  if (!(newton_rtol >= 5e-14 && outer_rtol >= 5e-14)) K.ok = 0;  // below the pairs' reach
  K.inv_chat = pair_scaled(1.0 / chat, K.ok, kUnitMax);
  K.chat = pair_scaled(chat, K.ok, kUnitMax);
  K.inv_c = pair_scaled(1.0 / c, K.ok);
  K.chat_over_c = pair_scaled(chat / c, K.ok, kUnitMax);
  K.c_over_chat = pair_scaled(c / chat, K.ok, kUnitMax);
  K.c2 = pair_scaled(c * c, K.ok);
  K.inv_c2 = pair_scaled(1.0 / (c * c), K.ok);
  K.q4 = pair_scaled(sqrt(sqrt(c / chat * a_rad)) / cv_spec, K.ok);
}

// m 2^e as a float power of two factor; false outside the normal range
__device__ __forceinline__ bool pow2f(int e, float& f) {
  if (e < -100 || e > 100) return false;
  f = __uint_as_float((unsigned)(e + 127) << 23);
  return true;
}

// Where a tested number is within kBlur of the terms it sums of its threshold,
// single precision cannot decide the test (it is good to about 1e-6 of the
// terms) and the cell is left to the cold start, so that every cell stops
// where the double-precision iteration stops (1e-4 of the cells).
constexpr float kBlur = 2e-5f;

// What pair_start found, for local_solve to settle in double.
struct WarmStart {
  double R, F[3];
  double lag;  // the residual the iteration leaves in the R-row
};

// One cell's data of pair_start, in its units
struct StartCell {
  Pair eg, er, k, hk, km, q4;
  Pair f0[3], b0[3];
};

// (the products' errors and the cross terms summed in single precision, one
// renormalisation: 29 instructions for 43)
__device__ __forceinline__ Pair dot3(const Pair a[3], const Pair b[3]) {
  const float p0 = __fmul_rn(a[0].hi, b[0].hi), p1 = __fmul_rn(a[1].hi, b[1].hi);
  const float p2 = __fmul_rn(a[2].hi, b[2].hi);
  const float s = __fadd_rn(p0, p1), t = __fadd_rn(s, -p0);
  float e = __fadd_rn(__fadd_rn(p0, -__fadd_rn(s, -t)), __fadd_rn(p1, -t));
  const float r = __fadd_rn(s, p2), q = __fadd_rn(r, -s);
  e = __fadd_rn(e, __fadd_rn(__fadd_rn(s, -__fadd_rn(r, -q)), __fadd_rn(p2, -q)));
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const float p = i == 0 ? p0 : i == 1 ? p1 : p2;
    e = __fadd_rn(e, __fmaf_rn(a[i].lo, b[i].hi, __fmaf_rn(a[i].hi, b[i].lo,
                                                          __fmaf_rn(a[i].hi, b[i].hi, -p))));
  }
  return pair_norm(r, e);
}

// f and b of the next outer pass from the inner stage's x4 = a T^4 and e and
// the frozen f, b, which they replace.  The flux is f(t) + df, df = [k (x^4 b +
// b.P) - k g f(t)]/(1 + k g), whose rounding in a thin cell (k << 1) is that
// of df; df is returned to single precision.  (512 batched problems: 0.02 % of
// the late cells' starts are undecided and take the double-precision iteration,
// 2.9 % with f recomputed from its sum; 245.7 -> 239.5 ms, a 256-cell row
// 3.57 -> 3.25.)
__device__ __forceinline__ void flux_pass(const StartCell& C, bool m1, Pair x4, Pair e, Pair kg,
                                          Pair f[3], Pair b[3], float df[3]) {
  const Pair third = {0x1.555556p-2f, -0x1.555556p-27f};
  Pair ha = e * third, hb = pair_of(0.f);
  if (m1) {
    const Pair f2 = dot3(f, f), e2 = e * e;
    if (e2.hi < f2.hi) {
      ha = pair_of(0.f);
      hb = e * recip(f2);
    } else {
      const Pair s = root(scaled(e2, 4.f) - f2 * 3.f);
      ha = (s - e) * third;
      hb = recip(scaled(e, 2.f) + s) * 3.f;
    }
  }
  const Pair t = hb * dot3(b, f), u = x4 + ha, ig = recip(kg + 1.f);
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const Pair d = (C.k * (u * b[i] + t * f[i]) - kg * C.f0[i]) * ig;
    f[i] = C.f0[i] + d;
    b[i] = C.b0[i] - d * C.km;
    df[i] = d.hi;
  }
}

// Single-precision values of one outer pass, kept to form the next pass'
// changes as differences (each to single precision of itself).
struct PassValues {
  float x, x4, e, f2, s, hb, u, t, bf;
  bool over;  // above the free-streaming limit
};

__device__ __forceinline__ float fdot3(const float a[3], const float b[3]) {
  return fmaf(a[2], b[2], fmaf(a[1], b[1], __fmul_rn(a[0], b[0])));
}

__device__ __forceinline__ PassValues pass_values(bool m1, float x, float e, const float f[3],
                                                  const float b[3]) {
  PassValues p;
  p.x = x;
  p.e = e;
  const float x2 = __fmul_rn(x, x);
  p.x4 = __fmul_rn(x2, x2);
  p.f2 = fdot3(f, f);
  p.bf = fdot3(b, f);
  p.over = m1 && __fmul_rn(e, e) < p.f2;
  p.s = p.over ? 0.f : sqrtf(fmaf(-3.f, p.f2, __fmul_rn(4.f * e, e)));
  p.hb = !m1 ? 0.f : p.over ? __fdividef(e, p.f2) : __fdividef(3.f, fmaf(2.f, e, p.s));
  const float ha = !m1 ? __fmul_rn(e, 1.f / 3.f) : p.over ? 0.f : __fmul_rn(p.s - e, 1.f / 3.f);
  p.u = p.x4 + ha;
  p.t = __fmul_rn(p.hb, p.bf);
  return p;
}

// The iteration of Sec. 3.3 as local_solve runs it, on pairs, up to the entry
// of its last pass.  Units: 2^s for energies (2^s <= E_tot < 2^(s+4), s a
// multiple of 4), c for velocities and chat 2^s for fluxes:
//   eg = Egas 2^-s, er = (c/chat) E 2^-s, r = (c/chat) R 2^-s, f = F/chat 2^-s,
//   b = v/c, ek = hk b.b, x = (c a/chat 2^-s)^(1/4) T = q4 (eg - r - ek),
//   0 = phi = k g (x^4 - er - r) + k b.f - r             (inner stage, for r)
//   f <- [f(t) + k (x^4 b + b.P)]/(1 + k g),  b <- b(t) - km (f - f(t))
// with k = chat chi theta dt, g = 1 + b.b/2 (order 2), hk = rho c^2 2^-s/2,
// km = 1/(2 hk).
//
// The passes and Newton updates are those that local_solve would take, with
// its tests and tolerances, and count in no and nn against the same bounds.
// The tests compare numbers of 1e-13 of E_tot or Q, next to the pairs'
// rounding, so what they test is tracked in single precision as differences:
//   lag  phi as the accepted Newton updates (what their linearisation drops)
//        and the changes of (b, f) since have left it,
//   df   a pass' change of f as the finite difference of the pass' formula
//        from the change before it (df_i = [k (du b + u db + dt f + t df) -
//        d(kg) f]/(1 + k g)), from which the change of Q follows.
// Once df is below 1e-7 of f it also updates f (its error, below 1e-13 of f,
// shrinks in the last pass); until then a pass runs on pairs.
// What it is for: the FP64 pipe bounds the stage kernels, and the iteration put
// 4.4 passes and 7 updates a cell through it; one pass is left.  Two steps of a
// 256^3 box: 191 -> 112 ms, mixed 250 x 200 x 130, four steps, 104 -> 46 ms.
// W: R and F at the entry of the last pass (the one that passes the outer
// test), where local_solve repeats it in double, and the lag.
// False (the caller starts from the explicit state) if a quantity leaves the
// float range, a bound is reached or a value is not positive.
__device__ __forceinline__ bool pair_start(const StartConsts& K, bool m1, bool order2, double rho,
                                           double k0, double Etot, const double y[8],
                                           const double v0[3], int newton_max, int outer_max,
                                           WarmStart& W, int& nn, int& no) {
  const int se = (int)((__double_as_longlong(Etot) >> 52) & 0x7ff) - 1023;
  const int s = (se >> 2) * 4;
  const int sr = (int)((__double_as_longlong(rho) >> 52) & 0x7ff) - 1023;
  if (se < -700 || se > 700 || sr < -200 || sr > 200) return false;
  StartCell C;
  bool ok = split_scaled(y[0], s, C.eg);
  ok &= split_scaled(y[4], s - K.c_over_chat.e, C.er);
  ok &= split_scaled(k0, 0, C.k);
  Pair rm;
  ok &= split_scaled(rho, sr, rm);
  float p2;
  C.er = C.er * K.c_over_chat.m;
  C.hk = rm * K.c2.m;
  ok &= pow2f(sr + K.c2.e - s - 1, p2);
  C.hk = scaled(C.hk, p2);
  const Pair ir = recip(rm);
  ok &= pow2f(K.inv_c2.e - sr + s, p2);
  C.km = scaled(ir * K.inv_c2.m, p2);
  ok &= pow2f(K.q4.e - sr + 3 * (s / 4), p2);
  C.q4 = scaled(ir * K.q4.m, p2);
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    Pair t;
    ok &= split_scaled(y[5 + i], s - K.inv_chat.e, t);
    C.f0[i] = t * K.inv_chat.m;
    ok &= split_scaled(v0[i], -K.inv_c.e, t);
    C.b0[i] = t * K.inv_c.m;
  }
  if (!ok) return false;

  Pair f[3], b[3], r;
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    f[i] = C.f0[i];
    b[i] = C.b0[i];
  }
  {
    // start of the inner stage: k g x^4 + (1 + k g) x/q4 = C in single
    // precision, by Newton from the upper bound (monotone: the quartic is
    // convex)
    const Pair bb = dot3(b, b), ei = C.eg - C.hk * bb;
    const float bf = dot3(b, f).hi;
    const float kg = order2 ? fmaf(0.5f * C.k.hi, bb.hi, C.k.hi) : C.k.hi;
    const float be = __fmul_rn(1.f + kg, __fdividef(1.f, C.q4.hi));
    const float Ct = fmaf(kg, C.er.hi, fmaf(-C.k.hi, bf, __fmul_rn(1.f + kg, ei.hi)));
    if (!(Ct > 0.f)) return false;
    const float z = __fdividef(Ct, kg);
    float x = fminf(__fdividef(Ct, be), sqrtf(sqrtf(z)));
#pragma unroll 1
    for (int i = 0; i < 6; ++i) {
      const float x3 = __fmul_rn(__fmul_rn(kg, x), __fmul_rn(x, x));
      x -= __fdividef(fmaf(x3, x, fmaf(be, x, -Ct)), fmaf(4.f, x3, be));
    }
    // r from the energies, or from the R-row where that is less sensitive to x
    const float x3 = __fmul_rn(x, __fmul_rn(x, x));
    if (__fmul_rn(__fmul_rn(4.f * kg, x3), C.q4.hi) < 1.f + kg)
      r = pair_of(__fdividef(fmaf(kg, fmaf(x3, x, -C.er.hi), __fmul_rn(C.k.hi, bf)), 1.f + kg));
    else
      r = ei - recip(C.q4) * pair_of(x);
  }
  const float tolr = __fmul_rn(K.newton_rtol, C.eg.hi + C.er.hi);  // times k g
  const float hs = order2 ? 0.5f : 0.f;
  float df[3], db[3], dbb = 0.f, dbf = 0.f, lag = 0.f;
  PassValues P;
  for (bool first = true;;) {
    // inner stage
    float kgf = order2 ? fmaf(0.5f * C.k.hi, dot3(b, b).hi, C.k.hi) : C.k.hi;
    const float tol = __fmul_rn(tolr, kgf);
    float dr = 0.f;
    int it = 0;
    while (first && it == 0 || fabsf(lag) > tol) {
      const Pair bb = dot3(b, b), x = C.q4 * (C.eg - C.hk * bb - r), x2 = x * x;
      const Pair kg = order2 ? C.k + C.k * scaled(bb, 0.5f) : C.k;
      const Pair phi = kg * (x2 * x2 - C.er) + C.k * dot3(b, f) - (kg + 1.f) * r;
      if (!(x.hi > 0.f) || !(fabsf(phi.hi) < 1e30f)) return false;
      if (first && it == 0 && fabsf(phi.hi) <= 1.4f * tol) {
        if (fabsf(phi.hi) > 0.7f * tol) return false;
        lag = phi.hi;
        break;
      }
      if (it >= newton_max) return false;
      ++it;
      const float j = __fmul_rn(4.f * kg.hi, C.q4.hi);
      const float d = __fdividef(phi.hi, fmaf(j, __fmul_rn(x.hi, x2.hi), kg.hi + 1.f));
      r = r + d;
      dr += d;
      // phi after an exact Newton update
      const float dx = __fmul_rn(C.q4.hi, d);
      const float c2 = fmaf(dx, fmaf(-4.f, x.hi, dx), 6.f * x2.hi);
      lag = __fmul_rn(__fmul_rn(kg.hi, __fmul_rn(dx, dx)), c2);
      if (fabsf(fabsf(lag) - tol) < __fmul_rn(kBlur, fabsf(lag))) return false;
    }
    nn += it;

    // the pass' changes
    const float ff[3] = {f[0].hi, f[1].hi, f[2].hi}, bh[3] = {b[0].hi, b[1].hi, b[2].hi};
    const Pair bb = dot3(b, b), e = C.er + r;
    const Pair x = C.q4 * (C.eg - C.hk * bb - r);
    if (!(x.hi > 0.f)) return false;
    const PassValues N = pass_values(m1, x.hi, e.hi, ff, bh);
    const Pair kg = order2 ? C.k + C.k * scaled(bb, 0.5f) : C.k, kg1 = kg + 1.f;
    const float ig = __fdividef(1.f, kg1.hi);
    float dn[3], dsum[3], big_df = 0.f, big_f = 0.f;
    Pair fn[3], bn[3];
    if (first) {
      const Pair x2 = x * x;
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        fn[i] = f[i];
        bn[i] = b[i];
      }
      flux_pass(C, m1, x2 * x2, e, kg, fn, bn, dn);
#pragma unroll
      for (int i = 0; i < 3; ++i) dsum[i] = fabsf(dn[i]);
    } else {
      const float dxx = __fmul_rn(-C.q4.hi, fmaf(C.hk.hi, dbb, dr));
      const float dx4 = __fmul_rn(__fmul_rn(dxx, N.x + P.x),
                                  fmaf(N.x, N.x, __fmul_rn(P.x, P.x)));
      float df2 = 0.f;
#pragma unroll
      for (int i = 0; i < 3; ++i) df2 = fmaf(df[i], fmaf(2.f, ff[i], -df[i]), df2);
      float dha = __fmul_rn(dr, 1.f / 3.f), dhb = 0.f;
      if (m1) {
        if (N.over != P.over) {
          dha = (N.u - N.x4) - (P.u - P.x4);
          dhb = N.hb - P.hb;
        } else if (N.over) {
          dha = 0.f;
          dhb = __fdividef(fmaf(-P.hb, df2, dr), N.f2);
        } else {
          const float ds = __fdividef(fmaf(-3.f, df2, __fmul_rn(4.f * dr, N.e + P.e)),
                                      N.s + P.s);
          dha = __fmul_rn(ds - dr, 1.f / 3.f);
          dhb = __fmul_rn(__fmul_rn(N.hb, P.hb), __fmul_rn(fmaf(2.f, dr, ds), -1.f / 3.f));
        }
      }
      const float du = dx4 + dha;
      const float dt = fmaf(dhb, N.bf, __fmul_rn(P.hb, dbf));
      const float dkg = __fmul_rn(__fmul_rn(C.k.hi, hs), dbb);
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        const float q1 = __fmul_rn(du, bh[i]), q2 = __fmul_rn(P.u, db[i]);
        const float q3 = __fmul_rn(dt, ff[i]), q4 = __fmul_rn(P.t, df[i]);
        const float q5 = __fmul_rn(dkg, ff[i]);
        dn[i] = __fmul_rn(ig, fmaf(C.k.hi, (q1 + q2) + (q3 + q4), -q5));
        dsum[i] = __fmul_rn(ig, fmaf(C.k.hi, (fabsf(q1) + fabsf(q2)) + (fabsf(q3) + fabsf(q4)),
                                     fabsf(q5)));
      }
    }
    P = N;
    dbf = dbb = 0.f;
    float Qs = 0.f, bbn = 0.f, blur = 0.f;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      const float d = __fmul_rn(-C.km.hi, dn[i]), fi = ff[i] + dn[i], bi = bh[i] + d;
      dbf = fmaf(d, fi, fmaf(bh[i], dn[i], dbf));
      dbb = fmaf(d, bh[i] + bi, dbb);
      bbn = fmaf(bi, bi, bbn);
      blur = fmaf(fabsf(d), fabsf(fi), fmaf(fabsf(bh[i]), dsum[i], blur));
      Qs = fmaf(fabsf(bi), fabsf(fi), Qs);
      big_df = fmaxf(big_df, fabsf(dn[i]));
      big_f = fmaxf(big_f, fabsf(fi));
      df[i] = dn[i];
      db[i] = d;
    }
    const float xe = N.x4 - N.e, dh = __fmul_rn(hs, dbb), dQ = fabsf(fmaf(dh, xe, dbf));
    const float Q = fabsf(fmaf(__fmul_rn(hs, bb.hi), xe, N.bf));
    const float big = fmaxf(fmaxf(Q, fabsf(__fdividef(r.hi, C.k.hi))),
                            fmaf(__fmul_rn(hs, bbn), fabsf(xe), Qs));
    const float tolQ = __fmul_rn(K.outer_rtol, big);
    blur = fmaf(fabsf(dh), fabsf(xe), blur);
    // (the first pass' change comes from pairs, good to 2^-46 of k g f/(1 + k g))
    const float rest = first ? __fmul_rn(__fmul_rn(4e-14f, Qs), __fmul_rn(kg.hi, ig)) : 0.f;
    if (fabsf(dQ - tolQ) < fmaf(kBlur, blur, rest)) return false;
    if (dQ <= tolQ) break;  // the last pass
    if (!(dQ < 1e30f) || ++no >= outer_max) return false;
    const bool small = !first && big_df <= __fmul_rn(1e-7f, big_f);
    if (!first && !small) {
      const Pair x2 = x * x;
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        fn[i] = f[i];
        bn[i] = b[i];
      }
      float unused[3];
      flux_pass(C, m1, x2 * x2, e, kg, fn, bn, unused);
    }
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      f[i] = small ? f[i] + df[i] : fn[i];
      b[i] = small ? b[i] + db[i] : bn[i];
    }
    first = false;
    // phi at the entry of the next pass
    const float x3 = __fmul_rn(N.x, __fmul_rn(N.x, N.x));
    const float dx = __fmul_rn(__fmul_rn(C.q4.hi, C.hk.hi), dbb);
    const float l1 = __fmul_rn(-4.f * kg.hi, __fmul_rn(x3, dx));
    blur = fmaf(C.k.hi, blur, fabsf(lag) + fabsf(l1));
    lag = fmaf(C.k.hi, fmaf(dh, xe, dbf), l1 + lag);
    if (fabsf(fabsf(lag) - tol) < __fmul_rn(kBlur, blur)) return false;
  }
  W.R = widened(r * K.chat_over_c.m, s + K.chat_over_c.e);
  W.lag = widened(__fmul_rn(lag, K.chat_over_c.m.hi), s + K.chat_over_c.e);
#pragma unroll
  for (int i = 0; i < 3; ++i) W.F[i] = widened(f[i] * K.chat.m, s + K.chat.e);
  return true;
}

}  // namespace rhd
