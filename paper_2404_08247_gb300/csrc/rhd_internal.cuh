// rhd_internal.cuh -- device-side building blocks of the IMEX PD-ARS step.
//
// Internal to the library (csrc/*.cu).  Every routine cites the passage of
// He, Wibking & Krumholz (2024) it implements; readings of passages the paper
// leaves open are the library's documented choices (M1 closure, PLM with the
// monotonised-central limiter, symmetric HLL speeds floored at chat/sqrt(3),
// E_tot = Egas + (c/chat) E, energy closure E = E(t) - (chat/c) dEgas).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "rhd.h"
#include "rhd_start.cuh"

namespace rhd {

// evolved-field slots of a state buffer (NY * ncell doubles, slot-major)
enum { Y_EGAS = 0, Y_MX, Y_MY, Y_MZ, Y_ERAD, Y_FX, Y_FY, Y_FZ, NY };

// Device status block: the first failing launch records its step, stage and
// the smallest failing cell; every later kernel of the batch sees the key and
// skips its work, so the last good ping-pong buffer is never overwritten.
struct DevStatus {
  unsigned long long fail_key;  // (cell << 8) | rhd_status, ~0ull if none
  int fail_step;
  int fail_stage;
  int max_newton;
  int max_outer;
  unsigned long long sum_newton;
  unsigned long long n_solves;
  unsigned long long sum_outer;
};

// Index checks of the bounds-checked build (-DRHD_BOUNDS_CHECK).  chk_index
// returns whether 0 <= i < n; an index outside records RHD_ERR_BOUNDS in the
// status block, with the index in place of the cell (its low 56 bits), and
// the caller skips the access (a load gives 0).  Nothing traps: the context
// stays usable and the step reports the status.  The default build compiles
// the plain accesses.
#ifdef RHD_BOUNDS_CHECK
__device__ __forceinline__ bool chk_index(DevStatus* st, long long i, long long n) {
  if (i >= 0 && i < n) return true;
  atomicMin(&st->fail_key, (((unsigned long long)i & 0x00ffffffffffffffull) << 8) | 8ull);
  return false;
}
#define RHD_LDG(st, p, i, n) (chk_index((st), (i), (n)) ? __ldg((p) + (i)) : 0.0)
#define RHD_LD(st, p, i, n) (chk_index((st), (i), (n)) ? (p)[i] : 0.0)
#define RHD_ST(st, p, i, n, v)                  \
  do {                                          \
    if (chk_index((st), (i), (n))) (p)[i] = (v); \
  } while (0)
#else
#define RHD_LDG(st, p, i, n) __ldg((p) + (i))
#define RHD_LD(st, p, i, n) ((p)[i])
#define RHD_ST(st, p, i, n, v) ((p)[i] = (v))
#endif

struct Geometry {
  int ndim;
  int n[3];
  int stride[3];
  int ncell;
  int bc[3][2];
  double dx[3];
  double inv_dx[3];
  double bc_state[3][2][4];  // ghost E, Fx, Fy, Fz of RHD_BC_INFLOW faces
};

struct Physics {
  double c, chat, a_rad;
  double cv_spec;       // kB_over_mu / (gamma - 1): C_v = rho cv_spec
  double inv_c;         // 1/c
  double c_over_chat;   // c/chat
  double chat_over_c;   // chat/c
  double inv_c2;        // 1/c^2
  double inv_cchat;     // 1/(c chat)
  int closure, vc_order, hll_mode;
  double newton_rtol, outer_rtol;
  double outer_settle;  // the outer tolerance and the pairs' rounding (local_solve)
  int newton_max, outer_max;
  int scheme;              // rhd_scheme
  double kappa_T_exp;      // chi = kappa rho (T / T_ref)^kappa_T_exp
  double inv_kappa_T_ref;  // 1 / T_ref
  int kappa_T_int;         // kappa_T_exp where it is a whole number up to 8, else 0
  double kappa_P_ratio;    // chi_0P / chi_0E
  double kappa_F_ratio;    // chi_0F / chi_0E
  int reconstruction;      // rhd_recon
  double inv_cv_spec;      // 1/cv_spec
  StartConsts start;       // constants of pair_start
};

struct StageArgs {
  Geometry g;
  Physics ph;
  double dt;
  int step;            // step index within the batch (for the status block)
  const double* rho;
  const double* kappa;
  const double* yt[NY];  // state whose transport s(.) is taken, one pointer per slot
  const double* yn[NY];  // y(n) (stage 2 only)
  double* yo[NY];        // stage output
  const double* eps[3];  // TAU mode: per-face optical-depth factors, or null
                         // (then computed from kappa and rho on the fly)
  // weights of the face flux differences in the update of E and of the
  // physical F: u theta dt/dx_d, and c times that, with u the unit of the flux
  // (chat/2 in FP64, 1 mixed) and theta dt = 1 for rates (stage 0), dt in stage
  // 1, dt/2 in stage 2 (flux_weights)
  double wE[3], wF[3];
  double* rate[4];       // transport-only launch: dE/dt, dFx/dt, dFy/dt, dFz/dt
  long long cell_base;   // added to cell indices in failure reports (batched pools)
  DevStatus* st;
  // RHD_BC_HALO z faces: the ghost planes the neighbouring slabs supplied,
  // per side [4 fields E, Fx, Fy, Fz][HALO_PLANES planes][n0 n1], planes in
  // z order (low side: z = -3..-1; high side: z = n2..n2+2); and the TAU
  // factors of the low slab face (n0 n1)
  const double* halo[2] = {nullptr, nullptr};
  const double* eps_zlo = nullptr;
  // the cells [lo, hi) of the launch along the slowest axis (z in 3-D, y in 2-D,
  // x in 1-D) and the planes a 3-D block marches through, its last one fewer
  int lo = 0, hi = 0, lz = 1;
};

// The planes [k0, k1) of block b of a 3-D launch over the planes [lo, hi): the
// last block stops at the launch's end.  Launches over parts of one grid run
// side by side (rhd_step_host), and the planes beyond belong to another one,
// whose inputs this one has not waited for.
__host__ __device__ inline void block_planes(int b, int lo, int hi, int lz, int& k0, int& k1) {
  k0 = lo + b * lz;
  k1 = k0 + lz < hi ? k0 + lz : hi;
}

// ghost planes a HALO face holds (the widest face stencil: PPM's 3)
constexpr int HALO_PLANES = 3;

inline void flux_weights(const Geometry& g, const Physics& ph, bool mixed, double tdt,
                         double wE[3], double wF[3]) {
  for (int d = 0; d < 3; ++d) {
    wE[d] = (mixed ? 1.0 : 0.5 * ph.chat) * g.inv_dx[d] * tdt;
    wF[d] = ph.c * wE[d];
  }
}

// slot pointers of a slot-major buffer of NY * n doubles
template <typename P>
inline void slots_of(P* out, P base, int n) {
  for (int q = 0; q < NY; ++q) out[q] = base + (size_t)q * n;
}

// ------------------------------------------------- FP64 off the FP64 pipe
// On this GPU the FP64 pipe, which limits the FP64 step, also executes double
// compares, minima and conversions (about one FMA slot each), and division
// and square root take about ten.  The helpers below give the same answers
// with the integer pipe doing what it can:
//  * non-negative, non-NaN doubles order like their IEEE bit patterns as
//    signed 64-bit integers, so their compares and minima are integer ops;
//  * rcp_pos / rsqrt_pos / sqrt_pos: 1/x, 1/sqrt(x) and sqrt(x) for x > 0 by
//    one Newton step (r + r (1 - x r); y + y (1 - x y^2)/2; t + (x - t^2) y/2
//    with t = x y) from a seed of 2^-44.  The seed is a single-precision one
//    corrected in single precision by the binomial series of its residual,
//    formed from the 24 leading bits and the rest of x; its bits are put
//    together by integer operations.  2, 3 and 3 FP64 operations, where the
//    series from the bare seed (2^-21) takes 3, 5 and 5 and two Newton steps 4,
//    7 and 8; within 1 ulp.  Two steps of a 256^3 box 91.8 -> 87.8 ms, a 512^2
//    gradient 38.5 -> 36.6, with PPM 17.7 -> 17.4.  Near the ends of the double
//    range (2^-1019, 2^1017) IEEE operations are used, 1/sqrt in two roundings.
constexpr long long kMag = 0x7fffffffffffffffll;
constexpr long long kInfBits = 0x7ff0000000000000ll;

__device__ __forceinline__ long long dbits(double x) { return __double_as_longlong(x); }
// x > 0 and finite (false for NaN)
__device__ __forceinline__ bool pos_finite(double x) {
  long long b = dbits(x);
  return b > 0 && b < kInfBits;
}
__device__ __forceinline__ bool finite_bits(double x) { return (dbits(x) & kMag) < kInfBits; }
// |x|, and a < b / a <= b / max(a, b) for a, b >= 0 (not NaN)
__device__ __forceinline__ long long abs_bits(double x) { return dbits(x) & kMag; }
__device__ __forceinline__ bool lt_nn(double a, double b) { return dbits(a) < dbits(b); }
__device__ __forceinline__ bool le_nn(double a, double b) { return dbits(a) <= dbits(b); }
__device__ __forceinline__ double max_nn(double a, double b) {
  return __longlong_as_double(max(dbits(a), dbits(b)));
}

__device__ __forceinline__ bool seed_range(double x) {
  int e = (int)(dbits(x) >> 52);  // biased exponent of x > 0
  return e > 1023 - 120 && e < 1023 + 120;
}
// x as a float with the mantissa truncated (x > 0 within seed_range)
__device__ __forceinline__ float seed_float(double x) {
  return __int_as_float((int)((dbits(x) >> 29) - (896ll << 23)));
}
// a positive normal float widened exactly
__device__ __forceinline__ double seed_double(float f) {
  return __longlong_as_double(((long long)__float_as_int(f) + (896ll << 23)) << 29);
}
// One rounding each, never contracted with a neighbour: a cell's solve gives the
// same bits in every kernel that runs it.
__device__ __forceinline__ double mul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ double add(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ double sub(double a, double b) { return __dadd_rn(a, -b); }
__device__ __forceinline__ double dot3(const double a[3], const double b[3]) {
  return fma(a[2], b[2], fma(a[1], b[1], mul(a[0], b[0])));
}

// The magnitude bits of x/2 and x/4, rounded as the products by 1/2 and 1/4 are:
// the exponent field lowered on the integer pipe, or, where the result is below
// the normal range, the bits shifted.  (A product for that range would issue,
// predicated off, with every use: 32 slots of the FP64 pipe a cell.)
__host__ __device__ __forceinline__ long long half_mag(long long a) {
  if (a >= kInfBits) return a;
  if (a >= (2ll << 52)) return a - (1ll << 52);
  return (a >> 1) + (a & (a >> 1) & 1);  // a units of 2^-1074: half of them, to even
}
__host__ __device__ __forceinline__ long long quarter_mag(long long a) {
  if (a >= kInfBits) return a;
  if (a >= (3ll << 52)) return a - (2ll << 52);
  if (a >= (2ll << 52)) return half_mag(a - (1ll << 52));  // twice that many units
  return (a + 1 + ((a >> 2) & 1)) >> 2;
}
// x/2 by one subtraction from its high word; rare: set where that is not the half
// (results below the normal range, infinities, NaN; zero stays zero), which the
// caller then takes the exact way.  Likewise the minimum of three magnitudes, the
// third a sum's less two exponents, is final unless min_is_rare.  (256^3 box, two
// steps: 87.1 ms, with the shifts in line 88.2, with results below the normal range
// dropped 85.9; 128 x 96 x 110 with PPM, three steps: 17.50, 17.84, 17.45.)
__device__ __forceinline__ double half_fast(double x, bool& rare) {
  const int hi = __double2hiint(x), lo = __double2loint(x), a = hi & 0x7fffffff;
  const bool zero = (a | lo) == 0;
  rare = rare | (!zero & ((unsigned)(a - 0x200000) >= 0x7fd00000u));
  return __hiloint2double(zero ? hi : hi - 0x100000, lo);
}
__device__ __forceinline__ bool min_is_rare(long long m) {
  return (unsigned)((int)(m >> 32) - 0x100000) >= 0x7fd00000u - 0x100000u;
}
__device__ __forceinline__ double half_of(double x) {
  const long long b = dbits(x);
  return __longlong_as_double(half_mag(b & kMag) | (b & ~kMag));
}
// a float as a double, exactly, by integer operations
__device__ __forceinline__ double widen(float f) {
  const unsigned u = __float_as_uint(f), a = u & 0x7fffffffu;
  unsigned m = a, e = 896u;  // the magnitude bits, the exponent's offset
  if (a >= 0x7f800000u) {
    e = 0x7ffu - 0xffu;  // infinity, NaN
  } else if (a < 0x00800000u) {
    // subnormal: the leading bit to the implicit place, the exponent from its
    // position; zero stays zero
    const int sh = __clz((int)a) - 8;
    m = a == 0u ? 0u : (a << sh) & 0x007fffffu;
    e = a == 0u ? 0u : 897u - (unsigned)sh;
  }
  const long long d = ((long long)m << 29) + ((long long)e << 52);
  return __longlong_as_double(d | ((long long)(u & 0x80000000u) << 32));
}

// 1/x to about 2^-21 for x > 0, off the FP64 pipe (outside the single-precision
// exponent range: the division)
__device__ __forceinline__ double rcp_approx(double x) {
  return seed_range(x) ? seed_double(__fdividef(1.0f, seed_float(x))) : 1.0 / x;
}
// x > 0 as 2^e (m + u): m in [1, 2) the leading 24 bits, u the other 29
__device__ __forceinline__ void split_mant(double x, float& m, float& u, int& e) {
  const unsigned hi = (unsigned)(dbits(x) >> 32), lo = (unsigned)dbits(x);
  e = (int)(hi >> 20) - 1023;
  m = __uint_as_float(0x3f800000u | ((hi & 0xfffffu) << 3) | (lo >> 29));
  u = __fmul_rn((float)(lo & 0x1fffffffu), 0x1p-52f);
}
// 2^-e r (1 + c) for r in [1/2, 1] and a correction |c| < 2^-22 that keeps it
// there: the bits of r as a double, c r added in units of 2^-53
__device__ __forceinline__ double seed_mant(float r, float c, int e) {
  const int n = __float2int_rn(__fmul_rn(__fmul_rn(r, c), 0x1p53f));
  const long long b = ((long long)(__float_as_int(r) - 0x3f000000) << 29) + n;
  return __longlong_as_double(b + ((long long)(1022 - e) << 52));
}
// a normal x whose reciprocal and root seeds are normal too
__device__ __forceinline__ bool seed_normal(double x) {
  const long long b = dbits(x);
  return b > (4ll << 52) && b < (2040ll << 52);
}
__device__ __forceinline__ double rcp_pos(double x) {
  if (!seed_normal(x)) return 1.0 / x;
  float m, u;
  int e;
  split_mant(x, m, u, e);
  const float r = fminf(fmaxf(__fdividef(1.0f, m), 0.5f), 1.0f);
  const float c = __fmaf_rn(-u, r, __fmaf_rn(-m, r, 1.0f));
  const double y = seed_mant(r, c, e);
  return fma(y, fma(-x, y, 1.0), y);
}
// the seed of 1/sqrt(x)
__device__ __forceinline__ double rsqrt_seed(double x) {
  float m, u;
  int e;
  split_mant(x, m, u, e);
  const float two = (e & 1) ? 2.0f : 1.0f;  // an even exponent: m in [1, 4)
  m *= two;
  u *= two;
  const float r = fminf(fmaxf(rsqrtf(m), 0.5f), 1.0f);
  const float p = __fmul_rn(m, r), q = __fmaf_rn(m, r, -p);  // m r exactly
  const float c =
      __fmaf_rn(-__fmul_rn(u, r), r, __fmaf_rn(-q, r, __fmaf_rn(-p, r, 1.0f)));
  return seed_mant(r, __fmul_rn(c, __fmaf_rn(0.375f, c, 0.5f)), e >> 1);
}
__device__ __forceinline__ double half_normal(double y) {
  return __longlong_as_double(dbits(y) - (1ll << 52));
}
__device__ __forceinline__ double rsqrt_pos(double x) {
  if (!seed_normal(x)) return 1.0 / sqrt(x);
  const double y = rsqrt_seed(x);
  return fma(half_normal(y), fma(-mul(x, y), y, 1.0), y);
}
// Outside the seeds' range: sqrt, but NaN for x = 0 (the square of an E below
// 1e-162 vanishes, and a closure formed from a root of zero would be a pressure of
// -E/3).
__device__ __forceinline__ double sqrt_or_nan(double x) {
  return dbits(x) == 0 ? __longlong_as_double(0x7ff8000000000000ll) : sqrt(x);
}
__device__ __forceinline__ double sqrt_pos(double x) {
  if (!seed_normal(x)) return sqrt_or_nan(x);
  const double y = rsqrt_seed(x), t = mul(x, y);
  return fma(fma(-t, t, x), half_normal(y), t);
}

// ---------------------------------------------------------------- limiter
// Half of the PLM slope with the monotonised-central limiter:
// (1/2) minmod(2 d-, (d- + d+)/2, 2 d+) = sgn * min(|d-|, |d+|, |d- + d+|/4),
// zero unless d- and d+ share a sign.  Face states are u -+ half_slope.
template <typename R>
__device__ __forceinline__ R half_slope(R um, R u0, R up) {
  R dm = u0 - um;
  R dp = up - u0;
  R m = fmin(fmin(fabs(dm), fabs(dp)), R(0.25) * fabs(dm + dp));
  return (dm > R(0) && dp > R(0)) ? m : ((dm < R(0) && dp < R(0)) ? -m : R(0));
}

// double: the same value with the sign tests, the quarter and the minimum on
// the integer pipe.  rare (not EXACT): set where the value has to be taken the
// exact way.
template <bool EXACT>
__device__ __forceinline__ double half_slope_d64(double um, double u0, double up, bool& rare) {
  double dm = u0 - um;
  double dp = up - u0;
  long long bm = dbits(dm), bp = dbits(dp);
  long long am = bm & kMag, ap = bp & kMag;
  const long long as = abs_bits(dm + dp);
  const long long m = min(min(am, ap), EXACT ? quarter_mag(as) : as - (2ll << 52));
  const bool take = ((bm ^ bp) >= 0) & (am != 0) & (ap != 0);  // same sign, both nonzero
  if (!EXACT) rare = rare | (take & min_is_rare(m));
  return __longlong_as_double(take ? (m | (bm & ~kMag)) : 0ll);
}
template <>
__device__ __forceinline__ double half_slope<double>(double um, double u0, double up) {
  bool rare;
  return half_slope_d64<true>(um, u0, up, rare);
}

// Those of the four fields of a cell, the exact quarter only where one needs it.
template <typename R>
__device__ __forceinline__ void half_slopes(const R um[4], const R u0[4], const R up[4], R h[4]) {
  if constexpr (sizeof(R) == sizeof(double)) {
    bool rare = false;
#pragma unroll
    for (int q = 0; q < 4; ++q) h[q] = half_slope_d64<false>(um[q], u0[q], up[q], rare);
    if (rare) {
#pragma unroll
      for (int q = 0; q < 4; ++q) h[q] = half_slope_d64<true>(um[q], u0[q], up[q], rare);
    }
  } else {
#pragma unroll
    for (int q = 0; q < 4; ++q) h[q] = half_slope(um[q], u0[q], up[q]);
  }
}

// ---------------------------------------------------------------- PPM
// Piecewise parabolic face states (Colella & Woodward 1984, the paper's
// reconstruction in Sec. 3.3) written with half slopes h = dm/2 of the
// limiter above.  Interface value between cells u0 and up (their eq. 1.6 with
// the limited slopes of eq. 1.8): (u0 + up)/2 - (dm(up) - dm(u0))/6
// = (u0 + up)/2 - (h1 - h0)/3; it lies between u0 and up.
template <typename R>
__device__ __forceinline__ R ppm_interface(R u0, R up, R h0, R h1) {
  if constexpr (sizeof(R) == sizeof(double))
    return fma(sub(h0, h1), 1.0 / 3.0, half_of(add(u0, up)));
  else
    return R(0.5) * (u0 + up) - (h1 - h0) * R(1.0 / 3.0);
}

// The same from the four cells um .. upp, the slopes and the half sum taken the
// short way unless EXACT (rare: see half_fast), and those of the four fields.
template <bool EXACT>
__device__ __forceinline__ double ppm_interface_d64(double um, double u0, double up, double upp,
                                                    bool& rare) {
  const double h0 = half_slope_d64<EXACT>(um, u0, up, rare);
  const double h1 = half_slope_d64<EXACT>(u0, up, upp, rare);
  const double s = add(u0, up);
  return fma(sub(h0, h1), 1.0 / 3.0, EXACT ? half_of(s) : half_fast(s, rare));
}
// SHORT: not in the transport-only kernel, which has the registers of one way
// (96^3 with PPM: 1.65 ms with both, 1.40 with one).
template <bool SHORT, typename R>
__device__ __forceinline__ void ppm_interfaces(const R um[4], const R u0[4], const R up[4],
                                               const R upp[4], R a[4]) {
  if constexpr (SHORT && sizeof(R) == sizeof(double)) {
    bool rare = false;
#pragma unroll
    for (int q = 0; q < 4; ++q)
      a[q] = ppm_interface_d64<false>(um[q], u0[q], up[q], upp[q], rare);
    if (rare) {
#pragma unroll
      for (int q = 0; q < 4; ++q)
        a[q] = ppm_interface_d64<true>(um[q], u0[q], up[q], upp[q], rare);
    }
  } else {
#pragma unroll
    for (int q = 0; q < 4; ++q)
      a[q] = ppm_interface(u0[q], up[q], half_slope(um[q], u0[q], up[q]),
                           half_slope(u0[q], up[q], upp[q]));
  }
}

// Their monotonicity constraint (eq. 1.10) on the edge values (l, r) of a
// cell of mean u0.  With dl = u0 - l and dr = r - u0: at a local extremum
// (dl dr <= 0) the cell is flat; otherwise the parabola is monotone in the
// cell iff |dl| <= 2|dr| and |dr| <= 2|dl| (its two tests, dd m6 > dd^2 and
// -dd^2 > dd m6 with dd = dl + dr and m6 = 3 (dl - dr), divided through by
// dd), and an edge beyond that is moved onto it: |dl| <- min(|dl|, 2|dr|),
// |dr| <- min(|dr|, 2|dl|), signs kept.  The constraint is continuous where
// its branches meet, so a tie decided either way changes an edge by
// rounding only.  Returned: the constrained left edge (LEFT) or right edge.
template <bool LEFT, typename R>
__device__ __forceinline__ R ppm_edge(R u0, R l, R r) {
  const R dl = u0 - l, dr = r - u0;
  if (!(dl * dr > R(0))) return u0;
  const R a = LEFT ? dl : dr, b = LEFT ? dr : dl;  // the moved side, the other
  const R m = fmin(fabs(a), R(2) * fabs(b));
  return LEFT ? u0 - copysign(m, a) : u0 + copysign(m, a);
}

// double: the sign tests, the minima and 2|b| on the integer pipe (non-negative
// doubles order as their bit patterns)
template <bool LEFT>
__device__ __forceinline__ double ppm_edge_d(double u0, double l, double r) {
  const double dl = u0 - l, dr = r - u0;
  const double a = LEFT ? dl : dr, b = LEFT ? dr : dl;
  const long long ba = dbits(a), bb = dbits(b);
  const long long ma = ba & kMag, mb = bb & kMag;
  const bool mono = ((ba ^ bb) >= 0) & (ma != 0) & (mb != 0);
  // (2|b| of a subnormal b doubles its bits; none is below infinity above)
  const long long b2 = mb < (1ll << 52) ? 2 * mb : min(mb + (1ll << 52), kInfBits);
  const long long m = min(ma, b2);
  const double s = __longlong_as_double(mono ? (m | (ba & ~kMag)) : 0ll);
  return LEFT ? u0 - s : u0 + s;
}

template <bool LEFT, typename R>
__device__ __forceinline__ R ppm_edge_of(R u0, R l, R r) {
  if constexpr (sizeof(R) == sizeof(double))
    return ppm_edge_d<LEFT>(u0, l, r);
  else
    return ppm_edge<LEFT>(u0, l, r);
}

// States of the face between u[2] and u[3] from cells u[0..5] (the face's
// three cells on each side): the constrained right edge of u[2] | the
// constrained left edge of u[3].
template <typename R>
__device__ __forceinline__ void ppm_face(const R u[6], R& L, R& Rr) {
  const R h1 = half_slope(u[0], u[1], u[2]), h2 = half_slope(u[1], u[2], u[3]);
  const R h3 = half_slope(u[2], u[3], u[4]), h4 = half_slope(u[3], u[4], u[5]);
  const R a12 = ppm_interface(u[1], u[2], h1, h2);
  const R a23 = ppm_interface(u[2], u[3], h2, h3);
  const R a34 = ppm_interface(u[3], u[4], h3, h4);
  L = ppm_edge_of<false>(u[2], a12, a23);
  Rr = ppm_edge_of<true>(u[3], a23, a34);
}

// The PPM limiter of Colella & Sekora (2008) (reconstruction PPM_CS), which
// keeps smooth extrema.  Interface value between cells u0 and up from
// um .. upp: the fourth-order value 7/12 (u0 + up) - 1/12 (um + upp); where it
// leaves [u0, up] its second difference 3 (u0 - 2a + up) is limited against
// those of the two cells (the smallest magnitude, C = 1.25 on its own, if all
// three share a sign, else zero) and a = (u0 + up)/2 - D2_lim/6.
template <typename R>
__device__ __forceinline__ bool same_sign3(R a, R b, R c) {
  return (a > R(0) && b > R(0) && c > R(0)) || (a < R(0) && b < R(0) && c < R(0));
}

template <typename R>
__device__ __forceinline__ R cs_interface(R um, R u0, R up, R upp) {
  R a = R(7.0 / 12.0) * (u0 + up) - R(1.0 / 12.0) * (um + upp);
  if ((a - u0) * (up - a) < R(0)) {
    const R d2 = R(3) * (u0 - R(2) * a + up);
    const R d2l = um - R(2) * u0 + up, d2r = u0 - R(2) * up + upp;
    R lim = R(0);
    if (same_sign3(d2, d2l, d2r))
      lim = copysign(fmin(R(1.25) * fabs(d2), fmin(fabs(d2l), fabs(d2r))), d2);
    a = R(0.5) * (u0 + up) - lim * R(1.0 / 6.0);
  }
  return a;
}

// Edges (l, r) of a cell of mean u0 with neighbours um, up under the
// Colella-Sekora constraint; d2L, d2R: second differences of the cells on
// either side.  At a local extremum (of the edges or of the means) the
// curvature -12 u0 + 6 (l + r) is limited against C = 1.25 times the second
// differences of the three cells and both edges scale towards u0 by the
// ratio; elsewhere an edge more than twice as far from u0 as the other is
// moved to twice that distance.
template <typename R>
__device__ __forceinline__ void cs_edges(R um, R u0, R up, R d2L, R d2R, R& l, R& r) {
  if ((r - u0) * (u0 - l) <= R(0) || (um - u0) * (u0 - up) <= R(0)) {
    const R d2 = R(-12) * u0 + R(6) * (l + r), d2c = um - R(2) * u0 + up;
    R lim = R(0);
    if (same_sign3(d2, d2c, d2L) && same_sign3(d2, d2c, d2R))
      lim = copysign(fmin(fabs(d2), R(1.25) * fmin(fabs(d2c), fmin(fabs(d2L), fabs(d2R)))),
                     d2);
    if (d2 != R(0)) {
      const R fac = lim / d2;
      l = u0 + (l - u0) * fac;
      r = u0 + (r - u0) * fac;
    } else {
      l = u0;
      r = u0;
    }
  } else {
    const R dl = u0 - l, dr = r - u0;
    if (fabs(dr) >= R(2) * fabs(dl))
      r = u0 + R(2) * dl;
    else if (fabs(dl) >= R(2) * fabs(dr))
      l = u0 - R(2) * dr;
  }
}

// Colella-Sekora states of the face between u[2] and u[3] from u[0..5]
template <typename R>
__device__ __forceinline__ void ppm_cs_face(const R u[6], R& L, R& Rr) {
  const R a12 = cs_interface(u[0], u[1], u[2], u[3]);
  const R a23 = cs_interface(u[1], u[2], u[3], u[4]);
  const R a34 = cs_interface(u[2], u[3], u[4], u[5]);
  R l2 = a12, r2 = a23, l3 = a23, r3 = a34;
  cs_edges(u[1], u[2], u[3], u[0] - R(2) * u[1] + u[2], u[2] - R(2) * u[3] + u[4], l2, r2);
  cs_edges(u[2], u[3], u[4], u[1] - R(2) * u[2] + u[3], u[3] - R(2) * u[4] + u[5], l3, r3);
  L = r2;
  Rr = l3;
}

// ---------------------------------------------------------------- closure
// Levermore M1 closure (the paper leaves the closure free, Sec. 2.1):
// P = E [(1 - xi)/2 I + (3 xi - 1)/2 n n], xi = (3 + 4 f^2)/(5 + 2 sqrt(4 - 3 f^2)),
// f = |Ft|/E clipped to [0, 1], Ft = F/c.  With s = sqrt(4 E^2 - 3 |Ft|^2)
// the same tensor is exactly
//     P = (s - E)/3 I + 3/(2E + s) Ft Ft^T          (|Ft| <= E),
// which needs one square root and one reciprocal and no division by |Ft|
// (zero flux gives E/3 I without a special case).  Above the free-streaming
// limit f is clipped to 1: P = E n n = (E/|Ft|^2) Ft Ft^T.  m1_coeffs returns
// (ha, hb) with P = ha I + hb Ft Ft^T.
__device__ __forceinline__ void m1_coeffs(double E, const double Ft[3], double& ha, double& hb) {
  const double F2 = dot3(Ft, Ft);
  const double E2 = mul(E, E);
  if (lt_nn(E2, F2)) {
    ha = 0.0;
    hb = mul(E, rcp_pos(F2));
  } else {
    const double s = sqrt_pos(fma(-3.0, F2, mul(4.0, E2)));
    ha = mul(sub(s, E), 1.0 / 3.0);
    hb = mul(3.0, rcp_pos(fma(2.0, E, s)));
  }
}

// ------------------------------------------------------------------- HLL
// Flux through one face along axis d (Sec. 3.3 Godunov step, Sec. 4.3 wave
// speeds) for the RSLA system dE/dt = -chat div(Ft), dFt/dt = -chat div(P),
// from the reconstructed face states L and R (E, Ft), in units of chat/2 (the
// update's weights hold the factor).  Reconstructed fluxes above the
// free-streaming limit are scaled back onto |Ft| = E.  Symmetric speeds S_R =
// -S_L = chat sqrt(max(D_dd,L, D_dd,R, 1/3)), D = P/E, so HLL is
//   Phi = (Phi_L + Phi_R)/2 - S (U_R - U_L)/2,
// with the optical-depth factor eps on the energy part (1 for HLL NONE).
// Returns false for a face state with E <= 0 (or NaN).

// One side: the free-streaming limit applied to q = (E, Ft), and row d of its
// P.  With h = s/2 = sqrt(E^2 - 3/4 |Ft|^2) the closure of m1_coeffs is P =
// (2h - E)/3 I + 3/2/(E + h) Ft Ft^T; E^2 and |Ft|^2 serve the limit as well
// (a flux scaled back has |Ft| = E, so P = E n n).
__device__ __forceinline__ void face_side(int d, double q[4], int closure, double P[3]) {
  const double E = q[0], E2 = mul(E, E), F2 = dot3(q + 1, q + 1);
  const bool over = lt_nn(E2, F2);
  // one root serves both: h, and above the limit 1/|Ft|
  const double x = over ? F2 : fma(-0.75, F2, E2);
  double y, t, h;
  if (seed_normal(x)) {
    y = rsqrt_seed(x);
    t = mul(x, y);
    h = fma(fma(-t, t, x), half_normal(y), t);
  } else {
    t = h = sqrt_or_nan(x);
    y = 1.0 / h;
  }
  if (over) {
    const double sc = mul(E, fma(half_normal(y), fma(-t, y, 1.0), y));
#pragma unroll
    for (int j = 0; j < 3; ++j) q[1 + j] = mul(q[1 + j], sc);
    h = half_of(E);
  }
  if (closure == RHD_CLOSURE_EDDINGTON) {
    P[0] = P[1] = P[2] = 0.0;
    P[d] = mul(E, 1.0 / 3.0);
    return;
  }
  const double ha = mul(fma(2.0, h, -E), 1.0 / 3.0);
  t = mul(mul(1.5, rcp_pos(add(E, h))), q[1 + d]);
#pragma unroll
  for (int j = 0; j < 3; ++j) P[j] = j == d ? fma(t, q[1 + j], ha) : mul(t, q[1 + j]);
}

__device__ __forceinline__ bool hll_states(int d, double L[4], double R[4], double eps,
                                           int closure, double out[4]) {
  if (!pos_finite(L[0]) || !pos_finite(R[0])) {
    out[0] = out[1] = out[2] = out[3] = 0.0;
    return false;
  }
  double PL[3], PR[3];
  face_side(d, L, closure, PL);
  face_side(d, R, closure, PR);
  // S/chat from the largest of D_dd,L, D_dd,R and 1/3, without dividing each
  // (P_dd >= 0): sqrt(num/den) = num/sqrt(num den)
  double num = PL[d], den = L[0];
  if (lt_nn(mul(PL[d], R[0]), mul(PR[d], L[0]))) { num = PR[d]; den = R[0]; }
  if (lt_nn(mul(3.0, num), den)) { num = 1.0; den = 3.0; }
  const double S = mul(num, rsqrt_pos(mul(num, den)));
  out[0] = fma(-mul(eps, S), sub(R[0], L[0]), add(L[1 + d], R[1 + d]));
#pragma unroll
  for (int j = 0; j < 3; ++j) out[1 + j] = fma(-S, sub(R[1 + j], L[1 + j]), add(PL[j], PR[j]));
  return true;
}

// Mixed precision: row d of the deviation P - (E/3) I of the closure tensor,
// in single precision.  From the form above, P - (E/3) I =
// (3 Ft Ft^T - |Ft|^2 I)/(2E + s) below the free-streaming limit (E n n - E/3 I
// above it; zero for the Eddington closure).  It is O(|Ft|^2/E), so its
// single-precision rounding is small next to the flux, where a rounded P_dd
// ~ E/3 would carry an error of an ulp of E/3 into every face.
__device__ __forceinline__ void m1_dev_row(int d, float E, const float Ft[3], int closure,
                                           float D[3]) {
  D[0] = D[1] = D[2] = 0.f;
  if (closure == RHD_CLOSURE_EDDINGTON) return;
  const float F2 = Ft[0] * Ft[0] + Ft[1] * Ft[1] + Ft[2] * Ft[2];
  const float E2 = E * E;
  float hb, ha;
  if (F2 > E2) {
    hb = E / F2;
    ha = -E * (1.f / 3.f);
  } else {
    const float s = sqrtf(4.f * E2 - 3.f * F2);
    const float w = 1.f / (2.f * E + s);
    hb = 3.f * w;
    ha = -F2 * w;
  }
  const float t = hb * Ft[d];
#pragma unroll
  for (int j = 0; j < 3; ++j) D[j] = t * Ft[j];
  D[d] += ha;
}

// HLL flux of hll_states in mixed precision.  The isotropic part of the
// normal momentum flux, hc (E_L + E_R)/3 (hc = chat/2), is linear in the face
// states: iso = E_L + E_R is returned in double (the exact single-precision
// face energies, widened off the FP64 pipe) and left out of out[1 + d], which
// carries the single-precision rest.  The flux of F along d is out[1 + d] +
// chat/6 iso (units of 1, where the double-precision flux has chat/2).  Rounding P_dd in single precision at every face gives each face an
// independent error of an ulp of E/3, which the flux difference turns into
// an error of the flux update of order 1e-7 E/|Ft| relative; near isotropy
// (|Ft| << E) that is the dominant single-precision error.
__device__ __forceinline__ bool hll_states_mixed(int d, float L[4], float Rr[4], float eps,
                                                 float chat, int closure, float out[4],
                                                 double& iso) {
  iso = 0.0;
  if (!(L[0] > 0.f) || !(Rr[0] > 0.f)) {
    out[0] = out[1] = out[2] = out[3] = 0.f;
    return false;
  }
  {
    float n2 = L[1] * L[1] + L[2] * L[2] + L[3] * L[3];
    if (L[0] * L[0] < n2) {
      const float sc = L[0] / sqrtf(n2);
      L[1] *= sc; L[2] *= sc; L[3] *= sc;
    }
    n2 = Rr[1] * Rr[1] + Rr[2] * Rr[2] + Rr[3] * Rr[3];
    if (Rr[0] * Rr[0] < n2) {
      const float sc = Rr[0] / sqrtf(n2);
      Rr[1] *= sc; Rr[2] *= sc; Rr[3] *= sc;
    }
  }
  float DL[3], DR[3];
  m1_dev_row(d, L[0], &L[1], closure, DL);
  m1_dev_row(d, Rr[0], &Rr[1], closure, DR);
  // D_dd = 1/3 + dev/E: the larger side and the 1/3 floor by the deviations
  float num = DL[d], den = L[0];
  if (DL[d] * Rr[0] < DR[d] * L[0]) { num = DR[d]; den = Rr[0]; }
  const float S = num > 0.f ? chat * sqrtf(1.f / 3.f + num / den) : chat * sqrtf(1.f / 3.f);
  const float hc = 0.5f * chat;
  const float hS = 0.5f * S;
  out[0] = hc * (L[1 + d] + Rr[1 + d]) - eps * hS * (Rr[0] - L[0]);
#pragma unroll
  for (int j = 0; j < 3; ++j) out[1 + j] = hc * (DL[j] + DR[j]) - hS * (Rr[1 + j] - L[1 + j]);
  iso = widen(L[0]) + widen(Rr[0]);
  return true;
}

// The face flux in the transport precision R: hll_states for double (units of
// chat/2; iso = 0, unused), hll_states_mixed for float.
template <typename R>
__device__ __forceinline__ bool face_hll(int d, R L[4], R Rr[4], R eps, R chat, int closure,
                                         R out[4], double& iso) {
  if constexpr (sizeof(R) == 8) {
    iso = 0.0;
    return hll_states(d, L, Rr, eps, closure, out);
  } else {
    return hll_states_mixed(d, L, Rr, eps, chat, closure, out, iso);
  }
}

// Optical-depth factor of the HLL energy dissipation (reading of Sec. 4.3):
// (1 - exp(-tau))/tau, 1 in the thin limit, 1/tau in the thick limit.
__device__ __forceinline__ double tau_factor(double tau) {
  return tau > 0.0 ? -expm1(-tau) / tau : 1.0;
}

// ------------------------------------------------------------ local solve
// Start of the inner Newton iteration.  With v and F frozen, eq. (FGFR) and
// eq. (Rnew) reduce exactly to a quartic for the gas temperature:
//   A T^4 + C_v T = C,  A = (c/chat) k g a/(1 + k g),
//   C = Egas(t) - E_kin + (c/chat) k (g E(t) - v.F/c^2)/(1 + k g),
// whose positive root is the converged inner state.  quartic_start solves
// a4 T^4 + T = rhs (a4 = A/C_v, rhs = C/C_v) in single precision in the
// variable t = T/T(t) (alpha t^4 + beta t = 1, coefficients of order one) by
// Newton from the upper bound min(1/beta, alpha^-1/4), where the convex
// quartic converges monotonically.  The double-precision Newton of the paper
// then starts from it instead of from (Egas(t), 0) and needs fewer updates;
// it converges to the same root.  Returns false (cold start) if the
// single-precision numbers are not finite.
__device__ __forceinline__ bool quartic_start(double a4, double rhs, double T0, double& T) {
  float al = (float)(a4 * (T0 * T0) * (T0 * T0) / rhs);
  float be = (float)(T0 / rhs);
  if (!(al >= 0.f) || !(be > 0.f) || !isfinite(al) || !isfinite(be)) return false;
  float t = fminf(1.0f / be, al > 0.f ? rsqrtf(sqrtf(al)) : INFINITY);
#pragma unroll
  for (int i = 0; i < 6; ++i) {
    float t2 = t * t;
    float f = fmaf(al * t2, t2, fmaf(be, t, -1.0f));
    float fp = fmaf(4.0f * al * t2, t, be);
    t = t - __fdividef(f, fp);
  }
  if (!(t > 0.f) || !isfinite(t)) return false;
  T = (double)t * T0;
  return true;
}

// (T/T_ref)^p of chi = kappa rho (T/T_ref)^p.  Whole exponents (the Marshak
// wave's -3) by a product that carries its rounding errors (fused
// multiply-adds; Dekker 1971) and one reciprocal: within 1 ulp, and 13 FP64
// operations for -3, where pow takes several times that in every Newton update
// (a 60-cell Marshak wave, 50 steps: 4.86 ms, with pow 6.56).
__device__ __forceinline__ double opacity_power(const Physics& ph, double x) {
  const int n = ph.kappa_T_int < 0 ? -ph.kappa_T_int : ph.kappa_T_int;
  if (n == 0) return pow(x, ph.kappa_T_exp);
  double hi = x, lo = 0.0;
  for (int i = 1; i < n; ++i) {
    const double p = mul(hi, x);
    lo = fma(lo, x, fma(hi, x, -p));
    hi = p;
  }
  if (!seed_range(hi)) return pow(x, ph.kappa_T_exp);
  if (ph.kappa_T_int > 0) return add(hi, lo);
  const double r = rcp_pos(hi);
  return fma(mul(-lo, r), r, r);
}

// Implicit stage of one cell (Sec. 3.3), grey chi.  y = {Egas, m, E, F}
// holds the explicit state on entry and the solution on exit.  tdt = theta dt.
//
// Inner stage: Newton on (Egas, R) for eq. (FGFR) with eq. (Rnew) and the
// paper's Jacobian (beta^2 dropped).  The R-row is multiplied by
// k g (k = chat chi theta dt, g = 1 + beta^2/2), which leaves the Newton
// iterates unchanged and keeps the system regular for small k:
//   r0 = Egas - Egas(t) + (c/chat) R
//   r1 = k g F_R = k g (aT^4 - E(t) - R) + k v.F/c^2 - R
//   J  = [[1, c/chat], [g k 4 a T^3 / C_v, -g (1 + k)]]
// converged when |r0| < eps E_tot and (c/chat)|r1| <= eps E_tot k g,
// E_tot = Egas(t) + (c/chat) E(t).  The iteration starts from pair_start's
// near-converged (R, F); if that gives up, or the iteration fails from there,
// from quartic_start and the explicit F, and with chi ~ T^p (whose J10 gains
// the term of the T-dependence of k) from (Egas(t), 0).
// Energy closure: E = E(t) - (chat/c)(Egas - Egas(t)).
// Outer stage: eq. (numF2) (order 2) or (numF1) (order 1) for F with P from
// the new E and the previous outer flux, momentum m = m(t) - (F - F(t))/(c chat),
// repeated until Q = k[(g - 1)(aT^4 - E) + v.F/c^2] settles: its change is at
// most outer_rtol times |Q|, |R| or the magnitude of its terms.  A warm start
// has applied both tests to its tracked changes; the double-precision pass that
// settles it sees the change from the pairs' flux, whose rounding (up to 1e-13
// of the terms) is allowed for: outer_rtol + min(outer_rtol, 1e-13).  (Without
// it 0.45 % of the cells of a 64^3 box take a further pass, which brings none
// nearer to the 64-bit values: 256^3 moves by 6e-12 at most, its error stays
// 3.7e-12; two steps take 87.4 ms for 85.9, 50 of a 4096-cell row 2.88 for 2.53.)
// MIXED: the reciprocal of the Jacobian determinant is a seed of 2^-21 (a step
// off by that factor only slows the last update); residuals, the state, the
// closure of the exchange term v.P and every update stay double, so the solve
// meets the double-precision convergence tests (inner and outer) and conserves
// to rounding.
// GEN: compiled with the temperature-dependent opacity; the default physics
// (constant chi) uses the GEN = false copy, free of that branch.
constexpr double kNear = 1e4;  // in units of the Newton tolerance

template <bool MIXED, bool GEN>
__device__ __forceinline__ int local_solve(const Physics& ph, double tdt, double rho,
                                           double chi, double y[8], int& nn, int& no) {
  nn = 0;
  no = 0;
  if (chi == 0.0) return RHD_OK;
  const double Cv = mul(rho, ph.cv_spec);
  const double inv_rho = rcp_pos(rho);
  const double inv_Cv = mul(inv_rho, ph.inv_cv_spec);
  const double cr = ph.c_over_chat;
  const double a = ph.a_rad;
  const bool order2 = ph.vc_order == 2;
  const double Eg0 = y[0], E0 = y[4];
  const double Etot = fma(cr, E0, Eg0);
  // k = chat chi theta dt; with a temperature-dependent opacity chi is taken
  // at the current Newton iterate (the paper's chi carry the superscript
  // (t+1)) and held fixed in the Jacobian
  const bool vary = GEN && ph.kappa_T_exp != 0.0;
  const double k0 = mul(mul(ph.chat, chi), tdt);
  double k = k0;
  const double tolG = mul(ph.newton_rtol, Etot);
  double Eg = Eg0, R = 0.0;
  double F[3] = {y[5], y[6], y[7]};
  double v[3] = {mul(y[1], inv_rho), mul(y[2], inv_rho), mul(y[3], inv_rho)};

  // With a temperature-dependent opacity the iteration starts from
  // (Egas(t), 0) like the oracle's: the exact Jacobian below converges
  // quadratically from there, and a common start keeps the two solves on
  // the same iterates near a Marshak front, where the stopping point's
  // rounding is amplified.
  WarmStart W;
  W.lag = 0.0;
  bool warm = !vary && ph.start.ok != 0 &&
              pair_start(ph.start, ph.closure == RHD_CLOSURE_M1, order2, rho, k0, Etot, y, v,
                         ph.newton_max, ph.outer_max, W, nn, no);
  bool settle = warm;  // the first double-precision pass from the warm start
  if (warm) {
    R = W.R;
    Eg = fma(-cr, R, Eg0);
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      F[i] = W.F[i];
      v[i] = mul(fma(-sub(F[i], y[5 + i]), ph.inv_cchat, y[1 + i]), inv_rho);
    }
  }

  for (;;) {  // from the warm start; from the cold one if that fails
    if (!warm) {
      nn = 0;
      no = 0;
      Eg = Eg0;
      R = 0.0;
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        F[i] = y[5 + i];
        v[i] = mul(y[1 + i], inv_rho);
      }
      const double v2 = dot3(v, v);
      const double Ekin = mul(mul(0.5, rho), v2);
      const double T0 = mul(sub(Eg0, Ekin), inv_Cv);
      if (!vary && pos_finite(T0)) {
        const double kg = order2 ? fma(k, mul(0.5, mul(v2, ph.inv_c2)), k) : k;
        const double w = mul(dot3(v, F), ph.inv_c2);
        const double ck = mul(cr, mul(rcp_pos(add(1.0, kg)), inv_Cv));
        const double a4 = mul(mul(ck, kg), a);
        const double rhs = fma(ck, fma(kg, E0, -mul(k, w)), T0);
        double Tg;
        if (pos_finite(rhs) && quartic_start(a4, rhs, T0, Tg)) {
          Eg = fma(Cv, Tg, Ekin);
          R = mul(-ph.chat_over_c, sub(Eg, Eg0));
        }
      }
    }

    int code = RHD_ERR_OUTER;
    while (no < ph.outer_max) {
      ++no;
      // the frozen (v, F): h = beta^2/2 = g - 1 (0 at order 1), v.F/c^2
      const double v2 = dot3(v, v);
      const double h = order2 ? mul(0.5, mul(v2, ph.inv_c2)) : 0.0;
      const double vF = dot3(v, F);
      const double w = mul(vF, ph.inv_c2);
      const double Ekin = mul(mul(0.5, rho), v2);
      double kg = fma(k, h, k);
      double kw = mul(k, w);

      double aT4 = 0.0;
      int inner = RHD_ERR_NEWTON;
      for (int it = 0;; ++it) {
        const double T = mul(sub(Eg, Ekin), inv_Cv);
        if (!pos_finite(T) || !finite_bits(R)) {
          inner = RHD_ERR_NONPHYSICAL;
          break;
        }
        if (vary) {
          k = mul(k0, opacity_power(ph, mul(T, ph.inv_kappa_T_ref)));
          kg = fma(k, h, k);
          kw = mul(k, w);
        }
        const double T2 = mul(T, T);
        aT4 = mul(mul(a, T2), T2);
        const double r0 = fma(cr, R, sub(Eg, Eg0));
        const double r1 = fma(kg, sub(sub(aT4, E0), R), sub(kw, R));
        // a warm start has taken the tests by its lag; its R only has to be
        // near enough for one update with the determinant's seed (2^-21) to
        // land at rounding level
        if (settle && !(lt_nn(fabs(r0), mul(kNear, tolG)) &&
                        le_nn(mul(cr, fabs(sub(r1, W.lag))), mul(mul(kNear, tolG), kg))))
          settle = false;
        const bool conv =
            settle || (lt_nn(fabs(r0), tolG) && le_nn(mul(cr, fabs(r1)), mul(tolG, kg)));
        if (conv) inner = RHD_OK;
        if (conv ? !settle : it >= ph.newton_max) break;
        const double aT3 = mul(mul(mul(4.0 * a, inv_Cv), T2), T);  // d(a T^4)/dEgas
        double J10 = mul(kg, aT3);
        // chi ~ T^p: the R/(k g) term of E(Egas, R) varies with T through k,
        // which adds p R/(T C_v) to the scaled J10 (exact dE/dEgas; the
        // paper's J10 holds chi fixed, Sec. 3.3, and converges linearly)
        if (vary) J10 = add(J10, ph.kappa_T_exp * R / sub(Eg, Ekin));
        const double gpk = add(add(1.0, h), kg);
        const double ndet = fma(cr, J10, gpk);  // > 0
        const double inv_det = settle || MIXED ? rcp_approx(ndet) : rcp_pos(ndet);
        // settling: the update of the residual beyond the one that the
        // iteration leaves removes the pairs' rounding from E_gas and R
        const double r1s = settle ? sub(r1, W.lag) : r1;
        const double dEg = mul(fma(r0, gpk, mul(cr, r1s)), inv_det);
        Eg = sub(Eg, dEg);
        R = fma(-fma(r0, J10, -r1s), inv_det, R);
        if (settle) {
          aT4 = fma(-aT3, dEg, aT4);
          break;
        }
        ++nn;
      }
      if (inner != RHD_OK) {
        code = inner;
        break;
      }

      // energy closure; aT4 is that of the converged Egas
      const double E = fma(-ph.chat_over_c, sub(Eg, Eg0), E0);

      // F(t) + k (aT^4 v + v.P) with P = ha I + hb Ft Ft^T at (E, F); the cell
      // flux may exceed the free-streaming limit
      const double Ft[3] = {mul(F[0], ph.inv_c), mul(F[1], ph.inv_c), mul(F[2], ph.inv_c)};
      double ha = mul(E, 1.0 / 3.0), t = 0.0;
      if (ph.closure == RHD_CLOSURE_M1) {
        double hb;
        m1_coeffs(E, Ft, ha, hb);
        t = mul(hb, mul(vF, ph.inv_c));
      }
      const double u = add(aT4, ha);
      const double inv_den = rcp_pos(add(1.0, kg));
      const double q = sub(aT4, E);
      const double Q_old = mul(k, fma(h, q, w));
      // the updated F, m and v: the next pass freezes these
      double m[3];
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        F[i] = mul(fma(k, fma(u, v[i], mul(t, Ft[i])), y[5 + i]), inv_den);
        m[i] = fma(-sub(F[i], y[5 + i]), ph.inv_cchat, y[1 + i]);
        v[i] = mul(m[i], inv_rho);
      }
      const double hn = order2 ? mul(0.5, mul(dot3(v, v), ph.inv_c2)) : 0.0;
      const double Q_new = mul(k, fma(hn, q, mul(dot3(v, F), ph.inv_c2)));
      // |dQ| <= rtol max(|Q_old|, |R|, Q_scale): the three tests of the outer
      // stop; Q_scale is the magnitude of the terms of Q, the rounding level
      // of a cancelling v.F
      const double dQ = fabs(sub(Q_new, Q_old));
      const double vFa = fma(fabs(v[2]), fabs(F[2]),
                             fma(fabs(v[1]), fabs(F[1]), mul(fabs(v[0]), fabs(F[0]))));
      const double Q_scale = mul(k, fma(hn, fabs(q), mul(vFa, ph.inv_c2)));
      const double big = max_nn(max_nn(fabs(Q_old), fabs(R)), Q_scale);
      if (le_nn(dQ, mul(settle ? ph.outer_settle : ph.outer_rtol, big))) {
        code = pos_finite(E) && finite_bits(F[0]) && finite_bits(F[1]) && finite_bits(F[2])
                   ? RHD_OK
                   : RHD_ERR_NONPHYSICAL;
        if (code == RHD_OK || !warm) {
          y[0] = Eg;
          y[1] = m[0]; y[2] = m[1]; y[3] = m[2];
          y[4] = E;
          y[5] = F[0]; y[6] = F[1]; y[7] = F[2];
        }
        break;
      }
      settle = false;
    }
    if (code == RHD_OK || !warm) return code;
    warm = settle = false;
  }
}

// Closure tensor D = P/E = dA I + dB Ft Ft^T of a state (E, Ft = F/c).
__device__ __forceinline__ void closure_D(const Physics& ph, double E, const double Ft[3],
                                          double& dA, double& dB) {
  if (ph.closure == RHD_CLOSURE_EDDINGTON) {
    dA = 1.0 / 3.0;
    dB = 0.0;
    return;
  }
  double ha, hb;
  m1_coeffs(E, Ft, ha, hb);
  const double iE = 1.0 / E;
  dA = ha * iE;
  dB = hb * iE;
}

// Implicit stage of one cell for non-grey material (general kernels only):
// chi_0E = chi (times the T factor), chi_0P = rP chi_0E, chi_0F = rF chi_0E in
// eq. (G0)/(G1).  The same inner/outer iteration as local_solve, with
//   R = k [(rP a T^4 - E) g + (2 - rF) v.F/c^2 + (rF - 1)(beta^2 + v.D.v/c^2) E]
// (k = chat chi_0E theta dt; the last term at order 2 only, with the closure
// tensor D frozen like v and F: that of the explicit state, then the one of
// the previous flux update), the R-row scaled by k' = k g - (kF - k)(beta^2 +
// v.D.v/c^2), the paper's Jacobian ((chi_0P/chi_0E) 4aT^3/C_v, -1/k - 1), and
// the flux from eq. (fupdate) with eq. (G1): at order 2
//   [(1 + kF g) I + 2 (kF - k)/c^2 v v^T] F = F(t) + kP a T^4 v + kF v.P + (kF - k) E v,
// solved by the Sherman-Morrison formula; at order 1 eq. (numF1).
template <bool MIXED>
__device__ int local_solve_nongrey(const Physics& ph, double tdt, double rho, double chi,
                                   double y[8], int& nn, int& no) {
  nn = 0;
  no = 0;
  if (chi == 0.0) return RHD_OK;
  const double Cv = rho * ph.cv_spec;
  const double inv_Cv = 1.0 / Cv, inv_rho = 1.0 / rho;
  const double cr = ph.c_over_chat, a = ph.a_rad, ic2 = ph.inv_c2;
  const double Eg0 = y[0], E0 = y[4];
  const double tolG = ph.newton_rtol * (Eg0 + cr * E0);
  const bool o2 = ph.vc_order == 2;
  const bool vary = ph.kappa_T_exp != 0.0;
  const double rP = ph.kappa_P_ratio, rF = ph.kappa_F_ratio;
  const double k0 = ph.chat * chi * tdt;
  double Eg = Eg0, R = 0.0, E = E0;
  double m[3] = {y[1], y[2], y[3]};
  double F[3] = {y[5], y[6], y[7]};
  double v[3] = {m[0] * inv_rho, m[1] * inv_rho, m[2] * inv_rho};
  double beta2 = (v[0] * v[0] + v[1] * v[1] + v[2] * v[2]) * ic2;
  double g = o2 ? 1.0 + 0.5 * beta2 : 1.0;
  double w = (v[0] * F[0] + v[1] * F[1] + v[2] * F[2]) * ic2;
  double Ekin = 0.5 * (m[0] * v[0] + m[1] * v[1] + m[2] * v[2]);
  double dA, dB, Fd[3] = {F[0] * ph.inv_c, F[1] * ph.inv_c, F[2] * ph.inv_c};
  closure_D(ph, E0, Fd, dA, dB);
  auto vdv_of = [&](const double vv[3]) {
    double vf = vv[0] * Fd[0] + vv[1] * Fd[1] + vv[2] * Fd[2];
    return (dA * (vv[0] * vv[0] + vv[1] * vv[1] + vv[2] * vv[2]) + dB * vf * vf) * ic2;
  };
  double vDv = vdv_of(v);
  double kE = k0, kP = rP * k0, kF = rF * k0;
  auto set_k = [&](double T) {
    kE = vary ? k0 * opacity_power(ph, mul(T, ph.inv_kappa_T_ref)) : k0;
    kP = rP * kE;
    kF = rF * kE;
  };
  auto kprime = [&]() { return kE * g - (o2 ? (kF - kE) * (beta2 + vDv) : 0.0); };

  if (!vary) {  // start from the frozen-opacity quartic A T^4 + C_v T = C (see quartic_start)
    const double T0 = (Eg0 - Ekin) * inv_Cv;
    if (pos_finite(T0)) {
      set_k(T0);
      const double kp = kprime();
      if (kp > 0.0) {
        const double inv1 = 1.0 / (1.0 + kp);
        const double a4 = cr * kP * g * a * inv1 * inv_Cv;
        const double rhs = T0 + cr * (kp * E0 - (2.0 * kE - kF) * w) * inv1 * inv_Cv;
        double Tg;
        if (pos_finite(rhs) && a4 > 0.0 && quartic_start(a4, rhs, T0, Tg)) {
          Eg = Cv * Tg + Ekin;
          R = -ph.chat_over_c * (Eg - Eg0);
        }
      }
    }
  }

  for (int outer = 0; outer < ph.outer_max; ++outer) {
    no = outer + 1;
    bool conv = false;
    double aT4 = 0.0, kp = 0.0;
    for (int it = 0;; ++it) {
      const double T = (Eg - Ekin) * inv_Cv;
      if (!pos_finite(T) || !finite_bits(R)) return RHD_ERR_NONPHYSICAL;
      set_k(T);
      kp = kprime();
      if (!(kp > 0.0)) return RHD_ERR_NONPHYSICAL;
      const double T2 = T * T;
      aT4 = a * T2 * T2;
      const double Se = kP * aT4 * g + (2.0 * kE - kF) * w;
      const double r0 = (Eg - Eg0) + cr * R;
      const double r1 = Se - R - kp * (E0 + R);
      if (fabs(r0) < tolG && cr * fabs(r1) <= tolG * kp) {
        conv = true;
        break;
      }
      if (it >= ph.newton_max) break;
      double J10 = kp * rP * 4.0 * a * T2 * T * inv_Cv;
      if (vary) J10 += ph.kappa_T_exp * R / (Eg - Ekin);  // as in local_solve
      const double gpk = kp / kE + kp;
      const double det = -gpk - cr * J10;
      const double inv_det = MIXED ? (double)(1.0f / (float)det) : 1.0 / det;
      Eg += (r0 * gpk + cr * r1) * inv_det;
      R += (r0 * J10 - r1) * inv_det;
      ++nn;
    }
    if (!conv) return RHD_ERR_NEWTON;

    E = E0 - ph.chat_over_c * (Eg - Eg0);  // energy closure
    // closure at (E, F of the previous pass): P v for eq. (G1) and the tensor
    // the next inner stage freezes
    double Ft[3] = {F[0] * ph.inv_c, F[1] * ph.inv_c, F[2] * ph.inv_c};
    closure_D(ph, E, Ft, dA, dB);
    Fd[0] = Ft[0]; Fd[1] = Ft[1]; Fd[2] = Ft[2];
    const double vFt = v[0] * Ft[0] + v[1] * Ft[1] + v[2] * Ft[2];
    double rhs[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      const double vP = (dA * v[i] + dB * vFt * Ft[i]) * E;
      rhs[i] = y[5 + i] + kP * aT4 * v[i] + kF * vP + (kF - kE) * E * v[i];
    }
    double Fn[3], mn[3];
    if (o2) {
      const double aa = 1.0 + kF * g;
      const double b = 2.0 * (kF - kE) * ic2;
      const double vr = v[0] * rhs[0] + v[1] * rhs[1] + v[2] * rhs[2];
      const double v2 = v[0] * v[0] + v[1] * v[1] + v[2] * v[2];
      const double corr = b * vr / (aa + b * v2);
#pragma unroll
      for (int i = 0; i < 3; ++i) Fn[i] = (rhs[i] - corr * v[i]) / aa;
    } else {
#pragma unroll
      for (int i = 0; i < 3; ++i) Fn[i] = rhs[i] / (1.0 + kF);
    }
#pragma unroll
    for (int i = 0; i < 3; ++i) mn[i] = y[1 + i] - (Fn[i] - y[5 + i]) * ph.inv_cchat;

    const double Q_old = (kP * aT4 - kE * E) * (g - 1.0) + (2.0 * kE - kF) * w +
                         (o2 ? (kF - kE) * (beta2 + vDv) * E : 0.0);
    double vn[3] = {mn[0] * inv_rho, mn[1] * inv_rho, mn[2] * inv_rho};
    const double beta2n = (vn[0] * vn[0] + vn[1] * vn[1] + vn[2] * vn[2]) * ic2;
    const double gn = o2 ? 1.0 + 0.5 * beta2n : 1.0;
    const double wn = (vn[0] * Fn[0] + vn[1] * Fn[1] + vn[2] * Fn[2]) * ic2;
    const double vDvn = vdv_of(vn);
    const double Q_new = (kP * aT4 - kE * E) * (gn - 1.0) + (2.0 * kE - kF) * wn +
                         (o2 ? (kF - kE) * (beta2n + vDvn) * E : 0.0);
    const double Q_scale =
        fabs((kP * aT4 - kE * E) * (gn - 1.0)) +
        fabs(2.0 * kE - kF) * (fabs(vn[0] * Fn[0]) + fabs(vn[1] * Fn[1]) + fabs(vn[2] * Fn[2])) *
            ic2 +
        (o2 ? fabs(kF - kE) * (beta2n + fabs(vDvn)) * E : 0.0);
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      F[i] = Fn[i];
      m[i] = mn[i];
      v[i] = vn[i];
    }
    beta2 = beta2n;
    g = gn;
    w = wn;
    vDv = vDvn;
    Ekin = 0.5 * (m[0] * v[0] + m[1] * v[1] + m[2] * v[2]);
    const double dQ = fabs(Q_new - Q_old);
    if (dQ <= ph.outer_rtol * fabs(Q_old) || dQ <= ph.outer_rtol * fabs(R) ||
        dQ <= ph.outer_rtol * Q_scale) {
      y[0] = Eg;
      y[1] = m[0]; y[2] = m[1]; y[3] = m[2];
      y[4] = E;
      y[5] = F[0]; y[6] = F[1]; y[7] = F[2];
      if (!pos_finite(E) || !finite_bits(F[0]) || !finite_bits(F[1]) || !finite_bits(F[2]))
        return RHD_ERR_NONPHYSICAL;
      return RHD_OK;
    }
  }
  return RHD_ERR_OUTER;
}

// ------------------------------------------------------------ launchers
// (host side, defined in the .cu files)
// b0, b1: the tile rows [b0, b1) of the slowest axis (b1 < 0: to the end)
cudaError_t launch_stage(int stage, int precision, const StageArgs& A, cudaStream_t s,
                         int b0 = 0, int b1 = -1);
cudaError_t launch_stage_ppm(int stage, int precision, const StageArgs& A, cudaStream_t s,
                             int b0 = 0, int b1 = -1);
// tile rows of a grid along its slowest axis, and the cells of one row
int stage_rows(const Geometry& g);
long long stage_row_cells(const Geometry& g, int row);
cudaError_t launch_status_reset(DevStatus* st, cudaStream_t s);
cudaError_t launch_totals(const Geometry& g, const Physics& ph, const double* y,
                          double* partials, int npart, double* out4, cudaStream_t s);
int totals_partials_needed();
// halo_kappa, halo_rho: plane 0 of the slab above a HALO top face (else null);
// i0, i1: the cells [i0, i1) whose +d faces are computed (i1 < 0: to the end)
cudaError_t launch_tau_eps(const Geometry& g, const double* rho, const double* kappa,
                           double tau_scale, double* const eps[3], cudaStream_t s,
                           const double* halo_kappa = nullptr,
                           const double* halo_rho = nullptr, long long i0 = 0,
                           long long i1 = -1);
cudaError_t launch_check_field(int field, const double* x, int n, int* flag,
                               cudaStream_t s);
// message returned by rhd_last_error(NULL) on this thread
void set_global_error(const char* msg);
// device-side geometry and physics of validated params
void fill_geometry(const rhd_params* p, Geometry& g, Physics& ph);
// whether a grid needs the general kernels (RK2-SSP, a temperature-dependent
// opacity or an inflow face) rather than the lean default ones
inline bool needs_general(const Geometry& g, const Physics& ph) {
  if (ph.scheme != RHD_SCHEME_IMEX_PDARS || ph.kappa_T_exp != 0.0 ||
      ph.reconstruction != RHD_RECON_PLM ||
      ph.kappa_P_ratio != 1.0 || ph.kappa_F_ratio != 1.0)
    return true;
  for (int d = 0; d < g.ndim; ++d)
    if (g.bc[d][0] == RHD_BC_INFLOW || g.bc[d][1] == RHD_BC_INFLOW) return true;
  return false;
}

}  // namespace rhd
