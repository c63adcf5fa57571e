// Device-side physics of the ideal-MHD Godunov step: primitive recovery,
// MC-limited piecewise-linear reconstruction, the HLLD and HLL Riemann
// fluxes and the upwind constrained-transport edge average.
//
// The paper (Sec. 2.2) names the stages of the gPLUTO step -- reconstruction
// of primitive variables, the Riemann solve at each interface, the
// flux-conservative update and, for MHD, constrained transport -- but prints
// no formulas.  The arithmetic below follows the published methods those
// stages name:
//   * MC limiter: slope = minmod(2 dm, 2 dp, (dm + dp)/2) (van Leer 1977);
//   * HLLD: Miyoshi & Kusano, J. Comput. Phys. 208 (2005) 315, eqs. 38-66;
//   * HLL: Harten, Lax & van Leer (1983) with the Davis wave-speed bounds
//     S_L = min(u_L,u_R) - max(cf_L,cf_R), S_R = max(u_L,u_R) + max(cf_L,cf_R);
//   * CT edge EMF: Gardiner & Stone, J. Comput. Phys. 205 (2005) 509,
//     eqs. 41-50 (upwinded by the sign of the face mass flux).
// Template parameter R is the arithmetic type (double for the FP64 path,
// float for the mixed and FP32 paths).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace mhd {

template <typename R> struct Eps;
template <> struct Eps<double> { static constexpr double degen = 1e-12; };
template <> struct Eps<float> { static constexpr float degen = 1e-6f; };

// Comparisons.  FP32: the FP32 compare instructions.  FP64 on the device:
// integer comparisons of the IEEE bit patterns, which keep them off the FP64
// pipe (one warp-instruction per ~17 SM cycles on GB300; the integer pipes
// are nearly idle in the FP64 form).  For non-NaN x the signed 64-bit key
// k(x) = b ^ ((b >> 63) & 0x7fff...f), b the bit pattern, orders as x does
// (with -0 just below +0); tests against zero use the sign and the pattern
// directly, so +-0 compare as IEEE does.  NaN inputs are not ordered as
// IEEE orders them (min/max may drop a NaN, as fmin/fmax do).
template <typename R> __host__ __device__ __forceinline__ R rabs(R x) { return x < R(0) ? -x : x; }
template <typename R> __host__ __device__ __forceinline__ R rmin(R a, R b) { return a < b ? a : b; }
template <typename R> __host__ __device__ __forceinline__ R rmax(R a, R b) { return a > b ? a : b; }
template <typename R> __host__ __device__ __forceinline__ bool gt0(R x) { return x > R(0); }
template <typename R> __host__ __device__ __forceinline__ bool lt0(R x) { return x < R(0); }
template <typename R> __host__ __device__ __forceinline__ bool lt_(R a, R b) { return a < b; }
#ifdef __CUDA_ARCH__
__device__ __forceinline__ long long okey(double x) {
  const long long b = __double_as_longlong(x);
  return b ^ ((b >> 63) & 0x7fffffffffffffffLL);
}
template <> __device__ __forceinline__ double rabs<double>(double x) { return fabs(x); }
template <> __device__ __forceinline__ double rmin<double>(double a, double b) { return okey(a) < okey(b) ? a : b; }
template <> __device__ __forceinline__ double rmax<double>(double a, double b) { return okey(a) > okey(b) ? a : b; }
template <> __device__ __forceinline__ bool gt0<double>(double x) { return __double_as_longlong(x) > 0; }
template <> __device__ __forceinline__ bool lt0<double>(double x) {
  return (unsigned long long)__double_as_longlong(x) > 0x8000000000000000ull;
}
template <> __device__ __forceinline__ bool lt_<double>(double a, double b) { return okey(a) < okey(b); }
#endif
template <typename R> __host__ __device__ __forceinline__ bool ge0(R x) { return !lt0(x); }
template <typename R> __host__ __device__ __forceinline__ bool le0(R x) { return !gt0(x); }
template <typename R> __host__ __device__ __forceinline__ bool le_(R a, R b) { return !lt_(b, a); }

// Reciprocal, square root and reciprocal square root.  FP32: the hardware
// instructions (the FP32-bulk units are compiled with approximate divide and
// square root).  FP64 on the device: the PTX approximate seeds
// rcp.approx.ftz.f64 / rsqrt.approx.ftz.f64 (measured relative error ~1e-6)
// refined by one third-order step, which cubes that error (~1e-18, so the
// result is within a few ulp of the IEEE one), in three to five FP64-pipe
// operations instead of an IEEE-rounded sequence (GB300 issues one FP64
// warp-instruction per ~17 SM cycles).  The steps are the truncated series
//   1/x        = r0 / (1 - e)       ~ r0 (1 + e + e^2),          e = 1 - x r0
//   1/sqrt(x)  = y0 (1 - h)^(-1/2)  ~ y0 (1 + h/2 + 3 h^2/8),    h = 1 - x y0^2
// and sqrt(x) = x / sqrt(x).  Zero, subnormal, infinite, NaN and (for the
// roots) negative inputs, recognised with integer tests, take the IEEE
// operation.
__host__ __device__ __forceinline__ bool f64_plain(double x) {
#ifdef __CUDA_ARCH__
  const int e = __double2hiint(x) & 0x7ff00000;
  return e != 0 && e != 0x7ff00000;
#else
  return false;
#endif
}
__host__ __device__ __forceinline__ double rcp_(double x) {
#ifdef __CUDA_ARCH__
  if (!f64_plain(x)) return 1.0 / x;
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
  const double e = fma(-x, r, 1.0);
  return fma(r, fma(e, e, e), r);
#else
  return 1.0 / x;
#endif
}
__host__ __device__ __forceinline__ double rrsqrt_(double x) {
#ifdef __CUDA_ARCH__
  if (!f64_plain(x) || __double2hiint(x) < 0) return 1.0 / sqrt(x);
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double h = fma(-(x * y), y, 1.0);
  return fma(y, h * fma(0.375, h, 0.5), y);
#else
  return 1.0 / sqrt(x);
#endif
}
__host__ __device__ __forceinline__ double rsqrt_(double x) {   // square root
#ifdef __CUDA_ARCH__
  if (!f64_plain(x) || __double2hiint(x) < 0) return sqrt(x);
  return x * rrsqrt_(x);
#else
  return sqrt(x);
#endif
}
// The same three with fewer FP64-pipe operations again (rcp 2, rsqrt and root
// 3), where the result may round differently (the characteristic slopes and
// the lean solvers below), and no less exact.  With the residual e of the seed
// y (t = x y for the root) the result is y + y (1 + e) e (rcp), y + y/2 (1 +
// 3/4 e) e (rsqrt), t (1 + 3/8 e^2) + t/2 e (root).  What stands before the
// last e is needed to 2^-33 only: it is formed on the bits of y, and the step
// to the result is one fma.  Halving is an exponent decrement.  A face has
// nine of them.  Errors in ulps, largest / mean of random mantissas: rcp 0.507 /
// 0.250, rsqrt 0.999 / 0.276, root 1.25 / 0.352; the forms above 0.508 / 0.250,
// 0.999 / 0.276, 1.73 / 0.383.  Measured (GB300, stage 1 / 2): 128^3 HLLD 4887 /
// 4976 us with the forms above, 4619 / 4717 with these, HLL 4432 / 4505 and 4286 /
// 4355, characteristic 96x64x80 1983 / 1976 and 1843 / 1837.  (Steps on the bits
// of e, or of y for any y, need a test for the next binade: 128^3 6 % slower.)
#ifdef __CUDA_ARCH__
// y (1 + (EIGHTHS / 8) e) to 2^-40 of itself, for a hardware seed y (20 leading
// mantissa bits, the others zero) and its residual, |e| < 2^-19.8: e times y's
// mantissa, in FP32 (e below 2^-62 counts as that), as a number of 2^12 ulps (the
// integer in the low bits of a float of 1.5 x 2^23) added to y's bits.  Below a
// mantissa of 1.0 an ulp is half of one; no seed is closer to 2.0 than its e.
template <int EIGHTHS>
__device__ __forceinline__ double scaled_seed(double y, double e) {
  constexpr float kUnit = 0.125f * EIGHTHS * 1099511627776.0f;   // in 2^12 ulps of [1, 2)
  const unsigned my = ((unsigned)__double2hiint(y) << 3 & 0x007fffffu) | 0x3f800000u;
  const float up = __uint_as_float(my) * kUnit, down = my == 0x3f800000u ? 2.0f * kUnit : up;
  const int he = __double2hiint(e);
  const unsigned mag = max((unsigned)he & 0x7fffffffu, 0x3c100000u);
  const float step = fmaf(__uint_as_float((mag << 3) - (896u << 23)), he < 0 ? -down : up, 12582912.0f);
  return __longlong_as_double(__double_as_longlong(y) + (long long)(__float_as_int(step) - 0x4b400000) * 4096);
}
// y (1 + (EIGHTHS / 8) e^2), y normal, |e| < 1e-4, half an ulp from rounding: the
// last term, formed in FP32, as a number of ulps (a step into the next
// binade, one in 10^12, is off by at most the step)
template <int EIGHTHS>
__device__ __forceinline__ double plus_square(double y, double e) {
  const unsigned he = (unsigned)__double2hiint(e) & 0x7fffffffu;
  // |e| and y's mantissa in [1, 2), cut to FP32 (|e| to 0 below 2^-62: its square is below an ulp)
  const float ef = he < 0x3c100000u ? 0.0f : __uint_as_float((he << 3) - (896u << 23));
  const float my = __uint_as_float(((unsigned)__double2hiint(y) << 3 & 0x007fffffu) | 0x3f800000u);
  const int ulps = __float2int_rn(ef * ef * (my * (0.125f * EIGHTHS * 4503599627370496.0f)));
  return __longlong_as_double(__double_as_longlong(y) + ulps);
}
__device__ __forceinline__ double half_(double x) {   // normal x
  return __hiloint2double(__double2hiint(x) - 0x00100000, __double2loint(x));
}
#endif
__host__ __device__ __forceinline__ double qrcp_(double x) {
#ifdef __CUDA_ARCH__
  if (!f64_plain(x)) return 1.0 / x;
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
  const double e = fma(-x, r, 1.0);
  return fma(scaled_seed<8>(r, e), e, r);
#else
  return 1.0 / x;
#endif
}
__host__ __device__ __forceinline__ double qrsqrt_(double x) {
#ifdef __CUDA_ARCH__
  if (!f64_plain(x) || __double2hiint(x) < 0) return 1.0 / sqrt(x);
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double e = fma(-(x * y), y, 1.0);
  return fma(scaled_seed<6>(half_(y), e), e, y);
#else
  return 1.0 / sqrt(x);
#endif
}
__host__ __device__ __forceinline__ double qroot_(double x) {
#ifdef __CUDA_ARCH__
  if (!f64_plain(x) || __double2hiint(x) < 0) return sqrt(x);
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double t = x * y, e = fma(-t, y, 1.0);
  return fma(half_(t), e, plus_square<3>(t, e));
#else
  return sqrt(x);
#endif
}
__host__ __device__ __forceinline__ float rcp_(float x) { return 1.0f / x; }
__host__ __device__ __forceinline__ float rrsqrt_(float x) { return rsqrtf(x); }
__host__ __device__ __forceinline__ float rsqrt_(float x) { return sqrtf(x); }
__host__ __device__ __forceinline__ float qrcp_(float x) { return 1.0f / x; }
__host__ __device__ __forceinline__ float qrsqrt_(float x) { return rsqrtf(x); }
__host__ __device__ __forceinline__ float qroot_(float x) { return sqrtf(x); }

// Sign-bit helpers (integer operations: they keep the sign tests of the
// limiter off the FP64 pipe).
__host__ __device__ __forceinline__ bool opposite_signs(double a, double b) {
#ifdef __CUDA_ARCH__
  return (__double2hiint(a) ^ __double2hiint(b)) < 0;
#else
  return (a < 0.0) != (b < 0.0) && a != 0.0 && b != 0.0;
#endif
}
__host__ __device__ __forceinline__ bool opposite_signs(float a, float b) {
#ifdef __CUDA_ARCH__
  return (__float_as_int(a) ^ __float_as_int(b)) < 0;
#else
  return (a < 0.0f) != (b < 0.0f) && a != 0.0f && b != 0.0f;
#endif
}
// x with its sign flipped where f is set (on the integer pipe in FP64)
__host__ __device__ __forceinline__ double flip_(double x, bool f) {
#ifdef __CUDA_ARCH__
  return __hiloint2double(__double2hiint(x) ^ (f ? (int)0x80000000 : 0), __double2loint(x));
#else
  return f ? -x : x;
#endif
}

__host__ __device__ __forceinline__ double copysign_(double m, double s) { return copysign(m, s); }
__host__ __device__ __forceinline__ float copysign_(float m, float s) { return copysignf(m, s); }
__host__ __device__ __forceinline__ double fmin_(double a, double b) {
#ifdef __CUDA_ARCH__
  return rmin(a, b);
#else
  return fmin(a, b);
#endif
}
__host__ __device__ __forceinline__ float fmin_(float a, float b) { return fminf(a, b); }

// A quarter of a non-negative value.  FP64 on the device: two off the
// exponent, on the integer pipe (a multiplication would take a slot of the
// FP64 pipe); zero, the smallest exponents, infinity and NaN multiply.
__host__ __device__ __forceinline__ float quarter_(float x) { return 0.25f * x; }
__host__ __device__ __forceinline__ double quarter_(double x) {
#ifdef __CUDA_ARCH__
  const unsigned hi = (unsigned)__double2hiint(x);
  if (hi - 0x00300000u < 0x7ff00000u - 0x00300000u) return __hiloint2double((int)(hi - 0x00200000u), __double2loint(x));
  return (hi | (unsigned)__double2loint(x)) == 0u ? x : 0.25 * x;
#else
  return 0.25 * x;
#endif
}

// Half of the MC-limited slope of the middle of three values (a face takes
// the cell value plus or minus it): with dm = q0 - qm and dp = qp - q0, the MC
// slope is sign(dp) min(2|dm|, 2|dp|, |dm+dp|/2) when dm and dp have the same
// sign, else 0, and its half is sign(dp) min(|dm|, |dp|, |dm+dp|/4) -- the
// same value exactly, since scaling by powers of two is exact.  A zero
// difference makes the minimum zero, so only opposite signs need a test
// (which differs from testing dm dp > 0 only when that product would
// underflow).
template <typename R>
__host__ __device__ __forceinline__ R mc_lim_half(R dm, R dp) {
  R m = fmin_(fmin_(rabs(dm), rabs(dp)), quarter_(rabs(dm + dp)));
  m = opposite_signs(dm, dp) ? R(0) : m;
  return copysign_(m, dp);
}
template <typename R>
__host__ __device__ __forceinline__ R mc_half_slope(R qm, R q0, R qp) {
  return mc_lim_half(q0 - qm, qp - q0);
}

// Fast magnetosonic speed along the normal; w = (rho, vn, vt1, vt2, p, Bt1,
// Bt2); rinv = 1/rho.
template <typename R>
__host__ __device__ __forceinline__ R fast_speed_r(const R* w, R bn, R gamma, R rinv) {
  R a2 = gamma * w[4] * rinv;
  R b2 = (bn * bn + w[5] * w[5] + w[6] * w[6]) * rinv;
  R s = a2 + b2;
  R disc = s * s - R(4) * a2 * bn * bn * rinv;
  disc = gt0(disc) ? disc : R(0);
  return rsqrt_(R(0.5) * (s + rsqrt_(disc)));
}

template <typename R>
__host__ __device__ __forceinline__ R fast_speed(const R* w, R bn, R gamma) {
  return fast_speed_r(w, bn, gamma, rcp_(w[0]));
}

// Fast speeds of both states of a face from one reciprocal of rho_L rho_R.
template <typename R>
__host__ __device__ __forceinline__ void fast_speeds(const R* wl, const R* wr, R bn, R gamma, R& cl, R& cr) {
  const R r = rcp_(wl[0] * wr[0]);
  cl = fast_speed_r(wl, bn, gamma, wr[0] * r);
  cr = fast_speed_r(wr, bn, gamma, wl[0] * r);
}

// Physical flux along the normal (7 components, rotated order); igm1 is
// 1/(gamma - 1), taken once per solve so the energy needs no division.
template <typename R>
__host__ __device__ __forceinline__ void phys_flux_i(const R* w, R bn, R igm1, R* f) {
  R rho = w[0], u = w[1], v = w[2], ww = w[3], p = w[4], by = w[5], bz = w[6];
  R b2 = bn * bn + by * by + bz * bz;
  R pt = p + R(0.5) * b2;
  R e = p * igm1 + R(0.5) * rho * (u * u + v * v + ww * ww) + R(0.5) * b2;
  R vb = u * bn + v * by + ww * bz;
  R mu = rho * u;
  f[0] = mu;
  f[1] = mu * u + pt - bn * bn;
  f[2] = mu * v - bn * by;
  f[3] = mu * ww - bn * bz;
  f[4] = (e + pt) * u - bn * vb;
  f[5] = u * by - v * bn;
  f[6] = u * bz - ww * bn;
}

template <typename R>
__host__ __device__ __forceinline__ void phys_flux(const R* w, R bn, R gamma, R* f) {
  phys_flux_i(w, bn, R(1) / (gamma - R(1)), f);
}

template <typename R>
__host__ __device__ __forceinline__ R total_energy_i(const R* w, R bn, R igm1) {
  return w[4] * igm1 + R(0.5) * w[0] * (w[1] * w[1] + w[2] * w[2] + w[3] * w[3]) +
         R(0.5) * (bn * bn + w[5] * w[5] + w[6] * w[6]);
}

// HLL flux; ig = 1/(gamma - 1).
template <typename R>
__host__ __device__ __forceinline__ void hll_flux_g(const R* wl, const R* wr, R bn, R gamma, R ig, R* f,
                                                    R* cmax = nullptr) {
  R cl, cr;
  fast_speeds(wl, wr, bn, gamma, cl, cr);
  R cm = rmax(cl, cr);
  if (cmax) *cmax = cm;
  R sl = rmin(wl[1], wr[1]) - cm;
  R sr = rmax(wl[1], wr[1]) + cm;
  if (ge0(sl)) { phys_flux_i(wl, bn, ig, f); return; }
  if (le0(sr)) { phys_flux_i(wr, bn, ig, f); return; }
  R fl[7], fr[7];
  phys_flux_i(wl, bn, ig, fl);
  phys_flux_i(wr, bn, ig, fr);
  R ul[7] = {wl[0], wl[0] * wl[1], wl[0] * wl[2], wl[0] * wl[3], total_energy_i(wl, bn, ig), wl[5], wl[6]};
  R ur[7] = {wr[0], wr[0] * wr[1], wr[0] * wr[2], wr[0] * wr[3], total_energy_i(wr, bn, ig), wr[5], wr[6]};
  R inv = rcp_(sr - sl);
#pragma unroll
  for (int q = 0; q < 7; ++q) f[q] = (sr * fl[q] - sl * fr[q] + sl * sr * (ur[q] - ul[q])) * inv;
}

template <typename R>
__host__ __device__ __forceinline__ void hll_flux(const R* wl, const R* wr, R bn, R gamma, R* f, R* cmax = nullptr) {
  hll_flux_g(wl, wr, bn, gamma, R(1) / (gamma - R(1)), f, cmax);
}

// Star state of one side (Miyoshi & Kusano eqs. 43-48), with the outer
// state's total energy, total pressure and v.B (its flux reuses them).
template <typename R>
struct Star {
  R rho, v, w, by, bz, e, vb, sq, isq;   // sq = sqrt(rho*), isq = 1/sqrt(rho*)
  R eo, pto, vbo;
};


template <typename R>
__host__ __device__ __forceinline__ Star<R> star_side(const R* w, R bn, R igm1, R pt, R s, R sm, R pts) {
  Star<R> st;
  R rho = w[0], u = w[1], v = w[2], ww = w[3], by = w[5], bz = w[6];
  R sd = s - u;
  R ssm = s - sm;
  R num = rho * sd * ssm;
  R bn2 = bn * bn;
  R den = num - bn2;
  R scale = rmax(rabs(num), bn2);
  R inv_ssm;
  if (le_(rabs(den), Eps<R>::degen * scale)) {
    inv_ssm = rcp_(ssm);
    st.v = v; st.w = ww; st.by = by; st.bz = bz;
  } else {
    // 1/(S - S_M) and 1/den from one reciprocal of their product
    const R r = rcp_(ssm * den);
    inv_ssm = den * r;
    R iden = ssm * r;
    R c1 = bn * (sm - u) * iden;
    R c2 = (rho * sd * sd - bn2) * iden;
    st.v = v - by * c1;
    st.w = ww - bz * c1;
    st.by = by * c2;
    st.bz = bz * c2;
  }
  st.rho = rho * sd * inv_ssm;
  R vb = u * bn + v * by + ww * bz;
  st.vb = sm * bn + st.v * st.by + st.w * st.bz;
  R e = total_energy_i(w, bn, igm1);
  st.e = (sd * e - pt * u + pts * sm + bn * (vb - st.vb)) * inv_ssm;
  st.eo = e;
  st.pto = pt;
  st.vbo = vb;
  st.isq = rrsqrt_(st.rho);
  st.sq = st.rho * st.isq;
  return st;
}

// HLLD flux.  Ties at exactly zero take the first region in the order
// L, L*, L**, R**, R*, R; sign(0) = 0; degenerate star states (den ~ 0)
// keep the outer tangential values.
template <typename R>
__host__ __device__ __forceinline__ void hlld_flux_g(const R* wl, const R* wr, R bn, R gamma, R ig, R* f,
                                                     R* cmax = nullptr) {
  R cl, cr;
  fast_speeds(wl, wr, bn, gamma, cl, cr);
  R cm = rmax(cl, cr);
  if (cmax) *cmax = cm;
  R sl = rmin(wl[1], wr[1]) - cm;
  R sr = rmax(wl[1], wr[1]) + cm;
  if (gt0(sl)) { phys_flux_i(wl, bn, ig, f); return; }
  if (lt0(sr)) { phys_flux_i(wr, bn, ig, f); return; }
  R ptl = wl[4] + R(0.5) * (bn * bn + wl[5] * wl[5] + wl[6] * wl[6]);
  R ptr = wr[4] + R(0.5) * (bn * bn + wr[5] * wr[5] + wr[6] * wr[6]);
  R sdl = sl - wl[1], sdr = sr - wr[1];
  R sm = (sdr * wr[0] * wr[1] - sdl * wl[0] * wl[1] - ptr + ptl) * rcp_(sdr * wr[0] - sdl * wl[0]);
  R pts = ptl + wl[0] * sdl * (sm - wl[1]);
  Star<R> L = star_side(wl, bn, ig, ptl, sl, sm, pts);
  Star<R> Rr = star_side(wr, bn, ig, ptr, sr, sm, pts);
  R abn = rabs(bn);
  R ssl = sm - abn * L.isq;
  R ssr = sm + abn * Rr.isq;
  const bool left = ge0(sm);
  const R* w = left ? wl : wr;
  const Star<R>& S = left ? L : Rr;
  R so = left ? sl : sr;
  bool dbl = left ? lt0(ssl) : ge0(ssr);
  // the outer state's flux and conserved values, from the energy, total
  // pressure and v.B its star side already formed
  R fo[7];
  {
    const R mu = w[0] * w[1];
    fo[0] = mu;
    fo[1] = mu * w[1] + S.pto - bn * bn;
    fo[2] = mu * w[2] - bn * w[5];
    fo[3] = mu * w[3] - bn * w[6];
    fo[4] = (S.eo + S.pto) * w[1] - bn * S.vbo;
    fo[5] = w[1] * w[5] - w[2] * bn;
    fo[6] = w[1] * w[6] - w[3] * bn;
  }
  R uo[7] = {w[0], w[0] * w[1], w[0] * w[2], w[0] * w[3], S.eo, w[5], w[6]};
  R us[7] = {S.rho, S.rho * sm, S.rho * S.v, S.rho * S.w, S.e, S.by, S.bz};
#pragma unroll
  for (int q = 0; q < 7; ++q) f[q] = fo[q] + so * (us[q] - uo[q]);
  if (dbl) {
    R sgn = gt0(bn) ? R(1) : (lt0(bn) ? R(-1) : R(0));
    R isq = rcp_(L.sq + Rr.sq);
    R vss = (L.sq * L.v + Rr.sq * Rr.v + (Rr.by - L.by) * sgn) * isq;
    R wss = (L.sq * L.w + Rr.sq * Rr.w + (Rr.bz - L.bz) * sgn) * isq;
    R byss = (L.sq * Rr.by + Rr.sq * L.by + L.sq * Rr.sq * (Rr.v - L.v) * sgn) * isq;
    R bzss = (L.sq * Rr.bz + Rr.sq * L.bz + L.sq * Rr.sq * (Rr.w - L.w) * sgn) * isq;
    R vbss = sm * bn + vss * byss + wss * bzss;
    R ess = left ? S.e - S.sq * (S.vb - vbss) * sgn : S.e + S.sq * (S.vb - vbss) * sgn;
    R sso = left ? ssl : ssr;
    R uss[7] = {S.rho, S.rho * sm, S.rho * vss, S.rho * wss, ess, byss, bzss};
#pragma unroll
    for (int q = 0; q < 7; ++q) f[q] += sso * (uss[q] - us[q]);
  }
}

template <typename R>
__host__ __device__ __forceinline__ void hlld_flux(const R* wl, const R* wr, R bn, R gamma, R* f, R* cmax = nullptr) {
  hlld_flux_g(wl, wr, bn, gamma, R(1) / (gamma - R(1)), f, cmax);
}

// ---------------------------------------------------------------------------
// The same two solvers with fewer operations: the forms of the FP64 kernels,
// which are bound by the FP64 pipe (one warp-instruction per ~17 SM cycles,
// the other pipes nearly idle).  They equal the forms above up to rounding,
// times the conditioning of the star states.  FP32 fluxes keep the forms above:
// a change of FP32 rounding flips limiter and upwind choices here and there,
// which moves single cells by 1e-3.  As written, an HLLD solution takes 59
// additions and 85 multiplications instead of 107 and 169 (mean of random
// faces, fused ones counted apart; HLL 66 and 93 instead of 80 and 142), and
// fewer roots and reciprocals, by these identities:
//   * c_f^2 = T / (2 rho), T = gamma p + |B|^2 + sqrt((gamma p - |B|^2)^2 + 4 gamma p |B_t|^2):
//     the larger of two fast speeds is found by comparing T_L rho_R with
//     T_R rho_L, and one division and one outer root serve both states;
//   * the flux of every region has the form of the physical flux of that
//     region's state with its total pressure, so one evaluation on the
//     selected state replaces F + S (U* - U) + S* (U** - U*);
//   * rho* and sqrt(rho*) follow from one reciprocal root y of
//     m (S - S_M), m = rho (S - u): sqrt(rho*) = |m| y, 1/sqrt(rho*) = |S - S_M| y;
//   * across an Alfven wave v** - v* = +-sgn(bn) (B** - B*)/sqrt(rho*);
//   * only the side of S_M that holds the face forms its energy, and the
//     other side's star state is formed only where a double-star state needs it.
// Measured (GB300, 128^3, stage 1 / 2 in us): HLLD 6389 / 6480 with the plain
// solvers, 4619 / 4717 with these; HLL 4837 / 4901 and 4286 / 4355.

// The larger fast speed of two states, b2_* = |B|^2 and bt2_* = |B_t|^2 of each.
__host__ __device__ __forceinline__ double max_fast_speed(const double* wl, const double* wr, double b2_l, double b2_r,
                                                          double bt2_l, double bt2_r, double gamma) {
  const double g4 = 4.0 * gamma;
  const double x_l = gamma * wl[4] - b2_l, x_r = gamma * wr[4] - b2_r;
  const double t_l = gamma * wl[4] + b2_l + qroot_(x_l * x_l + (g4 * wl[4]) * bt2_l);
  const double t_r = gamma * wr[4] + b2_r + qroot_(x_r * x_r + (g4 * wr[4]) * bt2_r);
  const bool l = lt_(t_r * wl[0], t_l * wr[0]);
  const double t = l ? t_l : t_r, rho = l ? wl[0] : wr[0];
  // sqrt(t / (2 rho)) = t / sqrt(2 rho t)
  return t * (0.70710678118654752440 * qrsqrt_(rho * t));
}

// Whether a star state's denominator den = num - bn^2 counts as zero:
// |den| <= eps max(|num|, bn^2), as in star_side.  On the device, where
// the exponents already put |den| above 2^-38 bn^2, and so (|num| <= |den| +
// bn^2) above 1e-12 of both, no FP64 operation is needed.
__host__ __device__ __forceinline__ bool star_degenerate(double den, double num, double bn2) {
#ifdef __CUDA_ARCH__
  const unsigned hd = (unsigned)__double2hiint(den) & 0x7fffffffu, hb = (unsigned)__double2hiint(bn2);
  if (hd + (37u << 20) > hb) return false;
#endif
  return le_(rabs(den), Eps<double>::degen * rmax(rabs(num), bn2));
}

// Star state of one side as the lean solver needs it: m = rho (S - u), ssm =
// S - S_M, smu = S_M - u.
struct LeanStar {
  double v, w, by, bz, sq, isq, y;   // sq = sqrt(rho*), isq = 1/sqrt(rho*), y = 1/sqrt(m ssm)
  bool degen;
};
__host__ __device__ __forceinline__ LeanStar lean_star(double v, double w, double by, double bz, double bn, double bn2,
                                                       double m, double ssm, double smu) {
  LeanStar st;
  const double num = m * ssm, den = num - bn2;
  st.degen = star_degenerate(den, num, bn2);
  const double t = smu * qrcp_(den);
  const double c1 = st.degen ? 0.0 : bn * t;          // v* = v - B_t c1
  const double c2 = st.degen ? 1.0 : 1.0 + m * t;    // B_t* = B_t c2, c2 = (m (S - u) - bn^2) / den
  st.v = v - by * c1;
  st.w = w - bz * c1;
  st.by = by * c2;
  st.bz = bz * c2;
  st.y = qrsqrt_(num);
  st.sq = rabs(m) * st.y;
  st.isq = rabs(ssm) * st.y;
  return st;
}

// Flux of the state (rho, u, v, w, energy e, total pressure pt, transverse
// field by, bz, vb = v.B).
__host__ __device__ __forceinline__ void state_flux(double rho, double u, double v, double w, double e, double pt,
                                                    double by, double bz, double vb, double bn, double bn2, double* f) {
  const double mu = rho * u;
  f[0] = mu;
  f[1] = mu * u + (pt - bn2);
  f[2] = mu * v - bn * by;
  f[3] = mu * w - bn * bz;
  f[4] = (e + pt) * u - bn * vb;
  f[5] = u * by - bn * v;
  f[6] = u * bz - bn * w;
}

// Conserved hydro values and flux of one outer state.
__host__ __device__ __forceinline__ void lean_side(const double* w, double bn, double bn2, double b2, double ig,
                                                   double* u, double* f) {
  const double e = w[4] * ig + 0.5 * (w[0] * (w[1] * w[1] + w[2] * w[2] + w[3] * w[3]) + b2);
  const double vb = w[1] * bn + w[2] * w[5] + w[3] * w[6];
  state_flux(w[0], w[1], w[2], w[3], e, w[4] + 0.5 * b2, w[5], w[6], vb, bn, bn2, f);
  u[0] = w[0];
  u[1] = f[0];
  u[2] = w[0] * w[2];
  u[3] = w[0] * w[3];
  u[4] = e;
}

// HLLD flux; ig = 1/(gamma - 1).  Regions, ties and the degenerate star state
// as hlld_flux_g: a degenerate side keeps its outer tangential values, and
// its transverse induction flux the outer velocity.
__host__ __device__ __forceinline__ void hlld_flux_lean(const double* wl, const double* wr, double bn, double gamma,
                                                        double ig, double* f, double* cmax) {
  const double bn2 = bn * bn;
  const double bt2l = wl[5] * wl[5] + wl[6] * wl[6], bt2r = wr[5] * wr[5] + wr[6] * wr[6];
  const double b2l = bn2 + bt2l, b2r = bn2 + bt2r;
  const double ptl = wl[4] + 0.5 * b2l, ptr = wr[4] + 0.5 * b2r;
  const double cm = max_fast_speed(wl, wr, b2l, b2r, bt2l, bt2r, gamma);
  *cmax = cm;
  const double sl = rmin(wl[1], wr[1]) - cm, sr = rmax(wl[1], wr[1]) + cm;
  const bool out_l = gt0(sl), outside = out_l || lt0(sr);
  // the outer sides' S - u, m = rho (S - u) and the contact speed S_M
  const double sdl = sl - wl[1], sdr = sr - wr[1];
  const double ml = wl[0] * sdl, mr = wr[0] * sdr;
  const double sm = ((ptl - ptr) + mr * wr[1] - ml * wl[1]) * qrcp_(mr - ml);
  const bool left = outside ? out_l : ge0(sm);
  // A: the side that holds the face, B: the other one
  const double rho = left ? wl[0] : wr[0], u = left ? wl[1] : wr[1], p = left ? wl[4] : wr[4];
  const double va = left ? wl[2] : wr[2], wa = left ? wl[3] : wr[3];
  const double bya = left ? wl[5] : wr[5], bza = left ? wl[6] : wr[6];
  const double b2 = left ? b2l : b2r, pta = left ? ptl : ptr;
  const double vb = u * bn + va * bya + wa * bza;
  const double e = p * ig + 0.5 * (rho * (u * u + va * va + wa * wa) + b2);
  // the state whose flux this is
  double fr = rho, fu = u, fv = va, fw = wa, fby = bya, fbz = bza, fe = e, fvb = vb, fpt = pta;
  double smu = 0.0;
  bool degen = false;
  if (!outside) {
    const double s = left ? sl : sr, m = left ? ml : mr, sd = left ? sdl : sdr;
    const double ssm = s - sm;
    smu = sm - u;
    const LeanStar A = lean_star(va, wa, bya, bza, bn, bn2, m, ssm, smu);
    degen = A.degen;
    const double inv = A.y * A.y * m;   // 1 / (S - S_M)
    fpt = pta + m * smu;
    fr = m * inv;
    fu = sm;
    const double smbn = sm * bn;
    fvb = smbn + A.v * A.by + A.w * A.bz;
    fe = (sd * e - pta * u + fpt * sm + bn * (vb - fvb)) * inv;
    fv = A.v;
    fw = A.w;
    fby = A.by;
    fbz = A.bz;
    // beyond the Alfven wave of side A: S*_L < 0 (left), S*_R >= 0 (right)
    const double al = rabs(bn) * A.isq;
    if (left ? lt_(sm, al) : le_(-sm, al)) {
      const double sb = left ? sr : sl;
      const LeanStar B = lean_star(left ? wr[2] : wl[2], left ? wr[3] : wl[3], left ? wr[5] : wl[5],
                                      left ? wr[6] : wl[6], bn, bn2, left ? mr : ml, sb - sm,
                                      sm - (left ? wr[1] : wl[1]));
      const bool neg = lt0(bn) == left;   // sign of sgn(bn) (+ on the left, - on the right)
      const double is = qrcp_(A.sq + B.sq);
      const double ps = flip_(A.sq * B.sq, neg);
      fby = (A.sq * B.by + B.sq * A.by + ps * (B.v - A.v)) * is;
      fbz = (A.sq * B.bz + B.sq * A.bz + ps * (B.w - A.w)) * is;
      const double k = flip_(A.isq, neg);
      fv = A.v + k * (fby - A.by);
      fw = A.w + k * (fbz - A.bz);
      const double vbs = fvb;
      fvb = smbn + fv * fby + fw * fbz;
      fe = fe - flip_(A.sq, neg) * (vbs - fvb);
    }
  }
  state_flux(fr, fu, fv, fw, fe, fpt, fby, fbz, fvb, bn, bn2, f);
  if (degen) {   // outside the star region degen is false
    f[5] -= smu * bya;
    f[6] -= smu * bza;
  }
}

// HLL flux a F_L + b F_R + c (U_R - U_L) with the three weights formed once.
__host__ __device__ __forceinline__ void hll_flux_lean(const double* wl, const double* wr, double bn, double gamma,
                                                       double ig, double* f, double* cmax) {
  const double bn2 = bn * bn;
  const double bt2l = wl[5] * wl[5] + wl[6] * wl[6], bt2r = wr[5] * wr[5] + wr[6] * wr[6];
  const double b2l = bn2 + bt2l, b2r = bn2 + bt2r;
  const double cm = max_fast_speed(wl, wr, b2l, b2r, bt2l, bt2r, gamma);
  *cmax = cm;
  const double sl = rmin(wl[1], wr[1]) - cm, sr = rmax(wl[1], wr[1]) + cm;
  const double is = qrcp_(sr - sl);
  double a = sr * is, b = -(sl * is), c = sl * a;
  if (ge0(sl)) { a = 1.0; b = c = 0.0; }   // outside the fan: one side's flux
  else if (le0(sr)) { b = 1.0; a = c = 0.0; }
  double ul[5], ur[5], fl[7], fr[7];
  lean_side(wl, bn, bn2, b2l, ig, ul, fl);
  lean_side(wr, bn, bn2, b2r, ig, ur, fr);
#pragma unroll
  for (int q = 0; q < 7; ++q) {
    const double du = q < 5 ? ur[q] - ul[q] : wr[q] - wl[q];
    f[q] = a * fl[q] + (b * fr[q] + c * du);
  }
}

// Mass flux that orients the upwind EMF average: the face mass flux, or 0
// when it lies inside a rounding deadband eps (rho_L + rho_R)/2 c_max, so
// rounding noise of a vanishing mass flux selects the mean of both sides
// instead of an arbitrary side.
// FP64 on the device: where the exponents already put |f0| above the band
// (eps (rho_L + rho_R)/2 c_max < 2^(sum of the exponents + 3)), no FP64
// operation is needed.
template <typename R>
__host__ __device__ __forceinline__ R oriented_mass_flux(R f0, R rho_l, R rho_r, R cmax, R eps) {
#ifdef __CUDA_ARCH__
  if constexpr (sizeof(R) == 8) {
    const int er = max(__double2hiint((double)rho_l), __double2hiint((double)rho_r));
    const int ec = __double2hiint((double)cmax) >> 20, ee = __double2hiint((double)eps) >> 20;
    const int band = (er >> 20) + ec + ee - 2 * 1023 + 3;
    if (((__double2hiint((double)f0) & 0x7fffffff) >> 20) > band) return f0;
  }
#endif
  return le_(rabs(f0), eps * R(0.5) * (rho_l + rho_r) * cmax) ? R(0) : f0;
}

// Gardiner-Stone upwind selection by the sign of a face mass flux: the
// difference lo_a - lo_b of one side, hi_a - hi_b of the other, or their mean.
template <typename R>
__host__ __device__ __forceinline__ R upwind(R m, R lo_a, R lo_b, R hi_a, R hi_b) {
  const R lo = lo_a - lo_b, hi = hi_a - hi_b;
  return gt0(m) ? lo : (lt0(m) ? hi : R(0.5) * (lo + hi));
}
// The same for a mass flux that is not zero: select, then one difference.
template <typename R>
__host__ __device__ __forceinline__ R upwind_nz(R m, R lo_a, R lo_b, R hi_a, R hi_b) {
  const bool up = gt0(m);
  return (up ? lo_a : hi_a) - (up ? lo_b : hi_b);
}

// Edge EMF along c at the corner of the (a, b) plane (c, a, b cyclic), from
// the two a-face EMFs (fa_m at b-1, fa_p at b), the two b-face EMFs (fb_m at
// a-1, fb_p at a), the face mass fluxes, and the four cell-centred values
// e_mm (a-1,b-1), e_pm (a,b-1), e_mp (a-1,b), e_pp (a,b).  A mass flux of
// exactly zero is rare (rest, or inside the deadband), so FP64 forms the mean
// it asks for only where one of the four is: four differences instead of
// eight and no means, half of an edge's FP64 operations (128^3, stage 1 / 2:
// 4619 / 4717 us, without the branch 4759 / 4851).  FP32, where the selections
// cost as much as the differences they save, forms them all (256^3 mixed: 2386 /
// 2583 us, with the branch 2418 / 2604).  The values are the same either way.
template <typename R>
__host__ __device__ __forceinline__ R edge_emf(R fa_m, R fa_p, R ma_m, R ma_p, R fb_m, R fb_p, R mb_m, R mb_p,
                                      R e_mm, R e_pm, R e_mp, R e_pp, bool plain_mean) {
  R avg = R(0.25) * (fa_m + fa_p + fb_m + fb_p);
  if (plain_mean) return avg;
  R db_plus, db_minus, da_plus, da_minus;
  if (sizeof(R) == 8 && (gt0(ma_p) || lt0(ma_p)) && (gt0(ma_m) || lt0(ma_m)) &&
      (gt0(mb_p) || lt0(mb_p)) && (gt0(mb_m) || lt0(mb_m))) {
    db_plus = upwind_nz(ma_p, e_mp, fb_m, e_pp, fb_p);
    db_minus = upwind_nz(ma_m, fb_m, e_mm, fb_p, e_pm);
    da_plus = upwind_nz(mb_p, e_pm, fa_m, e_pp, fa_p);
    da_minus = upwind_nz(mb_m, fa_m, e_mm, fa_p, e_mp);
  } else {
    db_plus = upwind(ma_p, e_mp, fb_m, e_pp, fb_p);
    db_minus = upwind(ma_m, fb_m, e_mm, fb_p, e_pm);
    da_plus = upwind(mb_p, e_pm, fa_m, e_pp, fa_p);
    da_minus = upwind(mb_m, fa_m, e_mm, fa_p, e_mp);
  }
  return avg + R(0.25) * (db_minus - db_plus) + R(0.25) * (da_minus - da_plus);
}

// Half of the characteristic MC slope of the middle cell w0 of (wm, w0, wp), rotated
// primitives (rho, v_n, v_t1, v_t2, p, B_t1, B_t2), bn0 the middle cell's
// cell-centred normal field.  The one-sided differences are projected on the
// left eigenvectors of the primitive Jacobian at w0, limited wave by wave and
// projected back with the right eigenvectors (Roe & Balsara 1996
// normalisation: alpha_f, alpha_s, beta = B_t/|B_t|, sgn(bn) = 1 for bn >= 0;
// alpha_f = 1 when c_f = c_s and beta = (1, 1)/sqrt 2 when |B_t| vanishes,
// both to the precision's degeneracy tolerance).  Each +/- wave pair shares
// an even and an odd part of its projection, which the code forms once.
template <typename R>
__host__ __device__ __forceinline__ void char_half_slope(const R* wm, const R* w0, const R* wp, R bn0, R gamma,
                                                    R* slope) {
  const R rho = w0[0];
  const R ir = rcp_(rho);
  const R a2 = gamma * w0[4] * ir, a = rsqrt_(a2), sr = rsqrt_(rho), isr = rcp_(sr);
  const R bnr = bn0 * isr, b1 = w0[5] * isr, b2 = w0[6] * isr;
  const R bt2 = b1 * b1 + b2 * b2, bsq = bnr * bnr + bt2;
  // forms without cancellation: c_f^2 - c_s^2 = sqrt((a^2-b^2)^2 + 4 a^2 b_t^2),
  // c_s^2 = a^2 b_n^2 / c_f^2, and below c_f^2 - a^2, a^2 - c_s^2 as half-sums
  // with that root (alpha_s is otherwise the root of a rounding residue when
  // B_t vanishes)
  // IEEE square root here: sqrt(fl(d*d)) = |d| exactly when B_t = 0, which
  // makes c_f^2 - a^2 or a^2 - c_s^2 below exactly zero (a root with a few
  // ulp of error would leave a residue whose square root is ~1e-8)
  const R sq = sqrt((a2 - bsq) * (a2 - bsq) + R(4) * a2 * bt2);
  const R cf2 = R(0.5) * (a2 + bsq + sq);
  const R cs2 = gt0(cf2) ? a2 * bnr * bnr * rcp_(cf2) : R(0);
  const R cf = rsqrt_(cf2), cs = rsqrt_(cs2), bt = rsqrt_(bt2);
  R be1, be2;
  if (lt_(Eps<R>::degen * rsqrt_(a2 + bsq), bt)) {
    const R ib = rcp_(bt);
    be1 = b1 * ib;
    be2 = b2 * ib;
  } else {
    be1 = be2 = R(0.70710678118654752440);
  }
  R af, as;
  if (lt_(Eps<R>::degen * cf2, sq)) {
    const R id = rcp_(sq);
    const R fa = R(0.5) * (bsq - a2 + sq), as2 = R(0.5) * (a2 - bsq + sq);   // c_f^2 - a^2, a^2 - c_s^2
    af = rsqrt_((gt0(as2) ? as2 : R(0)) * id);
    as = rsqrt_((gt0(fa) ? fa : R(0)) * id);
  } else {
    af = R(1);
    as = R(0);
  }
  const R sg = ge0(bn0) ? R(1) : R(-1);
  const R ia2 = rcp_(a2);
  const R i2a2 = R(0.5) * ia2, i2r = i2a2 * ir, i2sa = R(0.5) * isr * rcp_(a), i2s = R(0.5) * isr;
  R dc[7];   // limited wave amplitudes: f-, a-, s-, e, s+, a+, f+
  {
    R m[7], q[7];
    const R* pairs[2][2] = {{wm, w0}, {w0, wp}};
#pragma unroll
    for (int side = 0; side < 2; ++side) {
      R d[7];
#pragma unroll
      for (int v = 0; v < 7; ++v) d[v] = pairs[side][1][v] - pairs[side][0][v];
      const R t = be1 * d[2] + be2 * d[3], bb = be1 * d[5] + be2 * d[6];
      const R xf = (af * cf * d[1] - as * cs * sg * t) * i2a2, yf = af * d[4] * i2r + as * bb * i2sa;
      const R xs = (as * cs * d[1] + af * cf * sg * t) * i2a2, ys = as * d[4] * i2r - af * bb * i2sa;
      const R xa = R(0.5) * sg * (be2 * d[2] - be1 * d[3]), ya = (be1 * d[6] - be2 * d[5]) * i2s;
      R* c = side == 0 ? m : q;
      c[0] = yf - xf;
      c[1] = ya - xa;
      c[2] = ys - xs;
      c[3] = d[0] - d[4] * ia2;
      c[4] = ys + xs;
      c[5] = ya + xa;
      c[6] = yf + xf;
    }
#pragma unroll
    for (int k = 0; k < 7; ++k) dc[k] = mc_lim_half(m[k], q[k]);
  }
  const R Fp = dc[6] + dc[0], Fm = dc[6] - dc[0];
  const R Sp = dc[4] + dc[2], Sm = dc[4] - dc[2];
  const R Ap = dc[5] + dc[1], Am = dc[5] - dc[1];
  slope[0] = rho * (af * Fp + as * Sp) + dc[3];
  slope[1] = af * cf * Fm + as * cs * Sm;
  const R tv = af * cf * Sm - as * cs * Fm;
  slope[2] = sg * (be1 * tv + be2 * Am);
  slope[3] = sg * (be2 * tv - be1 * Am);
  slope[4] = rho * a2 * (af * Fp + as * Sp);
  const R tb = a * sr * (as * Fp - af * Sp);
  slope[5] = be1 * tb - sr * be2 * Ap;
  slope[6] = be2 * tb + sr * be1 * Ap;
}

// The same in FP64, with a third fewer operations: reciprocals and roots from
// one reciprocal root each, the projection's coefficients formed once for both
// sides, and of c_f^2 - a^2 and a^2 - c_s^2 the smaller one from their product
// a^2 b_t^2 (exactly zero when B_t is), so that the root of the discriminant
// needs no correct rounding.  Measured (96x64x80, stage 1 / 2): 1843 / 1837 us,
// with the form above 2136 / 2131.
__host__ __device__ __forceinline__ void char_half_slope(const double* wm, const double* w0, const double* wp, double bn0,
                                                         double gamma, double* slope) {
  const double rho = w0[0], gp = gamma * w0[4];
  const double isr = qrsqrt_(rho), sr = rho * isr, ir = isr * isr;
  const double a2 = gp * ir, ra = qrsqrt_(a2), a = a2 * ra, ia2 = ra * ra;
  const double bnr = bn0 * isr, b1 = w0[5] * isr, b2 = w0[6] * isr;
  const double bt2 = b1 * b1 + b2 * b2, bsq = bnr * bnr + bt2;
  const double d = a2 - bsq, s = a2 + bsq, q = 4.0 * a2 * bt2, disc = d * d + q;
  double be1, be2;
  if (lt_(Eps<double>::degen * Eps<double>::degen * s, bt2)) {
    const double ib = qrsqrt_(bt2);
    be1 = b1 * ib;
    be2 = b2 * ib;
  } else {
    be1 = be2 = 0.70710678118654752440;
  }
  const double iq = gt0(disc) ? qrsqrt_(disc) : 0.0, sq = disc * iq;   // c_f^2 - c_s^2 and its reciprocal
  const double cf2 = 0.5 * (s + sq), icf = qrsqrt_(cf2);
  const double cf = cf2 * icf, cs = a * (rabs(bnr) * icf);
  double af, as;
  if (lt_(Eps<double>::degen * cf2, sq)) {
    const double big = 0.5 * (rabs(d) + sq), small = quarter_(q) * qrcp_(big);
    const bool pos = ge0(d);   // a^2 - c_s^2 is the larger one
    af = qroot_((pos ? big : small) * iq);
    as = qroot_((pos ? small : big) * iq);
  } else {
    af = 1.0;
    as = 0.0;
  }
  const bool neg = lt0(bn0);   // sgn(bn) = -1
  const double fc = af * cf, sc = as * cs, h = 0.5 * ia2, hs = 0.5 * isr, hr = h * ir, ha = hs * ra;
  const double x1 = fc * h, x2 = sc * h, y1 = af * hr, y2 = as * hr, z1 = af * ha, z2 = as * ha;
  const double e1 = flip_(0.5 * be1, neg), e2 = flip_(0.5 * be2, neg), g1 = be1 * hs, g2 = be2 * hs;
  const double x1s = flip_(x1, neg), x2s = flip_(x2, neg);
  double dc[7];   // limited wave amplitudes: f-, a-, s-, e, s+, a+, f+
  {
    double m[7], p[7];
#pragma unroll
    for (int side = 0; side < 2; ++side) {
      const double* lo = side == 0 ? wm : w0;
      const double* hi = side == 0 ? w0 : wp;
      double v[7];
#pragma unroll
      for (int k = 0; k < 7; ++k) v[k] = hi[k] - lo[k];
      const double t = be1 * v[2] + be2 * v[3], bb = be1 * v[5] + be2 * v[6];
      const double xf = x1 * v[1] - x2s * t, yf = y1 * v[4] + z2 * bb;
      const double xs = x2 * v[1] + x1s * t, ys = y2 * v[4] - z1 * bb;
      const double xa = e2 * v[2] - e1 * v[3], ya = g1 * v[6] - g2 * v[5];
      double* c = side == 0 ? m : p;
      c[0] = yf - xf;
      c[1] = ya - xa;
      c[2] = ys - xs;
      c[3] = v[0] - v[4] * ia2;
      c[4] = ys + xs;
      c[5] = ya + xa;
      c[6] = yf + xf;
    }
#pragma unroll
    for (int k = 0; k < 7; ++k) dc[k] = mc_lim_half(m[k], p[k]);
  }
  const double Fp = dc[6] + dc[0], Fm = dc[6] - dc[0];
  const double Sp = dc[4] + dc[2], Sm = dc[4] - dc[2];
  const double Ap = sr * (dc[5] + dc[1]), Am = dc[5] - dc[1];
  const double w = af * Fp + as * Sp;
  slope[0] = rho * w + dc[3];
  slope[1] = fc * Fm + sc * Sm;
  const double tv = fc * Sm - sc * Fm;
  slope[2] = flip_(be1 * tv + be2 * Am, neg);
  slope[3] = flip_(be2 * tv - be1 * Am, neg);
  slope[4] = gp * w;
  const double tb = (a * sr) * (as * Fp - af * Sp);
  slope[5] = be1 * tb - be2 * Ap;
  slope[6] = be2 * tb + be1 * Ap;
}

// Characteristic PLM of a face: as plm_face, with the slopes of c1 and c2
// taken in characteristic variables (bn1, bn2: their cell-centred normal
// fields).
template <typename R>
__host__ __device__ __forceinline__ void plm_face_char(const R* c0, const R* c1, const R* c2, const R* c3, R bn1,
                                                       R bn2, R gamma, R* wl, R* wr, R rho_floor, R p_floor) {
  R sl[7], sr_[7];
  char_half_slope(c0, c1, c2, bn1, gamma, sl);
  char_half_slope(c1, c2, c3, bn2, gamma, sr_);
#pragma unroll
  for (int q = 0; q < 7; ++q) {
    wl[q] = c1[q] + sl[q];
    wr[q] = c2[q] - sr_[q];
  }
  wl[0] = rmax(wl[0], rho_floor);
  wr[0] = rmax(wr[0], rho_floor);
  wl[4] = rmax(wl[4], p_floor);
  wr[4] = rmax(wr[4], p_floor);
}

// Reconstruct the two states of a face from four cells along the normal
// (c0, c1 | c2, c3), 7 rotated primitives each; face values of rho and p are
// floored (MC keeps them between the neighbouring cell values, so the floor
// only absorbs rounding next to a cell that sits at the floor).
template <typename R>
__host__ __device__ __forceinline__ void plm_face(const R* c0, const R* c1, const R* c2, const R* c3, R* wl, R* wr,
                                                  R rho_floor, R p_floor) {
#pragma unroll
  for (int q = 0; q < 7; ++q) {
    wl[q] = c1[q] + mc_half_slope(c0[q], c1[q], c2[q]);
    wr[q] = c2[q] - mc_half_slope(c1[q], c2[q], c3[q]);
  }
  wl[0] = rmax(wl[0], rho_floor);
  wr[0] = rmax(wr[0], rho_floor);
  wl[4] = rmax(wl[4], p_floor);
  wr[4] = rmax(wr[4], p_floor);
}

}  // namespace mhd
