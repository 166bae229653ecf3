// Device building blocks of the stage update: reconstruction from precomputed 1-d geometry
// tables, HLLC, the M1 closure, Planck group integrals and opacities.
//
// All functions are templated on the transport precision R (double for the plain FP64 path,
// float for the FP32 form).  Coupling arithmetic that the FP32 form keeps in FP64 takes double.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>

#include "fx_pair.cuh"
#include "fx_types.h"

namespace fx {

// Reciprocal: IEEE division in FP64; the hardware approximation (1 ulp) in FP32, one instruction
// (a division intrinsic adds range scaling that no caller needs).
__device__ __forceinline__ double frcp(double x) { return 1.0 / x; }
__device__ __forceinline__ float frcp(float x) { return rcp_approx(x); }

// ---------------------------------------------------------------------------------------------
// FP64 operations off the FP64 pipe where the result allows it.  The pipe does two lane operations
// per cycle per multiprocessor (1/64 of FP32), and a comparison, minimum or select of doubles
// takes a turn on it like any other operation, so the helpers below compare bit patterns with the
// integer units: doubles of one sign order as their bits do.
// ---------------------------------------------------------------------------------------------
// FP32 value of a double without the flush of denormal results, which the compiler adds as a
// comparison and a multiplication under flush-to-zero (every FP32 operation that takes the value flushes it)
__device__ __forceinline__ float to_f32(double x) {
  float y;
  asm("cvt.rn.f32.f64 %0, %1;" : "=f"(y) : "d"(x));
  return y;
}
__device__ __forceinline__ float to_f32(float x) { return x; }
// x > 0 and normal
__device__ __forceinline__ bool normal_pos(double x) { return __double2hiint(x) >= 0x00100000; }
// 1/x for normal positive x below 2^1022: the hardware seed y (relative error e, |e| < 2^-19)
// improved by one third-order step y (1 + e + e^2), the truncated geometric series of 1/(1 - e), whose
// error is e^3 < 2^-57 plus the roundings.
__device__ __forceinline__ double rcp64(double x) {
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double e = fma(-x, y, 1.0);
  return fma(y, fma(e, e, e), y);
}
// 1/x for positive x: as rcp64 below 2^1020, by division above (an infinity gives 0).
__device__ __forceinline__ double rcp_pos(double x) { return __double2hiint(x) < 0x7fb00000 ? rcp64(x) : 1.0 / x; }
// sqrt(a) for normal positive a: the hardware seed of 1/sqrt(a), one coupled Newton step on
// g ~ sqrt(a) and h ~ 1/(2 sqrt(a)) (Goldschmidt's iteration), and a last correction by the residual
// a - g^2.
__device__ __forceinline__ double sqrt64(double a) {
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(a));
  double g = a * y, h = 0.5 * y;
  const double r = fma(-g, h, 0.5);
  g = fma(g, r, g);
  h = fma(h, r, h);
  return fma(fma(-g, g, a), h, g);
}
// 1/sqrt(a) for normal positive a: the hardware seed y with e = 1 - a y^2, and the series of
// (1 - e)^(-1/2) to its second power, y (1 + e/2 + 3 e^2/8).
__device__ __forceinline__ double rsqrt64(double a) {
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(a));
  const double e = fma(-(a * y), y, 1.0);
  return fma(y * e, fma(e, 0.375, 0.5), y);
}
// 1 / max(t, 1)
__device__ __forceinline__ double rcp_ge1(double t) {
  const int hi = __double2hiint(t);
  return hi < 0x3ff00000 ? 1.0 : (hi >= 0x7fd00000 ? 0.0 : rcp64(t));
}
__device__ __forceinline__ F2 rcp_ge1(F2 t) { return F2(rcp_approx(fmaxf(t.x, 1.0f)), rcp_approx(fmaxf(t.y, 1.0f))); }

// Comparisons by bit patterns for the selects of the gas kernels: a and b of one sign and neither
// zero; of opposite signs and neither zero; the sign of |a| - |b|; the middle of three values.
__device__ __forceinline__ bool same_sign(float a, float b) { return a * b > 0.0f; }
__device__ __forceinline__ bool opposite_sign(float a, float b) { return a * b < 0.0f; }
__device__ __forceinline__ int cmp_abs(float a, float b) { return fabsf(a) < fabsf(b) ? -1 : (fabsf(a) == fabsf(b) ? 0 : 1); }
__device__ __forceinline__ float median(float x, float u, float v) { return fmaxf(fminf(u, v), fminf(fmaxf(u, v), x)); }
__device__ __forceinline__ bool nonzero64(double a) { return (__double_as_longlong(a) << 1) != 0; }
__device__ __forceinline__ bool nonzero(float a) { return a != 0.0f; }
__device__ __forceinline__ bool nonzero(double a) { return nonzero64(a); }
__device__ __forceinline__ bool differ(float a, float b) { return __float_as_int(a) != __float_as_int(b); }
__device__ __forceinline__ bool differ(double a, double b) { return __double_as_longlong(a) != __double_as_longlong(b); }
__device__ __forceinline__ bool same_sign(double a, double b) {
  return (__double2hiint(a) ^ __double2hiint(b)) >= 0 && nonzero64(a) && nonzero64(b);
}
__device__ __forceinline__ bool opposite_sign(double a, double b) {
  return (__double2hiint(a) ^ __double2hiint(b)) < 0 && nonzero64(a) && nonzero64(b);
}
__device__ __forceinline__ int cmp_abs(double a, double b) {
  const long long x = __double_as_longlong(a) & 0x7fffffffffffffffLL, y = __double_as_longlong(b) & 0x7fffffffffffffffLL;
  return x < y ? -1 : (x == y ? 0 : 1);
}
// order-preserving map of a double to a signed integer (negative numbers have their magnitude bits
// inverted)
__device__ __forceinline__ long long key64(double a) {
  const long long k = __double_as_longlong(a);
  return k ^ ((k >> 63) & 0x7fffffffffffffffLL);
}
__device__ __forceinline__ bool less64(double a, double b) { return key64(a) < key64(b); }
__device__ __forceinline__ double median(double x, double u, double v) {
  const long long kx = key64(x), ku = key64(u), kv = key64(v);
  const long long r = max(min(ku, kv), min(max(ku, kv), kx));
  return __longlong_as_double(r ^ ((r >> 63) & 0x7fffffffffffffffLL));
}
__device__ __forceinline__ float min_fast(float a, float b) { return fminf(a, b); }
__device__ __forceinline__ float max_fast(float a, float b) { return fmaxf(a, b); }
// (as fmin and fmax, the other operand where one is NaN: the sound speed of a state with negative pressure.
// The result of an operation, whose NaN is a quiet one, is told by its high word.)
__device__ __forceinline__ bool nan64(double a) { return ((unsigned)__double2hiint(a) << 1) > 0xffe00000u; }
__device__ __forceinline__ double min_fast(double a, double b) { return nan64(b) || (less64(a, b) && !nan64(a)) ? a : b; }
__device__ __forceinline__ double max_fast(double a, double b) { return nan64(a) || (less64(a, b) && !nan64(b)) ? b : a; }
// a >= 0 (false for NaN)
__device__ __forceinline__ bool nonneg(float a) { return a >= 0.0f; }
__device__ __forceinline__ bool nonneg(double a) { return (unsigned)__double2hiint(a) <= 0x7ff00000u || !nonzero64(a); }
// 1/x and sqrt(x) of any argument: the short forms on the normal range, the library's outside it
__device__ __forceinline__ float rcp_any(float x) { return rcp_approx(x); }
__device__ __forceinline__ double rcp_any(double x) {
  const unsigned e = (unsigned)__double2hiint(x) & 0x7fffffffu;
  return e >= 0x00400000u && e < 0x7fb00000u ? rcp64(x) : 1.0 / x;
}
__device__ __forceinline__ float sqrt_any(float x) { return sqrtf(x); }
__device__ __forceinline__ double sqrt_any(double x) {
  const int e = __double2hiint(x);
  return e >= 0x00400000 && e < 0x7fb00000 ? sqrt64(x) : sqrt(x);
}

// ---------------------------------------------------------------------------------------------
// Per-cell reconstruction/divergence table (one row per padded cell and direction), built on the
// host in FP64 from the coordinate moments <x^j> of each cell (Sec. 5.1, Eq. 14).
// ---------------------------------------------------------------------------------------------
enum TabEntry {
  T_WA0, T_WA1, T_WA2,  // system 1 (Eq. 15): lower-face value = WA . (p[i-1], p[i], p[i+1])
  T_WB0, T_WB1, T_WB2,  // system 1: upper-face value
  T_SL2, T_TL2,         // face-interval reset on (centroid i-1, centroid i): s^2 and (1-s)^2
  T_SR2, T_TR2,         // same on (centroid i, centroid i+1)
  T_AL0, T_AL1, T_AL2,  // system 2 (Eq. 16) slope at the lower face = AL . (a, m, b)
  T_AR0, T_AR1, T_AR2,  // slope at the upper face
  T_RHL, T_RHR,         // zero-slope resets: w^2/<(x-x_L)^2>, w^2/<(x-x_R)^2>
  T_IL, T_IR, T_IC,     // linear MC: 1/(c_i - c_{i-1}), 1/(c_{i+1} - c_i), 1/(c_{i+1} - c_{i-1})
  T_DL, T_DR,           // x_L - c_i, x_R - c_i   (c = centroid)
  T_FL, T_FR,           // divergence factor of the lower / upper face (area / volume)
  T_ELL,                // optical-depth length of the lower face (R9)
  T_VOL,                // 1-d volume factor of the cell
  // Separable finite-volume geometry (Sec. 4, Eq. 8; Appendix A).  For the faces of this
  // direction: area/volume factor of the lower/upper face for scalar fluxes (T_FL/T_FR above),
  // for the flux of covariant component 0 (T_FL1/T_FR1) and of component 1 (T_FL2/T_FR2).
  T_FL1, T_FR1, T_FL2, T_FR2,
  // Factors this direction contributes to the faces of the other direction (scalar, component
  // 0, component 1) and to their optical-depth length.
  T_XS, T_X1, T_X2, T_XH,
  // Scale factors h of components 0 and 1 (their product over directions gives the cell's).
  T_HA, T_HB,
  // Volume-averaged connection coefficients carried by this direction (Appendix D): radial
  // <Gamma^1_11>, <Gamma^2_21> = <Gamma^3_31>, <Gamma^1_22>; polar <Gamma^2_22>, <Gamma^3_32>.
  T_GA, T_GB, T_GC,
  // Radial map at the cell's lower face (spherical radial direction; 1 elsewhere): 1 / (dr/dx1)
  // and 1 / r, the factors that turn a face's physical velocity into coordinate components.
  T_QI, T_RI,
  NTAB
};

template <class R> struct Tab {
  const R* p;    // [NTAB][np] for one direction, np = n + 4 (two ghost layers each side)
  int np;
  const R* cst;  // the single row of a direction whose rows are all equal (uniform grids), else null
  // rows outside the table (cells of a tile that overhang the grid; never used) are clamped so
  // that every read stays inside the array
  __device__ __forceinline__ R operator()(int e, int ip) const {
    if (cst) return cst[e];
    ip = ip < 0 ? 0 : (ip >= np ? np - 1 : ip);
    return __ldg(p + e * np + ip);
  }
};

// The table of a Cartesian direction: one row (of the launch arguments) for every cell.
template <class R> struct TabRow {
  const R* row;
  __device__ __forceinline__ R operator()(int e, int) const { return row[e]; }
};

// One row of a direction's table, found once: a kernel that reads several entries of a row pays
// for the test, the clamp and the address of Tab's reads once per row instead of once per entry.
template <class R> struct TabAt {
  const R* p;  // entry 0 of the row
  int np;
  __device__ __forceinline__ TabAt(const R* tab, int n, int ip) : p(tab + min(max(ip, 0), n + 3)), np(n + 4) {}
  __device__ __forceinline__ R operator()(int e, int) const { return __ldg(p + e * np); }
};

// ---------------------------------------------------------------------------------------------
// Parabolic (n = 2) reconstruction of one variable in one cell (Sec. 5.1; readings R2-R4).
// ip: padded index of the cell (cell i -> i + 2).
// ---------------------------------------------------------------------------------------------
template <class T, class V>
__device__ __forceinline__ void recon_parabolic(const T& t, int ip, V pm, V p0, V pp, V& a, V& b) {
  const V dl = p0 - pm, dr = pp - p0;
  // decisions are selects over values computed for every cell, so that a warp runs one path; in FP64
  // they are integer comparisons
  const bool ext = !same_sign(dl, dr);
  V a0 = t(T_WA0, ip) * pm + t(T_WA1, ip) * p0 + t(T_WA2, ip) * pp;
  V b0 = t(T_WB0, ip) * pm + t(T_WB1, ip) * p0 + t(T_WB2, ip) * pp;
  // between the zero-slope values at the two centroids, whichever is the lower one
  a0 = median(a0, pm + dl * t(T_SL2, ip), p0 - dl * t(T_TL2, ip));
  b0 = median(b0, p0 + dr * t(T_SR2, ip), pp - dr * t(T_TR2, ip));
  const V sl = t(T_AL0, ip) * a0 + t(T_AL1, ip) * p0 + t(T_AL2, ip) * b0;
  const V sr = t(T_AR0, ip) * a0 + t(T_AR1, ip) * p0 + t(T_AR2, ip) * b0;
  const bool inc = opposite_sign(sl, sr);  // extremum inside the cell
  const int cmp = cmp_abs(sl, sr);
  const V bz = a0 + (p0 - a0) * t(T_RHL, ip);  // zero slope at the lower face
  const V az = b0 + (p0 - b0) * t(T_RHR, ip);  // zero slope at the upper face
  const V an = inc ? (cmp == 0 ? p0 : (cmp < 0 ? a0 : az)) : a0;
  const V bn = inc ? (cmp == 0 ? p0 : (cmp < 0 ? bz : b0)) : b0;
  a = ext ? p0 : an;
  b = ext ? p0 : bn;
}

// Coefficients of the linear MC reconstruction of one cell (shared by all its variables and
// groups): inverse centroid gaps and the face offsets from the centroid.
template <class R> struct MCCoef { R il, ir, ic, dl, dr; };
template <class R, class T> __device__ __forceinline__ MCCoef<R> mc_coef(const T& t, int ip) {
  return {t(T_IL, ip), t(T_IR, ip), t(T_IC, ip), t(T_DL, ip), t(T_DR, ip)};
}

// ---------------------------------------------------------------------------------------------
// HLLC (Sec. 5.2; Toro, Spruce & Speares 1994 with Batten et al. 1997 / Einfeldt speed bounds,
// reading R6).  States are primitive (rho, p, u_n, u_t1, u_t2) in the face-normal frame.
// Output: fluxes of (rho, rho u_n, rho u_t1, rho u_t2, rho e) per unit physical area and the
// contact speed (the particle velocity used to upwind radiation advection, Eq. 19).
// ---------------------------------------------------------------------------------------------
template <class R, int D>
__device__ __forceinline__ void hllc(R gam, const R* L, const R* Rs, R* f, R& vstar) {
  // Every division is a reciprocal, shared where the denominator is (the
  // FP64 form of a division costs twice a reciprocal's operations), and the choice among the
  // supersonic and star fluxes is a select: the side k (left when the face is supersonic to the
  // right or the contact moves right) and its plain flux F_k for every face; the star correction
  // S_k (U*_k - U_k) is added where the face is subsonic.
  const R igm1 = rcp_any(gam - R(1)), g1 = gam - R(1);
  const R rl = L[0], pl = L[1], ul = L[2], rr = Rs[0], pr = Rs[1], ur = Rs[2];
  R kl = ul * ul, kr = ur * ur;
#pragma unroll
  for (int q = 1; q < D; ++q) { kl += L[2 + q] * L[2 + q]; kr += Rs[2 + q] * Rs[2 + q]; }
  const R El = pl * igm1 + R(0.5) * rl * kl, Er = pr * igm1 + R(0.5) * rr * kr;
  const R irl = rcp_any(rl), irr = rcp_any(rr);
  const R al = sqrt_any(gam * pl * irl), ar = sqrt_any(gam * pr * irr);
  const R sl = sqrt_any(rl), sr = sqrt_any(rr), iw = rcp_any(sl + sr);
  const R Ht = (sl * ((El + pl) * irl) + sr * ((Er + pr) * irr)) * iw;
  const R ut = (sl * ul + sr * ur) * iw;
  R v2 = ut * ut;
#pragma unroll
  for (int q = 1; q < D; ++q) { const R vq = (sl * L[2 + q] + sr * Rs[2 + q]) * iw; v2 += vq * vq; }
  const R at2 = g1 * (Ht - R(0.5) * v2);
  const R at = sqrt_any(nonneg(at2) ? at2 : R(0));
  const R SL = min_fast(ul - al, ut - at), SR = max_fast(ur + ar, ut + at);
  const R dl = rl * (SL - ul), dr = rr * (SR - ur);
  const R Ss = (pr - pl + ul * dl - ur * dr) * rcp_any(dl - dr);
  vstar = Ss;
  const bool supL = nonneg(SL), supR = !supL && !nonneg(SR), sup = supL || supR;
  const bool left = supL || (!supR && nonneg(Ss));
  const R rk = left ? rl : rr, pk = left ? pl : pr, uk = left ? ul : ur;
  const R Ek = left ? El : Er, Sk = left ? SL : SR, irk = left ? irl : irr;
  const R sku = Sk - uk, m = rk * uk;
  const R fac = rk * sku * rcp_any(Sk - Ss);
  const R f1 = m * uk + pk;
  f[0] = sup ? m : m + Sk * (fac - rk);
  f[1] = sup ? f1 : f1 + Sk * (fac * Ss - m);
#pragma unroll
  for (int q = 1; q < D; ++q) {
    const R wq = left ? L[2 + q] : Rs[2 + q];
    const R fq = m * wq;
    f[1 + q] = sup ? fq : fq + Sk * (fac * wq - rk * wq);
  }
  const R Es = fac * (Ek * irk + (Ss - uk) * (Ss + pk * (irk * rcp_any(sku))));
  const R fE = (Ek + pk) * uk;
  f[1 + D] = sup ? fE : fE + Sk * (Es - Ek);
}

// Gas flux of one face by the selected solver (Sec. 5.2 names local Lax-Friedrichs, HLLE and
// HLLC; reading R21): 0 HLLC, 1 HLLE with the speed bounds of R6 (b_L = min(S_L, 0),
// b_R = max(S_R, 0)), 2 local Lax-Friedrichs with s = max(|u_L| + a_L, |u_R| + a_R).  vstar is
// always the HLLC contact speed of the two states (the upwind velocity of Eq. 19).
template <class R, int D>
__device__ __forceinline__ void gas_riemann(int solver, R gam, const R* L, const R* Rs, R* f, R& vstar) {
  hllc<R, D>(gam, L, Rs, f, vstar);
  if (solver == 0) return;
  const R gm1 = gam - R(1);
  const R rl = L[0], pl = L[1], ul = L[2], rr = Rs[0], pr = Rs[1], ur = Rs[2];
  R kl = ul * ul, kr = ur * ur;
#pragma unroll
  for (int q = 1; q < D; ++q) { kl += L[2 + q] * L[2 + q]; kr += Rs[2 + q] * Rs[2 + q]; }
  const R El = pl / gm1 + R(0.5) * rl * kl, Er = pr / gm1 + R(0.5) * rr * kr;
  const R al = sqrt(gam * pl / rl), ar = sqrt(gam * pr / rr);
  R UL[2 + D], UR[2 + D], FL[2 + D], FR[2 + D];
  UL[0] = rl; UR[0] = rr;
  FL[0] = rl * ul; FR[0] = rr * ur;
#pragma unroll
  for (int q = 0; q < D; ++q) {
    UL[1 + q] = rl * L[2 + q]; UR[1 + q] = rr * Rs[2 + q];
    FL[1 + q] = rl * ul * L[2 + q]; FR[1 + q] = rr * ur * Rs[2 + q];
  }
  FL[1] += pl; FR[1] += pr;
  UL[1 + D] = El; UR[1 + D] = Er;
  FL[1 + D] = (El + pl) * ul; FR[1 + D] = (Er + pr) * ur;
  if (solver == 2) {
    const R sm = fmax(fabs(ul) + al, fabs(ur) + ar);
#pragma unroll
    for (int v = 0; v < 2 + D; ++v) f[v] = R(0.5) * (FL[v] + FR[v]) - R(0.5) * sm * (UR[v] - UL[v]);
    return;
  }
  const R sl = sqrt(rl), sr = sqrt(rr), iw = R(1) / (sl + sr);
  const R Ht = (sl * ((El + pl) / rl) + sr * ((Er + pr) / rr)) * iw;
  const R ut = (sl * ul + sr * ur) * iw;
  R v2 = ut * ut;
#pragma unroll
  for (int q = 1; q < D; ++q) { const R vq = (sl * L[2 + q] + sr * Rs[2 + q]) * iw; v2 += vq * vq; }
  const R at2 = gm1 * (Ht - R(0.5) * v2);
  const R at = sqrt(at2 > R(0) ? at2 : R(0));
  const R bl = fmin(fmin(ul - al, ut - at), R(0)), br = fmax(fmax(ur + ar, ut + at), R(0));
  const R ib = R(1) / (br - bl);
#pragma unroll
  for (int v = 0; v < 2 + D; ++v) f[v] = (br * FL[v] - bl * FR[v] + bl * br * (UR[v] - UL[v])) * ib;
}

// ---------------------------------------------------------------------------------------------
// Powers with half-integer exponents: x^(h/2) = x^k sqrt(x)^(h mod 2), k = floor(h/2), by binary
// powers and one reciprocal for k < 0.  The exponent is the launch's: every branch is uniform, and
// the common |k| < 8 take no loop (with a loop and signed divisions the powers were a fifth of the
// interaction kernel's instructions).
// ---------------------------------------------------------------------------------------------
template <class R> __device__ __forceinline__ R hpow(R x, int h) {
  const int k = h >> 1, n = k < 0 ? -k : k;
  R r = n & 1 ? x : R(1);
  if (n > 1) {
    R b = x * x;
    if (n & 2) r = r * b;
    if (n > 3) {
      b = b * b;
      if (n & 4) r = r * b;
      for (int m = n >> 3; m; m >>= 1) {
        b = b * b;
        if (m & 1) r = r * b;
      }
    }
  }
  if (k < 0) r = rcp_any(r);
  return h & 1 ? r * sqrt_any(x) : r;
}

// ---------------------------------------------------------------------------------------------
// Planck integrals per group edge.  For an edge at x = eps/T the device evaluates
//   Q(x) = Int_0^x t^3/(e^t-1) dt   (x < XSPLIT, Bernoulli-number power series)
//   Q(x) = Int_x^inf t^3/(e^t-1) dt (x >= XSPLIT, sum_n e^{-nx} (x^3/n + 3x^2/n^2 + 6x/n^3 + 6/n^4))
// and w(x) = x^4/(e^x - 1) (for dB/dT).  A group band then combines its two edges without
// cancelling large tails.  Coefficients b_k = B_k/k! are generated on the host.
// ---------------------------------------------------------------------------------------------
struct PlanckCoef {
  double lo[NPLANCK_LO];  // b_{2m}/(2m+3), m = 1..NPLANCK_LO (D series, beyond 1/3 - x/8)
  double wd[NPLANCK_LO];  // b_{2m}, m = 1..NPLANCK_LO (w series, beyond 1 - x/2)
  double rn[NPLANCK_UP];  // 1/n, n = 1..NPLANCK_UP (exponential series)
};

template <class R> struct PlanckEdge { R Q, w; bool upper; };

// FP64 edge evaluation (used by the FP64 path and the final FP64 coupling arithmetic).
__device__ __forceinline__ PlanckEdge<double> planck_edge64(double x, const PlanckCoef& pc) {
  PlanckEdge<double> e;
  if (x < XSPLIT) {
    double x2 = x * x, x3 = x2 * x;
    double sd = pc.lo[NPLANCK_LO - 1], sw = pc.wd[NPLANCK_LO - 1];
#pragma unroll
    for (int m = NPLANCK_LO - 2; m >= 0; --m) { sd = fma(sd, x2, pc.lo[m]); sw = fma(sw, x2, pc.wd[m]); }
    e.Q = x3 * (1.0 / 3.0 - 0.125 * x + x2 * sd);
    e.w = x3 * (1.0 - 0.5 * x + x2 * sw);
    e.upper = false;
  } else {
    double y = exp(-x), yn = y, x2 = x * x, x3 = x2 * x, s = 0.0;
    const double a2 = 3.0 * x2, a1 = 6.0 * x;
    for (int n = 1; n <= NPLANCK_UP; ++n) {
      const double rn = pc.rn[n - 1];
      double t = yn * rn * (x3 + rn * (a2 + rn * (a1 + 6.0 * rn)));
      s += t;
      if (t <= 1e-17 * s) break;
      yn *= y;
    }
    e.Q = s;
    e.w = x3 * x * y / (1.0 - y);
    e.upper = true;
  }
  return e;
}

// The same from the table of polynomials (fx_planck.h) at x16 = 16 x: row n = round(16 x), t = 16 x - n.
// One edge takes 20 FP64 operations (seven Horner steps for the value, six for the derivative, and
// w = x dQ/dx up to sign from it), against 58 for the power series below XSPLIT and ~20 + 8 per term
// with the exponential series above it: the FP64 pipe is what the FP64 interaction is bound by.
// Rows past the table (x >= 64, and NaN) take the series.  The row is read as four 16-byte loads.
// Relative error of the edge's integral and of its weight: at most 5 and 8 units of 2^-53, measured 3.6 and
// 5.2 (the series: 6.4 and 9.3).
static __device__ __noinline__ PlanckEdge<double> planck_edge_far(double x, const PlanckCoef& pc) { return planck_edge64(x, pc); }
__device__ __forceinline__ PlanckEdge<double> planck_edge_tab(double x16, const double* __restrict__ tab, const PlanckCoef& pc) {
  if ((unsigned)__double2hiint(x16) >= 0x40900000u) return planck_edge_far(x16 * 0.0625, pc);  // 16 x >= 1024
  const double magic = 6755399441055744.0;  // 1.5 2^52: the sum's low word is the nearest integer
  const double s = x16 + magic;
  const int n = __double2loint(s);
  const double t = x16 - (s - magic);
  const double2* const r = reinterpret_cast<const double2*>(tab) + n * 4;
  const double2 a = __ldg(r), b = __ldg(r + 1), c = __ldg(r + 2), d = __ldg(r + 3);
  double p = d.y, q = d.y;
  p = fma(p, t, d.x);
  q = fma(q, t, p);
  p = fma(p, t, c.y);
  q = fma(q, t, p);
  p = fma(p, t, c.x);
  q = fma(q, t, p);
  p = fma(p, t, b.y);
  q = fma(q, t, p);
  p = fma(p, t, b.x);
  q = fma(q, t, p);
  p = fma(p, t, a.y);
  q = fma(q, t, p);  // dp/dt
  p = fma(p, t, a.x);
  PlanckEdge<double> e;
  e.upper = n >= PETAB_SPLIT;
  if (e.upper) {
    e.Q = p;
    e.w = -(x16 * q);
  } else {
    const double x3 = x16 * x16 * (x16 * (1.0 / 4096.0));
    e.Q = x3 * p;
    e.w = x3 * fma(x16, q, 3.0 * p);
  }
  return e;
}

// Band integral Int_{x_lo}^{x_hi} t^3/(e^t-1) dt from the two edge evaluations.
template <class R>
__device__ __forceinline__ R planck_band(const PlanckEdge<R>& lo, const PlanckEdge<R>& hi) {
  const R total = R(6.4939394022668291491);  // pi^4/15
  if (!lo.upper && !hi.upper) return hi.Q - lo.Q;
  if (lo.upper && hi.upper) return lo.Q - hi.Q;
  return (total - lo.Q) - hi.Q;
}

}  // namespace fx
