// Three neutrino species (Sec. 3.2; Sec. 5.3 in the core-collapse form): the composition rho Y_e
// and the two-equation interaction in (T, Y_e), on Cartesian and spherical grids.
//
// The radiation channels are the groups of the three species (nu_e, anti-nu_e, nu_x), species-
// major; the gas face and radiation/update kernels transport them like groups.  rho Y_e lives in
// a block after the radiation block.
//   comp_kernel: its finite-volume update and RK combination (the gas mass flux times the
//     reconstructed Y_e on the v* upwind side of each face, the HLLC passive-scalar flux);
//   couple_ye_kernel (FP64 state) and couple_ye32_kernel (FP32 state): the interaction, one thread
//     per cell, the iterate in FP64 in both; with the FP32 state the band energies B_g(T) come
//     from the FP32 Planck band table (as in the one-species FP32 interaction), the channel
//     arithmetic is FP32 and the iteration stops at FP32 resolution.  Inner backward-Euler update of
//     every channel at (T, Y_e), with the equilibrium energy w_s(Y_e) B_g(T), w = 2 Y_e,
//     2 (1 - Y_e), 1, and the lepton number per unit energy xi = -xi0/eps_g, +xi0/eps_g, 0;
//     outer residuals r_E = u(T) - u^- + sum dE and r_X = rho (Y_e - Y_e^-) - sum xi dE, solved
//     by Newton with the analytic Jacobian and backtracking on the scaled residual norm, with
//     alternating one-variable bisections as the fallback; then u and rho Y_e by conservation
//     and the flux absorption with its momentum and energy feedback.  The decisions follow the
//     oracle's two-equation interaction in the same order.
#pragma once
#include <cuda_runtime.h>

#include "fx_couple.cuh"
#include "fx_stage.cuh"

namespace fx {

// ---- composition ----------------------------------------------------------------------------
// One thread per cell.  Bound by instruction issue: the rows of the geometry tables are found once
// each (a Cartesian direction has one row, of the launch arguments); with a test, a clamp and an
// address per entry 512^2 cells took 29 us, now 10.
template <class R, int D, bool SPH>
__global__ void __launch_bounds__(256) comp_kernel(const __grid_constant__ StageArgs<R> A) {
  constexpr int NG = 2 + D;
  using TT = typename std::conditional<SPH, TabAt<R>, TabRow<R>>::type;
  auto row_of_dir = [&](int d, int i) -> TT {
    if constexpr (SPH) return TT(A.tab[d], A.g.n[d], bc_pad(i));
    else return TT{A.urow[d]};
  };
  const DevGrid& g = A.g;
  const uint32_t ncell = (uint32_t)g.ncell;
  const uint32_t c = blockIdx.x * 256u + threadIdx.x;
  if (c >= ncell) return;
  const int n0 = g.n[0], n1 = g.n[1], n2 = g.n[2];
  const int ix = (int)(c % (uint32_t)n0), iy = (int)((c / (uint32_t)n0) % (uint32_t)n1);
  const int iz = (int)(c / ((uint32_t)n0 * n1));
  const uint32_t XO = (uint32_t)(NG + (1 + D) * g.G) * ncell;
  // Y_e of the cell at offset k along direction d (ghosts from the boundary rules)
  auto ye = [&](int d, int k) -> R {
    int x3[3] = {ix, iy, iz};
    bool f = false;
    x3[d] = min(max(bc_map(x3[d] + k, g.n[d], g.bc_lo[d], g.bc_hi[d], f), 0), g.n[d] - 1);
    const uint32_t ci = ((uint32_t)x3[2] * n1 + x3[1]) * n0 + x3[0];
    return A.in[FXI(XO + ci, A.n_state)] / A.in[FXI(ci, A.n_state)];
  };
  R net = R(0);
#pragma unroll
  for (int d = 0; d < D; ++d) {
    const int i = d == 0 ? ix : (d == 1 ? iy : iz);
    const TT tt = row_of_dir(d, i);
    R y[5];
#pragma unroll
    for (int k = 0; k < 5; ++k) y[k] = ye(d, k - 2);
    R am, bm, a0, b0, ap, bp;
    recon_parabolic(row_of_dir(d, i - 1), 0, y[0], y[1], y[2], am, bm);
    recon_parabolic(tt, 0, y[1], y[2], y[3], a0, b0);
    recon_parabolic(row_of_dir(d, i + 1), 0, y[2], y[3], y[4], ap, bp);
    (void)am;
    (void)bp;
    const uint32_t ex = (uint32_t)(n0 + (d == 0)), ey = (uint32_t)(n1 + (d == 1));
    const uint32_t nf = ex * ey * (uint32_t)(n2 + (d == 2));
    const uint32_t lf = ((uint32_t)iz * ey + (uint32_t)iy) * ex + (uint32_t)ix;
    const uint32_t uf = lf + (d == 0 ? 1u : (d == 1 ? ex : ex * ey));
    const R* fr = A.faces + A.face_off[d];
    const uint32_t nfr = (uint32_t)(NG + 1 + (g.vterms ? D - 1 : 0)) * nf;  // this direction's block
    (void)nfr;
    const R mlo = fr[FXI(lf, nfr)], mhi = fr[FXI(uf, nfr)];
    const R vlo = fr[FXI((uint32_t)NG * nf + lf, nfr)], vhi = fr[FXI((uint32_t)NG * nf + uf, nfr)];
    const R flo = mlo * (vlo >= R(0) ? bm : a0), fhi = mhi * (vhi >= R(0) ? b0 : ap);
    // area/volume factors of the two faces (Eq. 8 with a separable volume element): this
    // direction's own, times the cross factors of the other directions (1 on Cartesian grids)
    R cross = R(1);
    if constexpr (SPH) {
#pragma unroll
      for (int e = 0; e < D; ++e)
        if (e != d) cross *= row_of_dir(e, e == 0 ? ix : iy)(T_XS, 0);
    }
    net += (fhi * tt(T_FR, 0) - flo * tt(T_FL, 0)) * cross;
  }
  const auto& K = A.k(R(0));  // the step and RK weights in R (no per-thread conversions)
  const R u = A.in[FXI(XO + c, A.n_state)] - K.dt * net;
  const bool stage2 = A.base != nullptr;
  const R r = stage2 ? K.alpha * A.base[FXI(XO + c, A.n_state)] + K.beta * u : u;
  if (!isfinite(r)) atomicOr(A.status, ST_NONFINITE);
  A.out[FXI(XO + c, A.n_state)] = r;
}

// ---- two-equation interaction ---------------------------------------------------------------
constexpr int CPLYE_THREADS = 128;

inline size_t couple_ye_smem_bytes(int G) { return (size_t)2 * CPLYE_THREADS * (size_t)(G + 1) * sizeof(double); }

__device__ __forceinline__ double ye_w(int s, double Y) { return s == 0 ? 2.0 * Y : (s == 1 ? 2.0 * (1.0 - Y) : 1.0); }
__device__ __forceinline__ double ye_dw(int s) { return s == 0 ? 2.0 : (s == 1 ? -2.0 : 0.0); }

template <int D>
__global__ void __launch_bounds__(CPLYE_THREADS) couple_ye_kernel(const __grid_constant__ StageArgs<double> A) {
  using R = double;
  constexpr int NG = 2 + D, NRV = 1 + D;
  extern __shared__ __align__(16) unsigned char ye_raw[];
  const DevGrid& g = A.g;
  const int G = g.G, Gs = g.Gs, RS = G + 1;
  // E^- of the cell's channels and the last evaluation's E
  double* Em = reinterpret_cast<double*>(ye_raw) + threadIdx.x * RS;
  double* En = Em + CPLYE_THREADS * RS;
  const uint32_t ncell = (uint32_t)g.ncell;
  const uint32_t c = blockIdx.x * CPLYE_THREADS + threadIdx.x;
  const GroupConst& gc = *A.gc;
  // 1 / eps_g of each group (centre sqrt(eps_{g-1/2} eps_{g+1/2})), once per block
  __shared__ double s_icen[MAXG];
  for (int j = threadIdx.x; j < Gs; j += CPLYE_THREADS) s_icen[FXI(j, MAXG)] = 1.0 / sqrt(gc.edge[j] * gc.edge[j + 1]);
  __syncthreads();
  if (c >= ncell) return;
  const double cl = g.c, dt = A.dts, cv = 1.0 / (g.gamma - 1.0), xi0 = g.xi0;
  R* U = A.out;
  const uint32_t rad = (uint32_t)NG * ncell, XO = (uint32_t)(NG + NRV * G) * ncell;
  unsigned st = 0;
  double rho = U[FXI(c, A.n_state)];
  if (rho < g.rho_floor) { rho = g.rho_floor; U[FXI(c, A.n_state)] = (R)rho; st |= ST_FLOOR; }
  // scale factors h_0, h_1 of the cell (1 on Cartesian grids): momentum and flux are covariant
  double hq[D];
#pragma unroll
  for (int q = 0; q < D; ++q) hq[q] = 1.0;
  if (g.geom != 0) {
    const int i3[3] = {(int)(c % (uint32_t)g.n[0]), (int)((c / (uint32_t)g.n[0]) % (uint32_t)g.n[1]), 0};
#pragma unroll
    for (int d = 0; d < D; ++d) {
      const Tab<R> td{A.tab[d], g.n[d] + 4, A.uniform[d] ? A.urow[d] : nullptr};
      hq[0] *= (double)td(T_HA, bc_pad(i3[d]));
      if (D > 1) hq[D > 1 ? 1 : 0] *= (double)td(T_HB, bc_pad(i3[d]));
    }
  }
  double ke = 0.0;
#pragma unroll
  for (int q = 0; q < D; ++q) { const double vh = U[FXI((1 + q) * ncell + c, A.n_state)] / (rho * hq[q]); ke += 0.5 * rho * vh * vh; }
  double u_m = U[FXI((NG - 1) * ncell + c, A.n_state)] - ke;
  const double u_floor = g.p_floor / (g.gamma - 1.0);
  if (u_m < u_floor) { u_m = u_floor; U[FXI((NG - 1) * ncell + c, A.n_state)] = (R)(ke + u_m); st |= ST_FLOOR; }
  const double X_m = U[FXI(XO + c, A.n_state)], Y_m = X_m / rho;
  double Esum = 0.0, Lsum = 0.0, fadd = 0.0;
  for (int k = 0; k < G; ++k) {
    double E = U[FXI(rad + c * (uint32_t)G + k, A.n_state)];
    if (E < g.E_floor) { fadd += g.E_floor - E; E = g.E_floor; }
    Em[k] = E;
    Esum += E;
    const int s = k / Gs;
    if (s < 2) Lsum += fabs(xi0 * s_icen[FXI(k % Gs, MAXG)]) * E;
  }
  const double norm = g.a_rad * 0.15398973382026502;  // a_R 15/pi^4
  const double kpre = g.kappa0 * hpow(rho, g.kap_rho_h);
  auto xi_of = [&](int k) -> double {
    const int s = k / Gs;
    const double xg = xi0 * s_icen[FXI(k % Gs, MAXG)];
    return s == 0 ? -xg : (s == 1 ? xg : 0.0);
  };
  // residuals and Jacobian at (T, Y); with keep, the channel energies into En.  A band edge is
  // evaluated once (the upper edge of group g is the lower edge of g + 1), and the backward-Euler
  // factor 1/(1 + tau) and xi once per group (the three species share the group's opacity)
  auto eval = [&](double T, double Y, double& rE, double& rX, double J[2][2], bool keep) {
    double dE = 0.0, dX = 0.0, eT = 0.0, eY = 0.0, xT = 0.0, xY = 0.0;
    const double invT = 1.0 / T, T3 = T * T * T;
    const double kT = kpre * hpow(T, g.kap_T_h);
    PlanckEdge<double> lo = planck_edge_tab(gc.edge[0] * invT * 16.0, A.pk.petab, A.pk.c64);
    for (int gg = 0; gg < Gs; ++gg) {
      const PlanckEdge<double> hi = planck_edge_tab(gc.edge[gg + 1] * invT * 16.0, A.pk.petab, A.pk.c64);
      const double I = planck_band(lo, hi);
      const double B = norm * T3 * T * I;
      const double dB = norm * (4.0 * T3 * I + T3 * (lo.w - hi.w));
      lo = hi;
      const double kap = kT * gc.efac[gg];
      const double tau = cl * dt * kap, dtau = tau * (0.5 * g.kap_T_h * invT);
      const double xg = xi0 * s_icen[FXI(gg, MAXG)];
      const double inv = rcp_pos(1.0 + tau);
      for (int s = 0; s < 3; ++s) {
        const int k = s * Gs + gg;
        const double w = ye_w(s, Y), dw = ye_dw(s), xi = s == 0 ? -xg : (s == 1 ? xg : 0.0);
        const double Eq = w * B;
        const double Ek = (Em[k] + tau * Eq) * inv;
        const double dT_ = (tau * w * dB + dtau * (Eq - Ek)) * inv;
        const double dY_ = tau * dw * B * inv;
        dE += Ek - Em[k];
        dX += xi * (Ek - Em[k]);
        eT += dT_;
        eY += dY_;
        xT += xi * dT_;
        xY += xi * dY_;
        if (keep) En[k] = Ek;
      }
    }
    rE = rho * cv * T - u_m + dE;
    rX = rho * (Y - Y_m) - dX;
    J[0][0] = rho * cv + eT;
    J[0][1] = eY;
    J[1][0] = -xT;
    J[1][1] = rho - xY;
  };
  const double rtol = g.newton_rtol, n2ok = 1e-28, n2fb = 1e-24;
  const double sE = u_m + Esum, sX = fabs(X_m) + Lsum + 1e-300;
  auto norm2 = [&](double rE, double rX) { const double a = rE / sE, b = rX / sX; return a * a + b * b; };
  double T = u_m / (rho * cv), Y = Y_m, rE, rX, J[2][2];
  eval(T, Y, rE, rX, J, false);
  bool ok = false;
  for (int it = 0; it < g.newton_maxit; ++it) {
    if (norm2(rE, rX) <= n2ok) { ok = true; break; }
    const double det = J[0][0] * J[1][1] - J[0][1] * J[1][0];
    const double dT = -(J[1][1] * rE - J[0][1] * rX) / det;
    const double dY = -(J[0][0] * rX - J[1][0] * rE) / det;
    if (fabs(dT) <= rtol * T && fabs(dY) <= rtol * fmax(Y, 1e-3)) {
      T = T + dT;
      Y = Y + dY;
      ok = true;
      break;
    }
    double lam = 1.0;
    bool acc = false;
    const double n0 = norm2(rE, rX);
    for (int ls = 0; ls < 40; ++ls) {
      const double Tt = T + lam * dT, Yt = Y + lam * dY;
      if (Tt > 0.0 && Yt >= 0.0 && Yt <= 1.0) {
        double rEt, rXt, Jt[2][2];
        eval(Tt, Yt, rEt, rXt, Jt, false);
        if (norm2(rEt, rXt) < n0) {
          T = Tt; Y = Yt; rE = rEt; rX = rXt;
          J[0][0] = Jt[0][0]; J[0][1] = Jt[0][1]; J[1][0] = Jt[1][0]; J[1][1] = Jt[1][1];
          acc = true;
          break;
        }
      }
      lam *= 0.5;
    }
    if (!acc) break;
  }
  if (!ok) {
    for (int round = 0; round < 20 && !ok; ++round) {
      double Jd[2][2], r1, r2, rh, rm;
      double lo = 0.5 * T, hi = 2.0 * T;
      eval(lo, Y, r1, r2, Jd, false);
      for (int k = 0; k < 200 && r1 > 0.0; ++k) { lo = 0.5 * lo; eval(lo, Y, r1, r2, Jd, false); }
      eval(hi, Y, rh, r2, Jd, false);
      for (int k = 0; k < 200 && rh < 0.0; ++k) { hi = 2.0 * hi; eval(hi, Y, rh, r2, Jd, false); }
      for (int k = 0; k < g.bisect_maxit && hi - lo > rtol * hi; ++k) {
        const double mid = 0.5 * (lo + hi);
        eval(mid, Y, rm, r2, Jd, false);
        if (rm > 0.0) hi = mid; else lo = mid;
      }
      T = 0.5 * (lo + hi);
      double ylo = 0.0, yhi = 1.0;
      for (int k = 0; k < g.bisect_maxit && yhi - ylo > rtol; ++k) {
        const double mid = 0.5 * (ylo + yhi);
        eval(T, mid, r1, rm, Jd, false);
        if (rm > 0.0) yhi = mid; else ylo = mid;
      }
      Y = 0.5 * (ylo + yhi);
      eval(T, Y, rE, rX, J, false);
      if (norm2(rE, rX) <= n2fb) ok = true;
    }
    if (!ok) st |= ST_NEWTON;
  }
  // channel energies at the accepted (T, Y_e); u and rho Y_e by conservation
  eval(T, Y, rE, rX, J, true);
  double dEsum = 0.0, dXsum = 0.0;
  for (int k = 0; k < G; ++k) {
    const double dk = En[k] - Em[k];
    dEsum += dk;
    dXsum += xi_of(k) * dk;
    U[FXI(rad + c * (uint32_t)G + k, A.n_state)] = (R)En[k];
  }
  // (kept in FP64 until the momentum feedback below, then stored once)
  double ue = ke + (u_m - dEsum);
  U[FXI(XO + c, A.n_state)] = (R)(X_m + dXsum);
  // flux absorption (Eq. 28) with its momentum and energy feedback (Eqs. 31-32)
  double vcon[D], dm[D], dwork = 0.0;
#pragma unroll
  for (int q = 0; q < D; ++q) { vcon[q] = U[FXI((1 + q) * ncell + c, A.n_state)] / (rho * hq[q] * hq[q]); dm[q] = 0.0; }
  const double sig = g.sigma0 * rho;
  const double kT = kpre * hpow(T, g.kap_T_h);
  for (int k = 0; k < G; ++k) {
    const double fac = rcp_pos(1.0 + cl * dt * (kT * gc.efac[k % Gs] + sig));
#pragma unroll
    for (int q = 0; q < D; ++q) {
      R* Fp = FXP(U, rad + (uint32_t)(1 + q) * ncell * (uint32_t)G + c * (uint32_t)G + k, A.n_state);
      const double F = *Fp, Fn = F * fac, dF = Fn - F;
      dm[q] += dF;
      dwork += vcon[q] * dF;
      *Fp = (R)Fn;
    }
  }
  const double ic2 = 1.0 / (cl * cl);
#pragma unroll
  for (int q = 0; q < D; ++q) U[FXI((1 + q) * ncell + c, A.n_state)] = (R)((double)U[FXI((1 + q) * ncell + c, A.n_state)] - dm[q] * ic2);
  ue -= dwork * ic2;
  U[FXI((NG - 1) * ncell + c, A.n_state)] = (R)ue;
  bool bad = !isfinite(ue) || !isfinite((double)U[FXI(XO + c, A.n_state)]);
  if (bad) st |= ST_NONFINITE;
  if (st) atomicOr(A.status, st);
  if (A.budget != nullptr) {
    // (reading R13) the energy the gas gives up to the flux absorption and the energy the E
    // floor adds, weighted as the RK combination weighs this stage's interaction; one add per
    // cell into the block's budget row (the budgets are a diagnostic, off in production runs)
    const double wv = cell_volume(A, c) * A.bw_cpl;
    double* row = A.budget + (size_t)(blockIdx.x % BUDGET_SLOTS) * NBUDGET;
    if (dwork != 0.0) atomicAdd(row + 6, dwork * ic2 * wv);
    if (fadd != 0.0) atomicAdd(row + 7, fadd * wv);
  }
}

// ---------------------------------------------------------------------------------------------
// The same interaction for the FP32 state.  It was bound by the FP64 pipe (85 % busy): per-channel
// sums, the flux absorption and the conserved updates in FP64 made ~1500 FP64 lane operations per
// cell of 24 channels, and its rows were read and written one thread per cell, uncoalesced.  Here
//   - the rows are staged through shared memory in coalesced copies (RowCopy);
//   - what was summed in FP64 over channels is summed in pairs of floats that keep every rounding
//     error (TwoSum), and the differences E - E^- and F_new - F are formed exactly as such pairs, so
//     FP64 is left to the iterate, the residuals, the Jacobian's solve and the gas and composition
//     updates;
//   - the absorption factor 1/(1 + tau) of a group is one FP64 argument split into a float pair, its
//     reciprocal corrected to a pair, so that F_new carries one FP32 rounding as before;
//   - dr_E/dY_e vanishes identically (the weights w of nu_e and anti-nu_e have opposite derivatives
//     and one opacity), so the 2 x 2 solve is two divisions;
//   - every evaluation keeps its channel energies, so a run that ends on the residual test needs no
//     evaluation more.
// 512^2 cells x 24 channels: 0.72 -> 0.17 ms per launch (with the composition kernel).
// ---------------------------------------------------------------------------------------------
struct FPair { float h, l; };  // the sum h + l
__device__ __forceinline__ void acc(FPair& a, float x) {
  float s, e;
  two_sum(a.h, x, s, e);
  a.h = s;
  a.l += e;
}
__device__ __forceinline__ void two_diff(float a, float b, float& s, float& e) {
  s = a - b;
  const float bv = s - a;
  e = (a - (s - bv)) - (b + bv);
}
// a += x - y, the difference exact
__device__ __forceinline__ void acc_diff(FPair& a, float x, float y) {
  float d, f, s, e;
  two_diff(x, y, d, f);
  two_sum(a.h, d, s, e);
  a.h = s;
  a.l += e + f;
}
// a += (x + xl) y, the product with its rounding errors
__device__ __forceinline__ void acc_mul(FPair& a, float x, float xl, float y) {
  const float p = __fmul_rn(x, y);
  acc(a, p);
  a.l += fmaf(xl, y, fmaf(x, y, -p));
}
__device__ __forceinline__ double val(FPair a) { return (double)a.h + (double)a.l; }

constexpr int couple_ye32_rows(int D) { return D > 2 ? D : 2; }
template <int D> inline size_t couple_ye32_smem_bytes(int G) {
  return (size_t)couple_ye32_rows(D) * CPL_THREADS * (size_t)(G + 1) * sizeof(float);
}

template <int D>
__global__ void __launch_bounds__(CPL_THREADS, 5) couple_ye32_kernel(const __grid_constant__ StageArgs<float> A) {
  constexpr int NG = 2 + D;
  extern __shared__ __align__(16) unsigned char ye_raw[];
  float* const srow = reinterpret_cast<float*>(ye_raw);  // E^- and E, then the F_q
  __shared__ float s_ef[MAXG], s_ed[MAXG + 1], s_xi[MAXG], s_xil[MAXG];  // (xi0/eps_g: s_xi + s_xil)
  __shared__ double s_efd[MAXG], s_xid[MAXG];
  const DevGrid& g = A.g;
  const int G = g.G, Gs = g.Gs, RS = G + 1, t = (int)threadIdx.x;
  const uint32_t ncell = (uint32_t)g.ncell;
  const uint32_t c0 = blockIdx.x * (uint32_t)CPL_THREADS, c = c0 + (uint32_t)t;
  const int nc = (int)min((uint32_t)CPL_THREADS, ncell - c0);
  const bool act = t < nc;
  for (int j = t; j <= Gs; j += CPL_THREADS) {
    s_ed[j] = A.gc->edge32[j];
    if (j < Gs) {
      s_ef[j] = A.gc->efac32[j];
      s_efd[j] = A.gc->efac[j];
      const double xi = g.xi0 * (1.0 / sqrt(A.gc->edge[j] * A.gc->edge[j + 1]));
      s_xid[j] = xi;
      s_xi[j] = (float)xi;
      s_xil[j] = (float)(xi - (double)s_xi[j]);
    }
  }
  const RowCopy rc(A.out + ((size_t)NG * ncell + (size_t)c0 * G), nc, G, RS);
  rc.run<true, false>(FXPR(A.out, (size_t)NG * ncell + (size_t)c0 * G, nc * G, A.n_state), srow);
  __syncthreads();
  float* const Em = srow + t * RS;
  float* const En = srow + (CPL_THREADS + t) * RS;
  float* const U = A.out;
  const uint32_t XO = (uint32_t)(NG + (1 + D) * G) * ncell;
  unsigned st = 0;
  double rho = 1.0, m[D], hq[D], ke = 0.0, ue = 0.0, T = 1.0, Xn = 0.0, kpre = 0.0, fadd = 0.0;
#pragma unroll
  for (int q = 0; q < D; ++q) { m[q] = 0.0; hq[q] = 1.0; }
  const double cdt = A.kd.cdts;
  if (act) {
    rho = U[FXI(c, A.n_state)];
    if (rho < g.rho_floor) { rho = g.rho_floor; st |= ST_FLOOR; }
    // scale factors h_0, h_1 of the cell (1 on Cartesian grids): momentum and flux are covariant
    if (g.geom != 0) {
      const int i3[3] = {(int)(c % (uint32_t)g.n[0]), (int)((c / (uint32_t)g.n[0]) % (uint32_t)g.n[1]), 0};
#pragma unroll
      for (int d = 0; d < D; ++d) {
        const Tab<float> td{A.tab[d], g.n[d] + 4, A.uniform[d] ? A.urow[d] : nullptr};
        hq[0] *= (double)td(T_HA, bc_pad(i3[d]));
        if (D > 1) hq[D > 1 ? 1 : 0] *= (double)td(T_HB, bc_pad(i3[d]));
      }
    }
    const double irho = rcp_any(rho);
#pragma unroll
    for (int q = 0; q < D; ++q) {
      m[q] = U[FXI((1 + q) * ncell + c, A.n_state)];
      const double vh = g.geom != 0 ? m[q] * irho / hq[q] : m[q] * irho;
      ke = fma(0.5 * rho * vh, vh, ke);
    }
    double u_m = (double)U[FXI((NG - 1) * ncell + c, A.n_state)] - ke;
    const double u_floor = A.kd.u_floor;
    if (u_m < u_floor) { u_m = u_floor; st |= ST_FLOOR; }
    const double X_m = U[FXI(XO + c, A.n_state)], Y_m = X_m * irho;
    // E^- with its silent floor, sum E^- and the tolerance's scale sum |xi| E^-
    FPair Es = {0.0f, 0.0f}, Ls = Es;
    const float flo = (float)g.E_floor;
    // (floored channels are rare: found by a minimum, and the energy the floor adds summed in FP64 apart
    // from the loop, where its conversions and sums would run for every channel)
    float least = Em[0];
    for (int k = 1; k < G; ++k) least = fminf(least, Em[k]);
    if (least < flo) {
#pragma unroll 1
      for (int k = 0; k < G; ++k)
        if (Em[k] < flo) {
          fadd += g.E_floor - (double)Em[k];
          Em[k] = flo;
        }
    }
    for (int gg = 0; gg < Gs; ++gg) {
#pragma unroll
      for (int s = 0; s < 3; ++s) {
        const float e = Em[s * Gs + gg];
        acc(Es, e);
        if (s < 2) acc_mul(Ls, s_xi[gg], s_xil[gg], e);
      }
    }
    kpre = A.kd.kappa0 * hpow(rho, g.kap_rho_h);
    const float kpref = to_f32(kpre), cdtf = A.kf.cdts;
    const double rcv = rho * A.kd.cv;
    // residuals r_E, r_X and dr_E/dT, dr_X/dT, dr_X/dY at (T, Y); the channel energies into En
    auto eval = [&](double Tq, double Yq, double& rE, double& rX, double& JT, double& JX, double& JY) {
      const float Tf = to_f32(Tq), Yf = to_f32(Yq);
      const PlanckAt pa = planck_at(A.ptab, A.kf.aN, Tf);
      const float kTf = cdtf * (kpref * hpow(Tf, g.kap_T_h)), hTf = 0.5f * (float)g.kap_T_h * pa.invT;
      const float w0 = 2.0f * Yf, w1 = 2.0f * (1.0f - Yf);
      FPair dE = {0.0f, 0.0f}, dX = dE, eT = dE, xT = dE, xY = dE;
      F2 B2(0.0f), dB2(0.0f);
      for (int gg = 0; gg < Gs; ++gg) {
        if ((gg & 1) == 0) planck_pair(A.ptab, pa, gg >> 1, Gs, s_ed, B2, dB2);
        const float Bf = gg & 1 ? B2.y : B2.x, dBf = gg & 1 ? dB2.y : dB2.x;
        const float tf = kTf * s_ef[gg], invf = frcp(1.0f + tf), xf = s_xi[gg];
        float d[3], dt_[3];
#pragma unroll
        for (int s = 0; s < 3; ++s) {
          const int k = s * Gs + gg;
          const float w = s == 0 ? w0 : (s == 1 ? w1 : 1.0f);
          const float Emk = Em[k], Eq = w * Bf;
          const float Ek = fmaf(tf, Eq, Emk) * invf;
          dt_[s] = tf * fmaf(hTf, Eq - Ek, w * dBf) * invf;
          d[s] = Ek - Emk;
          En[k] = Ek;
        }
        acc(dE, d[0] + d[1] + d[2]);
        acc(dX, xf * (d[1] - d[0]));
        acc(eT, dt_[0] + dt_[1] + dt_[2]);
        acc(xT, xf * (dt_[1] - dt_[0]));
        acc(xY, -4.0f * xf * (tf * Bf * invf));
      }
      rE = fma(rcv, Tq, -u_m) + val(dE);
      rX = fma(rho, Yq - Y_m, -val(dX));
      JT = rcv + val(eT);
      JX = -val(xT);
      JY = rho - val(xY);
    };
    // stopping tests at FP32 resolution (relative step 2e-7 at least, residual 1e-7)
    const double rtol = A.kd.rtol, n2ok = A.kd.atol * A.kd.atol;
    const double isE = rcp_any(u_m + val(Es)), isX = rcp_any(fabs(X_m) + val(Ls) + 1e-300);
    auto norm2 = [&](double rE, double rX) { const double a = rE * isE, b = rX * isX; return fma(a, a, b * b); };
    double Y = Y_m, rE, rX, JT, JX, JY;
    T = u_m * rcp_any(rcv);
    eval(T, Y, rE, rX, JT, JX, JY);
    bool ok = false, fresh = true;  // fresh: En holds the energies at (T, Y)
    double n0 = norm2(rE, rX);
    for (int it = 0; it < g.newton_maxit; ++it) {
      if (n0 <= n2ok) { ok = true; break; }
      const double dT = -rE * rcp_any(JT), dY = -fma(JX, dT, rX) * rcp_any(JY);
      if (fabs(dT) <= rtol * T && fabs(dY) <= rtol * fmax(Y, 1e-3)) {
        T = T + dT;
        Y = Y + dY;
        ok = true;
        fresh = false;
        break;
      }
      double lam = 1.0;
      bool got = false;
      for (int ls = 0; ls < 40; ++ls) {
        const double Tt = fma(lam, dT, T), Yt = fma(lam, dY, Y);
        if (Tt > 0.0 && Yt >= 0.0 && Yt <= 1.0) {
          double rEt, rXt, JTt, JXt, JYt;
          eval(Tt, Yt, rEt, rXt, JTt, JXt, JYt);
          const double nt = norm2(rEt, rXt);
          fresh = false;
          if (nt < n0) {
            T = Tt; Y = Yt; rE = rEt; rX = rXt; JT = JTt; JX = JXt; JY = JYt; n0 = nt;
            got = fresh = true;
            break;
          }
        }
        lam *= 0.5;
      }
      if (!got) break;
    }
    if (!ok) {
      // alternating bisections (reading R33)
      for (int round = 0; round < 20 && !ok; ++round) {
        double r1, r2, rh, rm, j0, j1, j2;
        double lo = 0.5 * T, hi = 2.0 * T;
        eval(lo, Y, r1, r2, j0, j1, j2);
        for (int k = 0; k < 200 && r1 > 0.0; ++k) { lo = 0.5 * lo; eval(lo, Y, r1, r2, j0, j1, j2); }
        eval(hi, Y, rh, r2, j0, j1, j2);
        for (int k = 0; k < 200 && rh < 0.0; ++k) { hi = 2.0 * hi; eval(hi, Y, rh, r2, j0, j1, j2); }
        for (int k = 0; k < g.bisect_maxit && hi - lo > rtol * hi; ++k) {
          const double mid = 0.5 * (lo + hi);
          eval(mid, Y, rm, r2, j0, j1, j2);
          if (rm > 0.0) hi = mid; else lo = mid;
        }
        T = 0.5 * (lo + hi);
        double ylo = 0.0, yhi = 1.0;
        for (int k = 0; k < g.bisect_maxit && yhi - ylo > rtol; ++k) {
          const double mid = 0.5 * (ylo + yhi);
          eval(T, mid, r1, rm, j0, j1, j2);
          if (rm > 0.0) yhi = mid; else ylo = mid;
        }
        Y = 0.5 * (ylo + yhi);
        eval(T, Y, rE, rX, j0, j1, j2);
        if (norm2(rE, rX) <= n2ok) ok = true;
      }
      fresh = true;
      if (!ok) st |= ST_NEWTON;
    }
    if (!fresh) eval(T, Y, rE, rX, JT, JX, JY);
    // u and rho Y_e by conservation from the accepted channel energies
    FPair dE = {0.0f, 0.0f};
    Xn = X_m;
    for (int gg = 0; gg < Gs; ++gg) {
      FPair d = {0.0f, 0.0f};  // the group's anti-nu_e less nu_e changes
#pragma unroll
      for (int s = 0; s < 3; ++s) {
        const float e1 = En[s * Gs + gg], e0 = Em[s * Gs + gg];
        acc_diff(dE, e1, e0);
        if (s == 0) acc_diff(d, e0, e1);
        if (s == 1) acc_diff(d, e1, e0);
      }
      Xn = fma(s_xid[gg], val(d), Xn);
    }
    ue = ke + (u_m - val(dE));
  }
  __syncthreads();
  // the new E back, then the F rows into the same shared rows
  rc.run<false, false>(FXPR(A.out, (size_t)NG * ncell + (size_t)c0 * G, nc * G, A.n_state), srow + CPL_THREADS * RS);
  __syncthreads();
#pragma unroll
  for (int q = 0; q < D; ++q)
    rc.run<true, false>(FXPR(A.out, (size_t)NG * ncell + ((size_t)(1 + q) * ncell + c0) * G, nc * G, A.n_state), srow + q * CPL_THREADS * RS);
  __syncthreads();
  double dwork = 0.0;
  if (act) {
    // flux absorption (Eq. 28) with its momentum and energy feedback (Eqs. 31-32)
    FPair dm[D];
#pragma unroll
    for (int q = 0; q < D; ++q) dm[q] = {0.0f, 0.0f};
    const double sig = g.sigma0 * rho, kT = kpre * hpow(T, g.kap_T_h);
    for (int gg = 0; gg < Gs; ++gg) {
      const double x = fma(cdt, fma(kT, s_efd[gg], sig), 1.0);
      const float xh = to_f32(x), xl = to_f32(x - (double)xh);
      // 1/x = fh + fl (0 where x is past FP32's range: its float is infinite there)
      const float fh = frcp(xh), fl = fh > 0.0f ? fh * (fmaf(-xh, fh, 1.0f) - xl * fh) : 0.0f;
#pragma unroll
      for (int s = 0; s < 3; ++s) {
#pragma unroll
        for (int q = 0; q < D; ++q) {
          float* const r = srow + (q * CPL_THREADS + t) * RS + s * Gs + gg;
          const float F = *r, Fn = fmaf(F, fh, F * fl);
          acc_diff(dm[q], Fn, F);
          *r = Fn;
        }
      }
    }
    const double ic2 = A.kd.ic2, irho = rcp_any(rho);
    double mn[D];
    bool bad = false;
#pragma unroll
    for (int q = 0; q < D; ++q) {
      const double d = val(dm[q]), v = g.geom != 0 ? m[q] * irho / (hq[q] * hq[q]) : m[q] * irho;
      dwork = fma(v, d, dwork);
      mn[q] = fma(-d, ic2, m[q]);
      bad |= !isfinite(mn[q]);
    }
    ue -= dwork * ic2;
    A.out[FXI(c, A.n_state)] = (float)rho;
#pragma unroll
    for (int q = 0; q < D; ++q) A.out[FXI((1 + q) * ncell + c, A.n_state)] = (float)mn[q];
    A.out[FXI((NG - 1) * ncell + c, A.n_state)] = (float)ue;
    A.out[FXI(XO + c, A.n_state)] = (float)Xn;
    bad |= !isfinite(ue) || !isfinite(Xn);
    if (bad) st |= ST_NONFINITE;
    if (st) atomicOr(A.status, st);
    if (A.budget != nullptr) {
      const double wv = cell_volume(A, c) * A.bw_cpl;
      double* row = A.budget + (size_t)(blockIdx.x % BUDGET_SLOTS) * NBUDGET;
      if (dwork != 0.0) atomicAdd(row + 6, dwork * ic2 * wv);
      if (fadd != 0.0) atomicAdd(row + 7, fadd * wv);
    }
  }
  __syncthreads();
#pragma unroll
  for (int q = 0; q < D; ++q)
    rc.run<false, false>(FXPR(A.out, (size_t)NG * ncell + ((size_t)(1 + q) * ncell + c0) * G, nc * G, A.n_state), srow + q * CPL_THREADS * RS);
}

}  // namespace fx
