// Hand-written adjoint of one SSP-RK2 stage (Cartesian grids).
//
// A stage maps (U_in, U_base) to U_out in three parts, and its adjoint runs them backwards:
//   forward                                             adjoint (this file)
//   L = -(1/V) sum_faces A F(U_in)   (Sec. 4, Eq. 8)    adj_rad_kernel, adj_gas_kernel
//   U_pre = a U_base + b (U_in + dt L)   (Sec. 4)       adj_cell_kernel: RK weights, prim -> cons
//   U_out = C(U_pre), the interaction (Sec. 5.3)        adj_couple_kernel: implicit function rule
// Given lam_out = dJ/dU_out the kernels produce dJ/dU_in, dJ/dU_base and the kappa0 derivative.
// The objective J (boundary energy outflow) enters as a source on the adjoint of the upper-x
// boundary fluxes.  The forward state of the stage (U_pre and the converged temperature) is
// recorded by the forward kernel during the recomputation of each checkpoint segment.
//
// The interaction's derivative follows from the implicit function theorem on the Newton
// residual r(T) = rho c_v T - u^- + sum_g (E_g(T) - E_g^-) (Eqs. 25-27): dT = -(dr/dtheta)/(dr/dT).
// The flux functions are differentiated in reverse, each by one pass forward and one backwards over its
// operations (hllc_adjoint, m1_adjoint); the reconstructions are linear forms on each of their
// branches (mc_form, parabola_form).  Every branch is the one that the forward functions of
// fx_device.cuh take, so that the gradient is the exact derivative of the step as computed.
#pragma once
#include "fx_stage.cuh"

namespace fx {

template <class R> struct AdjArgs {
  DevGrid g;
  const R* tab[3];
  R urow[3][NTAB];
  int uniform[3];
  const GroupConst* gc;
  PlanckParams pk;
  PlanckTable ptab;
  const R* in;        // stage input U_in (state layout)
  const R* pre;       // recorded pre-interaction state
  const R* tstar;     // recorded interaction temperature [ncell]
  const R* lam_out;   // dJ/dU_out
  R* lam_pre;         // dJ/dU_pre (written by adj_couple_kernel)
  R* lvs;             // adjoint of each face's contact speed (adj_rad_kernel; the space of the face
                      // records, which the stage kernels write anew)
  int64_t lvs_off[3]; // first face of each direction in `lvs`
  R* lam_w;           // primitive adjoints accumulated by adj_rad_kernel and adj_gas_kernel:
                      //   gas [2+D][ncell] (rho, p, v_0..v_{D-1}), radiation [1+D][ncell][G]
                      //   (E, F_0..), total opacity [ncell][G]
  R* lam_in;          // dJ/dU_in (adj_cell_kernel; accumulated when accumulate_in)
  R* lam_base;        // dJ/dU_base (stage 2; written)
  double* kpart;      // one partial dJ/dkappa0 per block, added to by every stage
  int accumulate_in;
  double dt, alpha;   // stage step and RK weight of U_base
  R wJ;               // weight of the boundary outflow of this stage in J (dt/2; 0 if unused)
#ifdef FX_BOUNDS_CHECK
  unsigned* status;   // status word, and the elements of a state, for the index checks of the
  int64_t n_state, n_lvs;  // debug build
#endif
  R phi_area;         // area of one upper-x boundary face
  Consts<double> kd;
  Consts<float> kf;
  __device__ __forceinline__ const Consts<double>& k(double) const { return kd; }
  __device__ __forceinline__ const Consts<float>& k(float) const { return kf; }
};

// Block sum of one double per thread (only lanes that carry a value contribute) added to
// kpart[blockIdx.x]; 256 threads.  A warp without any value (busy, the same for its lanes) skips the
// sum over its lanes: five FP64 additions of 16 cycles each, which were 40 % of the time of blocks that have
// nothing else to do (512^2 x 8: 34 -> 20 us per launch).
__device__ __forceinline__ void block_partial(double v, double* kpart, bool busy = true) {
  __shared__ double red[8];
  if (busy) {
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  }
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
    double s = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += red[w];
    if (nonzero(s)) kpart[blockIdx.x] += s;
  }
}

// ---------------------------------------------------------------------------------------------
// Adjoint of the interaction (energy: Eqs. 25-27, R12; momentum: Eqs. 28, 31-32).  One cell per
// segment of GP lanes, lane = group; lanes < 2+D also carry one gas variable.
// ---------------------------------------------------------------------------------------------
template <class R, int D, int GP>
__global__ void __launch_bounds__(256) adj_couple_kernel(const __grid_constant__ AdjArgs<R> A) {
  constexpr int NG = 2 + D;
  const DevGrid& g = A.g;
  const Consts<R>& KR = A.k(R(0));
  const int G = g.G;
  const int lane = threadIdx.x % GP;
  const int64_t cr = (int64_t)blockIdx.x * (256 / GP) + threadIdx.x / GP;
  const bool active = cr < g.ncell;
  const uint32_t ncell = (uint32_t)g.ncell;
  const uint32_t c = active ? (uint32_t)cr : ncell - 1;
  const bool has = lane < G;
  const int gl = has ? lane : 0;
  const int gv = lane < NG ? lane : 0;

  R u[NG], lo[NG], lEo = R(0), lFo[3] = {R(0), R(0), R(0)};
  const R lgas = A.lam_out[FXI(gv * ncell + c, A.n_state)];
  bool any = nonzero(lgas);
  if (has) {
    lEo = A.lam_out[FXI(NG * ncell + c * G + gl, A.n_state)];
    any = any || nonzero(lEo);
#pragma unroll
    for (int q = 0; q < D; ++q) {
      lFo[q] = A.lam_out[FXI(NG * ncell + ((1 + q) * ncell + c) * G + gl, A.n_state)];
      any = any || nonzero(lFo[q]);
    }
  }
  double lk = 0.0;  // the cell's dJ/dkappa0
  const bool busy = g.couple && __any_sync(0xffffffffu, any);
  if (!g.couple) {  // no interaction: U_out = U_pre
    if (active) {
      if (lane < NG) A.lam_pre[FXI(lane * ncell + c, A.n_state)] = A.lam_out[FXI(lane * ncell + c, A.n_state)];
      if (has) {
        A.lam_pre[FXI(NG * ncell + c * G + gl, A.n_state)] = lEo;
#pragma unroll
        for (int q = 0; q < D; ++q) A.lam_pre[FXI(NG * ncell + ((1 + q) * ncell + c) * G + gl, A.n_state)] = lFo[q];
      }
    }
  } else if (!busy) {
    // where nothing depends on the outputs of the warp's cells, nothing does on their inputs
    if (active) {
      if (lane < NG) A.lam_pre[FXI(lane * ncell + c, A.n_state)] = R(0);
      if (has) {
#pragma unroll
        for (int v = 0; v < 1 + D; ++v) A.lam_pre[FXI(NG * ncell + (v * ncell + c) * G + gl, A.n_state)] = R(0);
      }
    }
  } else {
    const R ugas = A.pre[FXI(gv * ncell + c, A.n_state)];
#pragma unroll
    for (int v = 0; v < NG; ++v) {
      u[v] = __shfl_sync(0xffffffffu, ugas, v, GP);
      lo[v] = __shfl_sync(0xffffffffu, lgas, v, GP);
    }
    R E = R(0), F[3] = {R(0), R(0), R(0)};
    if (has) {
      E = A.pre[FXI(NG * ncell + c * G + gl, A.n_state)];
#pragma unroll
      for (int q = 0; q < D; ++q) F[q] = A.pre[FXI(NG * ncell + ((1 + q) * ncell + c) * G + gl, A.n_state)];
    }
    // the interaction's silent positivity floor on E_g^-: a floored group's energy does not depend
    // on its input
    const bool floored = has && E < KR.E_floor;
    if (floored) E = KR.E_floor;
    const R T = A.tstar[FXI(c, ncell)], iT = rcp_any(T);
    const R rho = u[0], irho = rcp_any(rho), rhoe = u[NG - 1];
    R m[3] = {R(0), R(0), R(0)}, ke = R(0);
#pragma unroll
    for (int q = 0; q < D; ++q) { m[q] = u[1 + q]; ke += R(0.5) * m[q] * m[q] * irho; }
    const R ra = R(0.5) * R(g.kap_rho_h), tb = R(0.5) * R(g.kap_T_h);
    const R K0 = hpow(rho, g.kap_rho_h) * hpow(T, g.kap_T_h);  // kappa / (kappa0 eps^d)
    const GroupConst& gc = *A.gc;
    const R ef = has ? R(gc.efac_of(gl, R(0))) : R(0);
    const R kap = KR.kappa0 * K0 * ef;
    const R cdts = KR.cdts;
    const R tau = cdts * kap;
    const R i1 = rcp_any(R(1) + tau);
    // Planck group energy and its T derivative at the converged temperature
    R B, dB;
    {
      LanePlanck<GP, R> cp{A.pk, A.ptab, lane, has, (G == GP) && (lane == G - 1), KR.aN,
                           R(gc.edge_of(lane <= G ? lane : G, R(0))), R(gc.edge_of(lane < G ? lane + 1 : G, R(0)))};
      cp.planck(T, iT, B, dB);
      if (!has) { B = R(0); dB = R(0); }
    }
    const R Ep = (E + tau * B) * i1;
    const R fac = rcp_any(R(1) + cdts * (kap + KR.sigma0 * rho));
    R SdF[3] = {R(0), R(0), R(0)};
#pragma unroll
    for (int q = 0; q < D; ++q) SdF[q] = seg_sum<GP>(has ? F[q] * (fac - R(1)) : R(0));

    const R ic2 = KR.ic2;
    const R lre_o = lo[NG - 1];
    // rho e' = rho e - sum_g (E'_g - E_g) - ic2 sum_q (m_q / rho) sum_g dF_gq;  m'_q = m_q - ic2 sum_g dF_gq
    R lrho = lo[0], lm[3] = {R(0), R(0), R(0)}, ldF[3] = {R(0), R(0), R(0)};
#pragma unroll
    for (int q = 0; q < D; ++q) {
      ldF[q] = -ic2 * (lo[1 + q] + m[q] * irho * lre_o);
      lm[q] = lo[1 + q] - ic2 * SdF[q] * irho * lre_o;
      lrho += ic2 * m[q] * SdF[q] * irho * irho * lre_o;
    }
    // F' = F fac, dF = F (fac - 1)
    R lF[3] = {R(0), R(0), R(0)}, lfac = R(0);
#pragma unroll
    for (int q = 0; q < D; ++q) {
      lF[q] = lFo[q] * fac + ldF[q] * (fac - R(1));
      lfac += F[q] * (lFo[q] + ldF[q]);
    }
    // fac = 1 / (1 + cdts (kappa + sigma0 rho))
    R lkap = -fac * fac * cdts * lfac;
    lrho += KR.sigma0 * seg_sum<GP>(has ? lkap : R(0));
    // energy: E'_g = (E_g + tau B)/(1 + tau) at T*
    R lrhoe = lre_o;
    const R lEp = lEo - lre_o;
    R lE = lre_o + lEp * i1;
    const R ltau = lEp * (B - Ep) * i1;
    R lT = seg_sum<GP>(has ? lEp * tau * i1 * dB : R(0));
    lkap += ltau * cdts;
    // kappa = kappa0 K0(rho, T) eps^d
    const R Slk = seg_sum<GP>(has ? lkap * kap : R(0));
    lrho += ra * Slk * irho;
    lT += tb * Slk * iT;
    R lk0 = seg_sum<GP>(has ? lkap * K0 * ef : R(0));
    // T* from r(T*; rho, u^-, E^-, kappa0) = 0
    const R dtau = tau * tb * iT;
    const R drdT = rho * KR.cv + seg_sum<GP>(has ? (tau * dB + dtau * (B - Ep)) * i1 : R(0));
    const R lr = -lT * rcp_any(drdT);
    const R Sb = seg_sum<GP>(has ? (B - Ep) * i1 * tau : R(0));
    lrho += lr * (KR.cv * T + ra * Sb * irho);
    const R lum = -lr;
    lE += lr * (-tau * i1);
    lk0 += lr * seg_sum<GP>(has ? (B - Ep) * i1 * cdts * K0 * ef : R(0));
    // u^- = rho e - |m|^2 / (2 rho)
    lrhoe += lum;
#pragma unroll
    for (int q = 0; q < D; ++q) lm[q] -= lum * m[q] * irho;
    lrho += lum * ke * irho;

    if (active) {
      if (lane < NG) {
        R val = lrho;
#pragma unroll
        for (int q = 0; q < D; ++q) if (lane == 1 + q) val = lm[q];
        if (lane == NG - 1) val = lrhoe;
        A.lam_pre[FXI(lane * ncell + c, A.n_state)] = val;
      }
      if (has) {
        A.lam_pre[FXI(NG * ncell + c * G + gl, A.n_state)] = floored ? R(0) : lE;
#pragma unroll
        for (int q = 0; q < D; ++q) A.lam_pre[FXI(NG * ncell + ((1 + q) * ncell + c) * G + gl, A.n_state)] = lF[q];
      }
    }
    if (active && lane == 0) lk = (double)lk0;
  }
  block_partial(lk, A.kpart, busy);
}

// Adjoint of the M1 pressure row n at the state Q = (E, F): adds sum_q lam_q dP_nq/dQ to lQ (lam in
// units where P is c^2 P).  P is homogeneous of degree one in (E, F), so below the free-streaming
// limit everything is formed at the normalised state psi = F/(cE): with f^2 = psi.psi,
// s = sqrt(4 - 3f^2), q = 1/(2+s), a = lam_n and b = lam.psi the row's weighted sum is
//   Phi' = a (1/3 - f^2 q) + 3 q psi_n b,
// its derivative along f^2, with dq/df^2 = 3 q^2/(2s), H = -a (q + f^2 dq) + 3 psi_n b dq, and so
//   dPhi'/dpsi_j = 2 H psi_j + 3 q (psi_n lam_j + delta_jn b),  dPhi/dE = Phi' - psi.dPhi'/dpsi,
// which keeps FP32 finite for the tiny E_g of cold groups (1/E^2 would overflow), needs no special
// case at F = 0, and at E <= 0 (isotropic branch: psi = 0) leaves a/3.  One pass backwards over the
// row takes a third of the operations of its Jacobian in three tangent directions.  Where |F| > cE the
// closure clamps f to 1 and P = E n n with n = F/|F|; that branch is written out.
__device__ __forceinline__ double rcp_energy(double E) {
  const int hi = __double2hiint(E);
  return hi >= 0x00400000 && hi < 0x7fb00000 ? rcp64(E) : (E > 0.0 ? fmin(1.0 / E, 1e308) : 0.0);
}
__device__ __forceinline__ float rcp_energy(float E) { return E > 0.0f ? fminf(rcp_approx(E), 3e38f) : 0.0f; }
template <class R, int D>
__device__ __forceinline__ void m1_adjoint(R c, R ic, const R* Q, int n, const R* lam, R* lQ) {
  const R iE = rcp_energy(Q[0]);
  R psi[D], f2 = R(0), b = R(0);
#pragma unroll
  for (int q = 0; q < D; ++q) {
    psi[q] = Q[1 + q] * iE * ic;
    f2 += psi[q] * psi[q];
    b += lam[q] * psi[q];
  }
  bool clamped = f2 > R(1);
  if (clamped || f2 > R(1) - R(1e-5)) {
    // f = |F| / (cE) = (smax un / E) / c, compared with 1 without forming |F|^2 / E^2
    R smax = R(0), u[D], un2 = R(0);
#pragma unroll
    for (int q = 0; q < D; ++q) smax = fmax(smax, fabs(Q[1 + q]));
#pragma unroll
    for (int q = 0; q < D; ++q) { u[q] = Q[1 + q] / smax; un2 += u[q] * u[q]; }
    const R un = sqrt(un2);
    clamped = smax * un > c * Q[0];
    if (clamped) {
      const R EoF = Q[0] / (smax * un);
      R nv[D], bn = R(0);
#pragma unroll
      for (int q = 0; q < D; ++q) { nv[q] = u[q] / un; bn += lam[q] * nv[q]; }
      lQ[0] += nv[n] * bn;
#pragma unroll
      for (int j = 0; j < D; ++j)
        lQ[1 + j] += EoF * ((j == n ? bn : R(0)) + nv[n] * lam[j] - R(2) * nv[n] * bn * nv[j]);
      return;
    }
    f2 = f2 > R(1) ? R(1) : f2;
  }
  const R sq = sqrt_any(R(4) - R(3) * f2), qd = rcp_any(R(2) + sq), dq = R(1.5) * qd * qd * rcp_any(sq);
  const R a = lam[n], pn = psi[n], t3 = R(3) * qd;
  const R H2 = R(2) * (R(3) * pn * b * dq - a * (qd + f2 * dq));
  R gE = a * (R(1.0 / 3.0) - f2 * qd) + t3 * pn * b;
#pragma unroll
  for (int j = 0; j < D; ++j) {
    const R gj = H2 * psi[j] + t3 * (pn * lam[j] + (j == n ? b : R(0)));
    gE -= psi[j] * gj;
    lQ[1 + j] += ic * gj;
  }
  lQ[0] += gE;
}

// The face value p0 + s d of the MC-limited slope s at the offset d from the centroid, and the
// branch's derivatives k by the three values (the middle one is formed as 1 + ds/dp0 d before it
// meets an adjoint, so that a weight that vanishes does so exactly).
template <class R>
__device__ __forceinline__ R mc_form(const MCCoef<R>& c, R d, R pm, R p0, R pp, R* k) {
  const R sL = (p0 - pm) * c.il, sR = (pp - p0) * c.ir, sC = (pp - pm) * c.ic;
  const bool any = same_sign(sL, sR), right = cmp_abs(sR, sL) < 0;
  const R s2 = R(2) * (right ? sR : sL);
  const bool cen = cmp_abs(sC, s2) < 0;
  const R w = any ? (cen ? c.ic : R(2) * (right ? c.ir : c.il)) * d : R(0);
  k[0] = cen || !right ? -w : R(0);
  k[1] = cen ? R(1) : (right ? R(1) - w : R(1) + w);
  k[2] = cen || right ? w : R(0);
  return p0 + (any ? cen ? sC : s2 : R(0)) * d;
}

// The parabolic reconstruction's face values a (lower) and b (upper) of one variable
// (recon_parabolic) with the derivatives of one of them, the upper one if `up`, by the three
// values: each branch is a linear form, so its weights are selects of table entries and a handful of
// operations instead of tangents carried through every branch.
template <class R>
__device__ __forceinline__ R parabola_form(const Tab<R>& t, int ip, bool up, R pm, R p0, R pp, R* k) {
  const R dl = p0 - pm, dr = pp - p0;
  R ka[3] = {t(T_WA0, ip), t(T_WA1, ip), t(T_WA2, ip)}, kb[3] = {t(T_WB0, ip), t(T_WB1, ip), t(T_WB2, ip)};
  R a = ka[0] * pm + ka[1] * p0 + ka[2] * pp, b = kb[0] * pm + kb[1] * p0 + kb[2] * pp;
  {
    const R s = t(T_SL2, ip), u = t(T_TL2, ip), x = pm + dl * s, y = p0 - dl * u, m = median(a, x, y);
    if (differ(m, a)) {
      const bool first = !differ(m, x);
      ka[0] = first ? R(1) - s : u;
      ka[1] = first ? s : R(1) - u;
      ka[2] = R(0);
    }
    a = m;
  }
  {
    const R s = t(T_SR2, ip), u = t(T_TR2, ip), x = p0 + dr * s, y = pp - dr * u, m = median(b, x, y);
    if (differ(m, b)) {
      const bool first = !differ(m, x);
      kb[0] = R(0);
      kb[1] = first ? R(1) - s : u;
      kb[2] = first ? s : R(1) - u;
    }
    b = m;
  }
  const R sl = t(T_AL0, ip) * a + t(T_AL1, ip) * p0 + t(T_AL2, ip) * b;
  const R sr = t(T_AR0, ip) * a + t(T_AR1, ip) * p0 + t(T_AR2, ip) * b;
  const bool inc = opposite_sign(sl, sr);  // extremum inside the cell
  const int cmp = cmp_abs(sl, sr);
  const bool flat = !same_sign(dl, dr) || (inc && cmp == 0), reset = inc && (up ? cmp < 0 : cmp > 0);
  // the wanted face's value, or where its end slope is the one reset, the other's moved towards p0
  const R rh = t(up ? T_RHL : T_RHR, ip);
  const bool fb = up != reset;  // start from b
  R v = fb ? b : a;
#pragma unroll
  for (int m = 0; m < 3; ++m) k[m] = fb ? kb[m] : ka[m];
  if (reset) {
    v = v + (p0 - v) * rh;
#pragma unroll
    for (int m = 0; m < 3; ++m) k[m] = k[m] + ((m == 1 ? R(1) : R(0)) - k[m]) * rh;
  }
#pragma unroll
  for (int m = 0; m < 3; ++m) k[m] = flat ? (m == 1 ? R(1) : R(0)) : k[m];
  return flat ? p0 : v;
}

// ---------------------------------------------------------------------------------------------
// Adjoint of the face fluxes: the reconstructed states and fluxes of each face recomputed from the
// stage input, the flux adjoints taken from the two adjacent cells (and the objective at the
// upper-x boundary), and the adjoints of the four stencil cells' primitives and of the two cells'
// opacities scattered (atomics; ghost positions land on the cells they mirror, with the sign of
// mirrored normal components).  Two kernels, because the two parts want different threads:
//   adj_rad_kernel   one thread per face and group (runs of groups are contiguous: coalesced reads and
//                    atomics); the contact speed and opacity factors of a block's faces are
//                    computed by one thread per face first, and the adjoint of the contact speed is summed
//                    over the groups at the end and left in the face records' space;
//   adj_gas_kernel   one thread per face.
// A block, or a face of the gas kernel, whose flux adjoints all vanish is done at once: the objective sits on
// one boundary, so after n steps back only its neighbourhood has any.  Bound by the FP64 pipe where all
// faces have adjoints and by the latency of a block's chains on small grids (128 x 96 x 8 FP64: 61 and
// 42 us per launch).  One thread per face that looped over the groups and carried the tangents of
// both sides in forward mode held 255 registers, kept the pipe half busy and took 287 us; the two kernels
// without the early end and with HLLC in forward mode took 96 and 94 us.  Radiation blocks of 256
// threads take 76 us (the few busy blocks crowd some multiprocessors), of 64 threads 61 (as long: the
// gas values of 8 faces occupy a whole warp).
// ---------------------------------------------------------------------------------------------
constexpr int ADJ_RAD_THREADS = 128, ADJ_GAS_THREADS = 64;

// Position of face f of direction DIR: its index along DIR, and the stencil cells id-2 .. id+1 with
// the flips of mirrored ones.
template <int DIR>
__device__ __forceinline__ int adj_face_cells(const DevGrid& g, uint32_t f, uint32_t* ci, bool* fl) {
  const int n0 = g.n[0], n1 = g.n[1], nd = g.n[DIR];
  const uint32_t ex = (uint32_t)(n0 + (DIR == 0)), ey = (uint32_t)(n1 + (DIR == 1));
  const int i0 = (int)(f % ex), i1 = (int)((f / ex) % ey), i2 = (int)(f / (ex * ey));
  const int id = DIR == 0 ? i0 : (DIR == 1 ? i1 : i2);
#pragma unroll
  for (int m = 0; m < 4; ++m) {
    bool flip = false;
    const int cd = min(max(bc_map(id - 2 + m, nd, g.bc_lo[DIR], g.bc_hi[DIR], flip), 0), nd - 1);
    const int c0 = DIR == 0 ? cd : i0, c1 = DIR == 1 ? cd : i1, c2 = DIR == 2 ? cd : i2;
    ci[m] = ((uint32_t)c2 * n1 + c1) * n0 + c0;
    fl[m] = flip;
  }
  return id;
}
__host__ __device__ inline uint32_t adj_faces(const DevGrid& g, int d) {
  return (uint32_t)(g.n[0] + (d == 0)) * (uint32_t)(g.n[1] + (d == 1)) * (uint32_t)(g.n[2] + (d == 2));
}

// Primitives (rho, p, v) of cell c of the stage input, the normal velocity mirrored with flip.
template <class R, int D, int DIR>
__device__ __forceinline__ void adj_prim(const AdjArgs<R>& A, uint32_t c, bool flip, R* W) {
  constexpr int NG = 2 + D;
  const uint32_t ncell = (uint32_t)A.g.ncell;
  const Consts<R>& KR = A.k(R(0));
  R u[NG];
#pragma unroll
  for (int v = 0; v < NG; ++v) u[v] = A.in[FXI(v * ncell + c, A.n_state)];
  if (flip) u[1 + DIR] = -u[1 + DIR];
  const R rho = u[0], irho = rcp_any(rho);
  R ke = R(0);
#pragma unroll
  for (int q = 0; q < D; ++q) { W[2 + q] = u[1 + q] * irho; ke += u[1 + q] * W[2 + q]; }
  W[0] = rho;
  W[1] = KR.gm1 * (u[NG - 1] - R(0.5) * ke);
}

template <class R, int D, int DIR>
__device__ __forceinline__ void adj_rad_tile(const AdjArgs<R>& A, R (*sf)[ADJ_RAD_THREADS], R* sl) {
  constexpr int NG = 2 + D, NW = 2 + D, NRV = 1 + D;
  const DevGrid& g = A.g;
  const Consts<R>& KR = A.k(R(0));
  const int G = g.G, F = ADJ_RAD_THREADS / G, tid = (int)threadIdx.x, nd = g.n[DIR];
  const uint32_t ncell = (uint32_t)g.ncell, nf = adj_faces(g, DIR), f0 = blockIdx.x * (uint32_t)F;
  if (f0 >= nf) return;
  const Tab<R> t{A.tab[DIR], nd + 4, A.uniform[DIR] ? A.urow[DIR] : nullptr};
  // ---- flux adjoints of the thread's face and group; a block without any is done
  const int tf = tid / G, gg = tid - tf * G;
  const bool own = tf < F && f0 + tf < nf;
  uint32_t ci[4] = {0, 0, 0, 0};
  bool fl[4] = {false, false, false, false}, any = false;
  int id = 0;
  R lout[NRV];
#pragma unroll
  for (int v = 0; v < NRV; ++v) lout[v] = R(0);
  if (own) {
    id = adj_face_cells<DIR>(g, f0 + tf, ci, fl);
    // adjoint of the face flux of state variable j: dJ/dF = -b dt fr(L) lam_pre(L) + b dt fl(R) lam_pre(R)
    const bool inL = id >= 1, inR = id < nd;
    const R bdt = KR.beta * KR.dt;  // (1 - alpha) dt: the weights 1, 1/2 are exact in R
    const R cL = inL ? -bdt * t(T_FR, bc_pad(id - 1)) : R(0);
    const R cR = inR ? bdt * t(T_FL, bc_pad(id)) : R(0);
    const bool objective = DIR == 0 && id == nd && A.wJ != R(0);
    any = objective;
#pragma unroll
    for (int v = 0; v < NRV; ++v) {
      R lj = R(0);
      if (inL) lj += cL * A.lam_pre[FXI(NG * ncell + (v * ncell + ci[1]) * G + gg, A.n_state)];
      if (inR) lj += cR * A.lam_pre[FXI(NG * ncell + (v * ncell + ci[2]) * G + gg, A.n_state)];
      if (v == 0 && objective) lj += A.wJ * A.phi_area;
      lout[v] = lj;
      any = any || nonzero(lj);
    }
  }
  if (!__syncthreads_or(any)) {
    if (tid < F && f0 + tid < nf) A.lvs[FXI((uint32_t)A.lvs_off[DIR] + f0 + tid, A.n_lvs)] = R(0);
    return;
  }
  // ---- gas values of the block's faces: contact speed, and the opacity factors of the two adjacent
  // cells: K = kappa0 rho^a T^b (0 where T <= 0), S = sigma0 rho
  if (tid < F && f0 + tid < nf) {
    uint32_t ci[4];
    bool fl[4];
    const int id = adj_face_cells<DIR>(g, f0 + tid, ci, fl);
    R W[4][NW], Lr[NW], Rr[NW], fx_[NW], vs;
#pragma unroll
    for (int m = 0; m < 4; ++m) adj_prim<R, D, DIR>(A, ci[m], fl[m], W[m]);
#pragma unroll
    for (int v = 0; v < NW; ++v) {
      const int slot = v < 2 ? v : 2 + (v - 2 - DIR + D) % D;
      R x;
      recon_parabolic(t, bc_pad(id - 1), W[0][v], W[1][v], W[2][v], x, Lr[slot]);
      recon_parabolic(t, bc_pad(id), W[1][v], W[2][v], W[3][v], Rr[slot], x);
    }
    hllc<R, D>(KR.gamma, Lr, Rr, fx_, vs);
    sf[0][tid] = vs;
#pragma unroll
    for (int s = 0; s < 2; ++s) {
      const R rho = W[1 + s][0], T = W[1 + s][1] * rcp_any(rho);
      sf[1 + s][tid] = T > R(0) ? KR.kappa0 * hpow(rho, g.kap_rho_h) * hpow(T, g.kap_T_h) : R(0);
      sf[3 + s][tid] = KR.sigma0 * rho;
    }
  }
  __syncthreads();
  // ---- per group: forward face state and flux, then its adjoint
  R lvs = R(0);
  if (any) {
    const R vstar = sf[0][tf];
    R* const lw_rad = A.lam_w + (size_t)NW * ncell;
    R* const lw_chi = lw_rad + (size_t)NRV * ncell * G;
    R Q[4][NRV];
#pragma unroll
    for (int v = 0; v < NRV; ++v)
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        const R val = A.in[FXI(NG * ncell + (v * ncell + ci[m]) * G + gg, A.n_state)];
        Q[m][v] = (v == 1 + DIR && fl[m]) ? -val : val;
      }
    const MCCoef<R> mcL = mc_coef<R>(t, bc_pad(id - 1)), mcR = mc_coef<R>(t, bc_pad(id));
    R kL[NRV][3], kR[NRV][3], QL[NRV], QR[NRV];
#pragma unroll
    for (int v = 0; v < NRV; ++v) {
      QL[v] = mc_form(mcL, mcL.dr, Q[0][v], Q[1][v], Q[2][v], kL[v]);
      QR[v] = mc_form(mcR, mcR.dl, Q[1][v], Q[2][v], Q[3][v], kR[v]);
    }
    const R ef = R(A.gc->efac_of(gg, R(0)));
    const R chiL = sf[1][tf] * ef + sf[3][tf], chiR = sf[2][tf] * ef + sf[4][tf];
    const R ell = t(T_ELL, bc_pad(id));
    const R tau = R(0.5) * (chiL + chiR) * ell;
    const R eps = tau > R(1) ? rcp_any(tau) : R(1);
    const bool upL = nonneg(vstar);
    // transpose of the face formula (Eqs. 17-19; R8, R9)
    R lQL[NRV], lQR[NRV], lam[D];
    const R l0 = lout[0], hc0 = eps * KR.hc * l0;
    lQL[0] = hc0;
    lQR[0] = -hc0;
#pragma unroll
    for (int q = 0; q < D; ++q) {
      const R lq = lout[1 + q], h = KR.hc * lq, u = q == DIR ? R(0.5) * l0 : R(0);
      lam[q] = KR.hc2 * lq;
      lQL[1 + q] = u + h;
      lQR[1 + q] = u - h;
    }
#pragma unroll
    for (int v = 0; v < NRV; ++v) {
      const R lv = vstar * lout[v];
      lQL[v] += upL ? lv : R(0);
      lQR[v] += upL ? R(0) : lv;
      lvs += (upL ? QL[v] : QR[v]) * lout[v];
    }
    const R ic = KR.c * KR.ic2;
    m1_adjoint<R, D>(KR.c, ic, QL, DIR, lam, lQL);
    m1_adjoint<R, D>(KR.c, ic, QR, DIR, lam, lQR);
    if (tau > R(1)) {
      const R lchi = R(0.5) * ell * (KR.hc * (QR[0] - QL[0]) * l0) * eps * eps;
      if (nonzero(lchi)) {
        atomicAdd(FXP(lw_chi, (size_t)ci[1] * G + gg, (size_t)ncell * G), lchi);
        atomicAdd(FXP(lw_chi, (size_t)ci[2] * G + gg, (size_t)ncell * G), lchi);
      }
    }
    // reconstruction: left state from cells id-2..id, right state from id-1..id+1
#pragma unroll
    for (int v = 0; v < NRV; ++v) {
      const R l = lQL[v], r = lQR[v];
      const R lq[4] = {l * kL[v][0], l * kL[v][1] + r * kR[v][0], l * kL[v][2] + r * kR[v][1], r * kR[v][2]};
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        const R x = (v == 1 + DIR && fl[m]) ? -lq[m] : lq[m];
        if (nonzero(x)) atomicAdd(FXP(lw_rad, ((size_t)v * ncell + ci[m]) * G + gg, (size_t)NRV * ncell * G), x);
      }
    }
  }
  // ---- the contact speed's adjoint: the groups' terms summed in order
  sl[tid] = lvs;
  __syncthreads();
  if (tid < F && f0 + tid < nf) {
    R s = R(0);
    for (int j = 0; j < G; ++j) s += sl[tid * G + j];
    A.lvs[FXI((uint32_t)A.lvs_off[DIR] + f0 + tid, A.n_lvs)] = s;
  }
}

template <class R, int D>
__global__ void __launch_bounds__(ADJ_RAD_THREADS) adj_rad_kernel(const __grid_constant__ AdjArgs<R> A) {
  __shared__ R sf[5][ADJ_RAD_THREADS], sl[ADJ_RAD_THREADS];
  if (blockIdx.y == 0) adj_rad_tile<R, D, 0>(A, sf, sl);
  else if (D >= 2 && blockIdx.y == 1) adj_rad_tile<R, D, (D >= 2 ? 1 : 0)>(A, sf, sl);
  else if (D >= 3) adj_rad_tile<R, D, (D >= 3 ? 2 : 0)>(A, sf, sl);
}

// Adjoint of HLLC: bL, bR = the derivatives of lvs vstar + lf . f by the two states (hllc in
// fx_device.cuh, whose branches these are), by one pass forward and one backwards over its
// operations: an eighth of the work of carrying eight tangents.
template <class R, int D>
__device__ __forceinline__ void hllc_adjoint(R gam, const R* L, const R* Q, R lvs, const R* lf, R* bL, R* bR) {
  constexpr int NW = 2 + D;
  const R gm1 = gam - R(1), igm1 = rcp_any(gm1), half = R(0.5);
  const R rl = L[0], pl = L[1], ul = L[2], rr = Q[0], pr = Q[1], ur = Q[2];
  R kl = ul * ul, kr = ur * ur;
#pragma unroll
  for (int q = 1; q < D; ++q) { kl += L[2 + q] * L[2 + q]; kr += Q[2 + q] * Q[2 + q]; }
  const R El = pl * igm1 + half * rl * kl, Er = pr * igm1 + half * rr * kr;
  const R irl = rcp_any(rl), irr = rcp_any(rr);
  const R al = sqrt_any(gam * pl * irl), ar = sqrt_any(gam * pr * irr);
  const R sl = sqrt_any(rl), sr = sqrt_any(rr), iw = rcp_any(sl + sr);
  const R hl = (El + pl) * irl, hr = (Er + pr) * irr;
  const R Ht = (sl * hl + sr * hr) * iw;
  R X[D], v2 = R(0);  // density-weighted velocities
#pragma unroll
  for (int q = 0; q < D; ++q) { X[q] = (sl * L[2 + q] + sr * Q[2 + q]) * iw; v2 += X[q] * X[q]; }
  const R at2 = gm1 * (Ht - half * v2);
  const bool sonic = at2 > R(0);
  const R at = sonic ? sqrt_any(at2) : R(0);
  const bool avL = X[0] - at < ul - al, avR = X[0] + at > ur + ar;
  const R SL = avL ? X[0] - at : ul - al, SR = avR ? X[0] + at : ur + ar;
  const R xl = SL - ul, xr = SR - ur, dl = rl * xl, dr = rr * xr;
  const R idd = rcp_any(dl - dr), Ss = (pr - pl + ul * dl - ur * dr) * idd;
  // ---- the flux of the side k
  const bool supL = SL >= R(0), supR = !supL && SR < R(0);
  const bool left = supL || (!supR && Ss >= R(0));
  const R rk = left ? rl : rr, pk = left ? pl : pr, uk = left ? ul : ur, Ek = left ? El : Er;
  R tk[D];  // (entry 0 unused)
#pragma unroll
  for (int q = 1; q < D; ++q) tk[q] = left ? L[2 + q] : Q[2 + q];
  const R A0 = lf[0], A1 = lf[1], AE = lf[1 + D];
  R At = R(0);  // sum of the transverse flux adjoints times the velocities
#pragma unroll
  for (int q = 1; q < D; ++q) At += lf[1 + q] * tk[q];
  const R ru = rk * uk, A01 = A0 + A1 * uk + At;
  R bSs = lvs, bSk = R(0), mt = ru;  // mt: what the transverse velocities are carried by
  R br = A01 * uk, bp = A1 + AE * uk, bu = rk * (A01 + A1 * uk) + AE * (Ek + pk), bE = AE * uk;
  if (!supL && !supR) {
    // with z = Ss - u_k and d = z / (S_k - Ss) the star density is rho_k (1 + d), and the corrections
    // to the plain flux vanish exactly with z
    const R Sk = left ? SL : SR, sku = left ? xl : xr;
    const R irk = left ? irl : irr, isku = rcp_any(sku), idk = rcp_any(Sk - Ss);
    const R z = Ss - uk, d = z * idk, rd = rk * d, fac = rk + rd;
    const R w = pk * irk * isku, qq = Ss + w, zq = z * qq, s1 = z + d * Ss;
    mt += Sk * rd;
    bSk = (A0 + At) * rd + A1 * rk * s1 + AE * (Ek * d + fac * zq);
    br += Sk * ((A0 + At) * d + A1 * s1 + AE * (zq + d * zq));
    bE += AE * Sk * d;
    const R bd = Sk * (rk * (A0 + At + A1 * Ss) + AE * (Ek + rk * zq)), bz = Sk * (A1 * rk + AE * fac * qq) + bd * idk;
    const R bw = AE * Sk * fac * z, bsku = -bw * w * isku, bdk = -bd * d * idk;
    bSs += A1 * Sk * rd + bw + bz - bdk;
    bp += bw * irk * isku;
    br -= bw * w * irk;
    bSk += bsku + bdk;
    bu -= bz + bsku;
  }
  // ---- contact speed
  const R bN = bSs * idd, bD = -bN * Ss;
  const R bdl = bN * ul + bD, bdr = -bN * ur - bD;
  const R bSL = bdl * rl + (left ? bSk : R(0)), bSR = bdr * rr + (left ? R(0) : bSk);
  R b0l = (left ? br : R(0)) + bdl * xl, b0r = (left ? R(0) : br) + bdr * xr;
  R b1l = (left ? bp : R(0)) - bN, b1r = (left ? R(0) : bp) + bN;
  R b2l = (left ? bu : R(0)) + bN * dl - bdl * rl, b2r = (left ? R(0) : bu) - bN * dr - bdr * rr;
  R bEl = left ? bE : R(0), bEr = left ? R(0) : bE;
  // ---- wave speeds and the density-weighted averages
  const R bul = avL ? R(0) : bSL, bur = avR ? R(0) : bSR;
  b2l += bul;
  b2r += bur;
  R bX0 = (avL ? bSL : R(0)) + (avR ? bSR : R(0));
  const R bat = (avR ? bSR : R(0)) - (avL ? bSL : R(0));
  const R bat2 = sonic ? half * bat * rcp_any(at) : R(0), bHt = gm1 * bat2;
  R bsl = bHt * (hl - Ht), bsr = bHt * (hr - Ht);  // (times iw below)
#pragma unroll
  for (int q = 0; q < D; ++q) {
    const R b = (q == 0 ? bX0 : R(0)) - bHt * X[q];
    bsl += b * (L[2 + q] - X[q]);
    bsr += b * (Q[2 + q] - X[q]);
    const R bl = b * sl * iw, brr = b * sr * iw;
    if (q == 0) {
      b2l += bl;
      b2r += brr;
    } else {
      const R m = lf[1 + q] * mt;
      bL[2 + q] = bl + (left ? m : R(0));
      bR[2 + q] = brr + (left ? R(0) : m);
    }
  }
  const R bhl = bHt * sl * iw * irl, bhr = bHt * sr * iw * irr;  // adjoint of the enthalpies over rho
  bEl += bhl;
  bEr += bhr;
  b1l += bhl;
  b1r += bhr;
  b0l += half * bsl * iw * rcp_any(sl) - bhl * hl;
  b0r += half * bsr * iw * rcp_any(sr) - bhr * hr;
  // sound speeds (entering as -al, +ar)
  const R gl = al > R(0) ? half * gam * irl * rcp_any(al) * bul : R(0);
  const R gr = ar > R(0) ? half * gam * irr * rcp_any(ar) * bur : R(0);
  b1l -= gl;
  b1r += gr;
  b0l += gl * pl * irl;
  b0r -= gr * pr * irr;
  // energies
  const R cl = bEl * rl, cr = bEr * rr;
  bL[0] = b0l + half * bEl * kl;
  bR[0] = b0r + half * bEr * kr;
  bL[1] = b1l + bEl * igm1;
  bR[1] = b1r + bEr * igm1;
  bL[2] = b2l + cl * ul;
  bR[2] = b2r + cr * ur;
#pragma unroll
  for (int q = 1; q < D; ++q) {
    bL[2 + q] += cl * L[2 + q];
    bR[2 + q] += cr * Q[2 + q];
  }
  (void)NW;
}

// Gas part: HLLC (fluxes and contact speed) and the reconstruction of the primitives.
template <class R, int D, int DIR>
__device__ __forceinline__ void adj_gas_face(const AdjArgs<R>& A, uint32_t f) {
  constexpr int NG = 2 + D, NW = 2 + D;
  const DevGrid& g = A.g;
  const Consts<R>& KR = A.k(R(0));
  const uint32_t ncell = (uint32_t)g.ncell;
  const int nd = g.n[DIR];
  if (f >= adj_faces(g, DIR)) return;
  uint32_t ci[4];
  bool fl[4];
  const int id = adj_face_cells<DIR>(g, f, ci, fl);
  const Tab<R> t{A.tab[DIR], nd + 4, A.uniform[DIR] ? A.urow[DIR] : nullptr};
  // adjoint of the face flux of state variable j: dJ/dF = -b dt fr(L) lam_pre(L) + b dt fl(R) lam_pre(R)
  const bool inL = id >= 1, inR = id < nd;
  const R bdt = KR.beta * KR.dt;
  const R cL = inL ? -bdt * t(T_FR, bc_pad(id - 1)) : R(0);
  const R cR = inR ? bdt * t(T_FL, bc_pad(id)) : R(0);
  R lg[NG], lfl[NW];
#pragma unroll
  for (int v = 0; v < NG; ++v) {
    R lj = R(0);
    if (inL) lj += cL * A.lam_pre[FXI(v * ncell + ci[1], A.n_state)];
    if (inR) lj += cR * A.lam_pre[FXI(v * ncell + ci[2], A.n_state)];
    lg[v] = lj;
  }
  lfl[0] = lg[0];
#pragma unroll
  for (int q = 0; q < D; ++q) lfl[1 + q] = lg[1 + (DIR + q) % D];
  lfl[1 + D] = lg[NG - 1];
  const R lvs = A.lvs[FXI((uint32_t)A.lvs_off[DIR] + f, A.n_lvs)];
  bool any = nonzero(lvs);
#pragma unroll
  for (int v = 0; v < NG; ++v) any = any || nonzero(lg[v]);
  if (!any) return;  // nothing depends on this face
  // face states (upper face of id-1, lower face of id; component 2 the normal velocity) and their
  // derivatives by the values of three cells each
  R kL[NW][3], kR[NW][3], Ls[NW], Rs[NW], bL[NW], bR[NW];
  {
    R W[4][NW];
#pragma unroll
    for (int m = 0; m < 4; ++m) adj_prim<R, D, DIR>(A, ci[m], fl[m], W[m]);
#pragma unroll
    for (int v = 0; v < NW; ++v) {
      const int slot = v < 2 ? v : 2 + (v - 2 - DIR + D) % D;
      Ls[slot] = parabola_form(t, bc_pad(id - 1), true, W[0][v], W[1][v], W[2][v], kL[v]);
      Rs[slot] = parabola_form(t, bc_pad(id), false, W[1][v], W[2][v], W[3][v], kR[v]);
    }
  }
  hllc_adjoint<R, D>(KR.gamma, Ls, Rs, lvs, lfl, bL, bR);
#pragma unroll
  for (int v = 0; v < NW; ++v) {
    const int slot = v < 2 ? v : 2 + (v - 2 - DIR + D) % D;
    const R l = bL[slot], r = bR[slot];
    const R lw[4] = {l * kL[v][0], l * kL[v][1] + r * kR[v][0], l * kL[v][2] + r * kR[v][1], r * kR[v][2]};
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      const R x = (v == 2 + DIR && fl[m]) ? -lw[m] : lw[m];
      if (nonzero(x)) atomicAdd(FXP(A.lam_w, (size_t)v * ncell + ci[m], (size_t)NW * ncell), x);
    }
  }
}

template <class R, int D>
__global__ void __launch_bounds__(ADJ_GAS_THREADS) adj_gas_kernel(const __grid_constant__ AdjArgs<R> A) {
  const uint32_t e = blockIdx.x * (uint32_t)ADJ_GAS_THREADS + threadIdx.x;
  if (blockIdx.y == 0) adj_gas_face<R, D, 0>(A, e);
  else if (D >= 2 && blockIdx.y == 1) adj_gas_face<R, D, (D >= 2 ? 1 : 0)>(A, e);
  else if (D >= 3) adj_gas_face<R, D, (D >= 3 ? 2 : 0)>(A, e);
}

// ---------------------------------------------------------------------------------------------
// Per cell: fold the opacity adjoints into (rho, p) and kappa0, map primitive adjoints to the
// conserved variables, and apply the RK weights: dJ/dU_in = b lam_pre + (transport part),
// dJ/dU_base = a lam_pre.
// ---------------------------------------------------------------------------------------------
template <class R, int D, int GP>
__global__ void __launch_bounds__(256) adj_cell_kernel(const __grid_constant__ AdjArgs<R> A) {
  constexpr int NG = 2 + D, NW = 2 + D, NRV = 1 + D;
  const DevGrid& g = A.g;
  const Consts<R>& KR = A.k(R(0));
  const int G = g.G;
  const int lane = threadIdx.x % GP;
  const int64_t cr = (int64_t)blockIdx.x * (256 / GP) + threadIdx.x / GP;
  const bool active = cr < g.ncell;
  const uint32_t ncell = (uint32_t)g.ncell;
  const uint32_t c = active ? (uint32_t)cr : ncell - 1;
  const bool has = lane < G;
  const int gl = has ? lane : 0;
  const int gv = lane < NG ? lane : 0;
  const R* lw_gas = A.lam_w;
  const R* lw_rad = A.lam_w + (size_t)NW * ncell;
  const R* lw_chi = lw_rad + (size_t)NRV * ncell * G;

  const R lgas = lw_gas[FXI(gv * ncell + c, (size_t)NW * ncell)];
  const R lchi = has ? lw_chi[FXI((size_t)c * G + gl, (size_t)ncell * G)] : R(0);
  R lU[NG], lk0 = R(0);
#pragma unroll
  for (int v = 0; v < NG; ++v) lU[v] = R(0);
  if (__any_sync(0xffffffffu, nonzero(lgas) || nonzero(lchi))) {  // (else the map leaves zeros)
    R u[NG], lw[NW];
    {
      const R a = A.in[FXI(gv * ncell + c, A.n_state)], b = lgas;
#pragma unroll
      for (int v = 0; v < NG; ++v) {
        u[v] = __shfl_sync(0xffffffffu, a, v, GP);
        lw[v] = __shfl_sync(0xffffffffu, b, v, GP);
      }
    }
    const R rho = u[0], irho = rcp_any(rho);
    R v_[3] = {R(0), R(0), R(0)}, ke = R(0), v2 = R(0);
#pragma unroll
    for (int q = 0; q < D; ++q) { v_[q] = u[1 + q] * irho; ke += u[1 + q] * v_[q]; v2 += v_[q] * v_[q]; }
    const R p = KR.gm1 * (u[NG - 1] - R(0.5) * ke);
    const R T = p * irho;
    // opacity: chi_g = kappa0 rho^a T^b eps_g^d + sigma0 rho (kappa = 0 where T <= 0)
    R c1 = lchi * KR.sigma0, c2 = R(0), c3 = R(0);
    if (T > R(0) && has) {
      const R K0 = hpow(rho, g.kap_rho_h) * hpow(T, g.kap_T_h);
      const R ef = R(A.gc->efac_of(gl, R(0)));
      const R kapg = KR.kappa0 * K0 * ef;
      const R ra = R(0.5) * R(g.kap_rho_h), tb = R(0.5) * R(g.kap_T_h);
      c1 += lchi * (ra - tb) * kapg * irho;  // d/drho at fixed p (T = p / rho)
      c2 = lchi * tb * kapg * rcp_any(p);
      c3 = lchi * K0 * ef;
    }
    const R lrhoW = lw[0] + seg_sum<GP>(c1);
    const R lpW = lw[1] + seg_sum<GP>(c2);
    lk0 = seg_sum<GP>(c3);
    // primitive (rho, p, v) -> conserved (rho, m, rho e)
    lU[0] = lrhoW + lpW * KR.gm1 * R(0.5) * v2;
#pragma unroll
    for (int q = 0; q < D; ++q) {
      lU[0] -= lw[2 + q] * v_[q] * irho;
      lU[1 + q] = lw[2 + q] * irho - lpW * KR.gm1 * v_[q];
    }
    lU[NG - 1] = lpW * KR.gm1;
  }

  const R al = KR.alpha, be = KR.beta;
  if (active) {
    if (lane < NG) {
      R val = lU[0];
#pragma unroll
      for (int v = 1; v < NG; ++v) if (lane == v) val = lU[v];
      const size_t o = (size_t)lane * ncell + c;
      const R lp = A.lam_pre[FXI(o, A.n_state)];
      const R li = be * lp + val;
      if (A.accumulate_in) A.lam_in[FXI(o, A.n_state)] += li; else A.lam_in[FXI(o, A.n_state)] = li;
      if (A.lam_base) A.lam_base[FXI(o, A.n_state)] = al * lp;
    }
    if (has) {
#pragma unroll
      for (int v = 0; v < NRV; ++v) {
        const size_t o = (size_t)NG * ncell + ((size_t)v * ncell + c) * G + gl;
        const R lp = A.lam_pre[FXI(o, A.n_state)];
        const R li = be * lp + lw_rad[FXI(((size_t)v * ncell + c) * G + gl, (size_t)NRV * ncell * G)];
        if (A.accumulate_in) A.lam_in[FXI(o, A.n_state)] += li; else A.lam_in[FXI(o, A.n_state)] = li;
        if (A.lam_base) A.lam_base[FXI(o, A.n_state)] = al * lp;
      }
    }
  }
  block_partial((active && lane == 0) ? (double)lk0 : 0.0, A.kpart);
}

// Launchers (one translation unit per state type).  The couple and cell kernels use blocks of
// 256 threads, 256/GP cells each, and write one kappa0 partial per block to a.kpart; the face
// kernels take the faces of every direction.
inline unsigned adj_cell_blocks(int64_t ncell, int GP) {
  return (unsigned)((ncell + 256 / GP - 1) / (256 / GP));
}
template <class R, int D> cudaError_t adj_launch_couple(const AdjArgs<R>& a, int GP, cudaStream_t s);
template <class R, int D> cudaError_t adj_launch_face(const AdjArgs<R>& a, cudaStream_t s);
template <class R, int D> cudaError_t adj_launch_cell(const AdjArgs<R>& a, int GP, cudaStream_t s);

#ifdef FX_ADJOINT_DEFINE
template <class R, int D> cudaError_t adj_launch_couple(const AdjArgs<R>& a, int GP, cudaStream_t s) {
  const unsigned nb = adj_cell_blocks(a.g.ncell, GP);
  switch (GP) {
    case 8: adj_couple_kernel<R, D, 8><<<nb, 256, 0, s>>>(a); break;
    case 16: adj_couple_kernel<R, D, 16><<<nb, 256, 0, s>>>(a); break;
    case 32: adj_couple_kernel<R, D, 32><<<nb, 256, 0, s>>>(a); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}
template <class R, int D> cudaError_t adj_launch_face(const AdjArgs<R>& a, cudaStream_t s) {
  int64_t nfmax = 0;
  for (int d = 0; d < D; ++d) nfmax = nfmax > faces_along(a.g.n, d) ? nfmax : faces_along(a.g.n, d);
  const int F = ADJ_RAD_THREADS / a.g.G;  // faces per block
  adj_rad_kernel<R, D><<<dim3((unsigned)((nfmax + F - 1) / F), D, 1), ADJ_RAD_THREADS, 0, s>>>(a);
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  adj_gas_kernel<R, D><<<dim3((unsigned)((nfmax + ADJ_GAS_THREADS - 1) / ADJ_GAS_THREADS), D, 1), ADJ_GAS_THREADS, 0, s>>>(a);
  return cudaGetLastError();
}
template <class R, int D> cudaError_t adj_launch_cell(const AdjArgs<R>& a, int GP, cudaStream_t s) {
  const unsigned nb = adj_cell_blocks(a.g.ncell, GP);
  switch (GP) {
    case 8: adj_cell_kernel<R, D, 8><<<nb, 256, 0, s>>>(a); break;
    case 16: adj_cell_kernel<R, D, 16><<<nb, 256, 0, s>>>(a); break;
    case 32: adj_cell_kernel<R, D, 32><<<nb, 256, 0, s>>>(a); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}
#define FX_ADJ_INSTANTIATE(R, D)                                                              \
  template cudaError_t adj_launch_couple<R, D>(const AdjArgs<R>&, int, cudaStream_t);       \
  template cudaError_t adj_launch_face<R, D>(const AdjArgs<R>&, cudaStream_t);              \
  template cudaError_t adj_launch_cell<R, D>(const AdjArgs<R>&, int, cudaStream_t);
#endif

}  // namespace fx
