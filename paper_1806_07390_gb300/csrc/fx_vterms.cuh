// Velocity-dependent radiation terms (Sec. 3.2, the group form of the moment equations; Sec. 5.2;
// Step 2 of Sec. 6), Cartesian and spherical grids: one lane per group, after the radiation/update
// kernel and before the interaction.  For the stage input U and the cell's volume-averaged
// velocity gradient V_ij = <v^i_;j>, the terms are
//   dE_g/dt   = -V_ij P_g^ij + V_ij [(nu P^ij)_{g+1/2} - (nu P^ij)_{g-1/2}],
//   dF_gj/dt  = -V_ij F_g^i  + V_ik [(nu Q^kji)_{g+1/2} - (nu Q^kji)_{g-1/2}],
// with the M1 pressure tensor P, the heat-flux tensor Q = cE [(f - q)/2 (n d + d n + ...) +
// (5q - 3f)/2 n n n], q = f (2 + 3 chi)/5, and the intergroup values taken, per component pair
// (i, j), from the group below the edge when V_ij < 0 and from the group above otherwise, each
// the limited (MC) linear reconstruction of the spectral density P_g/dnu_g (Q_g/dnu_g) about the
// group's midpoint in nu, with no flux through the ends of the group range (of each species'
// range with three neutrino species: their groups form separate chains).  The terms belong to
// the stage's explicit operator, so the kernel adds w dt (terms of U) to the stage output in place
// (w = 1 in stage 1, 1/2 in stage 2: the weights of the SSP-RK2 combination).
//
// On Cartesian grids V_ij = (v^i on the upper j face - v^i on the lower j face) / dx_j, from the
// face velocities the gas face kernel stores: the contact speed v* as the normal component and the
// transverse components of the reconstructed state on the v* upwind side (the spherical form is
// described at the kernel).
#pragma once
#include <utility>

#include "fx_stage.cuh"

namespace fx {

// Number of distinct components of the symmetric P (rank 2) and Q (rank 3) in D dimensions, and
// the index of a component among them.
template <int D> struct VtComp {
  static constexpr int NP = D * (D + 1) / 2;
  static constexpr int NQ = D == 1 ? 1 : (D == 2 ? 4 : 10);
  static constexpr int NC = NP + NQ;
};
__host__ __device__ constexpr int vt_sym2(int i, int j, int D) {
  return (i <= j) ? i * D - i * (i - 1) / 2 + (j - i) : j * D - j * (j - 1) / 2 + (i - j);
}
__host__ __device__ constexpr int vt_sym3(int i, int j, int k, int D) {
  // sort a <= b <= c; triples with a smaller first index come first, then pairs (b, c) on [a, D)
  int a = i, b = j, c = k, t = 0;
  if (a > b) { t = a; a = b; b = t; }
  if (b > c) { t = b; b = c; c = t; }
  if (a > b) { t = a; a = b; b = t; }
  int idx = 0;
  for (int x = 0; x < a; ++x) idx += (D - x) * (D - x + 1) / 2;
  return idx + vt_sym2(b - a, c - a, D - a);
}

// f(integral constant) for every index of the sequence
template <int... I, class F> __device__ __forceinline__ void vt_each(std::integer_sequence<int, I...>, F f) {
  (f(std::integral_constant<int, I>{}), ...);
}

// Reciprocals and roots of the closure for a lane's groups, 0 where the group has no flux or no
// energy (then f = 0: P = E/3 isotropic, Q = 0).
__device__ __forceinline__ void vt_roots(F2 FF, F2 cE, F2& iF, F2& iE) {
  const bool a = FF.x > 0.0f && cE.x > 0.0f, b = FF.y > 0.0f && cE.y > 0.0f;
  iF = F2(a ? rsqrtf(FF.x) : 0.0f, b ? rsqrtf(FF.y) : 0.0f);
  iE = F2(a ? rcp_approx(cE.x) : 0.0f, b ? rcp_approx(cE.y) : 0.0f);
}
__device__ __forceinline__ void vt_roots(double FF, double cE, double& iF, double& iE) {
  const bool ok = FF > 0.0 && cE > 0.0;
  const int e = __double2hiint(FF);
  iF = !ok ? 0.0 : (e >= 0x00400000 && e < 0x7fb00000 ? rsqrt64(FF) : 1.0 / sqrt(FF));
  iE = ok ? rcp_any(cE) : 0.0;
}

// Components of P (units of E) and Q (units of F) of the lane's groups, in the order of vt_sym2 /
// vt_sym3: x[0 .. NP) = P, x[NP .. NC) = Q.  With s = sqrt(4 - 3 f^2) the closure is polynomial in s:
// (1 - chi)/2 = (s - 1)/3, (3 chi - 1)/2 = 2 - s, and with q = f (2 + 3 chi)/5 = f (7 - 2 s)/5,
// (f - q)/2 = f (s - 1)/5, (5 q - 3 f)/2 = f (2 - s): one reciprocal of cE, one inverse root of F^2,
// one square root.
template <int D, class V>
__device__ __forceinline__ void vt_moments(V c, V one, V p4, V m3, V E, const V* F, V* x) {
  using VC = VtComp<D>;
  V FF = F[0] * F[0];
#pragma unroll
  for (int q = 1; q < D; ++q) FF = vfma(F[q], F[q], FF);
  const V cE = E * c;
  V iF, iE;
  vt_roots(FF, cE, iF, iE);
  const V f = vmin((FF * iF) * iE, one);
  const V s = vsqrt(vfma(m3, f * f, p4)), s1 = s - one, b = (one + one) - s;
  using T = decltype(vget(E, 0));
  const V g = f * cE, a3 = E * s1 * T(1.0 / 3.0), bE = E * b, qa = g * s1 * T(0.2), qb = g * b;
  V n[D];
#pragma unroll
  for (int i = 0; i < D; ++i) n[i] = F[i] * iF;
  vt_each(std::make_integer_sequence<int, D * D>{}, [&](auto t) {
    constexpr int i = decltype(t)::value / D, j = decltype(t)::value % D;
    if constexpr (i <= j) {
      const V nn = n[i] * n[j];
      x[vt_sym2(i, j, D)] = i == j ? vfma(bE, nn, a3) : bE * nn;
      vt_each(std::make_integer_sequence<int, D>{}, [&](auto u) {
        constexpr int k = decltype(u)::value;
        if constexpr (k >= j) {
          constexpr int m = VC::NP + vt_sym3(i, j, k, D);
          V r = qb * nn * n[k];
          if constexpr (j == k) r = vfma(qa, n[i], r);
          if constexpr (i == k) r = vfma(qa, n[j], r);
          if constexpr (i == j) r = vfma(qa, n[k], r);
          x[m] = r;
        }
      });
    }
  });
}

// Per-group frequency constants of the limited reconstruction (host-computed): the reciprocal
// group width, the reciprocal midpoint distances to the lower neighbour, the upper neighbour and
// across both, and the distances from the midpoint to the lower and upper edge (the distances are
// zero for the first and last group, whose slope is zero).
struct VtConst {
  double c[6][MAXG];
  float c32[6][MAXG];
  __device__ __forceinline__ double of(int k, int j, double) const { return c[k][j]; }
  __device__ __forceinline__ float of(int k, int j, float) const { return c32[k][j]; }
};
enum { VT_INU = 0, VT_LMID, VT_HMID, VT_CMID, VT_MLO, VT_MHI };

inline void vt_constants(const double* edge, int G, VtConst& v) {
  for (int k = 0; k < 6; ++k)
    for (int j = 0; j < MAXG; ++j) v.c[k][j] = 0.0;
  for (int j = 0; j < G; ++j) {
    const double mid = 0.5 * (edge[j] + edge[j + 1]);
    v.c[VT_INU][j] = 1.0 / (edge[j + 1] - edge[j]);
    if (j > 0 && j + 1 < G) {
      const double mm = 0.5 * (edge[j - 1] + edge[j]), mp = 0.5 * (edge[j + 1] + edge[j + 2]);
      v.c[VT_LMID][j] = 1.0 / (mid - mm);
      v.c[VT_HMID][j] = 1.0 / (mp - mid);
      v.c[VT_CMID][j] = 1.0 / (mp - mm);
      v.c[VT_MLO][j] = mid - edge[j];
      v.c[VT_MHI][j] = edge[j + 1] - mid;
    }
  }
  for (int k = 0; k < 6; ++k)
    for (int j = 0; j < MAXG; ++j) v.c32[k][j] = (float)v.c[k][j];
}

// One lane per W groups (a packed pair in FP32, one group in FP64), GL = ceil(G / W) lanes per cell and
// 32 / GL cells of one x row per warp; a block's warps take VT_ROWS rows in turn, so that the
// per-group constants are read once for them.  Each lane forms its groups' P and Q components and
// spectral densities, takes its neighbours' (the lane below's last group, the lane above's first)
// through warp shuffles for the limited slopes, and the flux through its upper edge from the lane
// above; the edge between a lane's two groups needs no shuffle.
//
// The upwind choice of component pair (i, j) depends on the sign of V_ij, the cell's: a lane splits
// V_ij into max(V_ij, 0) and min(V_ij, 0), adds the pairs that share a symmetric component, and
// contracts them with the lower-edge values and with the values below the edge, without selects.
//
// Bound by instruction issue (63 % of cycles).  768^2 x 16 groups 0.125 -> 0.104 ms per launch, against a
// kernel with the closure's reciprocals in chi, a select per component pair and lanes padded to a power of
// two.
//
// SPH: the 2-d spherical (r, theta) grid.  The tensors are those of 3 dimensions (DT = 3, with
// F_phi = 0 and the V_phiphi entry), in physical components: the state's covariant flux
// F_q = h_q Fhat_q (cell scale factors) is divided by h_q on entry, and the physical derivative
// of Fhat_q multiplied by h_q on exit.  The gradient takes the coordinate components
// v^1 = vhat_r / h_1, v^2 = vhat_theta / h_2 on the faces (radial faces: the face's dr/dx1 and r;
// theta faces: the cell's h), differences them over the cell, adds the volume-averaged
// connection coefficients times the coordinate velocity at the centroid (linear profile between
// the two faces), and turns V^a_b into physical components V^a_b h_a / h_b.
constexpr int VT_THREADS = 256, VT_ROWS = 4;

// The cell's velocity gradient V (physical components, DT x DT) and the scale factors h of the
// flux components (1 on Cartesian grids), from the face velocities: component i of a face of
// direction j sits in row NG + ((i - j) mod D) of direction j's face block.
template <class R, int D, bool SPH, int DT>
__device__ __forceinline__ void vt_gradient(const StageArgs<R>& A, int ix, int iy, int iz, R (&V)[DT][DT],
                                            R (&h)[DT]) {
  constexpr int NG = 2 + D;
  const DevGrid& g = A.g;
  R vl[D][D], vu[D][D];  // [j][i]: lower / upper face of direction j, component i
#pragma unroll
  for (int j = 0; j < D; ++j) {
    const uint32_t ex = (uint32_t)(g.n[0] + (j == 0)), ey = (uint32_t)(g.n[1] + (j == 1));
    const uint32_t nf = ex * ey * (uint32_t)(g.n[2] + (j == 2));
    const uint32_t lf = ((uint32_t)iz * ey + (uint32_t)iy) * ex + (uint32_t)ix;
    const uint32_t uf = lf + (j == 0 ? 1u : (j == 1 ? ex : ex * ey));
    const R* fr = A.faces + A.face_off[j];
    const uint32_t nfr = (uint32_t)(NG + D) * nf;  // this direction's block (fluxes, v*, D-1 velocities)
    (void)nfr;
#pragma unroll
    for (int i = 0; i < D; ++i) {
      const uint32_t row = (uint32_t)(NG + (i - j + D) % D) * nf;
      vl[j][i] = __ldg(FXP(fr, row + lf, nfr));
      vu[j][i] = __ldg(FXP(fr, row + uf, nfr));
    }
  }
#pragma unroll
  for (int i = 0; i < DT; ++i)
#pragma unroll
    for (int j = 0; j < DT; ++j) V[i][j] = R(0);
#pragma unroll
  for (int q = 0; q < DT; ++q) h[q] = R(1);
  if constexpr (SPH) {
    const Tab<R> tr{A.tab[0], g.n[0] + 4, A.uniform[0] ? A.urow[0] : nullptr};
    const Tab<R> tq{A.tab[1], g.n[1] + 4, A.uniform[1] ? A.urow[1] : nullptr};
    const int ipr = ix + 2, ipt = iy + 2;
    const R idr = A.k(R(0)).idx[0], idt = A.k(R(0)).idx[1];
    h[0] = tr(T_HA, ipr);
    h[1] = tr(T_HB, ipr);
    const R ih1 = R(1) / h[0], ih2 = R(1) / h[1];
    // coordinate components on the radial faces (the faces' own dr/dx1 and r) ...
    const R u1l = vl[0][0] * tr(T_QI, ipr), u1r = vu[0][0] * tr(T_QI, ipr + 1);
    const R u2l = vl[0][1] * tr(T_RI, ipr), u2r = vu[0][1] * tr(T_RI, ipr + 1);
    // ... and on the theta faces (the cell's h)
    const R t1l = vl[1][0] * ih1, t1r = vu[1][0] * ih1;
    const R t2l = vl[1][1] * ih2, t2r = vu[1][1] * ih2;
    // centroid values of the linear profiles: the centroid lies (c - x_L) / dx along the cell
    const R v1 = u1l + (u1r - u1l) * (-tr(T_DL, ipr) * idr);
    const R v2 = t2l + (t2r - t2l) * (-tq(T_DL, ipt) * idt);
    const R g111 = tr(T_GA, ipr), g221 = tr(T_GB, ipr), g122 = tr(T_GC, ipr);
    const R g222 = tq(T_GA, ipt), g332 = tq(T_GB, ipt);
    V[0][0] = (u1r - u1l) * idr + g111 * v1;
    V[0][1] = ((t1r - t1l) * idt + g122 * v2) * (h[0] * ih2);
    V[1][0] = ((u2r - u2l) * idr + g221 * v2) * (h[1] * ih1);
    V[1][1] = (t2r - t2l) * idt + g221 * v1 + g222 * v2;
    V[2][2] = g221 * v1 + g332 * v2;
  } else {
#pragma unroll
    for (int j = 0; j < D; ++j) {
      const R idx = A.k(R(0)).idx[j];
#pragma unroll
      for (int i = 0; i < D; ++i) V[i][j] = (vu[j][i] - vl[j][i]) * idx;
    }
  }
}

// Volume of cell (ix, iy) (the budget's weight).
template <class R, int D, bool SPH>
__device__ __forceinline__ double vt_volume(const StageArgs<R>& A, int ix, int iy) {
  const DevGrid& g = A.g;
  if constexpr (SPH) {
    return (double)Tab<R>{A.tab[0], g.n[0] + 4, A.uniform[0] ? A.urow[0] : nullptr}(T_VOL, ix + 2) *
           (double)Tab<R>{A.tab[1], g.n[1] + 4, A.uniform[1] ? A.urow[1] : nullptr}(T_VOL, iy + 2);
  } else {
    double vol = 1.0;
    for (int d = 0; d < D; ++d) vol /= g.inv_dx[d];
    return vol;
  }
}

// x shuffled from the lane below (its last group) or above (its first group): the neighbouring
// groups of the lane's first and last group, as lane values of the groups below and above each
__device__ __forceinline__ F2 vt_below(F2 x) { return F2(__shfl_up_sync(0xffffffffu, x.y, 1), x.x); }
__device__ __forceinline__ F2 vt_above(F2 x) { return F2(x.y, __shfl_down_sync(0xffffffffu, x.x, 1)); }
__device__ __forceinline__ double vt_below(double x) { return __shfl_up_sync(0xffffffffu, x, 1); }
__device__ __forceinline__ double vt_above(double x) { return __shfl_down_sync(0xffffffffu, x, 1); }
// the same with zero where the lane's first (last) group has no neighbour below (above)
__device__ __forceinline__ F2 vt_keep(F2 x, bool k0, bool k1) { return F2(k0 ? x.x : 0.0f, k1 ? x.y : 0.0f); }
__device__ __forceinline__ double vt_keep(double x, bool k0, bool) { return k0 ? x : 0.0; }

// Whether component (a <= b <= c) of Q enters the flux equation q (with the pair of its other two
// indices; the pairs (0, 2) and (1, 2) of the gradient vanish on the spherical grid), or any of D.
__host__ __device__ constexpr bool vt_enters(int a, int b, int c, int q, bool sph) {
  return (q == a || q == b || q == c) && (!sph || (q == a ? b : a) == (q == c ? b : c) || (q == c ? b : c) < 2);
}
__host__ __device__ constexpr bool vt_needed(int a, int b, int c, int D, bool sph) {
  for (int q = 0; q < D; ++q)
    if (vt_enters(a, b, c, q, sph)) return true;
  return false;
}
template <class R, int D, bool SPH>
__global__ void __launch_bounds__(VT_THREADS, sizeof(R) == 4 ? (D == 3 || SPH ? 2 : 3) : 1) vterm_kernel(const __grid_constant__ StageArgs<R> A) {
  static_assert(!SPH || D == 2, "the spherical grid is 2-d");
  using V = typename LaneOf<R>::V;
  constexpr int W = LaneOf<R>::W;
  constexpr int DT = SPH ? 3 : D;  // dimension of the tensors
  using VC = VtComp<DT>;
  constexpr int NG = 2 + D, NP = VC::NP, NC = VC::NC;
  const DevGrid& g = A.g;
  const int G = g.G, GL = (G + W - 1) / W;
  const uint32_t ncell = (uint32_t)g.ncell;
  const int cpw = 32 / GL, wl = (int)threadIdx.x & 31, cw = wl / GL, lane = wl - cw * GL;
  const int x0 = (int)(blockIdx.y * (VT_THREADS / 32) + threadIdx.x / 32) * cpw + cw;
  const bool cok = cw < cpw && x0 < g.n[0];
  const int ga = lane * W, gb = ga + W - 1;
  const int ka = ga % g.Gs, kb = gb < G ? gb % g.Gs : 0;  // groups of the channels (species-major)
  const bool acta = cok && ga < G, actb = W == 2 && cok && gb < G;
  const int ix = cok ? x0 : g.n[0] - 1;  // every lane takes part in the shuffles
  // per-group frequency constants (the first and last groups and absent ones have zero midpoint
  // constants: zero slope), and the lower edges (no flux through the lower end of a species' range)
  const VtConst& vc = *A.vtc;
  auto cpair = [&](int e) { return vpair(acta ? vc.of(e, ka, R(0)) : R(0), actb ? vc.of(e, kb, R(0)) : R(0), V()); };
  const V inu = cpair(VT_INU), lm = cpair(VT_LMID), hm = cpair(VT_HMID), cm = cpair(VT_CMID);
  const V mlo = cpair(VT_MLO), mhi = cpair(VT_MHI);
  const bool lo_a = acta && ka > 0, lo_b = actb && kb > 0;
  const V el = vpair(lo_a ? A.gc->edge_of(ka, R(0)) : R(0), lo_b ? A.gc->edge_of(kb, R(0)) : R(0), V());
  // whether the channel above each group is its upper neighbour in frequency
  const bool up_a = W == 2 ? true : !(ga + 1 >= G || ka + 1 >= g.Gs);
  const bool up_b = W == 2 && !(gb + 1 >= G || kb + 1 >= g.Gs);
  const V one(R(1)), p4(R(4)), m3(R(-3)), cc_(A.k(R(0)).c);
  const R wdt = A.k(R(0)).dt * A.k(R(0)).beta;  // w = 1 (stage 1) or 1/2 (stage 2)
  const uint32_t rad = (uint32_t)NG * ncell, vstr = ncell * (uint32_t)G;
  const bool vec = A.rt.vec != 0;
  const int nrow = g.n[1] * g.n[2];
  double esum = 0.0;
  for (int row = (int)blockIdx.x * VT_ROWS; row < min((int)(blockIdx.x + 1) * VT_ROWS, nrow); ++row) {
    const int iy = D == 3 ? row % g.n[1] : row, iz = D == 3 ? row / g.n[1] : 0;
    // 32-bit offsets: the host keeps every state offset below 2^32
    const uint32_t gid = ((uint32_t)row * g.n[0] + (uint32_t)ix) * (uint32_t)G + (uint32_t)ga;
    // the stage output this lane updates, read first so that its latency overlaps the work, and
    // the groups of the stage input
    V o[1 + D], Q[1 + D];
#pragma unroll
    for (int v = 0; v < 1 + D; ++v) o[v] = Q[v] = V(R(0));
    if (acta) {
#pragma unroll
      for (int v = 0; v < 1 + D; ++v) {
        o[v] = ld_global_lane(FXP(A.out, rad + v * vstr + gid, A.n_state), vec, actb, V());
        Q[v] = ld_global_lane(FXP(A.in, rad + v * vstr + gid, A.n_state), vec, actb, V());
      }
    }
    R Vg[DT][DT], h[DT];
    vt_gradient<R, D, SPH, DT>(A, ix, iy, iz, Vg, h);
    V F[DT], x[NC];
#pragma unroll
    for (int q = 0; q < DT; ++q) F[q] = V(R(0));
#pragma unroll
    for (int q = 0; q < D; ++q) F[q] = SPH ? Q[1 + q] * rcp_any(h[q]) : Q[1 + q];  // physical components
    vt_moments<DT>(cc_, one, p4, m3, Q[0], F, x);
    // the split gradient per symmetric pair p = (i <= j): cp, cn the sums of the positive and
    // negative parts, and their total (the pairs (0, 2) and (1, 2) vanish on the spherical grid)
    R cp[NP], cn[NP];
#pragma unroll
    for (int i = 0; i < DT; ++i)
#pragma unroll
      for (int j = i; j < DT; ++j) {
        const int p = vt_sym2(i, j, DT);
        cp[p] = max_fast(Vg[i][j], R(0));
        cn[p] = min_fast(Vg[i][j], R(0));
        if (i != j) {
          cp[p] += max_fast(Vg[j][i], R(0));
          cn[p] += min_fast(Vg[j][i], R(0));
        }
      }
    // work terms V_ij P^ij and sum_i V_ij F^i
    V d[1 + D];
#pragma unroll
    for (int v = 0; v < 1 + D; ++v) d[v] = V(R(0));
#pragma unroll
    for (int i = 0; i < DT; ++i)
#pragma unroll
      for (int j = i; j < DT; ++j)
        if (!SPH || i == j || j < 2) d[0] = vfma(V(-(cp[vt_sym2(i, j, DT)] + cn[vt_sym2(i, j, DT)])), x[vt_sym2(i, j, DT)], d[0]);
#pragma unroll
    for (int j = 0; j < D; ++j)
#pragma unroll
      for (int i = 0; i < D; ++i) d[1 + j] = vfma(V(-Vg[i][j]), F[i], d[1 + j]);
    // fluxes through the groups' lower edges, component by component of P and Q: the spectral
    // density's limited slope, its value at the lower edge and the value of the group below at it
    V fl[1 + D];
#pragma unroll
    for (int v = 0; v < 1 + D; ++v) fl[v] = V(R(0));
    auto edge = [&](V xm, V& low, V& below) {
      const V xc = xm * inu;
      const V xb = vt_below(xc), xa = vt_above(xc);
      const V sl = mc_min((xc - xb) * lm, (xa - xc) * hm, (xa - xb) * cm, R(2));
      low = vfma(sl * R(-1), mlo, xc);
      below = vt_below(vfma(sl, mhi, xc));
    };
#pragma unroll
    for (int i = 0; i < DT; ++i)
#pragma unroll
      for (int j = i; j < DT; ++j) {
        if (SPH && i != j && j >= 2) continue;  // V_ij = 0 there
        const int p = vt_sym2(i, j, DT);
        V low, below;
        edge(x[p], low, below);
        fl[0] = vfma(V(cp[p]), low, vfma(V(cn[p]), below, fl[0]));
      }
    // Q^kji: the component (a <= b <= c) enters flux q for every split of it into q and a pair u <= w
    // (constant indices: an index computed in an unrolled loop left the components in local memory)
    vt_each(std::make_integer_sequence<int, DT * DT * DT>{}, [&](auto t) {
      constexpr int a = decltype(t)::value / (DT * DT), b = decltype(t)::value / DT % DT, c = decltype(t)::value % DT;
      if constexpr (a <= b && b <= c && vt_needed(a, b, c, D, SPH)) {
        constexpr int m = NP + vt_sym3(a, b, c, DT);
        V low, below;
        edge(x[m], low, below);
        vt_each(std::make_integer_sequence<int, D>{}, [&](auto qt) {
          constexpr int q = decltype(qt)::value, u = q == a ? b : a, w = q == c ? b : c, p = vt_sym2(u, w, DT);
          if constexpr (vt_enters(a, b, c, q, SPH)) fl[1 + q] = vfma(V(cp[p]), low, vfma(V(cn[p]), below, fl[1 + q]));
        });
      }
    });
    bool bad = false;
#pragma unroll
    for (int v = 0; v < 1 + D; ++v) {
      const V f = vt_keep(fl[v] * el, lo_a, lo_b);
      d[v] = d[v] + (vt_keep(vt_above(f), up_a, up_b) - f);  // upper-edge flux less lower-edge flux
      if (SPH && v >= 1) d[v] = d[v] * h[v - 1];             // covariant component
      const V r = vfma(V(wdt), d[v], o[v]);
      if (acta) {
        st_global_lane(FXP(A.out, rad + v * vstr + gid, A.n_state), r, vec, actb);
        bad |= !isfinite(vget(r, 0)) || (actb && !isfinite(vget(r, W - 1)));
      }
    }
    if (bad) atomicOr(A.status, ST_NONFINITE);
    if (A.budget != nullptr && acta)
      esum += ((double)vget(d[0], 0) + (actb ? (double)vget(d[0], W - 1) : 0.0)) * vt_volume<R, D, SPH>(A, ix, iy);
  }
  if (A.budget != nullptr) {
    // radiation energy the terms add, weighted as the RK combination weighs this stage
#pragma unroll
    for (int s = 16; s > 0; s >>= 1) esum += __shfl_xor_sync(0xffffffffu, esum, s);
    if (wl == 0) atomicAdd(A.budget + (blockIdx.x % BUDGET_SLOTS) * NBUDGET + 8, esum * A.bw_flux);
  }
}

}  // namespace fx
