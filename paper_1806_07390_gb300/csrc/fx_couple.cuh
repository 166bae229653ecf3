// Cell-local implicit matter-radiation interaction of the FP32 state as a kernel of its own, one
// thread per cell (Sec. 5.3: the backward-Euler group update of Eq. 25 inside the Newton iteration
// on T of Eqs. 26-27, the gas energy by conservation, then the flux absorption of Eq. 28 and its
// momentum and energy feedback, Eqs. 31-32; readings R10-R12).
//
// Inside the stage kernel a cell's groups are spread over the lanes of a segment, so the scalar
// part of the interaction (the iteration on T, its stopping tests, the gas update) is repeated by
// every lane or confined to one warp that the others wait for at block barriers.  GB300 executes
// two FP64 lane-operations per cycle per multiprocessor, so an FP64 warp instruction costs the same
// with one active lane as with 32.  Here a thread owns a cell: each FP64 instruction serves 32
// cells, the group loop runs in FP32 with the temperature-dependent parts of the Planck table
// interpolation and of the opacity computed once per evaluation, and no warp waits at a barrier.
// The stage kernel leaves the state after the explicit update and RK combination in its output;
// this kernel updates that state in place.
//
// NT is the type of the iterate T, the residual and the gas update: double for the FP32 form with
// the FP64 Newton, float for the all-FP32 form.  Group arithmetic is FP32 in both.
#pragma once
#include <cuda_runtime.h>

#include "fx_stage.cuh"

namespace fx {

constexpr int CPL_THREADS = 128;  // cells (threads) per block of couple_kernel

// Rows of couple_kernel's shared memory per cell: E, then the F_q (which hold the first
// evaluation's E_g and dE_g/dT during the Newton); at least three.
constexpr int couple_rows(int D) { return 1 + D > 3 ? 1 + D : 3; }

// Row stride of couple_kernel in floats: the groups' pairs, twice an odd number of them, so that the
// threads' 8-byte accesses to one pair of their rows fall into distinct banks.
__host__ __device__ constexpr int couple_stride(int G) { return 2 * (((G + 1) / 2) | 1); }
template <int D> inline size_t couple_smem_bytes(int G) {
  return (size_t)couple_rows(D) * CPL_THREADS * (size_t)couple_stride(G) * sizeof(float);
}

// Temperature-dependent part of one evaluation of the group energies: the position in the FP32
// Planck band tables (shared by all groups: the tables have common nodes in log2 T) and the powers
// of T.
struct PlanckAt {
  int mode;              // 0: every band in the Wien tail (B = 0); 1: table; 2: hot-limit series
  int i;                 // interval (mode 1)
  F2 t, t2, t15;         // position t in it, 2 t and 3 t/2
  float invT, aT3, aT4;  // 1/T, a_N T^3, a_N T^4
};

__device__ __forceinline__ PlanckAt planck_at(const PlanckTable& ptab, float aN, float T) {
  PlanckAt p;
  p.invT = frcp(T);
  const float T3 = T * T * T;
  p.aT3 = aN * T3;
  p.aT4 = p.aT3 * T;
  const float s = (__log2f(T) - ptab.u0) * float(PTAB_PER_OCT);
  p.mode = s < 0.0f ? 0 : (s >= float(ptab.nu - 1) ? 2 : 1);
  p.i = p.mode == 1 ? (int)s : 0;
  const float t = s - (float)p.i;  // (used in mode 1)
  p.t = F2(t);
  p.t2 = F2(2.0f * t);
  p.t15 = F2(1.5f * t);
  return p;
}

// A band outside the table (one group): 0 deep in the Wien tail; very hot, x = eps/T < 2^-14 at both
// edges, Int s^3/(e^s-1) ds = x^3/3 - x^4/8 + O(x^5).  Returns I and d ln I / d ln T.
static __device__ __noinline__ float2 planck_outside(int mode, float elo, float ehi, float invT) {
  if (mode == 0) return make_float2(0.0f, 0.0f);
  const float a = elo * invT, b = ehi * invT;
  const float a3 = a * a * a, b3 = b * b * b;
  const float I = (b3 - a3) * (1.0f / 3.0f) - (b3 * b - a3 * a) * 0.125f;
  return make_float2(I, ((a3 * a * (1.0f - 0.5f * a)) - (b3 * b * (1.0f - 0.5f * b))) * frcp(I));
}

// B_g(T) and dB_g/dT of the groups 2 pr, 2 pr + 1 (G groups; edge: their band edges) at the
// evaluation point p.
__device__ __forceinline__ void planck_pair(const PlanckTable& ptab, const PlanckAt& p, int pr, int G,
                                            const float* edge, F2& B, F2& dB) {
  F2 I, d;  // d: d ln I / d ln T = dL/du
  if (p.mode == 1) {
    const float4* const q = FXP_AT(ptab.status, ptab.tab, 2 * (p.i * ptab.si + pr * ptab.sg), ptab.n - 1);
    const float4 u = __ldg(q), v = __ldg(q + 1);
    const F2 c0(u.x, u.y), c1(u.z, u.w), c2(v.x, v.y), c3(v.z, v.w);
    const F2 L = vfma(vfma(vfma(c3, p.t, c2), p.t, c1), p.t, c0);
    I = F2(ex2_approx(L.x), ex2_approx(L.y)) * F2(planck_scale(c3.x), planck_scale(c3.y));
    d = vfma(p.t2, vfma(p.t15, c3, c2), c1) * float(PTAB_PER_OCT);
  } else {
    const int g = 2 * pr, g1 = min(g + 1, G - 1);
    const float2 a = planck_outside(p.mode, edge[g], edge[g + 1], p.invT);
    const float2 b = planck_outside(p.mode, edge[g1], edge[g1 + 1], p.invT);
    I = F2(a.x, b.x);
    d = F2(a.y, b.y);
  }
  B = I * p.aT4;
  dB = (I * p.aT3) * (d + 4.0f);  // d/dT (T^4 I) = T^3 I (4 + d ln I / d ln T)
}

// Copies between contiguous runs of nc*G floats in global memory (nc cells of G groups) and the
// block's per-cell shared rows (stride RS): coalesced, in float4 units when the run is 16-byte
// aligned and G is a multiple of 4 (a float4 then never straddles two rows).  EVEN: RS is even, and a
// float4 is two 8-byte shared accesses.  A thread's first element and its steps are the same for
// every run of the block, so they are divided out once.
struct RowCopy {
  int nc, G, RS;
  int row, col, drow, dcol, ncol;  // in units of one float4 or float
  bool v4;
  __device__ __forceinline__ RowCopy(const float* gmem, int nc_, int G_, int RS_) : nc(nc_), G(G_), RS(RS_) {
    v4 = G % 4 == 0 && (reinterpret_cast<uintptr_t>(gmem) & 15) == 0;
    ncol = v4 ? G / 4 : G;
    const int t = threadIdx.x;
    row = t / ncol;
    col = t - row * ncol;
    drow = CPL_THREADS / ncol;
    dcol = CPL_THREADS - drow * ncol;
  }
  template <bool TO_SHARED, bool EVEN> __device__ __forceinline__ void run(float* gmem, float* rows) const {
    int r = row, c = col;
    const int tot = nc * ncol;
    if (v4) {
      float4* const g4 = reinterpret_cast<float4*>(gmem);
#pragma unroll 4
      for (int e = threadIdx.x; e < tot; e += CPL_THREADS) {
        float* const s = rows + r * RS + 4 * c;
        if constexpr (EVEN) {
          float2* const s2 = reinterpret_cast<float2*>(s);
          if (TO_SHARED) {
            const float4 x = g4[e];
            s2[0] = make_float2(x.x, x.y);
            s2[1] = make_float2(x.z, x.w);
          } else {
            const float2 x = s2[0], y = s2[1];
            g4[e] = make_float4(x.x, x.y, y.x, y.y);
          }
        } else if (TO_SHARED) {
          const float4 x = g4[e];
          s[0] = x.x; s[1] = x.y; s[2] = x.z; s[3] = x.w;
        } else {
          g4[e] = make_float4(s[0], s[1], s[2], s[3]);
        }
        r += drow;
        c += dcol;
        if (c >= ncol) { c -= ncol; ++r; }
      }
    } else {
#pragma unroll 4
      for (int e = threadIdx.x; e < tot; e += CPL_THREADS) {
        if (TO_SHARED) rows[r * RS + c] = gmem[e];
        else gmem[e] = rows[r * RS + c];
        r += drow;
        c += dcol;
        if (c >= ncol) { c -= ncol; ++r; }
      }
    }
  }
};

// The groups run in pairs (packed FP32 arithmetic, fx_pair.cuh): an odd count's last pair carries a
// group of zero energy and zero opacity, which changes nothing.  Bound by latency (the table words,
// shared rows and FP64 steps of a cell's chain; FP64 pipe 40 %, DRAM 35 % busy), so seven resident
// blocks at 72 registers (at 0.118 ms for 1024^2 x 16, six took 0.123 and eight 0.116, where 256^3 x 12
// loses 6 %).  With two table words per group, scalar rows, divisions in the copies and powers and FP64
// comparisons, 1024^2 x 16 took 0.133 ms, now 0.111; 256^3 x 12 3.31 -> 2.45 ms, 75 x 61 x 50 x 20 0.129 ->
// 0.091 ms.
template <int D, class NT>
__global__ void __launch_bounds__(CPL_THREADS, 7) couple_kernel(const __grid_constant__ StageArgs<float> A) {
  using LT = float;
  constexpr int NG = 2 + D, NRV = 1 + D;
  const DevGrid& g = A.g;
  const int G = g.G;
  const uint32_t ncell = (uint32_t)g.ncell;
  const Consts<NT>& kn = A.k(NT(0));
  const Consts<float>& kl = A.kf;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float* const srow = reinterpret_cast<float*>(smem_raw);  // [rows][CPL_THREADS][RS]
  __shared__ float s_ed[MAXG + 1];
  __shared__ F2 s_ef[MAXG / 2];
  const int RS = couple_stride(G), NPR = (G + 1) / 2;
  const int t = threadIdx.x;
  const uint32_t c0 = blockIdx.x * (uint32_t)CPL_THREADS;
  const int nc = (int)min((uint32_t)CPL_THREADS, ncell - c0);
  const bool act = t < nc;
  const uint32_t cid = c0 + (uint32_t)t;

  for (int j = t; j <= G; j += CPL_THREADS) s_ed[j] = A.gc->edge32[j];
  for (int j = t; j < NPR; j += CPL_THREADS)
    s_ef[j] = F2(A.gc->efac32[2 * j], 2 * j + 1 < G ? A.gc->efac32[2 * j + 1] : 0.0f);
  if (G & 1)  // the pad group's rows
    for (int v = 0; v < couple_rows(D); ++v) srow[(v * CPL_THREADS + t) * RS + G] = 0.0f;
  // the block's E rows: the contiguous range [c0 G, (c0 + nc) G) (the F rows follow the Newton)
  // (runs of the variables lie ncell G floats apart: with G a multiple of 4 all are aligned alike)
  const RowCopy rc(A.out + ((size_t)NG * ncell + (size_t)c0 * G), nc, G, RS);
  rc.run<true, true>(FXPR(A.out, (size_t)NG * ncell + (size_t)c0 * G, nc * G, A.n_state), srow);
  float rho_f = 1.0f, m_f[3] = {0.0f, 0.0f, 0.0f}, rhoe_f = 1.0f;
  if (act) {
    rho_f = A.out[FXI(cid, A.n_state)];
#pragma unroll
    for (int q = 0; q < D; ++q) m_f[q] = A.out[FXI((1 + q) * ncell + cid, A.n_state)];
    rhoe_f = A.out[FXI((NG - 1) * ncell + cid, A.n_state)];
  }
  // covariant components: physical = m_q / h_q on the spherical (r, theta) grid
  const bool sph = (D == 2) && g.geom != 0;
  float h[2] = {1.0f, 1.0f};
  if (sph && act) {
    const int nx = g.n[0], ny = g.n[1];
    const int gx = (int)(cid % (uint32_t)nx), gy = (int)(cid / (uint32_t)nx);
    const Tab<float> tx{A.tab[0], nx + 4, A.uniform[0] ? A.urow[0] : nullptr};
    const Tab<float> ty{A.tab[1], ny + 4, A.uniform[1] ? A.urow[1] : nullptr};
    h[0] = tx(T_HA, bc_pad(gx)) * ty(T_HA, bc_pad(gy));
    h[1] = tx(T_HB, bc_pad(gx)) * ty(T_HB, bc_pad(gy));
  }
  __syncthreads();

  F2* const rE = reinterpret_cast<F2*>(srow + t * RS);
  F2* const rE0 = reinterpret_cast<F2*>(srow + (CPL_THREADS + t) * RS);       // first evaluation: E_g
  F2* const rD0 = reinterpret_cast<F2*>(srow + (2 * CPL_THREADS + t) * RS);   // first evaluation: dE_g/dT
  const bool work = act && g.couple;
  unsigned st = 0;
  // The density, its reciprocal, the kinetic energy and T^- are FP32: they come from the FP32
  // state and set only the FP32 evaluation points of the group energies.  The internal energy u^-
  // = (rho e)^- - kinetic, the iterate T - T^-, the residual and the gas energy update by
  // conservation are NT.
  float rr = 1.0f, ir = 1.0f, ke = 0.0f;
  // budget terms of this cell (reading R13; FP32 like the state they come from, summed in FP64
  // only when the budgets are on): the energy the E floor adds waits in shared memory while the
  // Newton runs (a register held across it cost the loop spills)
  __shared__ float s_floor[CPL_THREADS];
  float work_out = 0.0f;
  NT um = NT(0);
  LT Kc = LT(0), Sc = LT(0), Tst = LT(0);
  float eh = 0.0f, el = 0.0f;
  if (work) {
    // ---- floors, T^- = u^-/(rho c_v), the opacity factors of the (floored) density
    rr = rho_f;
    if (rr < kl.rho_floor) { rr = kl.rho_floor; st |= ST_FLOOR; }
    ir = frcp(rr);
#pragma unroll
    for (int q = 0; q < D; ++q) {
      const float mh = sph ? m_f[q] * frcp(h[q]) : m_f[q];
      ke += 0.5f * mh * mh * ir;
    }
    um = (NT)rhoe_f - (NT)ke;
    if (um < kn.u_floor) { um = kn.u_floor; st |= ST_FLOOR; }
    const LT rcv_f = rr * kl.cv;
    const NT rcv = (NT)rcv_f;
    const LT Tm = to_f32(um) * ir * kl.gm1;  // c_v = 1/(gamma - 1)
    // opacity factors (they only enter the FP32 group arithmetic)
    Kc = kl.kappa0 * hpow(rr, g.kap_rho_h);
    Sc = kl.sigma0 * rr;
    // E^- with its silent positivity floor (Wien tails), and its group sum
    F2 Es2(0.0f), fadd(0.0f);
    for (int j = 0; j < NPR; ++j) {
      F2 e = rE[j];
      if (e.x < kl.E_floor || e.y < kl.E_floor) {
        if (e.x < kl.E_floor) { fadd.x += kl.E_floor - e.x; e.x = kl.E_floor; }
        if (e.y < kl.E_floor && 2 * j + 1 < G) { fadd.y += kl.E_floor - e.y; e.y = kl.E_floor; }
        rE[j] = e;
      }
      Es2 = Es2 + e;
    }
    const LT Esum = Es2.x + Es2.y;
    if (A.budget != nullptr) s_floor[t] = fadd.x + fadd.y;
    const NT ats = (NT)(kl.atol * (to_f32(um) + Esum));
    const LT hh = LT(0.5) * (LT)g.kap_T_h;
    // one evaluation at T: the group sums of E_g(T) - E_g^- (Eq. 25) and of dE_g/dT; the first
    // one also keeps each group's E_g and dE_g/dT (most cells converge from it)
    auto eval = [&](LT Tl, LT& sa, LT& sb, bool keep) {
      const PlanckAt p = planck_at(A.ptab, kl.aN, Tl);
      const LT ck = kl.cdts * (Kc * hpow(Tl, g.kap_T_h));
      const LT hi = hh * p.invT;
      F2 a(0.0f), b(0.0f);
#pragma unroll 1  // (unrolled by two or four: 256^3 x 12 2.72 and 2.68 ms against 2.52)
      for (int j = 0; j < NPR; ++j) {
        F2 Bq, dBq;
        planck_pair(A.ptab, p, j, G, s_ed, Bq, dBq);
        const F2 Em = rE[j];
        const F2 tau = s_ef[j] * ck, inv = frcp(tau + 1.0f);
        const F2 Eg = vfma(tau, Bq, Em) * inv;
        const F2 dEg = (tau * inv) * vfma(F2(hi), Bq - Eg, dBq);
        if (keep) { rE0[j] = Eg; rD0[j] = dEg; }
        a = a + (Eg - Em);
        b = b + dEg;
      }
      sa = a.x + a.y;
      sb = b.x + b.y;
    };

    // ---- Newton with backtracking (Eqs. 26-27; reading R11).  The iterate dl = T - T^- and the
    // residual r are NT; the direction -r/(dr/dT) only needs FP32 (a Newton step is as good as
    // its residual), so dr/dT, the step and the step test are FP32.
    // An FP64 comparison or conversion holds the FP64 pipe for 16 cycles, so the residuals are compared by the
    // integer units (cmp_abs) and values go to FP32 without the compiler's flush test (to_f32): 1024^2 x 16 118 ->
    // 111 us, 256^3 x 12 2.54 -> 2.45 ms.
    NT dl = NT(0), dacc = NT(0), r;
    LT drf, dTf = LT(0), lam = LT(1);
    LT Tacc = Tm;      // T at the accepted point, in FP32
    LT lin = LT(0);    // linearised step added to the accepted group energies at convergence
    int it = 0, ls = 0;
    bool ok = false, done = false, need_dir = true, first = true;  // first: accepted point is T^-
    {
      LT a, b;
      eval(Tacc, a, b, true);
      r = (NT)a;
      drf = rcv_f + b;
    }
    const int guard = g.newton_maxit * 41 + 2;
    for (int kk = 0; kk < guard; ++kk) {
      if (need_dir) {
        if (it >= g.newton_maxit) { done = true; }
        else if (cmp_abs(r, ats) <= 0) { done = true; ok = true; }
        else {
          dTf = -to_f32(r) * frcp(drf);
          ++it;
          if (fabsf(dTf) <= kl.rtol * Tacc) {
            // converged: the group energies at T + dT follow from the linearisation
            dl += (NT)dTf;
            lin = dTf;
            done = true;
            ok = true;
          } else { lam = LT(1); ls = 0; need_dir = false; }
        }
      }
      if (done) break;
      const NT dtt = dl + (NT)(lam * dTf);
      const LT Ttr = Tm + to_f32(dtt);
      const bool valid = Ttr > LT(0);
      const LT Tl = valid ? Ttr : Tacc;
      LT a, b;
      eval(Tl, a, b, false);
      const NT rt = rcv * dtt + (NT)a;
      if (valid && cmp_abs(rt, r) < 0) {
        dl = dtt;
        dacc = dtt;
        Tacc = Tl;
        first = false;
        r = rt;
        drf = rcv_f + b;
        need_dir = true;
      } else {
        lam *= LT(0.5);
        if (++ls >= 40) done = true;
      }
    }
    // ---- bisection fallback on a bracket around [T^-, T_rad] (reading R11), in T - T^-
    if (!ok) {
      const NT Tmn = (NT)Tm;
      const NT Tr = sqrt(sqrt((NT)Esum / (kn.aN * NT(6.4939394022668291491))));  // (sum E / a_R)^(1/4)
      const NT Tc = Tmn + dl;
      NT lo = fmin(fmin(Tc, Tr), Tmn) - Tmn, hi = fmax(fmax(Tc, Tr), Tmn) - Tmn;
      int phase = 0, cnt = 0;
      bool brk = false;
      NT Te = lo;
      for (int kk = 0; kk < 400 + g.bisect_maxit + 4 && phase < 3; ++kk) {
        LT a, b;
        eval(to_f32(Tmn + Te), a, b, false);
        const NT rq = rcv * Te + (NT)a;
        if (phase == 0) {
          if (rq > NT(0) && cnt < 200) { lo = NT(0.5) * (lo + Tmn) - Tmn; ++cnt; }  // T_lo /= 2
          else { phase = 1; cnt = 0; brk = rq <= NT(0); }
        } else if (phase == 1) {
          if (rq < NT(0) && cnt < 200) { hi = NT(2) * (hi + Tmn) - Tmn; ++cnt; }  // T_hi *= 2
          else { brk = brk && rq >= NT(0); cnt = 0; phase = brk ? (g.bisect_maxit > 0 ? 2 : 3) : 3; }
        } else {
          if (rq > NT(0)) hi = Te; else lo = Te;
          ++cnt;
          if (hi - lo <= kn.rtol * (hi + Tmn)) { ok = true; phase = 3; }
          else if (cnt >= g.bisect_maxit) phase = 3;
        }
        Te = phase == 0 ? lo : (phase == 1 ? hi : (phase == 2 ? NT(0.5) * (lo + hi) : Te));
      }
      if (brk) dl = NT(0.5) * (lo + hi);
      dacc = dl;
      lin = LT(0);
      first = false;
    }
    if (!ok) st |= ST_NEWTON;
    Tst = Tm + to_f32(dl);
    if (A.tstar_out != nullptr) A.tstar_out[FXI(cid, ncell)] = Tst;

    // ---- the accepted group energies (from the kept first evaluation when it is the accepted
    // point, else evaluated again), and the group sum of their changes as a float pair (the sum
    // keeps its rounding errors, so the gas energy update sees the changes summed to about twice
    // FP32 precision)
    F2 eh2(0.0f), el2(0.0f);
    auto accept = [&](int j, F2 Eg) {
      F2 s, e;
      two_sum(eh2, Eg - rE[j], s, e);
      eh2 = s;
      el2 = el2 + e;
      rE[j] = Eg;
    };
    if (first) {
#pragma unroll 2
      for (int j = 0; j < NPR; ++j) accept(j, lin != LT(0) ? vfma(rD0[j], F2(lin), rE0[j]) : rE0[j]);
    } else {
      const LT Ta = Tm + to_f32(dacc);
      const PlanckAt p = planck_at(A.ptab, kl.aN, Ta);
      const LT ck = kl.cdts * (Kc * hpow(Ta, g.kap_T_h));
      const LT hi = hh * p.invT;
      for (int j = 0; j < NPR; ++j) {
        F2 Bq, dBq;
        planck_pair(A.ptab, p, j, G, s_ed, Bq, dBq);
        const F2 tau = s_ef[j] * ck, inv = frcp(tau + 1.0f);
        F2 Eg = vfma(tau, Bq, rE[j]) * inv;
        if (lin != LT(0)) Eg = vfma((tau * inv) * vfma(F2(hi), Bq - Eg, dBq), F2(lin), Eg);
        accept(j, Eg);
      }
    }
    // the two halves' sums, joined without loss
    two_sum(eh2.x, eh2.y, eh, el);
    el += el2.x + el2.y;
  }
  // the F rows (into the rows that held the first evaluation)
  __syncthreads();
#pragma unroll
  for (int v = 1; v < NRV; ++v)
    rc.run<true, true>(FXPR(A.out, (size_t)NG * ncell + ((size_t)v * ncell + c0) * G, nc * G, A.n_state), srow + v * CPL_THREADS * RS);
  __syncthreads();
  if (work) {
    // ---- flux absorption at the converged temperature (Eq. 28) and the group sums of the flux
    // changes (in FP32: they reach the gas momentum and energy scaled by 1/c^2, Eqs. 31-32)
    float fh[3] = {0.0f, 0.0f, 0.0f};
    {
      const LT kT = Kc * hpow(Tst, g.kap_T_h);
      F2 f2[D];
#pragma unroll
      for (int q = 0; q < D; ++q) f2[q] = F2(0.0f);
#pragma unroll 2
      for (int j = 0; j < NPR; ++j) {
        const F2 fac = frcp(vfma(F2(kl.cdts), vfma(F2(kT), s_ef[j], F2(Sc)), F2(1.0f)));
#pragma unroll
        for (int q = 0; q < D; ++q) {
          F2* const rF = reinterpret_cast<F2*>(srow + ((1 + q) * CPL_THREADS + t) * RS) + j;
          const F2 Fq = *rF, Fn = Fq * fac;
          f2[q] = f2[q] + (Fn - Fq);
          *rF = Fn;
        }
      }
#pragma unroll
      for (int q = 0; q < D; ++q) fh[q] = f2[q].x + f2[q].y;
    }
    // ---- gas energy by conservation (R12) in NT; the momentum and energy feedback of the flux
    // absorption (Eqs. 31-32) in FP32: it is scaled by 1/c^2, and the FP32 momentum it changes
    // would round it to FP32 anyway
    const NT dEsum = (NT)eh + (NT)el;
    const NT re = (NT)ke + (um - dEsum);
    float vdf = 0.0f;  // v . sum_g dF_g
#pragma unroll
    for (int q = 0; q < D; ++q) {
      vdf += (sph ? m_f[q] * frcp(h[q] * h[q]) : m_f[q]) * ir * fh[q];
      m_f[q] = fmaf(-fh[q], kl.ic2, m_f[q]);
    }
    rhoe_f = (float)(re - (NT)(vdf * kl.ic2));
    rho_f = rr;
    work_out = vdf * kl.ic2;
  }
  if (act) {
    // A NaN or inf anywhere in the cell's outputs makes chk non-finite: a non-finite E_g or F_g
    // reaches the gas energy (through the group sum of the energy changes) or the momentum
    // (through the group sums of the flux changes), so the rows need no scan of their own when
    // the interaction ran.
    float chk = rho_f + rhoe_f;
    A.out[FXI(cid, A.n_state)] = rho_f;
#pragma unroll
    for (int q = 0; q < D; ++q) { A.out[FXI((1 + q) * ncell + cid, A.n_state)] = m_f[q]; chk += m_f[q]; }
    A.out[FXI((NG - 1) * ncell + cid, A.n_state)] = rhoe_f;
    if (!work) {
      for (int v = 0; v < NRV; ++v) {
        const float* rv = srow + (v * CPL_THREADS + t) * RS;
        for (int j = 0; j < G; ++j) chk += rv[j] * 0.0f;
      }
    }
    if (!isfinite(chk)) st |= ST_NONFINITE;
    if (st) atomicOr(A.status, st);
  }
  if (A.budget != nullptr) {
    const double wv = work ? cell_volume(A, cid) * A.bw_cpl : 0.0;
    block_add2((double)work_out * wv, work ? (double)s_floor[t] * wv : 0.0, A.budget + (size_t)(blockIdx.x % BUDGET_SLOTS) * NBUDGET + 6);
  }
  __syncthreads();
  // write the rows back
#pragma unroll
  for (int v = 0; v < NRV; ++v)
    rc.run<false, true>(FXPR(A.out, (size_t)NG * ncell + ((size_t)v * ncell + c0) * G, nc * G, A.n_state), srow + v * CPL_THREADS * RS);
}

}  // namespace fx
