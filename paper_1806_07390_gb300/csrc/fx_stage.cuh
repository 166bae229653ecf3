// SSP-RK2 stage kernel: explicit transport (reconstruction, M1/HLL radiation fluxes, flux divergence
// of gas and radiation) + RK combine in one pass over HBM.  The gas faces run before it
// (gas_face_kernel, fx_gas.cuh) and the cell-local implicit interaction after it, as kernels of
// their own (couple_kernel in fx_couple.cuh for the FP32 state, one thread per cell; couple64_kernel in
// fx_couple64.cuh for the FP64 state, 1 to 16).  Ghost cells are index maps applied when cells are
// loaded (Sec. 7.5): no separate ghost-fill pass touches HBM.
#pragma once
#include <type_traits>

#include "fx_check.cuh"
#include "fx_device.cuh"
#include "fx_pair.cuh"

namespace fx {

// Coupling constants per handle (device memory, staged into shared memory per block).
struct GroupConst {
  double edge[MAXG + 1];   // eps_{g-1/2}, g = 0..G
  double efac[MAXG];       // eps_g^kap_eps_exp
  float edge32[MAXG + 1];
  float efac32[MAXG];
  __device__ __forceinline__ double edge_of(int j, double) const { return edge[j]; }
  __device__ __forceinline__ float edge_of(int j, float) const { return edge32[j]; }
  __device__ __forceinline__ double efac_of(int j, double) const { return efac[j]; }
  __device__ __forceinline__ float efac_of(int j, float) const { return efac32[j]; }
};

// Scalar constants of one launch in the arithmetic type T (filled on the host in FP64 and
// rounded once), so kernels never convert or divide doubles per cell.
template <class T> struct Consts {
  T gamma, gm1, cv, c, ic2, hc, hc2;       // gamma, gamma-1, 1/(gamma-1), c, 1/c^2, c/2, c^2/2
  T kappa0, sigma0, rho_floor, u_floor, E_floor, aN;  // aN = a_R 15/pi^4
  T cdts, dt, alpha, beta;                 // c * coupling step, stage step, RK weights
  T rtol, atol;                            // coupling convergence tolerances
  T idx[3];                                // 1 / cell width per direction (in x, the coordinate)
};

// Planck series coefficients (universal constants), passed by value in the kernel parameters.
struct PlanckParams {
  PlanckCoef c64;
  const double* petab;  // FP64 edge table (fx_planck.h) in device memory; null in the FP32 forms
};

// FP32 Planck band tables on nodes u0 + i/PTAB_PER_OCT of u = log2 T: per group and interval [i, i+1]
// the cubic Hermite polynomial of L(u) = log2 Int_{eps_g-1/2/T}^{eps_g+1/2/T} s^3/(e^s-1) ds through
// the nodes' values and slopes (built on the host in FP64), as
//   L - k = c0 + c1 t + c2 t^2 + c3 t^3,  k = floor(L) at the left node, t in [0, 1].
// The low eight bits of c3, whose term is below 3e-4, hold the exponent field of 2^k (0: 2^k below
// 2^-126, the band flushes to zero), so that small numbers are interpolated and the scale is exact.
// Two groups' coefficients are interleaved, (c0 c0' c1 c1'), (c2 c2' c3 c3'), so that an evaluation
// for both reads two 16-byte words straight into packed FP32 pairs (the nodes' values and slopes were
// four words for two groups).
struct PlanckTable {
  // interval i, pair p of groups at tab[2 (i * si + p * sg)]; the host picks the layout (node-major
  // si = pairs, sg = 1, or group-major si = 1, sg = nu)
  const float4* tab;
  int nu;            // nodes
  float u0;
  int si, sg;
#ifdef FX_BOUNDS_CHECK
  int n;             // words (2 x nu x pairs), for the index checks of the debug build
  unsigned* status;  // status word those checks report to
#endif
};

// Lane value of the stage kernel: a lane owns W groups, two as one packed FP32 pair, one in FP64.
template <class R> struct LaneOf;
template <> struct LaneOf<float> { using V = F2; static constexpr int W = 2; };
template <> struct LaneOf<double> { using V = double; static constexpr int W = 1; };

// Constants of the stage kernel as lane values (pairs of equal floats in FP32: a packed instruction
// takes both halves from registers, and a scalar would be copied into a pair at every use).
template <class V> struct LaneConst {
  V c, mc;              // c, -c
  V c3, mc3;            // c/3, -c/3
  V d1, d2;             // 1/(3c), 2/(3c)
  V m3, p4, q25;        // -3, 4, 1/4
  V hdt[3], mhdt[3];    // stage step / (2 cell width) and its negative
  V alpha, beta;        // RK weights
};

struct VtConst;  // frequency constants of the velocity-dependent terms (fx_vterms.cuh)

template <class R> struct StageArgs {
  DevGrid g;
  PlanckTable ptab;
  const R* faces;      // gas face fluxes and contact speeds [dir][NG+1][faces of dir], then, with
                       // the velocity terms on, D-1 rows of transverse face velocities
  R* faces_out;        // the same buffer, written by gas_face_kernel
  // Face records for the radiation fluxes, four values per face [dir][faces of dir][4]:
  // 2 max(v*, 0), 2 min(v*, 0) (the upwind advection, Eq. 19) and the two sums over the face's
  // cells that give the optical depth of group g (reading R9) as eps_g^d r2 + r3, with r2 =
  // (K_L + K_R) ell/2, K = kappa0 rho^a T^b, and r3 likewise from S = sigma0 rho.  gas_face_kernel
  // writes them, stage_kernel reads them as one 16-byte (FP32) copy per face.
  R* frec;
  int64_t rec_off[3];  // first face of each direction in `frec`
  RadTile rt;          // tile of the stage kernel's radiation blocks
  unsigned char* sflag;  // carbuncle guard (null when off): bit e of a cell's byte is set when a
                         // face of direction e of the cell lies in a shock (shock_flag_kernel)
  int64_t face_off[3]; // element offset of each direction's block in `faces`
  R urow[3][NTAB];     // the common table row of a uniform direction
  int uniform[3];      // direction d has identical table rows (Cartesian grids)
  const R* in;         // state the stencil reads (U^n in stage 1, U^(1) in stage 2)
  const R* base;       // U^n for the stage-2 combination (nullptr in stage 1)
  R* out;              // result (may alias neither input)
  const R* tab[3];     // per-direction reconstruction/divergence tables [NTAB][n_d + 4]
  const GroupConst* gc;
  const VtConst* vtc;  // per-group constants of the velocity-dependent terms
  PlanckParams pk;
  unsigned* status;
#ifdef FX_BOUNDS_CHECK
  int64_t n_state;     // elements of a state (in, base, out, pre_out) and faces in frec, for the index
  int64_t n_recs;      // checks of the debug build
#endif
  double dt;           // stage step
  double dts;          // coupling step (dt after stage 1, dt/2 after stage 2; reading R10)
  double alpha;        // 0 (stage 1) or 1/2 (stage 2)
  int chunk;           // planes per block along the march axis
  // Optional outputs (null when unused).  pre_out: the state after the explicit update and RK
  // combination, before the interaction (state layout); tstar_out: the interaction's converged
  // temperature per cell; phi_out: per row of upper-x boundary faces and group, the radiation
  // energy flux through the face times phi_area, the area of one such face (Cartesian).
  R* pre_out;
  R* tstar_out;
  R* phi_out;
  R phi_area;
  // Budgets (reading R13; null when not accumulated): [0] mass, [1..3] momentum (with the
  // radiation momentum / c^2), [4] total energy and [5] radiation energy that leave through the
  // non-periodic boundaries, [6] the energy the gas gives up to the flux absorption, [7] the
  // radiation energy the positivity floor of E_g adds, [8] the radiation energy the
  // velocity-dependent terms add.  bw_flux weighs this stage's boundary
  // fluxes (dt/2), bw_cpl its interaction (1/2 after stage 1, 1 after stage 2), as the RK
  // combination weighs them in U^(n+1).
  double* budget;
  double bw_flux, bw_cpl;
  int budget_bnd;  // the grid has a non-periodic boundary: the stage kernel adds its outflows
  Consts<double> kd;
  Consts<float> kf;
  LaneConst<typename LaneOf<R>::V> kl;
  __device__ __forceinline__ const Consts<double>& k(double) const { return kd; }
  __device__ __forceinline__ const Consts<float>& k(float) const { return kf; }
};

__device__ __forceinline__ float ex2_approx(float x) {  // 2^x, relative error about 2^-22
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
// 2^k from the low bits of c3
__device__ __forceinline__ float planck_scale(float c3) { return __uint_as_float((__float_as_uint(c3) << 23) & 0x7f800000u); }

__device__ __forceinline__ int bc_pad(int i) { return i + 2; }  // padded table row of cell i

// Map an index along one direction into the domain (ghost cells), Sec. 7.5.
__device__ __forceinline__ int bc_map(int i, int n, int lo, int hi, bool& flip) {
  if (i < 0) {
    if (lo == 1) return i + n;   // periodic
    if (lo == 0) return 0;       // outflow: zero-gradient copy
    flip = !flip;                // reflecting wall / polar axis: mirror, negate normal vectors
    return -1 - i;
  }
  if (i >= n) {
    if (hi == 1) return i - n;
    if (hi == 0) return n - 1;
    flip = !flip;
    return 2 * n - 1 - i;
  }
  return i;
}

}  // namespace fx
#include "fx_gas.cuh"
namespace fx {

template <int GP, class V> __device__ __forceinline__ V seg_sum(V v) {
#pragma unroll
  for (int o = GP / 2; o >= 1; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o, GP);
  return v;
}

// Error-free float addition (Knuth's TwoSum): s = fl(a + b) and s + e = a + b exactly.
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
  s = a + b;
  const float bv = s - a;
  e = (a - (s - bv)) + (b - bv);
}

// Finite-volume update of one conserved variable (Eq. 8), and the RK combination of stage 2:
//   u = cov + dt (src - net),  net = sum_k Fp_k Ap_k - sum_k Fm_k Am_k,  then alpha base + beta u,
// with Fp/Fm the fluxes through the upper/lower faces of each direction and Ap/Am their area over
// volume factors.  In FP32 (precision form (1)) the divergence is a compensated sum: the face
// terms are added with TwoSum and their rounding errors carried in a second float that joins the
// sum before the update (Neumaier's compensated summation), so the divergence is exact up to the
// rounding of each face term; in FP64 the plain sum.
template <int K>
__device__ __forceinline__ float fv_update(const float (&Fp)[K], const float (&Ap)[K], const float (&Fm)[K],
                                           const float (&Am)[K], float cov, float src, float dt,
                                           bool stage2, float base, float alpha, float beta) {
  float s = Fp[0] * Ap[0], c, t;
  two_sum(s, -(Fm[0] * Am[0]), t, c);
  s = t;
#pragma unroll
  for (int k = 1; k < K; ++k) {
    float e;
    two_sum(s, Fp[k] * Ap[k], t, e);
    s = t;
    c += e;
    two_sum(s, -(Fm[k] * Am[k]), t, e);
    s = t;
    c += e;
  }
  const float u = fmaf(dt, (src - s) - c, cov);
  return stage2 ? fmaf(alpha, base, beta * u) : u;
}
// The same for the two groups of a lane, in packed FP32 arithmetic (TwoSum is exact in the
// packed instructions as in the scalar ones: each is the correctly rounded scalar operation).
__device__ __forceinline__ void two_sum(F2 a, F2 b, F2& s, F2& e) {
  s = a + b;
  const F2 bv = s - a;
  e = (a - (s - bv)) + (b - bv);
}
// s = fl(a - b) and s + e = a - b exactly (TwoSum of a and -b, without forming -b).
__device__ __forceinline__ void two_diff(F2 a, F2 b, F2& s, F2& e) {
  s = a - b;
  const F2 bv = s - a;
  e = (a - (s - bv)) - (b + bv);
}
template <int K>
__device__ __forceinline__ F2 fv_update(const F2 (&Fp)[K], const float (&Ap)[K], const F2 (&Fm)[K],
                                        const float (&Am)[K], F2 cov, F2 src, float dt, bool stage2,
                                        F2 base, float alpha, float beta) {
  F2 s = Fp[0] * Ap[0], c, t;
  two_diff(s, Fm[0] * Am[0], t, c);
  s = t;
#pragma unroll
  for (int k = 1; k < K; ++k) {
    F2 e;
    two_sum(s, Fp[k] * Ap[k], t, e);
    s = t;
    c = c + e;
    two_diff(s, Fm[k] * Am[k], t, e);
    s = t;
    c = c + e;
  }
  const F2 u = vfma(F2(dt), (src - s) - c, cov);
  return stage2 ? vfma(F2(alpha), base, beta * u) : u;
}
template <int K>
__device__ __forceinline__ double fv_update(const double (&Fp)[K], const double (&Ap)[K], const double (&Fm)[K],
                                            const double (&Am)[K], double cov, double src, double dt,
                                            bool stage2, double base, double alpha, double beta) {
  double net = Fp[0] * Ap[0] - Fm[0] * Am[0];
#pragma unroll
  for (int k = 1; k < K; ++k) net = net + (Fp[k] * Ap[k] - Fm[k] * Am[k]);
  const double u = cov + dt * (src - net);
  return stage2 ? alpha * base + beta * u : u;
}

// ---------------------------------------------------------------------------------------------
// Planck group energy B_g(T) and dB_g/dT of one lane's group, for code that spreads a cell's
// groups over the lanes of a segment of GP lanes (the adjoint of the interaction): in FP32 from
// the band table of the group; in FP64 from the edge series, each lane evaluating its lower edge
// and taking its upper edge from the next lane (the last group's lane also evaluates the top
// edge).  All lanes of the segment take part.
// ---------------------------------------------------------------------------------------------
template <int GP, class LT>
struct LanePlanck {
  const PlanckParams& pk;
  const PlanckTable& ptab;
  int lane;
  bool has;       // lane < G
  bool top2;      // this lane also evaluates the top edge (G == GP)
  LT aN;          // a_R 15 / pi^4
  LT elo, etop;   // lower and upper edge of this lane's group

  // FP32 group energy B_g(T) and T dB_g/dT from the band table of this lane's group
  __device__ __forceinline__ void planck_tab(float T, float invT, float& B, float& dB) const {
    const float s = (__log2f(T) - ptab.u0) * float(PTAB_PER_OCT);
    float I, dLdu;
    if (s < 0.0f) {
      I = 0.0f;  // every band of this group is deep in the Wien tail
      dLdu = 0.0f;
    } else if (s >= float(ptab.nu - 1)) {
      // very hot: x = eps/T < 2^-14, so Int t^3/(e^t-1) = x^3/3 - x^4/8 + O(x^5)
      const float a = (float)elo * invT, b = (float)etop * invT;
      const float a3 = a * a * a, b3 = b * b * b;
      I = (b3 - a3) * (1.0f / 3.0f) - (b3 * b - a3 * a) * 0.125f;
      dLdu = ((a3 * a * (1.0f - 0.5f * a)) - (b3 * b * (1.0f - 0.5f * b))) * frcp(I);
    } else {
      const int i = (int)s;
      const float t = s - (float)i;
      const float* const c = reinterpret_cast<const float*>(FXP_AT(ptab.status, ptab.tab, 2 * (i * ptab.si + (lane >> 1) * ptab.sg), ptab.n - 1)) + (lane & 1);
      const float c0 = __ldg(c), c1 = __ldg(c + 2), c2 = __ldg(c + 4), c3 = __ldg(c + 6);
      const float dLdt = fmaf(fmaf(3.0f * c3, t, 2.0f * c2), t, c1);
      I = ex2_approx(fmaf(fmaf(fmaf(c3, t, c2), t, c1), t, c0)) * planck_scale(c3);
      dLdu = dLdt * float(PTAB_PER_OCT);
    }
    const float T2 = T * T, T3 = T2 * T;
    B = (float)aN * T3 * T * I;
    dB = (float)aN * T3 * I * (4.0f + dLdu);  // d/dT (T^4 I) = T^3 I (4 + d ln I / d ln T)
  }

  // this lane's group energy B_g(T) and dB_g/dT (all lanes of the segment take part: the FP64
  // form shares edge integrals between neighbouring lanes)
  __device__ __forceinline__ void planck(LT Tl, LT invT, LT& Bq, LT& dBq) const {
    if (sizeof(LT) == 4) {
      float B_, dB_;
      if (has) planck_tab((float)Tl, (float)invT, B_, dB_);
      else { B_ = 0.0f; dB_ = 0.0f; }
      Bq = (LT)B_;
      dBq = (LT)dB_;
    } else {
      PlanckEdge<double> lo = planck_edge_tab((double)(elo * invT) * 16.0, pk.petab, pk.c64);
      PlanckEdge<double> hi;
      hi.Q = __shfl_down_sync(0xffffffffu, lo.Q, 1, GP);
      hi.w = __shfl_down_sync(0xffffffffu, lo.w, 1, GP);
      hi.upper = __shfl_down_sync(0xffffffffu, (int)lo.upper, 1, GP) != 0;
      if (top2) hi = planck_edge_tab((double)(etop * invT) * 16.0, pk.petab, pk.c64);
      LT I = (LT)planck_band(lo, hi);
      LT T3 = Tl * Tl * Tl;
      Bq = aN * T3 * Tl * I;
      dBq = aN * T3 * (LT(4) * I + (LT)(lo.w - hi.w));
    }
  }
};

// Volume of cell cid (the product of its 1-d volume factors), for the budgets (reading R13).
template <class R> __device__ __forceinline__ double cell_volume(const StageArgs<R>& A, uint32_t cid) {
  const DevGrid& g = A.g;
  if (A.uniform[0] && (g.D < 2 || A.uniform[1]) && (g.D < 3 || A.uniform[2])) {
    // uniform spacing in every direction: every cell has the same volume
    double v = (double)A.urow[0][T_VOL];
    if (g.D >= 2) v *= (double)A.urow[1][T_VOL];
    if (g.D >= 3) v *= (double)A.urow[2][T_VOL];
    return v;
  }
  const uint32_t nx = (uint32_t)g.n[0], ny = (uint32_t)g.n[1];
  const int gx = (int)(cid % nx), gy = (int)((cid / nx) % ny), gz = (int)(cid / (nx * ny));
  double v = (double)Tab<R>{A.tab[0], g.n[0] + 4, A.uniform[0] ? A.urow[0] : nullptr}(T_VOL, bc_pad(gx));
  if (g.D >= 2) v *= (double)Tab<R>{A.tab[1], g.n[1] + 4, A.uniform[1] ? A.urow[1] : nullptr}(T_VOL, bc_pad(gy));
  if (g.D >= 3) v *= (double)Tab<R>{A.tab[2], g.n[2] + 4, A.uniform[2] ? A.urow[2] : nullptr}(T_VOL, bc_pad(gz));
  return v;
}

// Block sums of a and b (blocks of whole warps, at most 1024 threads) added to out[0], out[1] by
// one thread.  Every thread of the block calls it.
__device__ __forceinline__ void block_add2(double a, double b, double* out) {
  __shared__ double red[2][32];
#pragma unroll
  for (int o = 16; o >= 1; o >>= 1) {
    a += __shfl_xor_sync(0xffffffffu, a, o);
    b += __shfl_xor_sync(0xffffffffu, b, o);
  }
  if ((threadIdx.x & 31) == 0) {
    red[0][threadIdx.x >> 5] = a;
    red[1][threadIdx.x >> 5] = b;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double sa = 0.0, sb = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) { sa += red[0][w]; sb += red[1][w]; }
    if (sa != 0.0) atomicAdd(out, sa);
    if (sb != 0.0) atomicAdd(out + 1, sb);
  }
}

// Asynchronous global -> shared copies of single elements (cp.async, sm_80 and later): the
// stage kernel stages each march plane into shared memory one step ahead, without passing the
// values through registers.  A thread's copies are complete, and visible to that thread, after
// its wait; other threads see them after the next barrier.
template <class R> __device__ __forceinline__ void cp_async(R* smem, const R* gmem) {
  const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
  if constexpr (sizeof(R) == 4)
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(sa), "l"(gmem) : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(sa), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }

// cp.async of one lane value (the lane's groups: both values of a pair where they are 8-byte
// aligned in global memory and both exist, else one by one).
__device__ __forceinline__ void cp_async_lane(F2* s, const float* g, bool vec, bool h1) {
  const unsigned sa = (unsigned)__cvta_generic_to_shared(s);
  if (vec) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(sa), "l"(g) : "memory");
  } else {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(sa), "l"(g) : "memory");
    if (h1) asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(sa + 4), "l"(g + 1) : "memory");
  }
}
__device__ __forceinline__ void cp_async_lane(double* s, const double* g, bool, bool) { cp_async(s, g); }
__device__ __forceinline__ void cp_async16(void* s, const void* g) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"((unsigned)__cvta_generic_to_shared(s)), "l"(g) : "memory");
}

// ---------------------------------------------------------------------------------------------
// The stage kernel (one launch per RK stage, after gas_face_kernel).
//
// Radiation blocks.  A group's transport does not see the other groups, so a cell is served by
// exactly as many lanes as its groups need: GL = ceil(G / W) lanes of W groups, W = 2 as one packed
// FP32 pair (F2), W = 1 in FP64.  A block owns a tile of TX x TY cells (TY = 1 below 3-d),
// tid = cell * GL + lane, and marches along the slowest axis over a chunk of planes.  The tile is
// chosen at run time (fit_tile): all shared arrays are addressed by tid and compile-time
// capacities, so no group or tile count is a template parameter and no lane is padding.
//   ring   four planes of the tile's own cells [slot][v][NT]: a thread copies its own cell with
//          cp.async three planes ahead and reads its own march column from it;
//   halo   two cells on each in-plane side, two planes [parity][v][NH GL];
//   rec    the face records that gas_face_kernel wrote (upwind speeds and opacity sums), two planes;
//   xb, yb the state left of every in-plane face, overwritten by the face's flux.
// Per plane k:
//   A  issue the copies of plane k+3 (own cells), of plane k+1 (halo, records) and of the stage-2
//      base of plane k;
//   B  reconstruct each cell once per direction, the halo cells as extra tasks spread over the
//      block's threads;                                                             -- barrier
//   C  the fluxes through the cell's lower faces and its march face k+1/2, the tile's upper faces
//      as extra tasks; wait for the copies of A;                                    -- barrier
//   D  divergence, RK combination, store.
//
// On a Cartesian grid every direction is uniform, so the kernel needs no table: the half slopes
// of the limiter give the face states, and the divergence is formed from the differences of the
// two fluxes of a direction (exact as s + e by TwoSum in FP32), scaled by dt / (2 dx) and summed with
// all rounding errors (net_update): twice the flux is carried, which saves the halvings of the two-state
// averages.
//
// Gas blocks.  The gas update of a cell needs only the face fluxes in the face buffer: the last
// blocks of the grid do it, one thread per cell, in the slots that the radiation blocks leave free
// and as they finish (no launch of its own, and no gas variables in the radiation blocks).
//
// Bound by instruction issue and by the latency between the plane barriers (1024^2 x 16: 351 thread
// instructions per cell and group, issued in 66 % of cycles at 20 warps per multiprocessor; 128^3 x 12:
// 690 in 57 % at 16 warps; DRAM 1.1x the algorithmic bytes), the FP64 state by the FP64 pipe (87
// % busy, 224 operations per cell and group).  Measured (FP32 state unless noted, one launch):
// 1024^2 x 16 groups 0.455 -> 0.241 ms, 256^3 x 12 16.4 -> 6.6 ms, 640 x 128 x 20 spherical 0.124 ->
// 0.047 ms, 512^2 x 24 channels 0.23 -> 0.098 ms, 512^2 x 16 FP64 2.99 -> 1.84 ms, against one kernel
// with lanes padded to a power of two, geometry tables on every grid, and the gas update in its lanes.
// (The variants below were measured while the divergence took the shorter sum that net_update names.)
//
// Block sizes (StageCap).  A thread holds about 90 values at order 1, so 20 warps of 96 registers in
// 2-d (4 blocks of 160: 2 of 256 0.244 ms, 3 of 160 0.229 ms but the 24-channel and 400 x 300 grids
// 6 to 8 % slower, 5 of 160 0.264 ms) and, with the second in-plane direction, 16 warps of 128 in 3-d
// (256^3 x 12, 2 blocks of 256: 6.2 ms; 4 of 128 6.4, 3 of 192 spill 7.3, 1 of 512 6.5: larger tiles
// have less halo).
//
// VEC (FP32 below 3-d): an even group count on aligned buffers, so every lane's pair is complete and
// is copied and stored as one 8-byte word without a test (1024^2 x 16 234 -> 229 us with the slots
// rotated, 515 x 389 x 7 34.4 -> 32.4, 96 x 80 x 8 10.4 -> 8.8; in 3-d 0.6 % slower, so tested there).
//
// SPH selects the spherical (r, theta) geometry, RO the radiation reconstruction (1: linear with
// the MC limiter, the paper's; 2: the gas's parabola), BUD the boundary-outflow budgets (R13).
// ---------------------------------------------------------------------------------------------
template <class R, int D> struct StageCap {
  static constexpr int NT = sizeof(R) == 8 ? 256 : (D == 3 ? 256 : 160);  // most threads per block
  static constexpr int XP = sizeof(R) == 8 ? 128 : 64;  // room for the upper face of every row
  // ... and for the threads past the tile (at most 31), which run along on entries of their own
  static constexpr int XC = NT + XP + 32 + (D == 3 ? XP : 32);
  static constexpr int PB = D == 3 ? 1 : 2;             // planes of xb (and yb) in use at once
  static constexpr int MINB = sizeof(R) == 8 ? 2 : (D == 3 ? 2 : 4);  // resident blocks aimed at
};

// Halo cells per plane and face records per plane of a tile.
template <int D> __host__ __device__ inline int tile_halo(const RadTile& t) { return 4 * t.ty + (D == 3 ? 4 * t.tx : 0); }
template <int D> __host__ __device__ inline int tile_recs(const RadTile& t) {
  return (t.tx + 1) * t.ty + (D == 3 ? t.tx * (t.ty + 1) : 0) + (D >= 2 ? t.tx * t.ty : 0);
}

// Shared memory of stage_kernel: offsets in lane values (8 bytes), the records last.
template <class R, int D> struct StageLayout {
  using C = StageCap<R, D>;
  static constexpr int NRV = 1 + D;
  int ring, base, xb, yb, xr, yr, halo, rec, end;
  __host__ __device__ explicit StageLayout(const RadTile& t) {
    ring = 0;
    base = ring + (D == 1 ? 1 : 4) * NRV * C::NT;
    xb = base + NRV * C::NT;
    yb = xb + C::PB * NRV * C::XC;
    xr = yb + (D == 3 ? C::PB * NRV * C::XC : 0);
    yr = xr + NRV * t.ty * t.gl;
    halo = yr + (D == 3 ? NRV * t.tx * t.gl : 0);
    rec = (halo + (D == 3 ? 2 * NRV * tile_halo<D>(t) * t.gl : NRV * C::NT) + 1) & ~1;  // 16-byte aligned
    end = rec + 2 * tile_recs<D>(t) * (4 * (int)sizeof(R) / 8);
  }
};
template <class R, int D> inline size_t stage_smem_bytes(const RadTile& t) { return (size_t)StageLayout<R, D>(t).end * 8; }

// 1/(cE), s = sqrt(4 - 3 f^2) and f^2 of a radiation state, f = |F|/(cE); 1/(cE) is 0 for E <= 0.
template <int D>
__device__ __forceinline__ void m1_state(const LaneConst<F2>& K, F2 cE, const F2* F, F2& iE, F2& f2, F2& s) {
  F2 FF = F[0] * F[0];
#pragma unroll
  for (int q = 1; q < D; ++q) FF = vfma(F[q], F[q], FF);
  iE = F2(cE.x > 0.0f ? rcp_approx(cE.x) : 0.0f, cE.y > 0.0f ? rcp_approx(cE.y) : 0.0f);
  f2 = (FF * iE) * iE;
  s = vsqrt(vfma(K.m3, vmin(f2, F2(1.0f)), K.p4));
}
template <int D>
__device__ __forceinline__ void m1_state(const LaneConst<double>& K, double cE, const double* F, double& iE,
                                         double& f2, double& s) {
  double FF = F[0] * F[0];
#pragma unroll
  for (int q = 1; q < D; ++q) FF = fma(F[q], F[q], FF);
  iE = normal_pos(cE) ? rcp64(cE) : 0.0;
  f2 = (FF * iE) * iE;
  s = sqrt64(fma(K.m3, __double2hiint(f2) >= 0x3ff00000 ? 1.0 : f2, K.p4));
}
__device__ __forceinline__ F2 max1(F2 f2) { return vmax(f2, F2(1.0f)); }
__device__ __forceinline__ double max1(double f2) { return __double2hiint(f2) >= 0x3ff00000 ? f2 : 1.0; }  // f2 >= 0
__device__ __forceinline__ F2 rcp_fast(F2 x) { return F2(rcp_approx(x.x), rcp_approx(x.y)); }
// (x > 0; 0 for an infinite x: f^2 overflows where a flux meets a cell whose energy lies at its floor, and
// rcp64 has no value there)
__device__ __forceinline__ double rcp_fast(double x) { return __double2hiint(x) == 0x7ff00000 ? 0.0 : rcp64(x); }

// c^2 times row n of the M1 pressure tensor (reading R7) for the lane's groups.  With f = |F|/(cE)
// and s = sqrt(4 - 3 f^2), f^2 = (4 - s^2)/3 turns the closure's two coefficients into
//   (1 - chi)/2 = (s - 1)/3,   (3 chi - 1)/2 = 3 f^2/(2 + s),
// so c^2 P_nq = cE (c/3)(s - 1) delta_nq + F_n F_q / ((2 + s) cE/(3c)): one reciprocal of cE, one square
// root, one reciprocal.  f > 1 keeps the direction with f clamped to 1 (the factor max(f^2, 1) in
// the second reciprocal's argument, which is 0 where f^2 overflows); E <= 0 is isotropic (1/(cE) taken
// as 0).
template <int D, class V>
__device__ __forceinline__ void m1_c2row(const LaneConst<V>& K, V E, const V* F, int n, V* P) {
  const V cE = E * K.c;
  V iE, f2, s;
  m1_state<D>(K, cE, F, iE, f2, s);
  const V diag = cE * vfma(s, K.c3, K.mc3);
  const V w = rcp_fast(vfma(s, K.d1, K.d2) * max1(f2)) * iE * F[n];
#pragma unroll
  for (int q = 0; q < D; ++q) P[q] = q == n ? vfma(w, F[q], diag) : w * F[q];
}
// The entry of c^2 P perpendicular to F (the closure's isotropic part).
template <int D, class V> __device__ __forceinline__ V m1_c2perp(const LaneConst<V>& K, V E, const V* F) {
  const V cE = E * K.c;
  V iE, f2, s;
  m1_state<D>(K, cE, F, iE, f2, s);
  return cE * vfma(s, K.c3, K.mc3);
}

// dt times the divergence of a cell on a uniform grid, from twice the fluxes: x, (3-d) y, march; h the
// factors dt / (2 dx), mh their negatives.  In FP32 (precision form (1)) the sum is compensated
// throughout: each direction's difference is s + e exactly (TwoSum), its product with h is split by an
// FMA, the directions are added by TwoSum, and the errors of all three are summed beside (ml, the negated
// sum of what the high part n has lost) and join it at the end, so that directions that cancel leave no
// rounding of their parts.  Without the errors of the products and of the sum over directions, and with
// Dekker's shorter difference, the kernel took 229 us instead of 241 at 1024^2 x 16 groups and 6.24 ms
// instead of 6.57 at 256^3 x 12, but left 1e-7 of the parts where the directions cancel.
template <int D>
__device__ __forceinline__ F2 net_update(F2 xp, F2 xm, F2 yp, F2 ym, F2 mp, F2 mm, const F2* h, const F2* mh) {
  F2 s, e;
  two_diff(xp, xm, s, e);
  F2 n = s * h[0], ml = vfma(e, mh[0], vfma(s, mh[0], n));
  auto add = [&](F2 up, F2 lo, F2 hd, F2 mhd) {
    two_diff(up, lo, s, e);
    const F2 p = s * hd;
    F2 t, r;
    two_sum(n, p, t, r);
    n = t;
    ml = vfma(e, mhd, ml + (vfma(s, mhd, p) - r));
  };
  if (D == 3) add(yp, ym, h[1], mh[1]);
  if (D >= 2) add(mp, mm, h[D - 1], mh[D - 1]);
  return n - ml;
}
template <int D>
__device__ __forceinline__ double net_update(double xp, double xm, double yp, double ym, double mp, double mm, const double* h,
                                             const double*) {
  double n = (xp - xm) * h[0];
  if (D == 3) n = fma(yp - ym, h[1], n);
  if (D >= 2) n = fma(mp - mm, h[D - 1], n);
  return n;
}

// Gas update of one cell per thread (the gas blocks of stage_kernel): the divergence of the face
// fluxes, the geometric sources of the spherical grid, the RK combination and, with BUD, the
// boundary outflows.
template <class R, int D, bool SPH, bool BUD>
__device__ __forceinline__ void gas_update(const StageArgs<R>& A, uint32_t cid) {
  constexpr int NG = 2 + D, MD = D - 1;
  const DevGrid& g = A.g;
  const Consts<R>& KR = A.k(R(0));
  const uint32_t ncell = (uint32_t)g.ncell;
  if (cid >= ncell) return;
  const int nx = g.n[0], ny = g.n[1], nz = g.n[2];
  const int gx = D == 1 ? (int)cid : (int)(cid % (uint32_t)nx);
  const int gy = D == 1 ? 0 : (D == 2 ? (int)(cid / (uint32_t)nx) : (int)((cid / (uint32_t)nx) % (uint32_t)ny));
  const int gz = D == 3 ? (int)(cid / ((uint32_t)nx * ny)) : 0;
  const int gi[3] = {gx, gy, gz};
  const Tab<R> tx{A.tab[0], nx + 4, A.uniform[0] ? A.urow[0] : nullptr};
  const Tab<R> ty{A.tab[D >= 2 ? 1 : 0], (D >= 2 ? ny : nx) + 4, A.uniform[D >= 2 ? 1 : 0] ? A.urow[D >= 2 ? 1 : 0] : nullptr};
  const Tab<R> tz{A.tab[D >= 3 ? 2 : 0], (D >= 3 ? nz : nx) + 4, A.uniform[D >= 3 ? 2 : 0] ? A.urow[D >= 3 ? 2 : 0] : nullptr};
  const uint32_t nfd[3] = {(uint32_t)(nx + 1) * (D > 1 ? ny : 1) * (D > 2 ? nz : 1),
                           (uint32_t)nx * (ny + 1) * (D > 2 ? nz : 1), (uint32_t)nx * ny * (nz + 1)};
  const uint32_t fl[3] = {((uint32_t)gz * ny + gy) * (nx + 1) + gx, ((uint32_t)gz * (ny + 1) + gy) * nx + gx, cid};
  const uint32_t fs[3] = {1u, (uint32_t)nx, (uint32_t)nx * ny};  // to the upper face
  auto face = [&](int d, int v, uint32_t f) -> R {
    const R* const fr = A.faces + A.face_off[d];  // (64 bits: the blocks before this one may hold 2^32 elements)
    return __ldg(FXP(fr, v * nfd[d] + f, (NG + 1 + (g.vterms ? D - 1 : 0)) * nfd[d]));
  };
  R u0[NG];
#pragma unroll
  for (int v = 0; v < NG; ++v) u0[v] = A.in[FXI(v * ncell + cid, A.n_state)];
  R src[NG];
#pragma unroll
  for (int v = 0; v < NG; ++v) src[v] = R(0);
  const int ipx = bc_pad(gx), ipm = bc_pad(gy);
  if (SPH) {
    const R h0 = tx(T_HA, ipx) * ty(T_HA, ipm), h1 = tx(T_HB, ipx) * ty(T_HB, ipm);
    const R g111 = tx(T_GA, ipx), g221 = tx(T_GB, ipx), g122 = tx(T_GC, ipx);
    const R g222 = ty(T_GA, ipm), g332 = ty(T_GB, ipm);
    const R rho = u0[0], irho = frcp(rho);
    const R v1 = u0[1] * irho * frcp(h0), v2 = u0[2] * irho * frcp(h1);
    const R p = KR.gm1 * (u0[NG - 1] - R(0.5) * rho * (v1 * v1 + v2 * v2));
    const R r12 = h0 * frcp(h1), r21 = h1 * frcp(h0);
    src[1] = g111 * (rho * v1 * v1 + p) + g221 * (rho * v2 * v2 + p) + g221 * p;
    src[2] = g122 * (rho * v1 * v2 * r12) + g221 * (rho * v1 * v2 * r21) + g222 * (rho * v2 * v2 + p) + g332 * p;
  }
  const bool stage2 = A.base != nullptr;
  R chk = R(0);
  double out[NG];  // budgets
#pragma unroll
  for (int v = 0; v < NG; ++v) {
    R Fp[D], Ap[D], Fm[D], Am[D];
#pragma unroll
    for (int d = 0; d < D; ++d) {
      Fm[d] = face(d, v, fl[d]);
      Fp[d] = face(d, v, fl[d] + fs[d]);
    }
    // area/volume factors (Eq. 8): scalar variables, and covariant components 0 and 1
    const int eL[3] = {T_FL, T_FL1, T_FL2}, eR[3] = {T_FR, T_FR1, T_FR2}, eX[3] = {T_XS, T_X1, T_X2};
    const int c = (v >= 1 && v <= 2 && v <= D) ? v : 0;
    if (SPH) {
      Ap[0] = tx(eR[c], ipx) * ty(eX[c], ipm);
      Am[0] = tx(eL[c], ipx) * ty(eX[c], ipm);
      Ap[D - 1] = ty(eR[c], ipm) * tx(eX[c], ipx);
      Am[D - 1] = ty(eL[c], ipm) * tx(eX[c], ipx);
    } else {
      Ap[0] = tx(T_FR, ipx);
      Am[0] = tx(T_FL, ipx);
      if (D >= 2) { Ap[D >= 2 ? 1 : 0] = ty(T_FR, ipm); Am[D >= 2 ? 1 : 0] = ty(T_FL, ipm); }
      if (D == 3) { Ap[D == 3 ? 2 : 0] = tz(T_FR, bc_pad(gz)); Am[D == 3 ? 2 : 0] = tz(T_FL, bc_pad(gz)); }
    }
    const R b = stage2 ? A.base[FXI(v * ncell + cid, A.n_state)] : R(0);
    const R un = fv_update(Fp, Ap, Fm, Am, u0[v], src[v], KR.dt, stage2, b, KR.alpha, KR.beta);
    A.out[FXI(v * ncell + cid, A.n_state)] = un;
    if (A.pre_out != nullptr) A.pre_out[FXI(v * ncell + cid, A.n_state)] = un;
    chk += un * R(0);
    if (BUD) {
      double o = 0.0;
#pragma unroll
      for (int d = 0; d < D; ++d) {
        if (gi[d] == g.n[d] - 1 && g.bc_hi[d] != 1) o += (double)(Fp[d] * Ap[d]);
        if (gi[d] == 0 && g.bc_lo[d] != 1) o -= (double)(Fm[d] * Am[d]);
      }
      out[v] = o;
    }
  }
  if (!isfinite(chk)) atomicOr(A.status, ST_NONFINITE);
  if (BUD && A.budget != nullptr) {
    bool edge = false;
#pragma unroll
    for (int d = 0; d < D; ++d)
      edge |= (gi[d] == 0 && g.bc_lo[d] != 1) || (gi[d] == g.n[d] - 1 && g.bc_hi[d] != 1);
    if (edge) {
      double vol = (double)tx(T_VOL, ipx);
      if (D >= 2) vol *= (double)ty(T_VOL, ipm);
      if (D == 3) vol *= (double)tz(T_VOL, bc_pad(gz));
      const double bs = vol * A.bw_flux;
      double* const bud = A.budget + (size_t)(blockIdx.x % BUDGET_SLOTS) * NBUDGET;
#pragma unroll
      for (int v = 0; v < NG; ++v)
        if (out[v] != 0.0) atomicAdd(bud + (v == NG - 1 ? 4 : v), out[v] * bs);
    }
  }
  (void)MD;
}

template <class R, int D, bool SPH, int RO, bool BUD, bool VEC>
__global__ void __launch_bounds__((StageCap<R, D>::NT), (StageCap<R, D>::MINB))
stage_kernel(const __grid_constant__ StageArgs<R> A) {
  static_assert(!SPH || D == 2, "the spherical geometry is 2-d (r, theta)");
  using CP = StageCap<R, D>;
  using V = typename LaneOf<R>::V;
  constexpr int W = LaneOf<R>::W;
  constexpr int NG = 2 + D, NRV = 1 + D, MD = D - 1;
  constexpr int NT = CP::NT, XC = CP::XC, PB = CP::PB;
  constexpr bool TABLES = SPH || RO == 2;  // the reconstruction reads the geometry tables
  const int NTH = (int)blockDim.x, tid = (int)threadIdx.x;
  const RadTile& RT = A.rt;
  if (blockIdx.x >= (unsigned)RT.nrad) {  // gas blocks: cells in strides of the gas blocks' threads
    const uint32_t nthr = (gridDim.x - (unsigned)RT.nrad) * (uint32_t)NTH;
    for (uint32_t c = (blockIdx.x - (unsigned)RT.nrad) * (uint32_t)NTH + tid; c < (uint32_t)A.g.ncell; c += nthr)
      gas_update<R, D, SPH, BUD>(A, c);
    return;
  }
  const DevGrid& g = A.g;
  const Consts<R>& KR = A.k(R(0));
  const LaneConst<V>& KL = A.kl;
  const int G = g.G, GL = RT.gl, TX = RT.tx, TY = D == 3 ? RT.ty : 1, TC = TX * TY;
  const int nx = g.n[0], ny = g.n[1], nz = g.n[2];
  const uint32_t ncell = (uint32_t)g.ncell;  // the host keeps every state offset below 2^32
  // block -> tile and chunk
  const int bt = (int)blockIdx.x;
  const int btx = bt % RT.ntx, btr = bt / RT.ntx;
  const int bty = D == 3 ? btr % RT.nty : 0, bck = D == 3 ? btr / RT.nty : btr;
  const int x0 = btx * TX, y0 = D == 3 ? bty * TY : 0;
  const int nmarch = D == 1 ? 1 : g.n[MD];
  const int kbeg = D == 1 ? 0 : bck * A.chunk;
  const int kend = D == 1 ? 1 : min(kbeg + A.chunk, nmarch);
  const int tcell = tid / GL, lane = tid - tcell * GL;
  // the last warp's threads past the tile run along on a copy of cell 0 and entries of their own
  const bool act = tcell < TC;
  const int tc = act ? tcell : 0;
  const int lx = D == 3 ? tc % TX : tc, ly = D == 3 ? tc / TX : 0;
  const int g0 = lane * W;
  const bool h1 = W == 2 && (VEC || g0 + 1 < G);
  const bool vec = VEC || (D == 3 && RT.vec != 0);  // pairs copied and stored whole (all complete and aligned)

  extern __shared__ __align__(16) unsigned char smem_raw[];
  V* const sm = reinterpret_cast<V*>(smem_raw);
  const StageLayout<R, D> L(RT);
  const int NH = tile_halo<D>(RT), HS = NH * GL, NREC = tile_recs<D>(RT);
  V* const ring = sm + L.ring;
  V* const sbase = sm + L.base;
  V* const xb = sm + L.xb;
  V* const yb = sm + L.yb;
  V* const xr = sm + L.xr;
  V* const yr = sm + L.yr;
  V* const halo = sm + L.halo;
  R* const rec = reinterpret_cast<R*>(sm + L.rec);
  const int n_ring = (D == 1 ? 1 : 4) * NRV * NT, n_base = NRV * NT, n_xb = PB * NRV * XC;
  const int n_xr = NRV * TY * GL, n_yr = NRV * TX * GL, n_halo = D == 3 ? 2 * NRV * HS : NRV * NT, n_rec = 8 * NREC;
  // halo planes: variable stride and offset of the second plane (below 3-d the ring's stride, so that
  // both are read with the same immediate offsets; two planes fit in it, fit_tile)
  const int HV = D == 3 ? HS : NT, HPAR = D == 3 ? NRV * HS : HS;
  (void)n_ring; (void)n_base; (void)n_xb; (void)n_xr; (void)n_yr; (void)n_halo; (void)n_rec;

  // The geometry tables, a row at a time: a Cartesian direction has one row for every cell (of the
  // launch arguments).  On the spherical grid a thread keeps the address of its own cell's row and
  // takes the other rows (halo cells, planes) once for all their entries; every entry fetched
  // through the general reader (Tab) made 640 x 128 x 20 67 us instead of 50.
  using TT = typename std::conditional<SPH, TabAt<R>, TabRow<R>>::type;
  auto row_of_dir = [&](int d, int i) -> TT {
    if constexpr (SPH) return TT(A.tab[d], g.n[d], bc_pad(i));
    else return TT{A.urow[d]};
  };

  // ---- positions.  Ghost cells are index maps (Sec. 7.5); tiles may overhang the grid, their
  // cells past the first two ghosts are never used and clamped into the array.
  auto map_x = [&](int x, bool& f) { return min(max(bc_map(x, nx, g.bc_lo[0], g.bc_hi[0], f), 0), nx - 1); };
  auto map_y = [&](int y, bool& f) { return min(max(bc_map(y, ny, g.bc_lo[1], g.bc_hi[1], f), 0), ny - 1); };
  auto map_m = [&](int k, bool& f) {
    if (D == 1) return 0;
    return min(max(bc_map(k, nmarch, g.bc_lo[MD], g.bc_hi[MD], f), 0), nmarch - 1);
  };
  const uint32_t pcells = D == 1 ? 0u : (D == 2 ? (uint32_t)nx : (uint32_t)nx * ny);  // cells per plane
  auto inplane = [&](int sx, int sy, bool& fx, bool& fy) -> uint32_t {  // of tile cell (sx, sy)
    const uint32_t cx = (uint32_t)map_x(x0 + sx, fx);
    return D == 3 ? (uint32_t)map_y(y0 + sy, fy) * nx + cx : cx;
  };
  // t / GL for the task indices (t < 2^16: exact with mgl = ceil(2^32 / GL))
  auto div_gl = [&](int t) -> int { return GL == 1 ? t : (int)__umulhi((unsigned)t, RT.mgl); };
  // halo cell h: 4 per row (-2, -1, TX, TX+1), then (3-d) 4 rows of TX (-2, -1, TY, TY+1)
  auto halo_pos = [&](int h, int& sx, int& sy) {
    if (D < 3 || h < 4 * TY) { const int r = h >> 2, c = h & 3; sy = r; sx = c < 2 ? c - 2 : TX + (c - 2); }
    else { const int j = h - 4 * TY, r = j / TX; sx = j - r * TX; sy = r < 2 ? r - 2 : TY + (r - 2); }
  };
  bool fx_own = false, fy_own = false;
  const uint32_t cxy = inplane(lx, ly, fx_own, fy_own);
  const int gx = x0 + lx, gy = y0 + ly;
  const TT tx = row_of_dir(0, gx), ty = row_of_dir(D == 3 ? 1 : 0, gy);  // rows of the own cell
  const bool cell_in = act && gx < nx && (D < 3 || gy < ny);
  const uint32_t toff = cxy * (uint32_t)G + g0;  // the thread's elements in a plane of a radiation variable
  const uint32_t vstride = ncell * (uint32_t)G, pstride = pcells * (uint32_t)G;
  // The halo entries and face records that this thread copies: the first ones (one halo entry, two
  // in 3-d; two records) keep their element offsets in registers, more of them (tiles of few cells
  // with many lanes) recompute theirs.  Halo entries go to the threads from the last one down, so
  // that they and the records fall to different warps.
  constexpr int HP = D == 3 ? 2 : 1, RP = 2;
  const int ht0 = NTH - 1 - tid;
  auto halo_entry = [&](int t, uint32_t& off, bool& two) {
    const int h = div_gl(t), ln = t - h * GL;
    int sx, sy;
    bool f0 = false, f1 = false;
    halo_pos(h, sx, sy);
    off = inplane(sx, sy, f0, f1) * (uint32_t)G + ln * W;
    two = W == 2 && (VEC || ln * W + 1 < G);
  };
  uint32_t hoff[HP];
  bool hh1[HP];
#pragma unroll
  for (int p = 0; p < HP; ++p) {
    hoff[p] = 0;
    hh1[p] = false;
    if (ht0 + p * NTH < HS) halo_entry(ht0 + p * NTH, hoff[p], hh1[p]);
  }
  // records: x faces (TX+1 per row), (3-d) y faces, march faces (the cell's upper one); face on
  // plane 0 and faces per plane
  const int NXF = (TX + 1) * TY, NYF = D == 3 ? TX * (TY + 1) : 0;
  auto rec_entry = [&](int t, uint32_t& off, uint32_t& str) {
    if (t < NXF) {
      const int row = D == 3 ? t / (TX + 1) : 0, c = t - row * (TX + 1);
      str = D == 1 ? 0u : (D == 2 ? (uint32_t)(nx + 1) : (uint32_t)(nx + 1) * ny);
      off = (uint32_t)A.rec_off[0] + (D == 3 ? (uint32_t)min(y0 + row, ny - 1) * (nx + 1) : 0u) + (uint32_t)min(x0 + c, nx);
    } else if (t < NXF + NYF) {
      const int q = t - NXF, row = q / TX, c = q - row * TX;
      str = (uint32_t)(ny + 1) * nx;
      off = (uint32_t)A.rec_off[1] + (uint32_t)min(y0 + row, ny) * nx + (uint32_t)min(x0 + c, nx - 1);
    } else {
      const int q = t - NXF - NYF, row = D == 3 ? q / TX : 0, c = q - row * TX;
      str = pcells;
      off = (uint32_t)A.rec_off[D >= 2 ? MD : 0] + (D == 3 ? (uint32_t)min(y0 + row, ny - 1) * nx : 0u) + (uint32_t)min(x0 + c, nx - 1) + pcells;
    }
  };
  uint32_t roff[RP], rstr[RP];
#pragma unroll
  for (int p = 0; p < RP; ++p) {
    roff[p] = rstr[p] = 0;
    if (tid + p * NTH < NREC) rec_entry(tid + p * NTH, roff[p], rstr[p]);
  }
  if (W == 2 && !VEC && (G & 1)) {  // the pad component of an odd group count's last pair stays zero
    for (int i = tid; i < L.rec; i += NTH) sm[i] = V(R(0));
    __syncthreads();
  }

  // ---- copies.  A plane's address is block-uniform (the state's base, the variable, the plane)
  // plus the thread's fixed offset.
  auto plane_at = [&](const R* S, int v, uint32_t row) -> const R* { return S + ((size_t)NG * ncell + (size_t)v * vstride + row); };
  // ring slot of plane P (counted from the chunk's first plane, as are the parities of halo and
  // record planes)
  auto ring_slot = [&](int P) -> int { return D == 1 ? 0 : ((P - kbeg + 1) & 3) * NRV * NT; };
  auto row_of = [&](int P) -> uint32_t {  // first element of plane P in a variable (P >= 0: upper ghosts mapped)
    bool f = false;
    return (uint32_t)(P < nmarch && P >= 0 ? P : map_m(P, f)) * pstride;
  };
  auto issue_own = [&](int P, int slot) {
    const uint32_t row = row_of(P);
    const int s = slot + tid;
#pragma unroll
    for (int v = 0; v < NRV; ++v)
      cp_async_lane(&ring[FXI(s + v * NT, n_ring)], FXP(plane_at(A.in, v, row), toff, vstride - row), vec, h1);
  };
  auto issue_halo = [&](int P, int par) {
    const uint32_t row = row_of(P);
    auto one = [&](int t, uint32_t off, bool two) {
      const int s = par * HPAR + t;
#pragma unroll
      for (int v = 0; v < NRV; ++v)
        cp_async_lane(&halo[FXI(s + v * HV, n_halo)], FXP(plane_at(A.in, v, row), off, vstride - row), vec, two);
    };
#pragma unroll
    for (int p = 0; p < HP; ++p)
      if (ht0 + p * NTH < HS) one(ht0 + p * NTH, hoff[p], hh1[p]);
    if (D == 3 && HS > HP * NTH) {  // (fit_tile: never below 3-d)
      for (int t = ht0 + HP * NTH; t < HS; t += NTH) {
        uint32_t off;
        bool two;
        halo_entry(t, off, two);
        one(t, off, two);
      }
    }
  };
  auto issue_rec = [&](int P, int par) {
    auto one = [&](int t, uint32_t f) {
      R* const d = rec + FXI((par * NREC + t) * 4, n_rec);
      const R* const s = A.frec + (size_t)4 * FXI(f, A.n_recs);
      cp_async16(d, s);
      if (sizeof(R) == 8) cp_async16(d + 2, s + 2);
    };
#pragma unroll
    for (int p = 0; p < RP; ++p)
      if (tid + p * NTH < NREC) one(tid + p * NTH, roff[p] + (uint32_t)P * rstr[p]);
    if (D == 3 && NREC > RP * NTH) {
      for (int t = tid + RP * NTH; t < NREC; t += NTH) {
        uint32_t off, str;
        rec_entry(t, off, str);
        one(t, off + (uint32_t)P * str);
      }
    }
  };
  auto issue_base = [&](int P) {
    if (A.base == nullptr) return;
    const uint32_t row = (uint32_t)P * pstride;
#pragma unroll
    for (int v = 0; v < NRV; ++v)
      cp_async_lane(&sbase[FXI(v * NT + tid, n_base)], FXP(plane_at(A.base, v, row), toff, vstride - row), vec, h1);
  };
  // scale factor of component q of the cell with x index ix on plane k
  auto hfac = [&](int q, const TT& rx, const TT& rm) -> R {
    if (!SPH) return R(1);
    const int e = q == 0 ? T_HA : T_HB;
    return rx(e, 0) * rm(e, 0);
  };
  // after the wait, each thread finishes what it copied: the mirrored components of ghost cells
  // change sign, and on the spherical grid covariant flux components become physical.  Planes
  // inside the grid of blocks without mirrored in-plane ghosts need neither.
  const bool fin_xy = SPH || g.bc_lo[0] >= 2 || g.bc_hi[0] >= 2 || (D == 3 && (g.bc_lo[1] >= 2 || g.bc_hi[1] >= 2));
  auto finish_one = [&](V* p, int vs, bool fx, bool fy, bool fm, const TT& rx, const TT& rm) {
#pragma unroll
    for (int q = 0; q < D; ++q) {
      const bool fl = q == MD && D > 1 ? fm : (q == 0 ? fx : fy);
      V x = p[(1 + q) * vs];
      if (SPH) x = x * frcp(hfac(q, rx, rm));
      if (fl) x = -x;
      p[(1 + q) * vs] = x;
    }
  };
  auto finish_own = [&](int P, int slot) {
    bool fm = false;
    map_m(P, fm);
    if (SPH || fx_own || fy_own || fm)
      finish_one(&ring[FXI(slot + tid, n_ring)], NT, fx_own, fy_own, fm, tx, row_of_dir(MD, P));
  };
  auto finish_halo = [&](int P, int par) {
    bool fm = false;
    map_m(P, fm);
    const TT rm = row_of_dir(MD, P);
    for (int t = ht0; t < HS; t += NTH) {
      int sx, sy;
      bool f0 = false, f1 = false;
      halo_pos(div_gl(t), sx, sy);
      inplane(sx, sy, f0, f1);
      if (SPH || f0 || f1 || fm) finish_one(&halo[FXI(par * HPAR + t, n_halo)], HV, f0, f1, fm, row_of_dir(0, x0 + sx), rm);
    }
  };

  // ---- reads.  The in-plane neighbours of the own cell: in the ring, or for an edge cell in the
  // halo (other base and variable stride, both fixed along the march up to the plane's slot).
  auto own_ld = [&](int slot, V* Q) {
    const int s = slot + tid;
#pragma unroll
    for (int v = 0; v < NRV; ++v) Q[v] = ring[FXI(s + v * NT, n_ring)];
  };
  // o: a neighbour's offset in the plane of the ring (slot) or of the halo (par)
  auto nb_ld = [&](int slot, int par, bool in_halo, int o, V* Q) {
    const V* const p = in_halo ? halo + FXI(par * HPAR + o, n_halo) : ring + FXI(slot + o, n_ring);
    const int st = D == 3 && in_halo ? HV : NT;  // (below 3-d the same)
#pragma unroll
    for (int v = 0; v < NRV; ++v) Q[v] = p[v * st];
  };
  const bool xm_h = lx == 0, xp_h = lx == TX - 1, ym_h = D == 3 && ly == 0, yp_h = D == 3 && ly == TY - 1;
  const int otid = act ? tid : lane;
  const int xm_o = xm_h ? (4 * ly + 1) * GL + lane : otid - GL, xp_o = xp_h ? (4 * ly + 2) * GL + lane : otid + GL;
  const int ym_o = ym_h ? (4 * TY + TX + lx) * GL + lane : otid - TX * GL;
  const int yp_o = yp_h ? (4 * TY + 2 * TX + lx) * GL + lane : otid + TX * GL;
  // face states of one cell along a direction: a at its lower face, b at its upper face
  auto recon = [&](const TT& t, const V* Qm, const V* Q0, const V* Qp, V* a, V* b) {
    if constexpr (RO == 2) {
#pragma unroll
      for (int v = 0; v < NRV; ++v) {
        R a0, b0, a1 = R(0), b1 = R(0);
        recon_parabolic(t, 0, vget(Qm[v], 0), vget(Q0[v], 0), vget(Qp[v], 0), a0, b0);
        if (W == 2) recon_parabolic(t, 0, vget(Qm[v], 1), vget(Q0[v], 1), vget(Qp[v], 1), a1, b1);
        a[v] = vpair(a0, a1, V());
        b[v] = vpair(b0, b1, V());
      }
    } else if constexpr (SPH) {
      const MCCoef<R> c = mc_coef<R>(t, 0);
#pragma unroll
      for (int v = 0; v < NRV; ++v) {
        const V s = mc_min((Q0[v] - Qm[v]) * c.il, (Qp[v] - Q0[v]) * c.ir, (Qp[v] - Qm[v]) * c.ic, R(2));
        a[v] = vfma(s, V(c.dl), Q0[v]);
        b[v] = vfma(s, V(c.dr), Q0[v]);
      }
    } else {
#pragma unroll
      for (int v = 0; v < NRV; ++v) {
        const V dl = Q0[v] - Qm[v], dr = Qp[v] - Q0[v];
        const V s = mc_min(dl, dr, (dl + dr) * KL.q25, R(1));  // half the limited slope times dx
        a[v] = Q0[v] - s;
        b[v] = Q0[v] + s;
      }
    }
  };
  // twice the flux through a face of direction n from its two states; r: the face record
  // (2 max(v*, 0), 2 min(v*, 0), and the opacity sums so that tau_g = eps_g^d r2 + r3)
  auto face_flux = [&](int n, const V* QL, const V* QR, const R* r, V ef, V* out) {
    V PL[D], PR[D];
    m1_c2row<D>(KL, QL[0], QL + 1, n, PL);
    m1_c2row<D>(KL, QR[0], QR + 1, n, PR);
    const V tau = vfma(ef, V(r[2]), V(r[3]));
    const V ce = rcp_ge1(tau) * KL.mc;  // -c min(1, 1/tau)
    out[0] = vfma(V(r[1]), QR[0], vfma(V(r[0]), QL[0], vfma(ce, QR[0] - QL[0], QL[1 + n] + QR[1 + n])));
    const V kL = V(KR.c + r[0]), kR = V(r[1] - KR.c);
#pragma unroll
    for (int q = 0; q < D; ++q) out[1 + q] = vfma(kR, QR[1 + q], vfma(kL, QL[1 + q], PL[q] + PR[q]));
  };
  auto rec_ld = [&](int par, int i, R* r) {
    const R* const p = rec + FXI((par * NREC + i) * 4, n_rec);
    if constexpr (sizeof(R) == 4) {
      const float4 x = *reinterpret_cast<const float4*>(p);
      r[0] = x.x; r[1] = x.y; r[2] = x.z; r[3] = x.w;
    } else {
#pragma unroll
      for (int c = 0; c < 4; ++c) r[c] = p[c];
    }
  };
  auto ef_of = [&](int ln) -> V {
    const int ga = ln * W, gb = ga + 1 < G ? ga + 1 : ga;
    return vpair(A.gc->efac_of(ga, R(0)), A.gc->efac_of(W == 2 ? gb : ga, R(0)), V());
  };
  const V efv = ef_of(lane);
  // own lower faces in xb (TX+1 faces per row) and yb; the threads past the tile use the space
  // after the arrays' faces
  const int xo = act ? tid + ly * GL : NT + CP::XP + (tid & 31), yo = act ? tid : xo;

  // ---------------------------------------------------------------- prologue
  V bm0[NRV], rfm_old[NRV];  // upper march-face state of plane k, flux through its lower march face
#pragma unroll
  for (int v = 0; v < NRV; ++v) bm0[v] = rfm_old[v] = V(R(0));
  if constexpr (D == 1) {
    issue_own(0, 0);
    issue_halo(0, 0);
    issue_rec(0, 0);
    cp_async_commit();
    cp_async_wait_all();
    finish_own(0, 0);
    finish_halo(0, 0);
    __syncthreads();
  } else {
    for (int P = kbeg - 1; P <= kbeg + 2; ++P) issue_own(P, ring_slot(P));
    issue_halo(kbeg, 0);
    issue_rec(kbeg, 0);
    cp_async_commit();
    V Qa[NRV];  // own column of plane kbeg-2, straight from global memory
    {
      bool fm = false;
      const TT rm = row_of_dir(MD, kbeg - 2);
      const uint32_t o = NG * ncell + toff + (uint32_t)map_m(kbeg - 2, fm) * pstride;
#pragma unroll
      for (int v = 0; v < NRV; ++v) {
        const R e0 = A.in[FXI(o + v * vstride, A.n_state)], e1 = h1 ? A.in[FXI(o + v * vstride + 1, A.n_state)] : R(0);
        Qa[v] = vpair(e0, e1, V());
      }
#pragma unroll
      for (int q = 0; q < D; ++q) {
        const bool fl = q == MD ? fm : (q == 0 ? fx_own : fy_own);
        if (SPH) Qa[1 + q] = Qa[1 + q] * frcp(hfac(q, tx, rm));
        if (fl) Qa[1 + q] = -Qa[1 + q];
      }
    }
    R r[4];
    {
      const uint32_t f = (uint32_t)A.rec_off[MD] + (D == 3 ? (uint32_t)min(gy, ny - 1) * nx : 0u) + (uint32_t)min(gx, nx - 1) + (uint32_t)kbeg * pcells;
      const R* const s = A.frec + (size_t)4 * FXI(f, A.n_recs);
#pragma unroll
      for (int c = 0; c < 4; ++c) r[c] = s[c];
    }
    cp_async_wait_all();
    for (int P = kbeg - 1; P <= kbeg + 2; ++P) finish_own(P, ring_slot(P));
    finish_halo(kbeg, 0);
    __syncthreads();
    // march reconstruction of planes kbeg-1 (upper face) and kbeg, and the flux at kbeg-1/2
    V Qb[NRV], Qc[NRV], Qd[NRV], ta[NRV], tb[NRV], am[NRV];
    own_ld(ring_slot(kbeg - 1), Qb);
    own_ld(ring_slot(kbeg), Qc);
    own_ld(ring_slot(kbeg + 1), Qd);
    recon(row_of_dir(MD, kbeg - 1), Qa, Qb, Qc, ta, tb);
    recon(row_of_dir(MD, kbeg), Qb, Qc, Qd, am, bm0);
    face_flux(MD, tb, am, r, efv, rfm_old);
  }

  // the halo reconstructions as tasks, one per (row or column end, lane): the upper-face state of
  // cells -1 (left state of the tile's first face) and the lower-face state of cells TX, TY (right
  // state of its last face).  A task's ring entry of the edge cell, halo entry of the near halo
  // cell and step to the far one, and where the state goes:
  const int n1 = TY * GL, n2 = D == 3 ? TX * GL : 0, ntask = 2 * (n1 + n2);
  struct Task { int in, h, hs, dst; bool up, x; };
  auto task_of = [&](int t) -> Task {
    Task b;
    b.x = D < 3 || t < 2 * n1;
    const int u = b.x ? t : t - 2 * n1, nn = b.x ? n1 : n2;
    b.up = u >= nn;                      // the halo cell above the tile
    const int e = b.up ? u - nn : u;     // row (or column) * GL + lane
    const int c = div_gl(e), ln = e - c * GL;
    if (b.x) {
      b.in = (c * TX + (b.up ? TX - 1 : 0)) * GL + ln;
      b.h = (4 * c + (b.up ? 2 : 1)) * GL + ln;
      b.hs = b.up ? GL : -GL;
      b.dst = b.up ? e : c * (TX + 1) * GL + ln;
    } else {
      b.in = (b.up ? (TY - 1) * TX * GL : 0) + e;
      b.h = (4 * TY + (b.up ? 2 : 1) * TX) * GL + e;
      b.hs = b.up ? TX * GL : -TX * GL;
      b.dst = e;
    }
    return b;
  };
  auto run_task = [&](int slot, int par, int px, const Task& b_) {
    V Qi[NRV], Q0[NRV], Qo[NRV], a[NRV], b[NRV];
    nb_ld(slot, par, false, b_.in, Qi);
    nb_ld(slot, par, true, b_.h, Q0);
    nb_ld(slot, par, true, b_.h + b_.hs, Qo);
    if constexpr (TABLES) {
      const TT tt = b_.x ? row_of_dir(0, b_.up ? x0 + TX : x0 - 1) : ty;
      if (b_.up) recon(tt, Qi, Q0, Qo, a, b);
      else recon(tt, Qo, Q0, Qi, b, a);
    } else {
      // (uniform spacing: the other way round gives the mirrored states)
      recon(tx, Qi, Q0, Qo, a, b);
    }
    V* const d = b_.up ? (b_.x ? xr + FXI(b_.dst, n_xr) : yr + FXI(b_.dst, n_yr))
                       : (b_.x ? xb : yb) + FXI(px + b_.dst, n_xb);
    const int st = b_.up ? (b_.x ? n1 : n2) : XC;
#pragma unroll
    for (int v = 0; v < NRV; ++v) d[v * st] = a[v];
  };
  Task my{};
  if (tid < ntask) my = task_of(tid);
  // the fluxes through the tile's upper faces likewise, from the last threads down
  const int ct = NTH - 1 - tid;
  const bool task_c = ct < n1 + n2;
  const bool more_out = A.pre_out != nullptr || A.phi_out != nullptr;
  const bool stage2 = A.base != nullptr;

  // ---------------------------------------------------------------- march
  // (unrolled by four planes, with every slot a constant, the kernel lost 8 to 25 % to instruction
  // fetch)
  constexpr int SL = D == 1 ? 0 : NRV * NT;
  int par = 0, s0 = SL, s1 = 2 * SL, s2 = 3 * SL, s3 = 0;  // slots of planes k, k+1, k+2 and the one to fill
  for (int k = kbeg; k < kend; ++k) {
    if (D == 3) {  // (rotated below: 256^3 x 12 slower by 0.7 %, 2-d faster by 1 to 2 %)
      const int u = k - kbeg;
      par = u & 1;
      s0 = ((u + 1) & 3) * SL; s1 = ((u + 2) & 3) * SL; s2 = ((u + 3) & 3) * SL; s3 = (u & 3) * SL;
    }
    const bool more = D >= 2 && k + 1 < kend;
    if (more) {
      issue_own(k + 3, s3);
      issue_halo(k + 1, par ^ 1);
      issue_rec(k + 1, par ^ 1);
    }
    issue_base(k);
    cp_async_commit();
    const int px = PB == 2 ? par * NRV * XC : 0;  // this plane's half of xb and yb
    // ---- B
    V ax[NRV], ay[NRV], am1[NRV], bm1[NRV];
    {
      V Q0[NRV], Qm[NRV], Qp[NRV], b[NRV];
      own_ld(s0, Q0);
      nb_ld(s0, par, xm_h, xm_o, Qm);
      nb_ld(s0, par, xp_h, xp_o, Qp);
      recon(tx, Qm, Q0, Qp, ax, b);
#pragma unroll
      for (int v = 0; v < NRV; ++v) xb[FXI(px + v * XC + xo + GL, n_xb)] = b[v];
      if constexpr (D == 3) {
        nb_ld(s0, par, ym_h, ym_o, Qm);
        nb_ld(s0, par, yp_h, yp_o, Qp);
        recon(ty, Qm, Q0, Qp, ay, b);
#pragma unroll
        for (int v = 0; v < NRV; ++v) yb[FXI(px + v * XC + yo + TX * GL, n_xb)] = b[v];
      }
      if constexpr (D >= 2) {
        own_ld(s1, Qm);
        own_ld(s2, Qp);
        recon(row_of_dir(MD, k + 1), Q0, Qm, Qp, am1, bm1);
      }
    }
    if (tid < ntask) run_task(s0, par, px, my);
    if (D == 3 && ntask > NTH)
      for (int t = tid + NTH; t < ntask; t += NTH) run_task(s0, par, px, task_of(t));
    __syncthreads();
    // ---- C
    V rfm_new[NRV];
#pragma unroll
    for (int v = 0; v < NRV; ++v) rfm_new[v] = V(R(0));
    {
      V QL[NRV], out[NRV];
      R r[4];
#pragma unroll
      for (int v = 0; v < NRV; ++v) QL[v] = xb[FXI(px + v * XC + xo, n_xb)];
      rec_ld(par, ly * (TX + 1) + lx, r);
      face_flux(0, QL, ax, r, efv, out);
#pragma unroll
      for (int v = 0; v < NRV; ++v) xb[FXI(px + v * XC + xo, n_xb)] = out[v];
      if constexpr (D == 3) {
#pragma unroll
        for (int v = 0; v < NRV; ++v) QL[v] = yb[FXI(px + v * XC + yo, n_xb)];
        rec_ld(par, NXF + ly * TX + lx, r);
        face_flux(1, QL, ay, r, efv, out);
#pragma unroll
        for (int v = 0; v < NRV; ++v) yb[FXI(px + v * XC + yo, n_xb)] = out[v];
      }
      if constexpr (D >= 2) {
        rec_ld(par, NXF + NYF + tc, r);
        face_flux(MD, bm0, am1, r, efv, rfm_new);
      }
    }
    // the tile's upper faces, one task per row (column) and lane
    if (task_c) {
      const bool isx = D < 3 || ct < n1;
      const int e = isx ? ct : ct - n1;
      const int c = div_gl(e), ln = e - c * GL;
      V* const p = isx ? xb + FXI(px + (c * (TX + 1) + TX) * GL + ln, n_xb) : yb + FXI(px + TC * GL + e, n_xb);
      const V* const pr = isx ? xr + FXI(e, n_xr) : yr + FXI(e, n_yr);
      const int sr = isx ? n1 : n2;
      V QL[NRV], QR[NRV], out[NRV];
      R r[4];
#pragma unroll
      for (int v = 0; v < NRV; ++v) { QL[v] = p[v * XC]; QR[v] = pr[v * sr]; }
      rec_ld(par, isx ? c * (TX + 1) + TX : NXF + TY * TX + c, r);
      if (D < 3 || isx) face_flux(0, QL, QR, r, ef_of(ln), out);
      else face_flux(D == 3 ? 1 : 0, QL, QR, r, ef_of(ln), out);
#pragma unroll
      for (int v = 0; v < NRV; ++v) p[v * XC] = out[v];
    }
    cp_async_wait_all();
    if (more && (fin_xy || k + 3 >= nmarch)) {
      finish_own(k + 3, s3);
      finish_halo(k + 1, par ^ 1);
    }
    __syncthreads();
    // ---- D
    if (cell_in) {
      V Q0[NRV], U[NRV];
      own_ld(s0, Q0);
      const uint32_t cidx = cxy + (uint32_t)k * pcells;
      V xm[NRV], xp[NRV], ym[NRV], yp[NRV];
#pragma unroll
      for (int v = 0; v < NRV; ++v) {
        xm[v] = xb[FXI(px + v * XC + xo, n_xb)];
        xp[v] = xb[FXI(px + v * XC + xo + GL, n_xb)];
        if (D == 3) {
          ym[v] = yb[FXI(px + v * XC + yo, n_xb)];
          yp[v] = yb[FXI(px + v * XC + yo + TX * GL, n_xb)];
        }
      }
      if constexpr (SPH) {
        // area/volume factors of the two face pairs per flux class (half: twice the flux is
        // carried), and the geometric sources <Gamma^l_jk> T^k_l of the stage's input state (Eq. 9;
        // Appendix D)
        const TT tm = row_of_dir(MD, k);
        const R hq[2] = {hfac(0, tx, tm), hfac(1, tx, tm)};
        const R g111 = tx(T_GA, 0), g221 = tx(T_GB, 0), g122 = tx(T_GC, 0);
        const R g222 = tm(T_GA, 0), g332 = tm(T_GB, 0);
        const R rho = A.in[FXI(cidx, A.n_state)], irho = frcp(rho);
        const R v1 = A.in[FXI(ncell + cidx, A.n_state)] * irho * frcp(hq[0]), v2 = A.in[FXI(2 * ncell + cidx, A.n_state)] * irho * frcp(hq[1]);
        const R r12 = hq[0] * frcp(hq[1]), r21 = hq[1] * frcp(hq[0]);
        V P0[D], P1[D];
        m1_c2row<D>(KL, Q0[0], Q0 + 1, 0, P0);
        m1_c2row<D>(KL, Q0[0], Q0 + 1, 1, P1);
        // c^2 P33 is the closure's diagonal part: the trace c^2 E less the other two entries would
        // cancel for a beam, so it is formed as P11 less its beam part
        const V P33 = m1_c2perp<D>(KL, Q0[0], Q0 + 1);
        const V R11 = vfma(V(v1), Q0[1], P0[0]), R22 = vfma(V(v2), Q0[D >= 2 ? 2 : 0], P1[D - 1]);
        const V R21 = vfma(V(v2), Q0[1], P0[D - 1]) * r12, R12 = vfma(V(v1), Q0[D >= 2 ? 2 : 0], P0[D - 1]) * r21;
        V src[3] = {V(R(0)), R11 * g111 + (R22 + P33) * g221, R21 * g122 + R12 * g221 + R22 * g222 + P33 * g332};
        const int eL[3] = {T_FL, T_FL1, T_FL2}, eR[3] = {T_FR, T_FR1, T_FR2}, eX[3] = {T_XS, T_X1, T_X2};
#pragma unroll
        for (int v = 0; v < NRV; ++v) {
          const V Fp[2] = {xp[v], rfm_new[v]}, Fm[2] = {xm[v], rfm_old[v]};
          const R xs = R(0.5) * tm(eX[v], 0), ms = R(0.5) * tx(eX[v], 0);
          const R Ap[2] = {tx(eR[v], 0) * xs, tm(eR[v], 0) * ms};
          const R Am[2] = {tx(eL[v], 0) * xs, tm(eL[v], 0) * ms};
          const V cov = v >= 1 ? Q0[v] * hq[v - 1] : Q0[v];  // covariant F
          U[v] = fv_update(Fp, Ap, Fm, Am, cov, src[v], KR.dt, stage2, stage2 ? sbase[FXI(v * NT + tid, n_base)] : V(R(0)),
                           KR.alpha, KR.beta);
        }
      } else {
#pragma unroll
        for (int v = 0; v < NRV; ++v) {
          V u = Q0[v] - net_update<D>(xp[v], xm[v], yp[v], ym[v], rfm_new[v], rfm_old[v], KL.hdt, KL.mhdt);
          if (stage2) u = vfma(KL.alpha, sbase[FXI(v * NT + tid, n_base)], u * KL.beta);
          U[v] = u;
        }
      }
      // budgets (reading R13): the outward fluxes through this cell's faces on non-periodic
      // boundaries, times the face area (the area/volume factor times the cell volume) and the
      // stage's weight, added to one of BUDGET_SLOTS rows of accumulators (summed when read)
      if (BUD && A.budget != nullptr) {
        const bool xl = gx == 0 && g.bc_lo[0] != 1, xh = gx == nx - 1 && g.bc_hi[0] != 1;
        const bool yl = D == 3 && gy == 0 && g.bc_lo[1] != 1, yh = D == 3 && gy == ny - 1 && g.bc_hi[1] != 1;
        const bool ml = D >= 2 && k == 0 && g.bc_lo[MD] != 1, mh = D >= 2 && k == nmarch - 1 && g.bc_hi[MD] != 1;
        if (xl || xh || yl || yh || ml || mh) {
          const TT tm = row_of_dir(MD, k);
          double vol = (double)tx(T_VOL, 0);
          if (D == 3) vol *= (double)ty(T_VOL, 0);
          if (D >= 2) vol *= (double)tm(T_VOL, 0);
          const double bs = 0.5 * vol * A.bw_flux;  // (twice the flux is carried)
          double* const bud = A.budget + (size_t)(blockIdx.x % BUDGET_SLOTS) * NBUDGET;
          const int eL[3] = {T_FL, T_FL1, T_FL2}, eR[3] = {T_FR, T_FR1, T_FR2}, eX[3] = {T_XS, T_X1, T_X2};
#pragma unroll
          for (int v = 0; v < NRV; ++v) {
            const int c = SPH ? v : 0;
            const R sx = SPH ? tm(eX[c], 0) : R(1), sm_ = SPH ? tx(eX[c], 0) : R(1);
            double o = 0.0;
#pragma unroll
            for (int j = 0; j < W; ++j) {
              if (j == 1 && !h1) continue;
              if (xh) o += (double)(vget(xp[v], j) * (tx(eR[c], 0) * sx));
              if (xl) o -= (double)(vget(xm[v], j) * (tx(eL[c], 0) * sx));
              if (D == 3 && yh) o += (double)(vget(yp[v], j) * ty(T_FR, 0));
              if (D == 3 && yl) o -= (double)(vget(ym[v], j) * ty(T_FL, 0));
              if (D >= 2 && mh) o += (double)(vget(rfm_new[v], j) * (tm(eR[c], 0) * sm_));
              if (D >= 2 && ml) o -= (double)(vget(rfm_old[v], j) * (tm(eL[c], 0) * sm_));
            }
            if (o != 0.0) {
              if (v == 0) {
                atomicAdd(bud + 4, o * bs);
                atomicAdd(bud + 5, o * bs);
              } else {
                atomicAdd(bud + v, o * bs * (double)KR.ic2);
              }
            }
          }
        }
      }
      if (more_out) {
        // recording for the adjoint: the pre-interaction state
        if (A.pre_out != nullptr) {
          const uint32_t o = NG * ncell + cidx * G + g0;
#pragma unroll
          for (int v = 0; v < NRV; ++v) {
            A.pre_out[FXI(o + v * vstride, A.n_state)] = vget(U[v], 0);
            if (h1) A.pre_out[FXI(o + v * vstride + 1, A.n_state)] = vget(U[v], W - 1);
          }
        }
        // objective: energy flux through the upper x boundary face of the row, times its area
        if (A.phi_out != nullptr && gx == nx - 1) {
          const uint32_t row = D == 1 ? 0u : D == 2 ? (uint32_t)k : (uint32_t)k * ny + gy;
          const uint32_t n_phi = (uint32_t)(D >= 2 ? ny : 1) * (D >= 3 ? nz : 1) * G;
          (void)n_phi;
          A.phi_out[FXI(row * G + g0, n_phi)] = R(0.5) * vget(xp[0], 0) * A.phi_area;
          if (h1) A.phi_out[FXI(row * G + g0 + 1, n_phi)] = R(0.5) * vget(xp[0], W - 1) * A.phi_area;
        }
      }
      V chk = V(R(0));  // a NaN or inf anywhere in the outputs makes this sum non-finite
      const uint32_t row = (uint32_t)k * pstride;
#pragma unroll
      for (int v = 0; v < NRV; ++v) {
        st_global_lane(FXP(const_cast<R*>(plane_at(A.out, v, row)), toff, vstride - row), U[v], vec, h1);
        chk = vfma(U[v], V(R(0)), chk);
      }
      if (!isfinite(vget(chk, 0)) || (h1 && !isfinite(vget(chk, W - 1)))) atomicOr(A.status, ST_NONFINITE);
    }
    if (PB == 1) __syncthreads();  // the next plane's face states overwrite these fluxes
#pragma unroll
    for (int v = 0; v < NRV; ++v) {
      if (D >= 2) bm0[v] = bm1[v];
      rfm_old[v] = rfm_new[v];
    }
    if (D < 3) {
      const int s4 = s0;
      s0 = s1; s1 = s2; s2 = s3; s3 = s4;
      par ^= 1;
    }
  }
}

}  // namespace fx
