// pflb_kernels.cuh -- CUDA kernels of the PF-LB-FD time step (sm_103a).
//
// One fused kernel advances one time step of the low-Mach phase-field /
// lattice-Boltzmann / finite-difference model (arXiv 2310.17214, Sec. 3.3):
//   pull streaming of the pressure-based populations with the boundary rules,
//   moments with the implicit diffuse-interface drag (Sec. 3.2.1), FD
//   transport of T, Y_k and the solid temperature with the reaction source
//   (Sec. 3.2.2 eq. 8, Sec. 3.3 eqs. diffusion-heat-flux-3,
//   energy-transport-DI-version, 9), the divergence from the low-Mach
//   constraint, the source Xi (eq. body-force) and BGK collision (eqs.
//   eq-pop-f, eq-pop-g), and the FP64 reduction for P0 (Sec. 3.1) finished by
//   the last block to arrive.
//
// Layout: SoA in HBM, g[i*N + cell], Y[k*N + cell]; cell = x + nx*(y + ny*z).
// A block owns a tile of 32 columns of one or more z-planes (3-D:
// pflb_step3d.cuh).  It stages T, Y, phi, Ts of the tile plus a one-cell halo
// in shared memory and evaluates the per-cell properties (EOS density,
// viscosity, conductivity, diffusivity factor) once per staged cell; the FD
// stencils and grad(rho) then read their neighbours from shared memory.  The
// populations are pulled straight from HBM.  In FP32 a thread owns two
// neighbouring cells and works on them with packed arithmetic (pflb_vec.cuh).
// FP16-stored populations have their own update (pflb_half.cuh).
#pragma once

#include <cuda_fp16.h>
#include <stdint.h>

#include "pflb_vec.cuh"

namespace pflb {

constexpr int KMAX = 8;
constexpr int JMAX = 4;
constexpr int BLOCK = 256;  // threads per block (one cell each per plane)
// default bound of a device-side wait: 2^31 SM clock cycles, about a second
constexpr long long kDefaultWaitCycles = 1LL << 31;

enum { BC_PERIODIC = 0, BC_WALL = 1, BC_INLET = 2, BC_OUTLET = 3 };
enum { MODE_FP64 = 0, MODE_FP32 = 1, MODE_FP16 = 2 };

// ------------------------------------------------------------- lattices
// D2Q9 and D3Q19 velocity sets and weights (cs^2 = 1/3).  The direction
// order is the library's storage order (reported by pflb_lattice).
template <int DIM> struct Lattice;

template <> struct Lattice<2> {
  static constexpr int Q = 9;
  __host__ __device__ static constexpr int c(int i, int a) {
    constexpr int t[9][3] = {{0, 0, 0},  {1, 0, 0},  {0, 1, 0},   {-1, 0, 0}, {0, -1, 0},
                             {1, 1, 0},  {-1, 1, 0}, {-1, -1, 0}, {1, -1, 0}};
    return t[i][a];
  }
  __host__ __device__ static constexpr double w(int i) {
    return i == 0 ? 4.0 / 9.0 : (i < 5 ? 1.0 / 9.0 : 1.0 / 36.0);
  }
  __host__ __device__ static constexpr int opp(int i) {
    constexpr int t[9] = {0, 3, 4, 1, 2, 7, 8, 5, 6};
    return t[i];
  }
};

template <> struct Lattice<3> {
  static constexpr int Q = 19;
  __host__ __device__ static constexpr int c(int i, int a) {
    constexpr int t[19][3] = {{0, 0, 0},  {1, 0, 0},  {-1, 0, 0}, {0, 1, 0},   {0, -1, 0},
                              {0, 0, 1},  {0, 0, -1}, {1, 1, 0},  {-1, -1, 0}, {1, -1, 0},
                              {-1, 1, 0}, {1, 0, 1},  {-1, 0, -1}, {1, 0, -1}, {-1, 0, 1},
                              {0, 1, 1},  {0, -1, -1}, {0, 1, -1}, {0, -1, 1}};
    return t[i][a];
  }
  __host__ __device__ static constexpr double w(int i) {
    return i == 0 ? 1.0 / 3.0 : (i < 7 ? 1.0 / 18.0 : 1.0 / 36.0);
  }
  __host__ __device__ static constexpr int opp(int i) {
    constexpr int t[19] = {0, 2, 1, 4, 3, 6, 5, 8, 7, 10, 9, 12, 11, 14, 13, 16, 15, 18, 17};
    return t[i];
  }
};

// ------------------------------------------------------------ parameters
// FP64 chemistry data of the implicit integrator.
template <int K>
struct Chem64 {
  static constexpr int KK = K > 0 ? K : 1;
  double A[JMAX], b[JMAX], EaR[JMAX], dn[JMAX];
  int rev[JMAX];
  double order[JMAX][KK], rorder[JMAX][KK];
  double Ms[JMAX][KK];          // M_k s_kj
  double dS_R[JMAX], dH_R[JMAX];  // dS / R, dH / R
  double invM[KK], cp[KK];
  double ln_pref_R, rho_ref, dt;  // ln_pref_R = ln(p_ref / R)
  double H[JMAX], cM[JMAX];  // sum_k hf_k Ms_jk, sum_k cp_k Ms_jk
  double pref_R;             // p_ref / R
  int used;                  // bit k: species k enters a rate
  __device__ __forceinline__ bool active(int j) const { return A[j] != 0.0; }
};

// FP32 copy of the chemistry for the Newton fallback of the surrogate in FP32
// domains (rate constants as logarithms: ln k = ln A + b ln T - EaR / T).
template <int K>
struct Chem32 {
  static constexpr int KK = K > 0 ? K : 1;
  float lnA[JMAX], b[JMAX], EaR[JMAX], dn[JMAX], dS_R[JMAX], dH_R[JMAX];
  int on[JMAX], rev[JMAX];
  float order[JMAX][KK], rorder[JMAX][KK];
  float Ms[JMAX][KK];  // M_k s_kj
  float invM[KK], cp[KK];
  float ln_pref_R, dt;
  float H[JMAX], cM[JMAX];
  __device__ __forceinline__ bool active(int j) const { return on[j] != 0; }
};

// Everything in lattice units, converted once on the host (pflb_launch.cuh).
template <class Real, int K>
struct Params {
  static constexpr int KK = K > 0 ? K : 1;
  int nx, ny, nz, N;
  int bc[6];
  Real wall_u[6][3];
  Real wall_T[6];
  double eos_c;            // rho* = P0 Mw eos_c / T, eos_c = 1 / (R rho_ref)
  double inv_rho_ref;      // dP0 / rho_ref (J/kg) in the T equation
  Real eos_cr;             // eos_c in the compute type
  Real mu_lat;             // mu_ref dt / (rho_ref dx^2)
  int sutherland;
  Real inv_suth_T, suth_S, suth_TS;  // suth_TS = suth_T + suth_S
  Real inv_Pr;
  Real Au_eta2, AT_eta2;   // A_u / eta^2, A_T / eta^2
  Real Fb[3];
  int inlet_parabolic;
  Real u_in, T_in;
  Real Y_in[KK];
  Real M0, cp0;
  Real invM[KK], cp[KK], hf[KK];
  Real Dlat[KK], Dlat_h[KK];  // diffusivity in lattice units, half of it
  Real cpD[KK];            // cp_k Dlat_k (enthalpy-flux cross term)
  int D_Tdep;
  Real inv_DTref, D_exp;
  int Ts_field;
  Real Ts_uniform, Cs;     // solid rho cp / rho_ref
  Real Lams, Lams_h;       // lambda_s dt / (rho_ref dx^2), half of it
  Real phi_min;
  int chem, J;
  Real A_lat[JMAX];        // A dt / rho_ref
  Real b[JMAX], EaR[JMAX];
  Real order[JMAX][KK], stoichM[JMAX][KK];  // stoichM = s_kj M_k
  Real rho_ref_M[KK];      // rho_ref / M_k (concentration from rho* Y_k)
  Real g_scale, g_inv_scale;  // FP16 storage scale (power of two)
  // reversible reactions in the compute type (explicit rates)
  int rev[JMAX];
  Real rorder[JMAX][KK];
  Real dS_R[JMAX], dH_R[JMAX], dn[JMAX], p_ref_R;  // dS/R, dH/R, sum_k s_kj, p_ref/R
  // FP64 copy of the chemistry for the implicit Newton integrator (FP64 in
  // every precision mode: the stiff chemistry keeps double precision)
  Chem64<K> c64;
  Chem32<K> c32;
  // mixture-averaged transport (Sec. 4.4): species Sutherland laws (lattice
  // units), modified Eucken factors, Wilke's constant factors
  int mix;
  Real mu_lat_k[KK], inv_suth_Tk[KK], suth_Sk[KK], suth_TSk[KK], eucken_k[KK];
  Real wA[KK][KK];         // (M_j / M_k)^(1/4)
  Real wB[KK][KK];         // 1 / (sqrt(8) sqrt(1 + M_k / M_j))
  // inlet mass-flow feedback (Sec. 4.4.1): on, species index, and
  // feed_c = 1 / (rho_in / P0 Y_in[k] A) so that u_in = fuel feed_c / P0
  int feed, feed_k;
  double feed_c;
  // characteristic outlet (Sec. 4.1): on, and K = sigma cs / nx
  int nscbc;
  double nscbc_K;
  // moving solid (Sec. 2, interface velocity): rigid translation velocity
  int moving;
  Real u_s[3];
};

// Scalar state on the device.  The per-step quantities the cells need (P0,
// dP0/P0, dP0/rho_ref) are precomputed by the block that finishes the
// reduction, in FP64 and in FP32.
struct DevScalars {
  double P0, P0_prev, mass, I, flux_in, flux_out, mass_now;
  double flux_in_sum, flux_out_sum;  // inlet / outlet mass flux summed over the steps
  long long step;
  int status;
  int pad;
  double dlnP0, dP0r;
  float P0_f, dlnP0_f, dP0r_f, pad_f;
  // inlet peak speed of the next step and the consumption it was set from
  // (inlet feedback; otherwise u_in stays the description's value)
  double u_in, fuel;
  float u_in_f, pad_f2;
  // boundary pressure of the next step at the characteristic outlet
  double pb;
  float pb_f, pad_f3;
};

// FP16 storage keeps, per cell, the FP32 moments (P, j) = (sum g*, sum c g*)
// of the post-collision populations and, per direction, the FP16 residual
// h_i = (g*_i - w_i (P + 3 c_i . j)) S / w_i (the first-order equilibrium of
// the cell's own moments removed, so that the narrowed quantity is second
// order in u).  A reader adds w_i (P + 3 c_i . j) of the source cell back.
template <class Store> struct IsHalf { static constexpr bool value = false; };
template <> struct IsHalf<__half> { static constexpr bool value = true; };

template <class Real, class Store>
struct State {
  const Store* __restrict__ g_in;
  Store* __restrict__ g_out;
  const Real* __restrict__ M_in;   // FP16 storage: moments [DIM+1][N] of g_in (else null)
  Real* __restrict__ M_out;        // FP16 storage: moments of g_out
  const Real* __restrict__ T_in;
  Real* __restrict__ T_out;
  const Real* __restrict__ Y_in;
  Real* __restrict__ Y_out;
  const Real* __restrict__ Ts_in;
  Real* __restrict__ Ts_out;
  const Real* __restrict__ phi;
  const Real* __restrict__ src;  // precomputed chemistry increments [K+1][N] (implicit/surrogate)
  DevScalars* scal;
  double* partials;        // this step's block partials: [blocks][4]
  unsigned* counter;
  int even;                // pairs of cells are aligned words: nx even, arrays aligned
  Real* ob;                // characteristic outlet: P_h, u_x of columns nx-1 and nx-2 and rho
                           // of column nx-1 of this step, [5][ny nz] (else null)
};

// A domain of a batch's work list (pflb_batch.cuh).
template <int K, class Real, class Store>
struct BatchDom {
  Params<Real, K> P;
  State<Real, Store> S[2];  // S[q]: input state in ping-pong buffer q
  int p0_closed;
  int cur0;                 // buffer holding the input at even batch steps
};

// ----------------------------------------------------- storage codecs
template <class Store, class Real> struct Codec;
// raw: the stored value as a number (read-only path).
template <> struct Codec<double, double> {
  __device__ static double raw(const double* p) { return __ldg(p); }
  __device__ static void store(double* p, double v, double) { *p = v; }
};
template <> struct Codec<float, float> {
  __device__ static float raw(const float* p) { return __ldg(p); }
  __device__ static void store(float* p, float v, float) { *p = v; }
};
// FP16: residual r_i = g_i - w_i (P + 3 c_i . j), stored as h = r / w * scale
// (weights folded so every direction has the same range).  dec(raw, w/S, fo): the
// population from it and the first-order part fo of the source cell, one FMA,
// the same on every path that decodes, so that all paths round alike.
template <> struct Codec<__half, float> {
  __device__ static float raw(const __half* p) { return __half2float(__ldg(p)); }
  __device__ static float dec(float r, float w_over_scale, float fo) {
    return __fmaf_rn(r, w_over_scale, fo);
  }
  __device__ static void store(__half* p, float v, float scale_over_w) {
    *p = __float2half_rn(v * scale_over_w);
  }
};

template <class Real> __device__ __forceinline__ Real scal_P0(const DevScalars* s);
template <> __device__ __forceinline__ double scal_P0<double>(const DevScalars* s) { return s->P0; }
template <> __device__ __forceinline__ float scal_P0<float>(const DevScalars* s) { return s->P0_f; }
template <class Real> __device__ __forceinline__ Real scal_u_in(const DevScalars* s);
template <> __device__ __forceinline__ double scal_u_in<double>(const DevScalars* s) { return s->u_in; }
template <> __device__ __forceinline__ float scal_u_in<float>(const DevScalars* s) { return s->u_in_f; }
template <class Real> __device__ __forceinline__ Real scal_pb(const DevScalars* s);
template <> __device__ __forceinline__ double scal_pb<double>(const DevScalars* s) { return s->pb; }
template <> __device__ __forceinline__ float scal_pb<float>(const DevScalars* s) { return s->pb_f; }
template <class Real> __device__ __forceinline__ Real scal_dlnP0(const DevScalars* s);
template <> __device__ __forceinline__ double scal_dlnP0<double>(const DevScalars* s) { return s->dlnP0; }
template <> __device__ __forceinline__ float scal_dlnP0<float>(const DevScalars* s) { return s->dlnP0_f; }
template <class Real> __device__ __forceinline__ Real scal_dP0r(const DevScalars* s);
template <> __device__ __forceinline__ double scal_dP0r<double>(const DevScalars* s) { return s->dP0r; }
template <> __device__ __forceinline__ float scal_dP0r<float>(const DevScalars* s) { return s->dP0r_f; }

// ------------------------------------------------------------ physics
// The per-cell functions below are written over V: one cell (Real) or a pair
// of x-neighbours (float2), see pflb_vec.cuh.
// Viscosity: Sutherland (Sec. 4, eq. muT) or constant, lattice units.
template <class Real, int K, class V>
__device__ __forceinline__ V viscosity(const Params<Real, K>& P, V T) {
  if (!P.sutherland) return splat<V>(P.mu_lat);
  const V t = vmuls<V>(P.inv_suth_T, T);
  return vmul(vmul(vmuls<V>(P.mu_lat, t), fsqrt(t)),
              fdiv(splat<V>(P.suth_TS), vadds<V>(P.suth_S, T)));
}

// Viscosity and conductivity of the gas of composition Y at T (lattice
// units).  Single-gas mode: the viscosity law above and lambda = mu cp / Pr.
// Mixture mode (Sec. 4.4, eqs. muT_mix, phi_mix, conduct_mix): mole fractions
// X_k = Y_k Mw / M_k, species viscosities from their Sutherland laws,
// mu = sum_k mu_k X_k / sum_j Phi_kj X_j with
// Phi_kj = (1 + sqrt(mu_k / mu_j) (M_j / M_k)^(1/4))^2 / (sqrt(8) sqrt(1 + M_k / M_j)),
// lambda = (sum_k X_k lambda_k + 1 / sum_k X_k / lambda_k) / 2 with
// lambda_k = mu_k (1.32 cv_k + 1.77 R / M_k).
template <class Real, int K, class V>
__device__ __forceinline__ void transport(const Params<Real, K>& P, V T, const V* Y, V invMw, V cp,
                                          V& mu, V& lam) {
  const V one = splat<V>(Real(1));
  if constexpr (K > 0) {
    if (P.mix) {
      V X[K], m[K], sm[K], ism[K];
      const V Mw = vrcp(invMw);
#pragma unroll
      for (int k = 0; k < K; ++k) {
        X[k] = vmul(vmuls<V>(P.invM[k], Y[k]), Mw);
        const V t = vmuls<V>(P.inv_suth_Tk[k], T);
        m[k] = vmul(vmul(vmuls<V>(P.mu_lat_k[k], t), fsqrt(t)),
                    fdiv(splat<V>(P.suth_TSk[k]), vadds<V>(P.suth_Sk[k], T)));
        sm[k] = fsqrt(m[k]);
        ism[k] = vrcp(sm[k]);
      }
      V mm = splat<V>(Real(0)), l1 = mm, l2 = mm;
#pragma unroll
      for (int k = 0; k < K; ++k) {
        V den = splat<V>(Real(0));
#pragma unroll
        for (int j = 0; j < K; ++j) {
          const V a = vfma(vmuls<V>(P.wA[k][j], sm[k]), ism[j], one);
          den = vfma(vmul(a, a), vmuls<V>(P.wB[k][j], X[j]), den);
        }
        mm = vfma(vmul(m[k], X[k]), vrcp(den), mm);
        const V lk = vmuls<V>(P.eucken_k[k], m[k]);
        l1 = vfma(X[k], lk, l1);
        l2 = vfma(X[k], vrcp(lk), l2);
      }
      mu = mm;
      lam = vmuls<V>(Real(0.5), vadd(l1, vrcp(l2)));
      return;
    }
  }
  mu = viscosity<Real, K, V>(P, T);
  lam = vmuls<V>(P.inv_Pr, vmul(mu, cp));
}

template <class Real, int K, class V>
__device__ __forceinline__ V mixture_invMw(const Params<Real, K>& P, const V* Y) {
  if constexpr (K == 0) {
    return splat<V>(fdiv(Real(1), P.M0));
  } else {
    V s = vmuls<V>(P.invM[0], Y[0]);
#pragma unroll
    for (int k = 1; k < K; ++k) s = vfmas<V>(P.invM[k], Y[k], s);
    return s;
  }
}

template <class Real, int K, class V>
__device__ __forceinline__ V mixture_cp(const Params<Real, K>& P, const V* Y) {
  if constexpr (K == 0) {
    return splat<V>(P.cp0);
  } else {
    V s = vmuls<V>(P.cp[0], Y[0]);
#pragma unroll
    for (int k = 1; k < K; ++k) s = vfmas<V>(P.cp[k], Y[k], s);
    return s;
  }
}

// Explicit Arrhenius rates (Sec. 3.2.2 eq. 8, Sec. 3.3 eq. 9), per lattice
// step per rho_ref: om[k] = omega_k dt / rho_ref, omT likewise (J/kg).
template <class Real, int K, class V>
__device__ __forceinline__ void rates(const Params<Real, K>& P, V T, const V* Y, V rho, V invT,
                                      V* om, V& omT) {
  const V zero = splat<V>(Real(0));
#pragma unroll
  for (int k = 0; k < K; ++k) om[k] = zero;
  V C[Params<Real, K>::KK];
#pragma unroll
  for (int k = 0; k < K; ++k)
    C[k] = vmul(vmuls<V>(P.rho_ref_M[k], rho), vsel(vgt(Y[k], zero), Y[k], zero));
#pragma unroll 1
  for (int j = 0; j < P.J; ++j) {
    V kf = vmuls<V>(P.A_lat[j], fexp(vmuls<V>(-P.EaR[j], invT)));
    if (P.b[j] != Real(0)) kf = vmul(kf, fpow(T, P.b[j]));
    V q = kf;
#pragma unroll
    for (int k = 0; k < K; ++k) {
      const Real o = P.order[j][k];
      if (o == Real(1)) q = vmul(q, C[k]);
      else if (o == Real(2)) q = vmul(q, vmul(C[k], C[k]));
      else if (o != Real(0)) q = vmul(q, fpow(C[k], o));
    }
    if (P.rev[j]) {
      // k_r = k_f / K_c, K_c = exp(dS/R - dH/(R T)) (p_ref/(R T))^(sum s)
      const V Kc = vmul(fexp(vfmas<V>(-P.dH_R[j], invT, splat<V>(P.dS_R[j]))),
                        fpow(vmuls<V>(P.p_ref_R, invT), P.dn[j]));
      V qr = fdiv(kf, Kc);
#pragma unroll
      for (int k = 0; k < K; ++k) {
        const Real o = P.rorder[j][k];
        if (o == Real(1)) qr = vmul(qr, C[k]);
        else if (o == Real(2)) qr = vmul(qr, vmul(C[k], C[k]));
        else if (o != Real(0)) qr = vmul(qr, fpow(C[k], o));
      }
      q = vsub(q, qr);
    }
#pragma unroll
    for (int k = 0; k < K; ++k) om[k] = vfmas<V>(P.stoichM[j][k], q, om[k]);
  }
  V wt = zero;
#pragma unroll
  for (int k = 0; k < K; ++k) wt = vfmas<V>(-P.hf[k], om[k], wt);
  omT = wt;
}

// Solve A x = r in place (r <- x) by Gaussian elimination with partial
// pivoting; false if a pivot is zero.
template <int n, class LA>
__device__ __forceinline__ bool solve_pivoted(LA (*A)[n], LA* r) {
  LA dinv[n];
#pragma unroll
  for (int col = 0; col < n; ++col) {
    int piv = col;
    LA best = fabs(A[col][col]);
#pragma unroll
    for (int rr = col + 1; rr < n; ++rr) {
      const LA v = fabs(A[rr][col]);
      if (v > best) { best = v; piv = rr; }
    }
    if (best == LA(0)) return false;
#pragma unroll
    for (int rr = col + 1; rr < n; ++rr) {
      if (rr == piv) {
#pragma unroll
        for (int k = col; k < n; ++k) { const LA t = A[col][k]; A[col][k] = A[rr][k]; A[rr][k] = t; }
        const LA t = r[col]; r[col] = r[rr]; r[rr] = t;
      }
    }
    dinv[col] = LA(1) / A[col][col];
#pragma unroll
    for (int rr = col + 1; rr < n; ++rr) {
      const LA f = vmul(A[rr][col], dinv[col]);
#pragma unroll
      for (int k = col + 1; k < n; ++k) A[rr][k] = vfma(-f, A[col][k], A[rr][k]);
      r[rr] = vfma(-f, r[col], r[rr]);
    }
  }
#pragma unroll
  for (int rr = n - 1; rr >= 0; --rr) {
    LA s = r[rr];
#pragma unroll
    for (int k = rr + 1; k < n; ++k) s = vfma(-A[rr][k], r[k], s);
    r[rr] = vmul(s, dinv[rr]);
  }
  return true;
}

// ----------------------------------------------------- implicit chemistry
// One lattice step of the chemistry alone at frozen density (operator
// splitting), backward Euler: dY/dt = omega/rho, dT/dt = -sum hf omega / (rho
// cp(Y)), Newton with the analytic Jacobian (<= 30 iterations); if it fails
// the step is split into 2, 4, ..., 64 backward-Euler sub-steps.
//
// The species only move along the reactions: omega_k = sum_j M_k s_kj q_j, so
// after its first iteration the Newton iterate of the K + 1 unknowns (Y, T) is
// Y = Y_s + sum_j Ms_j xi_j, and the T row, with the rows of the reactions
// inserted, reads dT = R - sum_i a_i dxi_i with
//   R = -(T - T_s) - sum_j H_j xi_j / cp,  H_j = sum_k hf_k Ms_jk,
//   a_i = H_i / cp - (h / rho) (sum_j H_j q_j) / cp^2 sum_k cp_k Ms_ik.
// So the same iteration is carried by the J progress variables xi,
//   sum_i [delta_ji - hr (Q_ji - q_jT a_i)] dxi_i = hr (q_j + q_jT R) - xi_j,
//   Q_ji = sum_k dq_j/dY_k Ms_ik,  hr = h / rho,
// a J x J system (two reactions: 2 x 2) in place of the (K + 1) x (K + 1) one.
//
// FP64 domains do everything in FP64.  FP32 domains (LA = float) keep state,
// rates and right-hand side in FP64, form the factors of the Jacobian (powers,
// products before a factor, rate and heat derivatives, 1 / cp) in FP64 and
// narrow them, and take their products, the matrix, the solve and the update
// test in FP32: a direction off by about cond(A) x 6e-8 of itself still
// contracts, and the iteration stops where the FP64 right-hand side puts the
// root.  The FP64 pipe bounds this pre-pass (one warp instruction every 16
// cycles per SM, conversions and comparisons included), so the FP32 part takes
// its own copies of the constants, signs are tested on the bit pattern, and
// what an iteration needs only if another follows is left to that one (most
// cells are cold and take one).  2048 x 512 cells of the two-step bed, FP32
// domain, a step: 1.28 ms with the 7 x 7 system, 0.81 so (0.74 with the factors
// formed in FP32).

// Power C^o of a concentration for the reaction orders that occur (1, 2, 1/2:
// multiplications and a square root), pow() otherwise,
// with d = dC^o/dC for C > 0, in the precision LA of the Jacobian.
template <class R, class LA>
__device__ __forceinline__ R conc_power(R C, R o, LA& d) {
  if (o == R(1)) { d = LA(1); return C; }
  if (o == R(2)) { d = LA(2) * LA(C); return C * C; }
  if (o == R(0.5)) {
    const R s = sqrt(C);
    d = s > R(0) ? LA(0.5) / LA(s) : LA(0);
    return s;
  }
  const R p = pow(C, o);
  if constexpr (sizeof(R) == sizeof(LA)) d = C > R(0) ? o * R(pow(C, o - R(1))) : LA(0);
  else d = C > R(0) ? LA(o * p / C) : LA(0);
  return p;
}

// Rate constants of reaction j at T; k_r = 0 for an irreversible reaction.  FP32
// takes them as exponentials of their logarithms, so that neither over- nor
// underflows on the way.
template <int K>
__device__ __forceinline__ void rate_constants(const Chem64<K>& c, int j, double T, double invT,
                                               double& kf, double& kr) {
  kf = c.A[j] * exp(-c.EaR[j] * invT);
  if (c.b[j] != 0.0) kf *= pow(T, c.b[j]);
  kr = 0.0;
  if (c.rev[j]) {
    // 1 / K_c = exp(dH/(R T) - dS/R) (p_ref / (R T))^(-dn)
    double lnKi = vfma(c.dH_R[j], invT, -c.dS_R[j]);
    if (c.dn[j] == -0.5) {
      kr = kf * exp(lnKi) * sqrt(c.pref_R * invT);
    } else {
      if (c.dn[j] != 0.0) lnKi = vfma(-c.dn[j], vsub(c.ln_pref_R, log(T)), lnKi);
      kr = kf * exp(lnKi);
    }
  }
}
template <int K>
__device__ __forceinline__ void rate_constants(const Chem32<K>& c, int j, float T, float invT,
                                               float& kf, float& kr) {
  const float lnT = logf(T);
  const float lkf = vfma(-c.EaR[j], invT, vfma(c.b[j], lnT, c.lnA[j]));
  kf = expf(lkf);
  kr = 0.f;
  if (c.rev[j]) {
    const float lnKc = vfma(c.dn[j], vsub(c.ln_pref_R, lnT), vfma(-c.dH_R[j], invT, c.dS_R[j]));
    kr = expf(vsub(lkf, lnKc));
  }
}

// One Newton iteration's rates: q_j in Real, its derivatives dq_j/dT (qT) and
// along the reactions (Q[j][i]) in LA, from factors in Real.  C_k = rho Y_k / M_k
// and dC_k = rho / M_k are 0 where Y_k <= 0.  Species of order 0 are skipped (the
// orders are uniform).
template <int K, int J, class Real, class LA, class Chem, class ChemL>
__device__ __forceinline__ void reaction_rates(const Chem& c, const ChemL& cl, const Real* C,
                                               const LA* dC, Real T, Real invT, Real* q, LA* qT,
                                               LA (*Q)[J]) {
#pragma unroll
  for (int j = 0; j < J; ++j) {
    q[j] = Real(0);
    qT[j] = LA(0);
#pragma unroll
    for (int i = 0; i < J; ++i) Q[j][i] = LA(0);
    if (!c.active(j)) continue;
    Real kk[2];
    rate_constants<K>(c, j, T, invT, kk[0], kk[1]);
    Real dl = vmul(vfma(c.EaR[j], invT, c.b[j]), invT);  // d ln k / dT, forward
    Real dT = Real(0);
#pragma unroll
    for (int dir = 0; dir < 2; ++dir) {
      if (dir == 1 && !c.rev[j]) break;
      if (dir == 1) dl = vfma(-vfma(c.dH_R[j], invT, c.dn[j]), invT, dl);
      // prefix / suffix products: the product without factor k, no division
      LA Pw[K], pre[K], Dp[K], suf = LA(1);
      Real prod = dir == 0 ? kk[0] : -kk[1];
#pragma unroll
      for (int k = 0; k < K; ++k) {
        const Real o = dir == 0 ? c.order[j][k] : c.rorder[j][k];
        if (o == Real(0)) continue;
        pre[k] = LA(prod);
        const Real p = conc_power(C[k], o, Dp[k]);
        Pw[k] = LA(p);
        prod = vmul(prod, p);
      }
      q[j] = vadd(q[j], prod);
      dT = vfma(prod, dl, dT);
#pragma unroll
      for (int k = K - 1; k >= 0; --k) {
        const Real o = dir == 0 ? c.order[j][k] : c.rorder[j][k];
        if (o == Real(0)) continue;
        const LA d = vmul(vmul(pre[k], suf), vmul(Dp[k], dC[k]));
        suf = vmul(suf, Pw[k]);
#pragma unroll
        for (int i = 0; i < J; ++i) Q[j][i] = vfma(d, cl.Ms[i][k], Q[j][i]);
      }
    }
    qT[j] = LA(dT);
  }
}

// The system of one iteration (see above): matrix A, right-hand side r and the
// row a of dT.  hr = h / rho, icp = 1 / cp, w = hr (sum_j H_j q_j) / cp^2,
// rhs_j = hr q_j - xi_j, R.
template <int K, int J, class LA, class ChemL>
__device__ __forceinline__ void reaction_system(const ChemL& cl, LA hr, LA icp, LA w,
                                                const LA* rhs, const LA* qT, const LA (*Q)[J], LA R,
                                                LA (*A)[J], LA* r, LA* a) {
#pragma unroll
  for (int i = 0; i < J; ++i) a[i] = vfma(-w, cl.cM[i], vmul(cl.H[i], icp));
#pragma unroll
  for (int j = 0; j < J; ++j) {
    r[j] = vfma(vmul(hr, qT[j]), R, rhs[j]);
#pragma unroll
    for (int i = 0; i < J; ++i)
      A[j][i] = vfma(-hr, vfma(-qT[j], a[i], Q[j][i]), LA(i == j ? 1 : 0));
  }
}

// The least LA not below a threshold x: a value in LA is below it when it is
// below x.
template <class LA> __device__ __forceinline__ LA threshold(double x);
template <> __device__ __forceinline__ double threshold<double>(double x) { return x; }
template <> __device__ __forceinline__ float threshold<float>(double x) { return __double2float_ru(x); }

// z > 0 by its bits (a comparison would go through the FP64 pipe)
__device__ __forceinline__ bool positive(double z) { return __double_as_longlong(z) > 0; }

template <int K, int J, class LA, class ChemL>
__device__ __forceinline__ void chem_be_newton(const Chem64<K>& c, const ChemL& cl, double T0,
                                               const double* Y0, double rho, double* dY,
                                               double* dT) {
  const double inv_rho = 1.0 / rho;
  double acc[K], accT = 0.0;  // increments of the finished sub-steps
  int ok = -1;
#pragma unroll 1
  for (int nsub = 1; nsub <= 64 && ok != 0; nsub *= 2) {
#pragma unroll
    for (int k = 0; k < K; ++k) acc[k] = 0.0;
    accT = 0.0;
    ok = 0;
    const double hr = c.dt / nsub * inv_rho;
    const LA hrL = LA(hr);
#pragma unroll 1
    for (int sub = 0; sub < nsub && ok == 0; ++sub) {
      const double Ts = vadd(T0, accT);
      const LA tolT = threshold<LA>(1e-13 * Ts), tolY = threshold<LA>(1e-13);
      double xi[J], T = Ts, z[K];
#pragma unroll
      for (int j = 0; j < J; ++j) xi[j] = 0.0;
#pragma unroll
      for (int k = 0; k < K; ++k) z[k] = sub == 0 ? Y0[k] : vadd(Y0[k], acc[k]);
      ok = -1;
#pragma unroll 1
      for (int it = 0; it < 30; ++it) {
        double C[K], q[J], R = 0.0, cp = 0.0, Hq = 0.0;
        LA dC[K], qT[J], Q[J][J], A[J][J], r[J], a[J], rhs[J];
#pragma unroll
        for (int k = 0; k < K; ++k) {
          C[k] = 0.0;
          dC[k] = LA(0);
          if ((c.used & (1 << k)) && positive(z[k])) {
            const double d = vmul(rho, c.invM[k]);
            dC[k] = LA(d);
            C[k] = vmul(z[k], d);
          }
          cp = vfma(z[k], c.cp[k], cp);
        }
        reaction_rates<K, J, double, LA>(c, cl, C, dC, T, 1.0 / T, q, qT, Q);
        const double icp = 1.0 / cp;
        if (it > 0) {  // R = 0 in the first iteration
          double Hxi = 0.0;
#pragma unroll
          for (int j = 0; j < J; ++j) Hxi = vfma(c.H[j], xi[j], Hxi);
          R = vfma(-Hxi, icp, vsub(Ts, T));
        }
#pragma unroll
        for (int j = 0; j < J; ++j) {
          Hq = vfma(c.H[j], q[j], Hq);
          rhs[j] = LA(vfma(hr, q[j], -xi[j]));
        }
        const double w = vmul(vmul(hr, Hq), vmul(icp, icp));
        reaction_system<K, J, LA>(cl, hrL, LA(icp), LA(w), rhs, qT, Q, LA(R), A, r, a);
        if (!solve_pivoted<J, LA>(A, r)) break;
        LA ar = LA(0);
#pragma unroll
        for (int j = 0; j < J; ++j) {
          xi[j] = vadd(xi[j], double(r[j]));
          ar = vfma(a[j], r[j], ar);
        }
        const double dTn = vsub(R, double(ar));
        T = vadd(T, dTn);
        // update test: species absolute, temperature relative to the start
        const LA eT = fabs(LA(dTn));
        bool bad = !(eT == eT), done = eT < tolT;
#pragma unroll
        for (int k = 0; k < K; ++k) {
          LA e = LA(0);
#pragma unroll
          for (int j = 0; j < J; ++j) e = vfma(cl.Ms[j][k], r[j], e);
          e = fabs(e);
          if (!(e == e)) bad = true;
          if (!(e < tolY)) done = false;
        }
        if (bad || !positive(T)) break;
        if (done) { ok = 0; break; }
#pragma unroll
        for (int k = 0; k < K; ++k) {
          double d = 0.0;
#pragma unroll
          for (int j = 0; j < J; ++j) d = vfma(c.Ms[j][k], xi[j], d);
          z[k] = vadd(vadd(Y0[k], acc[k]), d);
        }
      }
#pragma unroll
      for (int k = 0; k < K; ++k) {
        double d = 0.0;
#pragma unroll
        for (int j = 0; j < J; ++j) d = vfma(c.Ms[j][k], xi[j], d);
        acc[k] = vadd(acc[k], d);
      }
      accT = vadd(accT, vsub(T, Ts));
    }
  }
  // differences of states, as a full iterate gives them: what the state cannot
  // resolve is no increment
#pragma unroll
  for (int k = 0; k < K; ++k) dY[k] = vsub(vadd(Y0[k], acc[k]), Y0[k]);
  *dT = accT;
}

// The same step in FP32 for the cells that the surrogate rejects in FP32
// domains.  FP32 cannot hold the root to the FP64 integrator's 1e-13: the
// unknowns are the sub-step's increments (small numbers keep their relative
// precision), and the iteration stops once every update is below
// 1e-5 |d_m| + 1e-6 |z_m| (a few units in the last place of the FP32 field
// that receives the increment).
template <int K, int J>
__device__ __forceinline__ void chem_be_newton32(const Chem32<K>& c, float T0, const float* Y0,
                                                 float rho, float* dY, float* dT) {
  const float inv_rho = 1.f / rho;
  float acc[K], accT = 0.f;
  int ok = -1;
#pragma unroll 1
  for (int nsub = 1; nsub <= 64 && ok != 0; nsub *= 2) {
#pragma unroll
    for (int k = 0; k < K; ++k) acc[k] = 0.f;
    accT = 0.f;
    ok = 0;
    const float hr = c.dt / float(nsub) * inv_rho;
#pragma unroll 1
    for (int sub = 0; sub < nsub && ok == 0; ++sub) {
      const float Ts = vadd(T0, accT);
      float xi[J], dTs = 0.f, d[K];
#pragma unroll
      for (int j = 0; j < J; ++j) xi[j] = 0.f;
#pragma unroll
      for (int k = 0; k < K; ++k) d[k] = 0.f;
      ok = -1;
#pragma unroll 1
      for (int it = 0; it < 30; ++it) {
        const float T = vadd(Ts, dTs);
        if (!(T > 0.f)) break;
        float Cc[K], dC[K], q[J], rhs[J], qT[J], Q[J][J], A[J][J], r[J], a[J], cp = 0.f, Hq = 0.f;
#pragma unroll
        for (int k = 0; k < K; ++k) {
          const float z = vadd(vadd(Y0[k], acc[k]), d[k]);
          dC[k] = z > 0.f ? rho * c.invM[k] : 0.f;
          Cc[k] = vmul(z, dC[k]);
          cp = vfma(z, c.cp[k], cp);
        }
        reaction_rates<K, J, float, float>(c, c, Cc, dC, T, 1.f / T, q, qT, Q);
        const float icp = 1.f / cp;
        float Hxi = 0.f;
#pragma unroll
        for (int j = 0; j < J; ++j) {
          Hxi = vfma(c.H[j], xi[j], Hxi);
          Hq = vfma(c.H[j], q[j], Hq);
          rhs[j] = vfma(hr, q[j], -xi[j]);
        }
        const float R = vfma(-Hxi, icp, -dTs);
        const float w = vmul(vmul(hr, Hq), vmul(icp, icp));
        reaction_system<K, J, float>(c, hr, icp, w, rhs, qT, Q, R, A, r, a);
        if (!solve_pivoted<J, float>(A, r)) break;
        float dTn = R;
#pragma unroll
        for (int j = 0; j < J; ++j) {
          xi[j] = vadd(xi[j], r[j]);
          dTn = vfma(-a[j], r[j], dTn);
        }
        dTs = vadd(dTs, dTn);
        bool bad = !(dTn == dTn);
        bool done = fabsf(dTn) <= 1e-5f * fabsf(dTs) + 1e-6f * Ts;
#pragma unroll
        for (int k = 0; k < K; ++k) {
          float e = 0.f, s = 0.f;
#pragma unroll
          for (int j = 0; j < J; ++j) {
            e = vfma(c.Ms[j][k], r[j], e);
            s = vfma(c.Ms[j][k], xi[j], s);
          }
          d[k] = s;
          if (!(e == e)) bad = true;
          if (fabsf(e) > 1e-5f * fabsf(s) + 1e-6f * fabsf(vadd(Y0[k], acc[k]))) done = false;
        }
        if (bad) break;
        if (done) { ok = 0; break; }
      }
#pragma unroll
      for (int k = 0; k < K; ++k) acc[k] = vadd(acc[k], d[k]);
      accT = vadd(accT, dTs);
    }
  }
#pragma unroll
  for (int k = 0; k < K; ++k) dY[k] = acc[k];
  *dT = accT;
}

// Moments read straight from global memory (the moments kernel, no staging).
template <class Real>
struct GlobalMom {
  const Real* M;
  int N;
  __device__ __forceinline__ Real mom(int a, int src, int, int, int) const {
    return M[(size_t)a * N + src];
  }
};

// First-order part w_i (P + 3 c_i . j) of direction i at the source cell
// (global index src, offset (dx, dy, dz) from the pulling cell).
template <int DIM, class Real, class MA>
__device__ __forceinline__ Real first_order(const MA& A, int i, int src, int dx, int dy, int dz) {
  using L = Lattice<DIM>;
  Real cj = 0;
#pragma unroll
  for (int a = 0; a < DIM; ++a) {
    if (L::c(i, a) > 0) cj = vadd(cj, A.mom(1 + a, src, dx, dy, dz));
    if (L::c(i, a) < 0) cj = vsub(cj, A.mom(1 + a, src, dx, dy, dz));
  }
  return vmul(Real(L::w(i)), vfma(Real(3), cj, A.mom(0, src, dx, dy, dz)));
}

template <class Real, int K>
__device__ __forceinline__ Real inlet_u(const Params<Real, K>& P, Real u, const int xyz[3],
                                        int dim) {
  if (P.inlet_parabolic != 1) return u;
  for (int a = 1; a < dim; ++a) {
    if (P.bc[2 * a] != BC_WALL) continue;
    Real n = Real(a == 1 ? P.ny : P.nz);
    Real s = Real(xyz[a]) + Real(0.5);
    u = vmul(u, fdiv(vmul(vmul(Real(4), s), vsub(n, s)), vmul(n, n)));
  }
  return u;
}

// The cell's own post-collision population of direction ib (bounce-back).
template <int DIM, class Real, class Store, int K, class MA>
__device__ __forceinline__ Real own_pop(const Params<Real, K>& P, const State<Real, Store>& S,
                                        int c, int ib, const MA& mom) {
  const Real r = Codec<Store, Real>::raw(S.g_in + (size_t)ib * P.N + c);
  if constexpr (IsHalf<Store>::value)
    return Codec<Store, Real>::dec(r, Real(Lattice<DIM>::w(ib)) * P.g_inv_scale,
                                   first_order<DIM, Real>(mom, ib, c, 0, 0, 0));
  else return r;
}

// Half-way bounce-back with the wall velocity for the directions entering
// through face F, when the cell lies on it (on) and it is a wall.
template <int DIM, int F, class Real, class Store, int K, class MA>
__device__ __forceinline__ void wall_pops(const Params<Real, K>& P, const State<Real, Store>& S,
                                          int c, bool on, Real rho_c, Real* gin, const MA& mom) {
  using L = Lattice<DIM>;
  constexpr int a = F >> 1, s = (F & 1) ? -1 : 1;
  if (!(on && P.bc[F] == BC_WALL)) return;
#pragma unroll
  for (int i = 0; i < L::Q; ++i) {
    if (L::c(i, a) != s) continue;
    Real cu = 0;
#pragma unroll
    for (int b = 0; b < DIM; ++b) {
      if (L::c(i, b) > 0) cu = vadd(cu, P.wall_u[F][b]);
      if (L::c(i, b) < 0) cu = vsub(cu, P.wall_u[F][b]);
    }
    gin[i] = vfma(vmul(Real(2 * L::w(i)), rho_c), cu,
                  own_pop<DIM, Real, Store>(P, S, c, L::opp(i), mom));
  }
}

// The boundary rules of a cell on non-periodic faces: directions that cross a
// non-periodic face are replaced, in the order outlet, inlet, walls (the wall
// of the lowest axis last, so it wins on edges and corners): half-way
// bounce-back on walls (moving walls add 2 w rho c.u_w), the inlet as a moving
// wall with the inlet velocity and inlet density, the outlet as
// anti-bounce-back at P_h = 0 with wall velocity uw.
template <int DIM, class Real, class Store, int K, class MA>
__device__ __forceinline__ void edge_rules(const Params<Real, K>& P, const State<Real, Store>& S,
                                           int c, const int xyz[3], Real rho_c, Real rho_in,
                                           const Real* uw, Real* gin, const MA& mom) {
  using L = Lattice<DIM>;
  const int x = xyz[0], y = xyz[1], z = DIM == 3 ? xyz[2] : 0;
  const bool per0 = P.bc[0] == BC_PERIODIC, per1 = P.bc[1] == BC_PERIODIC;
  const bool per2 = P.bc[2] == BC_PERIODIC, per3 = P.bc[3] == BC_PERIODIC;
  const bool per4 = P.bc[4] == BC_PERIODIC, per5 = P.bc[5] == BC_PERIODIC;
  // non-periodic faces the cell lies on
  const bool f0 = x == 0 && !per0, f1 = x == P.nx - 1 && !per1;
  const bool f2 = y == 0 && !per2, f3 = y == P.ny - 1 && !per3;
  const bool f4 = DIM == 3 && z == 0 && !per4, f5 = DIM == 3 && z == P.nz - 1 && !per5;
  if (!(f0 || f1 || f2 || f3 || f4 || f5)) return;
  if (f1 && P.bc[1] == BC_OUTLET) {
    Real uu = 0;
#pragma unroll
    for (int a = 0; a < DIM; ++a) uu = vfma(uw[a], uw[a], uu);
    const Real pb2 = P.nscbc ? Real(2) * scal_pb<Real>(S.scal) : Real(0);
#pragma unroll
    for (int i = 0; i < L::Q; ++i) {
      if (L::c(i, 0) != -1) continue;
      Real cu = 0;
#pragma unroll
      for (int a = 0; a < DIM; ++a) {
        if (L::c(i, a) > 0) cu = vadd(cu, uw[a]);
        if (L::c(i, a) < 0) cu = vsub(cu, uw[a]);
      }
      gin[i] = vfma(Real(L::w(i)), vfma(rho_c, vfma(vmul(Real(3), cu), cu, -uu), pb2),
                    -own_pop<DIM, Real, Store>(P, S, c, L::opp(i), mom));
    }
  }
  if (f0 && P.bc[0] == BC_INLET) {
    Real ui = inlet_u(P, P.feed ? scal_u_in<Real>(S.scal) : P.u_in, xyz, DIM);
    if (P.inlet_parabolic == 2) ui = vmul(ui, vsub(Real(1), S.phi[c]));
#pragma unroll
    for (int i = 0; i < L::Q; ++i) {
      if (L::c(i, 0) != 1) continue;
      gin[i] = vfma(vmul(Real(2 * L::w(i)), rho_in), ui,
                    own_pop<DIM, Real, Store>(P, S, c, L::opp(i), mom));
    }
  }
  // walls, the highest axis first so that the lowest axis wins on edges
  if (DIM == 3) {
    wall_pops<DIM, 5>(P, S, c, f5, rho_c, gin, mom);
    wall_pops<DIM, 4>(P, S, c, f4, rho_c, gin, mom);
  }
  wall_pops<DIM, 3>(P, S, c, f3, rho_c, gin, mom);
  wall_pops<DIM, 2>(P, S, c, f2, rho_c, gin, mom);
  wall_pops<DIM, 1>(P, S, c, f1, rho_c, gin, mom);
  wall_pops<DIM, 0>(P, S, c, f0, rho_c, gin, mom);
}

// Pull streaming of every population into the cell.  A cell off every face
// reads its upstream neighbours at fixed offsets.  On a face, along each axis
// the upstream neighbour coordinate wraps across a periodic face and is
// clamped to the cell itself across any other face; every direction is read
// from there.  Directions that cross a non-periodic face are then replaced by
// the boundary rules.
template <int DIM, class Real, class Store, int K, class MA>
__device__ __forceinline__ void pull(const Params<Real, K>& P, const State<Real, Store>& S, int c,
                                     const int xyz[3], Real rho_c, Real rho_in, const Real* uw,
                                     Real* gin, const MA& mom) {
  using L = Lattice<DIM>;
  constexpr bool FO = IsHalf<Store>::value;  // residual storage: add the first-order part
  // cells off every domain face: fixed offsets from the cell (the common case)
  const bool inner = xyz[0] > 0 && xyz[0] < P.nx - 1 && xyz[1] > 0 && xyz[1] < P.ny - 1 &&
                     (DIM == 2 || (xyz[2] > 0 && xyz[2] < P.nz - 1));
  if (inner) {
    const int sy = P.nx, sz = P.nx * P.ny;
#pragma unroll
    for (int i = 0; i < L::Q; ++i) {
      const int cx = L::c(i, 0), cy = L::c(i, 1), cz = DIM == 3 ? L::c(i, 2) : 0;
      const int src = c - cx - cy * sy - cz * sz;
      const Real r = Codec<Store, Real>::raw(S.g_in + (size_t)i * P.N + src);
      if constexpr (FO)
        gin[i] = Codec<Store, Real>::dec(r, Real(L::w(i)) * P.g_inv_scale,
                                         first_order<DIM, Real>(mom, i, src, -cx, -cy, -cz));
      else gin[i] = r;
    }
    return;
  }
  // upstream neighbour coordinates along each axis: m (coordinate - 1) and
  // p (coordinate + 1), wrapped across periodic faces, clamped otherwise
  const int x = xyz[0], y = xyz[1], z = DIM == 3 ? xyz[2] : 0;
  const bool per0 = P.bc[0] == BC_PERIODIC, per1 = P.bc[1] == BC_PERIODIC;
  const bool per2 = P.bc[2] == BC_PERIODIC, per3 = P.bc[3] == BC_PERIODIC;
  const bool per4 = P.bc[4] == BC_PERIODIC, per5 = P.bc[5] == BC_PERIODIC;
  const int xm = x > 0 ? x - 1 : (per0 ? P.nx - 1 : x);
  const int xp = x < P.nx - 1 ? x + 1 : (per1 ? 0 : x);
  const int ym = y > 0 ? y - 1 : (per2 ? P.ny - 1 : y);
  const int yp = y < P.ny - 1 ? y + 1 : (per3 ? 0 : y);
  const int zm = DIM == 3 ? (z > 0 ? z - 1 : (per4 ? P.nz - 1 : z)) : 0;
  const int zp = DIM == 3 ? (z < P.nz - 1 ? z + 1 : (per5 ? 0 : z)) : 0;
#pragma unroll
  for (int i = 0; i < L::Q; ++i) {
    const int cx = L::c(i, 0), cy = L::c(i, 1), cz = DIM == 3 ? L::c(i, 2) : 0;
    const int sx = cx > 0 ? xm : (cx < 0 ? xp : x);
    const int sy = cy > 0 ? ym : (cy < 0 ? yp : y);
    const int sz = cz > 0 ? zm : (cz < 0 ? zp : z);
    const int src = sx + P.nx * (sy + P.ny * sz);
    const Real r = Codec<Store, Real>::raw(S.g_in + (size_t)i * P.N + src);
    // a periodic source: the staged halo holds its image at the same offset
    if constexpr (FO)
      gin[i] = Codec<Store, Real>::dec(r, Real(L::w(i)) * P.g_inv_scale,
                                       first_order<DIM, Real>(mom, i, src, -cx, -cy, -cz));
    else gin[i] = r;
  }
  edge_rules<DIM>(P, S, c, xyz, rho_c, rho_in, uw, gin, mom);
}

// ----------------------------------------------------------- reductions
// Error-free sum of two floats (Knuth's two-sum).
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
  s = a + b;
  const float bb = s - a;
  e = (a - (s - bb)) + (b - bb);
}

// Block sum of one per-thread value into FP64 (result in thread 0).  FP32
// values are summed within the warp with compensation (the pair s + e is
// exact up to the final rounding), warps are combined in FP64.
// Warp part of the sums below (result in lane 0).
template <class V>
__device__ __forceinline__ double warp_sum(V v) {
  if constexpr (sizeof(typename Lanes<V>::S) == 4) {
    float s, e = 0.f;
    if constexpr (Lanes<V>::n == 2) two_sum(v.x, v.y, s, e);
    else s = v;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const float so = __shfl_down_sync(0xffffffffu, s, o);
      const float eo = __shfl_down_sync(0xffffffffu, e, o);
      float t, err;
      two_sum(s, so, t, err);
      s = t;
      e = e + eo + err;
    }
    return double(s) + double(e);
  } else {
    double w = v;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) w += __shfl_down_sync(0xffffffffu, w, o);
    return w;
  }
}

// The three sums of a tile (I, and the two fluxes when `bc` holds) with one
// barrier, grouped exactly as block_sum; results valid in thread 0.  `sh`
// holds 96 doubles and is free again after the block's next barrier.
// With `df` a fourth sum (of doubles: the fuel consumed), `sh` then 128 doubles.
template <class V, class Real>
__device__ __forceinline__ void block_sum4(V a, Real b, Real c, bool bc, double d, bool df,
                                           double* sh, double& ra, double& rb, double& rc,
                                           double& rd) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const double wa = warp_sum(a);
  const double wb = bc ? warp_sum(b) : 0.0, wc = bc ? warp_sum(c) : 0.0;
  if (lane == 0) {
    sh[wid] = wa;
    sh[32 + wid] = wb;
    sh[64 + wid] = wc;
  }
  if (df) {
    d = warp_sum(d);
    if (lane == 0) sh[96 + wid] = d;
  }
  __syncthreads();
  ra = rb = rc = rd = 0.0;
  if (wid == 0) {
    const bool in = lane < (int)(blockDim.x >> 5);
    double x = in ? sh[lane] : 0.0, y = in ? sh[32 + lane] : 0.0, z = in ? sh[64 + lane] : 0.0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      x += __shfl_down_sync(0xffffffffu, x, o);
      y += __shfl_down_sync(0xffffffffu, y, o);
      z += __shfl_down_sync(0xffffffffu, z, o);
    }
    ra = x;
    rb = bc ? y : 0.0;
    rc = bc ? z : 0.0;
    if (df) {
      double f = in ? sh[96 + lane] : 0.0;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) f += __shfl_down_sync(0xffffffffu, f, o);
      rd = f;
    }
  }
}

template <class V, class Real>
__device__ __forceinline__ void block_sum3(V a, Real b, Real c, bool bc, double* sh,
                                           double& ra, double& rb, double& rc) {
  double none = 0.0, rd;
  block_sum4(a, b, c, bc, none, false, sh, ra, rb, rc, rd);
}
template <class Real>
__device__ __forceinline__ double block_sum(Real v, double* sh) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  double w;
  if constexpr (sizeof(Real) == 4) {
    float s = v, e = 0.f;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const float so = __shfl_down_sync(0xffffffffu, s, o);
      const float eo = __shfl_down_sync(0xffffffffu, e, o);
      float t, err;
      two_sum(s, so, t, err);
      s = t;
      e = e + eo + err;
    }
    w = double(s) + double(e);
  } else {
    w = v;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) w += __shfl_down_sync(0xffffffffu, w, o);
  }
  if (lane == 0) sh[wid] = w;
  __syncthreads();
  double r = 0;
  if (wid == 0) {
    r = lane < (int)(blockDim.x >> 5) ? sh[lane] : 0.0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) r += __shfl_down_sync(0xffffffffu, r, o);
  }
  __syncthreads();
  return r;
}

// The scalar state after a step (or, is_init, of a new one) from its sums, by
// one thread: the P0 closure when the domain is closed, the diagnostics and the
// per-step constants the cells of the next step read.  With the inlet feedback
// (feed_c > 0, Sec. 4.4.1) the fuel the step consumed, phi_f (-omega_k) of its
// input state, sets the inlet peak speed of the next step, u_in = fuel feed_c /
// P0, held in [0, 0.3].
__device__ __forceinline__ void apply_sums(double I, double in, double out, double fuel,
                                           DevScalars* scal, int p0_closed, bool is_init,
                                           double init_P0, double eos_c, double inv_rho_ref,
                                           double feed_c) {
  double P0, P0p;
  if (is_init) {
    P0 = P0p = init_P0;
    scal->mass = init_P0 * I * eos_c;
    scal->flux_in = scal->flux_out = 0;
    scal->flux_in_sum = scal->flux_out_sum = 0;
    scal->step = 0;
    scal->status = 0;
  } else {
    P0p = scal->P0;
    P0 = P0p;
    if (p0_closed) P0 = scal->mass / (I * eos_c);
    scal->flux_in = in;
    scal->flux_out = out;
    scal->flux_in_sum += in;
    scal->flux_out_sum += out;
    scal->step += 1;
    // latch only the first failure (a timeout is not overwritten)
    if (scal->status == 0 && (!(I == I) || !(P0 == P0) || I <= 0.0)) scal->status = -5;
  }
  scal->P0_prev = P0p;
  scal->P0 = P0;
  scal->I = I;
  scal->mass_now = P0 * I * eos_c;
  scal->dlnP0 = (P0 - P0p) / P0;
  scal->dP0r = (P0 - P0p) * inv_rho_ref;
  scal->P0_f = float(P0);
  scal->dlnP0_f = float(scal->dlnP0);
  scal->dP0r_f = float(scal->dP0r);
  if (feed_c > 0.0) {
    double u = fuel * feed_c / P0;
    u = u > 0.3 ? 0.3 : (u > 0.0 ? u : 0.0);  // NaN -> 0
    scal->fuel = fuel;
    scal->u_in = u;
    scal->u_in_f = float(u);
  }
}

// Slots of one share of the combine by a block.
constexpr unsigned SLOT_RUN = 256;
// Slots that a lane has in flight: eight, so that a short list waits for memory
// once; four in the kernels without species, whose 64 registers eight would spill.
__host__ __device__ constexpr int slots_in_flight(int K) { return K == 0 ? 4 : 8; }

// The warp's sums over the shares w0, w0 + nw, ... of the slots (I, inlet and
// outlet flux and, FUEL, the fuel); valid in lane 0.  A lane adds every 32nd slot
// of a share in order, F of them in flight.  Only the slots that there are cost an
// addition: the FP64 pipe takes a warp's instruction every 16 cycles, and 32
// additions by every warp of a block were 1.5 to 3 us of it whatever the list.
template <bool FUEL, int F>
__device__ __forceinline__ void sum_slots(const double* partials, unsigned nb, unsigned w0,
                                          unsigned nw, double v[4]) {
  const unsigned lane = threadIdx.x & 31;
  v[0] = v[1] = v[2] = v[3] = 0.0;
  for (unsigned w = w0; w * SLOT_RUN < nb; w += nw) {
#pragma unroll 1
    for (unsigned s = w * SLOT_RUN; s < min(nb, (w + 1) * SLOT_RUN); s += 32 * F) {
      double2 a[F], c[F];
#pragma unroll
      for (int q = 0; q < F; ++q) {
        const unsigned b = s + 32 * q + lane;
        const double* p = partials + 4 * (size_t)b;
        a[q] = c[q] = make_double2(0.0, 0.0);
        if (b < nb) {
          a[q] = __ldcg(reinterpret_cast<const double2*>(p));
          if constexpr (FUEL) c[q] = __ldcg(reinterpret_cast<const double2*>(p) + 1);
          else c[q].x = __ldcg(p + 2);
        }
      }
#pragma unroll
      for (int q = 0; q < F; ++q) {
        if (s + 32 * q >= nb) break;
        v[0] += a[q].x;
        v[1] += a[q].y;
        v[2] += c[q].x;
        if constexpr (FUEL) v[3] += c[q].y;
      }
    }
  }
#pragma unroll
  for (int k = 0; k < (FUEL ? 4 : 3); ++k)
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v[k] += __shfl_down_sync(0xffffffffu, v[k], o);
}

// Combine the per-block partials of one step in a fixed order (strided sums,
// then a fixed shuffle tree) and update the scalar state: by one warp.
template <int F>
__device__ __forceinline__ void combine_partials(const double* partials, unsigned nb,
                                                 DevScalars* scal, int p0_closed, bool is_init,
                                                 double init_P0, double eos_c,
                                                 double inv_rho_ref, double feed_c = 0.0) {
  double v[4];
  if (feed_c > 0.0) sum_slots<true, F>(partials, nb, 0, 1, v);
  else sum_slots<false, F>(partials, nb, 0, 1, v);
  if ((threadIdx.x & 31) == 0)
    apply_sums(v[0], v[1], v[2], v[3], scal, p0_closed, is_init, init_P0, eos_c, inv_rho_ref,
               feed_c);
}

// The same for a fixed P0 by a whole block (every thread calls it; `sh` holds
// 96 doubles and is free again after the block's next barrier): one warp takes
// 25 us over the 4,096 slots of a 2048 x 512 domain.  Up to SLOT_RUN slots are
// left to the first warp; beyond, eight warps' shares are dealt to the warps that
// there are, so that the sums are the same bits under every block size.
template <int F>
__device__ __forceinline__ void combine_partials_block(const double* partials, unsigned nb,
                                                       DevScalars* scal, double eos_c,
                                                       double inv_rho_ref, double* sh) {
  const unsigned lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (nb <= SLOT_RUN) {
    if (wid == 0) combine_partials<F>(partials, nb, scal, 0, false, 0.0, eos_c, inv_rho_ref);
    return;
  }
#pragma unroll 1
  for (unsigned w = wid; w < 8 && w * SLOT_RUN < nb; w += blockDim.x / 32) {
    double v[4];
    sum_slots<false, F>(partials, nb, w, 8, v);
    if (lane == 0)
#pragma unroll
      for (int k = 0; k < 3; ++k) sh[32 * k + w] = v[k];
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double u[3] = {0.0, 0.0, 0.0};
    for (unsigned q = 0; q < 8 && q * SLOT_RUN < nb; ++q)
      for (int k = 0; k < 3; ++k) u[k] += sh[32 * k + q];
    apply_sums(u[0], u[1], u[2], 0.0, scal, 0, false, 0.0, eos_c, inv_rho_ref, 0.0);
  }
}

// Publish the block sums (valid in thread 0) of this step.  Closed domains
// need P0 of the next step before it starts, so the warp that draws the last
// arrival ticket combines at once (lane 0 fences its own writes before taking
// the ticket; the other warps retire).  With a fixed P0 the combine is
// deferred: the first block of the next launch, or the on-demand finalize kernel,
// does it, and the step ends without a serial tail.
// Write the sums into slot `bid`.
__device__ __forceinline__ void write_partials(double sI, double sIn, double sOut,
                                               double* partials, unsigned bid, double sF = 0.0) {
  if (threadIdx.x == 0) {
    partials[4 * bid + 3] = sF;
    partials[4 * bid + 0] = sI;
    partials[4 * bid + 1] = sIn;
    partials[4 * bid + 2] = sOut;
  }
}
// Count `n` slots that this block has written; the block that completes the
// `nb` slots combines them.  (First warp; the others pass.)
template <int F>
__device__ __forceinline__ void count_partials(double* partials, unsigned* counter,
                                               DevScalars* scal, int p0_closed, bool is_init,
                                               double init_P0, double eos_c, double inv_rho_ref,
                                               unsigned n, unsigned nb, double feed_c = 0.0) {
  if (threadIdx.x >= 32) return;
  const int lane = threadIdx.x;
  unsigned last = 0;
  if (lane == 0) {
    __threadfence();
    last = (atomicAdd(counter, n) == nb - n) ? 1u : 0u;
  }
  last = __shfl_sync(0xffffffffu, last, 0);
  if (!last) return;
  __threadfence();
  combine_partials<F>(partials, nb, scal, p0_closed, is_init, init_P0, eos_c, inv_rho_ref, feed_c);
  if (lane == 0) *counter = 0u;
}
// Publish into slot `bid` of `nb`; `now` combines at the last arrival.
template <int F>
__device__ __forceinline__ void publish_partials_at(double sI, double sIn, double sOut,
                                                    double* partials, unsigned* counter,
                                                    DevScalars* scal, int p0_closed, bool is_init,
                                                    double init_P0, double eos_c,
                                                    double inv_rho_ref, unsigned bid,
                                                    unsigned nb, bool now, double sF = 0.0,
                                                    double feed_c = 0.0) {
  write_partials(sI, sIn, sOut, partials, bid, sF);
  if (now)
    count_partials<F>(partials, counter, scal, p0_closed, is_init, init_P0, eos_c, inv_rho_ref, 1u,
                      nb, feed_c);
}

template <int F>
__device__ __forceinline__ void publish_partials(double sI, double sIn, double sOut,
                                                 double* partials, unsigned* counter,
                                                 DevScalars* scal, int p0_closed, bool is_init,
                                                 double init_P0, double eos_c,
                                                 double inv_rho_ref, double sF = 0.0,
                                                 double feed_c = 0.0) {
  publish_partials_at<F>(sI, sIn, sOut, partials, counter, scal, p0_closed, is_init, init_P0, eos_c,
                         inv_rho_ref, blockIdx.x, gridDim.x, p0_closed || is_init || feed_c > 0.0,
                         sF, feed_c);
}

// On-demand combine of the deferred partials of the last step (one block), to
// the same bits as the next step's: by the block, or by its first warp (FP16
// storage).
static __global__ void __launch_bounds__(BLOCK)
finalize_kernel(const double* partials, unsigned nb, DevScalars* scal, double eos_c,
                double inv_rho_ref, int one_warp) {
  __shared__ double sh[96];
  if (!one_warp)
    combine_partials_block<8>(partials, nb, scal, eos_c, inv_rho_ref, sh);
  else if (threadIdx.x < 32)
    combine_partials<8>(partials, nb, scal, 0, false, 0.0, eos_c, inv_rho_ref);
}

// ------------------------------------------------ runs of planes (3-D)
// Chunks of c planes (per tile) of the decreasing-size schedule that has
// reached plane zc: three quarters of what is left in the first class, the
// rest of it in the last (c <= 4).
__host__ __device__ inline int chunk_count(int nz, int zc, int c) {
  const int left = nz - zc;
  return c <= 4 ? (left + c - 1) / c : left * 3 / 4 / c;
}
__host__ __device__ inline int chunks_per_tile(int nz, int c) {
  int n = 0, zc = 0;
  for (;; c = c > 4 ? c / 2 : c) {
    const int k = chunk_count(nz, zc, c);
    n += k;
    zc += k * c;
    if (c <= 4) return n;
  }
}

// The run of planes of block b, which takes long chunks first and shorter ones
// last in launch order; chunk < 0: chunks of -chunk planes all along.
struct ZRun { int tile, z_begin, z_end; };
__device__ __forceinline__ ZRun z_run(int b, int tiles, int nz, int chunk) {
  if (chunk < 0) {
    const int z = b / tiles * -chunk;
    return {b % tiles, z, min(z - chunk, nz)};
  }
  int zc = 0, c = chunk;
#pragma unroll 1
  for (;; c = c > 4 ? c / 2 : c) {
    const int n = chunk_count(nz, zc, c);  // chunks of c planes per tile
    if (b < n * tiles || c <= 4) {
      zc += b / tiles * c;
      return {b % tiles, zc, min(zc + c, nz)};
    }
    b -= n * tiles;
    zc += n * c;
  }
}

// ------------------------------------------------------------ tiles
// A block owns TX x TY cells of a plane; a thread owns LN neighbouring cells
// in x (two in FP32 compute, one in FP64) in each of RPT rows.
//
// Two cells per thread in FP32: one cell per thread was bound by instruction
// issue, and a pair halves it -- packed f32x2 arithmetic, 64-bit shared-memory
// and global accesses, one set of addresses and parameter reads for two cells:
// 1,742 -> 847 warp instructions x 32 per cell of the 3-D bed.  Now bound by
// latency (10 to 16 warps per SM, a third of the issue slots used): 256 x 128 x
// 128 bed 394 -> 249 us a step, 1024 x 256 bed 17.5 -> 15.5, 48 channel beds 365
// -> 288.  FP64 is bound by the FP64 pipe; sharing te / to between opposite
// directions, the face sums and the reciprocals below took the 1001 x 251 bed
// from 410 to 320 us.
template <class Real> struct VecOf { using V = Real; };
template <> struct VecOf<float> { using V = float2; };

template <class V_, int TXv, int TYv, int RPTv = 1> struct Tile {
  using V = V_;
  static constexpr int LN = Lanes<V>::n;
  static constexpr int TX = TXv, TY = TYv;
  static constexpr int RPT = TX * TY / LN / RPTv > 256 ? TX * TY / LN / 256 : RPTv;
  static constexpr int NT = TX * TY / LN / RPT;  // threads
  static constexpr int TXT = TX / LN;            // threads per row
  // staged rows start LN cells left of the tile, so that a pair of cells is
  // an aligned 64-bit word of its row
  static constexpr int XO = LN;
  static constexpr int HX = TX + 2 * XO, HY = TY + 2, HP = HX * HY;
};

// ------------------------------------------------ staged tile (smem)
// Fields per staged cell: T, phi_s, rho, kappa_T = phi_f lambda, mu, f_D
// (diffusivity factor), Ts, phi_f rho f_D, then Y_k.
enum { F_T = 0, F_PHI, F_RHO, F_KT, F_MU, F_FD, F_TS, F_RF, F_Y0 };

// A pair / a cell of an array: `even` says that a pair is one aligned word
// (State::even), `two` that the second cell of the pair exists.
template <class V, class T>
__device__ __forceinline__ V load_cells(const T* __restrict__ p, bool even, bool two);
template <> __device__ __forceinline__ double load_cells<double, double>(const double* __restrict__ p, bool, bool) {
  return __ldg(p);
}
template <> __device__ __forceinline__ float load_cells<float, float>(const float* __restrict__ p, bool, bool) {
  return __ldg(p);
}
template <> __device__ __forceinline__ float2 load_cells<float2, float>(const float* __restrict__ p, bool even,
                                                                        bool two) {
  if (even) return __ldg(reinterpret_cast<const float2*>(p));
  return make_float2(__ldg(p), two ? __ldg(p + 1) : 0.f);
}
__device__ __forceinline__ void store_cells(double* p, double v, bool, bool) { *p = v; }
__device__ __forceinline__ void store_cells(float* p, float v, bool, bool) { *p = v; }
__device__ __forceinline__ void store_cells(float* p, float2 v, bool even, bool two) {
  if (even) {
    *reinterpret_cast<float2*>(p) = v;
  } else {
    p[0] = v.x;
    if (two) p[1] = v.y;
  }
}
// Values of the staged fields of one position (cell or pair) into the plane.
template <int K, class Real, class V, int HP>
__device__ __forceinline__ void stage_fields(const Params<Real, K>& P, Real* __restrict__ pl, int h,
                                             V T, V phis, V Ts, const V* Y, Real P0) {
  const V one = splat<V>(Real(1));
  const V phif = vsub(one, phis);
  const V invMw = mixture_invMw<Real, K, V>(P, Y);
  const V rho = fdiv(splat<V>(P0 * P.eos_cr), vmul(T, invMw));
  const V cp = mixture_cp<Real, K, V>(P, Y);
  V mu, lam;
  transport<Real, K, V>(P, T, Y, invMw, cp, mu, lam);
  V fD = one;
  if constexpr (K > 0) {
    if (P.D_Tdep) fD = fpow(vmuls<V>(P.inv_DTref, T), P.D_exp);
  }
  auto put = [&](int f, V v) { *reinterpret_cast<V*>(pl + f * HP + h) = v; };
  put(F_T, T);
  put(F_PHI, phis);
  put(F_RHO, rho);
  put(F_KT, vmul(phif, lam));
  put(F_MU, mu);
  put(F_FD, fD);
  put(F_TS, Ts);
  put(F_RF, vmul(vmul(phif, rho), fD));
#pragma unroll
  for (int k = 0; k < K; ++k) put(F_Y0 + k, Y[k]);
}

// Coordinate v of an axis of n cells: wrapped on periodic faces, else clamped.
__device__ __forceinline__ int wrap_or_clamp(int v, int n, bool per) {
  if (v < 0) v = per ? v + n : 0;
  if (v >= n) v = per ? v - n : n - 1;
  return v < 0 ? 0 : (v >= n ? n - 1 : v);  // tiles wider than n
}

// Stage plane z (may be -1 or nz: ghost plane) of the block's tile with its
// xy halo into `pl` ([fields][HP]).  Out-of-domain halo cells follow the ghost
// rules: periodic faces wrap; otherwise the adjacent cell's values, with the
// inlet state (T_in, Y_in) on the inlet face and the wall temperature on a
// wall that has one.
template <int DIM, int K, class Real, class T_>
__device__ __forceinline__ void stage_plane(const Params<Real, K>& P, const State<Real, Real>& S,
                                            Real* __restrict__ pl, int x0, int y0, int z, Real P0) {
  using V = typename T_::V;
  constexpr int LN = T_::LN, HP = T_::HP, PW = T_::HX / LN;
  constexpr int KK = Params<Real, K>::KK;
  // tiles whose halo lies inside the lattice need no ghost rules
  const bool inner = x0 >= LN && y0 >= 1 && x0 + T_::TX + LN <= P.nx && y0 + T_::TY < P.ny &&
                     (DIM == 2 || (z >= 0 && z < P.nz));
  const bool even = LN == 1 || S.even;
  struct Raw { V T, phis, Ts, Y[KK]; };
  auto load = [&](int p, Raw& R) {
    V &T = R.T, &phis = R.phis, &Ts = R.Ts, *Y = R.Y;
    const int hy = p / PW, hx = (p - hy * PW) * LN;
    const int x = x0 - LN + hx, y = y0 - 1 + hy;
    // source columns of the position's cells, start of the source row
    int xa = x, xb = x + 1, row = P.nx * (y + P.ny * z);
    if (!inner) {
      const bool per0 = P.bc[0] == BC_PERIODIC;
      xa = wrap_or_clamp(x, P.nx, per0);
      xb = wrap_or_clamp(x + 1, P.nx, per0);
      const int yc = wrap_or_clamp(y, P.ny, P.bc[2] == BC_PERIODIC);
      const int zc = DIM == 3 ? wrap_or_clamp(z, P.nz, P.bc[4] == BC_PERIODIC) : 0;
      row = P.nx * (yc + P.ny * zc);
    }
    if (LN == 1 || (even && xb == xa + 1 && (xa & 1) == 0)) {
      const int c = row + xa;
      T = load_cells<V>(S.T_in + c, true, true);
      phis = load_cells<V>(S.phi + c, true, true);
      Ts = P.Ts_field ? load_cells<V>(S.Ts_in + c, true, true) : splat<V>(P.Ts_uniform);
#pragma unroll
      for (int k = 0; k < K; ++k) Y[k] = load_cells<V>(S.Y_in + (size_t)k * P.N + c, true, true);
    } else {
      const int ca = row + xa, cb = row + xb;
      auto two = [&](const Real* b) {
        V v;
        set_lane(v, 0, __ldg(b + ca));
        set_lane(v, LN - 1, __ldg(b + cb));
        return v;
      };
      T = two(S.T_in);
      phis = two(S.phi);
      Ts = P.Ts_field ? two(S.Ts_in) : splat<V>(P.Ts_uniform);
#pragma unroll
      for (int k = 0; k < K; ++k) Y[k] = two(S.Y_in + (size_t)k * P.N);
    }
    if (!inner) {
      // one step outside exactly one non-periodic face: the face's ghost state
      const int fy = y < 0 ? 2 : (y >= P.ny ? 3 : -1);
      const int fz = DIM == 3 ? (z < 0 ? 4 : (z >= P.nz ? 5 : -1)) : -1;
      const bool gy = fy >= 0 && P.bc[fy] != BC_PERIODIC, gz = fz >= 0 && P.bc[fz] != BC_PERIODIC;
#pragma unroll
      for (int l = 0; l < LN; ++l) {
        const int fx = x + l < 0 ? 0 : (x + l >= P.nx ? 1 : -1);
        const bool gx = fx >= 0 && P.bc[fx] != BC_PERIODIC;
        if ((gx ? 1 : 0) + (gy ? 1 : 0) + (gz ? 1 : 0) != 1) continue;
        const int face = gx ? fx : (gy ? fy : fz);
        const int bc = P.bc[face];
        if (bc == BC_INLET) {
          set_lane(T, l, P.T_in);
#pragma unroll
          for (int k = 0; k < K; ++k) set_lane(Y[k], l, P.Y_in[k]);
        } else if (bc == BC_WALL && P.wall_T[face] > Real(0)) {
          set_lane(T, l, P.wall_T[face]);
        }
      }
    }
  };
  auto finish = [&](int p, const Raw& R) {
    const int hy = p / PW, hx = (p - hy * PW) * LN;
    stage_fields<K, Real, V, HP>(P, pl, hy * T_::HX + hx, R.T, R.phis, R.Ts, R.Y, P0);
  };
  if constexpr (DIM == 2 && K == 0) {
    // two positions' loads in flight (with species their registers spill)
    for (int p = threadIdx.x; p < PW * T_::HY; p += 2 * T_::NT) {
      Raw a, b;
      const bool second = p + T_::NT < PW * T_::HY;
      load(p, a);
      if (second) load(p + T_::NT, b);
      finish(p, a);
      if (second) finish(p + T_::NT, b);
    }
  } else {
    for (int p = threadIdx.x; p < PW * T_::HY; p += T_::NT) {
      Raw a;
      load(p, a);
      finish(p, a);
    }
  }
}

// Asynchronous copy of a cell or pair to shared memory, and the wait of the
// issuing thread for all of its own.
template <class V, class T>
__device__ __forceinline__ void cp_async_cells(T* dst, const T* src, bool even, bool two) {
  const unsigned d = static_cast<unsigned>(__cvta_generic_to_shared(dst));
  if (sizeof(V) == 8 && (sizeof(T) == 8 || even)) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(d), "l"(src) : "memory");
  } else {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(d), "l"(src) : "memory");
    if (two)
      asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(d + 4), "l"(src + 1) : "memory");
  }
}
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_all;" ::: "memory");
}

// Accessor of the update over the staged planes: own and neighbour values (a
// neighbour of a pair in x is half of the pair itself and one more cell).
template <class Real, class T_>
struct PlaneAcc {
  using V = typename T_::V;
  static constexpr int HP = T_::HP;
  const Real* __restrict__ cen;
  const Real* __restrict__ zm;
  const Real* __restrict__ zp;
  int h;
  const Real* src;  // this thread's chemistry increments in shared memory, or null
  __device__ __forceinline__ V c(int f) const {
    return *reinterpret_cast<const V*>(cen + f * HP + h);
  }
  __device__ __forceinline__ bool has_src() const { return src != nullptr; }
  __device__ __forceinline__ V increment(int k) const {
    return *reinterpret_cast<const V*>(src + k * T_::TX * T_::TY);
  }
  __device__ __forceinline__ V n(int f, int a, int s, V own) const {
    if (a == 0) {
      const Real v = cen[f * HP + h + (s < 0 ? -1 : T_::LN)];
      if constexpr (T_::LN == 1) return v;
      else return s < 0 ? make_float2(v, own.x) : make_float2(own.y, v);
    }
    if (a == 1) return *reinterpret_cast<const V*>(cen + f * HP + h + s * T_::HX);
    return *reinterpret_cast<const V*>((s < 0 ? zm : zp) + f * HP + h);
  }
};

// ------------------------------------------------------------ streaming
// Faces that a cell lies on and that are not periodic.
struct Faces {
  bool f[6];
  __device__ __forceinline__ bool any() const {
    return f[0] || f[1] || f[2] || f[3] || f[4] || f[5];
  }
};
template <int DIM, class Real, int K>
__device__ __forceinline__ Faces faces_of(const Params<Real, K>& P, int x, int y, int z) {
  Faces e;
  e.f[0] = x == 0 && P.bc[0] != BC_PERIODIC;
  e.f[1] = x == P.nx - 1 && P.bc[1] != BC_PERIODIC;
  e.f[2] = y == 0 && P.bc[2] != BC_PERIODIC;
  e.f[3] = y == P.ny - 1 && P.bc[3] != BC_PERIODIC;
  e.f[4] = DIM == 3 && z == 0 && P.bc[4] != BC_PERIODIC;
  e.f[5] = DIM == 3 && z == P.nz - 1 && P.bc[5] != BC_PERIODIC;
  return e;
}
// Populations that stream into the cell(s) starting at x: the upstream
// neighbour coordinate wraps across a periodic face and is clamped to the
// cell across any other face (the boundary rules then replace those values).
// Along x a pair reads columns x-1, x (directions to +x), x, x+1 (an aligned
// pair when rows are even) and x+1, x+2 (directions to -x).
template <int DIM, int K, class Real, class V>
__device__ __forceinline__ void load_pops(const Params<Real, K>& P, const State<Real, Real>& S,
                                          int x, int y, int z, V* __restrict__ out) {
  using L = Lattice<DIM>;
  constexpr int LN = Lanes<V>::n;
  const bool per0 = P.bc[0] == BC_PERIODIC, per2 = P.bc[2] == BC_PERIODIC,
             per4 = P.bc[4] == BC_PERIODIC;
  const int xm = x > 0 ? x - 1 : (per0 ? P.nx - 1 : x);
  const int x1 = x + 1 < P.nx ? x + 1 : (per0 ? 0 : x);
  const int x2 = x + 2 < P.nx ? x + 2 : (per0 ? x + 2 - P.nx : x1);
  const int ym = y > 0 ? y - 1 : (per2 ? P.ny - 1 : y);
  const int yp = y < P.ny - 1 ? y + 1 : (per2 ? 0 : y);
  int zz[3] = {0, 0, 0};
  if (DIM == 3) {
    zz[0] = z > 0 ? z - 1 : (per4 ? P.nz - 1 : z);
    zz[1] = z;
    zz[2] = z < P.nz - 1 ? z + 1 : (per4 ? 0 : z);
  }
  int row[3][3];  // [1 + dz][1 + dy]: start of the row
#pragma unroll
  for (int b = 0; b < 3; ++b) {
    if (DIM == 2 && b != 1) continue;
    row[b][0] = P.nx * (ym + P.ny * zz[b]);
    row[b][1] = P.nx * (y + P.ny * zz[b]);
    row[b][2] = P.nx * (yp + P.ny * zz[b]);
  }
  const bool even = S.even;
#pragma unroll
  for (int i = 0; i < L::Q; ++i) {
    const int cx = L::c(i, 0), r = row[DIM == 3 ? 1 - L::c(i, 2) : 1][1 - L::c(i, 1)];
    const Real* g = S.g_in + (size_t)i * P.N;
    if constexpr (LN == 1) {
      out[i] = __ldg(g + (r + (cx > 0 ? xm : (cx < 0 ? x1 : x))));
    } else if (cx == 0 && even) {
      out[i] = __ldg(reinterpret_cast<const float2*>(g + (r + x)));
    } else {
      out[i].x = __ldg(g + (r + (cx > 0 ? xm : (cx < 0 ? x1 : x))));
      out[i].y = __ldg(g + (r + (cx > 0 ? x : (cx < 0 ? x2 : x1))));
    }
  }
}

// ------------------------------------------------------ the fused step
// Where a thread's cell or pair lies: lattice index of the first cell, the
// coordinates, whether pairs are aligned words, whether a second cell exists.
struct CellPos {
  int c, x, y, z;
  bool even, two;
};

// Per cell: (a1) pull + moments + implicit drag, (c) reaction source,
// (b) FD transport of Y_k, T, Ts, low-Mach divergence, (a) source + BGK
// collision + store, (d) contribution to the FP64 reduction (returned per
// cell; fluxes through the inlet / outlet face in fin, fout; the fuel consumed is
// added to `fuel` with the inlet feedback).  `gin` holds the
// streamed populations (load_pops) and is overwritten.
template <int DIM, int K, class Real, class V, class Acc>
__device__ __forceinline__ V cell_update(const Params<Real, K>& P, const State<Real, Real>& S,
                                         const Acc& A, V* __restrict__ gin, const CellPos q,
                                         Real P0, Real dlnP0, Real dP0r, Real& fin, Real& fout,
                                         double& fuel) {
  using L = Lattice<DIM>;
  constexpr int Q = L::Q;
  constexpr int KK = Params<Real, K>::KK;
  constexpr int LN = Lanes<V>::n;
  constexpr Real CS2 = Real(1) / Real(3);
  using Mask = typename Lanes<V>::M;
  const V zero = splat<V>(Real(0)), one = splat<V>(Real(1));

  const V T0 = A.c(F_T), phis = A.c(F_PHI), rho = A.c(F_RHO), mu = A.c(F_MU);
  const V phif = vsub(one, phis);
  const V Kd = vmul(vmul(vmuls<V>(P.Au_eta2, mu), phif), vmul(phis, phis));

  // (a1) boundary rules of the streamed populations
  const V inv_rk = vrcp(vfmas<V>(Real(0.5), Kd, rho));
  const int xl = q.x + (LN == 2 && q.two ? 1 : 0);  // last cell
  const Faces e0 = faces_of<DIM>(P, q.x, q.y, q.z);
  const Faces e1 = faces_of<DIM>(P, xl, q.y, q.z);
  if (e0.any() || e1.any()) {
    Real rho_in = 0;
    if (P.bc[0] == BC_INLET) {
      Real Yin[KK];
#pragma unroll
      for (int k = 0; k < K; ++k) Yin[k] = P.Y_in[k];
      rho_in = fdiv(P0 * P.eos_cr, vmul(P.T_in, mixture_invMw<Real, K, Real>(P, Yin)));
    }
#pragma unroll
    for (int l = 0; l < LN; ++l) {
      if (l == 1 && !q.two) break;
      const int xyz[3] = {q.x + l, q.y, q.z};
      const Faces& e = l == 0 ? e0 : e1;
      if (!e.any()) continue;
      Real gl[Q], uw[3] = {0, 0, 0};
#pragma unroll
      for (int i = 0; i < Q; ++i) gl[i] = get_lane(gin[i], l);
      const GlobalMom<Real> gm{S.M_in, P.N};
      edge_rules<DIM>(P, S, q.c + l, xyz, get_lane(rho, l), rho_in, uw, gl, gm);
      if (e.f[1] && P.bc[1] == BC_OUTLET) {
        // the outlet rule again with the cell's own first-pass velocity
#pragma unroll
        for (int a = 0; a < DIM; ++a) {
          Real m = 0;
#pragma unroll
          for (int i = 0; i < Q; ++i) {
            if (L::c(i, a) > 0) m = vadd(m, gl[i]);
            if (L::c(i, a) < 0) m = vsub(m, gl[i]);
          }
          const Real d = vfma(get_lane(Kd, l), P.u_s[a], P.Fb[a]);
          uw[a] = vmul(vfma(Real(3), m, vmul(Real(0.5), d)), get_lane(inv_rk, l));
        }
        edge_rules<DIM>(P, S, q.c + l, xyz, get_lane(rho, l), rho_in, uw, gl, gm);
      }
#pragma unroll
      for (int i = 0; i < Q; ++i) set_lane(gin[i], l, gl[i]);
    }
  }
  // moments from the sums and differences of opposite populations
  V sg = gin[0], mraw[3] = {zero, zero, zero}, u[3] = {zero, zero, zero};
#pragma unroll
  for (int i = 1; i < Q; ++i) {
    const int j = L::opp(i);
    if (j < i) continue;
    const V d = vsub(gin[i], gin[j]);
    sg = vadd(sg, vadd(gin[i], gin[j]));
#pragma unroll
    for (int a = 0; a < DIM; ++a) {
      if (L::c(i, a) > 0) mraw[a] = i == 1 + (DIM == 2 ? a : 2 * a) ? d : vadd(mraw[a], d);
      if (L::c(i, a) < 0) mraw[a] = vsub(mraw[a], d);
    }
  }
#pragma unroll
  for (int a = 0; a < DIM; ++a) {
    const V d = vfmas<V>(P.u_s[a], Kd, splat<V>(P.Fb[a]));
    u[a] = vmul(vfmas<V>(Real(3), mraw[a], vmuls<V>(Real(0.5), d)), inv_rk);
  }

  const V Ts0 = A.c(F_TS), kc = A.c(F_KT), rf0 = A.c(F_RF);
  V Y0[KK];
#pragma unroll
  for (int k = 0; k < K; ++k) Y0[k] = A.c(F_Y0 + k);
  const V invMw = mixture_invMw<Real, K, V>(P, Y0);
  const V cp = mixture_cp<Real, K, V>(P, Y0);
  const V invT = vrcp(T0);
  const Mask fluid = vge(phif, splat<V>(P.phi_min));
  const Mask solid = vge(phis, splat<V>(P.phi_min));
  // exchange with the solid; kappa_T = phi_f lambda
  V SI = vmul(vmul(vmuls<V>(P.AT_eta2, kc), vmul(phis, phis)), vsub(Ts0, T0));
  SI = vsel(fluid, SI, zero);
  if (P.Ts_field) SI = vsel(solid, SI, zero);

  // (c) reaction source
  V om[KK], omT = zero;
#pragma unroll
  for (int k = 0; k < KK; ++k) om[k] = zero;
  if constexpr (K > 0) {
    if (P.chem == 1) rates<Real, K, V>(P, T0, Y0, rho, invT, om, omT);
    if (P.chem >= 2) {
      // increments of the chemistry pre-pass (implicit integrator or surrogate)
      if (A.has_src()) {
        cp_async_wait();
#pragma unroll
        for (int k = 0; k < K; ++k) om[k] = A.increment(k);
        omT = A.increment(K);
      } else {
#pragma unroll
        for (int k = 0; k < K; ++k)
          om[k] = load_cells<V>(S.src + (size_t)k * P.N + q.c, q.even, q.two);
        omT = load_cells<V>(S.src + (size_t)K * P.N + q.c, q.even, q.two);
      }
    }
  }

  if constexpr (K > 0) {
    if (P.feed) {
#pragma unroll
      for (int l = 0; l < LN; ++l) {
        if ((l == 1 && !q.two) || !(get_lane(phif, l) >= P.phi_min)) continue;
        Real w = 0;
#pragma unroll
        for (int k = 0; k < K; ++k)
          if (k == P.feed_k) w = get_lane(om[k], l);
        fuel += double(vmul(get_lane(phif, l), -w));
      }
    }
  }

  // 1 / (phi_f rho) and 1 / (phi_f rho cp), zero in frozen cells; the negated
  // velocity of the convection terms is zero there too, so that frozen cells
  // change nothing
  const V irc = vsel(fluid, vrcp(vmul(vmul(phif, rho), cp)), zero);
  const V iphr = vmul(irc, cp);
  V un[DIM];
  Mask up[DIM];
#pragma unroll
  for (int a = 0; a < DIM; ++a) {
    un[a] = vsel(fluid, vneg(u[a]), zero);
    up[a] = vgt(u[a], zero);
  }

  // (b) species; the face factors (phi_f rho f_D summed over the face; their
  // 1/2 sits in D_k) are shared by every species, and the central differences
  // of Y_k feed the enthalpy-flux cross term of the temperature equation and,
  // weighted with 1/M_k, the divergence
  V Yn[KK];
  V sYm = zero;     // sum_k (1/M_k) (dY_k + u.grad Y_k)
  V sx[DIM];        // sum_k cp_k D_k (Y_k(+) - Y_k(-)) per axis
#pragma unroll
  for (int a = 0; a < DIM; ++a) sx[a] = zero;
  if constexpr (K > 0) {
    V fm[DIM], fp[DIM], sI[DIM];
#pragma unroll
    for (int a = 0; a < DIM; ++a) {
      fm[a] = vneg(vadd(rf0, A.n(F_RF, a, -1, rf0)));
      fp[a] = vadd(rf0, A.n(F_RF, a, +1, rf0));
      sI[a] = zero;
    }
#pragma unroll
    for (int k = 0; k < K; ++k) {
      V adv = zero, dif = zero;
#pragma unroll
      for (int a = 0; a < DIM; ++a) {
        const V dm = vsub(Y0[k], A.n(F_Y0 + k, a, -1, Y0[k]));
        const V dp = vsub(A.n(F_Y0 + k, a, +1, Y0[k]), Y0[k]);
        const V sd = vadd(dp, dm);
        adv = vfma(un[a], vsel(up[a], dm, dp), adv);
        dif = vfma(fp[a], dp, dif);
        dif = vfma(fm[a], dm, dif);
        sI[a] = vfmas<V>(P.invM[k], sd, sI[a]);
        sx[a] = vfmas<V>(P.cpD[k], sd, sx[a]);
      }
      const V dY = vfma(iphr, vfmas<V>(P.Dlat_h[k], dif, vmul(phif, om[k])), adv);
      Yn[k] = vadd(Y0[k], dY);
      sYm = vfmas<V>(P.invM[k], dY, sYm);
    }
    V cen = zero;
#pragma unroll
    for (int a = 0; a < DIM; ++a) cen = vfma(un[a], sI[a], cen);
    sYm = vfmas<V>(Real(-0.5), cen, sYm);
  }

  // (b) temperature
  V Tn, dTm;
  {
    const V fD = A.c(F_FD);
    V adv = zero, dif = zero, cross = zero, cen = zero;
#pragma unroll
    for (int a = 0; a < DIM; ++a) {
      const V dm = vsub(T0, A.n(F_T, a, -1, T0)), dp = vsub(A.n(F_T, a, +1, T0), T0);
      const V sd = vadd(dp, dm);
      adv = vfma(un[a], vsel(up[a], dm, dp), adv);
      cen = vfma(un[a], sd, cen);
      dif = vfma(vadd(kc, A.n(F_KT, a, +1, kc)), dp, dif);
      dif = vfma(vneg(vadd(kc, A.n(F_KT, a, -1, kc))), dm, dif);
      if constexpr (K > 0) cross = vfma(sx[a], sd, cross);
    }
    V src = vadd(vadds<V>(dP0r, omT), SI);
    if constexpr (K > 0) src = vfma(vmul(rho, fD), vmuls<V>(Real(0.25), cross), src);
    const V dTn = vfma(irc, vfmas<V>(Real(0.5), dif, vmul(phif, src)), adv);
    // frozen cells take the solid temperature
    Tn = vsel(fluid, vadd(T0, dTn), Ts0);
    dTm = vsel(fluid, vfmas<V>(Real(-0.5), cen, dTn), vsub(Ts0, T0));  // plus u.grad T (central)
  }

  // solid temperature
  if (P.Ts_field) {
    V Tsn = Ts0;
    if (vany(solid)) {
      V dif = zero;
#pragma unroll
      for (int a = 0; a < DIM; ++a) {
        const V sm = vsub(Ts0, A.n(F_TS, a, -1, Ts0)), sp = vsub(A.n(F_TS, a, +1, Ts0), Ts0);
        dif = vfma(vadd(phis, A.n(F_PHI, a, +1, phis)), sp, dif);
        dif = vfma(vneg(vadd(phis, A.n(F_PHI, a, -1, phis))), sm, dif);
      }
      const V num = vfma(vneg(phif), SI, vmuls<V>(P.Lams_h, dif));
      V dTs = fdiv(num, vmuls<V>(P.Cs, phis));
      if (P.moving) {
        // a moving solid carries its temperature with u_s (upwind)
#pragma unroll
        for (int a = 0; a < DIM; ++a) {
          const Real us = P.u_s[a];
          if (us > Real(0)) dTs = vfmas<V>(-us, vsub(Ts0, A.n(F_TS, a, -1, Ts0)), dTs);
          else if (us < Real(0)) dTs = vfmas<V>(-us, vsub(A.n(F_TS, a, +1, Ts0), Ts0), dTs);
        }
      }
      Tsn = vsel(solid, vadd(Ts0, dTs), Ts0);
    }
    store_cells(S.Ts_out + q.c, Tsn, q.even, q.two);
  }

  // low-Mach divergence: continuity with the EOS at uniform P0,
  // D = (1/T) DT/Dt + Mw sum_k (1/M_k) DY_k/Dt - (1/P0) dP0/dt, the material
  // increments taken as the step's increments plus u.grad with central
  // differences, the gradient the source takes of rho (with the upwind
  // gradient the discrete continuity would keep a first-order mass defect)
  V D = vfma(dTm, invT, splat<V>(-dlnP0));
  if constexpr (K > 0) D = vadd(D, fdiv(sYm, invMw));

  // (a) source and BGK collision: omega = 1/tau = 2 rho / (rho + 6 mu)
  V G[DIM], F[DIM];
  V uG = zero;
#pragma unroll
  for (int a = 0; a < DIM; ++a) {
    G[a] = vmuls<V>(CS2 * Real(0.5), vsub(A.n(F_RHO, a, +1, rho), A.n(F_RHO, a, -1, rho)));
    F[a] = vfma(vneg(Kd), vadds<V>(-P.u_s[a], u[a]), splat<V>(P.Fb[a]));
    uG = vfma(u[a], G[a], uG);
  }
  // P_h: the pulled zeroth moment plus half the zeroth moment of the source,
  // sum_i Xi_i = u.G + rho cs^2 D, so that a step adds the whole source
  const V rho3 = vmuls<V>(CS2, rho);
  const V Ph = vfmas<V>(Real(0.5), vfma(rho3, D, uG), sg);
  if (P.nscbc && xl >= P.nx - 2) {
    // the two outlet columns of this step for the characteristic outlet
    const int NF = P.ny * P.nz, f = q.y + P.ny * q.z;
#pragma unroll
    for (int l = 0; l < LN; ++l) {
      if (l == 1 && !q.two) break;
      if (q.x + l < P.nx - 2) continue;
      const int col = q.x + l == P.nx - 1 ? 0 : 1;
      S.ob[(size_t)(2 * col) * NF + f] = get_lane(Ph, l);
      S.ob[(size_t)(2 * col + 1) * NF + f] = get_lane(u[0], l);
      if (col == 0) S.ob[(size_t)4 * NF + f] = get_lane(rho, l);
    }
  }
  const V omega = fdiv(vmuls<V>(Real(2), rho), vfmas<V>(Real(6), mu, rho));
  const V src_w = vfmas<V>(Real(-0.5), omega, one);
  const V keep = vsub(one, omega);
  // f_eq / rho - w = w e with e = 3 cu + 9/2 cu^2 - 3/2 uu;
  // g_eq = cs2 f_eq + w (P_h - rho cs2) = w (P_h + rho e / 3);
  // Xi = w [(c - u).(G e + F (1 + e)) + rho cs2 D] = w [(c.H - u.H) e + c.F - u.F + rho cs2 D]
  // with H = G + F.  Split into the parts even and odd in c, e = E + O:
  //   g* = keep g + w (te + to),  O = 3 cu,  E = O^2 / 2 - 3/2 uu,
  //   te = A0 + B E + c.Hs O,  to = B O + c.Hs E + c.Fs,
  // with s = 1 - omega / 2, Hs = s H, Fs = s F, B = omega rho cs2 - s u.H and
  // A0 = omega P_h + s (rho cs2 D - u.F); a direction and its opposite share
  // te and to.
  V u3[DIM], Hs[DIM], Fs[DIM];
  V uu = zero, uHs = zero, uFs = zero;
#pragma unroll
  for (int a = 0; a < DIM; ++a) {
    Fs[a] = vmul(src_w, F[a]);
    Hs[a] = vfma(src_w, G[a], Fs[a]);
    u3[a] = vmuls<V>(Real(3), u[a]);
    uu = vfma(u[a], u[a], uu);
    uHs = vfma(u[a], Hs[a], uHs);
    uFs = vfma(u[a], Fs[a], uFs);
  }
  const V uu15 = vmuls<V>(Real(-1.5), uu);
  const V or3 = vmul(omega, rho3);
  const V B = vsub(or3, uHs);
  V A0 = vfma(omega, Ph, vmul(src_w, vmul(rho3, D)));
  A0 = vsub(A0, uFs);
  gin[0] = vfma(keep, gin[0], vmuls<V>(Real(L::w(0)), vfma(uu15, B, A0)));
#pragma unroll
  for (int i = 1; i < Q; ++i) {
    const int j = L::opp(i);
    if (j < i) continue;  // done with its opposite
    V O = zero, cH = zero, cF = zero;
    bool first = true;
#pragma unroll
    for (int a = 0; a < DIM; ++a) {
      if (L::c(i, a) == 0) continue;
      if (first) {  // the first direction of a pair starts with +1
        O = u3[a];
        cH = Hs[a];
        cF = Fs[a];
        if (L::c(i, a) < 0) { O = vneg(O); cH = vneg(cH); cF = vneg(cF); }
        first = false;
      } else if (L::c(i, a) > 0) {
        O = vadd(O, u3[a]);
        cH = vadd(cH, Hs[a]);
        cF = vadd(cF, Fs[a]);
      } else {
        O = vsub(O, u3[a]);
        cH = vsub(cH, Hs[a]);
        cF = vsub(cF, Fs[a]);
      }
    }
    const V E = vfma(vmuls<V>(Real(0.5), O), O, uu15);
    const V te = vfma(E, B, vfma(cH, O, A0));
    const V to = vfma(O, B, vfma(cH, E, cF));
    const V p = vmuls<V>(Real(L::w(i)), te);
    const V gi = vfma(keep, gin[i], vfmas<V>(Real(L::w(i)), to, p));
    const V gj = vfma(keep, gin[j], vfmas<V>(Real(-L::w(i)), to, p));
    gin[i] = gi;
    gin[j] = gj;
  }
#pragma unroll
  for (int i = 0; i < Q; ++i)
    store_cells(S.g_out + (size_t)i * P.N + q.c, gin[i], q.even, q.two);
  store_cells(S.T_out + q.c, Tn, q.even, q.two);
#pragma unroll
  for (int k = 0; k < K; ++k) store_cells(S.Y_out + (size_t)k * P.N + q.c, Yn[k], q.even, q.two);

  // (d) contributions to the reduction
  fin = fout = Real(0);
  if (q.x == 0 && P.bc[0] == BC_INLET)
    fin = get_lane(phif, 0) * get_lane(rho, 0) * get_lane(u[0], 0);
  if (xl == P.nx - 1 && P.bc[1] == BC_OUTLET) {
    const int l = LN == 2 && q.two ? 1 : 0;
    fout = get_lane(phif, l) * get_lane(rho, l) * get_lane(u[0], l);
  }
  // 0 * P_h is NaN when any pulled population is: a NaN confined to the
  // populations reaches the FP64 reduction (and the status word) this step
  V r = vfma(zero, Ph, vmul(phif, vrcp(vmul(Tn, mixture_invMw<Real, K, V>(P, Yn)))));
  if (LN == 2 && !q.two) set_lane(r, 1, Real(0));
  return r;
}

// Resident threads per SM asked of the register allocator in 2-D.  FP32 pairs
// wait on latency, so more resident blocks pay until they spill: without
// species 64 registers (1024 threads; 48 beds: 359 us a step at 512 threads,
// 288 at 1024), with species 128 (512 threads; the 1024 x 256 bed: 15.5 us, 16.6
// at 640, 17.6 at 768).  FP64 is bound by the FP64 pipe: 128 registers.
template <int K, class T_> struct MinBlocks {
  static constexpr int value = (T_::LN == 2 && K == 0 ? 1024 : 512) / T_::NT;
};

// One 2-D tile of the fused step (tile (bx, by)): stages the tile in `pl`
// (shared memory), updates its cells and returns the block sums of the
// reduction in thread 0 (I, inlet flux, outlet flux).  Every thread of the
// block calls it.  The population loads of the thread's cells are issued
// before the staging, so the two load phases overlap.
template <int K, class Real, class T_>
__device__ __forceinline__ void step_tile(const Params<Real, K>& P, const State<Real, Real>& S,
                                          int bx, int by, Real* pl, double* red_sh, double& sI,
                                          double& sIn, double& sOut, double& sF) {
  using V = typename T_::V;
  constexpr int Q = Lattice<2>::Q, LN = T_::LN, RPT = T_::RPT, RS = T_::TY / RPT;
  const Real P0 = scal_P0<Real>(S.scal);
  const Real dlnP0 = scal_dlnP0<Real>(S.scal);
  const Real dP0r = scal_dP0r<Real>(S.scal);
  const int tx = (threadIdx.x % T_::TXT) * LN, ty = threadIdx.x / T_::TXT;
  const int x0 = bx * T_::TX, y0 = by * T_::TY;
  const int x = x0 + tx;
  const bool flux_block = (x0 == 0 && P.bc[0] == BC_INLET) ||
                          (x0 + T_::TX >= P.nx && P.bc[1] == BC_OUTLET);
  const bool even = LN == 1 || S.even;
  V accI = splat<V>(Real(0));
  Real accIn = 0, accOut = 0;
  double fuel = 0.0;
  V g[RPT][Q];
#pragma unroll
  for (int r = 0; r < RPT; ++r)
    if (x < P.nx && y0 + ty + r * RS < P.ny)
      load_pops<2, K, Real, V>(P, S, x, y0 + ty + r * RS, 0, g[r]);
  // the cell's chemistry increments travel to shared memory meanwhile: loaded
  // where the update uses them, they held up its 16 warps per SM (2048 x 512
  // cells with six species: 81 us a step, 65 so)
  Real* src = nullptr;
  if constexpr (K > 0) {
    if (P.chem >= 2) {
      src = pl + (F_Y0 + K) * T_::HP + threadIdx.x * LN;
#pragma unroll
      for (int r = 0; r < RPT; ++r) {
        const int yr = y0 + ty + r * RS;
        if (x < P.nx && yr < P.ny)
#pragma unroll
          for (int k = 0; k <= K; ++k)
            cp_async_cells<V>(src + k * T_::TX * T_::TY + r * T_::NT * LN,
                              S.src + (size_t)k * P.N + x + P.nx * yr, even, x + 1 < P.nx);
      }
    }
  }
  stage_plane<2, K, Real, T_>(P, S, pl, x0, y0, 0, P0);
  __syncthreads();
#pragma unroll
  for (int r = 0; r < RPT; ++r) {
    const int yr = y0 + ty + r * RS;
    if (x < P.nx && yr < P.ny) {
      const CellPos q{x + P.nx * yr, x, yr, 0, even, x + 1 < P.nx};
      const PlaneAcc<Real, T_> A{pl, nullptr, nullptr,
                                 (ty + r * RS + 1) * T_::HX + tx + T_::XO,
                                 src ? src + r * T_::NT * LN : nullptr};
      Real fi, fo;
      accI = vadd(accI, cell_update<2, K, Real, V>(P, S, A, g[r], q, P0, dlnP0, dP0r, fi, fo,
                                                     fuel));
      accIn += fi;
      accOut += fo;
    }
  }
  // (d) block partials in FP64 (one barrier)
  block_sum4(accI, accIn, accOut, flux_block, fuel, K > 0 && P.feed, red_sh, sI, sIn, sOut, sF);
}

template <int DIM, int K, class Real, class T_>
constexpr size_t step_smem_bytes() {
  return sizeof(Real) * ((F_Y0 + K) * T_::HP * (DIM == 3 ? 3 : 1) +
                         (DIM == 2 && K > 0 ? (K + 1) * T_::TX * T_::TY : 0));
}

// The previous step's deferred partials (fixed P0 only) are combined by the first
// block, which with `lead` = 1 does nothing else: the launch then has one block
// more than tiles, and no tile waits for the combine.  FP32: always so (in front of
// its tile the combine made steps of up to 608 tiles, one wave, 2 to 4 us longer:
// a 128 x 64 channel 10.9 us, 7.7 so; 400 x 200 bed 12.9, 10.0; several waves
// equal); without species at compile time, as both forms in one kernel spill.
// FP64: while an SM is left for it (a 128 x 64 channel 19.0 us a step, 18.0 so);
// beyond, it moves tiles among the SMs, which the FP64 pipe bounds (400 x 160 bed, 260 tiles:
// 97.7 us with the combine in front of the first tile, 102.4 in a block of its own).
template <int K, class Real>
__host__ __device__ constexpr bool always_lead() { return K == 0 && sizeof(Real) == 4; }

template <int K, class Real, class T_>
__global__ void __launch_bounds__(T_::NT, (MinBlocks<K, T_>::value))
step_kernel(const __grid_constant__ Params<Real, K> P, const State<Real, Real> S, int p0_closed,
            const double* __restrict__ prev_partials, unsigned prev_nb, int lead) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  Real* pl = reinterpret_cast<Real*>(smem_raw);
  __shared__ double red_sh[128];
  constexpr int F = slots_in_flight(K);

  int b = blockIdx.x, nb = gridDim.x;
  if (prev_partials) {
    constexpr int CF = always_lead<K, Real>() ? F : 8;
    if (b == 0) {
      combine_partials_block<CF>(prev_partials, prev_nb, S.scal, P.eos_c, P.inv_rho_ref, red_sh);
      if (always_lead<K, Real>() || lead) return;
    }
    const int off = always_lead<K, Real>() ? 1 : lead;
    b -= off;
    nb -= off;
  }
  const int gx = (P.nx + T_::TX - 1) / T_::TX;
  double sI, sIn, sOut, sF;
  step_tile<K, Real, T_>(P, S, b % gx, b / gx, pl, red_sh, sI, sIn, sOut, sF);
  // deterministic finish by the last block (closed P0, inlet feedback) or
  // deferred
  publish_partials_at<F>(sI, sIn, sOut, S.partials, S.counter, S.scal, p0_closed, false, 0.0,
                         P.eos_c, P.inv_rho_ref, (unsigned)b, (unsigned)nb,
                         p0_closed || (K > 0 && P.feed), sF, K > 0 && P.feed ? P.feed_c : 0.0);
}

// Persistent variant of the 2-D step: one grid of resident blocks walks the
// tiles, handed out by an atomic counter (one per step parity; each launch
// clears the other one for the next step), so no block waits for a second
// wave and cheap tiles do not leave SMs idle.  Reduction slots are the tile
// indices, as in step_kernel.
template <int K, class Real, class T_>
__global__ void __launch_bounds__(T_::NT, (MinBlocks<K, T_>::value))
step_persistent_kernel(const __grid_constant__ Params<Real, K> P, const State<Real, Real> S,
                       int p0_closed, const double* __restrict__ prev_partials, unsigned prev_nb,
                       unsigned* __restrict__ tile_ctr, int parity) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  Real* pl = reinterpret_cast<Real*>(smem_raw);
  __shared__ double red_sh[128];
  __shared__ int next_sh[2];

  if (prev_partials && blockIdx.x == 0)
    combine_partials_block<slots_in_flight(K)>(prev_partials, prev_nb, S.scal, P.eos_c,
                                               P.inv_rho_ref, red_sh);

  const int nbx = (P.nx + T_::TX - 1) / T_::TX;
  const int total = nbx * ((P.ny + T_::TY - 1) / T_::TY);
  unsigned* ctr = tile_ctr + parity;
  if (threadIdx.x == 0) {
    if (blockIdx.x == 0) tile_ctr[parity ^ 1] = 0u;  // the next step's counter
    next_sh[0] = (int)atomicAdd(ctr, 1u);
  }
  __syncthreads();
  int par = 0;
  for (int t = next_sh[0]; t < total; t = next_sh[par]) {
    // draw the next tile now; the tile's staging barrier publishes it
    par ^= 1;
    if (threadIdx.x == 0) next_sh[par] = (int)atomicAdd(ctr, 1u);
    double sI, sIn, sOut, sF;
    step_tile<K, Real, T_>(P, S, t % nbx, t / nbx, pl, red_sh, sI, sIn, sOut, sF);
    publish_partials_at<slots_in_flight(K)>(
        sI, sIn, sOut, S.partials, S.counter, S.scal, p0_closed, false, 0.0, P.eos_c, P.inv_rho_ref,
        (unsigned)t, (unsigned)total, p0_closed || (K > 0 && P.feed), sF,
        K > 0 && P.feed ? P.feed_c : 0.0);
  }
}

// The chemistry's constants in the precision of the Newton matrix.
template <class LA, class Real, int K>
__device__ __forceinline__ const auto& chem_const(const Params<Real, K>& P) {
  if constexpr (sizeof(LA) == 8) return P.c64;
  else return P.c32;
}

// ------------------------------------------- chemistry pre-pass (implicit)
// Per cell: backward-Euler Newton increments over the step at (T^n, Y^n,
// rho^n), stored as the FD source terms rho* dY_k and rho* cp dT.
template <int K, int J, class Real, class Store>
__global__ void __launch_bounds__(BLOCK)
chem_implicit_kernel(const __grid_constant__ Params<Real, K> P, const State<Real, Store> S,
                     Real* __restrict__ src) {
  constexpr int KK = K > 0 ? K : 1;
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= P.N) return;
  const Real T = S.T_in[c];
  Real Y[KK];
#pragma unroll
  for (int k = 0; k < K; ++k) Y[k] = S.Y_in[(size_t)k * P.N + c];
  const Real phif = Real(1) - S.phi[c];
  Real om[KK], omT = 0;
#pragma unroll
  for (int k = 0; k < KK; ++k) om[k] = 0;
  if (phif >= P.phi_min) {
    const Real P0 = scal_P0<Real>(S.scal);
    const Real rho = fdiv(P0 * P.eos_cr, T * mixture_invMw(P, Y));
    double Yd[KK], dY[KK], dT;
#pragma unroll
    for (int k = 0; k < K; ++k) Yd[k] = double(Y[k]);
    chem_be_newton<K, J, Real>(P.c64, chem_const<Real>(P), double(T), Yd, double(rho) * P.c64.rho_ref, dY, &dT);
#pragma unroll
    for (int k = 0; k < K; ++k) om[k] = rho * Real(dY[k]);
    omT = rho * mixture_cp(P, Y) * Real(dT);
  }
#pragma unroll
  for (int k = 0; k < K; ++k) src[(size_t)k * P.N + c] = om[k];
  src[(size_t)K * P.N + c] = omT;
}

// ------------------------------------------------ inlet feedback
// Sec. 4.4.1: the inflow of species feed_k is matched to its consumption.
// The FP32 / FP64 steps sum the consumption with their other reductions
// (combine_partials).  FP16 storage: after the step kernel of step n, whose
// inputs (T, Y and the pre-pass increments) are still in place, feed_kernel
// sums phi_f (-omega_k) of that state over the cells (FP64 block partials,
// grid-stride over at most kFeedBlocks blocks) and feed_combine_kernel sums
// the partials in a fixed order and sets the inlet peak speed of step n + 1.
constexpr int kFeedBlocks = 1024;

template <int K, class Real, class Store>
__global__ void __launch_bounds__(BLOCK)
feed_kernel(const Params<Real, K> P, const State<Real, Store> S, double* __restrict__ part) {
  constexpr int KK = Params<Real, K>::KK;
  __shared__ double red_sh[32];
  double acc = 0;
  if constexpr (K > 0) {
    const Real P0 = scal_P0<Real>(S.scal);
    for (int c = blockIdx.x * BLOCK + threadIdx.x; c < P.N; c += gridDim.x * BLOCK) {
      const Real phif = Real(1) - S.phi[c];
      if (!(phif >= P.phi_min)) continue;
      Real om[KK], omT = 0;
      if (P.chem == 1) {
        const Real T = S.T_in[c];
        Real Y[KK];
#pragma unroll
        for (int k = 0; k < K; ++k) Y[k] = S.Y_in[(size_t)k * P.N + c];
        const Real rho = fdiv(P0 * P.eos_cr, T * mixture_invMw(P, Y));
        rates(P, T, Y, rho, fdiv(Real(1), T), om, omT);
        acc += double(phif * -om[P.feed_k]);
      } else if (P.chem >= 2) {
        acc += double(phif * -S.src[(size_t)P.feed_k * P.N + c]);
      }
    }
  }
  const double s = block_sum<double>(acc, red_sh);
  if (threadIdx.x == 0) part[blockIdx.x] = s;
}

// One warp: u_in = fuel feed_c / P0, held in [0, 0.3].
static __global__ void feed_combine_kernel(const double* __restrict__ part, unsigned nb,
                                           DevScalars* scal, double feed_c) {
  const int lane = threadIdx.x;
  double v = 0;
  for (unsigned b = lane; b < nb; b += 32) v += part[b];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  if (lane == 0) {
    double u = v * feed_c / scal->P0;
    u = u > 0.3 ? 0.3 : (u > 0.0 ? u : 0.0);  // NaN -> 0
    scal->fuel = v;
    scal->u_in = u;
    scal->u_in_f = float(u);
  }
}

// The inlet speed of the first step (and no consumption yet); the
// characteristic outlet starts at the ambient pressure.
static __global__ void set_inlet_kernel(DevScalars* scal, double u_in) {
  scal->u_in = u_in;
  scal->u_in_f = float(u_in);
  scal->fuel = 0.0;
  scal->pb = 0.0;
  scal->pb_f = 0.f;
}

// ------------------------------------------------ moving solid
// Phase field of step n of a rigidly translating solid: the step-0 field phi0
// displaced by s = n u_s, multilinear interpolation between the cells around
// x - s; per axis the host passes the whole shift ish and the fraction fr in
// [0, 1).  Periodic axes wrap, other axes clamp.
template <int DIM, class Real>
__global__ void __launch_bounds__(BLOCK)
phase_shift_kernel(const Real* __restrict__ phi0, Real* __restrict__ phi, int nx, int ny, int nz,
                   int per_mask, int3 ish, Real fx, Real fy, Real fz) {
  const int c = blockIdx.x * BLOCK + threadIdx.x;
  const int N = nx * ny * nz;
  if (c >= N) return;
  const int xyz[3] = {c % nx, (c / nx) % ny, c / (nx * ny)};
  const int ext[3] = {nx, ny, nz}, sh[3] = {ish.x, ish.y, ish.z};
  const Real fr[3] = {fx, fy, fz};
  Real v = 0;
#pragma unroll
  for (int corner = 0; corner < (1 << DIM); ++corner) {
    Real w = 1;
    int q[3] = {xyz[0], xyz[1], xyz[2]};
#pragma unroll
    for (int a = 0; a < DIM; ++a) {
      const int up = (corner >> a) & 1;
      w *= up ? fr[a] : Real(1) - fr[a];
      int qa = xyz[a] - sh[a] - up;
      if ((per_mask >> a) & 1) qa = ((qa % ext[a]) + ext[a]) % ext[a];
      else qa = qa < 0 ? 0 : (qa >= ext[a] ? ext[a] - 1 : qa);
      q[a] = qa;
    }
    v += w * phi0[q[0] + nx * (q[1] + ny * q[2])];
  }
  phi[c] = v;
}

// ------------------------------------------------ characteristic outlet
// Sec. 4.1 (Poinsot and Lele): after a step, one block forms the face means
// of the outlet columns it wrote (fixed-order FP64 sums) and advances the
// boundary pressure, P_b <- P_b - (L5 + K P_b) / 2 with
// L5 = (u + cs)((P1 - P2) + rho cs (u1 - u2)).
template <class Real>
__global__ void __launch_bounds__(BLOCK)
outlet_kernel(const Real* __restrict__ ob, int NF, DevScalars* scal, double K) {
  __shared__ double red_sh[32];
  double v[5] = {0, 0, 0, 0, 0};
  for (int f = threadIdx.x; f < NF; f += BLOCK)
#pragma unroll
    for (int q = 0; q < 5; ++q) v[q] += double(ob[(size_t)q * NF + f]);
  double m[5];
#pragma unroll
  for (int q = 0; q < 5; ++q) m[q] = block_sum<double>(v[q], red_sh) / NF;
  if (threadIdx.x == 0) {
    const double cs = 0.57735026918962576;  // sqrt(1/3)
    const double P1 = m[0], u1 = m[1], P2 = m[2], u2 = m[3], r = m[4];
    const double pb = scal->pb;
    const double L5 = (u1 + cs) * ((P1 - P2) + r * cs * (u1 - u2));
    const double nb = pb - 0.5 * (L5 + K * pb);
    scal->pb = nb;
    scal->pb_f = float(nb);
  }
}

// ------------------------------------------------ initial equilibrium
// g = g_eq(P_h = 0, rho, u); reduction of I = sum phi_f Mw / T for the mass m.
template <int DIM, int K, class Real, class Store>
__global__ void __launch_bounds__(BLOCK)
init_kernel(const Params<Real, K> P, const State<Real, Store> S, const Real* __restrict__ u_init,
            double P0_init) {
  using L = Lattice<DIM>;
  __shared__ double red_sh[32];
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  Real acc = 0;
  if (c < P.N) {
    const Real T = S.T_in[c];
    Real Y[Params<Real, K>::KK];
#pragma unroll
    for (int k = 0; k < K; ++k) Y[k] = S.Y_in[(size_t)k * P.N + c];
    const Real invMw = mixture_invMw(P, Y);
    const Real rho = Real(P0_init) * Real(P.eos_c) / (T * invMw);
    Real u[3] = {0, 0, 0};
    if (u_init)
      for (int a = 0; a < DIM; ++a) u[a] = u_init[(size_t)a * P.N + c];
    Real uu = 0;
    for (int a = 0; a < DIM; ++a) uu += u[a] * u[a];
    // FP16 storage: moments P = 0, j = rho u / 3 of g_eq; the stored residual
    // drops the first-order part w rho c.u
    constexpr bool FO = IsHalf<Store>::value;
#pragma unroll
    for (int i = 0; i < L::Q; ++i) {
      const Real w = Real(L::w(i));
      Real cu = 0;
      for (int a = 0; a < DIM; ++a) cu += Real(L::c(i, a)) * u[a];
      const Real geq = w * rho * ((FO ? Real(0) : cu) + Real(1.5) * cu * cu - Real(0.5) * uu);
      Codec<Store, Real>::store(S.g_out + (size_t)i * P.N + c, geq, P.g_scale * Real(1.0 / L::w(i)));
    }
    if constexpr (FO) {
      S.M_out[c] = Real(0);
      for (int a = 0; a < DIM; ++a) S.M_out[(size_t)(1 + a) * P.N + c] = rho * u[a] * Real(1.0 / 3.0);
    }
    acc = (Real(1) - S.phi[c]) / (T * invMw);
  }
  const double s = block_sum<Real>(acc, red_sh);
  publish_partials<8>(s, 0.0, 0.0, S.partials, S.counter, S.scal, 0, true, P0_init, P.eos_c,
                      P.inv_rho_ref);
}

// --------------------------------------------------- moments (get_fields)
// u, rho and sum g that the next step sees (pull + boundary rules + drag).
// Written in the caller's type Out; a null output is skipped.
template <int DIM, int K, class Real, class Store, class Out>
__global__ void __launch_bounds__(BLOCK)
moments_kernel(const Params<Real, K> P, const State<Real, Store> S, Out* __restrict__ u_out,
               Out* __restrict__ rho_out, Out* __restrict__ ph_out) {
  using L = Lattice<DIM>;
  constexpr int Q = L::Q;
  constexpr int KK = Params<Real, K>::KK;
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= P.N) return;
  const Real P0 = Real(S.scal->P0);
  int xyz[3];
  xyz[0] = c % P.nx;
  xyz[1] = (c / P.nx) % P.ny;
  xyz[2] = DIM == 3 ? c / (P.nx * P.ny) : 0;
  const Real T = S.T_in[c];
  Real Y[KK];
#pragma unroll
  for (int k = 0; k < K; ++k) Y[k] = S.Y_in[(size_t)k * P.N + c];
  const Real rho = P0 * Real(P.eos_c) / (T * mixture_invMw(P, Y));
  const Real phis = S.phi[c];
  Real mu_c, lam_c;
  transport(P, T, Y, mixture_invMw(P, Y), mixture_cp(P, Y), mu_c, lam_c);
  const Real Kd = P.Au_eta2 * mu_c * (Real(1) - phis) * phis * phis;
  Real Yin[KK];
#pragma unroll
  for (int k = 0; k < K; ++k) Yin[k] = P.Y_in[k];
  const Real rho_in = P0 * Real(P.eos_c) / (P.T_in * mixture_invMw(P, Yin));
  const bool outlet_cell = P.bc[1] == BC_OUTLET && xyz[0] == P.nx - 1;
  Real gin[Q], u[3] = {0, 0, 0}, uw[3] = {0, 0, 0};
  for (int pass = 0; pass < (outlet_cell ? 2 : 1); ++pass) {
    pull<DIM>(P, S, c, xyz, rho, rho_in, uw, gin, GlobalMom<Real>{S.M_in, P.N});
    for (int a = 0; a < DIM; ++a) {
      Real m = 0;
      for (int i = 0; i < Q; ++i) m += Real(L::c(i, a)) * gin[i];
      u[a] = (m * Real(3) + Real(0.5) * (P.Fb[a] + Kd * P.u_s[a])) / (rho + Real(0.5) * Kd);
      uw[a] = u[a];
    }
  }
  Real sg = 0;
  for (int i = 0; i < Q; ++i) sg += gin[i];
  if (u_out)
    for (int a = 0; a < DIM; ++a) u_out[(size_t)a * P.N + c] = Out(u[a]);
  if (rho_out) rho_out[c] = Out(rho);
  if (ph_out) ph_out[c] = Out(sg);
}

// ------------------------------------------------- diagnostics (on demand)
// Per-cell terms of the domain diagnostics of the state the next step sees,
// summed per block in FP64: drag sum K_d u (the force of the fluid on the
// solid phase, Sec. 3.2.1), heat sum phi_f S_I (Sec. 3.3, eq.
// diffusion-heat-flux-3), fluid mass sum phi_f rho, and over the outlet
// column rho u_x cp T and rho u_x cp (mixing-cup temperature, Sec. 4.2).
constexpr int NDIAG = 8;
template <int DIM, int K, class Real, class Store>
__global__ void __launch_bounds__(BLOCK)
diag_kernel(const Params<Real, K> P, const State<Real, Store> S, double* __restrict__ part) {
  using L = Lattice<DIM>;
  constexpr int Q = L::Q;
  constexpr int KK = Params<Real, K>::KK;
  __shared__ double red_sh[32];
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  double v[NDIAG] = {0, 0, 0, 0, 0, 0, 0, 0};
  if (c < P.N) {
    const Real P0 = Real(S.scal->P0);
    int xyz[3];
    xyz[0] = c % P.nx;
    xyz[1] = (c / P.nx) % P.ny;
    xyz[2] = DIM == 3 ? c / (P.nx * P.ny) : 0;
    const Real T = S.T_in[c];
    Real Y[KK];
#pragma unroll
    for (int k = 0; k < K; ++k) Y[k] = S.Y_in[(size_t)k * P.N + c];
    const Real rho = P0 * Real(P.eos_c) / (T * mixture_invMw(P, Y));
    const Real phis = S.phi[c], phif = Real(1) - phis;
    const Real cp = mixture_cp(P, Y);
    Real mu, lam;
    transport(P, T, Y, mixture_invMw(P, Y), cp, mu, lam);
    const Real Kd = P.Au_eta2 * mu * phif * phis * phis;
    Real Yin[KK];
#pragma unroll
    for (int k = 0; k < K; ++k) Yin[k] = P.Y_in[k];
    const Real rho_in = P0 * Real(P.eos_c) / (P.T_in * mixture_invMw(P, Yin));
    const bool outlet_cell = P.bc[1] == BC_OUTLET && xyz[0] == P.nx - 1;
    Real gin[Q], u[3] = {0, 0, 0}, uw[3] = {0, 0, 0};
    for (int pass = 0; pass < (outlet_cell ? 2 : 1); ++pass) {
      pull<DIM>(P, S, c, xyz, rho, rho_in, uw, gin, GlobalMom<Real>{S.M_in, P.N});
      for (int a = 0; a < DIM; ++a) {
        Real m = 0;
        for (int i = 0; i < Q; ++i) m += Real(L::c(i, a)) * gin[i];
        u[a] = (m * Real(3) + Real(0.5) * (P.Fb[a] + Kd * P.u_s[a])) / (rho + Real(0.5) * Kd);
        uw[a] = u[a];
      }
    }
    for (int a = 0; a < DIM; ++a) v[a] = double(Kd * (u[a] - P.u_s[a]));
    const Real Ts = P.Ts_field ? S.Ts_in[c] : P.Ts_uniform;
    const bool fluid_on = phif >= P.phi_min;
    const bool solid_on = P.Ts_field ? (phis >= P.phi_min) : true;
    if (fluid_on && solid_on)
      v[3] = double(phif * (P.AT_eta2 * lam * phif * phis * phis * (Ts - T)));
    v[4] = double(phif * rho);
    if (outlet_cell) {
      v[5] = double(rho * u[0] * cp * T);
      v[6] = double(rho * u[0] * cp);
    }
  }
#pragma unroll
  for (int k = 0; k < NDIAG; ++k) {
    const double s = block_sum<double>(v[k], red_sh);
    if (threadIdx.x == 0) part[(size_t)blockIdx.x * NDIAG + k] = s;
  }
}

// Fixed-order sum of the block partials (one warp).
static __global__ void diag_combine_kernel(const double* __restrict__ part, int nb,
                                           double* __restrict__ out) {
  const int lane = threadIdx.x & 31;
  for (int k = 0; k < NDIAG; ++k) {
    double s = 0;
    for (int b = lane; b < nb; b += 32) s += part[(size_t)b * NDIAG + k];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if (lane == 0) out[k] = s;
  }
}

}  // namespace pflb
