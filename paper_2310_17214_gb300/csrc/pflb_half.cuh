// pflb_half.cuh -- the fused step of domains with FP16-stored populations.
//
// One cell per thread, scalar FP32 arithmetic.  The stored FP16 residuals turn
// a last-bit difference of the FP32 update into a step of the FP16 grid (1e-3
// of the residual, 7e-5 of the velocity after 40 steps of the 2-D bed), so this
// path keeps its own operation order: a run reproduces the runs it has to be
// compared with, checkpoints written earlier included.  The FP32 / FP64 path
// (two cells per thread in FP32, written-out rounding) is in pflb_kernels.cuh;
// what does not touch that order (the lattices, the packed operations, the
// reductions, the runs of planes) is shared with it.
#pragma once

#include "pflb_kernels.cuh"

namespace pflb {
namespace half_store {

using Real = float;
using Store = __half;

// Tile shape: TX x (256 / TX) RPT cells per plane, 256 threads; in 2-D every
// thread can own RPT rows and issues the population loads of its inner cells
// before the staging barrier, so the two load phases overlap.  The single-domain
// step takes 32 x 8 with one row per thread (two rows spill at the 64-register
// cap); the batched step lets its autotuner pick among shapes.  3-D blocks march
// over a run of planes.
template <int DIM, int TXv = 32, int RPTv = 1> struct Tile {
  static constexpr int RPT = RPTv;
  static constexpr int TX = TXv, TY = (256 / TXv) * RPT;
  static constexpr int HX = TX + 2, HY = TY + 2, HP = HX * HY;
  static constexpr int NPL = DIM == 3 ? 3 : 1;  // staged planes
};

// Viscosity: Sutherland (Sec. 4, eq. muT) or constant, lattice units.
template <int K>
__device__ __forceinline__ Real viscosity(const Params<Real, K>& P, Real T) {
  if (!P.sutherland) return P.mu_lat;
  Real t = T * P.inv_suth_T;
  return P.mu_lat * t * sqrt(t) * fdiv(P.suth_TS, T + P.suth_S);
}

// Viscosity and conductivity of the gas of composition Y at T (lattice
// units).  Single-gas mode: the viscosity law above and lambda = mu cp / Pr.
// Mixture mode (Sec. 4.4, eqs. muT_mix, phi_mix, conduct_mix): mole fractions
// X_k = Y_k Mw / M_k, species viscosities from their Sutherland laws,
// mu = sum_k mu_k X_k / sum_j Phi_kj X_j with
// Phi_kj = (1 + sqrt(mu_k / mu_j) (M_j / M_k)^(1/4))^2 / (sqrt(8) sqrt(1 + M_k / M_j)),
// lambda = (sum_k X_k lambda_k + 1 / sum_k X_k / lambda_k) / 2 with
// lambda_k = mu_k (1.32 cv_k + 1.77 R / M_k).
template <int K>
__device__ __forceinline__ void transport(const Params<Real, K>& P, Real T, const Real* Y,
                                          Real invMw, Real cp, Real& mu, Real& lam) {
  if constexpr (K > 0) {
    if (P.mix) {
      Real X[K], m[K], sm[K], ism[K];
      const Real Mw = fdiv(Real(1), invMw);
#pragma unroll
      for (int k = 0; k < K; ++k) {
        X[k] = Y[k] * P.invM[k] * Mw;
        const Real t = T * P.inv_suth_Tk[k];
        m[k] = P.mu_lat_k[k] * t * sqrt(t) * fdiv(P.suth_TSk[k], T + P.suth_Sk[k]);
        sm[k] = sqrt(m[k]);
        ism[k] = fdiv(Real(1), sm[k]);
      }
      Real mm = 0, l1 = 0, l2 = 0;
#pragma unroll
      for (int k = 0; k < K; ++k) {
        Real den = 0;
#pragma unroll
        for (int j = 0; j < K; ++j) {
          const Real a = Real(1) + sm[k] * ism[j] * P.wA[k][j];
          den += a * a * P.wB[k][j] * X[j];
        }
        mm += m[k] * X[k] * fdiv(Real(1), den);
        const Real lk = m[k] * P.eucken_k[k];
        l1 += X[k] * lk;
        l2 += X[k] * fdiv(Real(1), lk);
      }
      mu = mm;
      lam = Real(0.5) * (l1 + fdiv(Real(1), l2));
      return;
    }
  }
  mu = half_store::viscosity(P, T);
  lam = mu * cp * P.inv_Pr;
}

template <int K>
__device__ __forceinline__ Real mixture_invMw(const Params<Real, K>& P, const Real* Y) {
  if constexpr (K == 0) {
    return Real(1) / P.M0;
  } else {
    Real s = 0;
#pragma unroll
    for (int k = 0; k < K; ++k) s += Y[k] * P.invM[k];
    return s;
  }
}

template <int K>
__device__ __forceinline__ Real mixture_cp(const Params<Real, K>& P, const Real* Y) {
  if constexpr (K == 0) {
    return P.cp0;
  } else {
    Real s = 0;
#pragma unroll
    for (int k = 0; k < K; ++k) s += Y[k] * P.cp[k];
    return s;
  }
}

// Explicit Arrhenius rates (Sec. 3.2.2 eq. 8, Sec. 3.3 eq. 9), per lattice
// step per rho_ref: om[k] = omega_k dt / rho_ref, omT likewise (J/kg).
template <int K>
__device__ __forceinline__ void rates(const Params<Real, K>& P, Real T, const Real* Y, Real rho,
                                      Real invT, Real* om, Real& omT) {
#pragma unroll
  for (int k = 0; k < K; ++k) om[k] = 0;
  Real C[Params<Real, K>::KK];
#pragma unroll
  for (int k = 0; k < K; ++k) C[k] = rho * P.rho_ref_M[k] * (Y[k] > Real(0) ? Y[k] : Real(0));
#pragma unroll 1
  for (int j = 0; j < P.J; ++j) {
    Real kf = P.A_lat[j] * fexp(-P.EaR[j] * invT);
    if (P.b[j] != Real(0)) kf *= fpow(T, P.b[j]);
    Real q = kf;
#pragma unroll
    for (int k = 0; k < K; ++k) {
      const Real o = P.order[j][k];
      if (o == Real(1)) q *= C[k];
      else if (o == Real(2)) q *= C[k] * C[k];
      else if (o != Real(0)) q *= fpow(C[k], o);
    }
    if (P.rev[j]) {
      // k_r = k_f / K_c, K_c = exp(dS/R - dH/(R T)) (p_ref/(R T))^(sum s)
      const Real Kc = fexp(P.dS_R[j] - P.dH_R[j] * invT) * fpow(P.p_ref_R * invT, P.dn[j]);
      Real qr = fdiv(kf, Kc);
#pragma unroll
      for (int k = 0; k < K; ++k) {
        const Real o = P.rorder[j][k];
        if (o == Real(1)) qr *= C[k];
        else if (o == Real(2)) qr *= C[k] * C[k];
        else if (o != Real(0)) qr *= fpow(C[k], o);
      }
      q -= qr;
    }
#pragma unroll
    for (int k = 0; k < K; ++k) om[k] += P.stoichM[j][k] * q;
  }
  Real wt = 0;
#pragma unroll
  for (int k = 0; k < K; ++k) wt -= P.hf[k] * om[k];
  omT = wt;
}

// First-order part w_i (P + 3 c_i . j) of direction i at the source cell
// (global index src, offset (dx, dy, dz) from the pulling cell).
template <int DIM, class MA>
__device__ __forceinline__ Real first_order(const MA& A, int i, int src, int dx, int dy, int dz) {
  using L = Lattice<DIM>;
  Real cj = 0;
#pragma unroll
  for (int a = 0; a < DIM; ++a) {
    if (L::c(i, a) > 0) cj += A.mom(1 + a, src, dx, dy, dz);
    if (L::c(i, a) < 0) cj -= A.mom(1 + a, src, dx, dy, dz);
  }
  return Real(L::w(i)) * (A.mom(0, src, dx, dy, dz) + Real(3) * cj);
}

template <int K>
__device__ __forceinline__ Real inlet_u(const Params<Real, K>& P, Real u, const int xyz[3],
                                        int dim) {
  if (P.inlet_parabolic != 1) return u;
  for (int a = 1; a < dim; ++a) {
    if (P.bc[2 * a] != BC_WALL) continue;
    Real n = Real(a == 1 ? P.ny : P.nz);
    Real s = Real(xyz[a]) + Real(0.5);
    u *= Real(4) * s * (n - s) / (n * n);
  }
  return u;
}

// The cell's own post-collision population of direction ib (bounce-back).
template <int DIM, int K, class MA>
__device__ __forceinline__ Real own_pop(const Params<Real, K>& P, const State<Real, Store>& S,
                                        int c, int ib, const MA& mom) {
  const Real r = Codec<Store, Real>::raw(S.g_in + (size_t)ib * P.N + c);
  return Codec<Store, Real>::dec(r, Real(Lattice<DIM>::w(ib)) * P.g_inv_scale,
                                 half_store::first_order<DIM>(mom, ib, c, 0, 0, 0));
}

// Half-way bounce-back with the wall velocity for the directions entering
// through face F, when the cell lies on it (on) and it is a wall.
template <int DIM, int F, int K, class MA>
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
    for (int b = 0; b < DIM; ++b) cu += Real(L::c(i, b)) * P.wall_u[F][b];
    gin[i] = half_store::own_pop<DIM>(P, S, c, L::opp(i), mom) +
             Real(2) * Real(L::w(i)) * rho_c * cu;
  }
}

// Pull streaming of every population into the cell.  A cell off every face
// reads its upstream neighbours at fixed offsets.  On a face, along each axis
// the upstream neighbour coordinate wraps across a periodic face and is
// clamped to the cell itself across any other face; every direction is read
// from there.  Directions that cross a non-periodic face are then replaced by the
// boundary rules, in the order outlet, inlet, walls (the wall of the lowest
// axis last, so it wins on edges and corners): half-way bounce-back on walls
// (moving walls add 2 w rho c.u_w), the inlet as a moving wall with the inlet
// velocity and inlet density, the outlet as anti-bounce-back at P_h = 0 with
// wall velocity uw.
template <int DIM, int K, class MA>
__device__ __forceinline__ void pull(const Params<Real, K>& P, const State<Real, Store>& S, int c,
                                     const int xyz[3], Real rho_c, Real rho_in, const Real* uw,
                                     Real* gin, const MA& mom) {
  using L = Lattice<DIM>;
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
      gin[i] = Codec<Store, Real>::dec(r, Real(L::w(i)) * P.g_inv_scale,
                                       half_store::first_order<DIM>(mom, i, src, -cx, -cy, -cz));
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
    gin[i] = Codec<Store, Real>::dec(r, Real(L::w(i)) * P.g_inv_scale,
                                     half_store::first_order<DIM>(mom, i, src, -cx, -cy, -cz));
  }
  // non-periodic faces the cell lies on
  const bool f0 = x == 0 && !per0, f1 = x == P.nx - 1 && !per1;
  const bool f2 = y == 0 && !per2, f3 = y == P.ny - 1 && !per3;
  const bool f4 = DIM == 3 && z == 0 && !per4, f5 = DIM == 3 && z == P.nz - 1 && !per5;
  if (!(f0 || f1 || f2 || f3 || f4 || f5)) return;
  if (f1 && P.bc[1] == BC_OUTLET) {
    Real uu = 0;
#pragma unroll
    for (int a = 0; a < DIM; ++a) uu += uw[a] * uw[a];
    const Real pb2 = P.nscbc ? Real(2) * scal_pb<Real>(S.scal) : Real(0);
#pragma unroll
    for (int i = 0; i < L::Q; ++i) {
      if (L::c(i, 0) != -1) continue;
      Real cu = 0;
#pragma unroll
      for (int a = 0; a < DIM; ++a) cu += Real(L::c(i, a)) * uw[a];
      gin[i] = -half_store::own_pop<DIM>(P, S, c, L::opp(i), mom) +
               Real(L::w(i)) * (pb2 + rho_c * (Real(3) * cu * cu - uu));
    }
  }
  if (f0 && P.bc[0] == BC_INLET) {
    Real ui = half_store::inlet_u(P, P.feed ? scal_u_in<Real>(S.scal) : P.u_in, xyz, DIM);
    if (P.inlet_parabolic == 2) ui *= Real(1) - S.phi[c];
#pragma unroll
    for (int i = 0; i < L::Q; ++i) {
      if (L::c(i, 0) != 1) continue;
      gin[i] = half_store::own_pop<DIM>(P, S, c, L::opp(i), mom) +
               Real(2) * Real(L::w(i)) * rho_in * ui;
    }
  }
  // walls, the highest axis first so that the lowest axis wins on edges
  if (DIM == 3) {
    half_store::wall_pops<DIM, 5>(P, S, c, f5, rho_c, gin, mom);
    half_store::wall_pops<DIM, 4>(P, S, c, f4, rho_c, gin, mom);
  }
  half_store::wall_pops<DIM, 3>(P, S, c, f3, rho_c, gin, mom);
  half_store::wall_pops<DIM, 2>(P, S, c, f2, rho_c, gin, mom);
  half_store::wall_pops<DIM, 1>(P, S, c, f1, rho_c, gin, mom);
  half_store::wall_pops<DIM, 0>(P, S, c, f0, rho_c, gin, mom);
}

// ------------------------------------------------ staged tile (smem)
// Fields per staged cell as in the other step, then the moments (P, j).
template <int DIM, int K, int HP>
struct Plane {
  Real f[F_Y0 + K + DIM + 1][HP];
};

// Stage plane z (may be -1 or nz: ghost plane) of the block's tile with its
// xy halo.  Out-of-domain halo cells follow the ghost rules: periodic faces
// wrap; otherwise the adjacent cell's values, with the inlet state (T_in,
// Y_in) on the inlet face and the wall temperature on a wall that has one.
template <int DIM, int K, class T_>
__device__ __forceinline__ void stage_plane(const Params<Real, K>& P, const State<Real, Store>& S,
                                            Plane<DIM, K, T_::HP>& pl, int x0, int y0, int z,
                                            Real P0) {
  // tiles whose halo lies inside the lattice need no ghost rules
  const bool inner = x0 >= 1 && y0 >= 1 && x0 + T_::TX < P.nx && y0 + T_::TY < P.ny &&
                     (DIM == 2 || (z >= 0 && z < P.nz));
  for (int h = threadIdx.x; h < T_::HP; h += blockDim.x) {
    const int hx = h % T_::HX, hy = h / T_::HX;
    int q[3] = {x0 - 1 + hx, y0 - 1 + hy, z};
    int ghost_face = -1;
    int nout = 0;
#pragma unroll
    for (int a = 0; a < DIM; ++a) {
      if (inner) break;
      const int n = a == 0 ? P.nx : (a == 1 ? P.ny : P.nz);
      if (q[a] < 0 || q[a] >= n) {
        const int face = 2 * a + (q[a] >= n ? 1 : 0);
        if (P.bc[face] == BC_PERIODIC) {
          q[a] = q[a] < 0 ? q[a] + n : q[a] - n;
          if (q[a] < 0 || q[a] >= n) q[a] = q[a] < 0 ? 0 : n - 1;  // tiles wider than n
        } else {
          q[a] = q[a] < 0 ? 0 : n - 1;
          ghost_face = face;
          ++nout;
        }
      }
    }
    const int c = q[0] + P.nx * (q[1] + P.ny * q[2]);
    Real T = __ldg(S.T_in + c);
    const Real phis = __ldg(S.phi + c);
    const Real Ts = P.Ts_field ? __ldg(S.Ts_in + c) : P.Ts_uniform;
    Real Y[Params<Real, K>::KK];
#pragma unroll
    for (int k = 0; k < K; ++k) Y[k] = __ldg(S.Y_in + (size_t)k * P.N + c);
    if (nout == 1) {
      const int bc = P.bc[ghost_face];
      if (bc == BC_INLET) {
        T = P.T_in;
#pragma unroll
        for (int k = 0; k < K; ++k) Y[k] = P.Y_in[k];
      } else if (bc == BC_WALL && P.wall_T[ghost_face] > Real(0)) {
        T = P.wall_T[ghost_face];
      }
    }
    const Real phif = Real(1) - phis;
    const Real invMw = half_store::mixture_invMw(P, Y);
    const Real rho = fdiv(P0 * P.eos_cr, T * invMw);
    const Real cp = half_store::mixture_cp(P, Y);
    Real mu, lam;
    half_store::transport(P, T, Y, invMw, cp, mu, lam);
    Real fD = Real(1);
    if constexpr (K > 0) {
      if (P.D_Tdep) fD = fpow(T * P.inv_DTref, P.D_exp);
    }
    pl.f[F_T][h] = T;
    pl.f[F_PHI][h] = phis;
    pl.f[F_RHO][h] = rho;
    pl.f[F_KT][h] = phif * lam;
    pl.f[F_MU][h] = mu;
    pl.f[F_FD][h] = fD;
    pl.f[F_TS][h] = Ts;
    pl.f[F_RF][h] = phif * rho * fD;
#pragma unroll
    for (int k = 0; k < K; ++k) pl.f[F_Y0 + k][h] = Y[k];
#pragma unroll
    for (int a = 0; a <= DIM; ++a) pl.f[F_Y0 + K + a][h] = __ldg(S.M_in + (size_t)a * P.N + c);
  }
}

// Staged-plane accessor: own and neighbour values of the staged fields and
// properties.  2-D: the populations may be in registers already (pre); 3-D: the
// pulled populations wait in shared memory (st).  MF: the first moment field.
template <int DIM, class TL, int MF>
struct PlaneAcc {
  static constexpr int HP = TL::HP;
  static constexpr bool has_pops = DIM == 2;
  static constexpr bool kStash = DIM == 3;
  const Real* __restrict__ cen;
  const Real* __restrict__ zm;
  const Real* __restrict__ zp;
  int h;
  const Real* pre;
  bool pv;  // pre holds this cell's populations
  Real* st; // stash, [Q][BLOCK]
  __device__ __forceinline__ Real c(int f) const { return cen[f * HP + h]; }
  __device__ __forceinline__ Real n(int f, int a, int s) const {
    if (a == 0) return cen[f * HP + h + s];
    if (a == 1) return cen[f * HP + h + s * TL::HX];
    return (s < 0 ? zm : zp)[f * HP + h];
  }
  __device__ __forceinline__ Real pop(int i) const { return has_pops ? pre[i] : Real(0); }
  // moment a of the staged cell at offset (dx, dy, dz)
  __device__ __forceinline__ Real mom(int a, int, int dx, int dy, int dz) const {
    const Real* p = dz < 0 ? zm : (dz > 0 ? zp : cen);
    return p[(MF + a) * HP + h + dx + dy * TL::HX];
  }
};


// ------------------------------------------------------ the fused step
// Per cell: (a1) pull + moments + implicit drag, (c) reaction source,
// (b) FD transport of Y_k, T, Ts, low-Mach divergence, (a) source + BGK
// collision + store, (d) contribution to the FP64 reduction.
template <int DIM, int K, class Acc>
__device__ __forceinline__ Real cell_update(const Params<Real, K>& P, const State<Real, Store>& S,
                                            const Acc& A, int c, const int xyz[3], Real P0,
                                            Real dlnP0, Real dP0r, Real& fin, Real& fout) {
  using L = Lattice<DIM>;
  constexpr int Q = L::Q;
  constexpr int KK = Params<Real, K>::KK;
  constexpr Real CS2 = Real(1) / Real(3);
  auto at = [&](int f, int a, int s) -> Real { return A.n(f, a, s); };

  const Real T0 = A.c(F_T);
  const Real phis = A.c(F_PHI);
  const Real phif = Real(1) - phis;
  const Real rho = A.c(F_RHO);
  const Real mu = A.c(F_MU);
  const Real fD = A.c(F_FD);
  const Real Ts0 = A.c(F_TS);
  Real Y0[KK];
#pragma unroll
  for (int k = 0; k < K; ++k) Y0[k] = A.c(F_Y0 + k);
  const Real invMw = half_store::mixture_invMw(P, Y0);
  const Real cp = half_store::mixture_cp(P, Y0);
  const Real lam = mu * cp * P.inv_Pr;
  const Real Kd = P.Au_eta2 * mu * phif * phis * phis;
  const Real invT = fdiv(Real(1), T0);

  // cells on a non-periodic face (their pull takes the boundary rules)
  bool edge = (xyz[0] == 0 && P.bc[0] != BC_PERIODIC) ||
              (xyz[0] == P.nx - 1 && P.bc[1] != BC_PERIODIC) ||
              (xyz[1] == 0 && P.bc[2] != BC_PERIODIC) ||
              (xyz[1] == P.ny - 1 && P.bc[3] != BC_PERIODIC);
  if (DIM == 3)
    edge = edge || (xyz[2] == 0 && P.bc[4] != BC_PERIODIC) ||
           (xyz[2] == P.nz - 1 && P.bc[5] != BC_PERIODIC);

  // (a1) pull streaming, moments, implicit drag
  Real rho_in = 0;
  if (edge && P.bc[0] == BC_INLET) {
    Real Yin[KK];
#pragma unroll
    for (int k = 0; k < K; ++k) Yin[k] = P.Y_in[k];
    rho_in = fdiv(P0 * P.eos_cr, P.T_in * half_store::mixture_invMw(P, Yin));
  }
  Real gin[Q];
  Real u[3] = {0, 0, 0}, uw[3] = {0, 0, 0}, mraw[3] = {0, 0, 0};
  const bool outlet_cell = P.bc[1] == BC_OUTLET && xyz[0] == P.nx - 1;
  const Real inv_rk = fdiv(Real(1), rho + Real(0.5) * Kd);
  for (int pass = 0; pass < (outlet_cell ? 2 : 1); ++pass) {
    if (Acc::has_pops && A.pv) {  // populations prefetched for this cell
#pragma unroll
      for (int i = 0; i < Q; ++i) {
        // prefetched values are the scaled residuals as stored
        gin[i] = Codec<Store, Real>::dec(
            A.pop(i), Real(L::w(i)) * P.g_inv_scale,
            half_store::first_order<DIM>(A, i, 0, -L::c(i, 0), -L::c(i, 1),
                                         DIM == 3 ? -L::c(i, 2) : 0));
      }
    } else {
      half_store::pull<DIM>(P, S, c, xyz, rho, rho_in, uw, gin, A);
    }
#pragma unroll
    for (int a = 0; a < DIM; ++a) {
      Real m = 0;
#pragma unroll
      for (int i = 0; i < Q; ++i)
        if (L::c(i, a) != 0) m += Real(L::c(i, a)) * gin[i];
      mraw[a] = m;
      u[a] = (m * Real(3) + Real(0.5) * (P.Fb[a] + Kd * P.u_s[a])) * inv_rk;
      uw[a] = u[a];
    }
  }
  Real sg = 0;
#pragma unroll
  for (int i = 0; i < Q; ++i) sg += gin[i];

  // the pulled populations are needed again only by the collision: with a
  // stash they wait in shared memory instead of 9 / 19 registers
  if constexpr (Acc::kStash) {
#pragma unroll
    for (int i = 0; i < Q; ++i) A.st[i * BLOCK + threadIdx.x] = gin[i];
  }

  const bool fluid_on = phif >= P.phi_min;
  const bool solid_on = P.Ts_field ? (phis >= P.phi_min) : true;
  Real SI = 0;
  if (fluid_on && solid_on)
    SI = P.mix ? P.AT_eta2 * A.c(F_KT) * phis * phis * (Ts0 - T0)  // staged phi_f lambda
               : P.AT_eta2 * lam * phif * phis * phis * (Ts0 - T0);

  // (c) reaction source
  Real om[KK], omT = 0;
#pragma unroll
  for (int k = 0; k < KK; ++k) om[k] = 0;
  if constexpr (K > 0) {
    if (P.chem == 1) half_store::rates(P, T0, Y0, rho, invT, om, omT);
    if (P.chem >= 2) {
      // increments of the chemistry pre-pass (implicit integrator or surrogate)
#pragma unroll
      for (int k = 0; k < K; ++k) om[k] = __ldg(S.src + (size_t)k * P.N + c);
      omT = __ldg(S.src + (size_t)K * P.N + c);
    }
  }

  const Real iphr = fluid_on ? fdiv(Real(1), phif * rho) : Real(0);
  const Real rf0 = A.c(F_RF);

  // (b) species; the face factors (phi_f rho f_D averaged over the face) are
  // shared by every species, and the central differences of Y_k feed the
  // enthalpy-flux cross term of the temperature equation
  Real Yn[KK];
  Real sYm = 0;  // sum_k (1/M_k) DY_k/Dt dt for the divergence
  Real sx[3] = {0, 0, 0};  // sum_k cp_k D_k (Y_k(+) - Y_k(-)) per axis
  {
    Real fm[DIM], fp[DIM];
#pragma unroll
    for (int a = 0; a < DIM; ++a) {
      fm[a] = Real(0.5) * (rf0 + at(F_RF, a, -1));
      fp[a] = Real(0.5) * (rf0 + at(F_RF, a, +1));
    }
    // species in pairs with packed f32x2 arithmetic, the last one of an odd count
    // by itself
    constexpr int KP = (K / 2) * 2;
    if constexpr (KP > 0) {
      const float2 zero = splat<float2>(0.f);
      float2 sx2[3] = {zero, zero, zero}, sYm2 = zero;
      const float2 prf = splat<float2>(-phif * rho), pf = splat<float2>(phif);
      const float2 ip = splat<float2>(iphr);
#pragma unroll
      for (int k = 0; k < KP; k += 2) {
        const float2 y0 = make_float2(Y0[k], Y0[k + 1]);
        float2 adv = zero, dif = zero, cen = zero;
#pragma unroll
        for (int a = 0; a < DIM; ++a) {
          const float2 dm = vsub(y0, make_float2(at(F_Y0 + k, a, -1), at(F_Y0 + k + 1, a, -1)));
          const float2 dp = vsub(make_float2(at(F_Y0 + k, a, +1), at(F_Y0 + k + 1, a, +1)), y0);
          adv = vfma(splat<float2>(u[a]), u[a] > 0.f ? dm : dp, adv);
          dif = vfma(splat<float2>(fp[a]), dp, dif);
          dif = vfma(splat<float2>(-fm[a]), dm, dif);
          const float2 sd = vadd(dp, dm);
          cen = vfma(splat<float2>(u[a]), sd, cen);
          sx2[a] = vfma(make_float2(P.cpD[k], P.cpD[k + 1]), sd, sx2[a]);
        }
        float2 dY = vfma(prf, adv, vfma(make_float2(P.Dlat[k], P.Dlat[k + 1]), dif,
                                        vmul(pf, make_float2(om[k], om[k + 1]))));
        dY = fluid_on ? vmul(dY, ip) : splat<float2>(0.f);
        const float2 yn = vadd(y0, dY);
        Yn[k] = yn.x;
        Yn[k + 1] = yn.y;
        // material increment: the step's increment plus u.grad Y_k (central)
        const float2 dm2 = fluid_on ? vfma(splat<float2>(0.5f), cen, dY) : splat<float2>(0.f);
        sYm2 = vfma(make_float2(P.invM[k], P.invM[k + 1]), dm2, sYm2);
      }
#pragma unroll
      for (int a = 0; a < DIM; ++a) sx[a] += sx2[a].x + sx2[a].y;
      sYm += sYm2.x + sYm2.y;
    }
#pragma unroll
    for (int k = KP; k < K; ++k) {
      Real adv = 0, dif = 0, cen = 0;
#pragma unroll
      for (int a = 0; a < DIM; ++a) {
        const Real dm = Y0[k] - at(F_Y0 + k, a, -1), dp = at(F_Y0 + k, a, +1) - Y0[k];
        adv += u[a] * (u[a] > Real(0) ? dm : dp);
        dif += fp[a] * dp - fm[a] * dm;
        cen += u[a] * (dp + dm);
        sx[a] += P.cpD[k] * (dp + dm);
      }
      const Real dY = fluid_on ? (-phif * rho * adv + P.Dlat[k] * dif + phif * om[k]) * iphr
                               : Real(0);
      Yn[k] = Y0[k] + dY;
      // material increment: the step's increment plus u.grad Y_k (central)
      sYm += (fluid_on ? dY + Real(0.5) * cen : Real(0)) * P.invM[k];
    }
  }

  // (b) temperature
  Real Tn = Ts0, dTm = Ts0 - T0;  // frozen cells take the solid temperature
  if (fluid_on) {
    Real adv = 0, dif = 0, cross = 0, cen = 0;
    const Real kc = A.c(F_KT);
#pragma unroll
    for (int a = 0; a < DIM; ++a) {
      const Real tm = at(F_T, a, -1), tp = at(F_T, a, +1);
      adv += u[a] > Real(0) ? u[a] * (T0 - tm) : u[a] * (tp - T0);
      cen += u[a] * (tp - tm);
      const Real km = Real(0.5) * (kc + at(F_KT, a, -1));
      const Real kp = Real(0.5) * (kc + at(F_KT, a, +1));
      dif += kp * (tp - T0) - km * (T0 - tm);
      if constexpr (K > 0) cross += Real(0.25) * fD * sx[a] * (tp - tm);
    }
    const Real rhs = -phif * rho * cp * adv + dif + phif * (rho * cross + dP0r + omT + SI);
    const Real dTn = rhs * iphr * fdiv(Real(1), cp);
    Tn = T0 + dTn;
    dTm = dTn + Real(0.5) * cen;  // plus u.grad T (central)
  }

  // solid temperature
  if (P.Ts_field) {
    Real Tsn = Ts0;
    if (phis >= P.phi_min) {
      Real dif = 0;
#pragma unroll
      for (int a = 0; a < DIM; ++a) {
        const Real km = Real(0.5) * (phis + at(F_PHI, a, -1)) * P.Lams;
        const Real kp = Real(0.5) * (phis + at(F_PHI, a, +1)) * P.Lams;
        dif += kp * (at(F_TS, a, +1) - Ts0) - km * (Ts0 - at(F_TS, a, -1));
      }
      Tsn = Ts0 + fdiv(dif - phif * SI, phis * P.Cs);
      if (P.moving) {
        // a moving solid carries its temperature with u_s (upwind)
        Real advs = 0;
#pragma unroll
        for (int a = 0; a < DIM; ++a) {
          const Real us = P.u_s[a];
          if (us > Real(0)) advs += us * (Ts0 - at(F_TS, a, -1));
          else if (us < Real(0)) advs += us * (at(F_TS, a, +1) - Ts0);
        }
        Tsn -= advs;
      }
    }
    S.Ts_out[c] = Tsn;
  }

  // low-Mach divergence: continuity with the EOS at uniform P0,
  // D = (1/T) DT/Dt + Mw sum_k (1/M_k) DY_k/Dt - (1/P0) dP0/dt, the material
  // increments taken as the step's increments plus u.grad with central
  // differences, the gradient the source takes of rho (with the upwind
  // gradient the discrete continuity would keep a first-order mass defect)
  Real D = dTm * invT;
  if constexpr (K > 0) D += fdiv(sYm, invMw);
  D -= dlnP0;

  // (a) source and BGK collision: omega = 1/tau = 2 rho / (rho + 6 mu)
  Real G[3] = {0, 0, 0}, F[3] = {0, 0, 0};
#pragma unroll
  for (int a = 0; a < DIM; ++a) {
    G[a] = CS2 * Real(0.5) * (at(F_RHO, a, +1) - at(F_RHO, a, -1));
    F[a] = P.Fb[a] - Kd * (u[a] - P.u_s[a]);
  }
  // P_h: the pulled zeroth moment plus half the zeroth moment of the source,
  // sum_i Xi_i = u.G + rho cs^2 D, so that a step adds the whole source
  Real uG = 0;
#pragma unroll
  for (int a = 0; a < DIM; ++a) uG += u[a] * G[a];
  const Real Ph = sg + Real(0.5) * (rho * CS2 * D + uG);
  if (P.nscbc && xyz[0] >= P.nx - 2) {
    // the two outlet columns of this step for the characteristic outlet
    const int NF = P.ny * P.nz, f = xyz[1] + P.ny * xyz[2];
    const int col = xyz[0] == P.nx - 1 ? 0 : 1;
    S.ob[(size_t)(2 * col) * NF + f] = Ph;
    S.ob[(size_t)(2 * col + 1) * NF + f] = u[0];
    if (col == 0) S.ob[(size_t)4 * NF + f] = rho;
  }
  const Real omega = fdiv(Real(2) * rho, rho + Real(6) * mu);
  const Real src_w = Real(1) - Real(0.5) * omega;
  // f_eq / rho - w = w e with e = 3 cu + 9/2 cu^2 - 3/2 uu;
  // g_eq = cs2 f_eq + w (P_h - rho cs2) = w (P_h + rho e / 3);
  // Xi = w [(c - u).(G e + F (1 + e)) + rho cs2 D] = w [(c.H - u.H) e + c.F - u.F + rho cs2 D]
  // with H = G + F.  Collected per cell: g* = (1 - omega) g + w [A0 + B e + src_w x],
  // A0 = omega P_h + src_w rho cs2 D, B = omega rho cs2, x = (c.H - u.H) e + c.F - u.F.
  Real H[3] = {0, 0, 0};
  Real uu = 0, uH = 0, uF = 0;
#pragma unroll
  for (int a = 0; a < DIM; ++a) {
    H[a] = G[a] + F[a];
    uu += u[a] * u[a];
    uH += u[a] * H[a];
    uF += u[a] * F[a];
  }
  const Real rho3 = rho * CS2;
  const Real A0 = omega * Ph + src_w * (rho3 * D);
  const Real B = omega * rho3;
  const Real uu15 = Real(1.5) * uu;
  const Real keep = Real(1) - omega;
  // the post-collision moments of this cell in closed form
  // (sum_i w_i e_i = 0, sum_i w_i x_i = u.G, sum_i w_i c_i e_i = u,
  // sum_i w_i c_i x_i = F / 3 on the isotropic lattice); any values would do,
  // since readers add back exactly what is subtracted here, but these leave
  // a residual of second order in u
  const Real Pst = keep * sg + A0 + src_w * (uH - uF);
  Real jst[3] = {0, 0, 0};
#pragma unroll
  for (int a = 0; a < DIM; ++a) jst[a] = keep * mraw[a] + B * u[a] + src_w * CS2 * F[a];
  // a direction and its opposite are updated together with packed f32x2
  // arithmetic (c.u, c.H, c.F of the opposite are the negated ones), the rest
  // direction by itself
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    if (L::opp(i) < i) continue;  // done with its opposite
    Real cu = 0, cH = 0, cF = 0, cj = 0;
#pragma unroll
    for (int a = 0; a < DIM; ++a) {
      if (L::c(i, a) > 0) { cu += u[a]; cH += H[a]; cF += F[a]; cj += jst[a]; }
      if (L::c(i, a) < 0) { cu -= u[a]; cH -= H[a]; cF -= F[a]; cj -= jst[a]; }
    }
    Real gi = gin[i];
    if constexpr (Acc::kStash) gi = A.st[i * BLOCK + threadIdx.x];
    if (i > 0) {
      const int j = L::opp(i);
      Real gj = gin[j];
      if constexpr (Acc::kStash) gj = A.st[j * BLOCK + threadIdx.x];
      const float2 cu2 = make_float2(cu, -cu);
      const float2 e = vfma(cu2, vfma(cu2, splat<float2>(4.5f), splat<float2>(3.f)),
                            splat<float2>(-uu15));
      const float2 x = vfma(vsub(make_float2(cH, -cH), splat<float2>(uH)), e,
                            vsub(make_float2(cF, -cF), splat<float2>(uF)));
      float2 t = vfma(splat<float2>(B), e, splat<float2>(A0));
      t = vfma(splat<float2>(src_w), x, t);
      const float w = float(L::w(i));
      float2 g = vfma(splat<float2>(keep), make_float2(gi, gj), vmul(splat<float2>(w), t));
      g = vsub(g, vmul(splat<float2>(w), vfma(splat<float2>(3.f), make_float2(cj, -cj),
                                              splat<float2>(Pst))));
      Codec<Store, Real>::store(S.g_out + (size_t)i * P.N + c, g.x,
                                P.g_scale * Real(1.0 / L::w(i)));
      Codec<Store, Real>::store(S.g_out + (size_t)j * P.N + c, g.y,
                                P.g_scale * Real(1.0 / L::w(j)));
      continue;
    }
    const Real w = Real(L::w(i));
    const Real e = cu * (Real(3) + Real(4.5) * cu) - uu15;
    const Real x = (cH - uH) * e + (cF - uF);
    Real g = keep * gi + w * (A0 + B * e + src_w * x);
    g -= w * (Pst + Real(3) * cj);
    Codec<Store, Real>::store(S.g_out + (size_t)i * P.N + c, g, P.g_scale * Real(1.0 / L::w(i)));
  }
  S.M_out[c] = Pst;
#pragma unroll
  for (int a = 0; a < DIM; ++a) S.M_out[(size_t)(1 + a) * P.N + c] = jst[a];

  S.T_out[c] = Tn;
#pragma unroll
  for (int k = 0; k < K; ++k) S.Y_out[(size_t)k * P.N + c] = Yn[k];

  // (d) contributions to the reduction
  const Real fx = phif * rho * u[0];
  fin = (xyz[0] == 0 && P.bc[0] == BC_INLET) ? fx : Real(0);
  fout = outlet_cell ? fx : Real(0);
  // 0 * P_h is NaN when any pulled population is: a NaN confined to the
  // populations reaches the FP64 reduction (and the status word) this step
  return phif * fdiv(Real(1), Tn * half_store::mixture_invMw(P, Yn)) + Real(0) * Ph;
}

// Resident blocks per SM asked of the register allocator: 4 in 2-D (64
// registers); 2 in 3-D, whose decode holds the source cells' moments (128).
template <int DIM> constexpr int min_blocks() { return DIM == 2 ? 4 : 2; }

// One tile of the fused step (tile (bx, by) of the xy grid, planes z_begin to
// z_end in 3-D): stages the tile's planes in `planes` (shared memory), updates its
// cells and returns the block sums of the reduction in thread 0 (I, inlet
// flux, outlet flux).  Every thread of the block calls it.
template <int DIM, int K, class T_ = Tile<DIM>>
__device__ __forceinline__ void step_tile(const Params<Real, K>& P, const State<Real, Store>& S,
                                          int bx, int by, int z_begin, int z_end,
                                          Plane<DIM, K, T_::HP>* planes,
                                          double* red_sh,
                                          double& sI, double& sIn, double& sOut) {
  const Real P0 = scal_P0<Real>(S.scal);
  const Real dlnP0 = scal_dlnP0<Real>(S.scal);
  const Real dP0r = scal_dP0r<Real>(S.scal);

  const int tx = threadIdx.x % T_::TX, ty = threadIdx.x / T_::TX;
  const int x0 = bx * T_::TX, y0 = by * T_::TY;
  const int x = x0 + tx, y = y0 + ty;
  const int h = (ty + 1) * T_::HX + (tx + 1);
  const bool in_xy = x < P.nx && y < P.ny;
  const bool flux_block = (x0 == 0 && P.bc[0] == BC_INLET) ||
                          (x0 + T_::TX >= P.nx && P.bc[1] == BC_OUTLET);

  Real accI = 0, accIn = 0, accOut = 0;
  if constexpr (DIM == 2) {
    using L = Lattice<2>;
    constexpr int RPT = T_::RPT;
    constexpr int RS = T_::TY / RPT;  // row stride between a thread's cells
    // population loads of the thread's interior cells, issued before staging
    Real pre[RPT][L::Q];
    bool pv[RPT];
#pragma unroll
    for (int r = 0; r < RPT; ++r) {
      const int yr = y0 + ty + r * RS;
      pv[r] = x > 0 && x < P.nx - 1 && yr > 0 && yr < P.ny - 1;
      if (pv[r]) {
        const int c = x + P.nx * yr;
#pragma unroll
        for (int i = 0; i < L::Q; ++i)
          pre[r][i] = Codec<Store, Real>::raw(
              S.g_in + (size_t)i * P.N + c - L::c(i, 0) - L::c(i, 1) * P.nx);
      }
    }
    half_store::stage_plane<DIM, K, T_>(P, S, planes[0], x0, y0, 0, P0);
    __syncthreads();
#pragma unroll
    for (int r = 0; r < RPT; ++r) {
      const int yr = y0 + ty + r * RS;
      if (x < P.nx && yr < P.ny) {
        const int c = x + P.nx * yr;
        const int xyz[3] = {x, yr, 0};
        const int hr = (ty + r * RS + 1) * T_::HX + (tx + 1);
        Real fi, fo;
        const PlaneAcc<DIM, T_, F_Y0 + K> A{&planes[0].f[0][0], nullptr, nullptr, hr, pre[r],
                                            pv[r], nullptr};
        accI += half_store::cell_update<DIM, K>(P, S, A, c, xyz, P0, dlnP0, dP0r, fi, fo);
        accIn += fi;
        accOut += fo;
      }
    }
  } else {
    // ring of three staged planes: slot (z mod 3)
    half_store::stage_plane<DIM, K, T_>(P, S, planes[(z_begin + 2) % 3], x0, y0,
                                                 z_begin - 1, P0);
    half_store::stage_plane<DIM, K, T_>(P, S, planes[z_begin % 3], x0, y0, z_begin, P0);
    for (int z = z_begin; z < z_end; ++z) {
      half_store::stage_plane<DIM, K, T_>(P, S, planes[(z + 1) % 3], x0, y0, z + 1, P0);
      __syncthreads();
      if (in_xy) {
        const int c = x + P.nx * (y + P.ny * z);
        const int xyz[3] = {x, y, z};
        Real fi, fo;
        const PlaneAcc<DIM, T_, F_Y0 + K> A{
            &planes[z % 3].f[0][0], &planes[(z + 2) % 3].f[0][0], &planes[(z + 1) % 3].f[0][0], h,
            nullptr, false, reinterpret_cast<Real*>(planes + T_::NPL)};
        accI += half_store::cell_update<DIM, K>(P, S, A, c, xyz, P0, dlnP0, dP0r, fi, fo);
        accIn += fi;
        accOut += fo;
      }
      __syncthreads();
    }
  }

  // (d) block partials in FP64 (one barrier)
  block_sum3<Real>(accI, accIn, accOut, flux_block, red_sh, sI, sIn, sOut);
}

template <int DIM, int K>
__global__ void __launch_bounds__(BLOCK, min_blocks<DIM>())
step_kernel(const Params<Real, K> P, const State<Real, Store> S, int p0_closed,
            const double* __restrict__ prev_partials, unsigned prev_nb, int chunk) {
  using T_ = Tile<DIM>;
  using PL = Plane<DIM, K, T_::HP>;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  PL* planes = reinterpret_cast<PL*>(smem_raw);
  __shared__ double red_sh[96];

  // deferred combine of the previous step's partials (fixed P0 only) by the first
  // block's first warp: in 2-D in a block of its own, so that no tile waits for it
  // (in front of the first tile, a 500 x 500 domain without species 17.4 us a step,
  // 15.4 so), in 3-D while the other blocks start on their cells
  int b = blockIdx.x, nb = gridDim.x;
  if (prev_partials) {
    if (b == 0) {
      if (threadIdx.x < 32)
        combine_partials<4>(prev_partials, prev_nb, S.scal, 0, false, 0.0, P.eos_c, P.inv_rho_ref);
      if (DIM == 2) return;
    }
    if (DIM == 2) {
      --b;
      --nb;
    }
  }

  double sI, sIn, sOut;
  const int gx = (P.nx + T_::TX - 1) / T_::TX;
  int bx = b % gx, by = b / gx, z0 = 0, z1 = 1;
  if constexpr (DIM == 3) {
    const ZRun r = z_run(b, gx * ((P.ny + T_::TY - 1) / T_::TY), P.nz, chunk);
    bx = r.tile % gx;
    by = r.tile / gx;
    z0 = r.z_begin;
    z1 = r.z_end;
  }
  half_store::step_tile<DIM, K, T_>(P, S, bx, by, z0, z1, planes, red_sh, sI, sIn, sOut);
  // deterministic finish by the last block (closed P0) or deferred
  publish_partials_at<4>(sI, sIn, sOut, S.partials, S.counter, S.scal, p0_closed, false, 0.0,
                         P.eos_c, P.inv_rho_ref, (unsigned)b, (unsigned)nb, p0_closed);
}

// Persistent variant of the 2-D step: one grid of resident blocks walks the
// tiles, handed out by an atomic counter (one per step parity; each launch
// clears the other one for the next step), so no block waits for a second
// wave and cheap tiles do not leave SMs idle.  Reduction slots are the tile
// indices, as in step_kernel.
template <int DIM, int K, class T_>
__global__ void __launch_bounds__(BLOCK, (T_::RPT > 1 ? 3 : 4))
step_persistent_kernel(const Params<Real, K> P, const State<Real, Store> S, int p0_closed,
                       const double* __restrict__ prev_partials, unsigned prev_nb,
                       unsigned* __restrict__ tile_ctr, int parity) {
  static_assert(DIM == 2, "the persistent step walks 2-D tiles");
  using PL = Plane<DIM, K, T_::HP>;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  PL* planes = reinterpret_cast<PL*>(smem_raw);
  __shared__ double red_sh[96];
  __shared__ int next_sh[2];

  if (prev_partials && blockIdx.x == 0 && threadIdx.x < 32)
    combine_partials<4>(prev_partials, prev_nb, S.scal, 0, false, 0.0, P.eos_c, P.inv_rho_ref);

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
    double sI, sIn, sOut;
    half_store::step_tile<DIM, K, T_>(P, S, t % nbx, t / nbx, 0, 1, planes, red_sh, sI, sIn,
                                       sOut);
    publish_partials_at<4>(sI, sIn, sOut, S.partials, S.counter, S.scal, p0_closed, false, 0.0,
                        P.eos_c, P.inv_rho_ref, (unsigned)t, (unsigned)total, p0_closed != 0);
  }
}

// staged planes, and in 3-D the stash of the pulled populations
template <int DIM, int K, class T_ = Tile<DIM>>
constexpr size_t step_smem_bytes() {
  return sizeof(Plane<DIM, K, T_::HP>) * T_::NPL +
         (DIM == 3 ? sizeof(Real) * Lattice<DIM>::Q * BLOCK : 0);
}

// staged fields of the march
enum { G_T = 0, G_PHI, G_RHO, G_KT, G_TS, G_RF, G_Y0 };

__host__ __device__ constexpr int march_field(int f) {
  return f == F_T ? G_T : f == F_PHI ? G_PHI : f == F_RHO ? G_RHO : f == F_KT ? G_KT
       : f == F_TS ? G_TS : f == F_RF ? G_RF : G_Y0 + (f - F_Y0);
}

template <int K>
__host__ __device__ constexpr int march_nf() { return G_Y0 + K + 4; }  // species, moments

template <int K>
constexpr size_t march_smem_bytes() {
  return sizeof(Real) * (3 * march_nf<K>() * Tile<3>::HP + Lattice<3>::Q * BLOCK);
}

// Accessor of cell_update over the march's staged planes; mu and f_D are the
// cell's own values.
template <int K, bool PRE>
struct MarchAcc {
  using TL = Tile<3>;
  static constexpr int HP = TL::HP;
  static constexpr bool has_pops = PRE;
  static constexpr bool kStash = true;  // pulled populations wait in shared memory
  const Real* __restrict__ cen;
  const Real* __restrict__ zm;
  const Real* __restrict__ zp;
  int h;
  Real mu, fD;
  const Real* pre;
  bool pv;  // pre holds this cell's populations
  Real* st; // stash [Q][BLOCK]
  __device__ __forceinline__ Real c(int f) const {
    if (f == F_MU) return mu;
    if (f == F_FD) return fD;
    return cen[march_field(f) * HP + h];
  }
  __device__ __forceinline__ Real n(int f, int a, int s) const {
    const int g = march_field(f) * HP;
    if (a == 0) return cen[g + h + s];
    if (a == 1) return cen[g + h + s * TL::HX];
    return (s < 0 ? zm : zp)[g + h];
  }
  __device__ __forceinline__ Real pop(int i) const { return PRE ? pre[i] : Real(0); }
  __device__ __forceinline__ Real mom(int a, int, int dx, int dy, int dz) const {
    const Real* p = dz < 0 ? zm : (dz > 0 ? zp : cen);
    return p[(G_Y0 + K + a) * HP + h + dx + dy * TL::HX];
  }
};

// Stage plane z (may be -1 or nz: ghost plane) of the tile at (x0, y0) with
// its xy halo into `pl` ([NF][HP]), with the ghost rules of stage_plane.
template <int K>
__device__ __forceinline__ void march_stage(const Params<Real, K>& P, const State<Real, Store>& S,
                                            Real* __restrict__ pl, int x0, int y0, int z,
                                            Real P0) {
  using T_ = Tile<3>;
  constexpr int HP = T_::HP;
  const bool inner = x0 >= 1 && y0 >= 1 && x0 + T_::TX < P.nx && y0 + T_::TY < P.ny && z >= 0 &&
                     z < P.nz;
  for (int h = threadIdx.x; h < HP; h += blockDim.x) {
    const int hy = h / T_::HX, hx = h - hy * T_::HX;
    int q[3] = {x0 - 1 + hx, y0 - 1 + hy, z};
    int ghost_face = -1, nout = 0;
    if (!inner) {
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        const int n = a == 0 ? P.nx : (a == 1 ? P.ny : P.nz);
        if (q[a] < 0 || q[a] >= n) {
          const int face = 2 * a + (q[a] >= n ? 1 : 0);
          if (P.bc[face] == BC_PERIODIC) {
            q[a] = q[a] < 0 ? q[a] + n : q[a] - n;
            if (q[a] < 0 || q[a] >= n) q[a] = q[a] < 0 ? 0 : n - 1;
          } else {
            q[a] = q[a] < 0 ? 0 : n - 1;
            ghost_face = face;
            ++nout;
          }
        }
      }
    }
    const int c = q[0] + P.nx * (q[1] + P.ny * q[2]);
    Real T = __ldg(S.T_in + c);
    const Real phis = __ldg(S.phi + c);
    const Real Ts = P.Ts_field ? __ldg(S.Ts_in + c) : P.Ts_uniform;
    Real Y[Params<Real, K>::KK];
#pragma unroll
    for (int k = 0; k < K; ++k) Y[k] = __ldg(S.Y_in + (size_t)k * P.N + c);
    if (nout == 1) {
      const int bc = P.bc[ghost_face];
      if (bc == BC_INLET) {
        T = P.T_in;
#pragma unroll
        for (int k = 0; k < K; ++k) Y[k] = P.Y_in[k];
      } else if (bc == BC_WALL && P.wall_T[ghost_face] > Real(0)) {
        T = P.wall_T[ghost_face];
      }
    }
    const Real phif = Real(1) - phis;
    const Real invMw = half_store::mixture_invMw(P, Y);
    const Real rho = fdiv(P0 * P.eos_cr, T * invMw);
    const Real cp = half_store::mixture_cp(P, Y);
    Real mu, lam;
    half_store::transport(P, T, Y, invMw, cp, mu, lam);
    Real fD = Real(1);
    if constexpr (K > 0) {
      if (P.D_Tdep) fD = fpow(T * P.inv_DTref, P.D_exp);
    }
    pl[G_T * HP + h] = T;
    pl[G_PHI * HP + h] = phis;
    pl[G_RHO * HP + h] = rho;
    pl[G_KT * HP + h] = phif * lam;
    pl[G_TS * HP + h] = Ts;
    pl[G_RF * HP + h] = phif * rho * fD;
#pragma unroll
    for (int k = 0; k < K; ++k) pl[(G_Y0 + k) * HP + h] = Y[k];
#pragma unroll
    for (int a = 0; a < 4; ++a)
      pl[(G_Y0 + K + a) * HP + h] = __ldg(S.M_in + (size_t)a * P.N + c);
  }
}

// The 19 pulls of cell (x, y, z) with periodic faces wrapped; false (and
// nothing loaded) for a cell on a non-periodic face, whose pull needs the
// boundary rules.
template <int K>
__device__ __forceinline__ bool march_prefetch(const Params<Real, K>& P,
                                               const State<Real, Store>& S, int x, int y, int z,
                                               Real* __restrict__ out) {
  using L = Lattice<3>;
  const int n[3] = {P.nx, P.ny, P.nz};
  const int xyz[3] = {x, y, z};
  int v[3][3];  // v[a][1 + s]: coordinate a of the neighbour at offset s, wrapped
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const int lo = xyz[a] - 1, hi = xyz[a] + 1;
    if ((lo < 0 && P.bc[2 * a] != BC_PERIODIC) || (hi >= n[a] && P.bc[2 * a + 1] != BC_PERIODIC))
      return false;
    v[a][0] = lo < 0 ? lo + n[a] : lo;
    v[a][1] = xyz[a];
    v[a][2] = hi >= n[a] ? hi - n[a] : hi;
  }
#pragma unroll
  for (int i = 0; i < L::Q; ++i) {
    const int src =
        v[0][1 - L::c(i, 0)] + P.nx * (v[1][1 - L::c(i, 1)] + P.ny * v[2][1 - L::c(i, 2)]);
    out[i] = Codec<Store, Real>::raw(S.g_in + (size_t)i * P.N + src);
  }
  return true;
}

template <int K, bool PRE>
__global__ void __launch_bounds__(BLOCK, min_blocks<3>())
step3d_march_kernel(const Params<Real, K> P, const State<Real, Store> S, int p0_closed,
                    const double* __restrict__ prev_partials, unsigned prev_nb) {
  using T_ = Tile<3>;
  using L = Lattice<3>;
  constexpr int HP = T_::HP;
  constexpr int NF = march_nf<K>();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  Real* planes = reinterpret_cast<Real*>(smem_raw);  // [3][NF][HP]
  __shared__ double red_sh[96];

  if (prev_partials && blockIdx.x == 0 && threadIdx.x < 32)
    combine_partials<4>(prev_partials, prev_nb, S.scal, 0, false, 0.0, P.eos_c, P.inv_rho_ref);

  const Real P0 = scal_P0<Real>(S.scal);
  const Real dlnP0 = scal_dlnP0<Real>(S.scal);
  const Real dP0r = scal_dP0r<Real>(S.scal);

  const int tiles_x = (P.nx + T_::TX - 1) / T_::TX;
  const int tiles = tiles_x * ((P.ny + T_::TY - 1) / T_::TY);
  const long long total = (long long)tiles * P.nz;
  const long long g_end = total * (blockIdx.x + 1) / gridDim.x;
  const int tx = threadIdx.x % T_::TX, ty = threadIdx.x / T_::TX;
  const int h = (ty + 1) * T_::HX + (tx + 1);

  Real accI = 0, accIn = 0, accOut = 0;
  bool flux_block = false;
  for (long long gi = total * blockIdx.x / gridDim.x; gi < g_end;) {
    const int tile = (int)(gi / P.nz);
    const int z_begin = (int)(gi - (long long)tile * P.nz);
    const int z_end = (int)min((long long)P.nz, z_begin + (g_end - gi));
    gi += z_end - z_begin;
    const int x0 = (tile % tiles_x) * T_::TX, y0 = (tile / tiles_x) * T_::TY;
    const int x = x0 + tx, y = y0 + ty;
    const bool in_xy = x < P.nx && y < P.ny;
    flux_block = flux_block || (x0 == 0 && P.bc[0] == BC_INLET) ||
                 (x0 + T_::TX >= P.nx && P.bc[1] == BC_OUTLET);

    __syncthreads();  // the previous column is done with the planes
    half_store::march_stage<K>(P, S, planes + ((z_begin + 2) % 3) * NF * HP, x0, y0,
                                z_begin - 1, P0);
    half_store::march_stage<K>(P, S, planes + (z_begin % 3) * NF * HP, x0, y0, z_begin, P0);
    Real pre[L::Q], nxt[L::Q];
    bool have = false, have_nxt = false;
    if constexpr (PRE) {
      if (in_xy) have = half_store::march_prefetch<K>(P, S, x, y, z_begin, pre);
    }
    for (int z = z_begin; z < z_end; ++z) {
      half_store::march_stage<K>(P, S, planes + ((z + 1) % 3) * NF * HP, x0, y0, z + 1, P0);
      if constexpr (PRE) {
        have_nxt = in_xy && z + 1 < z_end &&
                   half_store::march_prefetch<K>(P, S, x, y, z + 1, nxt);
      }
      __syncthreads();
      if (in_xy) {
        const int c = x + P.nx * (y + P.ny * z);
        const int xyz[3] = {x, y, z};
        const Real* cen = planes + (z % 3) * NF * HP;
        const Real T0 = cen[G_T * HP + h];
        Real fD = Real(1);
        if constexpr (K > 0) {
          if (P.D_Tdep) fD = fpow(T0 * P.inv_DTref, P.D_exp);
        }
        Real mu0 = half_store::viscosity(P, T0);
        if constexpr (K > 0) {
          if (P.mix) {  // mixture-averaged viscosity of the cell's own composition
            Real Yo[K], lam0;
#pragma unroll
            for (int k = 0; k < K; ++k) Yo[k] = cen[(G_Y0 + k) * HP + h];
            half_store::transport(P, T0, Yo, half_store::mixture_invMw(P, Yo),
                                  half_store::mixture_cp(P, Yo), mu0, lam0);
          }
        }
        const MarchAcc<K, PRE> A{cen, planes + ((z + 2) % 3) * NF * HP,
                                       planes + ((z + 1) % 3) * NF * HP, h, mu0, fD,
                                       pre, PRE && have, planes + 3 * NF * HP};
        // a cell that prefetched nothing lies on a non-periodic face: the
        // update pulls with the boundary rules there
        Real fi, fo;
        accI += half_store::cell_update<3, K>(P, S, A, c, xyz, P0, dlnP0, dP0r, fi, fo);
        accIn += fi;
        accOut += fo;
      }
      __syncthreads();
      if constexpr (PRE) {
#pragma unroll
        for (int i = 0; i < L::Q; ++i) pre[i] = nxt[i];
        have = have_nxt;
      }
    }
  }
  double sI, sIn, sOut;
  block_sum3<Real>(accI, accIn, accOut, flux_block, red_sh, sI, sIn, sOut);
  publish_partials<4>(sI, sIn, sOut, S.partials, S.counter, S.scal, p0_closed, false, 0.0, P.eos_c,
                   P.inv_rho_ref);
}

// ------------------------------------------------------------ batch
template <int CFG> struct BatchShape;
template <> struct BatchShape<0> { using T = Tile<2, 32, 1>; };
template <> struct BatchShape<1> { using T = Tile<2, 32, 2>; };
template <> struct BatchShape<2> { using T = Tile<2, 64, 1>; };

template <int K, class T_>
__global__ void __launch_bounds__(BLOCK, (T_::RPT > 1 ? 3 : 4))
batch_step_kernel(const BatchDom<K, Real, Store>* __restrict__ doms,
                  const int* __restrict__ tile_begin, int /* run: 1 */, int ndom, int flip,
                  unsigned* __restrict__ tile_ctr) {
  using PL = Plane<2, K, T_::HP>;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  PL* planes = reinterpret_cast<PL*>(smem_raw);
  __shared__ double red_sh[96];
  __shared__ Params<Real, K> Psh;
  __shared__ State<Real, Store> Ssh;
  __shared__ int p0c_sh;
  __shared__ int next_sh[2];

  const int total = tile_begin[ndom];
  unsigned* ctr = tile_ctr + flip;
  if (threadIdx.x == 0) {
    if (blockIdx.x == 0) tile_ctr[flip ^ 1] = 0u;  // the next launch's counter
    next_sh[0] = (int)atomicAdd(ctr, 1u);
  }
  __syncthreads();
  int cur_dom = -1, par = 0;
  for (int t = next_sh[0]; t < total; t = next_sh[par]) {
    // domain of tile t: the last d with tile_begin[d] <= t
    int lo = 0, hi = ndom - 1;
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (__ldg(tile_begin + mid) <= t) lo = mid;
      else hi = mid - 1;
    }
    if (lo != cur_dom) {
      __syncthreads();  // the previous tile is done with the shared copies
      const BatchDom<K, Real, Store>& D = doms[lo];
      constexpr int PW = sizeof(Params<Real, K>) / 4;
      const uint32_t* src = reinterpret_cast<const uint32_t*>(&D.P);
      uint32_t* dst = reinterpret_cast<uint32_t*>(&Psh);
      for (int i = threadIdx.x; i < PW; i += blockDim.x) dst[i] = __ldg(src + i);
      if (threadIdx.x == 0) {
        Ssh = D.S[D.cur0 ^ flip];
        p0c_sh = D.p0_closed;
      }
      __syncthreads();
      cur_dom = lo;
    }
    // draw the next tile now; the tile's staging barrier publishes it
    par ^= 1;
    if (threadIdx.x == 0) next_sh[par] = (int)atomicAdd(ctr, 1u);
    const int lt = t - tile_begin[lo];
    const int nbx = (Psh.nx + T_::TX - 1) / T_::TX;
    double sI, sIn, sOut;
    half_store::step_tile<2, K, T_>(Psh, Ssh, lt % nbx, lt / nbx, 0, 1, planes, red_sh, sI, sIn,
                                     sOut);
    const unsigned nb = (unsigned)(tile_begin[lo + 1] - tile_begin[lo]);
    publish_partials_at<4>(sI, sIn, sOut, Ssh.partials, Ssh.counter, Ssh.scal, p0c_sh, false, 0.0,
                        Psh.eos_c, Psh.inv_rho_ref, (unsigned)lt, nb, true);
  }
}

}  // namespace half_store
}  // namespace pflb
