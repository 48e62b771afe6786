// pflb_step3d.cuh -- the fused step of 3-D lattices: blocks march along z.
//
// The same per-cell update as the 2-D step (cell_update), organised for D3Q19:
//   - work is cut into T = tiles x nz tile-planes, z innermost.  Long domains
//     (chunk > 0) hand out runs of planes to blocks in launch order, long runs
//     first and ever shorter ones last (chunk_count), so that tiles with
//     boundary cells, which cost more, do not leave SMs idle at the end; a run
//     stages two halo planes, about the work of two planes.  Short domains
//     (chunk = 0) take equal runs: block b of a resident grid owns
//     [b T / G, (b + 1) T / G).  Lengths and times: LauncherImpl::first_chunk;
//   - a ring of three staged planes in shared memory;
//   - PRE: the 19 populations of the plane are issued before the next plane is
//     staged, so the two load phases overlap; otherwise after the staging
//     barrier, which holds fewer registers across it.
// The block sums of the whole run are published once into slot blockIdx.x.
#pragma once

#include "pflb_kernels.cuh"

namespace pflb {

// The 3-D tile of the march and the resident blocks per SM it is compiled for:
// 32 x 8 cells, in FP32 a pair per thread (128 threads, 168 registers: the
// 256 x 128 x 128 bed takes 295 us a step in equal runs; 32 x 16 cells in 256
// threads at 128 registers spill, 405 us), in FP64 one.
template <class Real> struct MarchTile {
  using T = Tile<typename VecOf<Real>::V, 32, 8>;
  static constexpr int MINB = sizeof(Real) == 8 ? 1 : 3;
};

template <int K, class Real, bool PRE>
__global__ void __launch_bounds__(MarchTile<Real>::T::NT, MarchTile<Real>::MINB)
step3d_march_kernel(const __grid_constant__ Params<Real, K> P, const State<Real, Real> S,
                    int p0_closed, const double* __restrict__ prev_partials, unsigned prev_nb,
                    int chunk) {
  using T_ = typename MarchTile<Real>::T;
  using V = typename T_::V;
  constexpr int Q = Lattice<3>::Q, LN = T_::LN;
  constexpr int PLANE = (F_Y0 + K) * T_::HP;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  Real* planes = reinterpret_cast<Real*>(smem_raw);  // [3][fields][HP]
  __shared__ double red_sh[128];

  if (prev_partials && blockIdx.x == 0) {
    combine_partials_block<slots_in_flight(K)>(prev_partials, prev_nb, S.scal, P.eos_c,
                                               P.inv_rho_ref, red_sh);
    // the block's own sums go to red_sh next; a block without planes meets no
    // other barrier before them
    __syncthreads();
  }

  const Real P0 = scal_P0<Real>(S.scal);
  const Real dlnP0 = scal_dlnP0<Real>(S.scal);
  const Real dP0r = scal_dP0r<Real>(S.scal);

  const int tiles_x = (P.nx + T_::TX - 1) / T_::TX;
  const int tiles = tiles_x * ((P.ny + T_::TY - 1) / T_::TY);
  const long long total = (long long)tiles * P.nz;
  long long gi, g_end;
  if (chunk > 0) {
    const ZRun r = z_run(blockIdx.x, tiles, P.nz, chunk);
    gi = (long long)r.tile * P.nz + r.z_begin;
    g_end = gi + (r.z_end - r.z_begin);
  } else {
    gi = total * blockIdx.x / gridDim.x;
    g_end = total * (blockIdx.x + 1) / gridDim.x;
  }
  const int tx = (threadIdx.x % T_::TXT) * LN, ty = threadIdx.x / T_::TXT;
  const int h = (ty + 1) * T_::HX + tx + T_::XO;
  const bool even = LN == 1 || S.even;

  V accI = splat<V>(Real(0));
  Real accIn = 0, accOut = 0;
  double fuel = 0.0;
  bool flux_block = false;
  while (gi < g_end) {
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
    Real* pm = planes + ((z_begin + 2) % 3) * PLANE;
    Real* pc = planes + (z_begin % 3) * PLANE;
    Real* pp = planes + ((z_begin + 1) % 3) * PLANE;
    stage_plane<3, K, Real, T_>(P, S, pm, x0, y0, z_begin - 1, P0);
    stage_plane<3, K, Real, T_>(P, S, pc, x0, y0, z_begin, P0);
    for (int z = z_begin; z < z_end; ++z) {
      V g[Q];
      if (PRE && in_xy) load_pops<3, K, Real, V>(P, S, x, y, z, g);
      stage_plane<3, K, Real, T_>(P, S, pp, x0, y0, z + 1, P0);
      __syncthreads();
      if (in_xy) {
        if (!PRE) load_pops<3, K, Real, V>(P, S, x, y, z, g);
        const CellPos q{x + P.nx * (y + P.ny * z), x, y, z, even, x + 1 < P.nx};
        const PlaneAcc<Real, T_> A{pc, pm, pp, h, nullptr};
        Real fi, fo;
        accI = vadd(accI, cell_update<3, K, Real, V>(P, S, A, g, q, P0, dlnP0, dP0r, fi, fo,
                                                       fuel));
        accIn += fi;
        accOut += fo;
      }
      __syncthreads();
      Real* t = pm;
      pm = pc;
      pc = pp;
      pp = t;
    }
  }
  double sI, sIn, sOut, sF;
  block_sum4(accI, accIn, accOut, flux_block, fuel, K > 0 && P.feed, red_sh, sI, sIn, sOut, sF);
  publish_partials<slots_in_flight(K)>(sI, sIn, sOut, S.partials, S.counter, S.scal, p0_closed,
                                       false, 0.0, P.eos_c, P.inv_rho_ref, sF,
                                       K > 0 && P.feed ? P.feed_c : 0.0);
}

}  // namespace pflb
