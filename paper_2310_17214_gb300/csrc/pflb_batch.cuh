// pflb_batch.cuh -- many 2-D domains advanced by one persistent kernel.
//
// Every domain keeps its own arrays; the batch holds a device work list with
// one entry per domain (its lattice-unit parameters, the two ping-pong views
// of its state, its P0 mode) and, per tile shape, the prefix sums of the
// domains' counts of runs of consecutive tiles.  A launch is a
// resident grid that draws runs from an atomic counter (one per launch parity;
// each launch clears the other one for the next launch), so blocks that draw
// cheap tiles take more of them and no SM idles at the end.  A block finds a
// run's domain by binary search, copies that domain's parameters into shared
// memory when it changes domain, and runs the same per-tile code as the
// single-domain step.  Each domain's reduction slots are its tile indices.  A
// block makes a run's slots visible and counts them once, and the block whose
// count completes a domain combines its slots at once, so a batch step leaves
// no deferred work behind and every domain's P0 is current for the next launch.
//
// Runs of tiles: the blocks advance through the tiles side by side, so with
// single tiles nearly every draw changed domain (a search, a copy of the
// parameters, two barriers) and every tile paid a fence.  The length of the runs
// follows the work there is (LauncherImpl::batch_run).
#pragma once

#include "pflb_half.cuh"
#include "pflb_kernels.cuh"

namespace pflb {

// Tile shapes the batch can run.
constexpr int BATCH_SHAPES = 3;
template <class Real, int CFG> struct BatchShape;
template <class Real> struct BatchShape<Real, 0> { using T = Tile<typename VecOf<Real>::V, 32, 8>; };
template <class Real> struct BatchShape<Real, 1> { using T = Tile<typename VecOf<Real>::V, 32, 16>; };
template <class Real> struct BatchShape<Real, 2> { using T = Tile<typename VecOf<Real>::V, 64, 4>; };

__host__ __device__ constexpr int batch_tx(int cfg) { return cfg == 2 ? 64 : 32; }
__host__ __device__ constexpr int batch_ty(int cfg) { return cfg == 0 ? 8 : (cfg == 1 ? 16 : 4); }

// most tiles of a run
constexpr int BATCH_RUN = 4;

template <int K, class Real, class T_>
__global__ void __launch_bounds__(T_::NT, (MinBlocks<K, T_>::value))
batch_step_kernel(const BatchDom<K, Real, Real>* __restrict__ doms,
                  const int* __restrict__ run_begin, int run, int ndom, int flip,
                  unsigned* __restrict__ run_ctr) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  Real* pl = reinterpret_cast<Real*>(smem_raw);
  __shared__ double red_sh[96];
  __shared__ Params<Real, K> Psh;
  __shared__ State<Real, Real> Ssh;
  __shared__ int p0c_sh;
  __shared__ int next_sh[2];

  const int total = run_begin[ndom];
  if (threadIdx.x == 0) {
    if (blockIdx.x == 0) run_ctr[flip ^ 1] = 0u;  // the next launch's counter
    next_sh[0] = (int)atomicAdd(run_ctr + flip, 1u);
  }
  __syncthreads();
  int dom = -1, par = 0;
  for (int r = next_sh[0]; r < total; r = next_sh[par]) {
    // domain of run r: the last d with run_begin[d] <= r
    int lo = 0, hi = ndom - 1;
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (__ldg(run_begin + mid) <= r) lo = mid;
      else hi = mid - 1;
    }
    if (lo != dom) {
      __syncthreads();  // the previous tile is done with the shared copies
      const BatchDom<K, Real, Real>& D = doms[lo];
      constexpr int PW = sizeof(Params<Real, K>) / 4;
      const uint32_t* src = reinterpret_cast<const uint32_t*>(&D.P);
      uint32_t* dst = reinterpret_cast<uint32_t*>(&Psh);
      for (int i = threadIdx.x; i < PW; i += blockDim.x) dst[i] = __ldg(src + i);
      if (threadIdx.x == 0) {
        Ssh = D.S[D.cur0 ^ flip];
        p0c_sh = D.p0_closed;
      }
      __syncthreads();
      dom = lo;
    }
    // draw the next run now; a tile's staging barrier publishes it
    par ^= 1;
    if (threadIdx.x == 0) next_sh[par] = (int)atomicAdd(run_ctr + flip, 1u);
    const int first = (r - __ldg(run_begin + lo)) * run;
#pragma unroll 1
    for (int i = 0; i < run; ++i) {
      const int nbx = (Psh.nx + T_::TX - 1) / T_::TX;
      if (first + i >= nbx * ((Psh.ny + T_::TY - 1) / T_::TY)) break;
      double sI, sIn, sOut, sF;
      step_tile<K, Real, T_>(Psh, Ssh, (first + i) % nbx, (first + i) / nbx, pl, red_sh, sI, sIn,
                             sOut, sF);
      write_partials(sI, sIn, sOut, Ssh.partials, (unsigned)(first + i));
    }
    const int nb = ((Psh.nx + T_::TX - 1) / T_::TX) * ((Psh.ny + T_::TY - 1) / T_::TY);
    count_partials<slots_in_flight(K)>(Ssh.partials, Ssh.counter, Ssh.scal, p0c_sh, false, 0.0,
                                       Psh.eos_c, Psh.inv_rho_ref, (unsigned)min(run, nb - first),
                                       (unsigned)nb);
  }
}

}  // namespace pflb
