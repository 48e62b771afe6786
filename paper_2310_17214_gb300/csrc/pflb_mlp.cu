// pflb_mlp.cu -- training and inference kernels of the chemistry-surrogate MLP
// and their C ABI (pflb_mlp_*, declared in include/pflb.h).
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <new>
#include <vector>

#include "../../include/pflb.h"
#include "pflb_mlp.cuh"

using namespace pflb::mlp;

struct pflb_mlp {
  int device = 0;
  cudaStream_t stream = nullptr;
  float* theta = nullptr;  // FP32 master parameters
  float* m = nullptr;      // Adam moments
  float* v = nullptr;
  float* grad = nullptr;   // gradient
  float* part = nullptr;   // the blocks' partial gradients [MAX_PART][NPARAM]
  double* loss = nullptr;  // loss, then the blocks' partial losses [MAX_PART]
  __nv_bfloat16* wf = nullptr;
  __nv_bfloat16* wb = nullptr;
  float* bias = nullptr;
  long long t = 0;         // Adam step count
};

namespace {

// Programmatic dependent launch: a kernel launched that way may start while the
// kernel before it in the stream is finishing.  pdl_wait holds it until that
// kernel has completed and its writes are visible (nothing is read or written
// before); pdl_trigger lets the kernel after this one start once every block
// has called it or ended.  Both do nothing in an ordinary launch.  A training step
// is two short kernels that wait for each other; started this way they hide
// their launches and prologues (a step of 8,192 rows: 25 -> 20 us with the
// changes beside it).
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
template <class... P, class... A>
cudaError_t launch_dependent(void (*kern)(P...), dim3 grid, unsigned threads, size_t smem,
                             cudaStream_t st, const A&... args) {
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, P(args)...);
}

constexpr int TW = 4;                // warps per block in the training kernel
constexpr int TROWS = 16 * TW;       // rows per block and iteration
constexpr int HLD = 72;              // row stride of the BF16 tiles: ldmatrix without conflicts
constexpr int MAX_PART = 256;        // blocks (partial gradients) of one mini-batch

// Activations and output gradients of the block's rows, kept for the weight
// gradients; XLD (24) and 8 are free of conflicts too.
struct TrainSmem {
  SmemNet net;
  __nv_bfloat16 x[TROWS * XLD];
  __nv_bfloat16 h[3][TROWS * HLD];
  __nv_bfloat16 dz[3][TROWS * HLD];  // dZ1..dZ3
  __nv_bfloat16 dO[TROWS * 8];
  float db[TW][NPB];                 // bias gradients per warp (padded layout)
  double loss[TW];
};

// Padded BF16 copies of the FP32 parameters (both layouts) and biases.
__global__ void pack_kernel(const float* __restrict__ theta, __nv_bfloat16* __restrict__ wf,
                            __nv_bfloat16* __restrict__ wb, float* __restrict__ bias) {
  for (int idx = blockIdx.x * blockDim.x + threadIdx.x; idx < NPAD + NPB;
       idx += gridDim.x * blockDim.x) {
    if (idx >= NPAD) {
      const int q = idx - NPAD;
      int l = 0;
      while (l < NL - 1 && q >= pboff(l + 1)) ++l;
      const int o = q - pboff(l);
      bias[q] = o < dim(l + 1) ? theta[boff(l) + o] : 0.f;
      continue;
    }
    int l = 0;
    while (l < NL - 1 && idx >= poff(l + 1)) ++l;
    const int r = idx - poff(l), IN = pdim(l), OUT = pdim(l + 1);
    // forward layout: B fragments in lane order (see Net)
    {
      const int e = r & 3, lane = (r >> 2) & 31, tile = r >> 7, KT = IN / 16;
      const int j = tile / KT, kk = tile % KT;
      const int o = 8 * j + (lane >> 2);
      const int i = 16 * kk + 2 * (lane & 3) + (e & 1) + (e >= 2 ? 8 : 0);
      const float w = (i < dim(l) && o < dim(l + 1)) ? theta[woff(l) + i * dim(l + 1) + o] : 0.f;
      wf[idx] = __float2bfloat16_rn(w);
    }
    // backward layout [in][out]
    {
      const int i = r / OUT, o = r % OUT;
      const float w = (i < dim(l) && o < dim(l + 1)) ? theta[woff(l) + i * dim(l + 1) + o] : 0.f;
      wb[idx] = __float2bfloat16_rn(w);
    }
  }
}

// Stage 16 normalised input rows (features 0..7, 8..15 zero) into a BF16
// [16][XLD] tile.
__device__ __forceinline__ void stage_x(__nv_bfloat16* x16, const float* __restrict__ X,
                                        long long row0, long long n) {
  const int lane = threadIdx.x & 31;
  const int r = lane >> 1, half = lane & 1;
  const long long row = row0 + r;
  float v[4];
#pragma unroll
  for (int f = 0; f < 4; ++f) v[f] = row < n ? X[row * 8 + half * 4 + f] : 0.f;
  uint32_t* q = reinterpret_cast<uint32_t*>(x16 + r * XLD);
  q[2 * half] = pack_bf16(v[0], v[1]);
  q[2 * half + 1] = pack_bf16(v[2], v[3]);
  q[4 + 2 * half] = 0u;
  q[5 + 2 * half] = 0u;
}

__device__ __forceinline__ float bf(const __nv_bfloat16 v) { return __bfloat162float(v); }

// Four 8 x 8 BF16 matrices, transposed on the way (lane l passes the address of
// row l & 7 of matrix l >> 3).
__device__ __forceinline__ void ldsm_t(uint32_t r[4], const __nv_bfloat16* p) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(static_cast<unsigned>(__cvta_generic_to_shared(p))));
}

// acc[nt] += A^T dZ over the block's rows for inputs m0..m0+15 and the n-tiles
// n0 + 8 nt: A is [rows][LDA], dZ [rows][LDB] (contraction over rows, so both
// operands are read transposed).
template <int NT, int LDA, int LDB>
__device__ __forceinline__ void grad_w(const __nv_bfloat16* A, int m0, const __nv_bfloat16* dZ,
                                       int n0, float acc[NT][4]) {
  const int lane = threadIdx.x & 31, i = lane >> 3, r = lane & 7;
#pragma unroll
  for (int k0 = 0; k0 < TROWS; k0 += 16) {
    uint32_t a[4], b[4];
    ldsm_t(a, A + (k0 + r + (i >= 2 ? 8 : 0)) * LDA + m0 + (i & 1) * 8);
    if constexpr (NT == 1) {
      // one n-tile: its two k-halves (twice)
      ldsm_t(b, dZ + (k0 + r + (i & 1) * 8) * LDB + n0);
      mma16816(acc[0], a, b[0], b[1]);
    } else {
#pragma unroll
      for (int nt = 0; nt < NT; nt += 2) {
        ldsm_t(b, dZ + (k0 + r + (i & 1) * 8) * LDB + n0 + 8 * nt + (i >= 2 ? 8 : 0));
        mma16816(acc[nt], a, b[0], b[1]);
        mma16816(acc[nt + 1], a, b[2], b[3]);
      }
    }
  }
}

// Weight gradients of layer L held as fragments (inputs m0 + g, + 8) into the
// block's partial gradient.
template <int L, int NT>
__device__ __forceinline__ void store_w(float* __restrict__ part, int m0, int n0,
                                        const float acc[NT][4]) {
  const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
#pragma unroll
  for (int nt = 0; nt < NT; ++nt)
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int m = m0 + g + (e >> 1) * 8, n = n0 + 8 * nt + 2 * t + (e & 1);
      if (m < dim(L) && n < dim(L + 1)) part[woff(L) + m * dim(L + 1) + n] = acc[nt][e];
    }
}

// Bias gradient: column sums of the 16 x OUT fragment set (rows g, g + 8),
// added to the warp's own sums.
template <int L, int NT>
__device__ __forceinline__ void grad_b(const float acc[][4], float* db) {
  const int lane = threadIdx.x & 31, t = lane & 3;
#pragma unroll
  for (int j = 0; j < NT; ++j) {
    float s0 = acc[j][0] + acc[j][2], s1 = acc[j][1] + acc[j][3];
#pragma unroll
    for (int o = 4; o < 32; o <<= 1) {
      s0 += __shfl_xor_sync(0xffffffffu, s0, o);
      s1 += __shfl_xor_sync(0xffffffffu, s1, o);
    }
    if (lane < 4) {
      db[pboff(L) + 8 * j + 2 * t] += s0;
      db[pboff(L) + 8 * j + 2 * t + 1] += s1;
    }
  }
}

// Store a 16 x 64 fragment set as a BF16 [16][HLD] tile.
__device__ __forceinline__ void store_tile(__nv_bfloat16* T, const float acc[8][4]) {
  const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    *reinterpret_cast<uint32_t*>(T + g * HLD + 8 * j + 2 * t) = pack_bf16(acc[j][0], acc[j][1]);
    *reinterpret_cast<uint32_t*>(T + (g + 8) * HLD + 8 * j + 2 * t) =
        pack_bf16(acc[j][2], acc[j][3]);
  }
}

// dH = dZ_next W^T (dZ_next as A fragments, W from the backward layout), then
// dZ = dH (1 - H^2) with H read back from the warp's tile.
template <int L>
__device__ __forceinline__ void back_dx(const SmemNet& s, const uint32_t* a, const __nv_bfloat16* H,
                                        float acc[8][4]) {
  constexpr int IN = pdim(L), OUT = pdim(L + 1);  // W_L is IN x OUT; dX has IN = 64 columns
  const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const __nv_bfloat16* W = s.wb + poff(L);
#pragma unroll
  for (int j = 0; j < IN / 8; ++j) {
    acc[j][0] = acc[j][1] = acc[j][2] = acc[j][3] = 0.f;
#pragma unroll
    for (int kk = 0; kk < (OUT + 15) / 16; ++kk) {
      const __nv_bfloat16* wr = W + (8 * j + g) * OUT + 16 * kk + 2 * t;
      const uint32_t b0 = (16 * kk + 2 * t < OUT) ? *reinterpret_cast<const uint32_t*>(wr) : 0u;
      const uint32_t b1 = (16 * kk + 8 + 2 * t < OUT) ? *reinterpret_cast<const uint32_t*>(wr + 8) : 0u;
      mma16816(acc[j], a + 4 * kk, b0, b1);
    }
    const __nv_bfloat162 ha = *reinterpret_cast<const __nv_bfloat162*>(H + g * HLD + 8 * j + 2 * t);
    const __nv_bfloat162 hb =
        *reinterpret_cast<const __nv_bfloat162*>(H + (g + 8) * HLD + 8 * j + 2 * t);
    const float h0 = bf(ha.x), h1 = bf(ha.y), h2 = bf(hb.x), h3 = bf(hb.y);
    acc[j][0] *= 1.f - h0 * h0;
    acc[j][1] *= 1.f - h1 * h1;
    acc[j][2] *= 1.f - h2 * h2;
    acc[j][3] *= 1.f - h3 * h3;
  }
}

// Asynchronous 16-byte copies of NV vectors by the block.
template <int NV>
__device__ __forceinline__ void copy16(void* dst, const void* src) {
  for (int i = threadIdx.x; i < NV; i += TW * 32)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                     static_cast<unsigned>(__cvta_generic_to_shared(dst)) + 16u * i),
                 "l"(static_cast<const char*>(src) + 16 * (size_t)i)
                 : "memory");
}

// Forward + backward of mini-batch rows: the block's part of the gradient of
// the mean squared error (scaled by inv_norm = 1 / (rows x 6)) and of the loss,
// into slot blockIdx.x.
//
// A warp carries 16 rows through forward and backward in registers; the weight
// gradients contract over the block's 64 rows, each warp owning 16 inputs of
// every layer, and stay in registers over the block's iterations.  One partial
// gradient per block goes to memory; update_kernel sums them in a fixed order
// (with a shared-memory and a global atomic per element and tile instead, and
// the network loaded one dependent word at a time, a mini-batch of 8,192 rows
// took 73 us, and takes 20).  What is left is latency: a few hundred dependent
// tensor-core and tanh steps of one wave of blocks, twice a launch.
__global__ void __launch_bounds__(TW * 32, 1)
grad_kernel(Net net, const float* __restrict__ X, const float* __restrict__ Y, long long n,
            float inv_norm, float* __restrict__ part, double* __restrict__ loss) {
  extern __shared__ __align__(16) unsigned char smem[];
  TrainSmem& S = *reinterpret_cast<TrainSmem*>(smem);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  for (int i = lane; i < NPB; i += 32) S.db[warp][i] = 0.f;
  pdl_wait();  // the parameters of the update before
  pdl_trigger();
  // the network, every copy in flight at once
  copy16<NPAD * 2 / 16>(S.net.wf, net.wf);
  copy16<NPAD * 2 / 16>(S.net.wb, net.wb);
  copy16<NPB * 4 / 16>(S.net.bias, net.bias);
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncthreads();
  float w1[2][4] = {}, w2[8][4] = {}, w3[8][4] = {}, w4[1][4] = {};
  float lsum = 0.f;
  __nv_bfloat16* x = S.x + warp * 16 * XLD;
  __nv_bfloat16* dO = S.dO + warp * 16 * 8;
  auto H = [&](int l) { return S.h[l] + warp * 16 * HLD; };
  auto DZ = [&](int l) { return S.dz[l] + warp * 16 * HLD; };
  for (long long row_blk = (long long)blockIdx.x * TROWS; row_blk < n;
       row_blk += (long long)gridDim.x * TROWS) {
    const long long row0 = row_blk + warp * 16;
    stage_x(x, X, row0, n);
    __syncwarp();
    // forward, keeping H1..H3
    uint32_t a[16];
    x_frags(x, XLD, a);
    float acc[8][4];
    layer_fwd<0>(S.net.wf, S.net.bias, a, acc);
    to_a<true>(acc, a);
    store_tile(H(0), acc);
    layer_fwd<1>(S.net.wf, S.net.bias, a, acc);
    to_a<true>(acc, a);
    store_tile(H(1), acc);
    layer_fwd<2>(S.net.wf, S.net.bias, a, acc);
    to_a<true>(acc, a);
    store_tile(H(2), acc);
    float o[1][4];
    layer_fwd<3>(S.net.wf, S.net.bias, a, o);
    // output gradient 2 (o - y) / (rows x 6)
    const long long rr[2] = {row0 + g, row0 + g + 8};
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const long long row = rr[e >> 1];
      const int col = 2 * t + (e & 1);
      float d = 0.f;
      if (row < n && col < 6) {
        const float diff = o[0][e] - Y[row * 6 + col];
        lsum += diff * diff;
        d = 2.f * diff * inv_norm;
      }
      o[0][e] = d;
    }
    uint32_t ad[16];
    ad[0] = pack_bf16(o[0][0], o[0][1]);
    ad[1] = pack_bf16(o[0][2], o[0][3]);
    ad[2] = ad[3] = 0u;
    *reinterpret_cast<uint32_t*>(dO + g * 8 + 2 * t) = ad[0];
    *reinterpret_cast<uint32_t*>(dO + (g + 8) * 8 + 2 * t) = ad[1];
    __syncwarp();
    grad_b<3, 1>(o, S.db[warp]);
    back_dx<3>(S.net, ad, H(2), acc);  // dZ3
    store_tile(DZ(2), acc);
    grad_b<2, 8>(acc, S.db[warp]);
    to_a<false>(acc, ad);
    back_dx<2>(S.net, ad, H(1), acc);  // dZ2
    store_tile(DZ(1), acc);
    grad_b<1, 8>(acc, S.db[warp]);
    to_a<false>(acc, ad);
    back_dx<1>(S.net, ad, H(0), acc);  // dZ1
    store_tile(DZ(0), acc);
    grad_b<0, 8>(acc, S.db[warp]);
    __syncthreads();
    // weight gradients of the block's rows: inputs 16 warp .. 16 warp + 15 of
    // W2..W4, outputs 16 warp .. of W1
    grad_w<2, XLD, HLD>(S.x, 0, S.dz[0], 16 * warp, w1);
    grad_w<8, HLD, HLD>(S.h[0], 16 * warp, S.dz[1], 0, w2);
    grad_w<8, HLD, HLD>(S.h[1], 16 * warp, S.dz[2], 0, w3);
    grad_w<1, HLD, 8>(S.h[2], 16 * warp, S.dO, 0, w4);
    __syncthreads();
  }
  float* p = part + (size_t)blockIdx.x * NPARAM;
  store_w<0, 2>(p, 0, 16 * warp, w1);
  store_w<1, 8>(p, 16 * warp, 0, w2);
  store_w<2, 8>(p, 16 * warp, 0, w3);
  store_w<3, 1>(p, 16 * warp, 0, w4);
#pragma unroll
  for (int o2 = 16; o2 > 0; o2 >>= 1) lsum += __shfl_xor_sync(0xffffffffu, lsum, o2);
  if (lane == 0) S.loss[warp] = (double)lsum;
  __syncthreads();
  for (int q = threadIdx.x; q < NPB; q += TW * 32) {
    int l = 0;
    while (l < NL - 1 && q >= pboff(l + 1)) ++l;
    const int o = q - pboff(l);
    float v = 0.f;
#pragma unroll
    for (int w = 0; w < TW; ++w) v += S.db[w][q];
    if (o < dim(l + 1)) p[boff(l) + o] = v;
  }
  if (threadIdx.x == 0) {
    double v = 0.0;
#pragma unroll
    for (int w = 0; w < TW; ++w) v += S.loss[w];
    loss[blockIdx.x] = v;
  }
}

// Where parameter i sits in the padded layouts (see Net): forward and backward
// BF16 weights, or the bias (w = false, its index in f).
struct Place {
  bool w;
  int f, b;
};
__device__ __forceinline__ Place place_of(int i) {
  int l = 0;
  while (l < NL - 1 && i >= woff(l + 1)) ++l;
  const int r = i - woff(l), OUT = dim(l + 1);
  if (r >= dim(l) * OUT) return {false, pboff(l) + r - dim(l) * OUT, 0};
  const int in = r / OUT, o = r - in * OUT, KT = pdim(l) / 16;
  const int k = in & 15, h = k & 7;
  const int lane = (o & 7) * 4 + (h >> 1), e = (h & 1) + (k >= 8 ? 2 : 0);
  return {true, poff(l) + (((o >> 3) * KT + (in >> 4)) * 32 + lane) * 4 + e,
          poff(l) + in * pdim(l + 1) + o};
}

// Sum of the blocks' partial gradients (fixed order: eight slices of the
// blocks, then the slices) and, with ADAM, the parameter update and its copies
// in the network's layouts, with the loss of the mini-batch summed beside.
constexpr int UP = 32, US = 8;  // parameters and slices per block
template <bool ADAM>
__global__ void __launch_bounds__(UP * US)
update_kernel(const float* __restrict__ part, int nb, const double* __restrict__ block_loss,
              double* __restrict__ loss, float* __restrict__ grad, float* __restrict__ theta,
              float* __restrict__ m, float* __restrict__ v, __nv_bfloat16* __restrict__ wf,
              __nv_bfloat16* __restrict__ wb, float* __restrict__ bias, float lr, float c1,
              float c2) {
  __shared__ float sh[US][UP];
  const int q = threadIdx.x % UP, s = threadIdx.x / UP, i = blockIdx.x * UP + q;
  float sum = 0.f;
  pdl_wait();
  pdl_trigger();
  if (i < NPARAM) {
    const int b0 = nb * s / US, b1 = nb * (s + 1) / US;
#pragma unroll 16
    for (int b = b0; b < b1; ++b) sum += part[(size_t)b * NPARAM + i];
  }
  sh[s][q] = sum;
  __syncthreads();
  if (s == 0 && i < NPARAM) {
    const float gi = ((sh[0][q] + sh[1][q]) + (sh[2][q] + sh[3][q])) +
                     ((sh[4][q] + sh[5][q]) + (sh[6][q] + sh[7][q]));
    if constexpr (!ADAM) {
      grad[i] = gi;
    } else {
      const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
      const float mi = b1 * m[i] + (1.f - b1) * gi;
      const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
      m[i] = mi;
      v[i] = vi;
      const float th = theta[i] - lr * (mi * c1) / (sqrtf(vi * c2) + eps);
      theta[i] = th;
      const Place p = place_of(i);
      if (p.w) {
        const __nv_bfloat16 w = __float2bfloat16_rn(th);
        wf[p.f] = w;
        wb[p.b] = w;
      } else {
        bias[p.f] = th;
      }
    }
  }
  if (blockIdx.x == 0 && threadIdx.x < 32) {
    double l = 0.0;
    for (int b = threadIdx.x; b < nb; b += 32) l += block_loss[b];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) l += __shfl_down_sync(0xffffffffu, l, o);
    if (threadIdx.x == 0) *loss = l;
  }
}

// Stage 32 normalised input rows into a BF16 [32][XLD] tile (one row per
// lane; features 8..15 zero).
__device__ __forceinline__ void stage_x32(__nv_bfloat16* x, const float* __restrict__ X,
                                          long long row0, long long n) {
  const int lane = threadIdx.x & 31;
  const long long row = row0 + lane;
  float v[8];
  if (row < n) {
    const float4 p0 = *reinterpret_cast<const float4*>(X + row * 8);
    const float4 p1 = *reinterpret_cast<const float4*>(X + row * 8 + 4);
    v[0] = p0.x; v[1] = p0.y; v[2] = p0.z; v[3] = p0.w;
    v[4] = p1.x; v[5] = p1.y; v[6] = p1.z; v[7] = p1.w;
  } else {
#pragma unroll
    for (int f = 0; f < 8; ++f) v[f] = 0.f;
  }
  uint32_t* r = reinterpret_cast<uint32_t*>(x + lane * XLD);
#pragma unroll
  for (int f = 0; f < 4; ++f) r[f] = pack_bf16(v[2 * f], v[2 * f + 1]);
#pragma unroll
  for (int f = 4; f < 8; ++f) r[f] = 0u;
}

__global__ void __launch_bounds__(256, 2)
forward_kernel(Net net, const float* __restrict__ X, float* __restrict__ out, long long n) {
  __shared__ SmemFwd s;
  __shared__ __align__(16) __nv_bfloat16 xs[8][32 * XLD];
  load_fwd(s, net);
  __syncthreads();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const long long tiles = (n + 31) / 32;
  for (long long tile = (long long)blockIdx.x * 8 + warp; tile < tiles;
       tile += (long long)gridDim.x * 8) {
    stage_x32(xs[warp], X, tile * 32, n);
    __syncwarp();
    float o[2][4];
    forward32(s, xs[warp], o[0], o[1]);
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const long long row = tile * 32 + 16 * h + g + (e >> 1) * 8;
        const int col = 2 * t + (e & 1);
        if (row < n && col < 6) out[row * 6 + col] = o[h][e];
      }
    __syncwarp();
  }
}

int grid_for(long long rows, int per_block) {
  long long b = (rows + per_block - 1) / per_block;
  if (b < 1) b = 1;
  if (b > 1184) b = 1184;
  return (int)b;
}

Net net_of(const pflb_mlp* m) { return Net{m->wf, m->wb, m->bias, m->theta}; }

// The partial gradients of n rows; returns their number.
int launch_grad(pflb_mlp* m, const float* X, const float* Y, long long n) {
  const int nb = (int)std::min<long long>((n + TROWS - 1) / TROWS, MAX_PART);
  launch_dependent(grad_kernel, dim3(nb), TW * 32, sizeof(TrainSmem), m->stream, net_of(m), X,
                   Y, n, 1.f / (float)(n * 6), m->part, m->loss + 1);
  return nb;
}

}  // namespace

namespace pflb {
// Network pointers of a handle (used by the surrogate chemistry pre-pass).
Net mlp_net(const pflb_mlp* m) { return net_of(m); }
}  // namespace pflb

extern "C" {

int pflb_mlp_create(int device, void* stream, pflb_mlp** out) {
  if (!out) return PFLB_ERR_ARG;
  *out = nullptr;
  if (cudaSetDevice(device) != cudaSuccess) return PFLB_ERR_CUDA;
  pflb_mlp* m = new (std::nothrow) pflb_mlp();
  if (!m) return PFLB_ERR_OOM;
  m->device = device;
  m->stream = static_cast<cudaStream_t>(stream);
  bool ok = cudaMalloc(&m->theta, NPARAM * 4) == cudaSuccess &&
            cudaMalloc(&m->m, NPARAM * 4) == cudaSuccess &&
            cudaMalloc(&m->v, NPARAM * 4) == cudaSuccess &&
            cudaMalloc(&m->grad, NPARAM * 4) == cudaSuccess &&
            cudaMalloc(&m->part, sizeof(float) * MAX_PART * NPARAM) == cudaSuccess &&
            cudaMalloc(&m->loss, (1 + MAX_PART) * sizeof(double)) == cudaSuccess &&
            cudaMalloc(&m->wf, NPAD * 2) == cudaSuccess &&
            cudaMalloc(&m->wb, NPAD * 2) == cudaSuccess &&
            cudaMalloc(&m->bias, NPB * 4) == cudaSuccess;
  if (!ok) {
    pflb_mlp_destroy(m);
    return PFLB_ERR_OOM;
  }
  cudaMemset(m->theta, 0, NPARAM * 4);
  cudaMemset(m->m, 0, NPARAM * 4);
  cudaMemset(m->v, 0, NPARAM * 4);
  cudaMemset(m->grad, 0, NPARAM * 4);
  cudaMemset(m->wf, 0, NPAD * 2);
  cudaMemset(m->wb, 0, NPAD * 2);
  cudaMemset(m->bias, 0, NPB * 4);
  if (cudaFuncSetAttribute(grad_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)sizeof(TrainSmem)) != cudaSuccess) {
    pflb_mlp_destroy(m);
    return PFLB_ERR_CUDA;
  }
  *out = m;
  return PFLB_OK;
}

int pflb_mlp_set_params(pflb_mlp* m, const float* theta) {
  if (!m || !theta) return PFLB_ERR_ARG;
  cudaSetDevice(m->device);
  if (cudaMemcpyAsync(m->theta, theta, NPARAM * 4, cudaMemcpyHostToDevice, m->stream) != cudaSuccess)
    return PFLB_ERR_CUDA;
  cudaMemsetAsync(m->m, 0, NPARAM * 4, m->stream);
  cudaMemsetAsync(m->v, 0, NPARAM * 4, m->stream);
  cudaMemsetAsync(m->grad, 0, NPARAM * 4, m->stream);
  m->t = 0;
  pack_kernel<<<(NPAD + NPB + 255) / 256, 256, 0, m->stream>>>(m->theta, m->wf, m->wb, m->bias);
  if (cudaGetLastError() != cudaSuccess) return PFLB_ERR_CUDA;
  return cudaStreamSynchronize(m->stream) == cudaSuccess ? PFLB_OK : PFLB_ERR_CUDA;
}

int pflb_mlp_get_params(pflb_mlp* m, float* theta) {
  if (!m || !theta) return PFLB_ERR_ARG;
  cudaSetDevice(m->device);
  if (cudaMemcpyAsync(theta, m->theta, NPARAM * 4, cudaMemcpyDeviceToHost, m->stream) != cudaSuccess)
    return PFLB_ERR_CUDA;
  return cudaStreamSynchronize(m->stream) == cudaSuccess ? PFLB_OK : PFLB_ERR_CUDA;
}

int pflb_mlp_forward(pflb_mlp* m, const float* X, float* out, long long n) {
  if (!m || !X || !out || n < 0 || (reinterpret_cast<uintptr_t>(X) & 15)) return PFLB_ERR_ARG;
  if (n == 0) return PFLB_OK;
  cudaSetDevice(m->device);
  forward_kernel<<<grid_for(n, 256), 256, 0, m->stream>>>(net_of(m), X, out, n);
  return cudaGetLastError() == cudaSuccess ? PFLB_OK : PFLB_ERR_CUDA;
}

int pflb_mlp_gradient(pflb_mlp* m, const float* X, const float* Y, long long n, float* grad,
                      double* loss) {
  if (!m || !X || !Y || n <= 0) return PFLB_ERR_ARG;
  cudaSetDevice(m->device);
  const int nb = launch_grad(m, X, Y, n);
  update_kernel<false><<<(NPARAM + UP - 1) / UP, UP * US, 0, m->stream>>>(
      m->part, nb, m->loss + 1, m->loss, m->grad, nullptr, nullptr, nullptr, nullptr, nullptr,
      nullptr, 0.f, 0.f, 0.f);
  if (cudaGetLastError() != cudaSuccess) return PFLB_ERR_CUDA;
  double l = 0;
  if (grad && cudaMemcpyAsync(grad, m->grad, NPARAM * 4, cudaMemcpyDeviceToHost, m->stream) != cudaSuccess)
    return PFLB_ERR_CUDA;
  if (cudaMemcpyAsync(&l, m->loss, sizeof(double), cudaMemcpyDeviceToHost, m->stream) != cudaSuccess ||
      cudaStreamSynchronize(m->stream) != cudaSuccess)
    return PFLB_ERR_CUDA;
  if (loss) *loss = l / (double)(n * 6);
  return PFLB_OK;
}

int pflb_mlp_train(pflb_mlp* m, const float* X, const float* Y, long long n, int batch, int steps,
                   float lr, double* last_loss) {
  if (!m || !X || !Y || n <= 0 || batch <= 0 || steps < 0) return PFLB_ERR_ARG;
  cudaSetDevice(m->device);
  const long long nb = (n + batch - 1) / batch;
  for (int s = 0; s < steps; ++s) {
    const long long b = s % nb;
    const long long r0 = b * batch;
    const long long rows = (r0 + batch <= n) ? batch : n - r0;
    const bool last = s == steps - 1;
    const int nblk = launch_grad(m, X + r0 * 8, Y + r0 * 6, rows);
    m->t += 1;
    const float c1 = 1.f / (1.f - powf(0.9f, (float)m->t));
    const float c2 = 1.f / (1.f - powf(0.999f, (float)m->t));
    launch_dependent(update_kernel<true>, dim3((NPARAM + UP - 1) / UP), UP * US, 0, m->stream,
                     m->part, nblk, m->loss + 1, m->loss, (float*)nullptr, m->theta, m->m,
                     m->v, m->wf, m->wb, m->bias, lr, c1, c2);
    if (last && last_loss) {
      double l = 0;
      cudaMemcpyAsync(&l, m->loss, sizeof(double), cudaMemcpyDeviceToHost, m->stream);
      cudaStreamSynchronize(m->stream);
      *last_loss = l / (double)(rows * 6);
    }
  }
  return cudaGetLastError() == cudaSuccess ? PFLB_OK : PFLB_ERR_CUDA;
}

int pflb_mlp_destroy(pflb_mlp* m) {
  if (!m) return PFLB_OK;
  cudaSetDevice(m->device);
  cudaStreamSynchronize(m->stream);
  void* p[] = {m->theta, m->m, m->v, m->grad, m->part, m->loss, m->wf, m->wb, m->bias};
  for (void* q : p)
    if (q) cudaFree(q);
  delete m;
  return PFLB_OK;
}

}  // extern "C"
