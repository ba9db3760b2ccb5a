// The learned macro-step's network: forward pass, loss and gradient by
// backpropagation, and Adam, as hand-written kernels (bfloat16 matrices, FP32
// accumulation, on the tensor cores for the forward pass and for the weight
// gradients and propagated errors of the backward pass). Gradients are summed
// per block of 128 samples and the block partials in a fixed order, so results
// are reproducible.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cmath>
#include <new>
#include <string>
#include <vector>

#include "tfkt_fused.cuh"
#include "tfkt_mlp.cuh"

namespace tfkt {
namespace {

// Inference on raw samples: one warp per TC_ROWS samples, the network on the
// tensor cores (mlp_warp_tc).
__global__ void __launch_bounds__(128) forward_kernel(const float* __restrict__ master,
                                                      const __nv_bfloat16* __restrict__ wmat,
                                                      const float* __restrict__ X, int64_t n,
                                                      float* __restrict__ Y) {
  extern __shared__ __align__(16) unsigned char fw_smem[];
  MlpTc& s = *reinterpret_cast<MlpTc*>(fw_smem);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  float* Xw = reinterpret_cast<float*>(fw_smem + ((sizeof(MlpTc) + 15) & ~(size_t)15)) +
              (size_t)warp * TC_WARP_FLOATS;
  float* Ow = Xw + TC_ROWS * TC_XLD;
  mlp_stage_tc(s, master, wmat, threadIdx.x, blockDim.x);
  __syncthreads();
  const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;   // warp-uniform pass
  const bool ok = k < n;
  float* xr = Xw + lane * TC_XLD;
#pragma unroll
  for (int i = 0; i < NIN; ++i) xr[i] = ok ? (X[k * NIN + i] - s.mx[i]) * s.rsx[i] : 0.f;
#pragma unroll
  for (int i = NIN; i < TC_K1; ++i) xr[i] = 0.f;
  __syncwarp();
  mlp_warp_tc(s, Xw, Ow, lane);
  __syncwarp();
  if (ok) {
#pragma unroll
    for (int j = 0; j < NOUT; ++j) Y[k * NOUT + j] = Ow[lane * 4 + j] * s.st[j] + s.mt[j];
  }
}

// ---- training: forward and backward on the tensor cores
// A block of 8 warps takes TB = 128 samples at a time, one 16-row tile per warp, and
// the grid is at most one block per SM, so that a larger batch adds tiles to a block
// and no partials. The forward pass is the inference routine's (standardised inputs
// and GELU activations as bfloat16 high part plus remainder, bfloat16 weights, FP32
// accumulation), keeping activations and GELU derivatives per sample (the derivative
// shares its erff with the activation). Backward: the output layer, the bias sums and
// the GELU derivatives on the CUDA cores; the weight gradients dW2 = dz2^T h1 and
// dW1 = dz1^T x (sums over samples, in registers over all tiles of the block) and the
// propagated error dz2 W2 as mma.sync, both FP32 operands split into high part and
// remainder (three products per pair: high x high, high x remainder, remainder x high).
//
// Up to one tile per SM the launches, the wait for the loss and the chain through one
// tile (14 us, two warps per scheduler, a third of it the GELUs) bound a call, beyond
// that the tiles. 16384 samples took 72 us for loss, gradient and an Adam step with
// four warps per block, sums of 128 terms in one thread each (biases, output layer,
// loss, and the partials of all blocks per weight), strided loads of the samples and
// separate copies of loss and gradient; now 39. 65536 samples 196 and 81.
constexpr int TB = 128;          // samples of a tile
constexpr int TW = 8;            // warps of a block
constexpr int TT = 32 * TW;      // threads
constexpr int TR_LD = 68;        // FP32 row stride of the per-sample tables (float2-aligned)
constexpr int TQ = TT / NH;      // threads that share a column's sum over a tile's samples
constexpr int MAX_TRAIN_BLOCKS = 152;   // one per SM
static_assert(TB == 16 * TW && TT == 4 * NH, "tiling of the training kernel");

struct TrainTc {
  MlpTc net;                         // forward weights ([out][in] bfloat16) and normalisation
  __nv_bfloat16 w2t[NH * TC_W2LD];   // W2 transposed ([in][out]) for the propagated error
  float xs[TB * TC_XLD];             // standardised inputs; columns NIN .. TC_K1 - 1 zero
  // activations; GELU derivatives, then in their place dz1 and dz2
  float d1[TB * TR_LD], h1[TB * TR_LD], d2[TB * TR_LD], h2[TB * TR_LD];
  float o[TB * 4], dO[TB * 4];
  float part[TQ][5][NH];             // column sums of the threads that share a column
  float part3[TW][4];
  double lsum[TW];
};

// Fragment pair (p, q) of an FP32 table split into bfloat16 high part and remainder.
__device__ __forceinline__ void tr_split2(const float* p, const float* q, uint32_t& hi, uint32_t& lo) {
  tc_split(*p, *q, hi, lo);
}

// GELU(z) = z Phi(z) and its derivative Phi(z) + z phi(z).
__device__ __forceinline__ float gelu_and_grad(float z, float& d) {
  const float e = 1.0f + erff(z * 0.70710678118654752f);
  d = 0.5f * e + z * expf(-0.5f * z * z) * 0.39894228040143268f;
  return 0.5f * z * e;
}

// One hidden layer's activations and derivatives of the warp's rows r0 and r1 from
// its accumulators, kept in the tables h and d, and the next layer's operands.
__device__ __forceinline__ void train_activate(const float (&c)[8][4], float* h, float* d, int r0, int r1,
                                               int t, uint32_t (&ah)[4][4], uint32_t (&al)[4][4]) {
#pragma unroll
  for (int n = 0; n < 8; ++n) {
    const int col = 8 * n + 2 * t;
    float a[4], g[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) a[e] = gelu_and_grad(c[n][e], g[e]);
    *reinterpret_cast<float2*>(d + r0 * TR_LD + col) = make_float2(g[0], g[1]);
    *reinterpret_cast<float2*>(d + r1 * TR_LD + col) = make_float2(g[2], g[3]);
    *reinterpret_cast<float2*>(h + r0 * TR_LD + col) = make_float2(a[0], a[1]);
    *reinterpret_cast<float2*>(h + r1 * TR_LD + col) = make_float2(a[2], a[3]);
    const int k = n >> 1, half = (n & 1) * 2;
    tc_split(a[0], a[1], ah[k][half], al[k][half]);
    tc_split(a[2], a[3], ah[k][half + 1], al[k][half + 1]);
  }
}

// Operand fragments of rows r0 and r1 of an FP32 table, NK k-steps of 16 columns.
template <int NK, int LD>
__device__ __forceinline__ void train_rows(const float* x, int r0, int r1, int t, uint32_t (&ah)[NK][4],
                                           uint32_t (&al)[NK][4]) {
  const float* x0 = x + r0 * LD;
  const float* x1 = x + r1 * LD;
#pragma unroll
  for (int k = 0; k < NK; ++k) {
    const int c0 = 16 * k + 2 * t;
    tc_split(x0[c0], x0[c0 + 1], ah[k][0], al[k][0]);
    tc_split(x1[c0], x1[c0 + 1], ah[k][1], al[k][1]);
    tc_split(x0[c0 + 8], x0[c0 + 9], ah[k][2], al[k][2]);
    tc_split(x1[c0 + 8], x1[c0 + 9], ah[k][3], al[k][3]);
  }
}

// Forward pass of the warp's 16 samples (rows wb .. wb + 15 of the tables).
__device__ __forceinline__ void train_forward_warp(TrainTc& sh, int wb, int lane) {
  const MlpTc& s = sh.net;
  const int g = lane >> 2, t = lane & 3;
  const int r0 = wb + g, r1 = r0 + 8;
  uint32_t ah1[3][4], al1[3][4], ah[4][4], al[4][4];
  train_rows<3, TC_XLD>(sh.xs, r0, r1, t, ah1, al1);
  float c[8][4];
#pragma unroll
  for (int n = 0; n < 8; ++n) {
    c[n][0] = c[n][2] = s.b1[8 * n + 2 * t];
    c[n][1] = c[n][3] = s.b1[8 * n + 2 * t + 1];
  }
  tc_layer<3, 8, TC_W1LD>(c, ah1, al1, s.w1, g, t);
  train_activate(c, sh.h1, sh.d1, r0, r1, t, ah, al);
#pragma unroll
  for (int n = 0; n < 8; ++n) {
    c[n][0] = c[n][2] = s.b2[8 * n + 2 * t];
    c[n][1] = c[n][3] = s.b2[8 * n + 2 * t + 1];
  }
  tc_layer<4, 8, TC_W2LD>(c, ah, al, s.w2, g, t);
  train_activate(c, sh.h2, sh.d2, r0, r1, t, ah, al);
  float c3[1][4] = {{s.b3[2 * t], s.b3[2 * t + 1], s.b3[2 * t], s.b3[2 * t + 1]}};
  tc_layer<4, 1, TC_W2LD>(c3, ah, al, s.w3, g, t);
  if (2 * t < NOUT) {
    sh.o[r0 * 4 + 2 * t] = c3[0][0];
    sh.o[r1 * 4 + 2 * t] = c3[0][2];
  }
  if (2 * t + 1 < NOUT) {
    sh.o[r0 * 4 + 2 * t + 1] = c3[0][1];
    sh.o[r1 * 4 + 2 * t + 1] = c3[0][3];
  }
}

// c += sum over the tile's samples s of D[s][o] B[s][i] for o in 16 rows (o0 ..) and
// NN n-tiles of 8 columns i (i0 ..).
template <int NN>
__device__ __forceinline__ void train_weight_grad(float (&c)[NN][4], const float* D, const float* B,
                                                  int bld, int o0, int i0, int lane) {
  const int g = lane >> 2, t = lane & 3;
#pragma unroll 2
  for (int k = 0; k < TB / 16; ++k) {
    const int s0 = 16 * k + 2 * t;
    uint32_t ah[4], al[4];
    tr_split2(D + s0 * TR_LD + o0 + g, D + (s0 + 1) * TR_LD + o0 + g, ah[0], al[0]);
    tr_split2(D + s0 * TR_LD + o0 + g + 8, D + (s0 + 1) * TR_LD + o0 + g + 8, ah[1], al[1]);
    tr_split2(D + (s0 + 8) * TR_LD + o0 + g, D + (s0 + 9) * TR_LD + o0 + g, ah[2], al[2]);
    tr_split2(D + (s0 + 8) * TR_LD + o0 + g + 8, D + (s0 + 9) * TR_LD + o0 + g + 8, ah[3], al[3]);
#pragma unroll
    for (int n = 0; n < NN; ++n) {
      const int i = i0 + 8 * n + g;
      uint32_t bh0, bl0, bh1, bl1;
      tr_split2(B + s0 * bld + i, B + (s0 + 1) * bld + i, bh0, bl0);
      tr_split2(B + (s0 + 8) * bld + i, B + (s0 + 9) * bld + i, bh1, bl1);
      tc_mma(c[n], ah, bh0, bh1);
      tc_mma(c[n], ah, bl0, bl1);
      tc_mma(c[n], al, bh0, bh1);
    }
  }
}

// P[o * ld + i] = c for the columns i < ni.
template <int NN>
__device__ __forceinline__ void train_store(const float (&c)[NN][4], int o0, int i0, int ni, float* P, int ld,
                                            int lane) {
  const int g = lane >> 2, t = lane & 3;
#pragma unroll
  for (int n = 0; n < NN; ++n) {
    const int i = i0 + 8 * n + 2 * t;
    if (i < ni) {
      P[(o0 + g) * ld + i] = c[n][0];
      P[(o0 + g + 8) * ld + i] = c[n][2];
    }
    if (i + 1 < ni) {
      P[(o0 + g) * ld + i + 1] = c[n][1];
      P[(o0 + g + 8) * ld + i + 1] = c[n][3];
    }
  }
}

// Loss and gradient partials of a block's tiles of TB samples; partial[b][NWEIGHTS].
__global__ void __launch_bounds__(TT) loss_grad_kernel(const float* master,
                                                       const __nv_bfloat16* wmat,
                                                       const float* X,
                                                       const float* T, int64_t n,
                                                       float* __restrict__ partial,
                                                       double* __restrict__ lpart) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  TrainTc& sh = *reinterpret_cast<TrainTc*>(smem_raw);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int g = lane >> 2, t = lane & 3, wb = 16 * warp;
  let_successor_start();
  wait_for_predecessor();
  mlp_stage_tc(sh.net, master, wmat, tid, TT);
  for (int k = tid; k < NH * NH; k += TT) {   // (columns >= NH of w2t are never read)
    const int o = k / NH, i = k % NH;
    sh.w2t[i * TC_W2LD + o] = wmat[NH * NIN + k];
  }
  for (int k = tid; k < TB * (TC_XLD - NIN); k += TT)
    sh.xs[k / (TC_XLD - NIN) * TC_XLD + NIN + k % (TC_XLD - NIN)] = 0.0f;
  __syncthreads();
  const MlpTc& s = sh.net;
  const float inv_n = 1.0f / (float)n;
  // sums over the block's tiles: this warp's part of the matrices' gradients, and for
  // column `col` a quarter of the samples of db1, db2 and the three rows of dW3
  float cw1[3][4] = {}, cw2[4][4] = {};
  const int o0 = 16 * (warp & 3), half = warp >> 2;
  const int col = tid % NH, quarter = tid / NH;
  float sb1 = 0.0f, sb2 = 0.0f, sw3[NOUT] = {}, sb3[NOUT] = {};
  double lsq = 0.0;
  const int64_t ntiles = (n + TB - 1) / TB;
  for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    // ---- standardised inputs
    const int64_t k0 = tile * TB;
    const int rows = (int)(n - k0 < TB ? n - k0 : TB);
    for (int k = tid; k < TB * NIN; k += TT) {
      const int r = k / NIN, i = k % NIN;
      sh.xs[r * TC_XLD + i] = r < rows ? (X[k0 * NIN + k] - s.mx[i]) * s.rsx[i] : 0.0f;
    }
    __syncthreads();
    // ---- forward, and the error of the outputs, of the warp's own samples
    train_forward_warp(sh, wb, lane);
    __syncwarp();
    if (lane < 16) {
      const int r = wb + lane;
#pragma unroll
      for (int j = 0; j < NOUT; ++j) {
        float d = 0.0f;
        if (r < rows) {
          const float tj = (T[(k0 + r) * NOUT + j] - s.mt[j]) / s.st[j];
          const float e = sh.o[r * 4 + j] - tj;
          lsq += (double)e * (double)e;
          d = 2.0f * e * inv_n;
        }
        sh.dO[r * 4 + j] = d;
        sb3[j] += d;
      }
      sh.dO[r * 4 + 3] = 0.0f;
    }
    __syncwarp();
    // ---- dz2 = (W3^T dO) GELU'(z2), in place of the derivative
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int c = lane + 32 * u;
      float w[NOUT];
#pragma unroll
      for (int j = 0; j < NOUT; ++j) w[j] = __bfloat162float(s.w3[j * TC_W2LD + c]);
#pragma unroll 4
      for (int r = wb; r < wb + 16; ++r) {
        const float4 e = *reinterpret_cast<const float4*>(sh.dO + 4 * r);
        sh.d2[r * TR_LD + c] *= fmaf(w[2], e.z, fmaf(w[1], e.y, w[0] * e.x));
      }
    }
    __syncthreads();
    // ---- layer 2 and the output layer: dW2 = dz2^T h1, db2, dW3 = dO^T h2
    train_weight_grad<4>(cw2, sh.d2, sh.h1, TR_LD, o0, 32 * half, lane);
#pragma unroll 4
    for (int r = quarter * (TB / TQ); r < (quarter + 1) * (TB / TQ); ++r) {
      const float h = sh.h2[r * TR_LD + col];
      const float4 e = *reinterpret_cast<const float4*>(sh.dO + 4 * r);
      sw3[0] = fmaf(e.x, h, sw3[0]);
      sw3[1] = fmaf(e.y, h, sw3[1]);
      sw3[2] = fmaf(e.z, h, sw3[2]);
      sb2 += sh.d2[r * TR_LD + col];
    }
    // ---- dz1 = (dz2 W2) GELU'(z1) for the warp's samples, in place of the derivative
    {
      const int r0 = wb + g, r1 = r0 + 8;
      uint32_t ah[4][4], al[4][4];
      train_rows<4, TR_LD>(sh.d2, r0, r1, t, ah, al);
      float c[8][4] = {};
      tc_layer<4, 8, TC_W2LD>(c, ah, al, sh.w2t, g, t);
#pragma unroll
      for (int nn = 0; nn < 8; ++nn) {
        float2* z0 = reinterpret_cast<float2*>(sh.d1 + r0 * TR_LD + 8 * nn + 2 * t);
        float2* z1 = reinterpret_cast<float2*>(sh.d1 + r1 * TR_LD + 8 * nn + 2 * t);
        const float2 a = *z0, b = *z1;
        *z0 = make_float2(c[nn][0] * a.x, c[nn][1] * a.y);
        *z1 = make_float2(c[nn][2] * b.x, c[nn][3] * b.y);
      }
    }
    __syncthreads();
    // ---- layer 1: dW1 = dz1^T x (inputs padded to 48), db1
    train_weight_grad<3>(cw1, sh.d1, sh.xs, TC_XLD, o0, 24 * half, lane);
#pragma unroll 8
    for (int r = quarter * (TB / TQ); r < (quarter + 1) * (TB / TQ); ++r) sb1 += sh.d1[r * TR_LD + col];
    __syncthreads();   // the tables are overwritten by the next tile
  }
  // ---- the block's partials; shared sums in a fixed order
  float* P = partial + (size_t)blockIdx.x * TFKT_MLP_NWEIGHTS;
  train_store<4>(cw2, o0, 32 * half, NH, P + OW2, NH, lane);
  train_store<3>(cw1, o0, 24 * half, NIN, P + OW1, NIN, lane);
  sh.part[quarter][0][col] = sb1;
  sh.part[quarter][1][col] = sb2;
#pragma unroll
  for (int j = 0; j < NOUT; ++j) sh.part[quarter][2 + j][col] = sw3[j];
#pragma unroll
  for (int m = 8; m > 0; m >>= 1) {   // over the 16 lanes that hold samples
    lsq += __shfl_down_sync(0xffffffffu, lsq, m, 16);
#pragma unroll
    for (int j = 0; j < NOUT; ++j) sb3[j] += __shfl_down_sync(0xffffffffu, sb3[j], m, 16);
  }
  if (lane == 0) {
    sh.lsum[warp] = lsq;
#pragma unroll
    for (int j = 0; j < NOUT; ++j) sh.part3[warp][j] = sb3[j];
  }
  __syncthreads();
  for (int k = tid; k < 5 * NH; k += TT) {
    const int c = k % NH, v = k / NH;
    float a = sh.part[0][v][c];
#pragma unroll
    for (int q = 1; q < TQ; ++q) a += sh.part[q][v][c];
    P[v == 0 ? OB1 + c : (v == 1 ? OB2 + c : OW3 + (v - 2) * NH + c)] = a;
  }
  if (tid < NOUT) {
    float a = 0.0f;
    for (int w = 0; w < TW; ++w) a += sh.part3[w][tid];
    P[OB3 + tid] = a;
  }
  if (tid == 32) {
    double l = 0.0;
    for (int w = 0; w < TW; ++w) l += sh.lsum[w];
    lpart[blockIdx.x] = l;
  }
}

// grad[w] = sum over blocks of partial[b][w], eight threads per weight with an eighth
// of the blocks each, in a fixed order; loss = sum lpart / n by the last block. out:
// the caller's copy of the gradient, or null.
constexpr int RD_W = 32, RD_S = 8;   // weights and shares of a block
__global__ void __launch_bounds__(RD_W * RD_S) reduce_kernel(const float* partial, int nblocks,
                                                             float* __restrict__ grad,
                                                             float* __restrict__ out,
                                                             const double* lpart,
                                                             double* __restrict__ loss, int64_t n) {
  __shared__ float part[RD_S][RD_W];
  __shared__ double lp[RD_S];
  const int lane = threadIdx.x % RD_W, share = threadIdx.x / RD_W;
  let_successor_start();
  wait_for_predecessor();
  if (blockIdx.x == gridDim.x - 1) {   // the loss
    double l = 0.0;
    for (int b = threadIdx.x; b < nblocks; b += RD_W * RD_S) l += lpart[b];
#pragma unroll
    for (int m = 16; m > 0; m >>= 1) l += __shfl_down_sync(0xffffffffu, l, m);
    if (lane == 0) lp[share] = l;
    __syncthreads();
    if (threadIdx.x == 0) {
      double t = 0.0;
      for (int k = 0; k < RD_S; ++k) t += lp[k];
      *loss = t / (double)n;
    }
    return;
  }
  const int w = blockIdx.x * RD_W + lane;
  float a = 0.0f;
  if (w < TFKT_MLP_NWEIGHTS) {
    const int per = (nblocks + RD_S - 1) / RD_S;
    const int b1 = min(nblocks, (share + 1) * per);
#pragma unroll 8
    for (int b = share * per; b < b1; ++b) a += partial[(size_t)b * TFKT_MLP_NWEIGHTS + w];
  }
  part[share][lane] = a;
  __syncthreads();
  if (share == 0 && w < TFKT_MLP_NWEIGHTS) {
#pragma unroll
    for (int k = 1; k < RD_S; ++k) a += part[k][lane];
    grad[w] = a;
    if (out) out[w] = a;
  }
}

// Adam on the master weights; c1 = 1 / (1 - beta1^t), c2 = 1 / (1 - beta2^t).
__global__ void adam_kernel(float* master, __nv_bfloat16* __restrict__ wmat,
                            float* m, float* v,
                            const float* grad, float lr, float b1, float b2,
                            float eps, float c1, float c2) {
  const int w = blockIdx.x * blockDim.x + threadIdx.x;
  let_successor_start();
  wait_for_predecessor();
  if (w >= TFKT_MLP_NWEIGHTS) return;
  const float g = grad[w];
  const float mw = b1 * m[w] + (1.0f - b1) * g;
  const float vw = b2 * v[w] + (1.0f - b2) * g * g;
  m[w] = mw;
  v[w] = vw;
  const float p = master[w] - lr * (mw * c1) / (sqrtf(vw * c2) + eps);
  master[w] = p;
  int e = -1;
  if (w < OB1) e = w;                                   // W1
  else if (w >= OW2 && w < OB2) e = NH * NIN + (w - OW2);   // W2
  else if (w >= OW3 && w < OB3) e = NH * NIN + NH * NH + (w - OW3);   // W3
  if (e >= 0) wmat[e] = __float2bfloat16_rn(p);
}

__global__ void refresh_kernel(const float* __restrict__ master, __nv_bfloat16* __restrict__ wmat) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= NMAT) return;
  int w;
  if (e < NH * NIN) w = OW1 + e;
  else if (e < NH * NIN + NH * NH) w = OW2 + (e - NH * NIN);
  else w = OW3 + (e - NH * NIN - NH * NH);
  wmat[e] = __float2bfloat16_rn(master[w]);
}

tfkt_status cuda_err(cudaError_t e, const char* what) {
  return fail(TFKT_ECUDA, std::string(what) + ": " + cudaGetErrorString(e));
}

#define MLP_CUDA(...)                                          \
  do {                                                         \
    cudaError_t e_ = (__VA_ARGS__);                            \
    if (e_ != cudaSuccess) return cuda_err(e_, #__VA_ARGS__);  \
  } while (0)

// What only training needs, on its first use: the partial sums of nb blocks.
tfkt_status ensure_training(tfkt_mlp* net, int nb) {
  if (!net->lpart) MLP_CUDA(cudaMalloc(&net->lpart, (MAX_TRAIN_BLOCKS + 1) * sizeof(double)));
  if (nb <= net->partial_blocks) return TFKT_OK;
  if (net->partial) MLP_CUDA(cudaFree(net->partial));
  net->partial = nullptr;
  net->partial_blocks = 0;
  MLP_CUDA(cudaMalloc(&net->partial, (size_t)nb * TFKT_MLP_NWEIGHTS * sizeof(float)));
  net->partial_blocks = nb;
  return TFKT_OK;
}

}  // namespace

const MlpDev& mlp_dev(const tfkt_mlp* net) { return net->d; }

}  // namespace tfkt

using namespace tfkt;

extern "C" {

tfkt_status tfkt_mlp_create(const float* params, void* stream, tfkt_mlp** out) {
  if (!params || !out) return fail(TFKT_EINVAL, "NULL argument");
  *out = nullptr;
  tfkt_mlp* net = new (std::nothrow) tfkt_mlp();   // nothing may throw across the C interface
  if (!net) return fail(TFKT_ENOMEM, "host allocation failed");
  net->stream = (cudaStream_t)stream;
  auto bad = [&](cudaError_t e, const char* what) {
    tfkt_mlp_destroy(net);
    return cuda_err(e, what);
  };
  cudaError_t e;
  if ((e = cudaMalloc(&net->d.master, TFKT_MLP_NPARAM * sizeof(float))) != cudaSuccess ||
      (e = cudaMalloc(&net->d.wmat, NMAT * sizeof(__nv_bfloat16))) != cudaSuccess ||
      (e = cudaMalloc(&net->m, TFKT_MLP_NWEIGHTS * sizeof(float))) != cudaSuccess ||
      (e = cudaMalloc(&net->v, TFKT_MLP_NWEIGHTS * sizeof(float))) != cudaSuccess ||
      (e = cudaMalloc(&net->grad, TFKT_MLP_NWEIGHTS * sizeof(float))) != cudaSuccess) {
    tfkt_mlp_destroy(net);
    cudaGetLastError();   // clear the allocation error
    return fail(TFKT_ENOMEM, std::string("cudaMalloc: ") + cudaGetErrorString(e));
  }
  // Where reduce_kernel leaves the loss that the host reads: pinned host memory saves the copy (6
  // of 45 us at 16384 samples). Where there is none, the loss is copied from device memory.
  if (cudaMallocHost(&net->loss_host, sizeof(double)) != cudaSuccess) {
    net->loss_host = nullptr;
    cudaGetLastError();
  }
  if ((e = cudaMemsetAsync(net->m, 0, TFKT_MLP_NWEIGHTS * sizeof(float), net->stream)) != cudaSuccess ||
      (e = cudaMemsetAsync(net->v, 0, TFKT_MLP_NWEIGHTS * sizeof(float), net->stream)) != cudaSuccess ||
      (e = cudaMemsetAsync(net->grad, 0, TFKT_MLP_NWEIGHTS * sizeof(float), net->stream)) != cudaSuccess)
    return bad(e, "cudaMemsetAsync");
  tfkt_status s = tfkt_mlp_set(net, params);
  if (s != TFKT_OK) {
    tfkt_mlp_destroy(net);
    return s;
  }
  *out = net;
  return TFKT_OK;
}

tfkt_status tfkt_mlp_destroy(tfkt_mlp* net) {
  if (!net) return TFKT_OK;
  cudaError_t e = cudaStreamSynchronize(net->stream);
  void* ptrs[] = {net->d.master, net->d.wmat, net->m, net->v, net->grad, net->partial, net->lpart};
  for (void* p : ptrs)
    if (p) {
      cudaError_t f = cudaFree(p);
      if (e == cudaSuccess) e = f;
    }
  if (net->loss_host) {
    cudaError_t f = cudaFreeHost(net->loss_host);
    if (e == cudaSuccess) e = f;
  }
  delete net;
  if (e != cudaSuccess) return cuda_err(e, "destroy");
  return TFKT_OK;
}

tfkt_status tfkt_mlp_get(tfkt_mlp* net, float* params) {
  if (!net || !params) return fail(TFKT_EINVAL, "NULL argument");
  MLP_CUDA(cudaMemcpyAsync(params, net->d.master, TFKT_MLP_NPARAM * sizeof(float),
                           cudaMemcpyDeviceToHost, net->stream));
  MLP_CUDA(cudaStreamSynchronize(net->stream));
  return TFKT_OK;
}

tfkt_status tfkt_mlp_set(tfkt_mlp* net, const float* params) {
  if (!net || !params) return fail(TFKT_EINVAL, "NULL argument");
  for (int k = 0; k < NIN; ++k)
    if (!(params[OSX + k] > 0)) return fail(TFKT_EINVAL, "input scales sx must be > 0");
  for (int k = 0; k < NOUT; ++k)
    if (!(params[OST + k] > 0)) return fail(TFKT_EINVAL, "output scales st must be > 0");
  MLP_CUDA(cudaMemcpyAsync(net->d.master, params, TFKT_MLP_NPARAM * sizeof(float),
                           cudaMemcpyHostToDevice, net->stream));
  refresh_kernel<<<(NMAT + 255) / 256, 256, 0, net->stream>>>(net->d.master, net->d.wmat);
  MLP_CUDA(cudaGetLastError());
  // the host vector may be released as soon as this returns
  MLP_CUDA(cudaStreamSynchronize(net->stream));
  return TFKT_OK;
}

tfkt_status tfkt_mlp_forward(tfkt_mlp* net, const float* X, int64_t n, float* Y) {
  NvtxRange nvtx_range("tfkt_mlp_forward");
  if (!net || n < 0 || (n > 0 && (!X || !Y))) return fail(TFKT_EINVAL, "bad argument");
  if (n == 0) return TFKT_OK;
  const int64_t blocks = (n + 127) / 128;
  forward_kernel<<<(unsigned)blocks, 128, tc_smem_bytes(4), net->stream>>>(net->d.master, net->d.wmat,
                                                                          X, n, Y);
  MLP_CUDA(cudaGetLastError());
  return TFKT_OK;
}

tfkt_status tfkt_mlp_loss_grad(tfkt_mlp* net, const float* X, const float* T, int64_t n,
                               double* loss, float* grad) {
  NvtxRange nvtx_range("tfkt_mlp_loss_grad");
  if (!net || n < 1 || !X || !T) return fail(TFKT_EINVAL, "bad argument");
  const int64_t tiles = (n + TB - 1) / TB;
  if (tiles > (1 << 20)) return fail(TFKT_EINVAL, "batch too large (at most 2^27 samples)");
  const int nb = (int)(tiles < MAX_TRAIN_BLOCKS ? tiles : MAX_TRAIN_BLOCKS);
  tfkt_status st = ensure_training(net, nb);
  if (st != TFKT_OK) return st;
  double* at = net->loss_host ? net->loss_host : net->lpart + MAX_TRAIN_BLOCKS;
  const size_t smem = sizeof(TrainTc);
  MLP_CUDA(cudaFuncSetAttribute(loss_grad_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)smem));
  const bool dep = !stream_capturing(net->stream);
  MLP_CUDA(launch(loss_grad_kernel, dim3(nb), dim3(TT), smem, net->stream, dep,
                  (const float*)net->d.master, (const __nv_bfloat16*)net->d.wmat, X, T, n,
                  net->partial, net->lpart));
  MLP_CUDA(launch(reduce_kernel, dim3((TFKT_MLP_NWEIGHTS + RD_W - 1) / RD_W + 1), dim3(RD_W * RD_S), 0,
                  net->stream, dep, (const float*)net->partial, nb, net->grad, grad,
                  (const double*)net->lpart, at, n));
  if (loss) {
    if (at != net->loss_host)
      MLP_CUDA(cudaMemcpyAsync(loss, at, sizeof(double), cudaMemcpyDeviceToHost, net->stream));
    MLP_CUDA(cudaStreamSynchronize(net->stream));
    if (at == net->loss_host) *loss = *(volatile double*)net->loss_host;
  }
  return TFKT_OK;
}

tfkt_status tfkt_mlp_adam(tfkt_mlp* net, float lr, float beta1, float beta2, float eps) {
  NvtxRange nvtx_range("tfkt_mlp_adam");
  if (!net) return fail(TFKT_EINVAL, "NULL argument");
  if (!(lr >= 0) || !(beta1 >= 0 && beta1 < 1) || !(beta2 >= 0 && beta2 < 1) || !(eps > 0))
    return fail(TFKT_EINVAL, "bad Adam hyper-parameters");
  net->t += 1;
  const float c1 = (float)(1.0 / (1.0 - std::pow((double)beta1, (double)net->t)));
  const float c2 = (float)(1.0 / (1.0 - std::pow((double)beta2, (double)net->t)));
  MLP_CUDA(launch(adam_kernel, dim3((TFKT_MLP_NWEIGHTS + 127) / 128), dim3(128), 0, net->stream,
                  !stream_capturing(net->stream), net->d.master, net->d.wmat, net->m, net->v,
                  (const float*)net->grad, lr, beta1, beta2, eps, c1, c2));
  return TFKT_OK;
}

}  // extern "C"
