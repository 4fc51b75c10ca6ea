// Learned initial guess: per-atom features, a 32 -> 64 -> 64 -> 64 -> 1 SiLU network
// (forward, gradient, Adam), and the guess q0 = q_prev + scale * net(features).
//
// The paper has no learned component; the network and its features are the project's
// definition (see the FP64 oracle for the same definition written out).  Parameters are
// FP32 master values; with `bf16` set the forward and gradient use them rounded to BF16
// (FP32 accumulation throughout).
#include <cuda_bf16.h>
#include <math.h>

#include <algorithm>
#include <vector>

#include "phasor.cuh"

namespace cpm {

namespace {

constexpr int kF = CPM_MLP_FEATURES;  // 32
constexpr int kH = 64;
constexpr int kP = CPM_MLP_PARAMS;    // 10,497
// parameter offsets: W1 [64][32], b1, W2 [64][64], b2, W3 [64][64], b3, W4 [64], b4
constexpr int oW1 = 0, ob1 = oW1 + kH * kF, oW2 = ob1 + kH, ob2 = oW2 + kH * kH,
              oW3 = ob2 + kH, ob3 = oW3 + kH * kH, oW4 = ob3 + kH, ob4 = oW4 + kH;
static_assert(ob4 + 1 == kP, "parameter layout");

// SiLU and its derivative through the fast exponential and reciprocal (relative error
// ~1e-6, far inside what a guess needs and what the oracle comparison allows): the
// forward pass spends as many instructions on 192 activations per sample as on its
// 10,497 multiply-adds otherwise.
__device__ __forceinline__ float sigmoid(float z) { return __frcp_rn(1.0f + __expf(-z)); }
__device__ __forceinline__ float silu(float z) { return z * sigmoid(z); }

// Shell of every PCG-DC pattern entry (k - 1/2 <= r < k + 1/2, k = 1..8; 0 outside or
// for the atom itself).  The electrode is fixed, so this geometry is found once; the host
// then files the entries of each atom by shell.
__global__ void k_shell_codes(int n, const double* __restrict__ xyz, double lx, double ly,
                              double lz, const int64_t* __restrict__ off,
                              const int* __restrict__ idx, uint8_t* __restrict__ shell) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double xi = xyz[3 * i], yi = xyz[3 * i + 1], zi = xyz[3 * i + 2];
  for (int64_t e = off[i]; e < off[i + 1]; ++e) {
    const int j = idx[e];
    int k = 0;
    if (j != i) {
      double dx = xyz[3 * j] - xi, dy = xyz[3 * j + 1] - yi, dz = xyz[3 * j + 2] - zi;
      dx -= lx * rint(dx / lx);
      dy -= ly * rint(dy / ly);
      dz -= lz * rint(dz / lz);
      k = (int)floor(sqrt(dx * dx + dy * dy + dz * dz) + 0.5);
      if (k < 1 || k > 8) k = 0;
    }
    shell[e] = (uint8_t)k;
  }
}

__global__ void k_to_float(const double* __restrict__ v, int64_t len, double add,
                           float* __restrict__ out) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < len;
       e += (int64_t)gridDim.x * blockDim.x)
    out[e] = (float)(v[e] + add);
}

// The potentials of a frame as floats: (b - b_prev, b) per atom.
__global__ void k_guess_prep(int64_t len, const double* __restrict__ b,
                             const double* __restrict__ b_prev, float2* __restrict__ out) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < len;
       e += (int64_t)gridDim.x * blockDim.x)
    out[e] = make_float2((float)(b[e] - b_prev[e]), (float)b[e]);
}

// Features of atom i in frame f (unscaled): 0 the potential change Delta b = b - b_prev,
// 1-8 its means over the neighbour shells k = 1..8, 9 b, 10-17 the shell means of b,
// 18 chi, 19 the side of the electrode (+1 above the mean height), 20 (P Delta b) / k_e
// with the PCG-DC preconditioner's pattern entries, 21-31 zero.
constexpr int kFeatFrames = 4;     // frames per thread: index loads shared by them
constexpr int kFeatThreads = 128;  // atoms per block

__global__ void __launch_bounds__(kFeatThreads)
k_guess_features(int n, int frames, const float2* __restrict__ pot,
                 const double* __restrict__ chi, const double* __restrict__ xyz, double zmean,
                 const int64_t* __restrict__ sh_off, const int* __restrict__ sh_idx,
                 const int64_t* __restrict__ off, const int* __restrict__ idx,
                 const float* __restrict__ pf32, float* __restrict__ feat) {
  constexpr int FB = kFeatFrames;
  __shared__ float stage[kFeatThreads * (kF + 1)];
  const int i0 = blockIdx.x * kFeatThreads;
  const int i = i0 + threadIdx.x;
  const int f0 = blockIdx.y * FB;
  const bool live = i < n;
  float sd[FB][8], sb[FB][8], pz[FB];
#pragma unroll
  for (int u = 0; u < FB; ++u) {
    pz[u] = 0.f;
#pragma unroll
    for (int k = 0; k < 8; ++k) sd[u][k] = sb[u][k] = 0.f;
  }
  // a frame past the last reads frame 0 and is not written
  const float2* pf[FB];
#pragma unroll
  for (int u = 0; u < FB; ++u) pf[u] = pot + (int64_t)(f0 + u < frames ? f0 + u : 0) * n;
  int cnt[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) cnt[k] = 0;
  if (live) {
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const int64_t e0 = sh_off[(int64_t)i * 8 + k], e1 = sh_off[(int64_t)i * 8 + k + 1];
      cnt[k] = (int)(e1 - e0);
      for (int64_t e = e0; e < e1; ++e) {
        const int j = sh_idx[e];
#pragma unroll
        for (int u = 0; u < FB; ++u) {
          const float2 v = pf[u][j];
          sd[u][k] += v.x;
          sb[u][k] += v.y;
        }
      }
    }
    for (int64_t e = off[i]; e < off[i + 1]; ++e) {
      const int j = idx[e];
      const float w = pf32[e];
#pragma unroll
      for (int u = 0; u < FB; ++u) pz[u] = fmaf(w, pf[u][j].x, pz[u]);
    }
  }
  const float chi_i = live ? (float)chi[i] : 0.f;
  const float side = live && xyz[3 * i + 2] > zmean ? 1.f : -1.f;
  const int na = min(kFeatThreads, n - i0);
#pragma unroll
  for (int u = 0; u < FB; ++u) {
    if (f0 + u >= frames) break;  // uniform per block
    float* row = stage + threadIdx.x * (kF + 1);
    if (live) {
      const float2 self = pf[u][i];
      row[0] = self.x;
      row[9] = self.y;
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const float inv = cnt[k] ? 1.0f / (float)cnt[k] : 0.f;
        row[1 + k] = sd[u][k] * inv;
        row[10 + k] = sb[u][k] * inv;
      }
      row[18] = chi_i;
      row[19] = side;
      row[20] = pz[u] * (float)(1.0 / kKe);
#pragma unroll
      for (int c = 21; c < kF; ++c) row[c] = 0.f;
    }
    __syncthreads();
    // the block's atoms are consecutive: one contiguous, coalesced write per frame
    float* dst = feat + ((int64_t)(f0 + u) * n + i0) * kF;
    for (int e = threadIdx.x; e < na * kF; e += kFeatThreads)
      dst[e] = stage[(e / kF) * (kF + 1) + e % kF];
    __syncthreads();
  }
}

// y[s] = net((feat[s] - mean) * inv_std), 128 samples per tile.  Weights (transposed,
// unit index fastest) and the activations of a tile (feature-major) sit in shared memory;
// each thread owns 8 samples x 4 units of a layer, so every float4 of weights and of
// activations it loads feeds 32 (or 16) FMAs.  The float4 slot of an activation row is
// XOR-swizzled with the row's unit group, which keeps the transposed stores of a layer's
// output free of bank conflicts.
constexpr int kTs = 128;          // samples per tile
constexpr int kFwdThreads = 256;  // 16 unit groups x 16 sample groups
constexpr int kWT = kP + 3;       // transposed weights, padded to a float4 boundary
constexpr size_t kFwdSmem = sizeof(float) * (kWT + 2 * kH * kTs);

__device__ __forceinline__ int act_at(int row, int s) {
  return row * kTs + 4 * ((s >> 2) ^ ((row >> 2) & 7)) + (s & 3);
}

// acc[k][j] += sum_c W[c][4 ug + j] in[c][8 sg + k] over NIN rows, two samples a paired FMA
// (half the issue slots of scalar ones: 426,000 samples, forward pass 296 -> 290 us, gradient
// 812 -> 781).
template <int NIN>
__device__ __forceinline__ void tile_product(const float* __restrict__ W,
                                             const float* __restrict__ in, float (&acc)[8][4],
                                             int ug, int sg) {
  float2 a[4][4];
#pragma unroll
  for (int k = 0; k < 4; ++k)
#pragma unroll
    for (int j = 0; j < 4; ++j) a[k][j] = make_float2(acc[2 * k][j], acc[2 * k + 1][j]);
#pragma unroll 4
  for (int c = 0; c < NIN; ++c) {
    const float4 w = *reinterpret_cast<const float4*>(W + c * kH + 4 * ug);
    const float4 x0 = *reinterpret_cast<const float4*>(in + act_at(c, 8 * sg));
    const float4 x1 = *reinterpret_cast<const float4*>(in + act_at(c, 8 * sg + 4));
    const float2 xv[4] = {make_float2(x0.x, x0.y), make_float2(x0.z, x0.w),
                          make_float2(x1.x, x1.y), make_float2(x1.z, x1.w)};
    const float wv[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int k = 0; k < 4; ++k)
        a[k][j] = __ffma2_rn(xv[k], make_float2(wv[j], wv[j]), a[k][j]);
  }
#pragma unroll
  for (int k = 0; k < 4; ++k)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      acc[2 * k][j] = a[k][j].x;
      acc[2 * k + 1][j] = a[k][j].y;
    }
}

// acc = bias[a] + sum_c WT[c][a] in[c][s] for this thread's 8 x 4 block.
template <int NIN>
__device__ __forceinline__ void fwd_layer(const float* __restrict__ WT,
                                          const float* __restrict__ bias,
                                          const float* __restrict__ in, float (&acc)[8][4],
                                          int ug, int sg) {
#pragma unroll
  for (int k = 0; k < 8; ++k)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[k][j] = bias[4 * ug + j];
  tile_product<NIN>(WT, in, acc, ug, sg);
}

__device__ __forceinline__ void fwd_store(float* __restrict__ out, const float (&acc)[8][4],
                                          int ug, int sg) {
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int row = 4 * ug + j;
    *reinterpret_cast<float4*>(out + act_at(row, 8 * sg)) =
        make_float4(silu(acc[0][j]), silu(acc[1][j]), silu(acc[2][j]), silu(acc[3][j]));
    *reinterpret_cast<float4*>(out + act_at(row, 8 * sg + 4)) =
        make_float4(silu(acc[4][j]), silu(acc[5][j]), silu(acc[6][j]), silu(acc[7][j]));
  }
}

__global__ void __launch_bounds__(kFwdThreads, 2)
k_mlp_forward(const float* __restrict__ params, const float* __restrict__ norm, int bf16,
              int64_t samples, const float* __restrict__ feat, float* __restrict__ out,
              float scale, const double* __restrict__ q_prev, double* __restrict__ q0) {
  extern __shared__ __align__(16) float fsm[];
  float* WT1 = fsm;               // [kF][kH]
  float* WT2 = WT1 + kF * kH;     // [kH][kH]
  float* WT3 = WT2 + kH * kH;     // [kH][kH]
  float* bv = WT3 + kH * kH;      // b1, b2, b3, W4 [kH each], b4
  float* act0 = fsm + kWT;        // [kH][kTs]
  float* act1 = act0 + kH * kTs;  // [kH][kTs]
  const int t = threadIdx.x;
  for (int e = t; e < kP; e += kFwdThreads) {
    float v = params[e];
    if (bf16) v = __bfloat162float(__float2bfloat16_rn(v));
    int d;
    if (e < ob1) d = (e % kF) * kH + e / kF;                                  // W1[a][c]
    else if (e < oW2) d = kF * kH + 2 * kH * kH + (e - ob1);                 // b1
    else if (e < ob2) d = kF * kH + ((e - oW2) % kH) * kH + (e - oW2) / kH;  // W2
    else if (e < oW3) d = kF * kH + 2 * kH * kH + kH + (e - ob2);            // b2
    else if (e < ob3) d = kF * kH + kH * kH + ((e - oW3) % kH) * kH + (e - oW3) / kH;
    else if (e < oW4) d = kF * kH + 2 * kH * kH + 2 * kH + (e - ob3);        // b3
    else d = kF * kH + 2 * kH * kH + 3 * kH + (e - oW4);                     // W4, b4
    fsm[d] = v;
  }
  const int ug = t & 15, sg = t >> 4;
  const int64_t tiles = (samples + kTs - 1) / kTs;
  for (int64_t tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
    const int64_t s0 = tile * kTs;
    __syncthreads();  // weights written / the previous tile's reads of act0 done
    for (int e = t; e < kTs * kF; e += kFwdThreads) {
      const int s = e / kF, c = e % kF;
      const int64_t gs = s0 + s;
      act0[act_at(c, s)] = gs < samples ? (feat[gs * kF + c] - norm[c]) * norm[kF + c] : 0.f;
    }
    __syncthreads();
    float acc[8][4];
    fwd_layer<kF>(WT1, bv, act0, acc, ug, sg);
    fwd_store(act1, acc, ug, sg);
    __syncthreads();
    fwd_layer<kH>(WT2, bv + kH, act1, acc, ug, sg);
    __syncthreads();  // all reads of act0 (the features) are done
    fwd_store(act0, acc, ug, sg);
    __syncthreads();
    fwd_layer<kH>(WT3, bv + 2 * kH, act0, acc, ug, sg);
    // output unit: y = b4 + sum_a W4[a] silu(z3[a]), summed over the 16 unit groups
    float y[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      float v = 0.f;
#pragma unroll
      for (int j = 0; j < 4; ++j) v = fmaf(bv[3 * kH + 4 * ug + j], silu(acc[k][j]), v);
#pragma unroll
      for (int o = 1; o < 16; o <<= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
      y[k] = v + bv[4 * kH];
    }
    if (ug == 0)
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const int64_t gs = s0 + 8 * sg + k;
        if (gs < samples) {
          if (out) out[gs] = y[k];
          if (q0) q0[gs] = q_prev[gs] + (double)scale * (double)y[k];  // the guess, fused
        }
      }
  }
}

// Gradient of the mean squared error (1/S) sum_s (y_s - t_s)^2 over this call's samples and
// sum_s (y_s - t_s)^2: every block's share into part[block][kPart], summed by k_grad_finish.
//
// Persistent blocks (one an SM: 222 KB of shared memory) take tiles of 128 samples.  Every
// product of the pass is a register-tiled one on feature-major tiles with XOR-swizzled rows:
// the forward layers and the back-propagated ones in 8 samples x 4 units a thread (as
// k_mlp_forward; the thread that made a pre-activation also meets its gradient, so silu'
// stays in its registers), the weight gradients in 4 x 4 outputs over the tile's samples.
// The weight gradients of a tile (layers 1 to 3) are float sums over its 128 samples, added to a
// float pair a thread keeps over its tiles; the biases' and the output weights' are float sums of a
// thread's 8 samples a tile (registers are all taken).  A launch takes at most kGradTiles tiles a
// block, and the next one adds to its blocks' shares in FP64: with one launch for 1,000 tiles a
// block those sums, 8,000 terms long, were off by 6e-5 of a layer's largest entry where the samples
// were alike.  (The same inside the kernel, every 32 tiles, cost 1% and more of any batch.)  Blocks
// are added in FP64 in a fixed order.  Bound by FP32
// multiply-adds (29,000 a sample; 8 warps an SM).  One thread a sample with scalar loads of
// every operand and an atomic add per parameter and 128 samples took 3,702 us for 426,000
// samples (8% of the chip's FP32 rate); this takes 781 us (the sigmoids' exponentials and
// divisions issue as much as the products).
constexpr int kGradThreads = 256;
constexpr int kGradTiles = 32;
constexpr int kPart = kP + 1;  // the parameters' gradients, the loss
constexpr int oGW = kF * kH + 2 * kH * kH;   // WT1, WT2, WT3, then:
constexpr int oGB = oGW + 2 * kH * kH;       // W2, W3 as given, then b1, b2, b3, W4, b4
constexpr int oGX = oGB + 4 * kH + 4;        // tiles: X, H1, H2, GA, GB
constexpr size_t kGradSmem = sizeof(float) * (oGX + kF * kTs + 4 * kH * kTs);

__device__ __forceinline__ void tile_store(float* __restrict__ out, const float (&v)[8][4],
                                           int ug, int sg) {
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int row = 4 * ug + j;
    *reinterpret_cast<float4*>(out + act_at(row, 8 * sg)) =
        make_float4(v[0][j], v[1][j], v[2][j], v[3][j]);
    *reinterpret_cast<float4*>(out + act_at(row, 8 * sg + 4)) =
        make_float4(v[4][j], v[5][j], v[6][j], v[7][j]);
  }
}

// (h, l)[i][j] += sum_s G[4 ua + i][s] in[NC uc + j][s] over the tile's samples.
template <int NC>
__device__ __forceinline__ void tile_outer(const float* __restrict__ G,
                                           const float* __restrict__ in, float (&h)[4][NC],
                                           float (&l)[4][NC], int ua, int uc) {
  float2 acc[4][NC];  // even samples, odd samples
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < NC; ++j) acc[i][j] = make_float2(0.f, 0.f);
#pragma unroll 2
  for (int s = 0; s < kTs; s += 4) {
    float4 g[4], x[NC];
#pragma unroll
    for (int i = 0; i < 4; ++i)
      g[i] = *reinterpret_cast<const float4*>(G + act_at(4 * ua + i, s));
#pragma unroll
    for (int j = 0; j < NC; ++j)
      x[j] = *reinterpret_cast<const float4*>(in + act_at(NC * uc + j, s));
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < NC; ++j)
        acc[i][j] = __ffma2_rn(make_float2(g[i].z, g[i].w), make_float2(x[j].z, x[j].w),
                               __ffma2_rn(make_float2(g[i].x, g[i].y),
                                          make_float2(x[j].x, x[j].y), acc[i][j]));
  }
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < NC; ++j) pair_add1(h[i][j], l[i][j], acc[i][j].x + acc[i][j].y);
}

__global__ void __launch_bounds__(kGradThreads, 1)
k_mlp_grad(const float* __restrict__ params, const float* __restrict__ norm, int bf16,
           int64_t samples, double inv_s, const float* __restrict__ feat,
           const float* __restrict__ target, double* __restrict__ part, int add) {
  extern __shared__ __align__(16) float gsm[];
  float *WT1 = gsm, *WT2 = WT1 + kF * kH, *WT3 = WT2 + kH * kH;
  float *W2 = gsm + oGW, *W3 = W2 + kH * kH, *bv = gsm + oGB;
  float *X = gsm + oGX, *H1 = X + kF * kTs, *H2 = H1 + kH * kTs, *GA = H2 + kH * kTs,
        *GB = GA + kH * kTs;
  const int t = threadIdx.x;
  for (int e = t; e < kP; e += kGradThreads) {
    float v = params[e];
    if (bf16) v = __bfloat162float(__float2bfloat16_rn(v));
    if (e < ob1) {
      WT1[(e % kF) * kH + e / kF] = v;
    } else if (e < oW2) {
      bv[e - ob1] = v;
    } else if (e < ob2) {
      WT2[((e - oW2) % kH) * kH + (e - oW2) / kH] = v;
      W2[e - oW2] = v;
    } else if (e < oW3) {
      bv[kH + e - ob2] = v;
    } else if (e < ob3) {
      WT3[((e - oW3) % kH) * kH + (e - oW3) / kH] = v;
      W3[e - oW3] = v;
    } else if (e < oW4) {
      bv[2 * kH + e - ob3] = v;
    } else {
      bv[3 * kH + e - oW4] = v;  // W4, b4
    }
  }
  const int ug = t & 15, sg = t >> 4;  // units 4 ug .., samples 8 sg ..; outputs 4 ug, sg too
  float h3[4][4], l3[4][4], h2[4][4], l2[4][4], h1[4][2], l1[4][2];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
#pragma unroll
    for (int j = 0; j < 4; ++j) h3[i][j] = l3[i][j] = h2[i][j] = l2[i][j] = 0.f;
#pragma unroll
    for (int j = 0; j < 2; ++j) h1[i][j] = l1[i][j] = 0.f;
  }
  float b1[4] = {0, 0, 0, 0}, b2[4] = {0, 0, 0, 0}, b3[4] = {0, 0, 0, 0}, w4[4] = {0, 0, 0, 0};
  float b4 = 0.f, lossh = 0.f, lossl = 0.f;
  const float scale = (float)(2.0 * inv_s);
  const int64_t tiles = (samples + kTs - 1) / kTs;
  for (int64_t tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
    const int64_t s0 = tile * kTs;
    __syncthreads();  // weights written / the previous tile's reads of X done
    for (int e = t; e < kTs * kF; e += kGradThreads) {
      const int s = e / kF, c = e % kF;
      const int64_t gs = s0 + s;
      X[act_at(c, s)] = gs < samples ? (feat[gs * kF + c] - norm[c]) * norm[kF + c] : 0.f;
    }
    __syncthreads();
    float acc[8][4], d1[8][4], d2[8][4];  // d: silu' of layers 1 and 2
    auto bias = [&](int layer) {
#pragma unroll
      for (int k = 0; k < 8; ++k)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[k][j] = bv[layer * kH + 4 * ug + j];
    };
    auto activate = [&](float (&d)[8][4]) {
#pragma unroll
      for (int k = 0; k < 8; ++k)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const float z = acc[k][j], s = sigmoid(z);
          d[k][j] = s * (1.0f + z * (1.0f - s));
          acc[k][j] = z * s;
        }
    };
    bias(0);
    tile_product<kF>(WT1, X, acc, ug, sg);
    activate(d1);
    tile_store(H1, acc, ug, sg);
    __syncthreads();
    bias(1);
    tile_product<kH>(WT2, H1, acc, ug, sg);
    activate(d2);
    tile_store(H2, acc, ug, sg);
    __syncthreads();
    bias(2);
    tile_product<kH>(WT3, H2, acc, ug, sg);
    // y, dL/dy and dL/dz3 of the thread's 8 samples
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      float hv[4], dv[4], y = 0.f;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float z = acc[k][j], s = sigmoid(z);
        hv[j] = z * s;
        dv[j] = s * (1.0f + z * (1.0f - s));
        y = fmaf(bv[3 * kH + 4 * ug + j], hv[j], y);
      }
#pragma unroll
      for (int o = 1; o < 16; o <<= 1) y += __shfl_xor_sync(0xffffffffu, y, o);
      const int64_t gs = s0 + 8 * sg + k;
      const float diff = gs < samples ? y + bv[4 * kH] - target[gs] : 0.f;
      const float dy = scale * diff;
      if (ug == 0) {
        const float p = __fmul_rn(diff, diff);
        pair_add1(lossh, lossl, p);
        lossl += fmaf(diff, diff, -p);
        b4 += dy;
      }
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        w4[j] = fmaf(dy, hv[j], w4[j]);
        acc[k][j] = dy * bv[3 * kH + 4 * ug + j] * dv[j];
        b3[j] += acc[k][j];
      }
    }
    tile_store(GA, acc, ug, sg);
    __syncthreads();
    auto back = [&](const float* W, const float* G, const float (&d)[8][4], float (&b)[4]) {
#pragma unroll
      for (int k = 0; k < 8; ++k)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[k][j] = 0.f;
      tile_product<kH>(W, G, acc, ug, sg);
#pragma unroll
      for (int k = 0; k < 8; ++k)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          acc[k][j] *= d[k][j];
          b[j] += acc[k][j];
        }
    };
    back(W3, GA, d2, b2);
    tile_store(GB, acc, ug, sg);
    tile_outer<4>(GA, H2, h3, l3, ug, sg);
    __syncthreads();
    back(W2, GB, d1, b1);
    tile_store(GA, acc, ug, sg);
    tile_outer<4>(GB, H1, h2, l2, ug, sg);
    __syncthreads();
    tile_outer<2>(GA, X, h1, l1, ug, sg);
  }
  // the block's sums: weight gradients from their threads, the others over the 16 sample groups
  double* out = part + (int64_t)blockIdx.x * kPart;
  auto put = [&](int e, double x) { out[e] = add ? out[e] + x : x; };
#pragma unroll
  for (int i = 0; i < 4; ++i) {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int e = (4 * ug + i) * kH + 4 * sg + j;
      put(oW3 + e, (double)h3[i][j] + (double)l3[i][j]);
      put(oW2 + e, (double)h2[i][j] + (double)l2[i][j]);
    }
#pragma unroll
    for (int j = 0; j < 2; ++j)
      put(oW1 + (4 * ug + i) * kF + 2 * sg + j, (double)h1[i][j] + (double)l1[i][j]);
  }
  __syncthreads();
  float* red = GA;  // [4][16 sample groups][64 units]
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    red[(0 * 16 + sg) * kH + 4 * ug + j] = b1[j];
    red[(1 * 16 + sg) * kH + 4 * ug + j] = b2[j];
    red[(2 * 16 + sg) * kH + 4 * ug + j] = b3[j];
    red[(3 * 16 + sg) * kH + 4 * ug + j] = w4[j];
  }
  double* red2 = reinterpret_cast<double*>(GB);  // [16][2]
  if (ug == 0) {
    red2[2 * sg] = (double)b4;
    red2[2 * sg + 1] = (double)lossh + (double)lossl;
  }
  __syncthreads();
  {
    const int arr = t >> 6, u = t & 63;
    double s = 0.0;
    for (int g = 0; g < 16; ++g) s += (double)red[(arr * 16 + g) * kH + u];
    put((arr == 0 ? ob1 : arr == 1 ? ob2 : arr == 2 ? ob3 : oW4) + u, s);
    if (t < 2) {
      s = 0.0;
      for (int g = 0; g < 16; ++g) s += red2[2 * g + t];
      put(t == 0 ? ob4 : kP, s);
    }
  }
}

struct AdamStep {
  float *p, *m, *v;
  float lr, c1, c2;
};

__device__ __forceinline__ void adam_update(const AdamStep& a, int k, float gk) {
  const float mk = 0.9f * a.m[k] + 0.1f * gk;
  const float vk = 0.999f * a.v[k] + 0.001f * gk * gk;
  a.m[k] = mk;
  a.v[k] = vk;
  a.p[k] -= a.lr * (mk * a.c1) / (sqrtf(vk * a.c2) + 1e-8f);
}

// grad = sum of the blocks' shares in block order (eight interleaved sums, added in order),
// the loss likewise; with a.p, the Adam step on the same parameter.
constexpr int kFinishSlices = 8;

__global__ void __launch_bounds__(32 * kFinishSlices)
k_grad_finish(const double* __restrict__ part, int blocks, float* __restrict__ grad,
              double* __restrict__ loss, const AdamStep a) {
  __shared__ double red[kFinishSlices][32];
  const int lane = threadIdx.x & 31, sl = threadIdx.x >> 5;
  const int k = blockIdx.x * 32 + lane;
  double s = 0.0;
  if (k < kPart)
#pragma unroll 4
    for (int b = sl; b < blocks; b += kFinishSlices) s += part[(int64_t)b * kPart + k];
  red[sl][lane] = s;
  __syncthreads();
  if (sl != 0 || k >= kPart) return;
  for (int w = 1; w < kFinishSlices; ++w) s += red[w][lane];
  if (k == kP) {
    *loss = s;
    return;
  }
  grad[k] = (float)s;
  if (a.p) adam_update(a, k, (float)s);
}

__global__ void k_adam(const AdamStep a, const float* __restrict__ g) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k < kP) adam_update(a, k, g[k]);
}

__global__ void k_guess_apply(int64_t len, const float* __restrict__ y, float scale,
                              const double* __restrict__ q_prev, double* __restrict__ q0) {
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < len;
       k += (int64_t)gridDim.x * blockDim.x)
    q0[k] = q_prev[k] + (double)scale * (double)y[k];
}

// Device memory of the context's device (or managed memory): what these kernels may use.
bool dev_ok(const Ctx* c, const void* p) { return pointer_where(c, p) == 1; }

}  // namespace
}  // namespace cpm

using namespace cpm;

struct cpm_ctx : public cpm::Ctx {};

namespace {

int features_async(cpm_ctx* c, int frames, const double* b, const double* b_prev,
                   const double* chi, float* feat) {
  if (!c) return CPM_EINVAL;
  if (!c->built) return set_err(c, CPM_ENOTBUILT, "cpm_guess_features before cpm_build_E");
  if (c->solve_only)
    return set_err(c, CPM_EINVAL, "cpm_guess_features: a context built by cpm_build_E_copy");
  if (c->p.precond != CPM_PRECOND_DC || !c->nbr_off.ptr)
    return set_err(c, CPM_EINVAL, "cpm_guess_features needs the PCG-DC neighbour lists");
  if (frames < 1 || !dev_ok(c, b) || !dev_ok(c, b_prev) || !dev_ok(c, chi) || !dev_ok(c, feat))
    return set_err(c, CPM_EINVAL, "cpm_guess_features: frames >= 1 and device arrays");
  int st = CPM_OK;
  const int n = c->n;
  if (!c->shells_ready) {  // frame-independent geometry, once per electrode
    Buf codes;
    if ((st = buf_alloc(c, &codes, std::max<int64_t>(c->nnz, 1)))) return st;
    (k_shell_codes<<<(n + 127) / 128, 128, 0, c->stream>>>(
         n, (const double*)c->xyz.ptr, c->p.box[0], c->p.box[1], c->p.box[2],
         (const int64_t*)c->nbr_off.ptr, (const int*)c->nbr_idx.ptr, (uint8_t*)codes.ptr),
     note_launch());
    std::vector<double> hx(3 * (size_t)n);
    std::vector<int64_t> hoff(n + 1);
    std::vector<int> hidx(c->nnz);
    std::vector<uint8_t> hk(c->nnz);
    st = cuda_check(c, cudaMemcpyAsync(hx.data(), c->xyz.ptr, hx.size() * sizeof(double),
                                       cudaMemcpyDeviceToHost, c->stream), "xyz");
    if (!st) st = cuda_check(c, cudaMemcpyAsync(hoff.data(), c->nbr_off.ptr,
                                                hoff.size() * sizeof(int64_t),
                                                cudaMemcpyDeviceToHost, c->stream), "off");
    if (!st) st = cuda_check(c, cudaMemcpyAsync(hidx.data(), c->nbr_idx.ptr,
                                                hidx.size() * sizeof(int),
                                                cudaMemcpyDeviceToHost, c->stream), "idx");
    if (!st) st = cuda_check(c, cudaMemcpyAsync(hk.data(), codes.ptr, hk.size(),
                                                cudaMemcpyDeviceToHost, c->stream), "codes");
    if (!st) st = cuda_check(c, cudaStreamSynchronize(c->stream), "shell sync");
    buf_free(c, &codes);
    if (st) return st;
    // entries of atom i filed by shell: bucket (i, k) = sh_off[8 i + k] .. sh_off[8 i + k + 1]
    std::vector<int64_t> so(8 * (size_t)n + 1, 0);
    for (int i = 0; i < n; ++i)
      for (int64_t e = hoff[i]; e < hoff[i + 1]; ++e)
        if (hk[e]) ++so[8 * (size_t)i + hk[e]];
    for (size_t t = 1; t < so.size(); ++t) so[t] += so[t - 1];
    std::vector<int> sj(std::max<int64_t>(so.back(), 1));
    std::vector<int64_t> fill(so.begin(), so.end() - 1);
    for (int i = 0; i < n; ++i)
      for (int64_t e = hoff[i]; e < hoff[i + 1]; ++e)
        if (hk[e]) sj[fill[8 * (size_t)i + hk[e] - 1]++] = hidx[e];
    double zm = 0.0;
    for (int i = 0; i < n; ++i) zm += hx[3 * i + 2];
    c->zmean = zm / n;
    if ((st = buf_alloc(c, &c->shell_off, so.size() * sizeof(int64_t))) ||
        (st = buf_alloc(c, &c->shell_members, sj.size() * sizeof(int))))
      return st;
    st = cuda_check(c, cudaMemcpy(c->shell_off.ptr, so.data(), so.size() * sizeof(int64_t),
                                  cudaMemcpyHostToDevice), "shell offsets");
    if (!st) st = cuda_check(c, cudaMemcpy(c->shell_members.ptr, sj.data(), sj.size() * sizeof(int),
                                           cudaMemcpyHostToDevice), "shell members");
    if (st) return st;
    // the preconditioner's pattern values (Eq. 36, p_gap taken back out) as floats
    if ((st = buf_alloc(c, &c->p_f32, std::max<int64_t>(c->nnz, 1) * sizeof(float)))) return st;
    (k_to_float<<<256, 256, 0, c->stream>>>((const double*)c->prow.ptr, c->nnz, c->pgap,
                                           (float*)c->p_f32.ptr), note_launch());
    if ((st = cuda_check(c, cudaGetLastError(), "P float"))) return st;
    c->shells_ready = true;
  }
  const int64_t len = (int64_t)frames * n;
  if ((st = buf_reserve(c, &c->ws_guess, len * sizeof(float2)))) return st;
  (k_guess_prep<<<(int)std::min<int64_t>((len + 255) / 256, 8192), 256, 0, c->stream>>>(
       len, b, b_prev, (float2*)c->ws_guess.ptr), note_launch());
  dim3 grid((n + kFeatThreads - 1) / kFeatThreads, (frames + kFeatFrames - 1) / kFeatFrames);
  (k_guess_features<<<grid, kFeatThreads, 0, c->stream>>>(
       n, frames, (const float2*)c->ws_guess.ptr, chi, (const double*)c->xyz.ptr, c->zmean,
       (const int64_t*)c->shell_off.ptr, (const int*)c->shell_members.ptr,
       (const int64_t*)c->nbr_off.ptr, (const int*)c->nbr_idx.ptr,
       (const float*)c->p_f32.ptr, feat), note_launch());
  return cuda_check(c, cudaGetLastError(), "features");
}

// Gradient, loss and, with adam.p, the Adam step, on the context's stream: two launches up to
// kGradTiles tiles a block, one more for each as many.
int grad_async(cpm_ctx* c, const float* params, const float* norm, int bf16, int64_t samples,
               const float* feat, const float* target, float* grad, double* loss,
               const AdamStep& adam) {
  int sms = 0;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, c->device);
  int blocks = (int)std::min<int64_t>((samples + kTs - 1) / kTs, std::max(sms, 1));
  int st;  // (fewer blocks where the memory for their shares cannot be had)
  while ((st = buf_reserve(c, &c->ws_grad, (size_t)blocks * kPart * sizeof(double))) ==
             CPM_ENOMEM && blocks > 1)
    blocks /= 2;
  if (!st) st = cuda_check(c, cudaFuncSetAttribute(k_mlp_grad,
                                                   cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                   (int)kGradSmem), "grad smem");
  if (st) return st;
  const int64_t step = (int64_t)blocks * kGradTiles * kTs;
  for (int64_t s0 = 0; s0 < samples; s0 += step)
    (k_mlp_grad<<<blocks, kGradThreads, kGradSmem, c->stream>>>(
         params, norm, bf16, std::min(step, samples - s0), 1.0 / (double)samples, feat + s0 * kF,
         target + s0, (double*)c->ws_grad.ptr, s0 > 0),
     note_launch());
  (k_grad_finish<<<(kPart + 31) / 32, 32 * kFinishSlices, 0, c->stream>>>(
       (const double*)c->ws_grad.ptr, blocks, grad, loss, adam),
   note_launch());
  return cuda_check(c, cudaGetLastError(), "grad");
}

AdamStep adam_step(float* params, float* m, float* v, int step, float lr) {
  return {params, m, v, lr, 1.0f / (1.0f - powf(0.9f, (float)step)),
          1.0f / (1.0f - powf(0.999f, (float)step))};
}

}  // namespace

extern "C" {

int cpm_guess_features(cpm_ctx* c, int frames, const double* b, const double* b_prev,
                       const double* chi, float* feat) {
  int st = features_async(c, frames, b, b_prev, chi, feat);
  if (st) return st;
  return cuda_check(c, cudaStreamSynchronize(c->stream), "features sync");
}

int cpm_guess(cpm_ctx* c, const float* params, const float* norm, int bf16, int frames,
              const double* b, const double* b_prev, const double* chi, float scale,
              const double* q_prev, double* q0) {
  if (!c) return CPM_EINVAL;
  if (!c->built) return set_err(c, CPM_ENOTBUILT, "cpm_guess before cpm_build_E");
  if (frames < 1 || !dev_ok(c, params) || !dev_ok(c, norm) || !dev_ok(c, q_prev) ||
      !dev_ok(c, q0))
    return set_err(c, CPM_EINVAL, "cpm_guess: frames >= 1 and device arrays");
  const int64_t samples = (int64_t)frames * c->n;
  int st = buf_reserve(c, &c->ws_feat, samples * kF * sizeof(float));
  if (st) return st;
  float* feat = (float*)c->ws_feat.ptr;
  if ((st = features_async(c, frames, b, b_prev, chi, feat))) return st;
  if ((st = cuda_check(c, cudaFuncSetAttribute(k_mlp_forward,
                                               cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               (int)kFwdSmem), "forward smem")))
    return st;
  int sms = 0;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, c->device);
  const int64_t tiles = (samples + kTs - 1) / kTs;
  const int blocks = (int)std::min<int64_t>(tiles, 2 * (int64_t)std::max(sms, 1));
  (k_mlp_forward<<<blocks, kFwdThreads, kFwdSmem, c->stream>>>(params, norm, bf16, samples,
                                                               feat, nullptr, scale, q_prev,
                                                               q0), note_launch());
  if ((st = cuda_check(c, cudaGetLastError(), "guess"))) return st;
  return cuda_check(c, cudaStreamSynchronize(c->stream), "guess sync");
}

int cpm_mlp_forward(cpm_ctx* c, const float* params, const float* norm, int bf16,
                    int64_t samples, const float* feat, float* out) {
  if (!c) return CPM_EINVAL;
  if (samples < 1 || !dev_ok(c, params) || !dev_ok(c, norm) || !dev_ok(c, feat) ||
      !dev_ok(c, out))
    return set_err(c, CPM_EINVAL, "cpm_mlp_forward: samples >= 1 and device arrays");
  int st = cuda_check(c, cudaFuncSetAttribute(k_mlp_forward,
                                              cudaFuncAttributeMaxDynamicSharedMemorySize,
                                              (int)kFwdSmem), "forward smem");
  if (st) return st;
  int sms = 0;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, c->device);
  const int64_t tiles = (samples + kTs - 1) / kTs;
  const int blocks = (int)std::min<int64_t>(tiles, 2 * (int64_t)std::max(sms, 1));
  (k_mlp_forward<<<blocks, kFwdThreads, kFwdSmem, c->stream>>>(params, norm, bf16, samples,
                                                               feat, out, 0.f, nullptr,
                                                               nullptr), note_launch());
  if ((st = cuda_check(c, cudaGetLastError(), "forward"))) return st;
  return cuda_check(c, cudaStreamSynchronize(c->stream), "forward sync");
}

int cpm_mlp_grad(cpm_ctx* c, const float* params, const float* norm, int bf16,
                 int64_t samples, const float* feat, const float* target, float* grad,
                 double* loss) {
  if (!c) return CPM_EINVAL;
  if (samples < 1 || !dev_ok(c, params) || !dev_ok(c, norm) || !dev_ok(c, feat) ||
      !dev_ok(c, target) || !dev_ok(c, grad) || !dev_ok(c, loss))
    return set_err(c, CPM_EINVAL, "cpm_mlp_grad: samples >= 1 and device arrays");
  const AdamStep none = {nullptr, nullptr, nullptr, 0.f, 0.f, 0.f};
  if (int st = grad_async(c, params, norm, bf16, samples, feat, target, grad, loss, none)) return st;
  return cuda_check(c, cudaStreamSynchronize(c->stream), "grad sync");
}

int cpm_mlp_adam(cpm_ctx* c, float* params, float* m, float* v, const float* grad, int step,
                 float lr) {
  if (!c) return CPM_EINVAL;
  if (step < 1 || !dev_ok(c, params) || !dev_ok(c, m) || !dev_ok(c, v) || !dev_ok(c, grad))
    return set_err(c, CPM_EINVAL, "cpm_mlp_adam: step >= 1 and device arrays");
  (k_adam<<<(kP + 255) / 256, 256, 0, c->stream>>>(adam_step(params, m, v, step, lr), grad),
   note_launch());
  return cuda_check(c, cudaGetLastError(), "adam");
}

int cpm_guess_train_step(cpm_ctx* c, float* params, const float* norm, int bf16,
                         int64_t samples, const float* feat, const float* target, float* m,
                         float* v, float* grad, double* loss, int step, float lr,
                         double* loss_out) {
  if (!c) return CPM_EINVAL;
  if (samples < 1 || step < 1 || !dev_ok(c, params) || !dev_ok(c, norm) ||
      !dev_ok(c, feat) || !dev_ok(c, target) || !dev_ok(c, m) || !dev_ok(c, v) ||
      !dev_ok(c, grad) || !dev_ok(c, loss))
    return set_err(c, CPM_EINVAL,
                   "cpm_guess_train_step: samples >= 1, step >= 1 and device arrays");
  int st = grad_async(c, params, norm, bf16, samples, feat, target, grad, loss,
                      adam_step(params, m, v, step, lr));
  if (st) return st;
  if (loss_out) {
    double l = 0.0;
    if ((st = cuda_check(c, cudaMemcpyAsync(&l, loss, sizeof(double), cudaMemcpyDeviceToHost,
                                            c->stream), "train step loss")))
      return st;
    if ((st = cuda_check(c, cudaStreamSynchronize(c->stream), "train step sync"))) return st;
    *loss_out = l / (double)samples;
    return CPM_OK;
  }
  return cuda_check(c, cudaStreamSynchronize(c->stream), "train step sync");
}

int cpm_guess_apply(cpm_ctx* c, int64_t len, const float* y, float scale, const double* q_prev,
                    double* q0) {
  if (!c) return CPM_EINVAL;
  if (len < 1 || !dev_ok(c, y) || !dev_ok(c, q_prev) || !dev_ok(c, q0))
    return set_err(c, CPM_EINVAL, "cpm_guess_apply: len >= 1 and device arrays");
  (k_guess_apply<<<256, 256, 0, c->stream>>>(len, y, scale, q_prev, q0), note_launch());
  int st = cuda_check(c, cudaGetLastError(), "guess apply");
  if (st) return st;
  return cuda_check(c, cudaStreamSynchronize(c->stream), "guess sync");
}

}  // extern "C"
