// decoder_fp32.cu -- the decoder in FP32 on the CUDA cores: the accuracy
// anchor of the neural path (fabric_shade_neural with FABRIC_PREC_FP32), the
// forward and backward building blocks for torch.autograd, and the default
// training step's decoder (Sec. 4.2-4.3, loss of Eq. 9-11).
//
// Every layer is a small product over a tile of points with weights and
// activations in shared memory.  A thread owns 4 outputs of 4 or 8 points in
// registers, so that two 16-byte shared-memory reads feed 16 or 32
// multiply-adds (packed FP32x2 over adjacent points); each output is one
// chain of fma over the inputs in order from the bias, as a plain loop gives
// it.  Reductions run in a fixed order (bitwise repeatable).
#include <cmath>

#include <algorithm>

#include "f32x2.h"
#include "fabric_internal.h"
#include "train_common.cuh"

namespace fab {
namespace {

constexpr int kThreads = 256;      // forward
// Row strides of the weights in shared memory, [out][in] as in the flat
// parameters: multiples of four floats (16-byte reads along the inputs)
// whose consecutive rows start in different banks.
constexpr int kLd1 = 76;          // 71 inputs, the rest zero
constexpr int kLdH = kHidden + 4;
constexpr int kInRows = 72;       // decoder inputs, and one row of zeros

// offsets in floats of the staged parameters
constexpr int kSW1 = 0;
constexpr int kSW2 = kSW1 + kHidden * kLd1;
constexpr int kSW3 = kSW2 + kHidden * kLdH;
constexpr int kSW4 = kSW3 + kHidden * kLdH;
constexpr int kSB = kSW4 + kOut * kLdH;             // b1 b2 b3 b4
constexpr int kSParams = kSB + 3 * kHidden + kOut;
static_assert(kSParams % 4 == 0, "what follows the parameters stays 16-byte aligned");

// The flat parameters (float-aligned) into shared memory, by NT threads.
template <int NT>
__device__ __forceinline__ void stage_params(const float *__restrict__ dec, float *W) {
  for (int e = threadIdx.x; e < kHidden * kLd1; e += NT) {
    const int o = e / kLd1, i = e % kLd1;
    W[kSW1 + e] = i < kDecIn ? dec[kOffW1 + o * kDecIn + i] : 0.0f;
  }
  for (int e = threadIdx.x; e < kHidden * kHidden; e += NT) {
    const int o = e / kHidden, i = e % kHidden;
    W[kSW2 + o * kLdH + i] = dec[kOffW2 + e];
    W[kSW3 + o * kLdH + i] = dec[kOffW3 + e];
  }
  for (int e = threadIdx.x; e < kOut * kHidden; e += NT)
    W[kSW4 + (e / kHidden) * kLdH + e % kHidden] = dec[kOffW4 + e];
  for (int e = threadIdx.x; e < 3 * kHidden + kOut; e += NT)
    W[kSB + e] = e < kHidden       ? dec[kOffB1 + e]
                 : e < 2 * kHidden ? dec[kOffB2 + e - kHidden]
                 : e < 3 * kHidden ? dec[kOffB3 + e - 2 * kHidden]
                                   : dec[kOffB4 + e - 3 * kHidden];
}

// A thread's place in a layer: point group pg (points 4 pg .. 4 pg + 3) and
// output group og of 16 (outputs og, og + 16, ...).  A warp holds eight point
// groups (one 128-byte read) and four output groups (rows in different
// banks): warp w takes points 32 (w mod PB) .. and output groups 4 (w / PB) ...
template <int PB>
__device__ __forceinline__ int point_group() { return (threadIdx.x & 7) + 8 * ((threadIdx.x >> 5) % PB); }
template <int PB>
__device__ __forceinline__ int output_group() { return ((threadIdx.x >> 3) & 3) + 4 * ((threadIdx.x >> 5) / PB % 4); }

// out[o][p] = relu(b[o] + sum_k W[o][k] in[k][p]) for this thread's outputs of
// RP = 4 or 8 points (8: 4 pg .. and 64 + 4 pg ..); K a multiple of four.  SYNC: `out` may be `in` (a CTA
// barrier between the last read and the first write).
template <int RP, int PB, int K, int LDW, int LDX, bool SYNC>
__device__ __forceinline__ void layer_relu(const float *W, const float *b, const float *in, float *out) {
  const int pg = point_group<PB>(), og = output_group<PB>();
  uint64_t acc[4][RP / 2];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const float bias = b[og + 16 * q];
#pragma unroll
    for (int p = 0; p < RP / 2; ++p) acc[q][p] = pk2(bias, bias);
  }
#pragma unroll 8
  for (int k0 = 0; k0 < K; k0 += 4) {
    float4 w[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) w[q] = *reinterpret_cast<const float4 *>(W + (og + 16 * q) * LDW + k0);
#pragma unroll
    for (int kk = 0; kk < 4; ++kk) {
      uint64_t x[RP / 2];
#pragma unroll
      for (int h = 0; h < RP / 4; ++h) {
        const ulonglong2 t = *reinterpret_cast<const ulonglong2 *>(in + (k0 + kk) * LDX + 64 * h + 4 * pg);
        x[2 * h] = t.x;
        x[2 * h + 1] = t.y;
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const float wk = kk == 0 ? w[q].x : kk == 1 ? w[q].y : kk == 2 ? w[q].z : w[q].w;
        const uint64_t w2 = pk2(wk, wk);
#pragma unroll
        for (int p = 0; p < RP / 2; ++p) acc[q][p] = fma2(w2, x[p], acc[q][p]);
      }
    }
  }
  if (SYNC) __syncthreads();
#pragma unroll
  for (int q = 0; q < 4; ++q)
#pragma unroll
    for (int h = 0; h < RP / 4; ++h) {
      float4 r;
      upk2(acc[q][2 * h], r.x, r.y);
      upk2(acc[q][2 * h + 1], r.z, r.w);
      r.x = fmaxf(r.x, 0.0f);
      r.y = fmaxf(r.y, 0.0f);
      r.z = fmaxf(r.z, 0.0f);
      r.w = fmaxf(r.w, 0.0f);
      *reinterpret_cast<float4 *>(out + (og + 16 * q) * LDX + 64 * h + 4 * pg) = r;
    }
}

// This thread's part of the inputs of point p (column r of X): PARTS threads
// share a point, thread `part` taking 16/PARTS octaves of u and v, 32/PARTS
// latent values and a share of the rest.  Row kDecIn is zero.
template <int PARTS, int LDX>
__device__ __forceinline__ void build_inputs(const fabric_gbuffer &g, int64_t p, const float *__restrict__ lat,
                                             int part, float *X, int r) {
  constexpr int NL = kLatent / PARTS, NO = 16 / PARTS;
  const float coord = part < PARTS / 2 ? g.u[p] : g.v[p];
  if ((reinterpret_cast<uintptr_t>(lat) & 15) == 0) {
#pragma unroll
    for (int i = 0; i < NL / 4; ++i) {
      const float4 t = __ldg(reinterpret_cast<const float4 *>(lat + part * NL) + i);
      X[(part * NL + 4 * i) * LDX + r] = t.x;
      X[(part * NL + 4 * i + 1) * LDX + r] = t.y;
      X[(part * NL + 4 * i + 2) * LDX + r] = t.z;
      X[(part * NL + 4 * i + 3) * LDX + r] = t.w;
    }
  } else {
#pragma unroll
    for (int i = 0; i < NL; ++i) X[(part * NL + i) * LDX + r] = __ldg(lat + part * NL + i);
  }
  if (part == 0) {
    X[64 * LDX + r] = (logf(fmaxf(g.radius[p], kRFloor)) - kLogRC0) * kLogRInvC1;
#pragma unroll
    for (int i = 0; i < 3; ++i) X[(65 + i) * LDX + r] = g.wi[3 * p + i];
  }
  if (part == PARTS - 1) {
#pragma unroll
    for (int i = 0; i < 3; ++i) X[(68 + i) * LDX + r] = g.wo[3 * p + i];
    X[kDecIn * LDX + r] = 0.0f;
  }
  const float f0 = coord - floorf(coord);
  const int k0 = (part * NO) & 7;
#pragma unroll
  for (int k = 0; k < NO; ++k) {   // as octaves_accurate forms them
    const float sc = f0 * (float)(1 << (k0 + k));
    float s, c;
    sincospif(2.0f * (sc - floorf(sc)), &s, &c);
    X[(kLatent + 2 * (part * NO + k)) * LDX + r] = s;
    X[(kLatent + 2 * (part * NO + k) + 1) * LDX + r] = c;
  }
}

// ---------------------------------------------------------------------------
// Forward
// ---------------------------------------------------------------------------
struct FwdArgs {
  fabric_gbuffer g;
  const DevMaterial *mats;
  int n_mat;
  const float *latents;
  int n_lat;
  const float *dec;
  float *rgb, *comps, *y_raw;
  int *status;
};

template <int RP>
constexpr size_t fwd_smem_bytes() {
  return (size_t)(kSParams + kInRows * 16 * RP + kOut * 16 * RP) * 4;
}

// Persistent CTAs (two per SM) over tiles of 16 RP points; each layer's
// outputs replace its inputs in shared memory.
template <int RP>
__global__ void __launch_bounds__(kThreads, 2) decoder_fp32_kernel(const FwdArgs a) {
  constexpr int TILE = 16 * RP, PARTS = kThreads / TILE;
  extern __shared__ __align__(16) float sm[];
  float *W = sm, *X = sm + kSParams, *Y = X + kInRows * TILE;
  stage_params<kThreads>(a.dec, W);
  const int t = threadIdx.x, r = t % TILE, part = t / TILE;
  const int64_t n_tiles = (a.g.n + TILE - 1) / TILE;
  const int mat_limit = a.rgb ? min(a.n_lat, a.n_mat) : a.n_lat;
  for (int64_t tile = blockIdx.x; tile < n_tiles; tile += gridDim.x) {
    const int64_t p = tile * TILE + r;
    const bool in = p < a.g.n;
    const int mat = in ? a.g.material[p] : 0;
    const bool ok = in && mat < mat_limit;
    // points past the end and bad indices compute point 0's (or their own
    // query's) network with latent 0; nothing of it is stored
    build_inputs<PARTS, TILE>(a.g, in ? p : 0, a.latents + (int64_t)(ok ? mat : 0) * kLatent, part, X, r);
    __syncthreads();
    layer_relu<RP, 2, kInRows, kLd1, TILE, true>(W + kSW1, W + kSB, X, X);
    __syncthreads();
    layer_relu<RP, 2, kHidden, kLdH, TILE, true>(W + kSW2, W + kSB + kHidden, X, X);
    __syncthreads();
    layer_relu<RP, 2, kHidden, kLdH, TILE, true>(W + kSW3, W + kSB + 2 * kHidden, X, X);
    __syncthreads();
    // the head: kOut / PARTS outputs of one point per thread
#pragma unroll
    for (int q = 0; q < kOut / PARTS; ++q) {
      const int k = part * (kOut / PARTS) + q;
      float acc = W[kSB + 3 * kHidden + k];
      const float *w = W + kSW4 + k * kLdH;
#pragma unroll 4
      for (int i = 0; i < kHidden; i += 4) {
        const float4 c = *reinterpret_cast<const float4 *>(w + i);
        acc = fmaf(c.x, X[i * TILE + r], acc);
        acc = fmaf(c.y, X[(i + 1) * TILE + r], acc);
        acc = fmaf(c.z, X[(i + 2) * TILE + r], acc);
        acc = fmaf(c.w, X[(i + 3) * TILE + r], acc);
      }
      Y[k * TILE + r] = acc;
    }
    __syncthreads();
    if (part == 0 && in) {
      float y[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) y[k] = Y[k * TILE + r];
      if (!ok) {
        atomicOr(a.status, kStatusBadMaterial);
#pragma unroll
        for (int k = 0; k < 4; ++k) y[k] = __int_as_float(0x7FC00000);
      }
      if (a.y_raw) store_row4(a.y_raw, p, y[0], y[1], y[2], y[3]);
      if (a.comps || a.rgb) {
        const float nan = y[0];
        const float c0 = ok ? fmaxf(0.0f, y[0]) : nan, c1 = ok ? fmaxf(0.0f, y[1]) : nan;
        const float s0 = ok ? fmaxf(0.0f, expm1f(y[2]) / kSpecK) : nan, s1 = ok ? fmaxf(0.0f, expm1f(y[3]) / kSpecK) : nan;
        if (a.comps) store_row4(a.comps, p, c0, c1, s0, s1);
        if (a.rgb) {
          const DevMaterial &m = a.mats[ok ? mat : 0];
#pragma unroll
          for (int ch = 0; ch < 3; ++ch)
            a.rgb[3 * p + ch] = m.kd[0][ch] * c0 + m.kd[1][ch] * c1 + m.ks[0][ch] * s0 + m.ks[1][ch] * s1;
        }
      }
    }
    // the next tile's inputs overwrite X, which every thread has finished
    // reading; Y is next written three barriers on
  }
}

// ---------------------------------------------------------------------------
// Forward and backward
// ---------------------------------------------------------------------------
constexpr int kBwdThreads = 512;
constexpr int kBlock = 32;         // rows a warp's eight point groups cover
constexpr int kTR = 4 * kBlock;    // rows per tile
constexpr int kLdR = kTR + 4;      // row stride: rows in different banks for 16-byte reads along the rows

struct BwdArgs {
  fabric_gbuffer g;
  const float *latents;
  int n_lat;
  const float *dec;
  const float *dy;       // [n][4] or null
  const float *target;   // [n][4] or null
  int loss_mode;         // FABRIC_LOSS_EQ11 or FABRIC_LOSS_RENDERED
  float inv_batch;       // 1/B for the loss
  float *partial;        // [grid][kDecParams]
  double *loss_partial;  // [grid]
  float *dlat_rows;      // [n][32]
  int *status;
};

constexpr size_t kBwdSmem = (size_t)(kSParams + (kInRows + 4 * kHidden + kOut) * kLdR) * 4;
static_assert(kBwdSmem <= 232448, "one CTA per SM");

// din[i][r] = (sum_o W[o][i] dout[o][r]) (pre[i][r] > 0) for this thread's
// points 4 pg .. and inputs NI ig .. NI ig + NI - 1 (NI = 4 or 2).
template <int NI, int K, int LDW>
__device__ __forceinline__ void layer_input_grad(const float *W, const float *dout, const float *pre, float *din) {
  const int pg = point_group<4>(), ig = output_group<4>();
  uint64_t acc[NI][2];
#pragma unroll
  for (int q = 0; q < NI; ++q) acc[q][0] = acc[q][1] = 0ull;
#pragma unroll 8
  for (int o = 0; o < K; ++o) {
    float w[NI];
    if (NI == 4) {
      const float4 t = *reinterpret_cast<const float4 *>(W + o * LDW + 4 * ig);
      w[0] = t.x;
      w[1] = t.y;
      w[2 % NI] = t.z;
      w[3 % NI] = t.w;
    } else {
      const float2 t = *reinterpret_cast<const float2 *>(W + o * LDW + 2 * ig);
      w[0] = t.x;
      w[1] = t.y;
    }
    const ulonglong2 d = *reinterpret_cast<const ulonglong2 *>(dout + o * kLdR + 4 * pg);
#pragma unroll
    for (int q = 0; q < NI; ++q) {
      const uint64_t w2 = pk2(w[q], w[q]);
      acc[q][0] = fma2(w2, d.x, acc[q][0]);
      acc[q][1] = fma2(w2, d.y, acc[q][1]);
    }
  }
#pragma unroll
  for (int q = 0; q < NI; ++q) {
    const int i = NI * ig + q;
    float4 r;
    upk2(acc[q][0], r.x, r.y);
    upk2(acc[q][1], r.z, r.w);
    if (pre) {
      const float4 h = *reinterpret_cast<const float4 *>(pre + i * kLdR + 4 * pg);
      r.x = h.x > 0.0f ? r.x : 0.0f;
      r.y = h.y > 0.0f ? r.y : 0.0f;
      r.z = h.z > 0.0f ? r.z : 0.0f;
      r.w = h.w > 0.0f ? r.w : 0.0f;
    }
    *reinterpret_cast<float4 *>(din + i * kLdR + 4 * pg) = r;
  }
}

// Weight gradients live in registers for all of the CTA's blocks.  A thread's
// place is (og, ig): outputs og + 16 q, inputs ig + 16 s; the two halves of a
// warp share it and take the blocks 0, 1 and 2, 3 of a tile.  Each block's
// sum is a chain over its 32 rows in order, and the running sums add the
// blocks in order: half h keeps those of q = 2h, 2h + 1, and the halves
// exchange the others by shuffles.
__device__ __forceinline__ int grad_half() { return (threadIdx.x >> 4) & 1; }
__device__ __forceinline__ int grad_og() { return ((threadIdx.x >> 3) & 1) + 2 * ((threadIdx.x >> 5) & 7); }
__device__ __forceinline__ int grad_ig() { return (threadIdx.x & 7) + 8 * (threadIdx.x >> 8); }

template <int NS>
__device__ __forceinline__ void layer_weight_grad(const float *dout, const float *in, int nb, float (*dW)[NS]) {
  const int og = grad_og(), ig = grad_ig(), half = grad_half();
  float sum[2][4][NS];
#pragma unroll
  for (int j = 0; j < 2; ++j) {
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
      for (int s = 0; s < NS; ++s) sum[j][q][s] = 0.0f;
    if (j >= nb) break;
    const int r0 = kBlock * (2 * half + j);
#pragma unroll 2
    for (int r = r0; r < r0 + kBlock; r += 4) {
      float4 d[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) d[q] = *reinterpret_cast<const float4 *>(dout + (og + 16 * q) * kLdR + r);
#pragma unroll
      for (int s = 0; s < NS; ++s) {   // a fifth group covers inputs 64..71 only
        const float4 x = *reinterpret_cast<const float4 *>(in + (16 * s + (s == 4 ? ig & 7 : ig)) * kLdR + r);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          sum[j][q][s] = fmaf(d[q].x, x.x, sum[j][q][s]);
          sum[j][q][s] = fmaf(d[q].y, x.y, sum[j][q][s]);
          sum[j][q][s] = fmaf(d[q].z, x.z, sum[j][q][s]);
          sum[j][q][s] = fmaf(d[q].w, x.w, sum[j][q][s]);
        }
      }
    }
  }
#pragma unroll
  for (int q = 0; q < 2; ++q)
#pragma unroll
    for (int s = 0; s < NS; ++s) {
      float lo[2], hi[2];   // blocks 0, 1 and 2, 3 of output og + 16 (2 half + q)
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const float keep = half ? sum[j][q + 2][s] : sum[j][q][s];
        const float got = __shfl_xor_sync(0xFFFFFFFFu, half ? sum[j][q][s] : sum[j][q + 2][s], 16);
        lo[j] = half ? got : keep;
        hi[j] = half ? keep : got;
      }
      float w = dW[q][s] + lo[0];
      if (nb > 1) w += lo[1];
      if (nb > 2) w += hi[0];
      if (nb > 3) w += hi[1];
      dW[q][s] = w;
    }
}

// Bias gradients: thread (o, blk) = (t / 4, t % 4) of the first 4 n_out threads
// adds block blk's rows of output o in order; the blocks' sums are added in
// order in the lane of block 0.
__device__ __forceinline__ void bias_grad(const float *dout, int n_out, int nb, float &db) {
  const int t = threadIdx.x, blk = t & 3;
  if ((t & ~31) >= 4 * n_out) return;            // whole warps
  const float *d = dout + min(t >> 2, n_out - 1) * kLdR + kBlock * blk;
  float s = 0.0f;
#pragma unroll
  for (int k = 0; k < kBlock; k += 4) {
    const float4 v = *reinterpret_cast<const float4 *>(d + k);
    s += v.x;
    s += v.y;
    s += v.z;
    s += v.w;
  }
  db += s;
#pragma unroll
  for (int k = 1; k < 4; ++k) {
    const float o = __shfl_down_sync(0xFFFFFFFFu, s, k);
    if (k < nb) db += o;
  }
}

// One CTA of 16 warps per SM.  The batch is cut into blocks of 32 rows; CTA c
// takes blocks c, c + grid, ..., four of them at a time as one tile (warps
// without a block wait), so that 65 536 rows are 13 or 14 blocks a CTA.  The
// parameters, a tile's inputs, activations and gradients fill the shared
// memory (226 KB: dA2 takes H3's place, dA1 dA3's, the latent gradient H2's).
// Bound by shared-memory latency and bandwidth: with eight warps on 64-row
// tiles (165 KB) the kernel took 180 us for 65 536 rows.
__global__ void __launch_bounds__(kBwdThreads, 1) decoder_bwd_kernel(const BwdArgs a) {
  extern __shared__ __align__(16) float sm[];
  float *W = sm;
  float *X = W + kSParams;               // [72][kLdR]
  float *H1 = X + kInRows * kLdR;        // activations [64][kLdR]
  float *H2 = H1 + kHidden * kLdR;
  float *H3 = H2 + kHidden * kLdR;
  float *D = H3 + kHidden * kLdR;        // [64][kLdR]
  float *DY = D + kHidden * kLdR;        // [4][kLdR]
  grid_dependency_wait();
  grid_dependents_launch();
  stage_params<kBwdThreads>(a.dec, W);
  const int t = threadIdx.x, r = t % kTR, part = t / kTR;
  const int rb = (t >> 5) & 3;
  float dW1[2][5] = {}, dW2[2][4] = {}, dW3[2][4] = {}, dW4 = 0.0f;
  float db1 = 0.0f, db2 = 0.0f, db3 = 0.0f, db4 = 0.0f;
  double loss_acc = 0.0;
  const int64_t n_blocks = (a.g.n + kBlock - 1) / kBlock, stride = gridDim.x;
  for (int64_t b0 = blockIdx.x; b0 < n_blocks; b0 += 4 * stride) {
    const int nb = (int)min((int64_t)4, (n_blocks - b0 + stride - 1) / stride), rows = nb * kBlock;
    const bool busy = rb < nb;             // this warp's row block exists (layers)
    auto point = [&](int row) { return (b0 + (row / kBlock) * stride) * kBlock + row % kBlock; };
    const int64_t p = point(r);
    const bool in = r < rows;
    const int mat = in && p < a.g.n ? (int)a.g.material[p] : -1;
    bool ok = mat >= 0;
    if (mat >= a.n_lat) {
      if (part == 0) atomicOr(a.status, kStatusBadMaterial);
      ok = false;
    }
    if (ok) {
      build_inputs<4, kLdR>(a.g, p, a.latents + (int64_t)mat * kLatent, part, X, r);
    } else if (in) {
      for (int i = part * 18; i < part * 18 + 18; ++i) X[i * kLdR + r] = 0.0f;
    }
    __syncthreads();
    if (busy) layer_relu<4, 4, kInRows, kLd1, kLdR, false>(W + kSW1, W + kSB, X, H1);
    __syncthreads();
    if (busy) layer_relu<4, 4, kHidden, kLdH, kLdR, false>(W + kSW2, W + kSB + kHidden, H1, H2);
    __syncthreads();
    if (busy) layer_relu<4, 4, kHidden, kLdH, kLdR, false>(W + kSW3, W + kSB + 2 * kHidden, H2, H3);
    __syncthreads();
    // ---- head and output gradient: output `part` of row r
    if (in) {
      float y = W[kSB + 3 * kHidden + part];
      const float *w = W + kSW4 + part * kLdH;
#pragma unroll 4
      for (int i = 0; i < kHidden; i += 4) {
        const float4 c = *reinterpret_cast<const float4 *>(w + i);
        y = fmaf(c.x, H3[i * kLdR + r], y);
        y = fmaf(c.y, H3[(i + 1) * kLdR + r], y);
        y = fmaf(c.z, H3[(i + 2) * kLdR + r], y);
        y = fmaf(c.w, H3[(i + 3) * kLdR + r], y);
      }
      float d = 0.0f;
      if (ok)
        d = a.target ? loss_grad(part, y, a.target[4 * p + part], a.g.wi[3 * p + 2], a.loss_mode, a.inv_batch, &loss_acc)
                     : a.dy[4 * p + part];
      DY[part * kLdR + r] = d;
    }
    __syncthreads();
    // ---- backward
    if (busy) layer_input_grad<4, kOut, kLdH>(W + kSW4, DY, H3, D);        // dA3
    if (t < kOut * kHidden) {
      const float *d = DY + (t >> 6) * kLdR, *h = H3 + (t & 63) * kLdR;     // dW4[t / 64][t % 64]
      for (int blk = 0; blk < nb; ++blk, d += kBlock, h += kBlock) {
        float s = 0.0f;
#pragma unroll
        for (int k = 0; k < kBlock; k += 4) {
          const float4 u = *reinterpret_cast<const float4 *>(d + k), v = *reinterpret_cast<const float4 *>(h + k);
          s = fmaf(u.x, v.x, s);
          s = fmaf(u.y, v.y, s);
          s = fmaf(u.z, v.z, s);
          s = fmaf(u.w, v.w, s);
        }
        dW4 += s;
      }
    }
    bias_grad(DY, kOut, nb, db4);
    __syncthreads();
    layer_weight_grad<4>(D, H2, nb, dW3);
    bias_grad(D, kHidden, nb, db3);
    if (busy) layer_input_grad<4, kHidden, kLdH>(W + kSW3, D, H2, H3);     // dA2, over H3
    __syncthreads();
    layer_weight_grad<4>(H3, H1, nb, dW2);
    bias_grad(H3, kHidden, nb, db2);
    if (busy) layer_input_grad<4, kHidden, kLdH>(W + kSW2, H3, H1, D);     // dA1, over dA3
    __syncthreads();
    layer_weight_grad<5>(D, X, nb, dW1);
    bias_grad(D, kHidden, nb, db1);
    if (a.dlat_rows) {
      // d x[0:32] = W1[:, 0:32]^T dA1, over H2; then row by row, eight floats of one row per thread
      if (busy) layer_input_grad<2, kHidden, kLd1>(W + kSW1, D, nullptr, H2);
      __syncthreads();
      const int row = t >> 2, c0 = 8 * (t & 3);
      const int64_t q = point(row);
      if (row < rows && q < a.g.n) {
        float4 *dst = reinterpret_cast<float4 *>(a.dlat_rows + q * kLatent + c0);
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          const float *s = H2 + (c0 + 4 * k) * kLdR + row;
          dst[k] = make_float4(s[0], s[kLdR], s[2 * kLdR], s[3 * kLdR]);
        }
      }
    }
    __syncthreads();
  }
  float *out = a.partial + (int64_t)blockIdx.x * kDecParams;
  const int og = grad_og(), ig = grad_ig(), half = grad_half();
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const int o = og + 16 * (2 * half + q);
#pragma unroll
    for (int s = 0; s < 5; ++s) {
      const int i = 16 * s + ig;
      if (i < kDecIn) out[kOffW1 + o * kDecIn + i] = dW1[q][s];
    }
#pragma unroll
    for (int s = 0; s < 4; ++s) {
      out[kOffW2 + o * kHidden + 16 * s + ig] = dW2[q][s];
      out[kOffW3 + o * kHidden + 16 * s + ig] = dW3[q][s];
    }
  }
  if (t < kOut * kHidden) out[kOffW4 + t] = dW4;
  if (t < 4 * kHidden && (t & 3) == 0) {
    out[kOffB1 + t / 4] = db1;
    out[kOffB2 + t / 4] = db2;
    out[kOffB3 + t / 4] = db3;
    if (t < 4 * kOut) out[kOffB4 + t / 4] = db4;
  }
  // loss: lanes by a fixed tree, then the 16 warps in order
  double *loss_red = reinterpret_cast<double *>(X);
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) loss_acc += __shfl_down_sync(0xFFFFFFFFu, loss_acc, off);
  if ((t & 31) == 0) loss_red[t >> 5] = loss_acc;
  __syncthreads();
  if (t == 0) {
    double s = loss_red[0];
    for (int k = 1; k < kBwdThreads / 32; ++k) s += loss_red[k];
    a.loss_partial[blockIdx.x] = s;
  }
}

template <int RP>
cudaError_t launch_fwd(const FwdArgs &a, int sm_count, cudaStream_t s) {
  const cudaError_t e = ensure_max_dyn_smem(reinterpret_cast<const void *>(decoder_fp32_kernel<RP>), (int)fwd_smem_bytes<RP>());
  if (e != cudaSuccess) return e;
  const int64_t tiles = (a.g.n + 16 * RP - 1) / (16 * RP);
  const int64_t grid = std::min<int64_t>(tiles, 2 * (int64_t)(sm_count > 0 ? sm_count : 148));
  decoder_fp32_kernel<RP><<<(unsigned)grid, kThreads, fwd_smem_bytes<RP>(), s>>>(a);
  return cudaGetLastError();
}

// 128-point tiles, or 64-point ones while those leave CTAs without work.
cudaError_t launch_fwd(const FwdArgs &a, int sm_count, cudaStream_t s) {
  return a.g.n > 128 * 2 * (int64_t)(sm_count > 0 ? sm_count : 148) ? launch_fwd<8>(a, sm_count, s) : launch_fwd<4>(a, sm_count, s);
}

int bwd_grid(int64_t n, int sm_count) {
  const int64_t blocks = (n + kBlock - 1) / kBlock;
  return (int)std::max<int64_t>(1, std::min<int64_t>(blocks, sm_count > 0 ? sm_count : 148));
}

}  // namespace

cudaError_t launch_decoder_fp32(const fabric_gbuffer &g, const DevMaterial *mats, int n_mat, const float *latents,
                                const float *dec, float *rgb, float *comps, float *y_raw, int *status, int sm_count,
                                cudaStream_t s) {
  return launch_fwd(FwdArgs{g, mats, n_mat, latents, mats ? n_mat : 0, dec, rgb, comps, y_raw, status}, sm_count, s);
}

cudaError_t launch_decoder_raw(const fabric_gbuffer &g, const float *latents, int n_lat, const float *dec,
                               float *y_raw, int *status, int sm_count, cudaStream_t s) {
  return launch_fwd(FwdArgs{g, nullptr, 0, latents, n_lat, dec, nullptr, nullptr, y_raw, status}, sm_count, s);
}

// Work layout: [grid][kDecParams] floats | [grid] doubles | [n][32] floats.
size_t decoder_backward_work_bytes(int64_t n, int sm_count) {
  const int grid = bwd_grid(n, sm_count);
  size_t bytes = (size_t)grid * kDecParams * 4;
  bytes = (bytes + 15) & ~size_t(15);
  bytes += (size_t)grid * 8;
  bytes = (bytes + 15) & ~size_t(15);
  bytes += (size_t)n * kLatent * 4;
  return bytes + 64;
}

cudaError_t launch_decoder_backward(const fabric_gbuffer &g, const float *latents, int n_lat, const float *dec,
                                    const float *dy, const float *target, int loss_mode, float *ddec, float *dlat,
                                    double *loss, void *work, int sm_count, int *status, cudaStream_t s) {
  cudaError_t e = ensure_max_dyn_smem(reinterpret_cast<const void *>(decoder_bwd_kernel), (int)kBwdSmem);
  if (e != cudaSuccess) return e;
  const int grid = bwd_grid(g.n, sm_count);
  uint8_t *w = static_cast<uint8_t *>(work);
  float *partial = reinterpret_cast<float *>(w);
  size_t off = ((size_t)grid * kDecParams * 4 + 15) & ~size_t(15);
  double *loss_part = reinterpret_cast<double *>(w + off);
  off = (off + (size_t)grid * 8 + 15) & ~size_t(15);
  float *rows = reinterpret_cast<float *>(w + off);
  BwdArgs a;
  a.g = g;
  a.latents = latents;
  a.n_lat = n_lat;
  a.dec = dec;
  a.dy = dy;
  a.target = target;
  a.loss_mode = loss_mode;
  a.inv_batch = 1.0f / (float)(g.n > 0 ? g.n : 1);
  a.partial = partial;
  a.loss_partial = loss_part;
  a.dlat_rows = dlat ? rows : nullptr;
  a.status = status;
  e = launch_dependent(decoder_bwd_kernel, grid, kBwdThreads, kBwdSmem, s, a);
  if (e != cudaSuccess) return e;
  return launch_decoder_grad_finish(g, n_lat, partial, grid, kDecParams, loss_part, rows, ddec, loss, dlat, s);
}

}  // namespace fab
