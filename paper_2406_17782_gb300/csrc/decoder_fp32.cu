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

constexpr int kThreads = 256;
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

// The flat parameters (float-aligned) into shared memory.
__device__ __forceinline__ void stage_params(const float *__restrict__ dec, float *W) {
  for (int e = threadIdx.x; e < kHidden * kLd1; e += kThreads) {
    const int o = e / kLd1, i = e % kLd1;
    W[kSW1 + e] = i < kDecIn ? dec[kOffW1 + o * kDecIn + i] : 0.0f;
  }
  for (int e = threadIdx.x; e < kHidden * kHidden; e += kThreads) {
    const int o = e / kHidden, i = e % kHidden;
    W[kSW2 + o * kLdH + i] = dec[kOffW2 + e];
    W[kSW3 + o * kLdH + i] = dec[kOffW3 + e];
  }
  for (int e = threadIdx.x; e < kOut * kHidden; e += kThreads)
    W[kSW4 + (e / kHidden) * kLdH + e % kHidden] = dec[kOffW4 + e];
  for (int e = threadIdx.x; e < 3 * kHidden + kOut; e += kThreads)
    W[kSB + e] = e < kHidden       ? dec[kOffB1 + e]
                 : e < 2 * kHidden ? dec[kOffB2 + e - kHidden]
                 : e < 3 * kHidden ? dec[kOffB3 + e - 2 * kHidden]
                                   : dec[kOffB4 + e - 3 * kHidden];
}

// Thread t's place in a layer: point group pg (points 4 pg .. 4 pg + 3 of every
// 64) and output group og of 16 (outputs og, og + 16, ...).  A warp holds
// eight point groups (one 128-byte read) and four output groups (rows in
// different banks).
__device__ __forceinline__ int point_group() { return (threadIdx.x & 7) | ((threadIdx.x >> 2) & 8); }
__device__ __forceinline__ int output_group() { return ((threadIdx.x >> 3) & 3) | ((threadIdx.x >> 6) << 2); }

// out[o][p] = relu(b[o] + sum_k W[o][k] in[k][p]) for this thread's outputs of
// RP = 4 or 8 points; K a multiple of four.  SYNC: `out` may be `in` (a CTA
// barrier between the last read and the first write).
template <int RP, int K, int LDW, int LDX, bool SYNC>
__device__ __forceinline__ void layer_relu(const float *W, const float *b, const float *in, float *out) {
  const int pg = point_group(), og = output_group();
  uint64_t acc[4][RP / 2];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const float bias = b[og + 16 * q];
#pragma unroll
    for (int p = 0; p < RP / 2; ++p) acc[q][p] = pk2(bias, bias);
  }
#pragma unroll 2
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
  stage_params(a.dec, W);
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
    layer_relu<RP, kInRows, kLd1, TILE, true>(W + kSW1, W + kSB, X, X);
    __syncthreads();
    layer_relu<RP, kHidden, kLdH, TILE, true>(W + kSW2, W + kSB + kHidden, X, X);
    __syncthreads();
    layer_relu<RP, kHidden, kLdH, TILE, true>(W + kSW3, W + kSB + 2 * kHidden, X, X);
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
constexpr int kTR = 64;          // rows per tile
constexpr int kLdR = kTR + 4;    // row stride: rows in different banks for 16-byte reads along the rows

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

constexpr size_t kBwdSmem = (size_t)(kSParams + (kInRows + 3 * kHidden + 2 * kHidden + kOut) * kLdR) * 4;

// din[i][r] = (sum_o W[o][i] dout[o][r]) (pre[i][r] > 0) for this thread's
// points 4 pg .. and inputs NI ig .. NI ig + NI - 1 (NI = 4 or 2).
template <int NI, int K, int LDW>
__device__ __forceinline__ void layer_input_grad(const float *W, const float *dout, const float *pre, float *din) {
  const int pg = point_group(), ig = output_group();
  uint64_t acc[NI][2];
#pragma unroll
  for (int q = 0; q < NI; ++q) acc[q][0] = acc[q][1] = 0ull;
#pragma unroll 4
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

// Weight gradients live in registers for all of the CTA's tiles: thread
// (og, ig) owns outputs og + 16 q and inputs ig + 16 s.  dW[q][s] += sum_r
// dout[o][r] in[i][r] over one tile: even and odd rows in the two packed
// lanes, added to the running sum per tile.
template <int NS>
__device__ __forceinline__ void layer_weight_grad(const float *dout, const float *in, float (*dW)[NS]) {
  const int og = output_group(), ig = point_group();
  uint64_t acc[4][NS];
#pragma unroll
  for (int q = 0; q < 4; ++q)
#pragma unroll
    for (int s = 0; s < NS; ++s) acc[q][s] = 0ull;
#pragma unroll 2
  for (int r = 0; r < kTR; r += 4) {
    ulonglong2 d[4], x[NS];
#pragma unroll
    for (int q = 0; q < 4; ++q) d[q] = *reinterpret_cast<const ulonglong2 *>(dout + (og + 16 * q) * kLdR + r);
#pragma unroll
    for (int s = 0; s < NS; ++s)   // a fifth group covers inputs 64..71 only
      x[s] = *reinterpret_cast<const ulonglong2 *>(in + (16 * s + (s == 4 ? ig & 7 : ig)) * kLdR + r);
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
      for (int s = 0; s < NS; ++s) {
        acc[q][s] = fma2(d[q].x, x[s].x, acc[q][s]);
        acc[q][s] = fma2(d[q].y, x[s].y, acc[q][s]);
      }
  }
#pragma unroll
  for (int q = 0; q < 4; ++q)
#pragma unroll
    for (int s = 0; s < NS; ++s) {
      float e, o;
      upk2(acc[q][s], e, o);
      dW[q][s] += e + o;
    }
}

// Thread t's share of a layer's bias gradient: rows 16 (t & 3) .. of output t / 4.
__device__ __forceinline__ float bias_share(const float *dout) {
  const float *d = dout + (threadIdx.x >> 2) * kLdR + 16 * (threadIdx.x & 3);
  float s = 0.0f;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const float4 v = reinterpret_cast<const float4 *>(d)[k];
    s += (v.x + v.y) + (v.z + v.w);
  }
  return s;
}

// Persistent CTAs, one per SM (the parameters, a tile's inputs, activations
// and two gradient buffers take 165 KB of shared memory).
__global__ void __launch_bounds__(kThreads, 1) decoder_bwd_kernel(const BwdArgs a) {
  extern __shared__ __align__(16) float sm[];
  float *W = sm;
  float *X = W + kSParams;               // [72][kLdR]
  float *H1 = X + kInRows * kLdR;        // activations [64][kLdR]
  float *H2 = H1 + kHidden * kLdR;
  float *H3 = H2 + kHidden * kLdR;
  float *D1 = H3 + kHidden * kLdR;       // [64][kLdR]
  float *D2 = D1 + kHidden * kLdR;
  float *DY = D2 + kHidden * kLdR;       // [4][kLdR]
  __shared__ double loss_red[kThreads];
  stage_params(a.dec, W);
  const int t = threadIdx.x, r = t % kTR, part = t / kTR;
  float dW1[4][5] = {}, dW2[4][4] = {}, dW3[4][4] = {}, dW4 = 0.0f;
  float db1 = 0.0f, db2 = 0.0f, db3 = 0.0f, db4 = 0.0f;
  double loss_acc = 0.0;
  const int64_t n_tiles = (a.g.n + kTR - 1) / kTR;
  for (int64_t tile = blockIdx.x; tile < n_tiles; tile += gridDim.x) {
    const int64_t p = tile * kTR + r;
    const int mat = p < a.g.n ? (int)a.g.material[p] : -1;
    bool ok = mat >= 0;
    if (mat >= a.n_lat) {
      if (part == 0) atomicOr(a.status, kStatusBadMaterial);
      ok = false;
    }
    if (ok) {
      build_inputs<4, kLdR>(a.g, p, a.latents + (int64_t)mat * kLatent, part, X, r);
    } else {
      for (int i = part * 18; i < part * 18 + 18; ++i) X[i * kLdR + r] = 0.0f;
    }
    __syncthreads();
    layer_relu<4, kInRows, kLd1, kLdR, false>(W + kSW1, W + kSB, X, H1);
    __syncthreads();
    layer_relu<4, kHidden, kLdH, kLdR, false>(W + kSW2, W + kSB + kHidden, H1, H2);
    __syncthreads();
    layer_relu<4, kHidden, kLdH, kLdR, false>(W + kSW3, W + kSB + 2 * kHidden, H2, H3);
    __syncthreads();
    // ---- head and output gradient: output `part` of row r
    {
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
    layer_input_grad<4, kOut, kLdH>(W + kSW4, DY, H3, D1);                 // dA3
    {
      const float *d = DY + (t >> 6) * kLdR, *h = H3 + (t & 63) * kLdR;     // dW4[t / 64][t % 64]
      float s = 0.0f;
#pragma unroll 4
      for (int k = 0; k < kTR; k += 4) {
        const float4 u = *reinterpret_cast<const float4 *>(d + k), v = *reinterpret_cast<const float4 *>(h + k);
        s = fmaf(u.x, v.x, s);
        s = fmaf(u.y, v.y, s);
        s = fmaf(u.z, v.z, s);
        s = fmaf(u.w, v.w, s);
      }
      dW4 += s;
      if (t < 4 * kOut) db4 += bias_share(DY);
    }
    __syncthreads();
    layer_weight_grad<4>(D1, H2, dW3);
    db3 += bias_share(D1);
    layer_input_grad<4, kHidden, kLdH>(W + kSW3, D1, H2, D2);              // dA2
    __syncthreads();
    layer_weight_grad<4>(D2, H1, dW2);
    db2 += bias_share(D2);
    layer_input_grad<4, kHidden, kLdH>(W + kSW2, D2, H1, D1);              // dA1
    __syncthreads();
    layer_weight_grad<5>(D1, X, dW1);
    db1 += bias_share(D1);
    if (a.dlat_rows) {
      // d x[0:32] = W1[:, 0:32]^T dA1
      layer_input_grad<2, kHidden, kLd1>(W + kSW1, D1, nullptr, D2);
      __syncthreads();
      // row by row through D2 [32][rows]: eight floats of one row per thread
      const int row = t >> 2, c0 = 8 * (t & 3);
      const int64_t q = tile * kTR + row;
      if (q < a.g.n) {
        float4 *dst = reinterpret_cast<float4 *>(a.dlat_rows + q * kLatent + c0);
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          const float *s = D2 + (c0 + 4 * k) * kLdR + row;
          dst[k] = make_float4(s[0], s[kLdR], s[2 * kLdR], s[3 * kLdR]);
        }
      }
    }
    __syncthreads();
  }
  float *out = a.partial + (int64_t)blockIdx.x * kDecParams;
  const int og = output_group(), ig = point_group();
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int o = og + 16 * q;
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
  out[kOffW4 + t] = dW4;
  // biases: the four row shares of an output sit in neighbouring lanes
  db1 += __shfl_xor_sync(0xFFFFFFFFu, db1, 1);
  db2 += __shfl_xor_sync(0xFFFFFFFFu, db2, 1);
  db3 += __shfl_xor_sync(0xFFFFFFFFu, db3, 1);
  db4 += __shfl_xor_sync(0xFFFFFFFFu, db4, 1);
  db1 += __shfl_xor_sync(0xFFFFFFFFu, db1, 2);
  db2 += __shfl_xor_sync(0xFFFFFFFFu, db2, 2);
  db3 += __shfl_xor_sync(0xFFFFFFFFu, db3, 2);
  db4 += __shfl_xor_sync(0xFFFFFFFFu, db4, 2);
  if ((t & 3) == 0) {
    out[kOffB1 + t / 4] = db1;
    out[kOffB2 + t / 4] = db2;
    out[kOffB3 + t / 4] = db3;
    if (t < 4 * kOut) out[kOffB4 + t / 4] = db4;
  }
  loss_red[t] = loss_acc;
  __syncthreads();
  if (t == 0) {
    double s = 0.0;
    for (int k = 0; k < kThreads; ++k) s += loss_red[k];
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
  const int64_t tiles = (n + kTR - 1) / kTR;
  return (int)std::max<int64_t>(1, std::min<int64_t>(tiles, sm_count > 0 ? sm_count : 148));
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
  decoder_bwd_kernel<<<grid, kThreads, kBwdSmem, s>>>(a);
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  return launch_decoder_grad_finish(g, n_lat, partial, grid, kDecParams, loss_part, rows, ddec, loss, dlat, s);
}

}  // namespace fab
