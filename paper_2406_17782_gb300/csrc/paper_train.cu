// paper_train.cu -- FP32 training kernels of the paper's decoder structure
// (Sec. 4.2 "Decoder", Fig. 3; losses of Sec. 4.3, Eq. 9-11) and of its
// 64-wide parameter encoder, for fabric_paper_train_step.
//
// The decoder's layers run over the whole batch as FP32 products of row-major
// activation matrices on the CUDA cores: the forward pass keeps every
// post-activation matrix (a leaky ReLU keeps the sign, so its derivative is
// read from the output), the input gradients take the same kernel (the
// forward's weights are transposed first), and the weight gradients are partial sums over fixed
// chunks of the batch, summed in a fixed order, so every step is bitwise
// repeatable.  The head (four outputs), the loss, the head's input gradient
// and its weight gradient are one pass over the last activations.  The
// per-material latent gradient sums the first layer's gradient over each
// material's queries (listed, in a fixed order) and multiplies by the latent
// block of S1.
#include <algorithm>
#include <cmath>

#include "f32x2.h"
#include "fabric_internal.h"
#include "paper_net.h"
#include "train_common.cuh"

namespace fab {
namespace {

__device__ __forceinline__ void pn_copy16(float *dst, const float *src, bool in) {   // zeros when !in
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src),
               "r"(in ? 16 : 0)
               : "memory");
}
__device__ __forceinline__ void pn_copy_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void pn_copy_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// Both products give a thread 8 x 8 outputs.  Shared memory delivers 128
// bytes per cycle and SM into registers (about twice that where a warp reads
// one or two addresses), so 8 x 8 is the smallest tile whose reads fit
// beside the multiply-adds; operands arrive by asynchronous 16-byte copies in
// three stages, one barrier a stage.  The form before (stages of depth 8
// through registers, two CTAs of 256 threads) took 68 us for a 128-wide layer
// of 65 536 rows.
constexpr int kStages = 3;
constexpr int kDepth = 16;         // depth of one stage of a layer
constexpr int kRowDepth = 32;      // rows of one stage of a weight gradient

// Epilogue of a layer: forward (bias, residual, leaky ReLU) or input gradient
// (addend, leaky ReLU derivative of the layer's own output).
struct Epi {
  const float *bias;      // [N] (forward)
  const float *res;       // residual / addend [M][ld_res] or null
  int ld_res;
  const float *h;         // post-activation whose derivative multiplies (input gradient) or null
  int ld_h;
  float *out;
  int ld_out;
};

// out[i][j] = epi(sum_k A[i][k] B[k][j]) for i < M, j < BN; rows of A (length
// lda) and B (length ldb >= BN) contiguous and 16-byte aligned, K a multiple of
// four.  BM x BN outputs per CTA; thread (ty, tx) has rows ty + q BM/8 and
// columns 4 tx and BN/2 + 4 tx (and what follows).  A is staged as rows of 16
// at a stride of 20 and read four k at a time, B as it lies; one packed fma
// per two columns (with both operands read along k and scalar fma, two of a
// fma's registers share a register bank half of the time: 58 us for a
// 128-wide layer of 65 536 rows).  Every output is one chain of fma over k in
// order.  GRAD: input gradient.
template <int BM, int BN, bool GRAD>
__global__ void __launch_bounds__(BM *BN / 64, 3) pn_layer_kernel(const float *__restrict__ A, int lda,
                                                                  const float *__restrict__ B, int ldb, int64_t M,
                                                                  int K, Epi e) {
  constexpr int T = BM * BN / 64, TX = BN / 8, TY = BM / 8, LD = kDepth + 4;
  constexpr int PA = kDepth / 4, PR = T / PA;   // pieces of a row of A, rows copied per pass
  constexpr int PB = T / (BN / 4);       // rows of B copied per pass
  static_assert(BM % PR == 0 && kDepth % PB == 0, "copy layout");
  constexpr int kStageFloats = BM * LD + kDepth * BN;
  extern __shared__ __align__(16) float lsm[];   // [kStages][kStageFloats]
  const int tid = threadIdx.x, tx = tid % TX, ty = tid / TX;
  const int64_t i0 = (int64_t)blockIdx.x * BM;
  if (!GRAD) grid_dependency_wait();   // GRAD: waited for at the end (see launch_paper_train)
  grid_dependents_launch();
  const int steps = (K + kDepth - 1) / kDepth;
  const int cr = tid / PA, cp = 4 * (tid % PA), br = tid / (BN / 4), bc = 4 * (tid % (BN / 4));
  const float *ga = A + (i0 + cr) * lda + cp, *gb = B + br * ldb + bc;
  bool row_in[BM / PR];
#pragma unroll
  for (int q = 0; q < BM / PR; ++q) row_in[q] = i0 + cr + PR * q < M;
  auto load = [&](int step) {
    float *st = lsm + step % kStages * kStageFloats;
    const int left = K - step * kDepth;
#pragma unroll
    for (int q = 0; q < BM / PR; ++q) {
      const bool in = cp < left && row_in[q];
      pn_copy16(st + (cr + PR * q) * LD + cp, in ? ga + (int64_t)q * PR * lda : A, in);
    }
#pragma unroll
    for (int q = 0; q < kDepth / PB; ++q) {
      const bool in = br + PB * q < left;
      pn_copy16(st + BM * LD + (br + PB * q) * BN + bc, in ? gb + q * PB * ldb : B, in);
    }
    ga += kDepth;
    gb += kDepth * ldb;
  };
  uint64_t acc[8][4];
#pragma unroll
  for (int q = 0; q < 8; ++q)
#pragma unroll
    for (int t = 0; t < 4; ++t) acc[q][t] = 0ull;
  load(0);
  pn_copy_commit();
  if (steps > 1) load(1);
  pn_copy_commit();
  for (int step = 0; step < steps; ++step) {
    pn_copy_wait<1>();
    __syncthreads();
    if (step + 2 < steps) load(step + 2);
    pn_copy_commit();
    const float *sa = lsm + step % kStages * kStageFloats + ty * LD, *sb = lsm + step % kStages * kStageFloats + BM * LD + 4 * tx;
#pragma unroll 2
    for (int kk = 0; kk < kDepth / 4; ++kk) {
      float4 a[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) a[q] = *reinterpret_cast<const float4 *>(sa + q * TY * LD + 4 * kk);
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const ulonglong2 b0 = *reinterpret_cast<const ulonglong2 *>(sb + (4 * kk + k) * BN);
        const ulonglong2 b1 = *reinterpret_cast<const ulonglong2 *>(sb + (4 * kk + k) * BN + BN / 2);
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          const float av = k == 0 ? a[q].x : k == 1 ? a[q].y : k == 2 ? a[q].z : a[q].w;
          const uint64_t a2 = pk2(av, av);
          acc[q][0] = fma2(a2, b0.x, acc[q][0]);
          acc[q][1] = fma2(a2, b0.y, acc[q][1]);
          acc[q][2] = fma2(a2, b1.x, acc[q][2]);
          acc[q][3] = fma2(a2, b1.y, acc[q][3]);
        }
      }
    }
  }
#pragma unroll
  for (int hf = 0; hf < 2; ++hf) {
    const int j = hf * (BN / 2) + 4 * tx;
    float4 bias;
    if (!GRAD) bias = make_float4(e.bias[j], e.bias[j + 1], e.bias[j + 2], e.bias[j + 3]);
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int64_t i = i0 + ty + TY * q;
      if (i >= M) continue;
      float4 v;
      upk2(acc[q][2 * hf], v.x, v.y);
      upk2(acc[q][2 * hf + 1], v.z, v.w);
      if (!GRAD) {
        v.x += bias.x;
        v.y += bias.y;
        v.z += bias.z;
        v.w += bias.w;
      }
      if (e.res) {
        const float4 r = *reinterpret_cast<const float4 *>(e.res + i * e.ld_res + j);
        v.x += r.x;
        v.y += r.y;
        v.z += r.z;
        v.w += r.w;
      }
      if (!GRAD) {
        v.x = fmaxf(v.x, kPnSlope * v.x);
        v.y = fmaxf(v.y, kPnSlope * v.y);
        v.z = fmaxf(v.z, kPnSlope * v.z);
        v.w = fmaxf(v.w, kPnSlope * v.w);
      } else {
        const float4 h = *reinterpret_cast<const float4 *>(e.h + i * e.ld_h + j);
        v.x *= h.x > 0.0f ? 1.0f : kPnSlope;
        v.y *= h.y > 0.0f ? 1.0f : kPnSlope;
        v.z *= h.z > 0.0f ? 1.0f : kPnSlope;
        v.w *= h.w > 0.0f ? 1.0f : kPnSlope;
      }
      *reinterpret_cast<float4 *>(e.out + i * e.ld_out + j) = v;
    }
  }
  if (GRAD) grid_dependency_wait();
}

// Weight-gradient partial of one chunk of kChunkRows rows: part[i][j] = sum_r
// dZ[r][i] X[r][j] for i < W and j < K, part[i][K] = sum_r dZ[r][i] (row length
// K + 1).  dZ has W columns, X ldx (a multiple of four); a CTA has BM rows
// (blockIdx.y) and X's first BN columns, with EXTRA also the eight after them.
// Thread (ty, tx) has rows 4 ty (and BM/2 + 4 ty when RM = 8), columns 4 tx and
// BN/2 + 4 tx (and what follows), one packed FP32x2 fma per two columns; every
// output is a chain over the chunk's rows in order.
constexpr int kChunkRows = 256;

template <int W, int BM, int BN, int RM, bool EXTRA>
__global__ void __launch_bounds__(BM *BN / (8 * RM)) pn_wgrad_kernel(const float *__restrict__ dZ,
                                                                     const float *__restrict__ X, int ldx, int K,
                                                                     int64_t rows, float *__restrict__ part) {
  constexpr int T = BM * BN / (8 * RM), TX = BN / 8, LD = BM + BN + (EXTRA ? 8 : 0);
  constexpr int PA = BM / 4, PB = BN / 4;             // 16-byte pieces per row
  constexpr int RA = T / PA, RB = T / PB;             // rows copied per pass
  static_assert(kRowDepth % RA == 0 && kRowDepth % RB == 0 && T % PA == 0 && T % PB == 0, "copy layout");
  extern __shared__ __align__(16) float wsm[];        // [kStages][kRowDepth][LD]
  const int tid = threadIdx.x, tx = tid % TX, ty = tid / TX;
  const int i0 = blockIdx.y * BM;
  const int64_t r_begin = (int64_t)blockIdx.x * kChunkRows;
  const int n = (int)(rows - r_begin < kChunkRows ? rows - r_begin : kChunkRows);
  grid_dependents_launch();   // the kernel before is waited for at the end (see launch_paper_train)
  const int steps = (n + kRowDepth - 1) / kRowDepth;
  const int ra = tid / PA, ca = 4 * (tid % PA), rb = tid / PB, cb = 4 * (tid % PB);
  const float *ga = dZ + (r_begin + ra) * W + i0 + ca, *gb = X + (r_begin + rb) * ldx + cb;
  const bool cb_in = cb < ldx;
  auto load = [&](int step) {
    float *st = wsm + (step % kStages) * (kRowDepth * LD);
    const int left = n - step * kRowDepth;
#pragma unroll
    for (int q = 0; q < kRowDepth / RA; ++q) {
      const bool in = ra + RA * q < left;
      pn_copy16(st + (ra + RA * q) * LD + ca, in ? ga + q * RA * W : dZ, in);
    }
#pragma unroll
    for (int q = 0; q < kRowDepth / RB; ++q) {
      const bool in = rb + RB * q < left && cb_in;
      pn_copy16(st + (rb + RB * q) * LD + BM + cb, in ? gb + (int64_t)q * RB * ldx : X, in);
    }
    if (EXTRA && tid < 2 * kRowDepth) {
      const int r = tid / 2, c = BN + 4 * (tid % 2);
      const bool in = r < left && c < ldx;
      pn_copy16(st + r * LD + BM + c, in ? X + (r_begin + step * kRowDepth + r) * ldx + c : X, in);
    }
    ga += kRowDepth * W;
    gb += (int64_t)kRowDepth * ldx;
  };
  uint64_t acc[RM][4];
#pragma unroll
  for (int q = 0; q < RM; ++q)
#pragma unroll
    for (int t = 0; t < 4; ++t) acc[q][t] = 0ull;
  // the extra columns and the bias: each of a ty's threads takes one of them
  // for all, or an equal share, of the ty's rows
  constexpr int SH = TX / 8;                          // threads that share an extra column's rows
  constexpr int NE = RM / SH;
  static_assert(NE >= 1 && TX % 8 == 0, "extra columns");
  float ext[NE];
#pragma unroll
  for (int q = 0; q < NE; ++q) ext[q] = 0.0f;
  const int e0 = NE * (tx / 8);                       // first of this thread's rows of the extra column
  auto row_of = [&](int q) { return 4 * ty + (q & 3) + (q >> 2) * (BM / 2); };
  float rsum = 0.0f;
  const int bias_row = row_of(tx % RM);
  load(0);
  pn_copy_commit();
  if (steps > 1) load(1);
  pn_copy_commit();
  for (int step = 0; step < steps; ++step) {
    pn_copy_wait<1>();
    __syncthreads();
    if (step + 2 < steps) load(step + 2);
    pn_copy_commit();
    const float *st = wsm + (step % kStages) * (kRowDepth * LD);
#pragma unroll 4
    for (int r = 0; r < kRowDepth; ++r) {
      const float *row = st + r * LD;
      float av[RM];
      {
        const float4 t = *reinterpret_cast<const float4 *>(row + 4 * ty);
        av[0] = t.x;
        av[1] = t.y;
        av[2] = t.z;
        av[3] = t.w;
      }
      if (RM == 8) {
        const float4 t = *reinterpret_cast<const float4 *>(row + BM / 2 + 4 * ty);
        av[4 % RM] = t.x;
        av[5 % RM] = t.y;
        av[6 % RM] = t.z;
        av[7 % RM] = t.w;
      }
      const ulonglong2 b0 = *reinterpret_cast<const ulonglong2 *>(row + BM + 4 * tx);
      const ulonglong2 b1 = *reinterpret_cast<const ulonglong2 *>(row + BM + BN / 2 + 4 * tx);
#pragma unroll
      for (int q = 0; q < RM; ++q) {
        const uint64_t a2 = pk2(av[q], av[q]);
        acc[q][0] = fma2(a2, b0.x, acc[q][0]);
        acc[q][1] = fma2(a2, b0.y, acc[q][1]);
        acc[q][2] = fma2(a2, b1.x, acc[q][2]);
        acc[q][3] = fma2(a2, b1.y, acc[q][3]);
      }
      rsum += row[bias_row];
      if (EXTRA) {
        const float x = row[BM + BN + (tx & 7)];
        if (SH == 1) {
#pragma unroll
          for (int q = 0; q < NE; ++q) ext[q] = fmaf(av[q % RM], x, ext[q]);
        } else {
#pragma unroll
          for (int q = 0; q < NE; ++q) ext[q] = fmaf(row[row_of(e0 + q)], x, ext[q]);
        }
      }
    }
  }
  const int N = K + 1;
  float *out = part + ((int64_t)blockIdx.x * W + i0) * N;
#pragma unroll
  for (int q = 0; q < RM; ++q) {
    const int i = row_of(q);
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      const int j = 4 * tx + 2 * (t & 1) + (t >> 1) * (BN / 2);
      float v0, v1;
      upk2(acc[q][t], v0, v1);
      if (j < K) out[(int64_t)i * N + j] = v0;
      if (j + 1 < K) out[(int64_t)i * N + j + 1] = v1;
    }
  }
  if (tx < RM) out[(int64_t)bias_row * N + K] = rsum;
  if (EXTRA) {
    const int j = BN + (tx & 7);
    if (j < K) {
#pragma unroll
      for (int q = 0; q < NE; ++q) out[(int64_t)row_of(e0 + q) * N + j] = ext[q];
    }
  }
  grid_dependency_wait();
}

// out_w[i][j] = sum_c part[c][i][j] for j < K, out_b[i] = sum_c part[c][i][K]:
// four lanes per element, lane g summing the g-th quarter of the chunks in
// order, the quarters then added as (q0 + q1) + (q2 + q3).
__global__ void pn_reduce_chunks_kernel(const float *__restrict__ part, int chunks, int M, int K,
                                       float *__restrict__ out_w, float *__restrict__ out_b) {
  grid_dependency_wait();
  grid_dependents_launch();
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int e = (int)(t >> 2), g = (int)(t & 3);
  const int N = K + 1;
  const bool in = e < M * N;
  const int64_t mn = (int64_t)M * N;
  const int per = (chunks + 3) / 4;
  const int c1 = min(chunks, (g + 1) * per);
  float s = 0.0f;
  if (in) {
    int c = g * per;
    for (; c + 8 <= c1; c += 8) {
      float v[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) v[q] = part[(c + q) * mn + e];   // eight loads in flight, added in order
#pragma unroll
      for (int q = 0; q < 8; ++q) s += v[q];
    }
    for (; c < c1; ++c) s += part[c * mn + e];
  }
  // every lane forms the same (q0 + q1) + (q2 + q3): addition commutes exactly
  const float o1 = __shfl_xor_sync(0xffffffffu, s, 1);
  const float p = (g & 1) ? o1 + s : s + o1;
  const float o2 = __shfl_xor_sync(0xffffffffu, p, 2);
  const float tot = (g & 2) ? o2 + p : p + o2;
  if (!in || g != 0) return;
  const int i = e / N, j = e % N;
  if (j < K)
    out_w[i * K + j] = tot;
  else
    out_b[i] = tot;
}

// One-blob channel k (FP32, accurate exp) of the footprint: k < 8 the
// periodic Gaussians of frac u (nearest image and the one on the far side),
// 8..15 those of frac v, 16..23 the plain ones of the size coordinate.
__device__ __forceinline__ float pn_blob_channel(float u, float v, float r, int k) {
  const float c = ((k & 7) + 0.5f) * 0.125f;
  if (k >= 16) {
    const float t = (logf(fmaxf(r, kRFloor)) - kPnLnRLo) * kPnInvLnSpan;
    const float d = t - c;
    return expf(-32.0f * d * d);
  }
  const float x = k < 8 ? u : v;
  float d = (x - floorf(x)) - c;
  d -= rintf(d);
  const float e = 1.0f - fabsf(d);
  return expf(-32.0f * d * d) + expf(-32.0f * e * e);
}

// X0[b] = [z_mat (64) | spatial channels (24 one-blob, or 3 unencoded)]
// (row stride ld0) and the angular inputs (wi, wo.xy) at columns
// ang0..ang0+4 of the row of A (row stride lda): XA after the fused
// spatial feature, or X0 itself without the fusion.  One warp per row, so
// that every store of a row is coalesced: lanes copy the latent in two
// 32-float halves, lane k < 24 computes spatial channel k, lanes < 5 the
// angular inputs; the columns up to the next multiple of four are zero.
__global__ void __launch_bounds__(256) pn_inputs_kernel(fabric_gbuffer g, const float *__restrict__ z, int n_lat,
                                                        int ablation, float *__restrict__ X0, int ld0,
                                                        float *__restrict__ A, int lda, int ang0, int *status) {
  grid_dependency_wait();
  grid_dependents_launch();
  const int64_t b = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (b >= g.n) return;
  const int m = g.material[b];
  float *x = X0 + b * ld0;
  float *xa = A + b * lda;
  const int ks = paper_spatial_channels(ablation);
  if (A != X0 && kPnLatent + ks + lane < ld0) x[kPnLatent + ks + lane] = 0.0f;
  if (ang0 + kPnAng + lane < lda) xa[ang0 + kPnAng + lane] = 0.0f;
  if (m >= n_lat) {
    if (lane == 0) atomicOr(status, kStatusBadMaterial);
    x[lane] = 0.0f;
    x[32 + lane] = 0.0f;
    if (lane < ld0 - kPnLatent) x[kPnLatent + lane] = 0.0f;
    if (lane < lda - ang0) xa[ang0 + lane] = 0.0f;
    return;
  }
  x[lane] = z[(int64_t)m * kPnLatent + lane];
  x[32 + lane] = z[(int64_t)m * kPnLatent + 32 + lane];
  const float u = g.u[b], v = g.v[b], r = g.radius[b];
  if (ablation == kPnNoOneBlob) {
    if (lane < 3)
      x[kPnLatent + lane] = lane == 0   ? u - floorf(u)
                            : lane == 1 ? v - floorf(v)
                                        : (logf(fmaxf(r, kRFloor)) - kPnLnRLo) * kPnInvLnSpan;
  } else if (lane < kPnBlob) {
    x[kPnLatent + lane] = pn_blob_channel(u, v, r, lane);
  }
  if (lane < kPnAng) xa[ang0 + lane] = lane < 3 ? g.wi[3 * b + lane] : g.wo[3 * b + lane - 3];
}

// What the head kernel writes: training (target set) the loss partial and
// the head's weight-gradient partial of each CTA and the gradient of k4's
// pre-activation, else the components (C = max(0, y), S = max(0, expm1(y) /
// 100), the inverse of Eq. 9) and RGB by Eq. 8.
struct HeadArgs {
  const float *K4;        // [n][W] last activations
  const float *A5, *a5;   // [4][W], [4]
  int64_t n;
  const float *target, *wi;
  int mode;
  float inv_batch;
  float *dq4;             // [n][W]
  float *part;            // [grid][4][W + 1]
  double *loss_part;      // [grid]
  const uint16_t *mat;
  const DevMaterial *mats;
  int n_mat;
  float *rgb, *comps;
};

constexpr int kHeadRows = 64;
template <int W>
constexpr size_t head_smem() {
  return (size_t)(2 * kHeadRows * (W + 4) + 4 * W + 4 + 4 * kHeadRows) * 4;
}

// A CTA of 256 threads takes a chunk of kChunkRows rows of k4 in tiles of 64,
// the next tile on its way while one is worked on: thread (k, r) forms output
// k of row r (a chain over the inputs in order, then the bias), then its loss
// gradient; the threads then go over the tile again along its columns.  The
// head's weight gradients are chains over the chunk's rows in order.  Bound by
// reading k4 and writing its gradient.
// (As four products with four columns or rows, a loss kernel and its sums
// this took 137 us for 65 536 rows of width 128.)
template <int W, bool TRAIN>
__global__ void __launch_bounds__(256) pn_head_kernel(const HeadArgs a) {
  extern __shared__ __align__(16) float hsm[];
  constexpr int LD = W + 4;
  float *A5 = hsm + 2 * kHeadRows * LD, *b5 = A5 + 4 * W, *DY = b5 + 4;
  __shared__ double red[8];
  grid_dependency_wait();
  grid_dependents_launch();
  const int t = threadIdx.x, r = t & 63, k = t >> 6;
  for (int e = t; e < 4 * W; e += 256) A5[e] = a.A5[e];
  if (t < 4) b5[t] = a.a5[t];
  constexpr int G = 256 / W;                     // weight-gradient rows: thread (g, c) takes outputs g, g + G, ...
  const int c = t % W, g = t / W;
  float gw[4 / G], gb = 0.0f;
#pragma unroll
  for (int q = 0; q < 4 / G; ++q) gw[q] = 0.0f;
  double loss = 0.0;
  const int64_t first = (int64_t)blockIdx.x * kChunkRows;
  const int n = (int)(a.n - first < kChunkRows ? a.n - first : kChunkRows);
  auto load = [&](int tile) {
    float *dst = hsm + (tile & 1) * kHeadRows * LD;
    const int left = n - tile * kHeadRows;
    const float *src = a.K4 + (first + tile * kHeadRows) * W;
#pragma unroll 4
    for (int e = t; e < kHeadRows * (W / 4); e += 256) {
      const int rr = e / (W / 4), cc = 4 * (e % (W / 4));
      pn_copy16(dst + rr * LD + cc, rr < left ? src + rr * W + cc : a.K4, rr < left);
    }
  };
  load(0);
  pn_copy_commit();
  for (int tile = 0; tile * kHeadRows < n; ++tile) {
    const float *X = hsm + (tile & 1) * kHeadRows * LD;
    const int64_t b0 = first + tile * kHeadRows, b = b0 + r;
    const int rows = n - tile * kHeadRows < kHeadRows ? n - tile * kHeadRows : kHeadRows;
    if ((tile + 1) * kHeadRows < n) load(tile + 1);
    pn_copy_commit();
    pn_copy_wait<1>();
    __syncthreads();
    float y = 0.0f;
#pragma unroll 8
    for (int i = 0; i < W; i += 4) {
      const float4 x = *reinterpret_cast<const float4 *>(X + r * LD + i), w = *reinterpret_cast<const float4 *>(A5 + k * W + i);
      y = fmaf(x.x, w.x, y);
      y = fmaf(x.y, w.y, y);
      y = fmaf(x.z, w.z, y);
      y = fmaf(x.w, w.w, y);
    }
    y += b5[k];
    if (TRAIN) {
      float d = 0.0f;
      if (r < rows) {
        const float tg = a.target[4 * b + k], wz = a.wi[3 * b + 2];
        d = k == 0   ? loss_grad(0, y, tg, wz, a.mode, a.inv_batch, &loss)
            : k == 1 ? loss_grad(1, y, tg, wz, a.mode, a.inv_batch, &loss)
            : k == 2 ? loss_grad(2, y, tg, wz, a.mode, a.inv_batch, &loss)
                     : loss_grad(3, y, tg, wz, a.mode, a.inv_batch, &loss);
      }
      DY[k * kHeadRows + r] = d;
    } else {
      DY[k * kHeadRows + r] = y;
    }
    __syncthreads();
    if (TRAIN) {
      // dq4 = (dy A5) lrelu'(k4), four columns of a row per thread
      for (int e = t; e < rows * (W / 4); e += 256) {
        const int rr = e / (W / 4), cc = 4 * (e % (W / 4));
        const float4 x = *reinterpret_cast<const float4 *>(X + rr * LD + cc);
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const float dy = DY[q * kHeadRows + rr];
          const float4 w = *reinterpret_cast<const float4 *>(A5 + q * W + cc);
          v.x = fmaf(dy, w.x, v.x);
          v.y = fmaf(dy, w.y, v.y);
          v.z = fmaf(dy, w.z, v.z);
          v.w = fmaf(dy, w.w, v.w);
        }
        v.x *= x.x > 0.0f ? 1.0f : kPnSlope;
        v.y *= x.y > 0.0f ? 1.0f : kPnSlope;
        v.z *= x.z > 0.0f ? 1.0f : kPnSlope;
        v.w *= x.w > 0.0f ? 1.0f : kPnSlope;
        *reinterpret_cast<float4 *>(a.dq4 + (b0 + rr) * W + cc) = v;
      }
#pragma unroll 8
      for (int rr = 0; rr < kHeadRows; ++rr) {   // rows past the end have dy = 0
        const float x = X[rr * LD + c];
#pragma unroll
        for (int q = 0; q < 4 / G; ++q) gw[q] = fmaf(DY[(g + G * q) * kHeadRows + rr], x, gw[q]);
      }
      if (t < 4)
        for (int rr = 0; rr < kHeadRows; ++rr) gb += DY[t * kHeadRows + rr];
    } else if (t < rows) {
      const int m = a.mat[b0 + t];
      float c4[4];
      if (m >= a.n_mat) {
        c4[0] = c4[1] = c4[2] = c4[3] = __int_as_float(0x7FC00000);
      } else {
        c4[0] = fmaxf(0.0f, DY[t]);
        c4[1] = fmaxf(0.0f, DY[kHeadRows + t]);
        c4[2] = fmaxf(0.0f, expm1f(DY[2 * kHeadRows + t]) / kSpecK);
        c4[3] = fmaxf(0.0f, expm1f(DY[3 * kHeadRows + t]) / kSpecK);
      }
      if (a.comps) store_row4(a.comps, b0 + t, c4[0], c4[1], c4[2], c4[3]);
      if (a.rgb) {
        const DevMaterial &M = a.mats[m < a.n_mat ? m : 0];
        for (int ch = 0; ch < 3; ++ch)
          a.rgb[3 * (b0 + t) + ch] = M.kd[0][ch] * c4[0] + M.kd[1][ch] * c4[1] + M.ks[0][ch] * c4[2] + M.ks[1][ch] * c4[3];
      }
    }
    __syncthreads();
  }
  if (!TRAIN) return;
  float *out = a.part + (int64_t)blockIdx.x * 4 * (W + 1);
#pragma unroll
  for (int q = 0; q < 4 / G; ++q) out[(g + G * q) * (W + 1) + c] = gw[q];
  if (t < 4) out[t * (W + 1) + W] = gb;
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) loss += __shfl_down_sync(0xffffffffu, loss, off);
  if ((t & 31) == 0) red[t >> 5] = loss;
  __syncthreads();
  if (t == 0) {
    double s = red[0];
    for (int q = 1; q < 8; ++q) s += red[q];
    a.loss_part[blockIdx.x] = s;
  }
}

// One warp: lane l sums the partials l, l + 32, ... in order, then a fixed
// shuffle tree adds the lanes.
__global__ void pn_loss_final_kernel(const double *__restrict__ part, int n, double *__restrict__ loss) {
  grid_dependency_wait();
  grid_dependents_launch();
  const int lane = threadIdx.x & 31;
  double s = 0.0;
  for (int k = lane; k < n; k += 32) s += part[k];
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) s += __shfl_down_sync(0xffffffffu, s, off);
  if (lane == 0) *loss = s;
}

// ---------------------------------------------------------------- encoder
constexpr int kEH = 128;
constexpr int kEI = kPatternSlots + 6;   // 22 material features
constexpr int oE1 = 0, oe1 = oE1 + kEH * kEI, oE2 = oe1 + kEH, oe2 = oE2 + kEH * kEH, oE3 = oe2 + kEH,
              oe3 = oE3 + kPnLatent * kEH;
static_assert(oe3 + kPnLatent == kPnEncParams, "encoder layout");

__device__ __forceinline__ float elrelu(float x) { return x > 0.0f ? x : kPnSlope * x; }

// Four materials per CTA of 128 threads: features, h1, h2 (post-activation)
// and z; h1, h2 and the features are kept for the backward pass.  Thread j
// loads row j of a layer's weights into registers once (all loads in flight
// together) and applies it to the four materials; every output is a chain
// of fmaf over its inputs in order, from the bias.
constexpr int kEncG = 4;

__global__ void __launch_bounds__(kEH) pn_enc_fwd_kernel(const fabric_material *__restrict__ raw, int n_mat,
                                                         const float *__restrict__ enc, float *__restrict__ F,
                                                         float *__restrict__ H1, float *__restrict__ H2,
                                                         float *__restrict__ z) {
  grid_dependency_wait();
  grid_dependents_launch();
  __shared__ float f[kEncG][kEI];
  __shared__ float h1[kEncG][kEH], h2[kEncG][kEH];
  const int m0 = blockIdx.x * kEncG, j = threadIdx.x;
  const int nm = min(kEncG, n_mat - m0);
  for (int e = j; e < kEncG * kEI; e += kEH) {
    const int g = e / kEI, i = e % kEI;
    float v = 0.0f;
    if (g < nm) {
      const fabric_material &M = raw[m0 + g];
      if (i < kPatternSlots) {
        v = M.pattern_id == i ? 1.0f : 0.0f;
      } else {
        const int q = i - kPatternSlots;
        v = q == 0 ? M.twist_deg / 30.0f : q == 1 ? M.incl_deg / 45.0f : q == 2 ? M.alpha[0] : q == 3 ? M.beta[0]
          : q == 4 ? M.alpha[1] : M.beta[1];
      }
      if (F) F[(int64_t)(m0 + g) * kEI + i] = v;
    }
    f[g][i] = v;
  }
  __syncthreads();
  float a[kEncG];
  {
    float c[kEI];
#pragma unroll
    for (int i = 0; i < kEI; ++i) c[i] = enc[oE1 + j * kEI + i];
    const float b = enc[oe1 + j];
#pragma unroll
    for (int g = 0; g < kEncG; ++g) {
      a[g] = b;
#pragma unroll
      for (int i = 0; i < kEI; ++i) a[g] = fmaf(c[i], f[g][i], a[g]);
      h1[g][j] = elrelu(a[g]);
    }
  }
  __syncthreads();
  {
    float c[kEH];
    const float4 *w4 = reinterpret_cast<const float4 *>(enc + oE2 + j * kEH);
#pragma unroll
    for (int i4 = 0; i4 < kEH / 4; ++i4) {
      const float4 t = w4[i4];
      c[4 * i4] = t.x;
      c[4 * i4 + 1] = t.y;
      c[4 * i4 + 2] = t.z;
      c[4 * i4 + 3] = t.w;
    }
    const float b = enc[oe2 + j];
#pragma unroll
    for (int g = 0; g < kEncG; ++g) {
      a[g] = b + h1[g][j];   // skip before the last activation
#pragma unroll
      for (int i = 0; i < kEH; ++i) a[g] = fmaf(c[i], h1[g][i], a[g]);
      h2[g][j] = elrelu(a[g]);
      if (g < nm) {
        if (H1) H1[(int64_t)(m0 + g) * kEH + j] = h1[g][j];
        if (H2) H2[(int64_t)(m0 + g) * kEH + j] = h2[g][j];
      }
    }
  }
  __syncthreads();
  // z: thread j takes output k = j % 64 of materials g = j / 64 and g + 2
  {
    const int k = j % kPnLatent, g0 = j / kPnLatent;
    float c[kEH];
    const float4 *w4 = reinterpret_cast<const float4 *>(enc + oE3 + k * kEH);
#pragma unroll
    for (int i4 = 0; i4 < kEH / 4; ++i4) {
      const float4 t = w4[i4];
      c[4 * i4] = t.x;
      c[4 * i4 + 1] = t.y;
      c[4 * i4 + 2] = t.z;
      c[4 * i4 + 3] = t.w;
    }
    const float b = enc[oe3 + k];
#pragma unroll
    for (int gg = 0; gg < kEncG / 2; ++gg) {
      const int g = g0 + 2 * gg;
      float acc = b;
#pragma unroll
      for (int i = 0; i < kEH; ++i) acc = fmaf(c[i], h2[g][i], acc);
      if (g < nm) z[(int64_t)(m0 + g) * kPnLatent + k] = acc;
    }
  }
}

// Per material: the latent's gradient dz[m][k] = sum_j G[m][j] S1[j][k] (G the
// material's sums of the first layer's gradient, W of them), then da2, da1
// (pre-activation gradients).
__global__ void __launch_bounds__(kEH) pn_enc_bwd_kernel(const float *__restrict__ G, int W, const float *__restrict__ S1,
                                                         int ld1, const float *__restrict__ enc,
                                                         const float *__restrict__ H1, const float *__restrict__ H2,
                                                         float *__restrict__ dz, float *__restrict__ DA1,
                                                         float *__restrict__ DA2) {
  __shared__ float sg[128], sdz[kPnLatent], da2[kEH];
  const int m = blockIdx.x, j = threadIdx.x;
  grid_dependents_launch();   // the kernel before is waited for at the end (see launch_paper_train)
  if (j < W) sg[j] = G[(int64_t)m * W + j];
  __syncthreads();
  if (j < kPnLatent) {
    float v = 0.0f;
#pragma unroll 64
    for (int i = 0; i < W; ++i) v = fmaf(sg[i], S1[i * ld1 + j], v);
    sdz[j] = v;
    dz[m * kPnLatent + j] = v;
  }
  __syncthreads();
  float g = 0.0f;
#pragma unroll 64
  for (int k = 0; k < kPnLatent; ++k) g = fmaf(enc[oE3 + k * kEH + j], sdz[k], g);
  const float d2 = g * (H2[m * kEH + j] > 0.0f ? 1.0f : kPnSlope);
  da2[j] = d2;
  DA2[m * kEH + j] = d2;
  __syncthreads();
  g = d2;   // through the skip
#pragma unroll 64
  for (int o = 0; o < kEH; ++o) g = fmaf(enc[oE2 + o * kEH + j], da2[o], g);
  DA1[m * kEH + j] = g * (H1[m * kEH + j] > 0.0f ? 1.0f : kPnSlope);
  grid_dependency_wait();
}

// Encoder parameter gradients as sums over materials of outer products,
// G[o][i] = sum_m L[m][o] R[m][i] (R = 1 for a bias): E1 (da1, features),
// e1, E2 (da2, h1), e2, E3 (dz, h2), e3.  A CTA of 64 threads takes a 16 x 16
// tile of one block, stages 128 materials' slices of L and R in shared memory
// at a time (all copies in flight together), and thread (ty, tx) keeps outputs
// 2 ty, 2 ty + 1 of columns 2 tx, 2 tx + 1, each a chain of fmaf over the
// materials in order.  (32 x 32 tiles with four outputs per thread ran on 38
// SMs, bound by their shared-memory loads: 11.7 us for 256 materials, 9.3
// so.)
constexpr int kEncGradChunk = 128, kEncGradTile = 16, kEncGradThreads = 64;

__host__ __device__ constexpr int pn_tiles(int rows, int cols) {
  return rows / kEncGradTile * ((cols + kEncGradTile - 1) / kEncGradTile);
}
constexpr int kPnEncGradTiles = pn_tiles(kEH, kEI) + pn_tiles(kEH, 1) + pn_tiles(kEH, kEH) + pn_tiles(kEH, 1) +
                                pn_tiles(kPnLatent, kEH) + pn_tiles(kPnLatent, 1);
static_assert(kEH % kEncGradTile == 0 && kPnLatent % kEncGradTile == 0, "whole tiles of rows");

__global__ void __launch_bounds__(kEncGradThreads) pn_enc_grad_kernel(int n_mat, const float *__restrict__ F,
                                                          const float *__restrict__ H1, const float *__restrict__ H2,
                                                          const float *__restrict__ dz,
                                                          const float *__restrict__ DA1,
                                                          const float *__restrict__ DA2, float *__restrict__ genc) {
  grid_dependency_wait();
  grid_dependents_launch();
  __shared__ __align__(16) float sl[kEncGradChunk][kEncGradTile], sr[kEncGradChunk][kEncGradTile];
  // which block, and which tile of it
  const float *L = DA1, *R = F;
  int ldl = kEH, ldr = kEI, cols = kEI, out = oE1;
  int t = blockIdx.x;
  constexpr int t0 = pn_tiles(kEH, kEI), t1 = t0 + pn_tiles(kEH, 1), t2 = t1 + pn_tiles(kEH, kEH),
                t3 = t2 + pn_tiles(kEH, 1), t4 = t3 + pn_tiles(kPnLatent, kEH);
  if (t >= t4) {
    L = dz; ldl = kPnLatent; R = nullptr; cols = 1; out = oe3; t -= t4;
  } else if (t >= t3) {
    L = dz; ldl = kPnLatent; R = H2; ldr = kEH; cols = kEH; out = oE3; t -= t3;
  } else if (t >= t2) {
    L = DA2; R = nullptr; cols = 1; out = oe2; t -= t2;
  } else if (t >= t1) {
    L = DA2; R = H1; ldr = kEH; cols = kEH; out = oE2; t -= t1;
  } else if (t >= t0) {
    R = nullptr; cols = 1; out = oe1; t -= t0;
  }
  const int ct = (cols + kEncGradTile - 1) / kEncGradTile;
  const int r0 = (t / ct) * kEncGradTile, c0 = (t % ct) * kEncGradTile;
  const int tid = threadIdx.x, ty = tid >> 3, tx = tid & 7;
  float acc[2][2] = {{0.0f, 0.0f}, {0.0f, 0.0f}};
  for (int m0 = 0; m0 < n_mat; m0 += kEncGradChunk) {
    const int mc = min(kEncGradChunk, n_mat - m0);
    __syncthreads();
    for (int e = tid; e < 4 * mc; e += kEncGradThreads)
      pn_copy16(&sl[e >> 2][4 * (e & 3)], L + (int64_t)(m0 + (e >> 2)) * ldl + r0 + 4 * (e & 3), true);
    if (R && cols == kEH) {
      for (int e = tid; e < 4 * mc; e += kEncGradThreads)
        pn_copy16(&sr[e >> 2][4 * (e & 3)], R + (int64_t)(m0 + (e >> 2)) * ldr + c0 + 4 * (e & 3), true);
    } else {   // features (rows of 22), or ones
#pragma unroll 8
      for (int e = tid; e < kEncGradTile * mc; e += kEncGradThreads) {
        const int k = c0 + (e & 15);
        sr[e >> 4][e & 15] = !R ? 1.0f : k < cols ? R[(int64_t)(m0 + (e >> 4)) * ldr + k] : 0.0f;
      }
    }
    pn_copy_commit();
    pn_copy_wait<0>();
    __syncthreads();
#pragma unroll 8
    for (int mm = 0; mm < mc; ++mm) {
      const float2 a = reinterpret_cast<const float2 *>(sl[mm])[ty];
      const float2 x = reinterpret_cast<const float2 *>(sr[mm])[tx];
      acc[0][0] = fmaf(a.x, x.x, acc[0][0]);
      acc[0][1] = fmaf(a.x, x.y, acc[0][1]);
      acc[1][0] = fmaf(a.y, x.x, acc[1][0]);
      acc[1][1] = fmaf(a.y, x.y, acc[1][1]);
    }
  }
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const int c = c0 + 2 * tx + k;
      if (c < cols) genc[out + (r0 + 2 * ty + i) * cols + c] = acc[i][k];
    }
}

// The weights as the layer kernel reads them, packed once per pass: for the
// forward layers the transposes [inputs][W] (inputs padded to a multiple of
// four with zeros), for A1's input gradient its rows at a multiple of four.
struct PnWeights {
  float *TS1, *TS2, *TA1, *TA2, *TA3, *TA4, *A1;
};

constexpr int pad4(int k) { return (k + 3) & ~3; }

__global__ void __launch_bounds__(256) pn_weights_kernel(const float *__restrict__ dec, PaperOffsets o, int w, int k1, int ka1,
                                                         int train, PnWeights P) {
  grid_dependency_wait();
  grid_dependents_launch();
  int e = blockIdx.x * 256 + threadIdx.x;
  const int nt = w * w, n1 = pad4(k1) * w, na = pad4(ka1) * w;
  // T[k][j] = W[j][k]
  auto transpose = [&](float *T, int src, int k_in) {
    const int k = e / w, j = e % w;
    T[e] = k < k_in ? dec[src + j * k_in + k] : 0.0f;
  };
  if (e < n1) return transpose(P.TS1, o.S1, k1);
  e -= n1;
  if (e < na) return transpose(P.TA1, o.A1, ka1);
  e -= na;
  if (e < 4 * nt) {
    const int l = e / nt;
    e %= nt;
    return transpose(l == 0 ? P.TS2 : l == 1 ? P.TA2 : l == 2 ? P.TA3 : P.TA4, l == 0 ? o.S2 : l == 1 ? o.A2 : l == 2 ? o.A3 : o.A4, w);
  }
  e -= 4 * nt;
  if (train && e < na) {
    const int j = e / pad4(ka1), k = e % pad4(ka1);
    P.A1[e] = k < ka1 ? dec[o.A1 + j * ka1 + k] : 0.0f;
  }
}

int chunk_count(int64_t B) { return (int)((B + kChunkRows - 1) / kChunkRows); }

template <int BM, int BN, bool GRAD>
cudaError_t layer_of(const float *A, int lda, const float *B, int ldb, int64_t M, int K, const Epi &e, cudaStream_t s) {
  constexpr size_t smem = (size_t)kStages * (BM * (kDepth + 4) + kDepth * BN) * sizeof(float);
  const auto k = pn_layer_kernel<BM, BN, GRAD>;
  const cudaError_t err = ensure_max_dyn_smem(reinterpret_cast<const void *>(k), (int)smem);
  if (err != cudaSuccess) return err;
  return launch_dependent(k, dim3((unsigned)((M + BM - 1) / BM)), BM * BN / 64, smem, s, A, lda, B, ldb, M, K, e);
}
template <bool GRAD>
cudaError_t layer(const float *A, int lda, const float *B, int ldb, int64_t M, int K, int w, const Epi &e, cudaStream_t s) {
  return w == 128 ? layer_of<64, 128, GRAD>(A, lda, B, ldb, M, K, e, s) : layer_of<128, 64, GRAD>(A, lda, B, ldb, M, K, e, s);
}

// forward layer: out[b][j] = lrelu(sum_k X[b][k] T[k][j] + bias[j] (+ res[b][j])), T [K][w]
cudaError_t fwd(const float *X, int ldx, const float *T, const float *bias, int w, int64_t B, float *out, int ldo,
                const float *res, int ldr, cudaStream_t s) {
  return layer<false>(X, ldx, T, w, B, ldx, w, Epi{bias, res, ldr, nullptr, 0, out, ldo}, s);
}

// input gradient: dX[b][k] = (sum_j dZ[b][j] W[j][k] (+ add[b][k])) lrelu'(h[b][k]), k < w
cudaError_t bwd_in(const float *dZ, const float *W, int ldw, int w, int64_t B, float *out, const float *add, const float *h,
                   int ldh, cudaStream_t s) {
  return layer<true>(dZ, w, W, ldw, B, w, w, Epi{nullptr, add, w, h, ldh, out, w}, s);
}

template <int W, int BM, int BN, int RM, bool EXTRA>
cudaError_t wgrad_partials(const float *dZ, const float *X, int ldx, int K, int64_t B, float *part, cudaStream_t s) {
  constexpr size_t smem = (size_t)kStages * kRowDepth * (BM + BN + (EXTRA ? 8 : 0)) * sizeof(float);
  const auto k = pn_wgrad_kernel<W, BM, BN, RM, EXTRA>;
  const cudaError_t e = ensure_max_dyn_smem(reinterpret_cast<const void *>(k), (int)smem);
  if (e != cudaSuccess) return e;
  return launch_dependent(k, dim3((unsigned)chunk_count(B), W / BM), BM * BN / (8 * RM), smem, s, dZ, X, ldx, K, B, part);
}

cudaError_t reduce_chunks(const float *part, int chunks, int N, int K, float *dW, float *db, cudaStream_t s) {
  const int64_t tot = (int64_t)N * (K + 1);
  return launch_dependent(pn_reduce_chunks_kernel, dim3((unsigned)((4 * tot + 255) / 256)), 256, 0, s, part, chunks, N, K, dW, db);
}

// Chunk sums (see reduce_chunks) of the weight and bias gradients dW[j][k] = sum_b
// dZ[b][j] X[b][k] for k < K, db[j] = sum_b dZ[b][j]; X [B][ldx].
cudaError_t wgrad(const float *dZ, int w, const float *X, int ldx, int K, int64_t B, float *part, cudaStream_t s) {
  cudaError_t e;
  if (w == 128)
    e = K > 128 ? wgrad_partials<128, 64, 128, 8, true>(dZ, X, ldx, K, B, part, s)
                : wgrad_partials<128, 64, 128, 8, false>(dZ, X, ldx, K, B, part, s);
  else
    e = K > 72   ? wgrad_partials<64, 64, 128, 8, false>(dZ, X, ldx, K, B, part, s)
        : K > 64 ? wgrad_partials<64, 64, 64, 4, true>(dZ, X, ldx, K, B, part, s)
                 : wgrad_partials<64, 64, 64, 4, false>(dZ, X, ldx, K, B, part, s);
  return e;
}

template <bool TRAIN>
cudaError_t head(int w, const HeadArgs &a, cudaStream_t s) {
  const size_t smem = w == 128 ? head_smem<128>() : head_smem<64>();
  const auto k = w == 128 ? pn_head_kernel<128, TRAIN> : pn_head_kernel<64, TRAIN>;
  const cudaError_t e = ensure_max_dyn_smem(reinterpret_cast<const void *>(k), (int)smem);
  if (e != cudaSuccess) return e;
  return launch_dependent(k, dim3((unsigned)chunk_count(a.n)), 256, smem, s, a);
}

}  // namespace

// Largest training material table the step accepts, at any width.
int paper_train_max_materials(int) { return 1600; }

namespace {

// Activation buffers of one pass over a batch of B queries: the first
// layer's input X0 [B][ld0], the first layer's output H1, A1's input XA
// [B][lda] (the second layer's output, then the angular inputs with the
// spatial fusion), K1..K4; row lengths padded to multiples of four.
struct PnPass {
  int w, ablation, KX0, KA, ld0, lda;
  float *X0, *H1, *XA, *K1, *K2, *K3, *K4;
  PnWeights W;
};

// keep: every activation has its own buffer (training); else the last one
// takes H1's place.
template <class Take>
PnPass pn_pass_buffers(int w, int ablation, int64_t B, bool keep, Take take) {
  PnPass P;
  P.w = w;
  P.ablation = ablation;
  P.KX0 = paper_x0_inputs(ablation);
  P.KA = paper_a1_inputs(w, ablation);
  P.ld0 = pad4(P.KX0);
  P.lda = pad4(P.KA);
  P.X0 = take((size_t)B * P.ld0);
  P.H1 = take((size_t)B * w);
  P.XA = take((size_t)B * P.lda);
  P.K1 = take((size_t)B * w);
  P.K2 = take((size_t)B * w);
  P.K3 = take((size_t)B * w);
  P.K4 = keep ? take((size_t)B * w) : P.H1;
  P.W.TS1 = take((size_t)P.ld0 * w);
  P.W.TS2 = take((size_t)w * w);
  P.W.TA1 = take((size_t)P.lda * w);
  P.W.TA2 = take((size_t)w * w);
  P.W.TA3 = take((size_t)w * w);
  P.W.TA4 = take((size_t)w * w);
  P.W.A1 = keep ? take((size_t)w * P.lda) : nullptr;
  return P;
}

// Inputs and the forward pass of the structure (or its ablation) up to the
// head's input K4.
cudaError_t pn_forward(const PnPass &P, const fabric_gbuffer &q, const float *z, int n_mat, const float *dec,
                       bool train, int *status, cudaStream_t s) {
  const PaperOffsets o = paper_offsets_ablation(P.w, P.ablation);
  const int64_t B = q.n;
  const int w = P.w;
  cudaError_t e;
  const bool fusion = P.ablation != kPnNoFusion;
  const int items = w * (P.ld0 + P.lda + 4 * w + (train ? P.lda : 0));
  if ((e = launch_dependent(pn_weights_kernel, dim3((unsigned)((items + 255) / 256)), 256, 0, s, dec, o, w, P.KX0, P.KA,
                            train ? 1 : 0, P.W)) != cudaSuccess)
    return e;
  if ((e = launch_dependent(pn_inputs_kernel, dim3((unsigned)((B + 7) / 8)), 256, 0, s, q, z, n_mat, P.ablation, P.X0, P.ld0,
                            fusion ? P.XA : P.X0, fusion ? P.lda : P.ld0, fusion ? w : kPnLatent + kPnBlob, status)) != cudaSuccess)
    return e;
  if ((e = fwd(P.X0, P.ld0, P.W.TS1, dec + o.s1, w, B, P.H1, w, nullptr, 0, s)) != cudaSuccess) return e;
  if ((e = fwd(P.H1, w, P.W.TS2, dec + o.s2, w, B, P.XA, P.lda, nullptr, 0, s)) != cudaSuccess) return e;
  if ((e = fwd(P.XA, P.lda, P.W.TA1, dec + o.a1, w, B, P.K1, w, nullptr, 0, s)) != cudaSuccess) return e;
  if ((e = fwd(P.K1, w, P.W.TA2, dec + o.a2, w, B, P.K2, w, nullptr, 0, s)) != cudaSuccess) return e;
  if ((e = fwd(P.K2, w, P.W.TA3, dec + o.a3, w, B, P.K3, w, P.K1, w, s)) != cudaSuccess) return e;   // skip
  return fwd(P.K3, w, P.W.TA4, dec + o.a4, w, B, P.K4, w, nullptr, 0, s);
}

// Floats that `take` hands out for a pass, with its rounding.
struct Count {
  size_t f = 0;
  float *operator()(size_t n) {
    f += (n + 63) & ~size_t(63);
    return nullptr;
  }
};

// Buffers of a training step after the forward pass's.
struct PnTrain {
  float *D1, *D2, *D3, *part[2], *G, *dz, *F, *EH1, *EH2, *DA1, *DA2, *z;
  double *lpart;
};
template <class Take>
PnTrain pn_train_buffers(int w, int ablation, int64_t B, int n_mat, Take take) {
  PnTrain T;
  T.D1 = take((size_t)B * w);
  T.D2 = take((size_t)B * w);
  T.D3 = take((size_t)B * w);
  // weight-gradient partials of the widest layer
  const int k_max = std::max(paper_x0_inputs(ablation), paper_a1_inputs(w, ablation));
  for (float *&part : T.part) part = take((size_t)chunk_count(B) * w * (k_max + 1));
  T.G = take((size_t)n_mat * w);
  T.dz = take((size_t)n_mat * kPnLatent);
  T.F = take((size_t)n_mat * kEI);
  T.EH1 = take((size_t)n_mat * kEH);
  T.EH2 = take((size_t)n_mat * kEH);
  T.DA1 = take((size_t)n_mat * kEH);
  T.DA2 = take((size_t)n_mat * kEH);
  T.z = take((size_t)n_mat * kPnLatent);
  T.lpart = reinterpret_cast<double *>(take((size_t)chunk_count(B) * 2));
  return T;
}

}  // namespace

size_t paper_train_work_bytes(int w, int64_t B, int n_mat) {
  size_t most = 0;   // over the structures, whose buffers differ a little
  for (int ablation : {kPnFull, kPnNoOneBlob, kPnNoFusion}) {
    Count c;
    pn_pass_buffers(w, ablation, B, true, [&](size_t n) { return c(n); });
    pn_train_buffers(w, ablation, B, n_mat, [&](size_t n) { return c(n); });
    most = std::max(most, c.f);
  }
  return most * 4;
}

// One step's forward, loss and backward: grad [decoder | encoder] and the
// batch loss; raw = device copy of the training materials.
cudaError_t launch_paper_train(int w, int ablation, const fabric_gbuffer &q, const float *target, int loss_mode,
                               const fabric_material *raw, int n_mat, const float *dec, const float *enc,
                               float *grad, double *loss, void *work, int *status, cudaStream_t s) {
  const PaperOffsets o = paper_offsets_ablation(w, ablation);
  const int64_t B = q.n;
  float *p = static_cast<float *>(work);
  auto take = [&](size_t nfl) {
    float *r = p;
    p += (nfl + 63) & ~size_t(63);
    return r;
  };
  const PnPass P = pn_pass_buffers(w, ablation, B, true, take);
  const PnTrain T = pn_train_buffers(w, ablation, B, n_mat, take);
  float *D1 = T.D1, *D2 = T.D2, *D3 = T.D3, *const *part = T.part;
  float *gd = grad, *ge = grad + o.total;
  cudaError_t e;
#define PN_TRY(x)                     \
  do {                                \
    e = (x);                          \
    if (e != cudaSuccess) return e;   \
  } while (0)
  // ---- encoder, inputs and forward
  PN_TRY(launch_dependent(pn_enc_fwd_kernel, dim3((n_mat + kEncG - 1) / kEncG), kEH, 0, s, raw, n_mat, enc, T.F, T.EH1, T.EH2, T.z));
  PN_TRY(pn_forward(P, q, T.z, n_mat, dec, true, status, s));
  // ---- head, loss and their gradients
  HeadArgs h{};
  h.K4 = P.K4;
  h.A5 = dec + o.A5;
  h.a5 = dec + o.a5;
  h.n = B;
  h.target = target;
  h.wi = q.wi;
  h.mode = loss_mode;
  h.inv_batch = 1.0f / (float)B;
  h.dq4 = D1;
  h.part = part[0];
  h.loss_part = T.lpart;
  PN_TRY(head<true>(w, h, s));
  PN_TRY(reduce_chunks(part[0], chunk_count(B), 4, w, gd + o.A5, gd + o.a5, s));
  PN_TRY(launch_dependent(pn_loss_final_kernel, dim3(1), 32, 0, s, T.lpart, chunk_count(B), loss));
  // ---- backward (D1..D3 rotate as dq4, dq3, dq2, dq1, dg2, dg1)
  // Three launches per layer: chunk sums of its weight gradients, input
  // gradient, reduction of the sums.  Only the reduction waits for the kernel
  // before it first.  The chunk sums start under the reduction of the layer
  // before (whose own wait the input gradient they read had to pass; their
  // buffers alternate), the input gradient under the chunk sums, filling the SMs
  // as the last of those run, and each waits at its end for the kernel it
  // started under, so that its completion still implies that one's: one after
  // the other, 65 536 queries at width 128 took 1063 us a step, so 1000.
  const int chunks = chunk_count(B);
  PN_TRY(wgrad(D1, w, P.K3, w, w, B, part[1], s));
  PN_TRY(bwd_in(D1, dec + o.A4, w, w, B, D2, nullptr, P.K3, w, s));          // dq3
  PN_TRY(reduce_chunks(part[1], chunks, w, w, gd + o.A4, gd + o.a4, s));
  PN_TRY(wgrad(D2, w, P.K2, w, w, B, part[0], s));
  PN_TRY(bwd_in(D2, dec + o.A3, w, w, B, D3, nullptr, P.K2, w, s));          // dq2
  PN_TRY(reduce_chunks(part[0], chunks, w, w, gd + o.A3, gd + o.a3, s));
  PN_TRY(wgrad(D3, w, P.K1, w, w, B, part[1], s));
  PN_TRY(bwd_in(D3, dec + o.A2, w, w, B, D1, D2, P.K1, w, s));               // dq1 (+ dq3 through the skip)
  PN_TRY(reduce_chunks(part[1], chunks, w, w, gd + o.A2, gd + o.a2, s));
  PN_TRY(wgrad(D1, w, P.XA, P.lda, P.KA, B, part[0], s));
  PN_TRY(bwd_in(D1, P.W.A1, P.lda, w, B, D2, nullptr, P.XA, P.lda, s));      // dg2
  PN_TRY(reduce_chunks(part[0], chunks, w, P.KA, gd + o.A1, gd + o.a1, s));
  PN_TRY(wgrad(D2, w, P.H1, w, w, B, part[1], s));
  PN_TRY(bwd_in(D2, dec + o.S2, w, w, B, D3, nullptr, P.H1, w, s));          // dg1
  PN_TRY(reduce_chunks(part[1], chunks, w, w, gd + o.S2, gd + o.s2, s));
  // ---- latent gradient: per-material sums of dg1, times S1's latent block; encoder backward
  PN_TRY(wgrad(D3, w, P.X0, P.ld0, P.KX0, B, part[0], s));
  PN_TRY(launch_material_row_sums(q.material, B, n_mat, D3, w, T.G, s));
  PN_TRY(reduce_chunks(part[0], chunks, w, P.KX0, gd + o.S1, gd + o.s1, s));
  PN_TRY(launch_dependent(pn_enc_bwd_kernel, dim3(n_mat), kEH, 0, s, T.G, w, dec + o.S1, P.KX0, enc, T.EH1, T.EH2, T.dz, T.DA1, T.DA2));
  PN_TRY(launch_dependent(pn_enc_grad_kernel, dim3(kPnEncGradTiles), kEncGradThreads, 0, s, n_mat, T.F, T.EH1, T.EH2, T.dz, T.DA1, T.DA2, ge));
#undef PN_TRY
  return cudaSuccess;
}

size_t paper_forward_work_bytes(int w, int64_t B) {
  size_t most = 0;
  for (int ablation : {kPnFull, kPnNoOneBlob, kPnNoFusion}) {
    Count c;
    pn_pass_buffers(w, ablation, B, false, [&](size_t n) { return c(n); });
    most = std::max(most, c.f);
  }
  return most * 4;
}

// FP32 forward of the structure (or an ablation) over a G-buffer, with
// per-material latents z [n_mat][64]: components and RGB.
cudaError_t launch_paper_forward(int w, int ablation, const fabric_gbuffer &g, const float *z,
                                 const DevMaterial *mats, int n_mat, const float *dec, float *rgb, float *comps,
                                 void *work, int *status, cudaStream_t s) {
  float *p = static_cast<float *>(work);
  auto take = [&](size_t nfl) {
    float *r = p;
    p += (nfl + 63) & ~size_t(63);
    return r;
  };
  const PaperOffsets o = paper_offsets_ablation(w, ablation);
  const PnPass P = pn_pass_buffers(w, ablation, g.n, false, take);
  cudaError_t e = pn_forward(P, g, z, n_mat, dec, false, status, s);
  if (e != cudaSuccess) return e;
  HeadArgs h{};
  h.K4 = P.K4;
  h.A5 = dec + o.A5;
  h.a5 = dec + o.a5;
  h.n = g.n;
  h.mat = g.material;
  h.mats = mats;
  h.n_mat = n_mat;
  h.rgb = rgb;
  h.comps = comps;
  return head<false>(w, h, s);
}

cudaError_t launch_paper_encoder(const fabric_material *raw, int n_mat, const float *enc, float *z, cudaStream_t s) {
  return launch_dependent(pn_enc_fwd_kernel, dim3((n_mat + kEncG - 1) / kEncG), kEH, 0, s, raw, n_mat, enc, nullptr, nullptr, nullptr, z);
}

}  // namespace fab
