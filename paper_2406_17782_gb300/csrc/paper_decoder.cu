// paper_decoder.cu -- the paper's own decoder structure (Sec. 4.2, "Decoder";
// Fig. 3) on the 5th-generation tensor cores: the footprint's position and
// size one-blob encoded (3 -> 24 channels), fused with the material latent by
// two fully connected layers (the spatial feature), then, with the angular
// inputs wi (x, y, z) and wo (x, y), an angular decoder of five fully
// connected layers with one skip connection; leaky ReLU throughout; the four
// components of Eq. 7 become RGB by Eq. 8.
//
// Same execution scheme as the workload's decoder (decoder_tc.cu): a
// persistent CTA holds one copy of the packed 16-bit weights in shared memory
// (one bulk copy), and WG tile pipelines of H warpgroups each stream
// 128-point tiles, H threads per point.  Per pipeline, tensor memory holds two
// regions of W columns: a layer's FP32 accumulator D in one, its 16-bit A
// operand (two values per 32-bit column) in the other.  Seven MMA chains per
// tile:
//   L0  S1': [one-blob (24) | one-hot material] -> W     (latent folded: the
//       per-material column holds S1[:, :64] z_m + s1, exact algebra)
//   L1  S2 : h1 -> h                                    (bias in a constant-one column)
//   L2  A1 : [h | wi | wo.xy] -> k1
//   L3  A2 : k1 -> k2
//   L4  A3 : k2 -> k3, with the skip: k3 = lrelu(A3 k2 + a3 + k1), k1 kept
//       in registers as the 16-bit operand values written after L2
//   L5  A4 : k3 -> k4
//   L6  A5 : k4 -> y (N = 16, four used)
// The one-blob bins of the periodic footprint centre are Gaussians wrapped
// around the weave repeat (nearest image plus the one on the far side; the
// others weigh below exp(-32)).
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "f32x2.h"
#include "fabric_internal.h"
#include "paper_net.h"
#include "tc_ptx.h"

namespace fab {
namespace {

constexpr int kTile = 128;
// A layer's operand begins kColBias columns of its region after the packed
// values of the first 32 inputs: its K step W / 16, the bias input (and after
// the spatial fusion the angular ones).  Layer 0's operand begins there too.
constexpr uint32_t kColBias = 16;
constexpr long long kWaitCycles = 4000000000ll;   // ~2 s at 2 GHz
constexpr int kPnMaxK1 = 128;                     // layer-0 K: 24 + materials, padded to 16

// Packed operands of width W (bytes; identical in global and shared memory):
// seven K-major weight blocks, then the per-material albedos.
struct PnBlob {
  int k1, kh;
  uint32_t l[7];
  uint32_t alb, total;
};

__host__ __device__ constexpr PnBlob pn_blob(int w, int n_mat) {
  PnBlob b{};
  b.k1 = (kPnBlob + n_mat + 15) / 16 * 16;
  b.kh = w + 16;
  b.l[0] = 0;
  b.l[1] = b.l[0] + (uint32_t)w * b.k1 * 2u;
  for (int i = 2; i <= 6; ++i) b.l[i] = b.l[i - 1] + (uint32_t)w * b.kh * 2u;
  b.alb = b.l[6] + 16u * b.kh * 2u;
  b.total = b.alb + ((uint32_t)(n_mat * 12 * 4) + 15u) / 16u * 16u;
  return b;
}

__host__ __device__ constexpr int pn_cols(int w) { return w == 64 ? 128 : 256; }   // tensor-memory columns per pipeline

template <bool F16>
__device__ __forceinline__ void put_op(uint8_t *base, uint32_t off, float v) {
  if (F16)
    *reinterpret_cast<__half *>(base + off) = __float2half_rn(v);
  else
    *reinterpret_cast<__nv_bfloat16 *>(base + off) = __float2bfloat16_rn(v);
}

// Fold the latents into layer 0 and pack every layer into the canonical
// K-major layout; layers 1-6 carry their bias in input column W (A1: column
// W + 5, after the angular inputs), the rest of the K padding is zero.  One CTA.
template <int W, bool F16>
__global__ void __launch_bounds__(256) pn_pack_kernel(const float *__restrict__ p, const float *__restrict__ lat,
                                                      const DevMaterial *__restrict__ mats, int n_mat,
                                                      uint8_t *__restrict__ blob) {
  extern __shared__ float fold[];   // [n_mat][W]
  constexpr PaperOffsets o = paper_offsets(W);
  const PnBlob B = pn_blob(W, n_mat);
  for (int e = threadIdx.x; e < n_mat * W; e += blockDim.x) {
    const int m = e / W, r = e % W;
    float acc = p[o.s1 + r];
    for (int j = 0; j < kPnLatent; ++j) acc = fmaf(p[o.S1 + r * (kPnLatent + kPnBlob) + j], lat[m * kPnLatent + j], acc);
    fold[m * W + r] = acc;
  }
  __syncthreads();
  for (int e = threadIdx.x; e < W * B.k1; e += blockDim.x) {
    const int r = e / B.k1, c = e % B.k1;
    float v = 0.0f;
    if (c < kPnBlob)
      v = p[o.S1 + r * (kPnLatent + kPnBlob) + kPnLatent + c];
    else if (c < kPnBlob + n_mat)
      v = fold[(c - kPnBlob) * W + r];
    put_op<F16>(blob, B.l[0] + tc::core_offset(r, c, B.k1), v);
  }
  // layers 1..5: [W][kh]; layer 6: [16][kh]
  const int wofs[6] = {o.S2, o.A1, o.A2, o.A3, o.A4, o.A5};
  const int bofs[6] = {o.s2, o.a1, o.a2, o.a3, o.a4, o.a5};
  for (int l = 1; l <= 6; ++l) {
    const int rows = l == 6 ? 16 : W;
    const int rows_used = l == 6 ? 4 : W;
    const int in = l == 2 ? W + kPnAng : W;   // weight columns
    for (int e = threadIdx.x; e < rows * B.kh; e += blockDim.x) {
      const int r = e / B.kh, c = e % B.kh;
      float v = 0.0f;
      if (r < rows_used) {
        if (c < in)
          v = p[wofs[l - 1] + r * in + c];
        else if (c == in)
          v = p[bofs[l - 1] + r];
      }
      put_op<F16>(blob, B.l[l] + tc::core_offset(r, c, B.kh), v);
    }
  }
  float *alb = reinterpret_cast<float *>(blob + B.alb);
  for (int e = threadIdx.x; e < n_mat * 12; e += blockDim.x) {
    const int m = e / 12, q = e % 12;
    const DevMaterial &M = mats[m];
    alb[e] = q < 3 ? M.kd[0][q] : q < 6 ? M.kd[1][q - 3] : q < 9 ? M.ks[0][q - 6] : M.ks[1][q - 9];
  }
}

struct PnArgs {
  const float *u, *v, *radius, *wi, *wo;
  const uint16_t *material;
  int64_t n, n_tiles;
  const uint8_t *blob;
  int n_mat;
  float *rgb, *comps;
  int *status;
};

struct PnPoint {
  float u, v, r, wi0, wi1, wi2, wo0, wo1;
  int mat;   // -1: beyond the end
};

// What thread h of the point's H threads needs: the first u, the radius and
// the angular inputs, the last v.
template <int H>
__device__ __forceinline__ PnPoint pn_load(const PnArgs &a, int64_t p, int h) {
  PnPoint q;
  q.u = q.v = q.r = q.wi0 = q.wi1 = q.wi2 = q.wo0 = q.wo1 = 0.0f;
  q.mat = -1;
  if (p < a.n) {
    q.mat = __ldg(a.material + p);
    if (H == 1 || h == 0) {
      q.u = __ldg(a.u + p);
      q.r = __ldg(a.radius + p);
      q.wi0 = __ldg(a.wi + 3 * p);
      q.wi1 = __ldg(a.wi + 3 * p + 1);
      q.wi2 = __ldg(a.wi + 3 * p + 2);
      q.wo0 = __ldg(a.wo + 3 * p);
      q.wo1 = __ldg(a.wo + 3 * p + 1);
    }
    if (H == 1 || h == 1) q.v = __ldg(a.v + p);
  }
  return q;
}

__device__ __forceinline__ float ex2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// exp(-d^2 / (2 sigma^2)) with sigma = 1/8, i.e. 2^(-32 log2(e) d^2)
constexpr float kGaussK = -46.16624130844683f;

// Eight periodic one-blob bins of x (wrapped Gaussians around the unit
// interval), packed two per word into w[0..3].
template <bool F16>
__device__ __forceinline__ void blob_periodic(float x, uint32_t *w) {
  const float f = x - floorf(x);
  float b[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    float d = f - (i + 0.5f) * 0.125f;
    d -= rintf(d);                       // nearest image, |d| <= 1/2
    const float e = 1.0f - fabsf(d);     // the image on the far side
    b[i] = ex2_approx(kGaussK * d * d) + ex2_approx(kGaussK * e * e);
  }
#pragma unroll
  for (int k = 0; k < 4; ++k) w[k] = tc::pack2<F16>(b[2 * k], b[2 * k + 1]);
}

template <bool F16>
__device__ __forceinline__ void blob_plain(float t, uint32_t *w) {
  float b[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const float d = t - (i + 0.5f) * 0.125f;
    b[i] = ex2_approx(kGaussK * d * d);
  }
#pragma unroll
  for (int k = 0; k < 4; ++k) w[k] = tc::pack2<F16>(b[2 * k], b[2 * k + 1]);
}

// Named barriers over the N threads of a pipeline: OR-reducing `pred`, and
// split into the waiting side (the issuing warp) and the arriving one.
template <int N>
__device__ __forceinline__ bool pn_bar_or(int id, bool pred) {
  int r;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "setp.ne.b32 p, %1, 0;\n\t"
      "bar.red.or.pred q, %2, %3, p;\n\t"
      "selp.s32 %0, 1, 0, q;\n\t}"
      : "=r"(r)
      : "r"((int)pred), "r"(id), "n"(N)
      : "memory");
  return r != 0;
}
template <int N>
__device__ __forceinline__ void pn_bar_sync(int id) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "n"(N) : "memory");
}
template <int N>
__device__ __forceinline__ void pn_bar_arrive(int id) {
  asm volatile("bar.arrive %0, %1;" ::"r"(id), "n"(N) : "memory");
}

// Leaky ReLU of x to 16 bits as relu16(x) - relu16(-slope x), of which one is
// zero: two conversions with ReLU and a packed subtraction, instead of two
// maxima and a conversion, which kept the ALU pipe busier than any other: width
// 64, which instructions bound, 155 -> 146 us per 1080p FP16 frame.  Width 128
// has the longer products to wait for and keeps the shorter chain (301 us,
// 303 so, in one run).
template <bool F16>
__device__ __forceinline__ uint32_t sub16(uint32_t a, uint32_t b) {
  if (F16) {
    const __half2 d = __hsub2(*reinterpret_cast<const __half2 *>(&a), *reinterpret_cast<const __half2 *>(&b));
    return *reinterpret_cast<const uint32_t *>(&d);
  }
  const __nv_bfloat162 d = __hsub2(*reinterpret_cast<const __nv_bfloat162 *>(&a), *reinterpret_cast<const __nv_bfloat162 *>(&b));
  return *reinterpret_cast<const uint32_t *>(&d);
}

template <bool F16>
__device__ __forceinline__ float2 unpack2(uint32_t w) {
  if (F16) {
    return __half22float2(*reinterpret_cast<const __half2 *>(&w));
  } else {
    return make_float2(__uint_as_float(w << 16), __uint_as_float(w & 0xFFFF0000u));
  }
}

// W: network width; F16: FP16 (else BF16) operands; WG tile pipelines per CTA;
// H threads per point, each with two of the 32-column chunks of the
// accumulator (chunk c H + h in turn c, so that the chunks are done in order).
// Bound by the chain of a tile's seven layers, of which tensor memory holds two
// tiles per SM at width 128.  With one accumulator and one operand column set
// a layer's conversion (665 cycles) and its products (1090 with their issue)
// took turns; with the next layer's first products under the second half of
// the conversion, the next tile's encoding under the head and packed
// multiplies for the leaky ReLU: 1080p, 8 materials, width 128 363 -> 302 us,
// width 64 158 -> 155 us (issue-bound); with shared memory by offset and, at width
// 64, the leaky ReLU below 290 and 146 us (tensor pipe 62 and 36 %, issue 60 and
// 67 %).
template <int W, bool F16, int WG, int H>
__global__ void __launch_bounds__(kTile * WG * H, W == 64 ? 2 : 1) pn_decoder_kernel(const PnArgs a) {
  static_assert(W == 64 * H, "two chunks per thread");
  constexpr int PT = kTile * H;
  constexpr uint32_t COLS = pn_cols(W);
  static_assert(COLS == 2 * W, "two regions");
  constexpr int KH = W + 16;
  constexpr int HALF = W / 32;      // K steps of the first turn's chunks
  constexpr int FIT = (W - (int)kColBias) / 8;   // K steps of layer 0 beside D of layer 6
  static_assert(H == 1 || FIT >= kPnMaxK1 / 16, "further steps overwrite the head's columns, which h = 0 reads");
  extern __shared__ uint8_t smem_raw[];
  uint8_t *smem = smem_raw + (-tc::smem_addr(smem_raw) & 1023u);   // an offset: a rounded address would be generic
  uint64_t *bar_w = reinterpret_cast<uint64_t *>(smem);
  uint64_t *bar_mma = bar_w + 1;         // one per pipeline
  uint64_t *bar_drain = bar_mma + WG;    // one per pipeline: its products, after a failed wait
  uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(bar_drain + WG);
  const PnBlob B = pn_blob(W, a.n_mat);
  uint8_t *wts = smem + 1024;
  const int tid = threadIdx.x;
  const int warp = tid >> 5;
  const int warp_u = __shfl_sync(0xFFFFFFFFu, warp, 0);   // uniform to the compiler (see elect_one)
  const int wg = warp_u / (PT / 32);
  const int row = tid % kTile;
  const int h = H == 1 ? 0 : warp_u / (kTile / 32) % H;
  const bool lead = warp_u % (PT / 32) == 0;   // the warp that issues the pipeline's products
  uint64_t *my_bar = bar_mma + wg;
  const int bar0 = 1 + 2 * wg;   // named barriers of the two turns

  if (tid == 0) {
    tc::mbar_init(bar_w, 1);
    for (int g = 0; g < WG; ++g) {
      tc::mbar_init(bar_mma + g, 1);
      tc::mbar_init(bar_drain + g, 1);
    }
    tc::fence_mbar_init();
  }
  if (warp == 0) tc::tmem_alloc(tmem_slot, COLS * WG);
  tc::tc_fence_before();
  __syncthreads();
  tc::tc_fence_after();
  const uint32_t tmem = *tmem_slot + COLS * (uint32_t)wg;
  const uint32_t lane = (uint32_t)((warp & 3) * 32) << 16;

  if (tid == 0) {
    tc::mbar_arrive_expect_tx(bar_w, B.total);
    tc::bulk_g2s(wts, a.blob, B.total, bar_w);
  }
  const int64_t stride = (int64_t)gridDim.x * WG;
  int64_t tile = (int64_t)blockIdx.x * WG + wg;
  PnPoint pt = pn_load<H>(a, tile * kTile + row, h);
  bool ok = __all_sync(0xFFFFFFFFu, tc::mbar_wait_sleep(bar_w, 0, kWaitCycles));   // one outcome per warp
  const float *alb = reinterpret_cast<const float *>(wts + B.alb);
  const uint32_t w_base = tc::smem_addr(wts);
  const uint32_t idW = F16 ? tc::idesc_f16(128, W) : tc::idesc_bf16(128, W);
  const uint32_t id16 = F16 ? tc::idesc_f16(128, 16) : tc::idesc_bf16(128, 16);
  const uint32_t one16 = F16 ? 0x3C00u : 0x3F80u;
  const uint64_t slope = W == 64 ? pk2(-kPnSlope, -kPnSlope) : pk2(kPnSlope, kPnSlope);
  uint32_t phase = 0;
  uint32_t par = 0;   // 0 or W: the region of this tile's even accumulators

  // Layer l's accumulator is in region R(l), its operand in the other one, on
  // top of the accumulator it was made from: the values of chunk j in columns
  // 32 j .. 32 j + 15, the bias step in 16 .. 23.  So the products of a
  // layer's first inputs run while its last ones are still being converted.
  // Layer 0's operand lies in R(6), past the head's 16 columns; K steps that
  // do not fit are written into those once the head has been read.
  auto issue = [&](int layer, int turn) {
    if (tc::elect_one() && ok) {
      tc::tc_fence_after();
      const uint32_t rd = tmem + ((layer & 1) ? W - par : par), ra = tmem + ((layer & 1) ? par : W - par);
      const uint32_t id = layer == 6 ? id16 : idW;
      if (layer == 0) {
        const uint64_t bd = tc::smem_desc(w_base + B.l[0], 128u, (uint32_t)B.k1 * 16u);
#pragma unroll
        for (int kk = 0; kk < kPnMaxK1 / 16; ++kk) {
          if (16 * kk >= B.k1) break;
          tc::mma_f16_ts(rd, ra + (kk < FIT ? kColBias + 8u * kk : 8u * (kk - FIT)), bd + 16u * kk, id, kk > 0 ? 1u : 0u);
        }
      } else {
        const uint64_t bd = tc::smem_desc(w_base + B.l[layer], 128u, KH * 16u);
#pragma unroll
        for (int kk = turn * HALF; kk < (turn == 0 ? HALF : KH / 16); ++kk)
          tc::mma_f16_ts(rd, ra + (kk < W / 16 ? 16u * (kk & ~1) + 8u * (kk & 1) : kColBias), bd + 16u * kk, id, kk > 0 ? 1u : 0u);
      }
      if (turn == 1) tc::mma_commit(my_bar);
    }
    __syncwarp();
  };
  // This warp's stores of a turn are done: the issuing warp waits for the
  // others and issues, the others go on.  They cannot arrive twice in a turn:
  // the next one follows the wait for this layer's products, or, once such a
  // wait has expired, everybody waits here until the tile's end.
  auto hand_over = [&](int layer, int turn) {
    tc::tmem_st_wait();
    tc::tc_fence_before();
    if (lead) {
      pn_bar_sync<PT>(bar0 + turn);
      issue(layer, turn);
    } else if (ok) {
      pn_bar_arrive<PT>(bar0 + turn);
    } else {
      pn_bar_sync<PT>(bar0 + turn);
    }
  };
  // layer 0's operand of pt's point: one-blob (24 channels), one-hot material
  auto hot_words = [&](int c, int mat, uint32_t *w8) {   // K step c (16 features) of the one-hot part
    const int hot = kPnBlob + mat;
#pragma unroll
    for (int k = 0; k < 8; ++k) w8[k] = hot >> 1 == 8 * c + k ? one16 << (16 * (hot & 1)) : 0u;
  };
  auto encode = [&](uint32_t t_x) {
    if (pt.mat >= a.n_mat) {
      if (h == 0) atomicOr(a.status, kStatusBadMaterial);
      pt.mat = -2;
    }
    if (H == 1 || h == 0) {
      uint32_t wu[4] = {0u, 0u, 0u, 0u}, wr[4] = {0u, 0u, 0u, 0u};
      if (pt.mat >= 0) {
        blob_periodic<F16>(pt.u, wu);
        const float t = (__logf(fmaxf(pt.r, kRFloor)) - kPnLnRLo) * kPnInvLnSpan;
        blob_plain<F16>(t, wr);
      }
      tc::tmem_st4(t_x, wu);
      tc::tmem_st4(t_x + 8, wr);
    }
    if (H == 1 || h == 1) {
      uint32_t wv[4] = {0u, 0u, 0u, 0u}, w8[8];
      if (pt.mat >= 0) blob_periodic<F16>(pt.v, wv);
      tc::tmem_st4(t_x + 4, wv);
      hot_words(1, pt.mat, w8);
      tc::tmem_st4(t_x + 12, w8 + 4);       // features 24..31
      for (int c = 2; c < B.k1 / 16 && c < FIT; ++c) {
        hot_words(c, pt.mat, w8);
        tc::tmem_st8(t_x + 8 * c, w8);
      }
    }
  };
  // a tile's head outputs, written while the next tile's first products run
  float y[4] = {0.0f, 0.0f, 0.0f, 0.0f};
  int64_t done_p = a.n;
  int done_mat = -1, cur_mat = -1;
  auto write_out = [&] {
    if ((H == 1 || h == 0) && done_p < a.n) {
      float c4[4];
      if (done_mat < 0) {
        c4[0] = c4[1] = c4[2] = c4[3] = __int_as_float(0x7FC00000);
      } else {
        c4[0] = fmaxf(0.0f, y[0]);
        c4[1] = fmaxf(0.0f, y[1]);
        c4[2] = fmaxf(0.0f, (__expf(y[2]) - 1.0f) * (1.0f / kSpecK));
        c4[3] = fmaxf(0.0f, (__expf(y[3]) - 1.0f) * (1.0f / kSpecK));
      }
      if (a.comps) store_row4(a.comps, done_p, c4[0], c4[1], c4[2], c4[3]);
      const float4 *al = reinterpret_cast<const float4 *>(alb + (done_mat < 0 ? 0 : done_mat) * 12);
      const float4 k0 = al[0], k1 = al[1], k2 = al[2];
      a.rgb[3 * done_p + 0] = k0.x * c4[0] + k0.w * c4[1] + k1.z * c4[2] + k2.y * c4[3];
      a.rgb[3 * done_p + 1] = k0.y * c4[0] + k1.x * c4[1] + k1.w * c4[2] + k2.z * c4[3];
      a.rgb[3 * done_p + 2] = k0.z * c4[0] + k1.y * c4[1] + k2.x * c4[2] + k2.w * c4[3];
    }
  };

  encode(tmem + lane + W - par + kColBias);
  for (; tile < a.n_tiles; tile += stride) {
    cur_mat = pt.mat;
    // the angular inputs, with the constant one of A1's bias after them
    const uint32_t ang0 = tc::pack2<F16>(pt.wi0, pt.wi1), ang1 = tc::pack2<F16>(pt.wi2, pt.wo0);
    const uint32_t ang2 = tc::pack2<F16>(pt.wo1, 1.0f);
    if (H == 1 || h == 1) {
      for (int c = FIT; c < B.k1 / 16; ++c) {
        uint32_t w8[8];
        hot_words(c, cur_mat, w8);
        tc::tmem_st8(tmem + lane + W - par + 8 * (c - FIT), w8);
      }
    }
    tc::tmem_st_wait();
    tc::tc_fence_before();
    if (pn_bar_or<PT>(bar0, !ok)) {
      ok = false;
      goto teardown;
    }
    if (lead) issue(0, 1);
    pt = pn_load<H>(a, (tile + stride) * kTile + row, h);
    write_out();
    uint32_t skip[32];   // k1 as 16-bit operand pairs, for the residual block
#pragma unroll
    for (int layer = 0; layer < 6; ++layer) {
      ok = __all_sync(0xFFFFFFFFu, ok && tc::mbar_wait_sleep(my_bar, phase, kWaitCycles));
      phase ^= 1u;
      tc::tc_fence_after();
      const uint32_t t_d = tmem + lane + ((layer & 1) ? W - par : par);   // and the next operand
      float acc[2][32];
      tc::tmem_ld32(t_d + 32 * h, acc[0]);
      tc::tmem_ld_wait32(acc[0]);
      tc::tmem_ld32(t_d + 32 * (H + h), acc[1]);
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        if (c == 1) tc::tmem_ld_wait32(acc[1]);
        uint32_t w[16];
#pragma unroll
        for (int k = 0; k < 16; ++k) {
          uint64_t x = pk2(acc[c][2 * k], acc[c][2 * k + 1]);
          if (layer == 4) {
            const float2 s = unpack2<F16>(skip[16 * c + k]);
            x = add2(x, pk2(s.x, s.y));
          }
          float x0, x1, n0, n1;
          upk2(x, x0, x1);
          upk2(mul2(x, slope), n0, n1);
          w[k] = W == 64 ? sub16<F16>(tc::pack2_relu<F16>(x0, x1), tc::pack2_relu<F16>(n0, n1))
                         : tc::pack2<F16>(fmaxf(x0, n0), fmaxf(x1, n1));
          if (layer == 2) skip[16 * c + k] = w[k];
        }
        tc::tmem_st16(t_d + 32 * (c * H + h), w);
        if (c == 0 && h == 0) {
          uint32_t w8[8] = {one16, 0u, 0u, 0u, 0u, 0u, 0u, 0u};
          if (layer == 1) {
            w8[0] = ang0;
            w8[1] = ang1;
            w8[2] = ang2;
          }
          tc::tmem_st8(t_d + kColBias, w8);
        }
        hand_over(layer + 1, c);
      }
    }
    // under the head's products: the next tile's layer 0 operand
    encode(tmem + lane + par + kColBias);
    ok = __all_sync(0xFFFFFFFFu, ok && tc::mbar_wait_sleep(my_bar, phase, kWaitCycles));
    phase ^= 1u;
    tc::tc_fence_after();
    if (H == 1 || h == 0) {
      tc::tmem_ld4(tmem + lane + par, y);
      tc::tmem_ld_wait();
      done_p = tile * kTile + row;
      done_mat = cur_mat;
    }
    par = W - par;
  }
  if (ok) write_out();

  ok = !pn_bar_or<PT>(bar0, !ok);
teardown:
  if (!ok) {   // let the weights' copy and the pipeline's products land before the memory goes away
    if ((tid & 31) == 0) atomicOr(a.status, kStatusTimeout);
    if (lead && tc::elect_one()) tc::mma_commit(bar_drain + wg);
    tc::mbar_wait(bar_w, 0, kWaitCycles);
    tc::mbar_wait(bar_drain + wg, 0, kWaitCycles);
  }
  tc::tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc::tc_fence_after();
    tc::tmem_dealloc(*tmem_slot, COLS * WG);
  }
}

constexpr int kPnWG = 2;
// Threads per point.  Width 128: two, each with half of the 128 accumulator
// columns (1080p, 8 materials: 371 us, against 425 with one and 754 with four
// of 64 registers).  Width 64: one; two would leave 64 registers a thread at
// two CTAs per SM, and spill (167 us against 209).
constexpr int pn_threads(int w) { return w == 64 ? 1 : 2; }

// W = 64: two pipelines of 128 columns per CTA, two CTAs per SM (four CTAs
// of one pipeline would need four copies of the 57 KB of weights); W = 128:
// one CTA of two pipelines of 256 columns.  Either way the SM's 512
// tensor-memory columns are taken.
template <int W, bool F16>
const void *pn_kernel() {
  if (W == 64) return reinterpret_cast<const void *>(pn_decoder_kernel<64, F16, kPnWG, pn_threads(64)>);
  return reinterpret_cast<const void *>(pn_decoder_kernel<128, F16, kPnWG, pn_threads(128)>);
}

}  // namespace

int paper_k1(int n_mat) {
  const int k1 = (kPnBlob + n_mat + 15) / 16 * 16;
  return (n_mat >= 1 && k1 <= kPnMaxK1) ? k1 : -1;
}

size_t paper_blob_bytes(int w, int n_mat) { return pn_blob(w, n_mat).total; }

cudaError_t launch_paper_pack(int w, int precision, const float *params, const float *latents,
                              const DevMaterial *mats, int n_mat, void *blob, cudaStream_t s) {
  if (!paper_width_ok(w) || paper_k1(n_mat) < 0) return cudaErrorInvalidValue;
  const bool f16 = precision == FABRIC_PREC_FP16;
  const size_t smem = (size_t)n_mat * w * sizeof(float);
  uint8_t *out = static_cast<uint8_t *>(blob);
  const void *fn = w == 64 ? (f16 ? reinterpret_cast<const void *>(pn_pack_kernel<64, true>)
                                  : reinterpret_cast<const void *>(pn_pack_kernel<64, false>))
                           : (f16 ? reinterpret_cast<const void *>(pn_pack_kernel<128, true>)
                                  : reinterpret_cast<const void *>(pn_pack_kernel<128, false>));
  cudaError_t e = ensure_max_dyn_smem(fn, 64 * 1024);
  if (e != cudaSuccess) return e;
  void *args[] = {(void *)&params, (void *)&latents, (void *)&mats, (void *)&n_mat, (void *)&out};
  return cudaLaunchKernel(fn, dim3(1), dim3(256), args, smem, s);
}

cudaError_t launch_paper_decoder(int w, int precision, const fabric_gbuffer &g, const void *blob, int n_mat,
                                 float *rgb, float *comps, int *status, int sm_count, cudaStream_t s) {
  if (!paper_width_ok(w) || paper_k1(n_mat) < 0) return cudaErrorInvalidValue;
  const bool f16 = precision == FABRIC_PREC_FP16;
  const void *fn = w == 64 ? (f16 ? pn_kernel<64, true>() : pn_kernel<64, false>())
                           : (f16 ? pn_kernel<128, true>() : pn_kernel<128, false>());
  const int wg = kPnWG;
  PnArgs a = {};
  a.u = g.u;
  a.v = g.v;
  a.radius = g.radius;
  a.wi = g.wi;
  a.wo = g.wo;
  a.material = g.material;
  a.n = g.n;
  a.n_tiles = (g.n + kTile - 1) / kTile;
  a.blob = static_cast<const uint8_t *>(blob);
  a.n_mat = n_mat;
  a.rgb = rgb;
  a.comps = comps;
  a.status = status;
  // Shared memory: alignment slack, barriers, the blob; padded so that no
  // CTA beyond the ones whose tensor memory fits (it would wait for it) can
  // share an SM: width 64 two CTAs of two 128-column pipelines (at least
  // 80 KB each), width 128 one CTA of two 256-column pipelines (116 KB).
  const int per_sm = w == 64 ? 2 : 1;
  const size_t floor_smem = (size_t)(w == 64 ? 80 : 116) * 1024;
  size_t smem = 2048 + ((pn_blob(w, n_mat).total + 1023u) & ~1023u);
  if (smem < floor_smem) smem = floor_smem;
  cudaError_t e = ensure_max_dyn_smem(fn, 227 * 1024);
  if (e != cudaSuccess) return e;
  int64_t grid = (int64_t)sm_count * per_sm;
  const int64_t need = (a.n_tiles + wg - 1) / wg;
  if (grid > need) grid = need;
  if (grid < 1) grid = 1;
  void *args[] = {&a};
  return cudaLaunchKernel(fn, dim3((unsigned)grid), dim3(kTile * wg * pn_threads(w)), args, smem, s);
}

}  // namespace fab
