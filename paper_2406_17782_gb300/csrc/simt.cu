// simt.cu -- FP32 kernels on the CUDA cores: the encoder's forward and
// backward (Sec. 4.2), the sums over per-CTA gradient partials and per-row
// latent gradients, Adam, FP64 image-wide error reductions and the dataset
// shuffle.
//
// All reductions run in a fixed order (owner-computes partial sums per CTA,
// then a fixed-order sum over CTAs), so repeated runs are bitwise identical.
#include <cmath>
#include <cstring>
#include <type_traits>

#include <algorithm>

#include "f32x2.h"
#include "fabric_internal.h"

namespace fab {
namespace {

constexpr float kLeaky = 0.01f;       // encoder residual-block activation slope

// Column sums out[j] = sum_c partial[c][j].  A CTA takes 32 consecutive
// columns; its kSumSegs warps sum consecutive ranges of rows (in row order),
// then the range sums are added in range order: a fixed order, so the
// result does not change from run to run.
constexpr int kSumSegs = 8;
constexpr int kSumBatch = 24;   // one batch for up to 192 partials

__device__ void reduce_loss_warp(const double *__restrict__ part, int n, double *__restrict__ out);

// Columns [0, w0) go to out0, columns [w0, width) to out1.  One CTA past the
// column blocks (when loss_out is set) sums the loss partials instead, so
// that both reductions take one launch.
__global__ void __launch_bounds__(32 * kSumSegs) reduce_partials_kernel(const float *__restrict__ partial,
                                                                        int n_part, int stride, int width, int w0,
                                                                        float *__restrict__ out0,
                                                                        float *__restrict__ out1,
                                                                        const double *__restrict__ loss_part,
                                                                        double *__restrict__ loss_out) {
  grid_dependency_wait();
  grid_dependents_launch();
  __shared__ float seg_sum[kSumSegs][32];
  if (loss_out && blockIdx.x == gridDim.x - 1) {
    if (threadIdx.x < 32) reduce_loss_warp(loss_part, n_part, loss_out);
    return;
  }
  const int lane = threadIdx.x & 31, seg = threadIdx.x >> 5;
  const int j = blockIdx.x * 32 + lane;
  const int per = (n_part + kSumSegs - 1) / kSumSegs;
  const int c0 = min(n_part, seg * per), c1 = min(n_part, c0 + per);
  float s = 0.0f;
  if (j < width) {
    // kSumBatch loads in flight, then their sum in order
    for (int c = c0; c < c1; c += kSumBatch) {
      float t[kSumBatch];
#pragma unroll
      for (int q = 0; q < kSumBatch; ++q) t[q] = c + q < c1 ? partial[(int64_t)(c + q) * stride + j] : 0.0f;
#pragma unroll
      for (int q = 0; q < kSumBatch; ++q)
        if (c + q < c1) s += t[q];
    }
  }
  seg_sum[seg][lane] = s;
  __syncthreads();
  if (seg == 0 && j < width) {
    float tot = seg_sum[0][lane];
#pragma unroll
    for (int k = 1; k < kSumSegs; ++k) tot += seg_sum[k][lane];
    if (j < w0) out0[j] = tot;
    else out1[j - w0] = tot;
  }
}

// 32 threads (one warp) sum fixed strided subsets, then lane 0 sums the 32
// in order.
__device__ void reduce_loss_warp(const double *__restrict__ part, int n, double *__restrict__ out) {
  const int lane = threadIdx.x & 31;
  double s = 0.0;
  for (int c = lane; c < n; c += 32) s += part[c];
  double t = 0.0;
  for (int k = 0; k < 32; ++k) t += __shfl_sync(0xFFFFFFFFu, s, k);
  if (lane == 0) *out = t;
}

// dlat[m][i] = sum over rows with material m of rows[row][i], i < 32; one CTA per
// material.  The sums are those of 256 bins added in order, a bin's rows in
// row order: with V (ids read as 16-byte groups of eight) bin (row / 8) mod
// 256, the last n mod 8 rows going to bins 0..7, else bin row mod 256.  Warp w
// owns bins 32 w .. 32 w + 31: it looks through their ids, eight groups of 256
// rows in flight (lane l those of bin 32 w + l, so that only a lane's own order
// counts), lists the rows that match, a row per lane at a time, and adds the
// listed rows to their bins in shared memory with one lane per column and
// sixteen rows' loads in flight.  65 536 rows of 256 materials: 14.9 us (32 with
// a row at a time as it is found, 17.7 with a ballot for each of a group's
// eight rows and eight loads in flight).
constexpr int kSegWarps = 8;
constexpr int kSegList = 512;    // listed rows per warp, emptied when 32 more might not fit

template <bool V>
__global__ void __launch_bounds__(32 * kSegWarps) latent_sums_kernel(const uint16_t *__restrict__ mat, int64_t n,
                                                                     const float *__restrict__ rows,
                                                                     float *__restrict__ dlat, int early) {
  __shared__ float bins[32 * kSegWarps][kLatent];
  __shared__ uint32_t list[kSegWarps][kSegList];   // rows (fewer than 2^32: they are 128 bytes each)
  // early: the kernel before this one is the sum over the same partials'
  // kernel, which had completed when that one let this one start; it is waited
  // for at the end, so that this kernel's completion implies its
  if (!early) grid_dependency_wait();
  grid_dependents_launch();
  const uint32_t m = blockIdx.x, mm = m * 0x10001u;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (m > 0xFFFFu) {   // no 16-bit id names it (and mm has overflowed)
    if (threadIdx.x < kLatent) dlat[(int64_t)m * kLatent + threadIdx.x] = 0.0f;
    if (early) grid_dependency_wait();
    return;
  }
  const uint32_t below = (1u << lane) - 1u;
  for (int k = 0; k < 32; ++k) bins[32 * warp + k][lane] = 0.0f;
  const int64_t whole = V ? n & ~int64_t(7) : n;
  int count = 0;
  auto bin_of = [&](uint32_t r) { return 32 * warp + (int)(V ? (r < whole ? (r >> 3) & 31u : (uint32_t)(r - whole)) : r & 31u); };
  constexpr int kRowsInFlight = 16;
  auto add_listed = [&]() {
    __syncwarp();
    for (int e = 0; e < count; e += kRowsInFlight) {
      uint32_t r[kRowsInFlight];
      float v[kRowsInFlight];
#pragma unroll
      for (int q = 0; q < kRowsInFlight; ++q) r[q] = e + q < count ? list[warp][e + q] : 0u;
#pragma unroll
      for (int q = 0; q < kRowsInFlight; ++q) v[q] = e + q < count ? rows[(int64_t)r[q] * kLatent + lane] : 0.0f;
#pragma unroll
      for (int q = 0; q < kRowsInFlight; ++q)
        if (e + q < count) bins[bin_of(r[q])][lane] += v[q];
    }
    count = 0;
    __syncwarp();
  };
  // row of bit k of this lane in the group at `base`, and the groups' stride
  constexpr int64_t kGroup = 8 * 32 * kSegWarps;
  auto row_of = [&](int64_t base, int k) {
    return V ? base + 256 * warp + 8 * lane + k : base + 256 * k + 32 * warp + lane;
  };
  constexpr int kInFlight = 8;
  for (int64_t base0 = 0; base0 < whole; base0 += kInFlight * kGroup) {
    uint4 w[kInFlight];
#pragma unroll
    for (int q = 0; q < kInFlight; ++q) {
      const int64_t r = row_of(base0 + q * kGroup, 0);
      w[q] = V && r + 8 <= whole ? *reinterpret_cast<const uint4 *>(mat + r) : make_uint4(~mm, ~mm, ~mm, ~mm);
    }
    uint64_t bits = 0;   // bit 8 q + k: row k of group q
#pragma unroll
    for (int q = 0; q < kInFlight; ++q) {
      uint32_t b8 = 0;
      if (V) {
        const uint32_t word[4] = {w[q].x ^ mm, w[q].y ^ mm, w[q].z ^ mm, w[q].w ^ mm};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          if ((word[k] & 0xFFFFu) == 0) b8 |= 1u << (2 * k);
          if ((word[k] >> 16) == 0) b8 |= 2u << (2 * k);
        }
      } else {
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          const int64_t r = row_of(base0 + q * kGroup, k);
          if (r < n && mat[r] == m) b8 |= 1u << k;
        }
      }
      bits |= (uint64_t)b8 << (8 * q);
    }
    // each lane's rows (one bin's) in row order, a row per lane at a time
    uint32_t hit;
    while ((hit = __ballot_sync(0xFFFFFFFFu, bits != 0)) != 0) {
      if (count > kSegList - 32) add_listed();
      if (bits) {
        const int k = __ffsll(bits) - 1;
        bits &= bits - 1;
        list[warp][count + __popc(hit & below)] = (uint32_t)row_of(base0 + (k >> 3) * kGroup, k & 7);
      }
      count += __popc(hit);
    }
  }
  if (V && warp == 0) {   // the last n mod 8 rows
    if (count > kSegList - 32) add_listed();
    const int64_t r = whole + lane;
    const bool match = r < n && mat[r] == m;
    const uint32_t hit = __ballot_sync(0xFFFFFFFFu, match);
    if (match) list[warp][count + __popc(hit & below)] = (uint32_t)r;
    count += __popc(hit);
  }
  add_listed();
  __syncthreads();
  if (threadIdx.x < kLatent) {
    float s = 0.0f;
#pragma unroll 16
    for (int k = 0; k < 32 * kSegWarps; ++k) s += bins[k][threadIdx.x];
    dlat[(int64_t)m * kLatent + threadIdx.x] = s;
  }
  if (early) grid_dependency_wait();
}

// out[m][i] = sum over rows with material m of rows[row][i], i < 32 NF; one CTA
// per material.  The rows are summed in row order within segments of 512, and
// the segments' sums in order: a fixed order.  The CTA goes over 128 segments
// at a time, a warp over 16 of them: it looks through the ids 256 at a time
// (read as 16-byte loads where V), lists the rows that match in shared
// memory, and adds the listed rows with NF columns per lane and eight rows'
// loads in flight.
constexpr int kSegRows = 512;    // rows per segment
constexpr int kSegPerWarp = 16;

template <int NF>
struct Columns {
  float v[NF];
  __device__ __forceinline__ static Columns load(const float *p) {
    Columns c;
    if constexpr (NF == 4) {
      const float4 t = *reinterpret_cast<const float4 *>(p);
      c.v[0] = t.x;
      c.v[1] = t.y;
      c.v[2] = t.z;
      c.v[3] = t.w;
    } else {
      static_assert(NF == 2, "64 or 128 columns");
      const float2 t = *reinterpret_cast<const float2 *>(p);
      c.v[0] = t.x;
      c.v[1] = t.y;
    }
    return c;
  }
  __device__ __forceinline__ void add(const Columns &o) {
#pragma unroll
    for (int k = 0; k < NF; ++k) v[k] += o.v[k];
  }
};

template <bool V, int NF>
__global__ void __launch_bounds__(32 * kSegWarps) segment_sums_kernel(const uint16_t *__restrict__ mat, int64_t n,
                                                                        const float *__restrict__ rows,
                                                                        float *__restrict__ out) {
  constexpr int COLS = 32 * NF;
  extern __shared__ __align__(16) float seg_sum[];   // [kSegWarps * kSegPerWarp][COLS]
  __shared__ int list[kSegWarps][kSegList];
  __shared__ uint32_t present[kSegWarps];            // a warp's segments that have rows of the material
  // the kernel before wrote nothing that is read here; it is waited for at the
  // end, so that this kernel's completion implies its
  grid_dependents_launch();
  const uint32_t m = blockIdx.x, mm = m * 0x10001u;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t below = (1u << lane) - 1u;
  constexpr int kWarpRows = kSegPerWarp * kSegRows;
  float total = 0.0f;
  for (int64_t batch = 0; batch < n; batch += (int64_t)kSegWarps * kWarpRows) {
    const int64_t first = batch + warp * kWarpRows;
    const int last = first >= n ? 0 : (int)(n - first < kWarpRows ? n - first : kWarpRows);   // this warp's rows
    Columns<NF> acc = {};
    int count = 0, seg = 0;
    uint32_t mask = 0;
    auto close = [&](int s) {   // the sum of the current segment is complete
      if ((mask >> seg) & 1u) {
#pragma unroll
        for (int k = 0; k < NF; ++k) seg_sum[(warp * kSegPerWarp + seg) * COLS + NF * lane + k] = acc.v[k];
      }
      seg = s;
      acc = Columns<NF>{};
    };
    auto add = [&](int row, const Columns<NF> &v) {
      if (row / kSegRows != seg) close(row / kSegRows);
      mask |= 1u << seg;
      acc.add(v);
    };
    auto add_listed = [&]() {
      __syncwarp();
      const float *src = rows + first * COLS + NF * lane;
      int e = 0;
      for (; e + 8 <= count; e += 8) {
        int r[8];
        Columns<NF> v[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) r[q] = list[warp][e + q];
#pragma unroll
        for (int q = 0; q < 8; ++q) v[q] = Columns<NF>::load(src + r[q] * COLS);
#pragma unroll
        for (int q = 0; q < 8; ++q) add(r[q], v[q]);
      }
      for (; e < count; ++e) {
        const int r = list[warp][e];
        add(r, Columns<NF>::load(src + r * COLS));
      }
      count = 0;
      __syncwarp();
    };
    constexpr int kInFlight = 4;
    for (int base0 = 0; base0 < last; base0 += 256 * kInFlight) {
      uint4 w[kInFlight];
#pragma unroll
      for (int q = 0; q < kInFlight; ++q) {
        const int r = base0 + 256 * q + 8 * lane;
        w[q] = V && r + 8 <= last ? *reinterpret_cast<const uint4 *>(mat + first + r) : make_uint4(~mm, ~mm, ~mm, ~mm);
      }
#pragma unroll
      for (int q = 0; q < kInFlight; ++q) {
        // rows r .. r + 7 that match, as bits
        const int r = base0 + 256 * q + 8 * lane;
        const uint32_t word[4] = {w[q].x ^ mm, w[q].y ^ mm, w[q].z ^ mm, w[q].w ^ mm};
        uint32_t bits = 0;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          if ((word[k] & 0xFFFFu) == 0) bits |= 1u << (2 * k);
          if ((word[k] >> 16) == 0) bits |= 2u << (2 * k);
        }
        if (!V || (r < last && r + 8 > last)) {   // single ids: an unaligned array, or the last n % 8
          bits = 0;
#pragma unroll
          for (int k = 0; k < 8; ++k)
            if (r + k < last && mat[first + r + k] == m) bits |= 1u << k;
        }
        if (!__any_sync(0xFFFFFFFFu, bits != 0)) continue;
        int before = 0, hits = 0;   // matches of lower lanes, and of all
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          const uint32_t hit = __ballot_sync(0xFFFFFFFFu, (bits >> k) & 1u);
          before += __popc(hit & below);
          hits += __popc(hit);
        }
#pragma unroll
        for (int k = 0; k < 8; ++k)
          if ((bits >> k) & 1u) list[warp][count + before + __popc(bits & ((1u << k) - 1u))] = r + k;
        count += hits;
        if (count > kSegList - 256) add_listed();
      }
    }
    add_listed();
    close(0);
    if (lane == 0) present[warp] = mask;
    __syncthreads();
    if (threadIdx.x < COLS) {
      for (int w = 0; w < kSegWarps; ++w) {
        uint32_t p = present[w];
        while (p) {
          const int s = __ffs(p) - 1;
          p &= p - 1;
          total += seg_sum[(w * kSegPerWarp + s) * COLS + threadIdx.x];
        }
      }
    }
    __syncthreads();
  }
  if (threadIdx.x < COLS) out[(int64_t)m * COLS + threadIdx.x] = total;
  grid_dependency_wait();
}

// ---------------------------------------------------------------------------
// Encoder (parameters -> latent), kEncGroup materials per CTA of 128 threads.
// acts (optional) [n][2][128] = pre-activations a1, a2 for the backward pass.
// ---------------------------------------------------------------------------
__device__ __forceinline__ float lrelu(float x) { return x > 0.0f ? x : kLeaky * x; }

__device__ __forceinline__ void material_features(const fabric_material &m, float *f) {
#pragma unroll
  for (int k = 0; k < kPatternSlots; ++k) f[k] = (m.pattern_id == k) ? 1.0f : 0.0f;
  f[kPatternSlots + 0] = m.twist_deg / 30.0f;
  f[kPatternSlots + 1] = m.incl_deg / 45.0f;
  f[kPatternSlots + 2] = m.alpha[0];
  f[kPatternSlots + 3] = m.beta[0];
  f[kPatternSlots + 4] = m.alpha[1];
  f[kPatternSlots + 5] = m.beta[1];
}

// Materials per encoder CTA: thread j reads its weight row once for all of
// them and keeps one accumulator per material (each sum still runs over the
// inputs in order, as for a single material).
constexpr int kEncGroup = 4;
// Threads per unit, each with half of the group's materials: the kernels run
// one CTA per SM and wait on their own latencies (256 materials: forward 6.3
// -> 6.1 us, backward 4.9 us either way).  What more they gain comes from
// starting under the kernel before: the backward's weights and the forward's
// features are on their way before the wait (with the decoder's sums and
// Adam's operands, which do the same, eight BF16 steps 405 -> 384 us).
constexpr int kEncSplit = 2;
constexpr int kEncEach = kEncGroup / kEncSplit;
constexpr int kEncThreads = kEncHidden * kEncSplit;

// The encoder kernels stage the weights they read in shared memory with
// asynchronous copies issued at once, so that all of them are one round trip
// rather than one dependent round trip per few elements.  Rows read by one
// thread each (thread j: row j) are padded so that a warp's reads fall into
// distinct banks: E1 rows of kEncIn floats at a stride of kE1Ld (odd),
// E2 and E3 rows of 128 floats at a stride of 132 (read as float4: eight
// lanes of a quarter-warp cover the 32 banks).
constexpr int kE1Ld = kEncIn | 1;
constexpr int kERowLd = kEncHidden + 4;
constexpr size_t kEncFwdSmem = (size_t)(kEncHidden * kE1Ld + kEncHidden * kERowLd + kLatent * kERowLd) * 4;
constexpr size_t kEncBwdSmem = (size_t)(kEncHidden * kEncHidden + kLatent * kEncHidden) * 4;

__device__ __forceinline__ void cp_async4(float *dst, const float *src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}
__device__ __forceinline__ void cp_async16(float *dst, const float *src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// rows x cols floats at src (row stride cols) into dst (row stride ld), by
// all threads of the CTA; 16-byte copies when V (src, cols and ld multiples
// of four floats, src 16-byte aligned), else 4-byte ones
template <bool V>
__device__ __forceinline__ void stage_rows(float *dst, int ld, const float *src, int rows, int cols) {
  if (V) {
    const int c4 = cols / 4;
    for (int e = threadIdx.x; e < rows * c4; e += blockDim.x)
      cp_async16(dst + (e / c4) * ld + 4 * (e % c4), src + (e / c4) * cols + 4 * (e % c4));
  } else {
    for (int e = threadIdx.x; e < rows * cols; e += blockDim.x)
      cp_async4(dst + (e / cols) * ld + e % cols, src + e);
  }
}

// dot of a shared-memory weight row w (LEN floats; 16-byte aligned) with
// kEncEach vectors x[g][0..LEN), one accumulator per material, inputs in order
template <int LEN, int LD>
__device__ __forceinline__ void enc_dot_s(const float *w, const float (*x)[LD], float *acc) {
#pragma unroll 8
  for (int i4 = 0; i4 < LEN / 4; ++i4) {
    const float4 c = reinterpret_cast<const float4 *>(w)[i4];
#pragma unroll
    for (int g = 0; g < kEncEach; ++g) {
      acc[g] = fmaf(c.x, x[g][4 * i4], acc[g]);
      acc[g] = fmaf(c.y, x[g][4 * i4 + 1], acc[g]);
      acc[g] = fmaf(c.z, x[g][4 * i4 + 2], acc[g]);
      acc[g] = fmaf(c.w, x[g][4 * i4 + 3], acc[g]);
    }
  }
}

// Records of a material edit, passed with the launch instead of copied to the
// device first (a copy from pageable memory costs the edit an extra operation
// on the stream and its staging on the host).  As many as the tensor-core
// decoder takes materials, 7.5 of the 32 KB a launch may carry: encoding 33
// records 17.4 -> 13.3 us of host and device, 89 16.9 -> 14.1, and one record
// 12.7 with room for 89, 13.5 with room for 32.
constexpr int kInlineRecords = 89;
struct InlineRecords {
  fabric_material m[kInlineRecords];
};
struct NoRecords {};

// The input features come from `recs` when REC is InlineRecords, else from
// `raw` records on the device, or (raw null) from `feats`.
template <bool V, typename REC>
__global__ void __launch_bounds__(kEncThreads) encoder_fwd_kernel(const float *__restrict__ feats,
                                                                 const fabric_material *__restrict__ raw,
                                                                 float *__restrict__ feats_out, int n,
                                                                 const float *__restrict__ enc,
                                                                 float *__restrict__ z, float *__restrict__ acts,
                                                                 const __grid_constant__ REC recs) {
  extern __shared__ __align__(16) float enc_smem[];
  float *e1 = enc_smem;                             // [128][kE1Ld]
  float *e2 = e1 + kEncHidden * kE1Ld;              // [128][kERowLd]
  float *e3 = e2 + kEncHidden * kERowLd;            // [32][kERowLd]
  static_assert((kEncHidden * kE1Ld) % 4 == 0, "E2 rows 16-byte aligned in shared memory");
  __shared__ float f[kEncGroup][kEncIn];
  __shared__ __align__(16) float h1[kEncGroup][kEncHidden];
  __shared__ __align__(16) float h2[kEncGroup][kEncHidden];
  const int m0 = blockIdx.x * kEncGroup, tid = threadIdx.x;
  const int j = tid % kEncHidden, g0 = tid / kEncHidden * kEncEach;   // unit, first material of the group
  const int nm = min(kEncGroup, n - m0);
  // The records' features: before the wait where the records came with the
  // launch or are a training step's (long there; they are the ones whose
  // features are kept), after it where a copy on the stream has just brought them.
  const bool records = std::is_same<REC, InlineRecords>::value || raw;
  const bool early = std::is_same<REC, InlineRecords>::value || feats_out;
  auto features = [&] {
    if (tid >= kEncGroup) return;
    float t[kEncIn];
    if (tid < nm) {
      if constexpr (std::is_same<REC, InlineRecords>::value) material_features(recs.m[m0 + tid], t);
      else material_features(raw[m0 + tid], t);
    } else {
#pragma unroll
      for (int i = 0; i < kEncIn; ++i) t[i] = 0.0f;
    }
#pragma unroll
    for (int i = 0; i < kEncIn; ++i) f[tid][i] = t[i];
  };
  if (records && early) features();
  grid_dependency_wait();
  grid_dependents_launch();
  stage_rows<false>(e1, kE1Ld, enc + kOffE1, kEncHidden, kEncIn);
  stage_rows<V>(e2, kERowLd, enc + kOffE2, kEncHidden, kEncHidden);
  stage_rows<V>(e3, kERowLd, enc + kOffE3, kLatent, kEncHidden);
  if (records) {
    if (!early) features();
    if (tid < nm && feats_out) {
#pragma unroll
      for (int i = 0; i < kEncIn; ++i) feats_out[(int64_t)(m0 + tid) * kEncIn + i] = f[tid][i];
    }
  } else {
    for (int t = tid; t < kEncGroup * kEncIn; t += kEncThreads) {
      const int g = t / kEncIn, i = t % kEncIn;
      f[g][i] = g < nm ? feats[(int64_t)(m0 + g) * kEncIn + i] : 0.0f;
    }
  }
  const float b1 = enc[kOffEb1 + j], b2 = enc[kOffEb2 + j], b3 = enc[kOffEb3 + j % kLatent];
  cp_async_wait_all();
  __syncthreads();
  float a1[kEncEach], a2[kEncEach];
#pragma unroll
  for (int g = 0; g < kEncEach; ++g) a1[g] = b1;
#pragma unroll
  for (int i = 0; i < kEncIn; ++i) {
    const float c = e1[j * kE1Ld + i];
#pragma unroll
    for (int g = 0; g < kEncEach; ++g) a1[g] = fmaf(c, f[g0 + g][i], a1[g]);
  }
#pragma unroll
  for (int g = 0; g < kEncEach; ++g) h1[g0 + g][j] = lrelu(a1[g]);
  __syncthreads();
#pragma unroll
  for (int g = 0; g < kEncEach; ++g) a2[g] = b2 + h1[g0 + g][j];   // skip connection before the last activation
  enc_dot_s<kEncHidden, kEncHidden>(e2 + j * kERowLd, h1 + g0, a2);
#pragma unroll
  for (int g = 0; g < kEncEach; ++g) {
    h2[g0 + g][j] = lrelu(a2[g]);
    if (acts && g0 + g < nm) {
      acts[(int64_t)(m0 + g0 + g) * 2 * kEncHidden + j] = a1[g];
      acts[(int64_t)(m0 + g0 + g) * 2 * kEncHidden + kEncHidden + j] = a2[g];
    }
  }
  __syncthreads();
  // layer 3: thread j < 128 computes latent output k = j % 32 of material j / 32
  static_assert(kEncGroup * kLatent == kEncHidden, "one layer-3 output per thread");
  if (tid >= kEncHidden) return;
  const int k = j % kLatent, g = j / kLatent;
  float acc = b3;
  const float *w3 = e3 + k * kERowLd;
#pragma unroll 8
  for (int i4 = 0; i4 < kEncHidden / 4; ++i4) {
    const float4 c = reinterpret_cast<const float4 *>(w3)[i4];
    acc = fmaf(c.x, h2[g][4 * i4], acc);
    acc = fmaf(c.y, h2[g][4 * i4 + 1], acc);
    acc = fmaf(c.z, h2[g][4 * i4 + 2], acc);
    acc = fmaf(c.w, h2[g][4 * i4 + 3], acc);
  }
  if (g < nm) z[(int64_t)(m0 + g) * kLatent + k] = acc;
}

// Per material: back-propagated pre-activation gradients da1, da2 and the
// activations h1, h2 into work [n][4][128]; kEncGroup materials per CTA.
template <bool V>
__global__ void __launch_bounds__(kEncThreads) encoder_bwd_vec_kernel(const float *__restrict__ enc, int n,
                                                                     const float *__restrict__ acts,
                                                                     const float *__restrict__ dz,
                                                                     float *__restrict__ work) {
  // E2 and E3 staged as they are (thread j reads their column j: a warp's
  // reads are consecutive words), on their way before the kernel before this
  // one has finished: it never writes them (the sums of a training step, or
  // the encoder's forward pass)
  extern __shared__ __align__(16) float enc_smem[];
  float *e2 = enc_smem;                          // [128][128]
  float *e3 = e2 + kEncHidden * kEncHidden;      // [32][128]
  stage_rows<V>(e2, kEncHidden, enc + kOffE2, kEncHidden, kEncHidden);
  stage_rows<V>(e3, kEncHidden, enc + kOffE3, kLatent, kEncHidden);
  grid_dependency_wait();
  grid_dependents_launch();
  __shared__ float sdz[kEncGroup][kLatent], da2s[kEncGroup][kEncHidden];
  const int m0 = blockIdx.x * kEncGroup, tid = threadIdx.x;
  const int j = tid % kEncHidden, g0 = tid / kEncHidden * kEncEach;   // unit, first material of the group
  const int nm = min(kEncGroup, n - m0);
  float a1[kEncEach], a2[kEncEach];
#pragma unroll
  for (int g = 0; g < kEncEach; ++g) {
    const int64_t m = g0 + g < nm ? m0 + g0 + g : m0;
    a1[g] = acts[m * 2 * kEncHidden + j];
    a2[g] = acts[m * 2 * kEncHidden + kEncHidden + j];
  }
  if (tid < kEncGroup * kLatent) {
    const int k = tid % kLatent, g = tid / kLatent;
    sdz[g][k] = g < nm ? dz[(int64_t)(m0 + g) * kLatent + k] : 0.0f;
  }
  cp_async_wait_all();
  __syncthreads();
  float dh2[kEncEach], dh1[kEncEach];
#pragma unroll
  for (int g = 0; g < kEncEach; ++g) dh2[g] = 0.0f;
#pragma unroll 8
  for (int k = 0; k < kLatent; ++k) {
    const float w3 = e3[k * kEncHidden + j];
#pragma unroll
    for (int g = 0; g < kEncEach; ++g) dh2[g] = fmaf(w3, sdz[g0 + g][k], dh2[g]);
  }
#pragma unroll
  for (int g = 0; g < kEncEach; ++g) {
    const float da2 = dh2[g] * (a2[g] > 0.0f ? 1.0f : kLeaky);
    da2s[g0 + g][j] = da2;
    dh1[g] = da2;   // through the skip
  }
  __syncthreads();
#pragma unroll 8
  for (int o = 0; o < kEncHidden; ++o) {
    const float w2 = e2[o * kEncHidden + j];
#pragma unroll
    for (int g = 0; g < kEncEach; ++g) dh1[g] = fmaf(w2, da2s[g0 + g][o], dh1[g]);
  }
#pragma unroll
  for (int g = 0; g < kEncEach; ++g) {
    if (g0 + g >= nm) break;
    float *w = work + (int64_t)(m0 + g0 + g) * 4 * kEncHidden;
    w[j] = dh1[g] * (a1[g] > 0.0f ? 1.0f : kLeaky);
    w[kEncHidden + j] = da2s[g0 + g][j];
    w[2 * kEncHidden + j] = lrelu(a1[g]);
    w[3 * kEncHidden + j] = lrelu(a2[g]);
  }
}

// Encoder parameter gradients: every block is a sum over materials of outer
// products, out[r][c] = sum_m L[m][r] R[m][c] (R = 1 for the biases).  A CTA
// takes a 16 x 16 tile of one of them with two groups of 64 threads: group q
// sums over the q-th half of the materials, staging kGradChunk materials' rows
// of L and R at a time in shared memory (all of a chunk's copies in flight
// together), thread (ty, tx) accumulating rows 2 ty, 2 ty + 1 of columns 2 tx,
// 2 tx + 1 over its materials in order; the tile is then (first half) +
// (second half).  Bound by the shared-memory loads: four warps with two 8-byte
// loads a step on 112 SMs, instead of sixteen with a 16-byte and a 4-byte one
// on 33 (256 materials: 8.5 -> 5.7 us).
constexpr int kGradChunk = 128;
constexpr int kGradTile = 16;

// Adam (Kingma and Ba 2015) with bias correction, one parameter.
__device__ __forceinline__ void adam_update(float *p, float *m, float *v, float g, float lr, float bc1, float bc2) {
  const float mi = 0.9f * *m + 0.1f * g;
  const float vi = 0.999f * *v + 0.001f * g * g;
  *m = mi;
  *v = vi;
  *p -= lr * (mi / bc1) / (sqrtf(vi / bc2) + 1e-8f);
}

// Block cb of the decoder's gradient: columns 32 cb .. 32 cb + 31 summed over
// the partials exactly as reduce_partials_kernel sums them (kSumSegs
// segments of partials in order, then the segments in order), then Adam.
constexpr int kGradThreads = 128;
__device__ void dec_reduce_adam(const DecAdamArgs &d, int cb) {
  __shared__ float seg_sum[kSumSegs][32];
  const int lane = threadIdx.x & 31;
  const int j = cb * 32 + lane;
  const int per = (d.n_part + kSumSegs - 1) / kSumSegs;
#pragma unroll
  for (int seg = threadIdx.x >> 5; seg < kSumSegs; seg += kGradThreads / 32) {
    const int c0 = min(d.n_part, seg * per), c1 = min(d.n_part, c0 + per);
    float s = 0.0f;
    if (j < d.n) {
      for (int c = c0; c < c1; c += kSumBatch) {
        float t[kSumBatch];
#pragma unroll
        for (int q = 0; q < kSumBatch; ++q) t[q] = c + q < c1 ? d.partial[(int64_t)(c + q) * d.stride + j] : 0.0f;
#pragma unroll
        for (int q = 0; q < kSumBatch; ++q)
          if (c + q < c1) s += t[q];
      }
    }
    seg_sum[seg][lane] = s;
  }
  __syncthreads();
  if (threadIdx.x < 32 && j < d.n) {
    float tot = seg_sum[0][lane];
#pragma unroll
    for (int k = 1; k < kSumSegs; ++k) tot += seg_sum[k][lane];
    adam_update(d.p + j, d.m + j, d.v + j, tot, d.lr, d.bc1, d.bc2);
  }
}

struct GradBlock {
  int l_off, r_off;        // column offsets of L and R in their per-material rows (r_off < 0: R = 1)
  int l_src, r_src;        // 0: work rows (512 floats), 1: feats rows (kEncIn), 2: dz rows (kLatent)
  int rows, cols;          // extent of the whole parameter block
  int out;                 // offset of the block in the encoder parameters
};

__host__ __device__ constexpr int grad_tiles(int rows, int cols) {
  return rows / kGradTile * ((cols + kGradTile - 1) / kGradTile);
}
static_assert(kEncHidden % kGradTile == 0 && kLatent % kGradTile == 0, "whole tiles of rows");
constexpr int kGradTiles = grad_tiles(kEncHidden, kEncIn) + grad_tiles(kEncHidden, 1) +
                           grad_tiles(kEncHidden, kEncHidden) + grad_tiles(kEncHidden, 1) +
                           grad_tiles(kLatent, kEncHidden) + grad_tiles(kLatent, 1);

// The parameter block of tile t, and t's place in it: immediate operands (the
// table in constant memory was six dependent misses at each CTA's start).
__device__ __forceinline__ GradBlock grad_block(int &t) {
  constexpr int t1 = grad_tiles(kEncHidden, kEncIn), t2 = t1 + grad_tiles(kEncHidden, 1);
  constexpr int t3 = t2 + grad_tiles(kEncHidden, kEncHidden), t4 = t3 + grad_tiles(kEncHidden, 1);
  constexpr int t5 = t4 + grad_tiles(kLatent, kEncHidden);
  if (t < t1) return {0, 0, 0, 1, kEncHidden, kEncIn, kOffE1};                              // E1[j][i] = sum da1_j f_i
  if (t < t2) return t -= t1, GradBlock{0, -1, 0, 0, kEncHidden, 1, kOffEb1};               // e1[j]
  if (t < t3) return t -= t2, GradBlock{kEncHidden, 2 * kEncHidden, 0, 0, kEncHidden, kEncHidden, kOffE2};   // E2[j][i] = sum da2_j h1_i
  if (t < t4) return t -= t3, GradBlock{kEncHidden, -1, 0, 0, kEncHidden, 1, kOffEb2};      // e2[j]
  if (t < t5) return t -= t4, GradBlock{0, 3 * kEncHidden, 2, 0, kLatent, kEncHidden, kOffE3};   // E3[k][i] = sum dz_k h2_i
  return t -= t5, GradBlock{0, -1, 2, 0, kLatent, 1, kOffEb3};                              // e3[k]
}

__device__ __forceinline__ const float *grad_src(int src, const float *work, const float *feats, const float *dz,
                                                 int &ld) {
  ld = src == 0 ? 4 * kEncHidden : src == 1 ? kEncIn : kLatent;
  return src == 0 ? work : src == 1 ? feats : dz;
}

// dz_v: dz can be read as float4 (the work rows always can).
__global__ void __launch_bounds__(kGradThreads) encoder_grad_kernel(const float *__restrict__ feats, int n,
                                                                    const float *__restrict__ dz, int dz_v,
                                                                    const float *__restrict__ work,
                                                                    float *__restrict__ denc, const DecAdamArgs dec) {
  // The decoder's gradient sums and Adam update, without a wait: the kernel
  // that wrote the partials and the one that read the parameters had completed
  // when the encoder's backward, the kernel before this one, passed its wait.
  if (blockIdx.x >= kGradTiles) {
    dec_reduce_adam(dec, blockIdx.x - kGradTiles);
    return;
  }
  grid_dependency_wait();
  grid_dependents_launch();
  __shared__ __align__(16) float sl[2][kGradChunk][kGradTile];
  __shared__ __align__(16) float sr[2][kGradChunk][kGradTile];
  // which block, and which tile of it
  int t = blockIdx.x;
  const GradBlock B = grad_block(t);
  const int ct = (B.cols + kGradTile - 1) / kGradTile;
  const int r0 = (t / ct) * kGradTile, c0 = (t % ct) * kGradTile;
  int ldl, ldr;
  const float *L = grad_src(B.l_src, work, feats, dz, ldl) + B.l_off + r0;
  const float *R = grad_src(B.r_src, work, feats, dz, ldr) + B.r_off + c0;
  const int q = threadIdx.x >> 6, tid = threadIdx.x & 63, ty = tid >> 3, tx = tid & 7;
  const int half = (n + 1) / 2, m_begin = q == 0 ? 0 : half, m_end = q == 0 ? half : n;
  const int rounds = (half + kGradChunk - 1) / kGradChunk;   // the same for both groups (CTA barriers)
  // mc rows of 16 columns, `cols` of them there, into s
  auto stage = [&](float(*s)[kGradTile], const float *src, int ld, int mc, int cols, bool v) {
    if (v) {
      for (int e = tid; e < mc * (kGradTile / 4); e += 64) cp_async16(&s[e >> 2][4 * (e & 3)], src + (int64_t)(e >> 2) * ld + 4 * (e & 3));
    } else {
      for (int e = tid; e < mc * kGradTile; e += 64)
        if ((e & 15) < cols) cp_async4(&s[e >> 4][e & 15], src + (int64_t)(e >> 4) * ld + (e & 15));
    }
  };
  float acc[2][2] = {{0.0f, 0.0f}, {0.0f, 0.0f}};
  for (int k0 = 0; k0 < rounds; ++k0) {
    const int m0 = m_begin + k0 * kGradChunk;
    const int mc = max(0, min(kGradChunk, m_end - m0));
    __syncthreads();
    stage(sl[q], L + (int64_t)m0 * ldl, ldl, mc, kGradTile, B.l_src == 0 || dz_v);
    if (B.r_off >= 0) {
      stage(sr[q], R + (int64_t)m0 * ldr, ldr, mc, B.cols - c0, B.r_src == 0);
    } else {
      for (int mm = tid; mm < mc; mm += 64) sr[q][mm][0] = 1.0f;
    }
    cp_async_wait_all();
    __syncthreads();
#pragma unroll 8
    for (int mm = 0; mm < mc; ++mm) {
      const float2 a = reinterpret_cast<const float2 *>(sl[q][mm])[ty];
      const float2 x = reinterpret_cast<const float2 *>(sr[q][mm])[tx];
      acc[0][0] = fmaf(a.x, x.x, acc[0][0]);
      acc[0][1] = fmaf(a.x, x.y, acc[0][1]);
      acc[1][0] = fmaf(a.y, x.x, acc[1][0]);
      acc[1][1] = fmaf(a.y, x.y, acc[1][1]);
    }
  }
  // the second half's sums through shared memory, added to the first half's
  __syncthreads();
  float(*part)[kGradTile] = sl[0];
  if (q == 1) {
#pragma unroll
    for (int i = 0; i < 2; ++i) reinterpret_cast<float2 *>(part[2 * ty + i])[tx] = make_float2(acc[i][0], acc[i][1]);
  }
  __syncthreads();
  if (q == 0) {
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        const int c = c0 + 2 * tx + k;
        if (c < B.cols) denc[B.out + (r0 + 2 * ty + i) * B.cols + c] = acc[i][k] + part[2 * ty + i][2 * tx + k];
      }
  }
}

// ---------------------------------------------------------------------------
// Adam (Kingma and Ba 2015) with bias correction.
// ---------------------------------------------------------------------------
// Parameters [0, n0) live in p0 and [n0, n0 + n1) in p1; g, m and v hold
// both sets back to back.
__global__ void adam_kernel(float *__restrict__ p0, int64_t n0, float *__restrict__ p1, int64_t n1,
                            const float *__restrict__ g, float *__restrict__ m, float *__restrict__ v, float lr,
                            float bc1, float bc2) {
  // what is updated is read before the wait: the kernel before has not written
  // it (launch_adam's condition)
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  float *p = i < n0 ? p0 + i : p1 + (i - n0);
  float pi = 0.0f, mi = 0.0f, vi = 0.0f;
  if (i < n0 + n1) {
    pi = *p;
    mi = m[i];
    vi = v[i];
  }
  grid_dependency_wait();
  grid_dependents_launch();
  if (i >= n0 + n1) return;
  adam_update(&pi, &mi, &vi, g[i], lr, bc1, bc2);
  *p = pi;
  m[i] = mi;
  v[i] = vi;
}

// ---------------------------------------------------------------------------
// FP64 error statistics: fixed grid of partial sums, then one fixed-order sum.
// ---------------------------------------------------------------------------
constexpr int kErrBlocks = 608;   // one wave: 4 CTAs of 256 threads (64 registers) on each of 152 SMs
constexpr int kErrThreads = 256;

// Per element the kernel needs (w(a-b))^2, (w b)^2 and |w(a-b)| to FP64
// accuracy.  On this GPU FP64 instructions issue at a small fraction of the
// FP32 rate, so the main loop holds no FP64 arithmetic at all: the terms are
// formed with error-free FP32 transformations (Knuth's TwoSum, the FMA
// TwoProduct) as unevaluated sums hi + lo -- a - b is exact as a pair, its
// square exact to about 2^-48 relative -- and each thread adds runs of
// kErrRun terms in renormalised double-float form (error below
// kErrRun * 2^-47 of a run's sum) before adding the run into its FP64 sums.
// The maximum is kept as a pair too: |a - b| = |hi| + sign(hi) lo, compared
// lexicographically, which is exact because FP32 rounding is monotone (with
// weights, the pair carries the product to about 2^-47 relative).  Elements
// whose values fall outside [2^-40, 2^60] in magnitude (where a square could
// overflow or its low part leave the normal range), and non-finite ones,
// are skipped there and handled in FP64 by a second pass over the thread's
// share, which runs only in threads that met one.
constexpr int kErrRun = 32;
constexpr int kErrBatch = 8;   // loads in flight per thread

__device__ __forceinline__ void two_sum(float a, float b, float &s, float &e) {
  s = __fadd_rn(a, b);
  const float bv = __fsub_rn(s, a);
  const float av = __fsub_rn(s, bv);
  e = __fadd_rn(__fsub_rn(a, av), __fsub_rn(b, bv));
}
__device__ __forceinline__ void two_prod(float a, float b, float &p, float &e) {
  p = __fmul_rn(a, b);
  e = __fmaf_rn(a, b, -p);
}
// s = h + l (|l| <= ulp(h) / 2) += x + y, with x >= 0 and |y| << x
struct DFloat {
  float h = 0.0f, l = 0.0f;
  __device__ __forceinline__ void add(float x, float y) {
    float t, e;
    two_sum(h, x, t, e);
    e = __fadd_rn(e, __fadd_rn(l, y));
    h = __fadd_rn(t, e);                 // fast two-sum: t >= |e|
    l = __fsub_rn(e, __fsub_rn(h, t));
  }
};

__device__ __forceinline__ bool err_fast(float x) {
  const float ax = fabsf(x);
  return ax == 0.0f || (ax >= 0x1p-40f && ax <= 0x1p60f);
}

// w (a - b) as dh + dl and w b as bh + bl; true when the pairs' range holds
template <bool W>
__device__ __forceinline__ bool err_pairs(float ai, float bi, float wv, float &dh, float &dl, float &bh, float &bl) {
  two_sum(ai, -bi, dh, dl);
  if (W) {
    float th, te;
    two_prod(dh, wv, th, te);
    dl = __fmaf_rn(dl, wv, te);
    dh = th;
    two_prod(bi, wv, bh, bl);
  } else {
    bh = bi;
    bl = 0.0f;
  }
  return err_fast(dh) && err_fast(bh) && (!W || err_fast(wv));
}

// i / group for 0 <= i < 2^31: one multiplication (group = 1: mul 0, shift 0).
// mul = ceil(2^p / group) < 2^32 with p = 31 + ceil(log2 group), so mul group
// exceeds 2^p by less than 2^(p - 31) and the quotient is exact below 2^31.
// The weights' index takes two divisions per pair of elements, which the
// general division (about 25 instructions) dominated.
struct GroupDiv {
  int group;
  uint32_t mul, shift;
  __device__ __forceinline__ int64_t operator()(int i) const {
    return mul ? (int64_t)(__umulhi((uint32_t)i, mul) >> shift) : (int64_t)i;
  }
  __device__ __forceinline__ int64_t operator()(int64_t i) const { return i / group; }
};
GroupDiv group_div(int group) {
  GroupDiv d{group, 0u, 0u};
  if (group > 1) {
    int lg = 1;
    while ((1ll << lg) < group) ++lg;
    const int p = 31 + lg;
    d.mul = (uint32_t)(((1ull << p) + (uint64_t)group - 1) / (uint64_t)group);
    d.shift = (uint32_t)(p - 32);
  }
  return d;
}

// CTA totals in thread 0 through shared memory: a fixed tree, halving the
// threads that add (the largest value compares as an integer, since it is
// non-negative).
__device__ __forceinline__ void err_reduce(double (*s)[kErrThreads], double &e2, double &b2, double &mx) {
  const int t = threadIdx.x;
  s[0][t] = e2;
  s[1][t] = b2;
  s[2][t] = mx;
  __syncthreads();
  auto larger = [](double x, double y) {
    return __double_as_longlong(x) > __double_as_longlong(y) ? x : y;
  };
#pragma unroll
  for (int off = kErrThreads / 2; off >= 32; off >>= 1) {
    if (t < off) {
      s[0][t] = e2 = e2 + s[0][t + off];
      s[1][t] = b2 = b2 + s[1][t + off];
      s[2][t] = mx = larger(mx, s[2][t + off]);
    }
    __syncthreads();
  }
  if (t < 32) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
      e2 += __shfl_down_sync(0xFFFFFFFFu, e2, off);
      b2 += __shfl_down_sync(0xFFFFFFFFu, b2, off);
      mx = larger(mx, __shfl_down_sync(0xFFFFFFFFu, mx, off));
    }
  }
}

// A CTA's totals into its place among the partials, or, when it is the only
// one, to the output.
__device__ __forceinline__ void err_store(double e2, double b2, double mx, double *__restrict__ part,
                                          double *__restrict__ out) {
  __shared__ double s[3][kErrThreads];
  err_reduce(s, e2, b2, mx);
  if (threadIdx.x == 0) {
    double *o = gridDim.x == 1 ? out : part + 3 * blockIdx.x;
    o[0] = e2;
    o[1] = b2;
    o[2] = mx;
  }
}

// The sum over the partials, by one CTA: thread t takes partials t, t + 256,
// ... in order, then the fixed tree.  Launched under the kernel that writes
// them, so that it is ready when that one ends.  (The last CTA of that kernel
// doing it instead needs a counter that outlives the call, which two calls
// at once on two streams left at a value from which no later call recovered,
// and is no faster: a weighted 1080p RGB frame 24.8 us either way, 1000
// elements, one CTA that needs no sum, 6.2 against 8.3.)
__global__ void __launch_bounds__(kErrThreads) err_final_kernel(const double *__restrict__ part, int n,
                                                                double *__restrict__ out) {
  __shared__ double s[3][kErrThreads];
  grid_dependency_wait();
  double e2 = 0.0, b2 = 0.0, mx = 0.0;
  for (int k = threadIdx.x; k < n; k += kErrThreads) {
    e2 += part[3 * k];
    b2 += part[3 * k + 1];
    mx = fmax(mx, part[3 * k + 2]);
  }
  err_reduce(s, e2, b2, mx);
  if (threadIdx.x == 0) {
    out[0] = e2;
    out[1] = b2;
    out[2] = mx;
  }
}

// W: weights present; Idx: index type (32-bit when n and the strides fit).
template <bool W, typename Idx>
__global__ void __launch_bounds__(kErrThreads) err_partial_kernel(const float *__restrict__ a,
                                                                  const float *__restrict__ b, int64_t n_,
                                                                  const float *__restrict__ w, GroupDiv group,
                                                                  int w_stride, double *__restrict__ part,
                                                                  double *__restrict__ out) {
  grid_dependents_launch();   // the sum over the partials (err_final_kernel)
  const Idx n = (Idx)n_;
  const Idx stride = (Idx)gridDim.x * kErrThreads;
  const Idx start = (Idx)blockIdx.x * kErrThreads + threadIdx.x;
  double e2 = 0.0, b2 = 0.0;
  float mh = -1.0f, ml = 0.0f;   // largest |w(a-b)| so far as mh + ml (mh < 0: none)
  bool slow = false;
  for (Idx i0 = start; i0 < n; i0 += kErrRun * stride) {
    DFloat E, B;
#pragma unroll 1
    for (int r0 = 0; r0 < kErrRun; r0 += kErrBatch) {
      // a batch of loads in flight together; positions past n read as a = b = 0
      float av[kErrBatch], bv[kErrBatch], wv[kErrBatch];
#pragma unroll
      for (int q = 0; q < kErrBatch; ++q) {
        const Idx i = i0 + (Idx)(r0 + q) * stride;
        const bool in = i < n;
        av[q] = in ? a[i] : 0.0f;
        bv[q] = in ? b[i] : 0.0f;
        wv[q] = W && in ? w[group(i) * w_stride] : 1.0f;
      }
#pragma unroll
      for (int q = 0; q < kErrBatch; ++q) {
        float dh, dl, bh, bl;
        if (!err_pairs<W>(av[q], bv[q], wv[q], dh, dl, bh, bl)) {
          slow = true;
          continue;
        }
        float p, pe, qq, qe;
        two_prod(dh, dh, p, pe);
        two_prod(bh, bh, qq, qe);
        E.add(p, __fmaf_rn(2.0f * dh, dl, pe));   // (dh + dl)^2 without the dl^2 term (below 2^-48)
        B.add(qq, __fmaf_rn(2.0f * bh, bl, qe));
        const float sh = fabsf(dh);
        if (sh >= mh) {   // rare once the running maximum has grown: one compare per element
          const float sl = dh < 0.0f ? -dl : dl;
          if (sh > mh || sl > ml) {
            mh = sh;
            ml = sl;
          }
        }
      }
    }
    e2 += (double)E.h + (double)E.l;
    b2 += (double)B.h + (double)B.l;
  }
  double mx = mh < 0.0f ? 0.0 : (double)mh + (double)ml;
  if (slow) {
    for (Idx i = start; i < n; i += stride) {
      const float ai = a[i], bi = b[i];
      const float wv = W ? w[group(i) * w_stride] : 1.0f;
      float dh, dl, bh, bl;
      if (err_pairs<W>(ai, bi, wv, dh, dl, bh, bl)) continue;
      const double wi = (double)wv;
      const double d = ((double)ai - (double)bi) * wi;
      const double bb = (double)bi * wi;
      e2 += d * d;
      b2 += bb * bb;
      mx = fmax(mx, fabs(d));
    }
  }
  err_store(e2, b2, mx, part, out);
}

// ---- the same reduction on pairs of elements with packed FP32x2
// instructions (add/sub/mul/fma.rn.f32x2: one instruction for two lanes),
// which halves the arithmetic instruction count of the error-free
// transformations; used when a and b are 8-byte aligned.  Lane 0 of every
// packed value carries the even element of a pair, lane 1 the odd one; each
// lane has its own double-float run sums.
// No element is range-checked in the main loop.  Where the FP32 pairs cannot
// carry a term exactly, the thread's results show it: a square or sum that
// overflows (or a non-finite input) makes its FP64 sums non-finite, and a
// square whose low part falls below the normal range loses at most 2^-149
// absolutely, which is below 2^-49 of the thread's sum unless its largest
// |w(a-b)| (or |w b|) is under sqrt(elements) 2^-50.  A thread in either
// case redoes its whole share in FP64 instead.  One whose largest value is
// exactly zero need not where its sums are then exact: without weights, and
// with them unless it met a nonzero weight and a nonzero a - b (or b), whose
// product may have underflowed (three ORs a pair: a weighted 1080p RGB frame
// 24.5 -> 24.8 us, 2^25 elements 84.3 -> 86.4).
constexpr int kErrRun2 = 16;    // pairs per run
constexpr int kErrBatch2 = 4;   // pair loads in flight per thread (eight without weights)
constexpr int kErrPerSm2 = 4;   // resident CTAs per SM
constexpr int kErrBlocks2 = 152 * kErrPerSm2;   // one wave on 152 SMs

constexpr uint64_t kSign2 = 0x8000000080000000ull;   // both lanes' sign bits

// Packed DFloat: (h, l) += (x, y) per lane, as DFloat::add.
__device__ __forceinline__ void dadd2(uint64_t &h, uint64_t &l, uint64_t x, uint64_t y) {
  const uint64_t t = add2(h, x);
  const uint64_t bv = sub2(t, h);
  const uint64_t av = sub2(t, bv);
  uint64_t e = add2(sub2(h, av), sub2(x, bv));
  e = add2(e, add2(l, y));
  h = add2(t, e);
  l = sub2(e, sub2(h, t));
}

// Both lanes of a run's packed sums in FP64, but for `rest`: the lanes' parts
// are joined by TwoSums in FP32, whose last terms (2^-48 of the sum) collect
// there for the whole thread, so that a run costs two FP64 conversions and
// one addition instead of four and three (FP64 instructions issue at about a
// fifteenth of a cycle each per SM, and at frame sizes a thread has only one
// or two runs: a weighted 1080p RGB frame 24.8 us, 26.8 with all of it in
// FP64 and the same error, 6.5e-16 of the exact sum; 50 001 elements 1.1e-16,
// and 2.8e-16 without those terms).
__device__ __forceinline__ double lanes_sum(uint64_t h, uint64_t l, float &rest) {
  float h0, h1, l0, l1, s, e, a, r1, b, r2;
  upk2(h, h0, h1);
  upk2(l, l0, l1);
  two_sum(h0, h1, s, e);
  two_sum(l0, l1, a, r1);
  two_sum(e, a, b, r2);
  rest = __fadd_rn(rest, __fadd_rn(r1, r2));
  return (double)s + (double)b;
}
__device__ __forceinline__ bool finite64(double x) { return (__double2hiint(x) & 0x7FF00000) != 0x7FF00000; }

template <bool W, typename Idx>
__global__ void __launch_bounds__(kErrThreads, kErrPerSm2) err_partial2_kernel(const float *__restrict__ a,
                                                                   const float *__restrict__ b, int64_t n_,
                                                                   const float *__restrict__ w, GroupDiv group,
                                                                   int w_stride, double *__restrict__ part,
                                                                   double *__restrict__ out) {
  grid_dependents_launch();   // the sum over the partials (err_final_kernel)
  const uint64_t *a2 = reinterpret_cast<const uint64_t *>(a);
  const uint64_t *b2 = reinterpret_cast<const uint64_t *>(b);
  const Idx n = (Idx)n_;
  const Idx np = n / 2;   // pairs; an odd last element is added by the FP64 pass of thread 0
  const Idx stride = (Idx)gridDim.x * kErrThreads;
  const Idx start = (Idx)blockIdx.x * kErrThreads + threadIdx.x;
  const uint64_t two = pk2(2.0f, 2.0f);
  double e2 = 0.0, b2s = 0.0;
  float e_rest = 0.0f, b_rest = 0.0f;
  float mh = -1.0f, ml = 0.0f, bmax = 0.0f;
  uint32_t any_d = 0, any_b = 0, any_w = 0;   // W: all bits of a - b, b and w
  auto bits2 = [](uint64_t x) { return (uint32_t)x | (uint32_t)(x >> 32); };
  for (Idx j0 = start; j0 < np; j0 += kErrRun2 * stride) {
    uint64_t EH = 0, EL = 0, BH = 0, BL = 0;
    constexpr int NB = W ? kErrBatch2 : 2 * kErrBatch2;
#pragma unroll 1
    for (int r0 = 0; r0 < kErrRun2 && j0 + (Idx)r0 * stride < np; r0 += NB) {
      uint64_t av[NB], bv[NB], wv[NB];
#pragma unroll
      for (int q = 0; q < NB; ++q) {
        const Idx j = j0 + (Idx)(r0 + q) * stride;
        const bool in = j < np;
        av[q] = in ? __ldg(a2 + j) : 0ull;
        bv[q] = in ? __ldg(b2 + j) : 0ull;
        if (W) {
          const float w0 = in ? w[group((Idx)(2 * j)) * w_stride] : 1.0f;
          const float w1 = in ? w[group((Idx)(2 * j + 1)) * w_stride] : 1.0f;
          wv[q] = pk2(w0, w1);
        }
      }
#pragma unroll
      for (int q = 0; q < NB; ++q) {
        // w (a - b) as D + E exactly (TwoSum, then the FMA TwoProduct by w)
        uint64_t D = sub2(av[q], bv[q]);
        const uint64_t BV = sub2(D, av[q]);
        const uint64_t AV = sub2(D, BV);
        uint64_t E = sub2(sub2(av[q], AV), add2(bv[q], BV));
        uint64_t Bh = bv[q], Bl = 0;
        if (W) {
          any_d |= bits2(D);
          any_b |= bits2(bv[q]);
          any_w |= bits2(wv[q]);
          const uint64_t P = mul2(D, wv[q]);
          const uint64_t PE = fma2(D, wv[q], P ^ kSign2);
          E = fma2(E, wv[q], PE);
          D = P;
          Bh = mul2(bv[q], wv[q]);
          Bl = fma2(bv[q], wv[q], Bh ^ kSign2);
        }
        float dh0, dh1, bh0, bh1;
        upk2(D, dh0, dh1);
        upk2(Bh, bh0, bh1);
        // PP and QQ go into additions (dadd2), where the assembler could join
        // them (see mul2_rounded) and the sums would be off by 1e-8; it does
        // not here: the same bits as with mul2_rounded, which with weights
        // costs 2 %
        const uint64_t PP = mul2(D, D);
        const uint64_t X = fma2(mul2(D, two), E, fma2(D, D, PP ^ kSign2));
        const uint64_t QQ = mul2(Bh, Bh);
        const uint64_t Y = W ? fma2(mul2(Bh, two), Bl, fma2(Bh, Bh, QQ ^ kSign2)) : fma2(Bh, Bh, QQ ^ kSign2);
        dadd2(EH, EL, PP, X);
        dadd2(BH, BL, QQ, Y);
        bmax = fmaxf(bmax, fmaxf(fabsf(bh0), fabsf(bh1)));
        float dl0, dl1;
        upk2(E, dl0, dl1);
#pragma unroll
        for (int lane = 0; lane < 2; ++lane) {
          const float dh = lane ? dh1 : dh0, dl = lane ? dl1 : dl0;
          const float sh = fabsf(dh);
          if (sh >= mh) {
            const float sl = dh < 0.0f ? -dl : dl;
            if (sh > mh || sl > ml) {
              mh = sh;
              ml = sl;
            }
          }
        }
      }
    }
    const double e_run = lanes_sum(EH, EL, e_rest), b_run = lanes_sum(BH, BL, b_rest);
    if (!W && j0 == start) {   // (2^25 elements 67.1 -> 63.9 us; weighted 87.2 -> 88.4, so not there)
      e2 = e_run;
      b2s = b_run;
    } else {
      e2 += e_run;
      b2s += b_run;
    }
  }
  e2 += (double)e_rest;
  b2s += (double)b_rest;
  double mx = mh < 0.0f ? 0.0 : (double)mh + (double)ml;
  {
    const float pairs = (float)((np - (start < np ? start : np) + stride - 1) / stride);   // this thread's pairs
    const float floor_v = 1.001f * sqrtf(2.0f * pairs) * 0x1p-50f;
    const bool weighed = W && (any_w << 1) != 0;   // a nonzero weight
    const bool slow = !finite64(e2) || !finite64(b2s) ||
                      (mh < floor_v && (mh > 0.0f || (weighed && (any_d << 1) != 0))) ||
                      (bmax < floor_v && (bmax > 0.0f || (weighed && (any_b << 1) != 0)));
    if (slow) {   // the thread's whole share again, in FP64
      e2 = 0.0;
      b2s = 0.0;
      mx = 0.0;
    }
    auto fp64 = [&](Idx i) {
      const float ai = a[i], bi = b[i];
      const double wi = W ? (double)w[group(i) * w_stride] : 1.0;
      const double d = ((double)ai - (double)bi) * wi;
      const double bb = (double)bi * wi;
      e2 += d * d;
      b2s += bb * bb;
      mx = fmax(mx, fabs(d));
    };
    if (slow)
      for (Idx j = start; j < np; j += stride) {
        fp64(2 * j);
        fp64(2 * j + 1);
      }
    if ((n & 1) && blockIdx.x == 0 && threadIdx.x == 0) fp64(n - 1);   // the odd last element
  }
  err_store(e2, b2s, mx, part, out);
}

}  // namespace

cudaError_t launch_material_row_sums(const uint16_t *material, int64_t n, int n_mat, const float *rows, int cols,
                                     float *out, cudaStream_t s) {
  const bool v = (reinterpret_cast<uintptr_t>(material) & 15) == 0;
  const auto k = cols == 128 ? (v ? segment_sums_kernel<true, 4> : segment_sums_kernel<false, 4>)
                             : (v ? segment_sums_kernel<true, 2> : segment_sums_kernel<false, 2>);
  const size_t smem = (size_t)kSegWarps * kSegPerWarp * cols * sizeof(float);
  const cudaError_t e = ensure_max_dyn_smem(reinterpret_cast<const void *>(k), (int)smem);
  if (e != cudaSuccess) return e;
  return launch_dependent(k, n_mat, 32 * kSegWarps, smem, s, material, n, rows, out);
}

namespace {
cudaError_t latent_sums(const fabric_gbuffer &g, int n_lat, const float *rows, float *dlat, bool early, cudaStream_t s) {
  const auto k = (reinterpret_cast<uintptr_t>(g.material) & 15) == 0 ? latent_sums_kernel<true> : latent_sums_kernel<false>;
  return launch_dependent(k, n_lat, 32 * kSegWarps, 0, s, g.material, g.n, rows, dlat, (int)early);
}
}  // namespace

cudaError_t launch_decoder_grad_finish(const fabric_gbuffer &g, int n_lat, const float *partial, int grid, int width,
                                      const double *loss_part, const float *rows, float *ddec, double *loss,
                                      float *dlat, cudaStream_t s) {
  // width > kDecParams: the per-CTA partials already hold the per-material
  // latent-gradient sums after the decoder's columns
  const bool folded = width > kDecParams;
  bool sums = false;   // the sums over the partials were launched
  if (ddec) {
    sums = true;
    const int cols = dlat ? width : kDecParams;
    launch_dependent(reduce_partials_kernel, (cols + 31) / 32 + (loss ? 1 : 0), 32 * kSumSegs, 0, s, partial, grid,
                     width, cols, kDecParams, ddec, dlat, loss_part, loss);
  } else {   // only the latent columns (folded) and the loss
    const int cols = dlat && folded ? width - kDecParams : 0;
    sums = cols > 0 || loss;
    if (sums)
      launch_dependent(reduce_partials_kernel, (cols + 31) / 32 + (loss ? 1 : 0), 32 * kSumSegs, 0, s,
                       partial + kDecParams, grid, width, cols, 0, static_cast<float *>(nullptr), dlat, loss_part,
                       loss);
  }
  if (dlat && !folded) latent_sums(g, n_lat, rows, dlat, sums, s);
  return cudaGetLastError();
}

namespace {
template <typename REC>
cudaError_t encoder_fwd(const float *feats, const fabric_material *raw, float *feats_out, int n, const float *enc,
                        float *z, float *acts, const REC &recs, cudaStream_t s) {
  const int grid = (n + kEncGroup - 1) / kEncGroup;
  const auto k = (reinterpret_cast<uintptr_t>(enc) & 15) == 0 ? encoder_fwd_kernel<true, REC> : encoder_fwd_kernel<false, REC>;
  const cudaError_t e = ensure_max_dyn_smem(reinterpret_cast<const void *>(k), (int)kEncFwdSmem);
  if (e != cudaSuccess) return e;
  return launch_dependent(k, grid, kEncThreads, kEncFwdSmem, s, feats, raw, feats_out, n, enc, z, acts, recs);
}
}  // namespace

bool encoder_takes_inline(int n) { return n <= kInlineRecords; }

cudaError_t launch_encoder_inline(const fabric_material *host, int n, const float *enc, float *z, cudaStream_t s) {
  InlineRecords recs;
  std::memcpy(recs.m, host, (size_t)n * sizeof(fabric_material));
  std::memset(recs.m + n, 0, (size_t)(kInlineRecords - n) * sizeof(fabric_material));
  return encoder_fwd(nullptr, nullptr, nullptr, n, enc, z, nullptr, recs, s);
}

cudaError_t launch_encoder_feats(const float *feats, int n, const float *enc, float *z, float *acts,
                                 cudaStream_t s) {
  return encoder_fwd(feats, nullptr, nullptr, n, enc, z, acts, NoRecords{}, s);
}

cudaError_t launch_encoder_raw(const fabric_material *raw, int n, const float *enc, float *feats_out, float *z,
                               float *acts, cudaStream_t s) {
  return encoder_fwd(nullptr, raw, feats_out, n, enc, z, acts, NoRecords{}, s);
}

size_t encoder_backward_work_floats(int n) { return (size_t)n * 2 * kEncHidden + (size_t)n * 4 * kEncHidden; }

cudaError_t launch_encoder_backward(const float *feats, int n, const float *enc, const float *acts_in,
                                    const float *dz, float *denc, float *work, cudaStream_t s,
                                    const DecAdamArgs *dec_adam) {
  // work: [n][2][128] activations (recomputed when acts_in is null) | [n][4][128]
  float *acts = work;
  float *vec = work + (size_t)n * 2 * kEncHidden;
  if (!acts_in) {
    // recompute the forward pass to obtain the pre-activations (z discarded into vec)
    const cudaError_t e = encoder_fwd(feats, nullptr, nullptr, n, enc, vec, acts, NoRecords{}, s);
    if (e != cudaSuccess) return e;
    acts_in = acts;
  }
  const bool v = (reinterpret_cast<uintptr_t>(enc) & 15) == 0;
  const void *k = v ? reinterpret_cast<const void *>(encoder_bwd_vec_kernel<true>)
                    : reinterpret_cast<const void *>(encoder_bwd_vec_kernel<false>);
  {
    const cudaError_t e = ensure_max_dyn_smem(k, (int)kEncBwdSmem);
    if (e != cudaSuccess) return e;
  }
  const int grid = (n + kEncGroup - 1) / kEncGroup;
  if (v)
    launch_dependent(encoder_bwd_vec_kernel<true>, grid, kEncThreads, kEncBwdSmem, s, enc, n, acts_in, dz, vec);
  else
    launch_dependent(encoder_bwd_vec_kernel<false>, grid, kEncThreads, kEncBwdSmem, s, enc, n, acts_in, dz, vec);
  DecAdamArgs d{};
  int extra = 0;
  if (dec_adam) {
    d = *dec_adam;
    extra = (d.n + 31) / 32;
  }
  launch_dependent(encoder_grad_kernel, kGradTiles + extra, kGradThreads, 0, s, feats, n, dz,
                   (int)((reinterpret_cast<uintptr_t>(dz) & 15) == 0), vec, denc, d);
  return cudaGetLastError();
}

void adam_bias(int64_t step, float *bc1, float *bc2) {
  *bc1 = (float)(1.0 - std::pow(0.9, (double)step));
  *bc2 = (float)(1.0 - std::pow(0.999, (double)step));
}

cudaError_t launch_adam(float *p0, int64_t n0, float *p1, int64_t n1, const float *grad, float *m, float *v, float lr,
                        int64_t step, cudaStream_t s) {
  float bc1, bc2;
  adam_bias(step, &bc1, &bc2);
  launch_dependent(adam_kernel, (unsigned)((n0 + n1 + 255) / 256), 256, 0, s, p0, n0, p1, n1, grad, m, v, lr, bc1, bc2);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Dataset shuffle: a pseudo-random permutation of [0, n) from a four-round
// Feistel network on [0, 4^k) (balanced halves of k bits, 4^k >= n) with
// the SplitMix64 finaliser of (seed, round, half) as round function; values
// at or past n are walked along their cycle (the network is a bijection of
// [0, 4^k), so the walk returns to [0, n)).
// ---------------------------------------------------------------------------
namespace {
__device__ __forceinline__ uint64_t shuffle_mix(uint64_t z) {
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

__device__ __forceinline__ uint64_t feistel(uint64_t x, int k, uint64_t seed) {
  const uint64_t mask = (1ull << k) - 1ull;
  uint64_t l = x >> k, r = x & mask;
#pragma unroll
  for (int round = 0; round < 4; ++round) {
    const uint64_t f = shuffle_mix(seed + 0x9E3779B97F4A7C15ull * (uint64_t)(round + 1) + r) & mask;
    const uint64_t t = l ^ f;
    l = r;
    r = t;
  }
  return (l << k) | r;
}

__global__ void shuffle_dataset_kernel(const fabric_train_batch src, const fabric_dataset_out dst, int k,
                                       uint64_t seed) {
  const int64_t n = src.queries.n;
  for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < n; p += (int64_t)gridDim.x * blockDim.x) {
    uint64_t j = feistel((uint64_t)p, k, seed);
    while (j >= (uint64_t)n) j = feistel(j, k, seed);
    const fabric_gbuffer &g = src.queries;
    dst.u[p] = g.u[j];
    dst.v[p] = g.v[j];
    dst.radius[p] = g.radius[j];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      dst.wi[3 * p + c] = g.wi[3 * j + c];
      dst.wo[3 * p + c] = g.wo[3 * j + c];
    }
    dst.material[p] = g.material[j];
    if (dst.target) {
#pragma unroll
      for (int c = 0; c < 4; ++c) dst.target[4 * p + c] = src.target[4 * j + c];
    }
  }
}
}  // namespace

cudaError_t launch_shuffle_dataset(const fabric_train_batch &src, const fabric_dataset_out &dst, uint64_t seed,
                                   int sm_count, cudaStream_t s) {
  const int64_t n = src.queries.n;
  int k = 1;
  while ((1ll << (2 * k)) < n) ++k;
  const int64_t blocks = std::min<int64_t>((n + 255) / 256, (int64_t)(sm_count > 0 ? sm_count : 148) * 8);
  shuffle_dataset_kernel<<<(unsigned)blocks, 256, 0, s>>>(src, dst, k, seed);
  return cudaGetLastError();
}

// [blocks][3] partials
size_t error_stats_work_bytes(int64_t) { return (size_t)kErrBlocks * 3 * sizeof(double); }

cudaError_t launch_error_stats(const float *a, const float *b, int64_t n, const float *w, int group, int w_stride,
                               double *out, void *work, cudaStream_t s) {
  double *part = static_cast<double *>(work);
  const bool small = n + (int64_t)kErrRun * kErrBlocks * kErrThreads < ((int64_t)1 << 31);
  const bool packed = ((reinterpret_cast<uintptr_t>(a) | reinterpret_cast<uintptr_t>(b)) & 7u) == 0;
  const auto kernel = packed ? (w ? (small ? err_partial2_kernel<true, int> : err_partial2_kernel<true, int64_t>)
                                  : (small ? err_partial2_kernel<false, int> : err_partial2_kernel<false, int64_t>))
                             : (w ? (small ? err_partial_kernel<true, int> : err_partial_kernel<true, int64_t>)
                                  : (small ? err_partial_kernel<false, int> : err_partial_kernel<false, int64_t>));
  // one wave of CTAs, or as many as give each thread an element or pair (two
  // are added in double-float, one not at all: 50 001 elements with two 3.6e-16
  // off the exact sum, so 1.1e-16; 300 000 10.3 us, so 14.4)
  const int64_t items = packed ? n / 2 : n, wave = packed ? kErrBlocks2 : kErrBlocks;
  const int blocks = (int)std::max<int64_t>(1, std::min<int64_t>(wave, (items + kErrThreads - 1) / kErrThreads));
  kernel<<<blocks, kErrThreads, 0, s>>>(a, b, n, w, group_div(group), w_stride, part, out);
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess || blocks == 1) return e;
  return launch_dependent(err_final_kernel, dim3(1), kErrThreads, 0, s, static_cast<const double *>(part), blocks, out);
}

}  // namespace fab
