// reference.cu -- supersampled footprint integral of the woven-fabric shading
// model (the plain method): Eq. 3-5 estimated with spp_x * spp_y stratified
// samples per shading point, shaded with Eq. 1-2, split into the components
// of Eq. 7 and recombined by Eq. 8.
//
// Work mapping: L lanes (L = 1..32, a power of two) share one shading point;
// each lane takes samples lane, lane + L, ... and the five running sums are
// combined with warp shuffles.  The kernel is bound by the issue slots (83 %
// busy; no pipe above 53 %), so its design is about instructions: 181 for
// each sample of a warp at 256 spp, where the first form took 275 (1080p
// frame 4.42 -> 2.94 ms).  Every discrete decision (cell, gap, visible
// yarn) is taken in 0.32 fixed-point integers from a SplitMix64 jitter
// (Steele, Lea and Flood 2014) so that it is exactly reproducible; the
// shading itself runs in FP32.
#include <algorithm>

#include "f32x2.h"
#include "fabric_internal.h"

namespace fab {
namespace {

constexpr float kPi = 3.14159265358979323846f;
constexpr float kHalfPiRest = (float)(1.57079632679489661923 - (double)(0.5f * kPi));   // pi / 2 past its FP32 value
constexpr float kTwoNeg32 = 2.3283064365386963e-10f;   // 2^-32

__device__ __forceinline__ uint64_t splitmix_finalise(uint64_t z) {
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

// Footprint centre in 0.32 fixed-point pattern coordinates (mod one repeat).
__device__ __forceinline__ uint32_t centre_fixed(float u) {
  const float f = __fsub_rn(u, floorf(u));
  return (uint32_t)(unsigned long long)__float2ll_rn(__fmul_rn(f, 4294967296.0f));
}

// Footprints below this half side keep every offset's 0.32 value within 32
// signed bits.
constexpr float kSmallRadius = 0.45f;

// sin and cos for |x| <= pi/2 from their Maclaurin series up to x^11 and
// x^12 (truncation below 6e-8 and 7e-9 there), Horner form with FMA.  The
// frame's angles (pi x / 2 across a yarn, theta along a float) stay in that
// range; the series keep the normal's error near one FP32 rounding, where the
// fast intrinsics' absolute error (about 4e-7) reached 2e-4 relative in the
// components of rays grazing the yarns.
__device__ __forceinline__ float sin_half_pi(float x) {
  const float x2 = x * x;
  float p = -2.505210838544172e-08f;     // -1/11!
  p = fmaf(p, x2, 2.7557319223985893e-06f);
  p = fmaf(p, x2, -1.984126984126984e-04f);
  p = fmaf(p, x2, 8.333333333333333e-03f);
  p = fmaf(p, x2, -1.6666666666666666e-01f);
  return fmaf(p * x2, x, x);
}
__device__ __forceinline__ float cos_half_pi(float x) {
  const float x2 = x * x;
  float p = 2.08767569878681e-09f;       // 1/12!
  p = fmaf(p, x2, -2.755731922398589e-07f);
  p = fmaf(p, x2, 2.48015873015873e-05f);
  p = fmaf(p, x2, -1.388888888888889e-03f);
  p = fmaf(p, x2, 4.1666666666666664e-02f);
  p = fmaf(p, x2, -0.5f);
  return fmaf(p, x2, 1.0f);
}
// Both of one angle: the two series side by side in the packed lanes.
__device__ __forceinline__ void sincos_half_pi(float x, float &sn, float &cs) {
  const float x2 = x * x;
  const uint64_t xx = pk2(x2, x2);
  uint64_t p = pk2(-2.505210838544172e-08f, fmaf(2.08767569878681e-09f, x2, -2.755731922398589e-07f));
  p = fma2(p, xx, pk2(2.7557319223985893e-06f, 2.48015873015873e-05f));
  p = fma2(p, xx, pk2(-1.984126984126984e-04f, -1.388888888888889e-03f));
  p = fma2(p, xx, pk2(8.333333333333333e-03f, 4.1666666666666664e-02f));
  p = fma2(p, xx, pk2(-1.6666666666666666e-01f, -0.5f));
  float ps, pc;
  upk2(p, ps, pc);
  sn = fmaf(ps * x2, x, x);
  cs = fmaf(pc, x2, 1.0f);
}

// One hardware operation each (relative error about 2^-23), without the
// range checks and fix-up branches of the IEEE forms.  What is the same in all
// samples of a point does not average out and is kept exact instead: the
// factor of the position across a yarn carries its remainder, and w / (pi wi.z)
// the remainder of pi.  The diffuse components of a 256 spp frame lie 6.2e-8
// (median) and 6.4e-7 (99 %) off FP64 so, in relative L2 8.6e-8; without the
// two remainders 7.6e-8, 9.8e-7 and 1.18e-7; with IEEE operations throughout
// and no remainders 7.3e-8, 8.3e-7 and 1.16e-7, for 2.94, 2.91 and 4.42 ms.
// IEEE divisions, square roots or expm1 in addition change none of these
// figures and take 6 % each; a Newton step on 1 / |N| 2 % for 5.9e-8.
__device__ __forceinline__ float rsqrt_hw(float x) {
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ float sqrt_hw(float x) {
  float r;
  asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ float lg2_hw(float x) {
  float r;
  asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ float cos_hw(float x) {
  float r;
  asm("cos.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ float ex2_hw(float x) {
  float r;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ float rcp_hw(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

// What every sample of one shading point reads.
struct PointMaterial {
  const DevMaterial *m;
  uint32_t rows, cols, gap, gap_span;   // gap_span: 2^32 - 1 - 2 gap, the body's extent past the gap
  float inv_1mg, cos_psi, sin_psi;
  float one_mg;                         // 1 - gap: the body's half width in cell units of [-1, 1]
  float across_off, across_lo;          // pi / (2 (1 - gap)), and what its rounding leaves
  float across_mul;                     // the march's pi x / 2 = across_mul * (0.32 fixed point) - across_off
};

struct PointDirs {
  float3 wi, wo;
  float h_inv;       // 1 / |wi + wo|, or 0 when wi + wo = 0 (no half vector, no specular term)
  float diff_k, diff_c;
};

struct Sums {
  float c0, c1, s0, s1, a;
};

// ---- the proposed inter-yarn visibility model (V of Eq. 3-5).  The surface
// is the height field whose slopes the frame below uses, in repeat units:
// on a top yarn's body beta w cos(pi x / 2) plus the float's rise (the
// integral of tan(theta) along it); under a gap the under-yarn, level, one
// cross-section height below the top yarns' edges, beta' w' (cos(pi x'/2) - 1).
// V(x_p, w) = 1 when a march from (p, H(p)) along w, with horizontal steps
// of 1 / (16 max(rows, cols)) repeats, stays above H until the ray rises
// above the material's largest height (at most 4096 steps); 0 otherwise and
// below the horizon.  Steps are integer multiples of one 0.32 fixed-point
// increment per ray.
constexpr int kVisMaxSteps = 4096;

// The cell that holds (pu, pv) and the local coordinates inside it.
struct CellHit {
  WeaveCell c;
  bool warp_top, body;
  uint32_t s_top, s_along;   // across the yarn on top, and along it
};
__device__ __forceinline__ CellHit locate(const PointMaterial &pm, uint32_t pu, uint32_t pv) {
  const uint32_t j = __umulhi(pu, pm.cols), su = pu * pm.cols;
  const uint32_t i = __umulhi(pv, pm.rows), sv = pv * pm.rows;
  const float4 q = __ldg(reinterpret_cast<const float4 *>(pm.m->cell) + (i * pm.cols + j));
  CellHit h;
  h.c.theta0 = q.x;
  h.c.theta1 = q.y;
  h.c.top_bound = q.z;
  h.c.rise = q.w;
  h.warp_top = __float_as_int(q.z) < 0;
  h.s_top = h.warp_top ? su : sv;
  h.s_along = h.warp_top ? sv : su;
  h.body = h.s_top - pm.gap <= pm.gap_span;   // gap <= s_top <= 2^32 - 1 - gap
  return h;
}

__device__ __forceinline__ float surface_height(const PointMaterial &pm, uint32_t pu, uint32_t pv) {
  const CellHit q = locate(pm, pu, pv);
  if (q.body) {
    const float s = (float)q.s_top * kTwoNeg32;
    const float x = (2.0f * s - 1.0f) * pm.inv_1mg;
    float h = __ldg(&pm.m->crest[q.warp_top ? 0 : 1]) * cosf(x * (0.5f * kPi));
    if (q.c.rise != 0.0f) {
      h += q.c.rise * (logf(cosf(q.c.theta0 - q.c.theta1 * (float)q.s_along)) - __ldg(&pm.m->lncos_incl));
    }
    return h;
  }
  const float s2 = (float)q.s_along * kTwoNeg32;
  const float x = fminf(1.0f, fmaxf(-1.0f, (2.0f * s2 - 1.0f) * pm.inv_1mg));
  return __ldg(&pm.m->crest[q.warp_top ? 1 : 0]) * (cosf(x * (0.5f * kPi)) - 1.0f);
}

// One direction's march, prepared once per point.  steps: -1 at or below the
// horizon (never visible), 0 straight up (always visible), else 1.
struct alignas(16) MarchDir {
  uint32_t inc_u, inc_v;         // position increments, 0.32 fixed point
  float dz;                      // height gained per step
  float cell_u, cell_v;          // just under 1 / (local cell coordinate per step), for skipping
  int steps;
  int pad[2];
};

__device__ __forceinline__ MarchDir march_dir(const DevMaterial *__restrict__ m, float3 w) {
  MarchDir d = {};
  d.steps = -1;
  if (!(w.z > 0.0f)) return d;
  const float rho2 = w.x * w.x + w.y * w.y;
  d.steps = 0;
  if (rho2 == 0.0f) return d;
  d.steps = 1;
  const float rho = sqrtf(rho2);
  const float delta = m->v_delta;
  d.inc_u = (uint32_t)(unsigned long long)__float2ll_rn(w.x / rho * delta * 4294967296.0f);
  d.inc_v = (uint32_t)(unsigned long long)__float2ll_rn(w.y / rho * delta * 4294967296.0f);
  d.dz = delta * (w.z / rho);
  // |increment| * cells <= 2^28, since delta is a sixteenth of the finer cell
  const int du = abs((int)(d.inc_u * m->cols)), dv = abs((int)(d.inc_v * m->rows));
  d.cell_u = du ? 0.999999f / (float)du : 3.0e38f;
  d.cell_v = dv ? 0.999999f / (float)dv : 3.0e38f;
  return d;
}

// The state of a march between its steps.
struct March {
  uint32_t qu, qv;               // position of the last step
  int k, K;                      // steps taken, and in all
  float h0;
  MarchDir d;
};

__device__ __forceinline__ void march_start(March &r, const DevMaterial *__restrict__ m, const MarchDir &d, uint32_t pu,
                                            uint32_t pv, float h0) {
  r.qu = pu;
  r.qv = pv;
  r.k = 0;
  r.h0 = h0;
  r.d = d;
  const float span = (__ldg(&m->h_max) - h0) / d.dz;
  int K = span < (float)kVisMaxSteps ? (int)floorf(span) + 1 : kVisMaxSteps;
  if (K < 1) K = 1;
  r.K = d.steps > 0 ? K : 0;
}

// One step of a march (k < K), or several that cannot meet the surface; true
// when the surface is above the ray there.  The decision at a step is that of
// surface_height(q) > h0 + k dz, reached in most cases without it:
//  - Over a cell the height is at most top_bound - crest xn^2 (xn in [-1, 1]
//    across the yarn on top; cos(pi xn / 2) <= 1 - xn^2) and at most 0 in the
//    gaps beyond |xn| = 1.  A ray at z >= 0 outside the band |xn| <
//    sqrt((top_bound - z) / crest) cannot be below the surface until it
//    enters the band, which it can only leave narrower since z rises: all
//    steps up to there, or to the cell's edge, are skipped at once.
//  - Inside, the height from the hardware cosine and logarithm decides, unless
//    the ray is within v_margin of it, a bound on its error that the host
//    computes per material; only there is surface_height evaluated.
__device__ __forceinline__ bool march_step(March &r, const PointMaterial &pm) {
  r.qu += r.d.inc_u;
  r.qv += r.d.inc_v;
  ++r.k;
  const float z = fmaf((float)r.k, r.d.dz, r.h0);
  const uint32_t j = __umulhi(r.qu, pm.cols), su = r.qu * pm.cols;
  const uint32_t i = __umulhi(r.qv, pm.rows), sv = r.qv * pm.rows;
  const float4 c = __ldg(reinterpret_cast<const float4 *>(pm.m->cell) + (i * pm.cols + j));
  const float2 crest = __ldg(reinterpret_cast<const float2 *>(pm.m->crest));
  const bool warp_top = __float_as_int(c.z) < 0;
  const uint32_t s_top = warp_top ? su : sv, s_along = warp_top ? sv : su;
  const float above = fabsf(c.z) - z, crest_top = warp_top ? crest.x : crest.y;
  const float xs = fmaf((float)s_top, 2.0f * kTwoNeg32, -1.0f);   // [-1, 1] across the cell
  // half width of the band in xs, enlarged past the rounding here
  const float band = above > 0.0f
                         ? fmaf(sqrt_hw(fminf(1.0f, above * rcp_hw(crest_top))), 1.0001f * pm.one_mg, 1e-5f)
                         : -1.0f;
  if (z >= 0.0f && fabsf(xs) > band) {
    const int inc_top = (int)(warp_top ? r.d.inc_u : r.d.inc_v), inc_along = (int)(warp_top ? r.d.inc_v : r.d.inc_u);
    // 0.32 distances to go: to the band when moving towards it, else to the cell's edge; and to the edge along the yarn
    const bool towards = band >= 0.0f && (xs > 0.0f) == (inc_top < 0);
    const float to_edge = (float)(inc_top < 0 ? s_top : ~s_top);
    const float go_top = towards ? (fabsf(xs) - band) * 2147483648.0f : to_edge;
    const float go_along = (float)(inc_along < 0 ? s_along : ~s_along);
    const int n = min(min(__float2int_rz(go_top * (warp_top ? r.d.cell_u : r.d.cell_v)),
                          __float2int_rz(go_along * (warp_top ? r.d.cell_v : r.d.cell_u))), r.K - r.k);
    r.qu += (uint32_t)n * r.d.inc_u;
    r.qv += (uint32_t)n * r.d.inc_v;
    r.k += n;
    return false;
  }
  const bool body = s_top - pm.gap <= pm.gap_span;
  if (!body && z >= 0.0f) return false;
  const float xh = fminf(0.5f * kPi, fmaxf(-0.5f * kPi, fmaf((float)(body ? s_top : s_along), pm.across_mul, -pm.across_off)));
  float h = cos_half_pi(xh);
  if (body) {
    h = fmaf(c.w, fmaf(lg2_hw(cos_hw(fmaf(-c.y, (float)s_along, c.x))), 0.6931471805599453f, -__ldg(&pm.m->lncos_incl)),
             h * crest_top);
  } else {
    h = (h - 1.0f) * (warp_top ? crest.y : crest.x);
  }
  const float d = h - z;
  if (fabsf(d) > __ldg(&pm.m->v_margin)) return d > 0.0f;
  return surface_height(pm, r.qu, r.qv) > z;
}

// The integrand of Eq. 3-5 at one sample.  With hc the height profile's
// slope, a / c the directions along / across the visible yarn and N = -hc
// cos(theta) c - sin(theta) a + cos(theta) z the unnormalised ply normal
// (|N|^2 = 1 + (hc cos theta)^2 = 1 / inv^2), a direction w enters through
//   N.w,   t0.w = cos(theta) w_a + sin(theta) w_z,
//   t_p.w = cos(psi) t0.w -+ sin(psi) inv (w_c + hc cos(theta) (cos(theta) w_z - sin(theta) w_a)),
// and the half vector mostly needs
// none of its own, t_p.h = (t_p.wi + t_p.wo) / |wi + wo|.  1 / inv cancels out of
// A = <wo.n_p> / <n_s.n_p> = N.wo / cos(theta) and, with X' = sigma_i N.wo +
// sigma_o N.wi, out of the specular term
//   D (1 - exp(-2 (L_i + L_o))) (N.wi N.wo / X') / (4 cos theta),
//   L_i + L_o = X' / (inv N.wi N.wo).
struct Shaded {
  float coJ, diff, spec;   // A's term, diffuse and specular numerators
  bool weft, ci_pos;
};
template <bool OPPOSITE>
__device__ __forceinline__ Shaded shade(const PointMaterial &pm, const PointDirs &d, uint32_t pu, uint32_t pv) {
  const CellHit q = locate(pm, pu, pv);
  Shaded r;
  r.weft = q.warp_top != q.body;   // in the gap of the top yarn the yarn underneath shows
  const float4 yc = __ldg(reinterpret_cast<const float4 *>(pm.m->yarn) + (r.weft ? 1 : 0));
  // pi x / 2 across the visible yarn (the clamp acts in gaps only); the
  // inclination along the float of a yarn on top, level in a gap
  const float xs = fmaf((float)(q.body ? q.s_top : q.s_along), 2.0f * kTwoNeg32, -1.0f);
  const float xh = fminf(0.5f * kPi, fmaxf(-0.5f * kPi, fmaf(xs, pm.across_off, xs * pm.across_lo)));
  float st, ct;
  sincos_half_pi(fmaf(-q.c.theta1, (float)q.s_along, q.c.theta0), st, ct);
  st = q.body ? st : 0.0f;
  ct = q.body ? ct : 1.0f;
  const float hct = yc.x * sin_half_pi(xh) * ct;   // hc cos(theta)
  const float n2 = fmaf(hct, hct, 1.0f);
  const float inv = rsqrt_hw(n2);
  const float ia = r.weft ? d.wi.x : d.wi.y, ic = r.weft ? d.wi.y : d.wi.x;
  const float oa = r.weft ? d.wo.x : d.wo.y, oc = r.weft ? d.wo.y : d.wo.x;
  const float Bi = fmaf(ct, d.wi.z, -st * ia), Bo = fmaf(ct, d.wo.z, -st * oa);   // cos(theta) w_z - sin(theta) w_a
  const float ni = fmaxf(0.0f, fmaf(-hct, ic, Bi)), no = fmaxf(0.0f, fmaf(-hct, oc, Bo));
  float rct = rcp_hw(ct);                                 // one Newton step: within an ulp of 1 / cos(theta)
  rct = fmaf(rct, fmaf(-ct, rct, 1.0f), rct);
  const float ci = ni * inv;
  r.coJ = no * rct;
  r.ci_pos = ci > 0.0f;
  r.diff = fmaf(d.diff_k, ci, d.diff_c) * ci * r.coJ;
  r.spec = 0.0f;
  const float cc = ni * no;
  if (cc > 0.0f && d.h_inv > 0.0f) {   // where the product vanishes in FP32, so does the term (and 1 / X may overflow)
    const float sp = (r.weft ? pm.sin_psi : -pm.sin_psi) * inv;
    const float ti = fmaf(sp, fmaf(hct, Bi, ic), pm.cos_psi * fmaf(ct, ia, st * d.wi.z));
    const float to = fmaf(sp, fmaf(hct, Bo, oc), pm.cos_psi * fmaf(ct, oa, st * d.wo.z));
    float tau = (ti + to) * d.h_inv;
    if (OPPOSITE && d.h_inv > 1.0f) {   // nearly opposite directions: the sum would lose what 1 / |wi + wo| magnifies
      const float hx = (d.wi.x + d.wo.x) * d.h_inv, hy = (d.wi.y + d.wo.y) * d.h_inv, hz = (d.wi.z + d.wo.z) * d.h_inv;
      const float ha = r.weft ? hx : hy, hcr = r.weft ? hy : hx;
      tau = fmaf(sp, fmaf(hct, fmaf(ct, hz, -st * ha), hcr), pm.cos_psi * fmaf(ct, ha, st * hz));
    }
    const float qd = fmaf(tau * tau, yc.y, 1.0f);         // D = 1 / (pi alpha q^2)
    const float si = sqrt_hw(fmaxf(0.0f, fmaf(-yc.z * ti, ti, 1.0f)));
    const float so = sqrt_hw(fmaxf(0.0f, fmaf(-yc.z * to, to, 1.0f)));
    const float X = fmaf(si, no, so * ni);
    // Eq. 2 with T rho = 2: 1 - exp(-y).  Above y = 1 the hardware exp2's
    // error is below an ulp of the difference; below, expm1 keeps its digits
    const float y = X * rcp_hw(cc) * (2.0f * (n2 * inv));
    const float E = y > 1.0f ? 1.0f - ex2_hw(-1.4426950408889634f * y) : -expm1f(-y);
    r.spec = (yc.w * rct) * (cc * E) * rcp_hw(qd * qd * X);
  }
  return r;
}

__device__ __forceinline__ void accumulate(const Shaded &r, Sums &acc) {
  if (!r.weft) {
    acc.c0 += r.diff;
    acc.s0 += r.spec;
  } else {
    acc.c1 += r.diff;
    acc.s1 += r.spec;
  }
}

struct RefArgs {
  const float *u, *v, *radius, *wi, *wo;
  const uint16_t *material;
  int64_t n;
  const DevMaterial *mats;
  int n_mat;
  int nx, ny;
  int rounds;          // points per group of L lanes
  int split;           // visibility, L = 32: warps of a CTA that share each point
  float two_over_nx, two_over_ny;
  uint64_t seed;
  float *rgb, *comps;
  int *status;
};

constexpr int kRefThreads = 256;
constexpr int kRefWarps = kRefThreads / 32;

// What the samples of one point share, prepared by one lane and read by all
// lanes of the point's group (16-byte loads).
struct alignas(16) PointRecord {
  uint64_t hash;                 // per-point jitter stream
  uint32_t cu, cv;               // footprint centre, 0.32 fixed point
  float wi_x, wo_x, wi_y, wo_y;
  float wi_z, wo_z, h_inv, diff_k;
  float diff_c, r;
  int mat;                       // -1: no such point, or a bad material index
  int pad;
};
static_assert(sizeof(PointRecord) == 64, "four 16-byte loads");

__device__ __forceinline__ PointRecord load_point(const RefArgs &a, int64_t p) {
  PointRecord R;
  R.mat = a.material[p];
  if (R.mat >= a.n_mat) {
    atomicOr(a.status, kStatusBadMaterial);
    R.mat = -1;
    return R;
  }
  const float u = a.u[p], v = a.v[p], r = a.radius[p];
  const float3 wi = make_float3(a.wi[3 * p], a.wi[3 * p + 1], a.wi[3 * p + 2]);
  const float3 wo = make_float3(a.wo[3 * p], a.wo[3 * p + 1], a.wo[3 * p + 2]);
  const float w = a.mats[R.mat].w_blend;
  R.wi_x = wi.x;
  R.wi_y = wi.y;
  R.wi_z = wi.z;
  R.wo_x = wo.x;
  R.wo_y = wo.y;
  R.wo_z = wo.z;
  const float3 h = make_float3(wi.x + wo.x, wi.y + wo.y, wi.z + wo.z);
  const float hn2 = h.x * h.x + h.y * h.y + h.z * h.z;
  R.h_inv = hn2 > 0.0f ? rsqrtf(hn2) : 0.0f;
  // w / (pi wi.z) to the last bit: pi's FP32 value is 2.8e-8 too large, and
  // this factor is in all samples of the brightest points
  const float z = fmaxf(wi.z, 1e-3f), den = kPi * z, rest = fmaf(kPi, z, -den) + 2.0f * kHalfPiRest * z;
  const float k = w / den;
  R.diff_k = k + (fmaf(-k, den, w) - k * rest) / den;
  R.diff_c = (1.0f - w) / kPi;
  R.cu = centre_fixed(u);
  R.cv = centre_fixed(v);
  R.hash = splitmix_finalise(a.seed + 0x9E3779B97F4A7C15ull * (uint64_t)(p + 1));
  R.r = r;
  R.pad = 0;
  return R;
}

// Stratum (ix, iy) of sample k = iy nx + ix as a packed pair of floats (both
// below 2^13, exact), stepped by the group's `stride` samples at a time.
struct SamplePlan {
  int spp, stride;
  uint64_t first, step, wrap, two_over_n;
  float nx;
};

// One point as its samples read it, and lane lane_g's place in its sequence.
// WIDE: footprints of any size (64-bit conversions).
template <bool WIDE>
struct PointSampler {
  PointMaterial pm;
  PointDirs d;
  uint64_t hp, rr, strat;
  uint32_t cu, cv;
  int k;

  __device__ __forceinline__ PointSampler(const RefArgs &a, const PointRecord &R, const SamplePlan &sp, int first) {
    pm.m = a.mats + max(R.mat, 0);
    const uint4 m0 = __ldg(reinterpret_cast<const uint4 *>(pm.m));
    const float4 m1 = __ldg(reinterpret_cast<const float4 *>(pm.m) + 1);
    pm.rows = m0.x;
    pm.cols = m0.y;
    pm.gap = m0.z;
    pm.gap_span = 0xFFFFFFFFu - 2u * pm.gap;
    pm.inv_1mg = m1.x;
    pm.cos_psi = m1.y;
    pm.sin_psi = m1.z;
    pm.one_mg = 1.0f / m1.x;
    pm.across_off = 0.5f * kPi * m1.x;
    pm.across_lo = fmaf(0.5f * kPi, m1.x, -pm.across_off) + kHalfPiRest * m1.x;
    pm.across_mul = pm.across_off * (2.0f * kTwoNeg32);
    d.wi = make_float3(R.wi_x, R.wi_y, R.wi_z);
    d.wo = make_float3(R.wo_x, R.wo_y, R.wo_z);
    d.h_inv = R.h_inv;
    d.diff_k = R.diff_k;
    d.diff_c = R.diff_c;
    hp = R.hash;
    const float r32 = WIDE ? R.r : R.r * 4294967296.0f;   // a power of two: exact
    rr = pk2(r32, r32);
    cu = R.cu;
    cv = R.cv;
    strat = sp.first;
    k = first;
  }

  // The position of sample k; moves on to sample k + stride.
  __device__ __forceinline__ void next(const SamplePlan &sp, uint32_t &pu, uint32_t &pv) {
    const uint64_t hk = splitmix_finalise(hp + (uint64_t)k);
    // ((k + xi) (2/n) - 1) r, rounded at every step as the oracle rounds it
    // (xi has 24 bits, so the product of the fma is exact; the first product
    // has to be kept from joining the subtraction, which moved the samples
    // wherever 2/n is no power of two)
    const uint64_t xi = pk2((float)(uint32_t)(hk >> 40), (float)(uint32_t)((hk >> 16) & 0xFFFFFFu));
    const uint64_t minus1 = pk2(-1.0f, -1.0f), xi_scale = pk2(5.9604644775390625e-08f, 5.9604644775390625e-08f);   // 2^-24
    const uint64_t t = mul2(add2(mul2_rounded(fma2(xi, xi_scale, strat), sp.two_over_n), minus1), rr);
    float ou, ov;
    upk2(t, ou, ov);
    if (WIDE) {
      pu = cu + (uint32_t)(unsigned long long)__float2ll_rn(__fmul_rn(ou, 4294967296.0f));
      pv = cv + (uint32_t)(unsigned long long)__float2ll_rn(__fmul_rn(ov, 4294967296.0f));
    } else {   // rr carries the 2^32, |offset| < 2^31: one 32-bit conversion
      pu = cu + (uint32_t)__float2int_rn(ou);
      pv = cv + (uint32_t)__float2int_rn(ov);
    }
    strat = add2(strat, sp.step);
    float ix, iy;
    upk2(strat, ix, iy);
    if (ix >= sp.nx) strat = add2(strat, sp.wrap);
    k += sp.stride;
  }
};

// Lane lane_g's samples of one point, V = 1.  OPPOSITE: directions that may
// be nearly opposite.  A lane alone with its point adds its samples in blocks,
// so that its sums round no more often than those of several lanes do.
constexpr int kLaneBlock = 4;
template <bool WIDE, bool OPPOSITE, int L>
__device__ __forceinline__ void integrate(const RefArgs &a, const PointRecord &R, const SamplePlan &sp, int lane_g,
                                          Sums &acc) {
  PointSampler<WIDE> s(a, R, sp, lane_g);
  auto add_samples = [&](int end, Sums &t) {
    do {
      uint32_t pu, pv;
      s.next(sp, pu, pv);
      const Shaded r = shade<OPPOSITE>(s.pm, s.d, pu, pv);
      t.a += r.coJ;                                    // A of Eq. 4
      accumulate(r, t);
    } while (s.k < end);
  };
  if (L == 1) {
    while (s.k < sp.spp) {
      Sums t = {0.f, 0.f, 0.f, 0.f, 0.f};
      add_samples(min(sp.spp, s.k + kLaneBlock), t);
      acc.c0 += t.c0;
      acc.c1 += t.c1;
      acc.s0 += t.s0;
      acc.s1 += t.s1;
      acc.a += t.a;
    }
  } else if (s.k < sp.spp) {
    add_samples(sp.spp, acc);
  }
}

// The same with the visibility model: V(x_p, wo) weighs A and the numerators,
// V(x_p, wi) the numerators (and is not marched with <wi.n_p> = 0).  Marches
// differ in length from lane to lane, from one step to hundreds, so the
// lanes are not kept in step: each takes its samples in order on its own.
// While most lanes are marching the warp steps their marches; when kRefill of
// them have none, those shade their next sample first.  Each lane's sums run
// in sample order whatever the others do.  1080p frame at 256 spp: 59.8 ms
// with the lanes in step and every height evaluated; with this loop and
// march_step's skipping 25.6 ms at kRefill = 8 and three CTAs per SM, 21.8 ms
// at 20 and four (starting the second march only together with the next
// samples: 23.6 ms).
constexpr int kRefill = 20;

__device__ __forceinline__ void integrate_visible(const RefArgs &a, const PointRecord &R, const MarchDir &to_i,
                                                  const MarchDir &to_o, const SamplePlan &sp, int first, Sums &acc) {
  PointSampler<true> s(a, R, sp, first);
  const int spp = R.mat >= 0 && to_o.steps >= 0 ? sp.spp : 0;   // wo below the horizon: every term is zero
  Shaded r = {};
  March m = {};
  uint32_t pu = 0, pv = 0;
  bool marching = false, on_wi = false;
  for (;;) {
    if (!marching && s.k < spp) {
      s.next(sp, pu, pv);
      r = shade<true>(s.pm, s.d, pu, pv);
      if (r.coJ > 0.0f) {
        march_start(m, s.pm.m, to_o, pu, pv, surface_height(s.pm, pu, pv));
        marching = true;
        on_wi = false;
      }
    }
    const unsigned busy = __ballot_sync(0xFFFFFFFFu, marching), left = __ballot_sync(0xFFFFFFFFu, s.k < spp);
    if (!(busy | left)) break;
    const int enough = min(kRefill, __popc(left));
    for (;;) {
      if (marching) {
        if (m.k < m.K && march_step(m, s.pm)) {
          marching = false;                             // hidden
        } else if (m.k >= m.K) {                        // above the surface all the way
          marching = false;
          if (!on_wi) {
            acc.a += r.coJ;                             // A of Eq. 4
            if (!r.ci_pos) {
              accumulate(r, acc);
            } else if (to_i.steps >= 0) {
              march_start(m, s.pm.m, to_i, pu, pv, m.h0);
              marching = on_wi = true;
            }
          } else {
            accumulate(r, acc);
          }
        }
      }
      const unsigned now = __ballot_sync(0xFFFFFFFFu, marching);
      if (now == 0 || (left && __popc(left & ~now) >= enough)) break;
    }
  }
}

// A warp owns 32/L * rounds consecutive points.  Its lanes first prepare one
// point each (G-buffer loads, jitter stream, half vector: about 300
// instructions that a group of L lanes would otherwise all repeat for every
// point, 37 a sample at 256 samples on 32 lanes), then each group of L lanes
// integrates its points one after the other, and at the end the lanes again
// take one point each to divide, recombine and store.
// Four CTAs per SM (64 registers): the V = 1 kernel needs no more, and with
// the visibility model the extra warps on the divergent marches outweigh a
// few spilled registers.
template <int L, bool VIS>
__global__ void __launch_bounds__(kRefThreads, 4) reference_kernel(const RefArgs a) {
  constexpr int G = 32 / L;
  // a lane that integrates its own point keeps everything in registers
  constexpr bool kStaged = L > 1;
  __shared__ PointRecord recs[kStaged ? kRefWarps : 1][kStaged ? 32 : 1];
  __shared__ MarchDir dirs[2][VIS && kStaged ? kRefWarps : 1][VIS && kStaged ? 32 : 1];
  __shared__ float sums[kStaged ? kRefWarps : 1][5][kStaged ? 32 : 1];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int lane_g = lane & (L - 1), group = lane / L;
  const int n_pts = G * a.rounds;
  // warps part, part + 1, ... of `split` share their points, each taking every split-th 32 samples
  const int split = VIS && L == 32 ? a.split : 1, part = warp % split;
  const int64_t p0 = ((int64_t)blockIdx.x * (kRefWarps / split) + warp / split) * n_pts;
  PointRecord own;
  own.mat = -1;
  own.r = own.h_inv = 0.0f;
  if (lane < n_pts && p0 + lane < a.n) own = load_point(a, p0 + lane);
  MarchDir own_i = {}, own_o = {};
  if (VIS && own.mat >= 0) {
    own_i = march_dir(a.mats + own.mat, make_float3(own.wi_x, own.wi_y, own.wi_z));
    own_o = march_dir(a.mats + own.mat, make_float3(own.wo_x, own.wo_y, own.wo_z));
  }
  if (kStaged) {
    if (lane < n_pts) {
      recs[warp][lane] = own;
      if (VIS) {
        dirs[0][warp][lane] = own_i;
        dirs[1][warp][lane] = own_o;
      }
    }
    __syncwarp();
  }
  SamplePlan sp;
  sp.spp = a.nx * a.ny;
  sp.stride = L * split;
  sp.step = pk2((float)(sp.stride % a.nx), (float)(sp.stride / a.nx));
  sp.wrap = pk2(-(float)a.nx, 1.0f);
  const int first = lane_g + L * part;
  sp.first = pk2((float)(first % a.nx), (float)(first / a.nx));
  sp.two_over_n = pk2(a.two_over_nx, a.two_over_ny);
  sp.nx = (float)a.nx;
  Sums total = {0.f, 0.f, 0.f, 0.f, 0.f};
  for (int round = 0; round < a.rounds; ++round) {
    const int pt = round * G + group;
    Sums acc = {0.f, 0.f, 0.f, 0.f, 0.f};
    const PointRecord &R = kStaged ? recs[warp][pt] : own;
    // V = 1: the loop's variant is chosen for the whole warp, so that its groups stay
    // together: with one point per warp both tests are taken out of the
    // loop (about six instructions a sample), with several only the width
    // (points with |wi + wo| < 1 are a few in a hundred, so most warps of
    // eight or more points hold one).
    if (VIS) {
      if (kStaged) integrate_visible(a, R, dirs[0][warp][pt], dirs[1][warp][pt], sp, first, acc);
      else integrate_visible(a, R, own_i, own_o, sp, first, acc);
    } else if (__all_sync(0xFFFFFFFFu, R.mat < 0 || (fabsf(R.r) < kSmallRadius && (L < 32 || R.h_inv <= 1.0f)))) {
      if (R.mat >= 0) integrate<false, (L < 32), L>(a, R, sp, lane_g, acc);
    } else {
      if (R.mat >= 0) integrate<true, true, L>(a, R, sp, lane_g, acc);
    }
    __syncwarp();
    // reduction inside each group of L lanes
#pragma unroll
    for (int off = L / 2; off > 0; off >>= 1) {
      acc.c0 += __shfl_xor_sync(0xFFFFFFFFu, acc.c0, off);
      acc.c1 += __shfl_xor_sync(0xFFFFFFFFu, acc.c1, off);
      acc.s0 += __shfl_xor_sync(0xFFFFFFFFu, acc.s0, off);
      acc.s1 += __shfl_xor_sync(0xFFFFFFFFu, acc.s1, off);
      acc.a += __shfl_xor_sync(0xFFFFFFFFu, acc.a, off);
    }
    if (!kStaged) {
      total = acc;
    } else if (lane_g == 0) {
      sums[warp][0][pt] = acc.c0;
      sums[warp][1][pt] = acc.c1;
      sums[warp][2][pt] = acc.s0;
      sums[warp][3][pt] = acc.s1;
      sums[warp][4][pt] = acc.a;
    }
  }
  const int64_t p = p0 + lane;
  if (split > 1) __syncthreads();
  else if (kStaged) __syncwarp();
  if (lane >= n_pts || p >= a.n || part != 0) return;
  const int mat = own.mat;
  if (kStaged) {
    for (int w = warp; w < warp + split; ++w) {
      total.c0 += sums[w][0][lane];
      total.c1 += sums[w][1][lane];
      total.s0 += sums[w][2][lane];
      total.s1 += sums[w][3][lane];
      total.a += sums[w][4][lane];
    }
  }
  float c[4], rgb[3];
  if (mat < 0) {
    c[0] = c[1] = c[2] = c[3] = rgb[0] = rgb[1] = rgb[2] = __int_as_float(0x7FC00000);
  } else {
    const bool seen = total.a > 0.0f;
    const float up = total.a < 0x1p-64f ? 0x1p64f : 1.0f;   // the reciprocal of a subnormal A overflows
    const float ia = seen ? 1.0f / (total.a * up) : 0.0f;
    c[0] = seen ? total.c0 * up * ia : 0.0f;
    c[1] = seen ? total.c1 * up * ia : 0.0f;
    c[2] = seen ? total.s0 * up * ia : 0.0f;
    c[3] = seen ? total.s1 * up * ia : 0.0f;
    const DevMaterial *m = a.mats + mat;
#pragma unroll
    for (int ch = 0; ch < 3; ++ch)
      rgb[ch] = m->kd[0][ch] * c[0] + m->kd[1][ch] * c[1] + m->ks[0][ch] * c[2] + m->ks[1][ch] * c[3];
  }
  if (a.comps) store_row4(a.comps, p, c[0], c[1], c[2], c[3]);
#pragma unroll
  for (int ch = 0; ch < 3; ++ch) a.rgb[3 * p + ch] = rgb[ch];
}

template <int L>
void launch_lanes(const RefArgs &a, unsigned blocks, bool visibility, cudaStream_t s) {
  if (visibility) reference_kernel<L, true><<<blocks, kRefThreads, 0, s>>>(a);
  else reference_kernel<L, false><<<blocks, kRefThreads, 0, s>>>(a);
}

}  // namespace

// A whole warp for large sample counts: its lanes' samples are neighbouring
// strata, which mostly fall into the same cell and yarn, so the branches stay
// together (1080p frame, 1024 spp: 10.8 ms with 32 lanes, 11.7 with 8, 12.4
// with one; 256 spp: 2.91, 3.00, 3.11 ms).  With fewer samples the reduction and
// the warp's rounds outweigh that (64 spp: 0.79 ms with 4 lanes, 0.80 with 8,
// 0.84 with 16, 0.92 with 32; 16 spp: 0.22 ms with one, 0.26 with 8; 4 spp:
// 0.076 with one, 0.105 with 4), but the lines lie where a lane's chain of
// additions does not yet cost digits: with 4 lanes the median error of the
// diffuse components at 64 and 120 spp is 6 and 12 % above that with 16, with 8
// lanes 2 %; one lane's 16 samples are added in blocks of four (4 % above 16
// lanes, one chain 15 %; 0.224 -> 0.227 ms).  Small G-buffers take more lanes,
// until the resident threads (1024 per SM) are used twice.
int reference_lanes(int64_t n, int spp, bool visibility, int sm_count) {
  if (visibility) {
    // as many lanes as there are samples: the marches' lengths vary most from
    // point to point, and a warp with several points waits for the longest
    // (1080p, 64 spp: 5.7 ms with 32 lanes, 8.2 with 16, 13.5 with 4)
    int L = 1;
    while (L < 32 && 2 * L <= spp) L *= 2;
    return L;
  }
  int L = spp >= 256 ? 32 : spp >= 96 ? 16 : spp >= 32 ? 8 : spp > 16 ? 4 : 1;
  const int64_t threads = (int64_t)(sm_count > 0 ? sm_count : 148) * 2048;
  while (L < 32 && 2 * L <= spp && n * L < threads) L *= 2;
  return L;
}

cudaError_t launch_reference(const fabric_gbuffer &g, const DevMaterial *mats, int n_mat, int spp_x, int spp_y,
                             uint64_t seed, float *rgb, float *comps, int *status, int lanes_per_point,
                             int sm_count, cudaStream_t s, bool visibility) {
  RefArgs a;
  a.u = g.u;
  a.v = g.v;
  a.radius = g.radius;
  a.wi = g.wi;
  a.wo = g.wo;
  a.material = g.material;
  a.n = g.n;
  a.mats = mats;
  a.n_mat = n_mat;
  a.nx = spp_x;
  a.ny = spp_y;
  a.two_over_nx = 2.0f / (float)spp_x;
  a.two_over_ny = 2.0f / (float)spp_y;
  a.seed = seed;
  a.rgb = rgb;
  a.comps = comps;
  a.status = status;
  // Points per warp: as many as its lanes can prepare at once (32), fewer
  // where the grid would not fill the resident warps (32 per SM) twice.
  const int L = lanes_per_point, G = 32 / L;
  const int64_t groups = (g.n + G - 1) / G, resident = (int64_t)(sm_count > 0 ? sm_count : 148) * 32;
  a.rounds = (int)std::max<int64_t>(1, std::min<int64_t>(L, groups / (2 * resident)));
  // With the visibility model one point's marches can outlast the rest of the
  // grid (grazing directions over wide footprints), so several warps share a
  // point once each lane still has a few samples: 8190 queries at 2048 spp
  // 2.9 ms with one warp a point, 1.6 with 4, 1.3 with 8; 4000 points at 1024
  // spp 0.95, 0.35, 0.27 ms; 30 000 at 256 spp 1.15, 0.79, 0.79 ms.  Large grids
  // at 256 spp hide the long points and keep one warp (2.07 M points 21.8 ms,
  // 27.5 with 4; 300 000 points the same with either), as 64 spp does (60 000
  // points 0.30 ms, 0.49 with 4); at 1024 spp 8 warps cost a large grid nothing
  // (2.07 M points 84.1 and 85.6 ms; 100 000 points 8.5 and 7.0 ms).
  const int spp = spp_x * spp_y;
  a.split = !visibility || L < 32 ? 1 : spp >= 1024 ? 8 : spp >= 256 && g.n < 64 * resident ? 4 : 1;
  if (a.split > 1) a.rounds = 1;
  const int64_t per_cta = (int64_t)(kRefWarps / a.split) * G * a.rounds;
  const unsigned blocks = (unsigned)((g.n + per_cta - 1) / per_cta);
  switch (L) {
    case 1: launch_lanes<1>(a, blocks, visibility, s); break;
    case 2: launch_lanes<2>(a, blocks, visibility, s); break;
    case 4: launch_lanes<4>(a, blocks, visibility, s); break;
    case 8: launch_lanes<8>(a, blocks, visibility, s); break;
    case 16: launch_lanes<16>(a, blocks, visibility, s); break;
    default: launch_lanes<32>(a, blocks, visibility, s); break;
  }
  return cudaGetLastError();
}

}  // namespace fab
