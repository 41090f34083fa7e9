// tm_lookup.cuh -- the per-pixel arithmetic shared by the lookup kernels: one
// field folded into the fusion of Eq. 3, and the colour restoration of Eq. 12.
#pragma once

#include "tm_common.cuh"

namespace tmk {

// Running sums of the fusion of Eq. 3 over the fields.
struct Fusion {
  float wsum = 0.f, acc = 0.f, mean = 0.f;
};

// Eq. 1, 2 and 4 of a field, folded into the sums of Eq. 3. kFast: the
// quotient of Eq. 4 without the division's handling of tiny denominators
// (P.fast: every eps is at least 1e-30); the same bits.
template <bool kFast>
__device__ __forceinline__ void fuse_field(const DevParams &P, int f, unsigned cnt, float rarea, float var, Fusion &fu,
                                           float &Wf, float &Lf) {
  const float Pf = (float)cnt * rarea;                                  // Eq. 1
  Lf = fmaf(P.ld_max - P.ld_min, Pf, P.ld_min);                         // Eq. 2
  Wf = kFast ? (P.alpha[f] * var) * rcp_normal(var + P.eps[f])
             : __fdividef(P.alpha[f] * var, var + P.eps[f]);            // Eq. 4
  fu.wsum += Wf;
  fu.acc = fmaf(Wf, Lf, fu.acc);
  fu.mean += Lf;
}

// Eq. 3 from the sums.
__device__ __forceinline__ float fused_value(const DevParams &P, const Fusion &fu) {
  return fu.wsum > 0.f ? __fdividef(fu.acc, fu.wsum) : __fdividef(fu.mean, (float)P.n_fields);
}

// The factors (C / i)^sat of Eq. 12 (restore_channel without L). kFast: ratios
// in the normal range take the base-2 logarithm and exponential without their
// handling of denormals (P.fast: sat <= 0.9, so the exponent stays within
// +-126); the same bits. Returns the channels (bits) whose result is 0
// whatever L: those without a positive ratio, unless sat = 0.
template <bool kFast>
__device__ __forceinline__ unsigned colour_powers(const DevParams &P, const float *rgb, float *pw) {
  const float inv_i = __fdividef(1.f, luminance(rgb[0], rgb[1], rgb[2]));
  const float a = rgb[0] * inv_i, b = rgb[1] * inv_i, c = rgb[2] * inv_i;
  constexpr float kMin = 1.17549435e-38f;
  if (kFast && a >= kMin && b >= kMin && c >= kMin) {
    pw[0] = exp2_normal(P.sat * log2_normal(a));
    pw[1] = exp2_normal(P.sat * log2_normal(b));
    pw[2] = exp2_normal(P.sat * log2_normal(c));
    return 0u;
  }
  pw[0] = a > 0.f ? exp2f(P.sat * __log2f(a)) : 1.f;
  pw[1] = b > 0.f ? exp2f(P.sat * __log2f(b)) : 1.f;
  pw[2] = c > 0.f ? exp2f(P.sat * __log2f(c)) : 1.f;
  return P.sat == 0.f ? 0u : (a > 0.f ? 0u : 1u) | (b > 0.f ? 0u : 2u) | (c > 0.f ? 0u : 4u);
}

// Field f of pixel (x, y) with Eq. 1 numerator cnt: Eq. 2 and Eq. 4 folded
// into the Eq. 3 sums (the same arithmetic as fuse_fields, one field at a
// time, so no per-field state is kept).
// mom (or null): receives the window's variance and mean of lhat for the
// backward (inv_scale = 2^-Q). kPlain: no debug planes and no literal area,
// and moments only under kMom (the other paths are then not compiled in);
// kSmall as for window_variance.
template <bool kPlain = false, bool kMom = false, int kSmall = -1>
__device__ __forceinline__ void fold_field(const DevParams &P, int f, int x, int y, int W, int H,
                                           unsigned cnt, const longlong2 *__restrict__ s12, int qbits,
                                           float inv_scale2, Fusion &fu, const DebugPlanes &dbg,
                                           float2 *mom = nullptr, float inv_scale = 0.f) {
  const WinMoments m = window_moments<!kPlain, kSmall>(P, f, x, y, W, H, s12, qbits, inv_scale2);
  const float rarea = m.rarea, var = m.var;
  if (kPlain ? kMom : mom != nullptr)
    mom[(size_t)f * W * H + (size_t)y * W + x] = make_float2(var, window_mean(m.q1, rarea, inv_scale));
  float Wf, Lf;
  fuse_field<false>(P, f, cnt, rarea, var, fu, Wf, Lf);
  if (!kPlain && dbg.l) {
    const long long N = (long long)W * H, pix = (long long)y * W + x;
    dbg.cnt[f * N + pix] = cnt;
    dbg.sigma2[f * N + pix] = var;
    dbg.weight[f * N + pix] = Wf;
    dbg.lf[f * N + pix] = Lf;
  }
}

// Eq. 3 and Eq. 12 for one pixel from the folded sums. kDt: the dtype of
// both images when known at compile time (-1: read from the descriptors).
template <bool kPlain = false, int kDt = -1>
__device__ __forceinline__ void finish_pixel(const Image &in, const Image &out, const DevParams &P,
                                             int x, int y, const Fusion &fu, const DebugPlanes &dbg) {
  const float L = fused_value(P, fu);
  float r, g, b;
  load_rgb<kDt>(in, x, y, r, g, b);
  const float inv_i = __fdividef(1.f, luminance(r, g, b));
  store_rgb<kDt>(out, x, y, restore_channel(r, inv_i, P.sat, L), restore_channel(g, inv_i, P.sat, L),
                 restore_channel(b, inv_i, P.sat, L), (P.flags & kFlagSrgb) != 0);
  if (!kPlain && dbg.l) dbg.l[(long long)y * in.W + x] = L;
}

}  // namespace tmk
