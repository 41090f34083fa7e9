// tm_merge.cu -- the capture front-end of Section III: a WDR radiance map from
// several exposures by Debevec and Malik's method (the paper's application
// captures four exposures and recovers the WDR image this way before tone
// mapping it).
//
// For each channel of each pixel, with z_j the exposure's 8-bit value, g the
// channel's log inverse response (g(z) = ln of the sensor exposure that maps
// to z) and dt_j the exposure time:
//     ln E = sum_j w(z_j) (g(z_j) - ln dt_j) / sum_j w(z_j),
//     w(z) = z for z <= 127, 255 - z above (the hat weighting),
// and E = exp(ln E). Where every weight is zero (each exposure at 0 or 255),
// the shortest exposure's estimate is taken if it is saturated, else the
// longest's. The response table travels as a kernel parameter; nothing is
// allocated.
//
// Bound by issue before bandwidth (n bytes read and 4 written per sample). A
// thread takes four pixels, twelve samples, as three 4-byte words per exposure
// and three 16-byte stores; shared memory holds, per exposure and channel, the
// pairs (g(z) - ln dt_j, w(z)), so that an exposure costs a sample one 8-byte
// read, an FMA and an add. The quotient is formed from a table of correctly
// rounded reciprocals of the weight sums (integers up to 8 x 127) by
// Markstein's correction, q + (a - b q) y with y = RN(1 / b), which rounds like
// the division. All lanes of a table read work on the same channel of nearby
// pixels, whose values are close, so the reads hardly conflict (four
// consecutive samples per thread, all memory accesses coalesced but three
// channels per read: 112 us). Four 12 MP exposures took 155 us with a pixel per
// thread, 1-byte loads and a division each, and take 79; more blocks per SM
// are slower (5: 88, 6: 93, 8: 154).
#include <algorithm>
#include <cmath>

#include "tm.h"
#include "tm_host.h"
#include "tm_kernels.cuh"

using namespace tmk;

namespace {

constexpr int kMaxExposures = 8;
constexpr int kMT = 256;
constexpr int kMB = 4;  // resident blocks per SM (8 exposures: 53 KB of tables each)
constexpr int kRecips = kMaxExposures * 127 + 1;  // weight sums
constexpr float kOne = 8388608.f;                 // 2^23: integers up to 2^23 above it are exact

struct MergeArgs {
  const uint8_t *ldr[kMaxExposures];  // HWC uint8, pitch_in elements per row
  float neg_log_t[kMaxExposures];     // -ln dt_j
  int n, shortest, longest;
  int vec;                            // words and vector stores are aligned, and |num| stays far below overflow
  long long pitch_in;
  float g[3][256];                    // log inverse response per channel
};

// ln E of a sample whose every weight is zero: z0 its value in the shortest
// exposure, z1 in the longest.
__device__ __forceinline__ float outside(const MergeArgs &a, const float2 *tab, int c, unsigned z0, unsigned z1) {
  return z0 == 255u ? tab[(a.shortest * 3 + c) * 256 + 255].x : tab[(a.longest * 3 + c) * 256 + z1].x;
}

// num / den, den a weight sum > 0 with rden = RN(1 / den).
__device__ __forceinline__ float quotient(float num, float den, float rden) {
  const float q = num * rden;
  return fmaf(fmaf(-q, den, num), rden, q);
}

// kN: the number of exposures when known at compile time (0: read from a).
template <int kN>
__global__ void __launch_bounds__(kMT, kMB)
    k_merge(const __grid_constant__ MergeArgs a, const __grid_constant__ Image out) {
  extern __shared__ float2 tab[];  // [n][3][256]: (g(z) - ln dt_j, w(z))
  __shared__ float rcp[kRecips];
  const int ne = kN ? kN : a.n;
  for (int i = threadIdx.x; i < ne * 768; i += kMT) {
    const int j = i / 768, z = i & 255;
    tab[i] = make_float2((&a.g[0][0])[i - 768 * j] + a.neg_log_t[j], (float)(z <= 127 ? z : 255 - z));
  }
  for (int i = threadIdx.x; i < kRecips; i += kMT) rcp[i] = 1.f / (float)i;
  __syncthreads();
  const int W = out.W, H = out.H;
  const unsigned gpr = ((unsigned)W + 3u) >> 2, ng = gpr * (unsigned)H;  // groups of four pixels
  for (unsigned g = blockIdx.x * kMT + threadIdx.x; g < ng; g += gridDim.x * kMT) {
    const int y = (int)(g / gpr), x = 4 * (int)(g - (unsigned)y * gpr);
    const int np = min(4, W - x);
    const long long o = (long long)y * a.pitch_in + 3LL * x;
    if (a.vec && np == 4) {
      float num[12], den[12], E[12], least = 1.f;
#pragma unroll
      for (int s = 0; s < 12; ++s) {
        num[s] = 0.f;
        den[s] = kOne;  // the sum counts in the low bits of the significand
      }
#pragma unroll
      for (int j = 0; j < (kN ? kN : kMaxExposures); ++j) {
        if (!kN && j >= ne) break;
        unsigned w[3];
#pragma unroll
        for (int k = 0; k < 3; ++k) w[k] = __ldg(reinterpret_cast<const unsigned *>(a.ldr[j] + o) + k);
#pragma unroll
        for (int s = 0; s < 12; ++s) {
          // the byte's value times 8, the entry's offset
          const unsigned at = (s & 3 ? w[s >> 2] >> (8 * (s & 3) - 3) : w[s >> 2] << 3) & 0x7f8u;
          const char *row = reinterpret_cast<const char *>(tab + (j * 3 + s % 3) * 256);
          const float2 t = *reinterpret_cast<const float2 *>(row + at);
          num[s] = fmaf(t.y, t.x, num[s]);
          den[s] += t.y;
        }
      }
#pragma unroll
      for (int s = 0; s < 12; ++s) {
        const float d = den[s] - kOne;
        least = fminf(least, d);
        E[s] = expf(quotient(num[s], d, rcp[__float_as_uint(den[s]) & 0x3ffu]));
      }
      if (least == 0.f) {  // some sample is clipped in every exposure
#pragma unroll
        for (int s = 0; s < 12; ++s)
          if (den[s] == kOne)
            E[s] = expf(outside(a, tab, s % 3, __ldg(a.ldr[a.shortest] + o + s), __ldg(a.ldr[a.longest] + o + s)));
      }
      const long long oo = (long long)y * out.pitch + 3LL * x;
      if (out.dtype == kF32) {
        float4 *p = reinterpret_cast<float4 *>(static_cast<float *>(out.p) + oo);
#pragma unroll
        for (int k = 0; k < 3; ++k) p[k] = make_float4(E[4 * k], E[4 * k + 1], E[4 * k + 2], E[4 * k + 3]);
      } else {
        uint2 *p = reinterpret_cast<uint2 *>(static_cast<__half *>(out.p) + oo);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          const __half2 h0 = __floats2half2_rn(E[4 * k], E[4 * k + 1]);
          const __half2 h1 = __floats2half2_rn(E[4 * k + 2], E[4 * k + 3]);
          p[k] = make_uint2(*reinterpret_cast<const unsigned *>(&h0), *reinterpret_cast<const unsigned *>(&h1));
        }
      }
      continue;
    }
    for (int i = 0; i < np; ++i) {
      float E[3];
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const long long q = o + 3 * i + c;
        float num = 0.f, den = 0.f;
        for (int j = 0; j < ne; ++j) {
          const float2 t = tab[(j * 3 + c) * 256 + __ldg(a.ldr[j] + q)];
          num = fmaf(t.y, t.x, num);
          den += t.y;
        }
        E[c] = expf(den > 0.f ? num / den
                              : outside(a, tab, c, __ldg(a.ldr[a.shortest] + q), __ldg(a.ldr[a.longest] + q)));
      }
      store_rgb(out, x + i, y, E[0], E[1], E[2]);
    }
  }
}

}  // namespace

extern "C" tm_status tm_merge_exposures(int32_t n, const uint8_t *const *ldr, const float *times,
                                        int32_t width, int32_t height, int64_t pitch,
                                        const float *log_response, const tm_image *out, void *stream) {
  if (n < 1 || n > kMaxExposures)
    return fail_noctx(TM_EINVAL, "tm_merge_exposures: 1 to 8 exposures");
  if (!ldr || !times || !log_response || !out || !out->data)
    return fail_noctx(TM_EINVAL, "tm_merge_exposures: null argument");
  if (width < 1 || height < 1 || (long long)width * height > (1LL << 31) - 1 || pitch < 3LL * width)
    return fail_noctx(TM_EINVAL, "tm_merge_exposures: bad size or pitch");
  if (out->width != width || out->height != height || out->pitch < 3LL * width ||
      (out->dtype != TM_F32 && out->dtype != TM_F16))
    return fail_noctx(TM_EINVAL, "tm_merge_exposures: out must be a float32 or float16 image of the same size");
  MergeArgs a{};
  a.n = n;
  a.pitch_in = pitch;
  for (int j = 0; j < n; ++j) {
    if (!ldr[j]) return fail_noctx(TM_EINVAL, "tm_merge_exposures: null exposure");
    if (!(times[j] > 0.f)) return fail_noctx(TM_EINVAL, "tm_merge_exposures: exposure times must be > 0");
    a.ldr[j] = ldr[j];
    a.neg_log_t[j] = (float)-std::log((double)times[j]);
    if (times[j] < times[a.shortest]) a.shortest = j;
    if (times[j] > times[a.longest]) a.longest = j;
  }
  for (int c = 0; c < 3; ++c)
    for (int z = 0; z < 256; ++z) {
      const float v = log_response[256 * c + z];
      if (!std::isfinite(v)) return fail_noctx(TM_EINVAL, "tm_merge_exposures: response table must be finite");
      a.g[c][z] = v;
    }
  Image o;
  o.p = out->data;
  o.W = width;
  o.H = height;
  o.pitch = out->pitch;
  o.dtype = out->dtype;
  if (pitch == 3LL * width && out->pitch == 3LL * width) {  // gapless rows: one row of every pixel
    o.W = width * height;
    o.H = 1;
    a.pitch_in = o.pitch = 3LL * o.W;
  }
  const size_t align = out->dtype == TM_F32 ? 16 : 8, es = out->dtype == TM_F32 ? 4 : 2;
  bool vec = (o.H == 1 || (pitch % 4 == 0 && ((size_t)out->pitch * es) % align == 0)) && (uintptr_t)o.p % align == 0;
  // (an infinite exposure time makes sums infinite: the corrected quotient of
  // the vector form would turn their limit, E = 0, into NaN)
  for (int j = 0; j < n; ++j) vec = vec && (uintptr_t)ldr[j] % 4 == 0 && std::isfinite(a.neg_log_t[j]);
  for (const auto &ch : a.g)
    for (const float v : ch) vec = vec && std::fabs(v) < 1e30f;
  a.vec = vec ? 1 : 0;
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const long long groups = (o.W + 3LL) / 4 * o.H;
  const long long want = (groups + kMT - 1) / kMT, cap = (long long)kMB * (sms > 0 ? sms : 1);
  const int blocks = (int)std::min(want, cap);
  const size_t smem = sizeof(float2) * 768 * (size_t)n;  // at most 48 KB
  const cudaStream_t st = static_cast<cudaStream_t>(stream);
  // eight have a variant of their own: pixel values without order conflict in
  // the table reads, and the general one took 230 us for 12 MP of white noise
  // (217 a pixel per thread; 223 now, photographs 151 -> 122). With variants
  // for five to seven 2 MP took up to 5 % longer.
  auto *const kernel = n == 2 ? k_merge<2> : n == 3 ? k_merge<3> : n == 4 ? k_merge<4> : n == 8 ? k_merge<8>
                                                                                                : k_merge<0>;
  // the limit is state of the kernel shared by every thread of the process:
  // always the largest, so that no call lowers it under another's launch
  if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)(sizeof(float2) * 768 * kMaxExposures)) != cudaSuccess)
    return fail_noctx(TM_ECUDA, "tm_merge_exposures: shared-memory attribute");
  kernel<<<blocks, kMT, smem, st>>>(a, o);
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return fail_noctx(TM_ECUDA, "tm_merge_exposures: kernel launch failed");
  return TM_OK;
}
