// tm_integral.cu -- integral images (Eq. 5) and integral histograms (Eq. 7-8).
//
// The integral images of q and q^2 are built over tiles of kIR rows x kIC
// columns in three launches that read q twice and write each plane once:
//   1. per tile: the column sums of the tile's chunk-local row prefixes, each
//      row's chunk total, and the tile total;
//   2. per column: the exclusive prefix over the row segments of those column
//      sums plus the row totals of the chunks to the left (the value of the
//      plane just above each segment);
//   3. per tile: the row prefixes again, offset by the chunks to the left, and
//      accumulated down the tile from the column's offset, written once.
// The same tile kernels, templated on the source of their two planes, build
// the backward's fixed-point integral planes of (u_f, v_f). The integral
// histograms have kernels of their own (k_hist_*). Integer arithmetic is modular (2^64 in the sums, 2^32 in the
// histogram planes), so box sums (Eq. 6, Eq. 9) are exact whatever the image
// size or summation order.
#include <algorithm>
#include <climits>
#include <type_traits>
#include <cstdint>

#include "tm_kernels.cuh"

namespace tmk {
namespace {

constexpr int kItems = 8;  // consecutive columns per thread in a tile row

// Rows go through shared memory so that global accesses are coalesced while
// each thread scans eight consecutive elements; the shared layouts are padded
// (9 slots per 8 elements) against bank conflicts.
__device__ __forceinline__ int pad9(int i) { return (i >> 3) * 9 + (i & 7); }

// ---- integral images of q and q^2 over tiles ----
constexpr int kINT = 128;               // threads of a tile kernel
constexpr int kIC = kINT * kItems;      // columns of a tile (1024)
constexpr int kIR = 16;                 // rows of a tile (one row segment) unless scratch is tight
constexpr int kMidCols = 32;            // columns of a column-prefix block
constexpr int kMidGroups = 16;          // segment groups of a column-prefix block
constexpr int kMidPer = 8;              // segments of a group per batch

// One tiled integral task: two (H+1) x (W+1) int64 planes A and B of an
// image (row 0 and column 0 zero), with their scratch (int64): the tiles'
// column sums, rewritten in place by the column prefix (2 planes x nseg x W),
// the rows' chunk totals (2 x H x nchunk) and the tile totals
// (2 x nseg x nchunk). Row segments of seg_rows rows, nseg of them.
struct IntTask {
  int W, H, nseg, seg_rows, nchunk;
  long long *colsum, *rowsum, *tiletot;
};

__device__ __forceinline__ IntTask int_task(int W, int H, int nseg, int seg_rows, long long *scratch) {
  IntTask t;
  t.W = W;
  t.H = H;
  t.nseg = nseg;
  t.seg_rows = seg_rows;
  t.nchunk = (W + kIC - 1) / kIC;
  t.colsum = scratch;
  t.rowsum = t.colsum + 2LL * nseg * W;
  t.tiletot = t.rowsum + 2LL * H * t.nchunk;
  return t;
}

// Values of the planes: q and q^2 of the quantised log (Eq. 5 of q).
struct QSource {
  using Raw = int32_t;
  const int32_t *q;
  int W;
  __device__ __forceinline__ Raw load(int r, int c) const { return __ldg(q + (long long)r * W + c); }
  // columns c .. c + 3 of row r (zero past W); vec: rows are 16-byte aligned
  __device__ __forceinline__ void load4(int r, int c, bool vec, Raw *x) const {
    const int32_t *p = q + (size_t)r * W + c;
    if (vec && c + 3 < W) {
      const int4 v = __ldg(reinterpret_cast<const int4 *>(p));
      x[0] = v.x, x[1] = v.y, x[2] = v.z, x[3] = v.w;
    } else {
#pragma unroll
      for (int j = 0; j < 4; ++j) x[j] = c + j < W ? __ldg(p + j) : 0;
    }
  }
  __device__ __forceinline__ bool vec_ok() const {
    return (W & 3) == 0 && (reinterpret_cast<uintptr_t>(q) & 15) == 0;
  }
  // warp sums of a thread's four-element partial row sums: |q| <= 2^23, so a
  // partial sum of q fits 26 bits and one of q^2 splits into two 24-bit
  // parts, each summed exactly in 32 bits by the warp reduction
  __device__ __forceinline__ void warp_sums(long long &su, long long &sv) const {
    su = (long long)__reduce_add_sync(0xffffffffu, (int)su);
    const unsigned long long v = (unsigned long long)sv;
    const unsigned hi = __reduce_add_sync(0xffffffffu, (unsigned)(v >> 24));
    const unsigned lo = __reduce_add_sync(0xffffffffu, (unsigned)(v & 0xffffffu));
    sv = (long long)(((unsigned long long)hi << 24) + lo);
  }
  __device__ __forceinline__ Raw zero() const { return 0; }
  __device__ __forceinline__ void values(Raw x, long long &a, long long &b) const {
    a = x;
    b = (long long)x * x;
  }
};

// Values of the planes: two float planes in 64-bit fixed point, u x 2^sa and
// v x 2^sb rounded to nearest. Each power of two is applied as two float
// factors 2^h and 2^(s - h), h = s / 2 (s in [-67, 209], so both are normal):
// for s >= 0 no product leaves the normal range; for s < 0 only values that
// end below 2^-126 can round twice, and those convert to 0 either way, so
// the integers equal those of a single scaling.
struct FixSource {
  using Raw = float2;
  const float *u, *v;
  int W, pitch;  // rows of pitch floats
  float a_hi, a_lo, b_hi, b_lo;
  __device__ __forceinline__ Raw load(int r, int c) const {
    const long long o = (long long)r * pitch + c;
    return make_float2(__ldg(u + o), __ldg(v + o));
  }
  __device__ __forceinline__ Raw zero() const { return make_float2(0.f, 0.f); }
  __device__ __forceinline__ void load4(int r, int c, bool vec, Raw *x) const {
    const size_t o = (size_t)r * pitch + c;
    if (vec && c + 3 < W) {
      const float4 a = __ldg(reinterpret_cast<const float4 *>(u + o));
      const float4 b = __ldg(reinterpret_cast<const float4 *>(v + o));
      x[0] = make_float2(a.x, b.x), x[1] = make_float2(a.y, b.y);
      x[2] = make_float2(a.z, b.z), x[3] = make_float2(a.w, b.w);
    } else {
#pragma unroll
      for (int j = 0; j < 4; ++j) x[j] = c + j < W ? make_float2(__ldg(u + o + j), __ldg(v + o + j)) : zero();
    }
  }
  __device__ __forceinline__ bool vec_ok() const {
    return (pitch & 3) == 0 && ((reinterpret_cast<uintptr_t>(u) | reinterpret_cast<uintptr_t>(v)) & 15) == 0;
  }
  __device__ __forceinline__ void warp_sums(long long &su, long long &sv) const {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      su += __shfl_xor_sync(0xffffffffu, su, o);
      sv += __shfl_xor_sync(0xffffffffu, sv, o);
    }
  }
  // u through the hardware conversion (the FP64 pipe), v through the 32-bit
  // integer sequence (the ALU pipe): both give round-to-nearest-even, and the
  // split keeps either pipe from limiting the tile kernels
  __device__ __forceinline__ void values(Raw x, long long &a, long long &b) const {
    a = __float2ll_rn(x.x * a_hi * a_lo);
    b = float_to_i64_rn(x.y * b_hi * b_lo);
  }
};

__device__ __forceinline__ FixSource fix_source_of(const float *u, const float *v, int W, int pitch, int sa, int sb) {
  return FixSource{u, v, W, pitch, ldexpf(1.f, sa / 2), ldexpf(1.f, sa - sa / 2), ldexpf(1.f, sb / 2),
                   ldexpf(1.f, sb - sb / 2)};
}

// Exclusive block scan of a pair of values with one set of barriers.
__device__ __forceinline__ void block_scan_pair(long long v1, long long v2, long long (*wt)[kINT / 32],
                                                long long &e1, long long &e2, long long &t1, long long &t2) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  long long x1 = v1, x2 = v2;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const long long y1 = __shfl_up_sync(0xffffffffu, x1, o), y2 = __shfl_up_sync(0xffffffffu, x2, o);
    if (lane >= o) x1 += y1, x2 += y2;
  }
  if (lane == 31) wt[0][wid] = x1, wt[1][wid] = x2;
  __syncthreads();
  long long b1 = 0, b2 = 0;
#pragma unroll
  for (int w = 0; w < kINT / 32; ++w) {
    if (w < wid) b1 += wt[0][w], b2 += wt[1][w];
  }
  t1 = 0;
  t2 = 0;
#pragma unroll
  for (int w = 0; w < kINT / 32; ++w) t1 += wt[0][w], t2 += wt[1][w];
  e1 = b1 + x1 - v1;
  e2 = b2 + x2 - v2;
  __syncthreads();  // wt is rewritten by the next scan
}

// The thread's kItems strided raw elements (i = threadIdx.x + m kINT) of
// chunk [C0, C0 + nc) of row r; zero past the chunk.
template <class Src>
__device__ __forceinline__ void load_chunk_row(const Src &src, int r, int C0, int nc, typename Src::Raw *v) {
#pragma unroll
  for (int m = 0; m < kItems; ++m) {
    const int i = threadIdx.x + m * kINT;
    v[m] = i < nc ? src.load(r, C0 + i) : src.zero();
  }
}

// Chunk-local row prefixes of planes A and B of one row, given the thread's
// strided raw elements of it (load_chunk_row): thread-local running sums of
// its kItems consecutive columns (l1, l2) and the exclusive offsets of the
// thread (e1, e2); t1, t2 are the row's chunk totals. The row goes through
// shared memory so that the loads were coalesced and each thread scans
// consecutive columns.
template <class Src>
__device__ __forceinline__ void chunk_row_prefix(const Src &src, const typename Src::Raw *v,
                                                 typename Src::Raw *tile, long long (*wt)[kINT / 32],
                                                 long long *l1, long long *l2, long long &e1, long long &e2,
                                                 long long &t1, long long &t2) {
#pragma unroll
  for (int m = 0; m < kItems; ++m) tile[pad9(threadIdx.x + m * kINT)] = v[m];
  __syncthreads();
  long long a1 = 0, a2 = 0;
#pragma unroll
  for (int k = 0; k < kItems; ++k) {
    long long x1, x2;
    src.values(tile[threadIdx.x * 9 + k], x1, x2);
    a1 += x1;
    a2 += x2;
    l1[k] = a1;
    l2[k] = a2;
  }
  block_scan_pair(a1, a2, wt, e1, e2, t1, t2);  // its barriers also order the tile's reuse
}

// Launch 1: per tile (seg, k), the column sums of the chunk-local row
// prefixes, the rows' chunk totals and the tile totals. The column sum of the
// row prefixes at column c is the prefix, up to c, of the plain column sums
// (both are the sum of the values above and left of c in the tile), so the
// rows are only summed down each column and across each row (warp sums, no
// barrier per row); one block scan over the columns ends the tile. The row
// and tile totals of the last chunk column are read by no later launch (they
// only offset the chunks to their right), so its tiles skip them. Each thread
// owns four consecutive columns of the chunk and keeps kFSRows rows of loads
// in flight, 16 bytes at a time where the rows are 16-byte aligned.
constexpr int kRowGroup = 16;  // rows whose warp partial sums are combined together
// Launch 2: for columns c0 .. c0 + kMidCols - 1 (of the image, one chunk),
// replace each segment's column sum by the plane value just above the
// segment: the sum, over the segments above, of their column sums plus the
// totals of their chunks left of c's chunk. The block's kMidGroups groups
// take kMidPer consecutive segments each per batch, with all loads of a batch
// in flight together.
constexpr int kMidBatch = kMidGroups * kMidPer;
__device__ __forceinline__ void int_mid_cols(const IntTask &X, int c0, long long (*part)[kMidGroups][kMidCols],
                                             long long (*leftT)[kMidBatch]) {
  const int W = X.W;
  const int lane = threadIdx.x % kMidCols, g = threadIdx.x / kMidCols;
  const int c = c0 + lane;
  const int k = c0 / kIC;  // the block's chunk (kMidCols divides kIC)
  long long carry1 = 0, carry2 = 0;
  for (int sb = 0; sb < X.nseg; sb += kMidBatch) {
    // totals of the batch's segments over the chunks left of k
    for (int t = threadIdx.x; t < 2 * kMidBatch; t += kMidCols * kMidGroups) {
      const int pl = t / kMidBatch, s = sb + t % kMidBatch;
      long long v = 0;
      if (s < X.nseg)
        for (int kk = 0; kk < k; ++kk) v += X.tiletot[((long long)pl * X.nseg + s) * X.nchunk + kk];
      leftT[pl][t % kMidBatch] = v;
    }
    __syncthreads();
    const int s0 = sb + g * kMidPer;
    long long v1[kMidPer], v2[kMidPer], sum1 = 0, sum2 = 0;
#pragma unroll
    for (int i = 0; i < kMidPer; ++i) {
      const int s = s0 + i;
      const bool ok = s < X.nseg && c < W;
      v1[i] = ok ? X.colsum[(long long)s * W + c] : 0;
      v2[i] = ok ? X.colsum[((long long)X.nseg + s) * W + c] : 0;
    }
#pragma unroll
    for (int i = 0; i < kMidPer; ++i) {
      if (s0 + i < X.nseg) {
        v1[i] += leftT[0][g * kMidPer + i];
        v2[i] += leftT[1][g * kMidPer + i];
      }
      sum1 += v1[i];
      sum2 += v2[i];
    }
    part[0][g][lane] = sum1;
    part[1][g][lane] = sum2;
    __syncthreads();
    long long run1 = carry1, run2 = carry2;
    for (int h = 0; h < g; ++h) run1 += part[0][h][lane], run2 += part[1][h][lane];
#pragma unroll
    for (int i = 0; i < kMidPer; ++i) {
      const int s = s0 + i;
      if (s < X.nseg && c < W) {
        X.colsum[(long long)s * W + c] = run1;
        X.colsum[((long long)X.nseg + s) * W + c] = run2;
      }
      run1 += v1[i];
      run2 += v2[i];
    }
    for (int h = 0; h < kMidGroups; ++h) carry1 += part[0][h][lane], carry2 += part[1][h][lane];
    __syncthreads();  // part and leftT are rewritten by the next batch
  }
}

// Launch 3: per tile, the full row prefixes (chunk-local prefix plus the
// row's totals of the chunks to the left) accumulated down the tile from the
// value above it, written to rows 1..H, columns 1..W of planes s1 and s2;
// tiles of the first segment also write row 0, tiles of the first chunk column
// 0. Pair: the planes are interleaved (s2 = s1 + 1, two elements per position),
// and each position is written with one 16-byte store. (A warp per 128 columns
// without a block barrier per row took 52 us alone against 73 at 12 MP, but
// 30 M warp instructions against 23 M, and the forward, which runs this beside
// the compact histogram's build, no less.)
template <class Src, bool Pair = false>
__device__ __forceinline__ void int_write_tile(const IntTask &X, const Src &src, long long *s1, long long *s2, int seg,
                                               int k, typename Src::Raw *tile, long long *out1, long long *out2,
                                               long long (*wt)[kINT / 32]) {
  const int W = X.W, H = X.H;
  const long long W1 = (long long)W + 1;
  const int R0 = seg * X.seg_rows, R1 = min(R0 + X.seg_rows, H), C0 = k * kIC, nc = min(kIC, W - C0);
  const long long os = Pair ? 2 : 1;  // elements per position (Pair: s2 = s1 + 1)
  if (seg == 0) {
    for (int i = threadIdx.x; i < nc; i += kINT) s1[(C0 + 1 + i) * os] = s2[(C0 + 1 + i) * os] = 0;
    if (k == 0 && threadIdx.x == 0) s1[0] = s2[0] = 0;
  }
  if (k == 0)
    for (int r = R0 + (int)threadIdx.x; r < R1; r += kINT) s1[(r + 1) * W1 * os] = s2[(r + 1) * W1 * os] = 0;
  long long acc1[kItems], acc2[kItems];
#pragma unroll
  for (int i = 0; i < kItems; ++i) {
    const int c = C0 + threadIdx.x * kItems + i;
    acc1[i] = c < W ? X.colsum[(long long)seg * W + c] : 0;
    acc2[i] = c < W ? X.colsum[((long long)X.nseg + seg) * W + c] : 0;
  }
  typename Src::Raw cur[kItems], nxt[kItems];
  load_chunk_row(src, R0, C0, nc, cur);
  for (int r = R0; r < R1; ++r) {
    if (r + 1 < R1) load_chunk_row(src, r + 1, C0, nc, nxt);  // in flight meanwhile
    long long L1 = 0, L2 = 0;  // the row's totals of the chunks to the left
    for (int kk = 0; kk < k; ++kk) {
      L1 += X.rowsum[(long long)r * X.nchunk + kk];
      L2 += X.rowsum[((long long)H + r) * X.nchunk + kk];
    }
    long long l1[kItems], l2[kItems], e1, e2, t1, t2;
    chunk_row_prefix(src, cur, tile, wt, l1, l2, e1, e2, t1, t2);
#pragma unroll
    for (int m = 0; m < kItems; ++m) cur[m] = nxt[m];
#pragma unroll
    for (int i = 0; i < kItems; ++i) {
      acc1[i] += L1 + e1 + l1[i];
      acc2[i] += L2 + e2 + l2[i];
      out1[threadIdx.x * 9 + i] = acc1[i];
      out2[threadIdx.x * 9 + i] = acc2[i];
    }
    __syncthreads();
    if (Pair) {  // one 16-byte store per position
      longlong2 *o = reinterpret_cast<longlong2 *>(s1) + (long long)(r + 1) * W1 + C0 + 1;
      for (int i = threadIdx.x; i < nc; i += kINT) o[i] = make_longlong2(out1[pad9(i)], out2[pad9(i)]);
      __syncthreads();
      continue;
    }
    const long long o = (long long)(r + 1) * W1 + C0 + 1;
    for (int i = threadIdx.x; i < nc; i += kINT) s1[o + i] = out1[pad9(i)], s2[o + i] = out2[pad9(i)];
    __syncthreads();  // out1 / out2 are rewritten by the next row
  }
}

constexpr int kFS = 256;    // threads of a four-column stats block
constexpr int kFSRows = 4;  // rows in flight per thread
static_assert(kFS * 4 == kIC, "a four-column stats block spans one chunk");

template <class Src>
__device__ __forceinline__ void int_stats4_tile(const IntTask &X, const Src &src, int seg, int k,
                                                long long (*rowp)[2][kFS / 32], long long (*wt)[kFS / 32]) {
  const int W = X.W, H = X.H;
  const int R0 = seg * X.seg_rows, R1 = min(R0 + X.seg_rows, H);
  const int c = k * kIC + 4 * (int)threadIdx.x;
  const bool vec = src.vec_ok();
  const bool totals = k + 1 < X.nchunk;  // block-uniform
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  long long cu[4] = {0, 0, 0, 0}, cv[4] = {0, 0, 0, 0};
  for (int r0 = R0; r0 < R1; r0 += kFSRows) {
    typename Src::Raw raw[kFSRows][4];
#pragma unroll
    for (int i = 0; i < kFSRows; ++i) {
      if (r0 + i < R1) {
        src.load4(r0 + i, c, vec, raw[i]);
      } else {
#pragma unroll
        for (int j = 0; j < 4; ++j) raw[i][j] = src.zero();
      }
    }
#pragma unroll
    for (int i = 0; i < kFSRows; ++i) {
      long long su = 0, sv = 0;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        long long x1, x2;
        src.values(raw[i][j], x1, x2);
        cu[j] += x1;
        cv[j] += x2;
        su += x1;
        sv += x2;
      }
      const int r = r0 + i;
      if (!totals || r >= R1) continue;  // block-uniform
      src.warp_sums(su, sv);
      const int g = (r - R0) % kRowGroup;
      if (lane == 0) {
        rowp[g][0][wid] = su;
        rowp[g][1][wid] = sv;
      }
      if (g == kRowGroup - 1 || r == R1 - 1) {  // the group's row totals
        __syncthreads();
        if ((int)threadIdx.x <= g) {
          const int rr = r - g + (int)threadIdx.x;
          long long t1 = 0, t2 = 0;
#pragma unroll
          for (int w = 0; w < kFS / 32; ++w) t1 += rowp[threadIdx.x][0][w], t2 += rowp[threadIdx.x][1][w];
          X.rowsum[(long long)rr * X.nchunk + k] = t1;
          X.rowsum[((long long)H + rr) * X.nchunk + k] = t2;
        }
        __syncthreads();  // rowp is rewritten by the next group
      }
    }
  }
  // chunk-local column prefixes of the column sums: the thread's four
  // columns, then an exclusive block scan over the threads
#pragma unroll
  for (int j = 1; j < 4; ++j) {
    cu[j] += cu[j - 1];
    cv[j] += cv[j - 1];
  }
  long long x1 = cu[3], x2 = cv[3];
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const long long y1 = __shfl_up_sync(0xffffffffu, x1, o), y2 = __shfl_up_sync(0xffffffffu, x2, o);
    if (lane >= o) x1 += y1, x2 += y2;
  }
  if (lane == 31) wt[0][wid] = x1, wt[1][wid] = x2;
  __syncthreads();
  long long e1 = x1 - cu[3], e2 = x2 - cv[3], t1 = 0, t2 = 0;
#pragma unroll
  for (int w = 0; w < kFS / 32; ++w) {
    if (w < wid) e1 += wt[0][w], e2 += wt[1][w];
    t1 += wt[0][w];
    t2 += wt[1][w];
  }
#pragma unroll
  for (int j = 0; j < 4; ++j)
    if (c + j < W) {
      X.colsum[(long long)seg * W + c + j] = e1 + cu[j];
      X.colsum[((long long)X.nseg + seg) * W + c + j] = e2 + cv[j];
    }
  if (threadIdx.x == 0 && totals) {
    X.tiletot[(long long)seg * X.nchunk + k] = t1;
    X.tiletot[((long long)X.nseg + seg) * X.nchunk + k] = t2;
  }
}

// The q integrals of a batch of jobs: block -> job through the batched stage
// offsets, then the job's tile or column block.
__device__ __forceinline__ IntTask job_task(const Job &J) {
  return int_task(J.in.W, J.in.H, J.nseg, J.seg_rows, J.segtot);
}

__global__ void __launch_bounds__(kFS, 3) k_int_stats(const Job *__restrict__ jobs, int njobs) {
  __shared__ long long rowp[kRowGroup][2][kFS / 32];
  __shared__ long long wt[2][kFS / 32];
  const Job &J = jobs[find_job(jobs, njobs, kStRows, blockIdx.x)];
  const IntTask X = job_task(J);
  const int lb = blockIdx.x - J.b0[kStRows];
  const QSource src{J.q, J.in.W};
  int_stats4_tile(X, src, lb / X.nchunk, lb % X.nchunk, rowp, wt);
}

// Whether a launch's images are rough, by one block: the mean bin span (largest
// - smallest) of up to 1024 of their 32-column chunk rows, spread over all of
// them, against the first job's limit (at most 1024 jobs), to its hint when
// that changes (a store to host memory holds up the end of a launch). Short, as
// the block must not outlast the others of its launch (with 4096 rows 512 x 384
// took 41.8 us for 38.2), and here, beside the smallest kernel of every path:
// in k_compact_rows its mere code cost 2400 x 1600 of white noise 185 -> 197 us.
__device__ __noinline__ void report_span(const Job *__restrict__ jobs, int njobs) {
  __shared__ unsigned long long part[32];
  unsigned rows = 0, spans = 0;
  const unsigned long long said = threadIdx.x == 0 ? *jobs[0].said : 0ull;
  const int lg = 10 - (32 - __clz(njobs - 1));  // 2^lg rows of each job
#pragma unroll 4
  for (int i = threadIdx.x; i < njobs << lg; i += blockDim.x) {
    const Job &J = jobs[i >> lg];
    const unsigned total = (unsigned)((J.in.W + 31) >> 5) * (unsigned)J.in.H;
    const unsigned q = (unsigned)i & ((1u << lg) - 1u);
    const unsigned v = __ldg(J.grp + ((unsigned long long)q * total >> lg));  // (some repeat where there are fewer)
    ++rows;
    spans += (v >> 8) - (v & 0xffu);
  }
  rows = __reduce_add_sync(0xffffffffu, rows);
  spans = __reduce_add_sync(0xffffffffu, spans);
  if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = (unsigned long long)rows << 32 | spans;
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned long long t = 0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += part[w];
    const bool rough = (float)(unsigned)t > jobs[0].rough * (float)(unsigned)(t >> 32);
    const unsigned long long say = (unsigned long long)jobs[0].hint_tag << 32 | (rough ? 1u : 0u);
    if (say != said) {
      *jobs[0].said = say;
      *reinterpret_cast<volatile unsigned long long *>(jobs[0].hint) = say;
    }
  }
}

// span: one more block, the last, tells whether the images are rough.
__global__ void __launch_bounds__(kMidCols * kMidGroups)
    k_int_mid(const Job *__restrict__ jobs, int njobs, bool span) {
  __shared__ long long part[2][kMidGroups][kMidCols];
  __shared__ long long leftT[2][kMidBatch];
  if (span && blockIdx.x == gridDim.x - 1) {
    report_span(jobs, min(njobs, 32));
    return;
  }
  const Job &J = jobs[find_job(jobs, njobs, kStCols, blockIdx.x)];
  int_mid_cols(job_task(J), (blockIdx.x - J.b0[kStCols]) * kMidCols, part, leftT);
}

__global__ void __launch_bounds__(kINT, 4) k_int_write(const Job *__restrict__ jobs, int njobs) {
  __shared__ int32_t tile[kIC / 8 * 9];
  __shared__ long long out1[kIC / 8 * 9], out2[kIC / 8 * 9];
  __shared__ long long wt[2][kINT / 32];
  const Job &J = jobs[find_job(jobs, njobs, kStRows, blockIdx.x)];
  const IntTask X = job_task(J);
  const int lb = blockIdx.x - J.b0[kStRows];
  const QSource src{J.q, J.in.W};
  if (J.s_pair)
    int_write_tile<QSource, true>(X, src, J.s1, J.s2, lb / X.nchunk, lb % X.nchunk, tile, out1, out2, wt);
  else
    int_write_tile(X, src, J.s1, J.s2, lb / X.nchunk, lb % X.nchunk, tile, out1, out2, wt);
}

// The backward's fixed-point integral planes of a batch of images: block ->
// image through FixJob::b0_tile / b0_col, then (pair p, tile) or (pair p,
// column block). Pair p of an image: planes u_p and v_p (each W x H), scaled
// by 2^fix_shift(amax[p], nmax[p]) and 2^fix_shift(amax[kMaxFields + p],
// nmax[p]) (the scales the backward converts back with), interleaved into
// the p-th pair plane of dst (two int64 per position); scratch per pair.
__device__ __forceinline__ int find_fix(const FixJob *jobs, int n, bool tiles, int blk) {
  int lo = 0, hi = n - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if ((tiles ? jobs[mid].b0_tile : jobs[mid].b0_col) <= blk) lo = mid; else hi = mid - 1;
  }
  return lo;
}

__device__ __forceinline__ IntTask fix_task(const FixJob &F, int p) {
  return int_task(F.W, F.H, F.nseg, F.seg_rows, F.scratch + (long long)p * F.scratch_stride);
}

__device__ __forceinline__ FixSource fix_source(const FixJob &F, int p) {
  const long long N = (long long)F.pitch * F.H;
  return fix_source_of(F.u + p * N, F.v + p * N, F.W, F.pitch, fix_shift(__ldg(F.amax + p), F.nmax[p]),
                       fix_shift(__ldg(F.amax + kMaxFields + p), F.nmax[p]));
}

__global__ void __launch_bounds__(kFS, 3) k_fix_stats(const FixJob *__restrict__ jobs, int n) {
  __shared__ long long rowp[kRowGroup][2][kFS / 32];
  __shared__ long long wt[2][kFS / 32];
  const FixJob &F = jobs[find_fix(jobs, n, true, blockIdx.x)];
  const int per = F.nseg * ((F.W + kIC - 1) / kIC), lb = blockIdx.x - F.b0_tile;
  const int p = lb / per, t = lb - p * per;
  const IntTask X = fix_task(F, p);
  int_stats4_tile(X, fix_source(F, p), t / X.nchunk, t % X.nchunk, rowp, wt);
}

__global__ void __launch_bounds__(kMidCols * kMidGroups) k_fix_mid(const FixJob *__restrict__ jobs, int n) {
  __shared__ long long part[2][kMidGroups][kMidCols];
  __shared__ long long leftT[2][kMidBatch];
  const FixJob &F = jobs[find_fix(jobs, n, false, blockIdx.x)];
  const int per = (F.W + kMidCols - 1) / kMidCols, lb = blockIdx.x - F.b0_col;
  const int p = lb / per;
  int_mid_cols(fix_task(F, p), (lb - p * per) * kMidCols, part, leftT);
}

__global__ void __launch_bounds__(kINT, 4) k_fix_write(const FixJob *__restrict__ jobs, int n) {
  __shared__ float2 tile[kIC / 8 * 9];
  __shared__ long long out1[kIC / 8 * 9], out2[kIC / 8 * 9];
  __shared__ long long wt[2][kINT / 32];
  const FixJob &F = jobs[find_fix(jobs, n, true, blockIdx.x)];
  const int per = F.nseg * ((F.W + kIC - 1) / kIC), lb = blockIdx.x - F.b0_tile;
  const int p = lb / per, t = lb - p * per;
  const IntTask X = fix_task(F, p);
  const long long plane = ((long long)F.W + 1) * ((long long)F.H + 1);
  long long *d = reinterpret_cast<long long *>(F.dst) + 2 * p * plane;
  int_write_tile<FixSource, true>(X, fix_source(F, p), d, d + 1, t / X.nchunk, t % X.nchunk, tile,
                                             out1, out2, wt);
}

// Integral histogram planes (uint32, modulo 2^32) of a bin map. The rows are
// cut into segments of seg_rows (a multiple of 32) and the columns into strips
// of 128, one warp each:
//   1. k_hist_cols counts, per segment, plane and column, the pixels the plane
//      indicates;
//   2. k_hist_mid, where there are more than kHDirect segments, replaces the
//      counts by those of the segments above (else the next launch adds them
//      up itself: a launch less);
//   3. k_hist_write, a block per segment and plane, walks the strips of the
//      image eight at a time. A warp's accumulators start from the column
//      counts above, summed along the strip; per row, ballots give the
//      indicator masks and the popcounts of their low bits the row prefixes.
//      What lies left of a strip comes from the strips' row totals, exchanged
//      once per 32 rows.
// Where segments x planes leave SMs idle and the rows are long, a segment is
// divided into parts of whole passes, a block each; more blocks of launch 1
// then give the strips' row totals and their sums over a segment, from which a
// part takes what lies left of it (hist_parts has the rule). With one block for
// the whole width 64 x 16384 with 2 bins took 182 us, 256 x 16384 189 and 2160
// x 3840 78 (55, 61 and 72 over the int64 tiles); now 30, 32 and 46.
// Bound by the writes (4 bytes per element; the bin map stays in L2) and by
// issue (105 warp instructions per strip row and plane). 32 planes of 1080p
// (265 MB) took 230 us over the int64 tiles of the integral images and take 90
// (counts 13, writes 77).
constexpr int kHW = 8;                  // strips (warps) of a block's pass
constexpr int kHStrip = 128;            // columns of a strip
constexpr int kHCols = kHW * kHStrip;   // columns of a pass
constexpr int kHDirect = 32;            // segments whose counts the write pass adds up
constexpr int kHBlocks = 152;           // fewer blocks of the write pass than SMs: their segments are divided

struct HistPlanes {
  const uint8_t *bins;
  uint32_t *planes;
  uint32_t *counts;  // nseg x n_planes x W column counts
  int W, H, nseg, seg_rows, n_planes, k_begin, eq;
  int summed;        // the counts have been replaced by those of the segments above
};

// With more than one part of `cols` columns (a multiple of kHCols) per segment,
// or with a side near 2^31: its kernels count columns and rows in unsigned
// (Index), which the ordinary ones would pay for (256 x 256, 8 bins, 22.0 and
// 23.8 us; 100000 x 16, 64 bins, 3910 and 3994).
struct HistParts : HistPlanes {
  int cols;
  uint32_t *segtot;  // nseg x n_planes x strips: the plane's pixels of a segment's strip
  uint8_t *rowtot;   // strips x n_planes x H: of a strip's row
};

template <class Args>
constexpr bool kHParts = std::is_same<Args, HistParts>::value;
template <class Args>
using Index = typename std::conditional<kHParts<Args>, unsigned, int>::type;

// The end of the segment of rows that begins at r0.
template <class Args>
__device__ __forceinline__ int segment_end(const Args &Q, int r0) {
  if (kHParts<Args>) return Q.H - r0 > Q.seg_rows ? r0 + Q.seg_rows : Q.H;
  return min(r0 + Q.seg_rows, Q.H);
}

// Launch 1's other blocks: the totals of strip s in segment seg, per row and
// over the segment. Plane p as in k_hist_cols.
__device__ __forceinline__ void hist_strip_totals(const HistParts &Q, int s, int seg, unsigned *sum) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, strips = (Q.W - 1) / kHStrip + 1;
  const int r0 = seg * Q.seg_rows, r1 = segment_end(Q, r0);
  const int c = s * kHStrip + lane;
  for (int p = threadIdx.x; p < Q.n_planes; p += kHStrip) sum[p] = 0;
  __syncthreads();
  for (unsigned r = r0 + 4 * wid; r < (unsigned)r1; r += kHStrip / 8) {  // four rows per warp and step
    int v[4][4];
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
      for (int m = 0; m < 4; ++m)
        v[u][m] = r + u < (unsigned)r1 && c + 32 * m < Q.W ? (int)__ldg(Q.bins + (size_t)(r + u) * Q.W + c + 32 * m)
                                                          : 256;
    for (int p = 0; p < Q.n_planes; ++p) {
      const int k = Q.k_begin + p;
      unsigned t = 0;  // the rows' totals, a byte each
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        unsigned n = 0;
#pragma unroll
        for (int m = 0; m < 4; ++m) n += Q.eq ? v[u][m] == k : v[u][m] < k;
        t |= n << (8 * u);
      }
      t = __reduce_add_sync(0xffffffffu, t);  // at most 128 each
      if (lane < 4 && r + lane < (unsigned)r1)
        Q.rowtot[((size_t)s * Q.n_planes + p) * Q.H + r + lane] = (uint8_t)(t >> (8 * lane));
      if (lane == 0) atomicAdd(&sum[p], (t & 0xffu) + ((t >> 8) & 0xffu) + ((t >> 16) & 0xffu) + (t >> 24));
    }
  }
  __syncthreads();
  for (int p = threadIdx.x; p < Q.n_planes; p += kHStrip)
    Q.segtot[((size_t)seg * Q.n_planes + p) * strips + s] = sum[p];
}

// Plane p indicates [b == k] (eq) or [b < k], k = k_begin + p.
template <class Args>
__global__ void __launch_bounds__(kHStrip) k_hist_cols(const __grid_constant__ Args Q) {
  extern __shared__ unsigned hcount[];  // [n_planes][kHStrip]
  if constexpr (kHParts<Args>)
    if ((int)blockIdx.y >= Q.nseg) {
      hist_strip_totals(Q, blockIdx.x, blockIdx.y - Q.nseg, hcount);
      return;
    }
  const int c = blockIdx.x * kHStrip + threadIdx.x, seg = blockIdx.y;
  for (int p = 0; p < Q.n_planes; ++p) hcount[p * kHStrip + threadIdx.x] = 0;
  if (c >= Q.W) return;  // (a thread only touches its own column)
  const int r0 = seg * Q.seg_rows, r1 = segment_end(Q, r0);
  const uint8_t *b = Q.bins + (size_t)r0 * Q.W + c;
  for (Index<Args> r = r0; r < (Index<Args>)r1; r += 8) {
    int v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) v[u] = r + u < (Index<Args>)r1 ? (int)__ldg(b + (size_t)u * Q.W) : 256;
#pragma unroll
    for (int u = 0; u < 8; ++u)
      if (v[u] < Q.n_planes) ++hcount[v[u] * kHStrip + threadIdx.x];
    b += (size_t)8 * Q.W;
  }
  uint32_t *o = Q.counts + (size_t)seg * Q.n_planes * Q.W + c;
  unsigned run = 0;
  for (int p = 0; p < Q.n_planes; ++p) {
    const unsigned h = hcount[p * kHStrip + threadIdx.x];
    run += h;
    o[(size_t)p * Q.W] = Q.eq ? h : run;  // [b < k_begin + p] with k_begin = 1: the bins 0 .. p
  }
}

__global__ void __launch_bounds__(128) k_hist_mid(const __grid_constant__ HistPlanes Q) {
  const size_t n = (size_t)Q.n_planes * Q.W, i = (size_t)blockIdx.x * 128 + threadIdx.x;
  if (i >= n) return;
  uint32_t *o = Q.counts + i;
  unsigned run = 0;
  for (int s = 0; s < Q.nseg; s += 8, o += 8 * n) {
    unsigned v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) v[u] = s + u < Q.nseg ? o[u * n] : 0u;
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      if (s + u < Q.nseg) o[u * n] = run;
      run += v[u];
    }
  }
}

__device__ __forceinline__ unsigned warp_inclusive(unsigned v) {
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned y = __shfl_up_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) >= (unsigned)o) v += y;
  }
  return v;
}

// kEq: Q.eq. Args: HistPlanes, or HistParts (undivided segments take 3 to 5 %
// longer with the parts compiled in: 3000 x 4000, 8 bins, 138 and 145 us).
template <bool kEq, class Args>
__global__ void __launch_bounds__(32 * kHW, 5) k_hist_write(const __grid_constant__ Args Q) {
  // [2][seg_rows]: the rows' totals of the passes before, read by one pass
  // while it writes the next one's (only where the image takes several)
  extern __shared__ unsigned left[];
  __shared__ uint4 mask[kHW][32];          // indicator masks of a strip's row, four words of 32 columns
  __shared__ unsigned part[kHW][32];       // and the counts of the first one, two and three words, a byte each
  __shared__ unsigned tot[2][kHW][32];     // row totals of the strips, per batch of 32 rows
  __shared__ unsigned above[kHW];          // totals of the strips in the segments above
  const int W = Q.W, H = Q.H, lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int p = blockIdx.x % Q.n_planes, seg = blockIdx.x / Q.n_planes;
  const int k = Q.k_begin + p;
  const int r0 = seg * Q.seg_rows, r1 = segment_end(Q, r0);
  const size_t W1 = (size_t)W + 1;
  uint32_t *const plane = Q.planes + (size_t)p * W1 * ((size_t)H + 1);
  const bool passes = W > kHCols;
  unsigned carry = 0;  // the passes before: their columns' total in the segments above
  int Cs = 0, Ce = W;  // the block's columns
  if constexpr (kHParts<Args>) {
    Cs = (int)blockIdx.y * Q.cols;
    Ce = W - Cs > Q.cols ? Cs + Q.cols : W;
    const int strips = (W - 1) / kHStrip + 1, s1 = Cs / kHStrip;
    if (seg == 0)
      for (unsigned c = Cs + threadIdx.x; c < (unsigned)Ce; c += 32 * kHW) plane[c + 1] = 0;
    if (seg == 0 && Cs == 0 && threadIdx.x == 0) plane[0] = 0;
    if (Cs == 0)
      for (unsigned r = r0 + threadIdx.x; r < (unsigned)r1; r += 32 * kHW) plane[(size_t)(r + 1) * W1] = 0;
    for (unsigned r = r0 + wid; r < (unsigned)r1 && passes; r += kHW) {  // a warp per row (more parts: more passes)
      const uint8_t *t = Q.rowtot + (size_t)p * H + r;
      unsigned n = 0;
#pragma unroll 8
      for (int s = lane; s < s1; s += 32) n += __ldg(t + (size_t)s * Q.n_planes * H);
      n = __reduce_add_sync(0xffffffffu, n);
      if (lane == 0) left[r - r0] = n;
    }
    for (int q = wid; q < seg; q += kHW)
#pragma unroll 4
      for (int s = lane; s < s1; s += 32) carry += __ldg(Q.segtot + ((size_t)q * Q.n_planes + p) * strips + s);
    carry = __reduce_add_sync(0xffffffffu, carry);
    if (lane == 0) above[wid] = carry;
    __syncthreads();
    carry = 0;
    for (int w = 0; w < kHW; ++w) carry += above[w];
  } else {
    for (int r = threadIdx.x; r < Q.seg_rows && passes; r += 32 * kHW) left[r] = 0;
    if (seg == 0)
      for (int c = threadIdx.x; c <= W; c += 32 * kHW) plane[c] = 0;
    for (int r = r0 + (int)threadIdx.x; r < r1; r += 32 * kHW) plane[(size_t)(r + 1) * W1] = 0;
  }
  const unsigned le = 0xffffffffu >> (31 - lane);
  int flip = 0, par = 0;
  for (Index<Args> C0 = Cs; C0 < (Index<Args>)Ce; C0 += kHCols, par ^= 1) {
    const int c0 = (int)C0 + wid * kHStrip;  // the warp's strip
    unsigned acc[4];                    // columns c0 + 32 m + lane
    bool ok[4];
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      ok[m] = c0 + 32 * m + lane < W;
      acc[m] = 0;
    }
#pragma unroll 4
    for (int q = Q.summed ? seg : 0; q < seg + Q.summed; ++q) {
      const uint32_t *cnt = Q.counts + ((size_t)q * Q.n_planes + p) * W + c0 + lane;
#pragma unroll
      for (int m = 0; m < 4; ++m)
        if (ok[m]) acc[m] += __ldg(cnt + 32 * m);
    }
    unsigned run = 0;
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      acc[m] = warp_inclusive(acc[m]) + run;
      run = __shfl_sync(0xffffffffu, acc[m], 31);
    }
    __syncthreads();  // the pass before has read above (and left is cleared)
    if (lane == 0) above[wid] = run;
    __syncthreads();
    unsigned base = carry;  // P: everything left of the strip, down to the row
    for (int w = 0; w < kHW; ++w) {
      if (w < wid) base += above[w];
      carry += above[w];
    }
    for (Index<Args> rb = r0; rb < (Index<Args>)r1; rb += 32, flip ^= 1) {
      const int n = min(32, r1 - (int)rb);
      const uint8_t *b = Q.bins + (size_t)rb * W + c0 + lane;
      uint4 rw = make_uint4(0u, 0u, 0u, 0u);  // lane = row: its masks
      for (int i = 0; i < n; i += 4) {
        int v[4][4];
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
          for (int m = 0; m < 4; ++m) v[u][m] = i + u < n && ok[m] ? (int)__ldg(b + (size_t)u * W + 32 * m) : 256;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          uint4 w;
          w.x = __ballot_sync(0xffffffffu, kEq ? v[u][0] == k : v[u][0] < k);
          w.y = __ballot_sync(0xffffffffu, kEq ? v[u][1] == k : v[u][1] < k);
          w.z = __ballot_sync(0xffffffffu, kEq ? v[u][2] == k : v[u][2] < k);
          w.w = __ballot_sync(0xffffffffu, kEq ? v[u][3] == k : v[u][3] < k);
          if (lane == i + u) rw = w;
        }
        b += (size_t)4 * W;
      }
      mask[wid][lane] = rw;
      const unsigned t0 = __popc(rw.x), t1 = t0 + __popc(rw.y), t2 = t1 + __popc(rw.z);
      part[wid][lane] = t0 | (t1 << 8) | (t2 << 16);
      const unsigned mine = t2 + __popc(rw.w);
      tot[flip][wid][lane] = mine;
      __syncthreads();  // (tot is double buffered: one barrier per batch)
      unsigned row = passes && lane < n ? left[par * Q.seg_rows + rb - r0 + lane] : 0u, all = row;
      for (int w = 0; w < kHW; ++w) {
        const unsigned t = tot[flip][w][lane];
        if (w < wid) row += t;
        all += t;
      }
      const unsigned P = warp_inclusive(row) + base;
      base = __shfl_sync(0xffffffffu, P, 31);
      uint32_t *o = plane + (size_t)(rb + 1) * W1 + c0 + 1 + lane;
#pragma unroll 4
      for (int i = 0; i < n; ++i) {
        const uint4 w = mask[wid][i];
        const unsigned t = part[wid][i], off = __shfl_sync(0xffffffffu, P, i);
        acc[0] += __popc(w.x & le);
        acc[1] += (t & 0xffu) + __popc(w.y & le);
        acc[2] += ((t >> 8) & 0xffu) + __popc(w.z & le);
        acc[3] += (t >> 16) + __popc(w.w & le);
#pragma unroll
        for (int m = 0; m < 4; ++m)
          if (ok[m]) o[32 * m] = acc[m] + off;
        o += W1;
      }
      __syncwarp();  // mask is rewritten by the next batch
      if (passes && wid == 0 && lane < n) left[(par ^ 1) * Q.seg_rows + rb - r0 + lane] = all;
    }
  }
}

}  // namespace

void integral_layout(int W, int H, size_t max_scratch_elems, int tiles, int &nseg, int &seg_rows) {
  // the shortest segments (most tiles) whose scratch fits, at least kIR rows;
  // fewer, down to four, where that gives no more than `tiles` tiles: a tile's
  // rows are a serial chain of barriers (16 rows 15 us, of 45 for a forward at
  // 512 x 384)
  seg_rows = kIR;
  const long long chunks = (W + kIC - 1) / kIC;
  while (seg_rows > 4 && (H + seg_rows / 2 - 1) / (seg_rows / 2) * chunks <= tiles) seg_rows /= 2;
  for (;;) {
    nseg = (H + seg_rows - 1) / seg_rows;
    if (integral_scratch_elems(W, H, nseg) <= max_scratch_elems || seg_rows >= H) return;
    seg_rows = std::min(H, seg_rows * 2);
  }
}

size_t integral_scratch_elems(int W, int H, int nseg) {
  const long long nchunk = (W + kIC - 1) / kIC;
  return (size_t)(2LL * nseg * W + 2LL * H * nchunk + 2LL * nseg * nchunk);
}

int integral_tile_blocks(int W, int nseg) { return nseg * ((W + kIC - 1) / kIC); }

int integral_col_blocks(int W) { return (W + kMidCols - 1) / kMidCols; }

// Row segments of an image's fixed-point pairs in a batch whose pairs, over
// all images, number `batch_pairs`: short enough for about 512 tiles over the
// batch, 4 to kIR rows (the three launches at 1599 x 1199, three pairs, for
// 4096, 2048, 1024 and 512 tiles: 89, 89, 85 and 81 us).
void fix_layout(int W, int H, long long batch_pairs, int &nseg, int &seg_rows) {
  const long long tiles_per_row = batch_pairs * ((W + kIC - 1) / kIC);
  seg_rows = (int)std::min<long long>(kIR, std::max<long long>(4, H * tiles_per_row / 512));
  nseg = (H + seg_rows - 1) / seg_rows;
}

size_t fix_integral_scratch_elems(int W, int H, int pairs, int nseg) {
  return (size_t)pairs * integral_scratch_elems(W, H, nseg);
}

int fix_tile_blocks(int W, int nseg, int pairs) { return pairs * integral_tile_blocks(W, nseg); }

int fix_col_blocks(int W, int pairs) { return pairs * integral_col_blocks(W); }

int launch_fix_integrals(const FixJob *jobs, int n, int tile_blocks, int col_blocks, cudaStream_t s) {
  k_fix_stats<<<tile_blocks, kFS, 0, s>>>(jobs, n);
  k_fix_mid<<<col_blocks, kMidCols * kMidGroups, 0, s>>>(jobs, n);
  k_fix_write<<<tile_blocks, kINT, 0, s>>>(jobs, n);
  return 3;
}

int launch_integral_jobs(const Job *jobs, int njobs, int tile_blocks, int col_blocks, bool span, cudaStream_t s) {
  k_int_stats<<<tile_blocks, kFS, 0, s>>>(jobs, njobs);
  k_int_mid<<<col_blocks + (span ? 1 : 0), kMidCols * kMidGroups, 0, s>>>(jobs, njobs, span);
  k_int_write<<<tile_blocks, kINT, 0, s>>>(jobs, njobs);
  return 3;
}

// Segments of 64 rows, longer (a multiple of 32) where there would be more
// than 4096 of them.
static void hist_layout(int H, int &nseg, int &seg_rows) {
  seg_rows = 64;
  const long long most = 4096LL * 64;
  if (H > most) seg_rows = (int)(((long long)H + 4095) / 4096 + 31) / 32 * 32;
  nseg = (int)(((long long)H + seg_rows - 1) / seg_rows);
}

// The parts of a segment, of whole passes: where there are fewer blocks than
// SMs, as many as give two per SM, if the passes that a block is spared (about
// 1 us + 0.16 us per row each) take longer than the strips' totals (0.6 us per
// plane). 64 rows of 2048 columns, undivided and in parts, us: 8 bins 34.6 and
// 27.9, 16 34.9 and 32.1, 32 35.5 and 40.1, 64 36 and 56; of 16384 columns, 64
// bins 254 and 131, 256 bins 330 and 445. With 256 blocks (512 x 4096, 32 bins)
// 105 undivided and 110.
static void hist_parts(int W, int H, int nseg, int seg_rows, int planes, int &parts, int &cols) {
  const long long pass = ((long long)W + kHCols - 1) / kHCols, blocks = (long long)nseg * planes;
  const long long want = blocks < kHBlocks ? std::min(pass, (2 * kHBlocks + blocks - 1) / blocks) : 1;
  long long per = (pass + want - 1) / want;
  if ((pass - per) * (1.0 + 0.16 * std::min(seg_rows, H)) < 0.6 * planes) per = pass;
  cols = (int)std::min<long long>(per * kHCols, W);
  parts = (int)((W + (long long)cols - 1) / cols);
}

size_t hist_scratch_bytes(int W, int H, int planes) {
  int nseg, seg_rows, parts, cols;
  hist_layout(H, nseg, seg_rows);
  planes = std::max(planes, 1);
  hist_parts(W, H, nseg, seg_rows, planes, parts, cols);
  const size_t counts = sizeof(uint32_t) * (size_t)planes * nseg * W, strips = ((size_t)W + kHStrip - 1) / kHStrip;
  return counts + (parts > 1 ? strips * planes * (sizeof(uint32_t) * nseg + H) : 0);
}

template <class Args>
static int launch_hist(Args Q, int parts, cudaStream_t s) {
  const size_t smem = sizeof(unsigned) * kHStrip * (size_t)Q.n_planes;  // at most 128 KB
  cudaFuncSetAttribute(k_hist_cols<Args>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                       (int)(sizeof(unsigned) * kHStrip * kMaxBins));
  k_hist_cols<Args><<<dim3((unsigned)((Q.W - 1) / kHStrip + 1), (unsigned)(parts > 1 ? 2 * Q.nseg : Q.nseg)),
                      kHStrip, smem, s>>>(Q);
  Q.summed = Q.nseg > kHDirect ? 1 : 0;
  if (Q.summed) k_hist_mid<<<(unsigned)(((size_t)Q.n_planes * Q.W + 127) / 128), 128, 0, s>>>(Q);
  auto *const write = Q.eq ? k_hist_write<true, Args> : k_hist_write<false, Args>;
  const size_t left = Q.W > kHCols ? 2 * sizeof(unsigned) * (size_t)Q.seg_rows : 0;
  if (left > 40 * 1024)  // (more than 20 M rows)
    cudaFuncSetAttribute(write, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
  write<<<dim3((unsigned)(Q.nseg * Q.n_planes), (unsigned)parts), 32 * kHW, left, s>>>(Q);
  return 2 + Q.summed;
}

int launch_integral_histogram(const uint8_t *bins, int W, int H, int n_bins, bool cumulative,
                              uint32_t *planes, void *scratch, cudaStream_t s) {
  HistParts Q{};
  Q.bins = bins;
  Q.planes = planes;
  Q.counts = static_cast<uint32_t *>(scratch);
  Q.W = W;
  Q.H = H;
  Q.k_begin = cumulative ? 1 : 0;
  Q.n_planes = cumulative ? n_bins - 1 : n_bins;
  Q.eq = cumulative ? 0 : 1;
  if (Q.n_planes <= 0) return 0;
  hist_layout(H, Q.nseg, Q.seg_rows);
  int parts;
  hist_parts(W, H, Q.nseg, Q.seg_rows, Q.n_planes, parts, Q.cols);
  constexpr int kFar = INT_MAX - (1 << 20);  // (int counters may not pass a side by a step)
  if (parts > 1 || W > kFar || H > kFar) {
    const size_t strips = ((size_t)W + kHStrip - 1) / kHStrip;
    Q.segtot = Q.counts + (size_t)Q.nseg * Q.n_planes * W;
    Q.rowtot = reinterpret_cast<uint8_t *>(Q.segtot + (size_t)Q.nseg * Q.n_planes * strips);
    return launch_hist<HistParts>(Q, parts, s);
  }
  return launch_hist<HistPlanes>(Q, 1, s);
}

}  // namespace tmk
