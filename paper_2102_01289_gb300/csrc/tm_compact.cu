// tm_compact.cu -- the Eq. 1 numerators from a compact form of the cumulative
// integral histogram.
//
// For a threshold k let C_k(u, p) be the integral histogram in cumulative form
// (Eq. 7-8 summed over the bins below k): the pixels of the first p rows and
// first u columns whose bin is below k. Eq. 9 takes four of its values per
// field and pixel. Written out it is n - 1 planes of the image's size (3 GB at
// 12 MP with 64 bins); here it is kept per 32-column chunk instead, as
//     C_k(u, p) = PT + o m + B[o]          c = u / 32, o = u mod 32,
// a record per (chunk c, row position p, threshold k) with
//     PT  the pixels below k of the first p rows in the chunks left of c,
//     m   the rows (of the first p) in which all of chunk c lies below k, and
//     the count j of the rows in which chunk c holds bins on both sides of k
//     ("mixed" rows), which names the vector
//     B[o] (slot j of the chunk and threshold): the sum over those rows of the
//         chunk's pixels below k left of column o.
// A vector is written only at a mixed row, so column work is paid only where a
// bin edge crosses a chunk: at 12 MP, 64 bins, the records are 192 MB and the
// vectors of one photograph-like scene about 40 MB. Forwards, against the
// sweep: 12 MP, 64 bins, 736 -> 502 us; with noise of 0.3 decades 1006 -> 709;
// 1080p, 32 bins, 199 -> 116. White noise (every chunk row mixed for every
// threshold) is its worst case: 1080p 281 -> 238, but 12 MP 1733 -> 2538 (the
// automatic path measures such images and leaves them to the sweep).
// Differences between two rows are taken modulo the width of m and B, so B is
// 16 bits wide unless a window is taller than 65535 / 31 rows.
//
// Three launches per group of images:
//   1. k_compact_rows: the prefix over the chunks of each row's counts below k
//      (lanes = thresholds, walking along the row);
//   2. k_compact_cols, a cluster of CTAs per chunk and group of
//      thresholds: its warps take consecutive row segments twice (lanes =
//      thresholds, walking down the rows), once for the segments' totals and,
//      after a scan of the totals over the segments, to write records and
//      vectors;
//   3. k_lookup_compact, a thread per column and a few rows: four records and
//      up to four vector entries per field and pixel, then the lookup's
//      arithmetic.
// Thresholds come in groups of KL (64, or 4, 8, 16, 32 where n - 1 is no
// larger), a group of 64 two adjacent ones to a lane.
// The bin ranges of the chunks come from the group summary of the bin pass.
#include <cooperative_groups.h>

#include <algorithm>

#include "tm_kernels.cuh"
#include "tm_lookup.cuh"

namespace tmk {
namespace {

constexpr int kRowWarps = 8;  // warps of a k_compact_rows block
// Rows of a segment of k_compact_cols, at most (up to eight CTAs per chunk): 16
// uneven images, up to 4096 x 3072, took 3171 us with segments of 192 rows, 3055
// with 96, 3085 and 3093 with 64 and 48.
constexpr int kSegRows = 96;
// A group of KL thresholds takes T adjacent ones per lane (lanes past KL / T
// hold none).
template <int KL>
struct Shape {
  static constexpr int T = KL == 64 ? 2 : 1;
  static constexpr int Step = 4;                         // rows or chunks in flight together
  // the column pass loads the next rows while it works on these, where the
  // registers allow (31 thresholds, 1080p: the build 55 -> 50 us; 63, 12 MP:
  // spills, 194 -> 214)
  static constexpr bool Ahead = T == 1;
  static constexpr int ColWarps = 16;                    // row segments of a CTA
  static constexpr int MinBlocks = 2;                    // 64 registers
  // column CTAs share a chunk's rows until the launch has this many warps.
  // 12 MP, 63 thresholds, a forward with clusters of 2, 4, 8: 549, 536, 563
  // us; 1080p, 31 thresholds, 4 and 8: 127 and 133; 32 1080p images in one
  // launch, 1 and 4: 9.49 and 9.75 ms per 120 (short segments pay more for
  // their totals, long ones leave the rows of a vertical edge to one warp);
  // the pyramid at 12 MP, 4 thresholds, up to 4000, 8000 and 16000 warps: the
  // build 89, 81 and 87 us (125 with eight segments to a warp).
  static constexpr int Fill = KL == 64 ? 4864 : KL == 32 ? 3600 : 8000;
};

// Whether a chunk row with bins in [g & 255, g >> 8] has bins on both sides of
// some threshold of the group (k0 + 1 .. k0 + KL).
template <int KL>
__device__ __forceinline__ bool mixed_range(unsigned g, int k0) {
  return max((int)(g & 0xffu), k0) < min((int)(g >> 8), k0 + KL);
}

// Its thresholds k0 + 1 + t are t0 <= t < t1.
template <int KL>
__device__ __forceinline__ void mixed_thresholds(unsigned g, int k0, int &t0, int &t1) {
  t0 = max((int)(g & 0xffu) - k0, 0);
  t1 = min((int)(g >> 8) - k0, KL);
}

constexpr unsigned kNoRow = 0xffffu;  // a bin range on no threshold's lower side

// T adjacent uint16 as one load, and T records as one store.
template <int T>
__device__ __forceinline__ void load_prefix(const uint16_t *p, unsigned *v) {
  if (T == 2) {
    const unsigned w = __ldg(reinterpret_cast<const unsigned *>(p));
    v[0] = w & 0xffffu;
    v[T - 1] = w >> 16;
  } else {
    v[0] = __ldg(p);
  }
}
template <int T>
__device__ __forceinline__ void store_records(uint2 *p, const unsigned *pt, const unsigned *mc) {
  if (T == 2) *reinterpret_cast<uint4 *>(p) = make_uint4(pt[0], mc[0], pt[T - 1], mc[T - 1]);
  else *p = make_uint2(pt[0], mc[0]);
}

// Rows: a warp per row, lane = T thresholds, walking along the row's chunks.
template <int KL>
__global__ void __launch_bounds__(32 * kRowWarps) k_compact_rows(const Job *__restrict__ jobs, int njobs, int K) {
  using S = Shape<KL>;
  constexpr int T = S::T;
  const Job &J = jobs[find_job(jobs, njobs, kStCRows, blockIdx.x)];
  const int lane = threadIdx.x & 31;
  const int W = J.in.W, H = J.in.H, G = (W + 31) >> 5, Gp = (W >> 5) + 1;
  const int rb = (H + kRowWarps - 1) / kRowWarps;
  const int lb = blockIdx.x - J.b0[kStCRows];
  const int kg = lb / rb, k0 = KL * kg;
  const int v = (lb - kg * rb) * kRowWarps + (threadIdx.x >> 5);
  if (v >= H) return;
  const bool own = T * lane < KL;
  const unsigned k8 = (unsigned)(k0 + 1 + T * lane) << 8;  // the lane's first threshold
  const uint8_t *__restrict__ bins = J.bins + (size_t)v * W + lane;
  const uint16_t *__restrict__ grow = J.grp + (size_t)v * G;
  const size_t cstride = (size_t)H * KL;
  uint16_t *__restrict__ dst = J.c_row + ((size_t)kg * Gp * H + v) * KL + T * lane;
  unsigned run[T];
#pragma unroll
  for (int z = 0; z < T; ++z) run[z] = 0;
  for (int cb = 0; cb < Gp; cb += 32) {
    const unsigned gl = cb + lane < G ? (unsigned)__ldg(grow + cb + lane) : kNoRow;
    const unsigned mixed = __ballot_sync(0xffffffffu, mixed_range<KL>(gl, k0));  // bit = chunk of the batch
    const int n = min(32, Gp - cb);
    const auto fetch = [&](int i, int *b) {  // the lane's bins of chunks i .. of the batch, where they are mixed
#pragma unroll
      for (int u = 0; u < S::Step; ++u) {
        const int col = 32 * (cb + i + u);
        b[u] = 256;
        if (i + u < 32 && ((mixed >> ((i + u) & 31)) & 1u) && col + lane < W) b[u] = (int)__ldg(bins + col);
      }
    };
    int nb[S::Step];
    fetch(0, nb);
    for (int i = 0; i < n; i += S::Step) {
      int b[S::Step];
#pragma unroll
      for (int u = 0; u < S::Step; ++u) b[u] = nb[u];
      fetch(i + S::Step, nb);  // in flight meanwhile
#pragma unroll
      for (int u = 0; u < S::Step; ++u) {
        if (i + u >= n) break;
        const unsigned g = __shfl_sync(0xffffffffu, gl, i + u);
        if (own) {
          if (T == 2) *reinterpret_cast<unsigned *>(dst) = run[0] | (run[T - 1] << 16);
          else *dst = (uint16_t)run[0];
        }
        dst += cstride;
        unsigned cc[T];
#pragma unroll
        for (int z = 0; z < T; ++z) cc[z] = g < k8 + 256u * z ? 32u : 0u;  // every bin of the chunk below k
        if ((mixed >> (i + u)) & 1u) {
          int t0, t1;
          mixed_thresholds<KL>(g, k0, t0, t1);
          for (int t = t0 / T * T; t < t1; t += T) {
#pragma unroll
            for (int z = 0; z < T; ++z) {
              const unsigned mask = __ballot_sync(0xffffffffu, b[u] <= k0 + t + z);  // bins below k0 + 1 + t + z
              if (lane == t / T) cc[z] = (unsigned)__popc(mask);
            }
          }
        }
#pragma unroll
        for (int z = 0; z < T; ++z) run[z] += cc[z];
      }
    }
  }
}

// The lane's state over its rows: T thresholds' pt and mc = m | (mixed rows)
// << 16, and mh, the mixed rows wholly below the threshold (first pass only).
template <int T>
struct ColState {
  unsigned pt[T], mc[T], mh[T];
};

// A warp's pass over rows [row0, rend) of chunk c: lane = T thresholds. kWrite:
// write records and vectors; sB[t][o] holds the vectors (lane = column o
// there). Else sB counts, per t and column, the pixels of the mixed rows with
// bin k0 + t (k0 or less for t = 0).
template <int KL, class BT, bool kWrite>
__device__ __forceinline__ void col_pass(const Job &J, int c, int kg, int K, int row0, int rend, BT *sB,
                                         ColState<Shape<KL>::T> &st) {
  using S = Shape<KL>;
  constexpr int T = S::T;
  const int lane = threadIdx.x & 31;
  const int W = J.in.W, H = J.in.H, G = (W + 31) >> 5, Gp = (W >> 5) + 1;
  const int k0 = KL * kg;
  const unsigned k8 = (unsigned)(k0 + 1 + T * lane) << 8;
  const bool own = T * lane < KL;
  const unsigned lt = (1u << lane) - 1u;
  const bool colok = 32 * c + lane < W;
  const uint8_t *__restrict__ bins = J.bins + (size_t)row0 * W + 32 * c + lane;
  const uint16_t *__restrict__ grp = J.grp + (size_t)(row0 + lane) * G + c;
  const size_t plane = (size_t)kg * Gp + c;
  const uint16_t *__restrict__ row = J.c_row + (plane * H + row0) * KL + T * lane;
  uint2 *__restrict__ rec = J.c_rec + (plane * (H + 1) + row0 + 1) * KL + T * lane;
  BT *__restrict__ vec = static_cast<BT *>(J.c_vec) + ((size_t)c * K + k0) * (H + 1) * 32 + lane;
  const unsigned vstep = (unsigned)(H + 1);
  for (int rb = row0; rb < rend; rb += 32) {
    const int n = min(32, rend - rb);
    const unsigned gl = c < G && lane < n ? (unsigned)__ldg(grp) : kNoRow;
    grp += (size_t)32 * G;
    const unsigned mixed = __ballot_sync(0xffffffffu, mixed_range<KL>(gl, k0));  // bit = row of the batch
    const auto fetch = [&](int i, unsigned (*rp)[T], int *b) {  // rows i .. of the batch: prefixes, mixed rows' bins
#pragma unroll
      for (int u = 0; u < S::Step; ++u) {
#pragma unroll
        for (int z = 0; z < T; ++z) rp[u][z] = 0;
        if (own && i + u < n) load_prefix<T>(row + (i + u) * KL, rp[u]);
        b[u] = 256;
        if (i + u < 32 && ((mixed >> ((i + u) & 31)) & 1u) && colok)
          b[u] = (int)__ldg(bins + (size_t)(unsigned)(i + u) * W);
      }
    };
    unsigned nrp[S::Step][T];
    int nb[S::Step];
    if (S::Ahead) fetch(0, nrp, nb);
    for (int i = 0; i < n; i += S::Step) {
      unsigned rp[S::Step][T];
      int b[S::Step];
      if (S::Ahead) {
#pragma unroll
        for (int u = 0; u < S::Step; ++u) {
#pragma unroll
          for (int z = 0; z < T; ++z) rp[u][z] = nrp[u][z];
          b[u] = nb[u];
        }
        fetch(i + S::Step, nrp, nb);
      } else {
        fetch(i, rp, b);
      }
#pragma unroll
      for (int u = 0; u < S::Step; ++u) {
        // (rows past the segment have no bins below or on both sides)
        const unsigned g = __shfl_sync(0xffffffffu, gl, i + u);
#pragma unroll
        for (int z = 0; z < T; ++z) {
          st.pt[z] += rp[u][z];
          if (g < k8 + 256u * z) ++st.mc[z];
        }
        if ((mixed >> (i + u)) & 1u) {
#pragma unroll
          for (int z = 0; z < T; ++z) {
            const unsigned kz = k8 + 256u * z;
            if (g >= kz && ((g & 0xffu) << 8) < kz) st.mc[z] += 0x10000u;  // bins on both sides
            if (!kWrite && g < kz) ++st.mh[z];
          }
          if (!kWrite) {
            const int h = max(b[u] - k0, 0);
            if (h < KL) {
              BT *const s = sB + h * 32 + lane;
              *s = (BT)(*s + 1);
            }
          } else {
            int t0, t1;
            mixed_thresholds<KL>(g, k0, t0, t1);
            for (int t = t0 / T * T; t < t1; t += T) {
              BT *const s = sB + t * 32 + lane;
              unsigned slot[T];
              BT val[T];
#pragma unroll
              for (int z = 0; z < T; ++z) {
                const unsigned mask = __ballot_sync(0xffffffffu, b[u] <= k0 + t + z);
                slot[z] = __shfl_sync(0xffffffffu, st.mc[z], t / T) >> 16;
                val[z] = (BT)(s[z * 32] + __popc(mask & lt));
              }
#pragma unroll
              for (int z = 0; z < T; ++z)
                if (t + z >= t0 && t + z < t1) {
                  s[z * 32] = val[z];
                  vec[(size_t)((unsigned)(t + z) * vstep + slot[z]) * 32] = val[z];
                }
            }
          }
        }
        if (kWrite && own && i + u < n) store_records<T>(rec + u * KL, st.pt, st.mc);
      }
      rec += S::Step * KL;
    }
    row += 32 * KL;
    bins += (size_t)32 * W;
  }
}

// Columns: cluster -> (image, chunk, threshold group), CTA -> a share of the
// rows, a segment of them per warp.
template <int KL, class BT>
__global__ void __launch_bounds__(32 * Shape<KL>::ColWarps, KL == 64 && sizeof(BT) == 4 ? 1 : Shape<KL>::MinBlocks)
    k_compact_cols(const Job *__restrict__ jobs, int njobs, int K) {
  using S = Shape<KL>;
  constexpr int T = S::T, NW = S::ColWarps;
  namespace cg = cooperative_groups;
  extern __shared__ __align__(16) unsigned char smem[];
  BT *const sB = reinterpret_cast<BT *>(smem);                  // [NW][KL][32]
  BT *const sT = sB + NW * KL * 32;                             // [KL][32]: the CTA's totals
  uint2 *const tot = reinterpret_cast<uint2 *>(sT + KL * 32);   // [NW + 1][KL], the last: the CTA's totals
  cg::cluster_group cluster = cg::this_cluster();
  const int rank = (int)cluster.block_rank(), nc = (int)cluster.num_blocks();
  const Job &J = jobs[find_job(jobs, njobs, kStCCols, blockIdx.x / nc)];
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int H = J.in.H, Gp = (J.in.W >> 5) + 1;
  const int lb = blockIdx.x / nc - J.b0[kStCCols];
  const int kg = lb / Gp, c = lb - kg * Gp;
  const bool own = T * lane < KL;
  const int share = (H + nc - 1) / nc, per = (share + NW - 1) / NW;
  const int row0 = rank * share + wid * per, rend = min(min(row0 + per, (rank + 1) * share), H);
  BT *const mine = sB + wid * KL * 32;
  for (int i = lane; i < KL * 32 * (int)sizeof(BT) / 4; i += 32) reinterpret_cast<unsigned *>(mine)[i] = 0;
  __syncwarp();
  ColState<T> st{};
  col_pass<KL, BT, false>(J, c, kg, K, row0, rend, mine, st);
  uint2 *const mytot = tot + wid * KL + T * lane;
#pragma unroll
  for (int z = 0; z < T; ++z)
    if (own) mytot[z] = make_uint2(st.pt[z], st.mc[z]);
  // per segment: the vectors' totals from the column counts (the pixels of
  // mixed rows below k, less those of rows wholly below it, left of o)
  unsigned any[T];
#pragma unroll
  for (int z = 0; z < T; ++z) any[z] = __ballot_sync(0xffffffffu, own && (st.mc[z] >> 16));
  if (any[0] | any[T - 1]) {
    __syncwarp();
    unsigned below = 0;
#pragma unroll 2
    for (int t = 0; t < KL / T; ++t) {
#pragma unroll
      for (int z = 0; z < T; ++z) {
        BT *const s = mine + (T * t + z) * 32 + lane;
        below += *s;
        unsigned e = 0;
        if ((any[z] >> t) & 1u) {
          const unsigned v = below - __shfl_sync(0xffffffffu, st.mh[z], t);
          e = v;
#pragma unroll
          for (int o = 1; o < 32; o <<= 1) {
            const unsigned y = __shfl_up_sync(0xffffffffu, e, o);
            if (lane >= o) e += y;
          }
          e -= v;
        }
        *s = (BT)e;
      }
    }
  }
  __syncthreads();
  for (int e = tid; e < KL * 32; e += 32 * NW) {
    unsigned t = 0;
#pragma unroll 4
    for (int w = 0; w < NW; ++w) t += sB[w * KL * 32 + e];
    sT[e] = (BT)t;
  }
  if (tid < KL) {
    uint2 t = make_uint2(0u, 0u);
    for (int w = 0; w < NW; ++w) {
      const uint2 x = tot[w * KL + tid];
      t.x += x.x, t.y += x.y;
    }
    tot[NW * KL + tid] = t;
  }
  cluster.sync();
  // exclusive scans over the cluster's segments
  for (int e = tid; e < KL * 32; e += 32 * NW) {
    unsigned run = 0;
    for (int r = 0; r < rank; ++r) run += cluster.map_shared_rank(sT, r)[e];
#pragma unroll 4
    for (int w = 0; w < NW; ++w) {
      BT *const s = sB + w * KL * 32 + e;
      const unsigned v = *s;
      *s = (BT)run;
      run += v;
    }
  }
  if (tid < KL) {
    uint2 run = make_uint2(0u, 0u);
    for (int r = 0; r < rank; ++r) {
      const uint2 x = cluster.map_shared_rank(tot, r)[NW * KL + tid];
      run.x += x.x, run.y += x.y;
    }
    for (int w = 0; w < NW; ++w) {
      const uint2 x = tot[w * KL + tid];
      tot[w * KL + tid] = run;
      run.x += x.x, run.y += x.y;
    }
  }
  cluster.sync();  // also: no CTA ends while another reads its totals
  if (rank == 0 && wid == 0) {
    uint2 *const rec = J.c_rec + ((size_t)kg * Gp + c) * (H + 1) * KL;
    for (int t = lane; t < KL; t += 32) rec[t] = make_uint2(0u, 0u);
    // slot 0 of every threshold: no mixed row yet
    BT *vec = static_cast<BT *>(J.c_vec) + (size_t)c * K * (H + 1) * 32 + lane;
    for (int t = KL * kg; t < min(KL * kg + KL, K); ++t) vec[(size_t)t * (H + 1) * 32] = 0;
  }
#pragma unroll
  for (int z = 0; z < T; ++z) {
    const uint2 x = own ? mytot[z] : make_uint2(0u, 0u);
    st.pt[z] = x.x;
    st.mc[z] = x.y;
  }
  col_pass<KL, BT, true>(J, c, kg, K, row0, rend, mine, st);
}

// What a launch does beside writing the output image.
// kOut: nothing; kOutKeep: also the count planes and window moments for the
// backward; kCountsOnly: only the count planes, no output; kCountsMom: the
// count planes and moments, no output.
enum { kOut = 0, kOutKeep = 1, kCountsOnly = 2, kCountsMom = 3 };

// The images of a lookup launch travel as kernel parameters: every block reads
// its image's pointers and sizes from constant memory, as uniform values.
struct LookJob {
  Image in, out;
  const uint8_t *bins;
  const uint2 *rec;
  const void *vec;
  const longlong2 *s12;
  unsigned *cnt;      // count planes (or null), field f's at cnt + f * cnt_step
  float2 *mom;        // window moments (or null)
  DebugPlanes dbg;
  long long cnt_step;
  int qbits, shift, b0, pad;
};
struct LookPack {
  LookJob j[kCompactImages];
  int n, rows;
};

// A block covers 128 columns x `rows` rows, a thread one column: what depends
// on the column (the windows' left and right edges, their chunks) is formed
// once for its rows, and what depends on the row is uniform. kPlain: no debug
// planes and the literal area is off; kSmall as for window_variance; kDt as
// for k_lookup_counts. kMode: kOut the output only; kOutKeep also the count
// planes and window moments for the backward; kCountsOnly only the count
// planes.
// Bound by issue (72 % of the active cycles), the L1's wavefronts (63 %) and
// load latency; a pixel takes 12 record, 12 vector and 12 corner loads. At
// 12 MP, three fields, seven blocks per SM (72 registers) and three fields'
// loads in flight took 252 us; 6, 8, 9 and 10 blocks 290, 265, 265 and 298; two
// fields at a time 283. Before the moments moved between the records and the
// vectors and the powers behind the vectors' loads it took 272, with
// descriptors read from global memory instead of the parameters 372.
constexpr int kLookCols = 128;
constexpr int kFieldBatch = 3;

template <int NF, class BT, bool kPlain, int kSmall, int kDt, int kMode>
__global__ void __launch_bounds__(kLookCols, 7)
    k_lookup_compact(const __grid_constant__ DevParams P, const __grid_constant__ LookPack L) {
  int jb = 0;
  while (jb + 1 < L.n && L.j[jb + 1].b0 <= (int)blockIdx.x) ++jb;
  const LookJob &J = L.j[jb];
  const int W = J.in.W, H = J.in.H;
  const int bx = (W + kLookCols - 1) / kLookCols;
  const int lb = blockIdx.x - J.b0, by = lb / bx;
  const int x = (lb - by * bx) * kLookCols + (int)threadIdx.x;
  if (x >= W) return;
  const int K = P.n_bins - 1, incl = (P.flags & kFlagCdfIncl) ? 1 : 0, shift = J.shift;
  const unsigned cstep = (unsigned)(H + 1) << shift;         // records per chunk
  const unsigned gstep = ((unsigned)(W >> 5) + 1u) * cstep;  // per threshold group
  const unsigned slots = (unsigned)(H + 1);                  // vectors per threshold
  const uint2 *__restrict__ rec = J.rec;
  const BT *__restrict__ vec = static_cast<const BT *>(J.vec);
  const float inv_scale = ldexpf(1.f, -J.qbits);
  const float inv_scale2 = inv_scale * inv_scale;
  const int y0 = by * L.rows, yend = min(y0 + L.rows, H);
  int t = (int)__ldg(J.bins + ((unsigned)y0 * (unsigned)W + (unsigned)x)) + incl;
#pragma unroll 1
  for (int y = y0; y < yend; ++y) {
    const unsigned pix = (unsigned)y * (unsigned)W + (unsigned)x;
    const bool look = t > 0 && t <= K;
    const unsigned k = look ? (unsigned)(t - 1) : 0u;  // (record and vector loads of threshold 1 where none is needed)
    const bool whole = t > K;
    if (y + 1 < yend) t = (int)__ldg(J.bins + pix + W) + incl;
    const unsigned kofs = (k >> 6) * gstep + (k & 63u);  // (one group up to 64 thresholds)
    float rgb[3], pw[3];
    unsigned black = 0;
    if (kMode < kCountsOnly) load_rgb<kDt>(J.in, x, y, rgb[0], rgb[1], rgb[2]);
    Fusion fu;
    // fields in batches whose loads are in flight together: all records, the
    // moments while they arrive, all vector entries (slot 0 where no row is
    // mixed), and the colour powers while those arrive
#pragma unroll
    for (int f0 = 0; f0 < NF; f0 += kFieldBatch) {
      unsigned cnt[kFieldBatch];
      uint2 r[kFieldBatch][4];
      unsigned e[kFieldBatch][4];
      float var[kFieldBatch], rarea[kFieldBatch];
#pragma unroll
      for (int i = 0; i < kFieldBatch && f0 + i < NF; ++i) {
        const int f = f0 + i;
        const unsigned ul = (unsigned)max(x - P.rx[f], 0), ur = (unsigned)min(x + P.rx[f], W - 1) + 1u;
        const unsigned p0 = (unsigned)max(y - P.ry[f], 0), p1 = (unsigned)min(y + P.ry[f], H - 1) + 1u;
        const unsigned cl = (ul >> 5) * cstep + kofs, cr = (ur >> 5) * cstep + kofs;
        const uint2 *ra = rec + (size_t)(p0 << shift), *rb = rec + (size_t)(p1 << shift);
        r[i][0] = __ldg(ra + cl);
        r[i][1] = __ldg(rb + cl);
        r[i][2] = __ldg(ra + cr);
        r[i][3] = __ldg(rb + cr);
      }
      if (kMode != kCountsOnly) {
#pragma unroll
        for (int i = 0; i < kFieldBatch && f0 + i < NF; ++i) {
          const WinMoments m = window_moments<!kPlain, kSmall>(P, f0 + i, x, y, W, H, J.s12, J.qbits, inv_scale2);
          var[i] = m.var;
          rarea[i] = m.rarea;
          if (kPlain ? kMode == kOutKeep || kMode == kCountsMom : J.mom != nullptr)
            J.mom[(size_t)(f0 + i) * W * H + pix] = make_float2(m.var, window_mean(m.q1, m.rarea, inv_scale));
        }
      }
#pragma unroll
      for (int i = 0; i < kFieldBatch && f0 + i < NF; ++i) {
        const int f = f0 + i;
        const unsigned ul = (unsigned)max(x - P.rx[f], 0), ur = (unsigned)min(x + P.rx[f], W - 1) + 1u;
        const unsigned ol = ul & 31u, orr = ur & 31u;
        // C(ur, p1) - C(ur, p0) - (C(ul, p1) - C(ul, p0))
        cnt[i] = (r[i][3].x - r[i][2].x) - (r[i][1].x - r[i][0].x) + orr * ((r[i][3].y - r[i][2].y) & 0xffffu) -
                 ol * ((r[i][1].y - r[i][0].y) & 0xffffu);
        const unsigned vl = ((ul >> 5) * (unsigned)K + k) * slots, vr = ((ur >> 5) * (unsigned)K + k) * slots;
        const BT *pl = vec + (size_t)vl * 32 + ol, *pr = vec + (size_t)vr * 32 + orr;
        // no vectors where no row is mixed between the two positions; checked
        // where it pays: with 16-bit vectors at 12 MP 254 -> 249 us; with the
        // pyramid's wide windows, which rarely skip, 433 -> 485, and where the
        // moments are kept 16 MP 370 -> 395
        const bool check = sizeof(BT) == 2 && kMode == kOut;
        e[i][0] = e[i][1] = e[i][2] = e[i][3] = 0;
        if (!check || (r[i][0].y ^ r[i][1].y) >> 16) {
          e[i][0] = __ldg(pl + (r[i][0].y >> 16) * 32);
          e[i][1] = __ldg(pl + (r[i][1].y >> 16) * 32);
        }
        if (!check || (r[i][2].y ^ r[i][3].y) >> 16) {
          e[i][2] = __ldg(pr + (r[i][2].y >> 16) * 32);
          e[i][3] = __ldg(pr + (r[i][3].y >> 16) * 32);
        }
      }
      if (f0 == 0 && kMode < kCountsOnly) black = colour_powers<kPlain>(P, rgb, pw);
#pragma unroll
      for (int i = 0; i < kFieldBatch && f0 + i < NF; ++i) {
        const int f = f0 + i;
        cnt[i] += (unsigned)(BT)(e[i][3] - e[i][2]) - (unsigned)(BT)(e[i][1] - e[i][0]);
        if (!look) {  // threshold n takes the whole window, threshold 0 nothing
          const Win w = window_of(P, f, x, y, W, H);
          cnt[i] = whole ? (unsigned)((w.x1 - w.x0 + 1) * (w.y1 - w.y0 + 1)) : 0u;
        }
        if (kMode >= kCountsOnly || (kPlain ? kMode == kOutKeep : J.cnt != nullptr))
          J.cnt[f * J.cnt_step + pix] = cnt[i];
        if (kMode < kCountsOnly) {
          float Wf, Lf;
          fuse_field<kPlain>(P, f, cnt[i], rarea[i], var[i], fu, Wf, Lf);
          if (!kPlain && J.dbg.l) {
            const size_t N = (size_t)W * H;
            J.dbg.cnt[f * N + pix] = cnt[i];
            J.dbg.sigma2[f * N + pix] = var[i];
            J.dbg.weight[f * N + pix] = Wf;
            J.dbg.lf[f * N + pix] = Lf;
          }
        }
      }
    }
    if (kMode < kCountsOnly) {
      const float Lc = fused_value(P, fu);
      rgb[0] = pw[0] * Lc, rgb[1] = pw[1] * Lc, rgb[2] = pw[2] * Lc;
      if (black) {
        if (black & 1u) rgb[0] = 0.f;
        if (black & 2u) rgb[1] = 0.f;
        if (black & 4u) rgb[2] = 0.f;
      }
      store_rgb<kDt>(J.out, x, y, rgb[0], rgb[1], rgb[2], (P.flags & kFlagSrgb) != 0);
      if (!kPlain && J.dbg.l) J.dbg.l[pix] = Lc;
    }
  }
}

template <int KL, class BT>
int launch_cols(const Job *jobs, int njobs, int blocks, int tall, int K, cudaStream_t s) {
  using S = Shape<KL>;
  const size_t smem = (size_t)(S::ColWarps + 1) * KL * (32 * sizeof(BT) + sizeof(uint2));
  if (cudaFuncSetAttribute(k_compact_cols<KL, BT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) !=
      cudaSuccess)
    return -1;
  int nc = 1;  // CTAs that share a chunk's rows
  while (nc < 8 && (blocks * S::ColWarps * nc < S::Fill || tall > kSegRows * S::ColWarps * nc)) nc *= 2;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)(blocks * nc));
  cfg.blockDim = dim3(32 * S::ColWarps);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = (unsigned)nc;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_compact_cols<KL, BT>, jobs, njobs, K) == cudaSuccess ? 1 : -1;
}

template <int KL>
int launch_build(const Job *jobs, int njobs, int row_blocks, int col_blocks, int tall, int K, bool wide,
                 cudaStream_t s) {
  k_compact_rows<KL><<<row_blocks, 32 * kRowWarps, 0, s>>>(jobs, njobs, K);
  const int r = wide ? launch_cols<KL, uint32_t>(jobs, njobs, col_blocks, tall, K, s)
                     : launch_cols<KL, uint16_t>(jobs, njobs, col_blocks, tall, K, s);
  return r < 0 ? -1 : 2;
}

// Thresholds per group for K of them (log2).
int group_shift(int K) { return K <= 4 ? 2 : K <= 8 ? 3 : K <= 16 ? 4 : K <= 32 ? 5 : 6; }

}  // namespace

bool plan_compact(const DevParams &P, int W, int H, CompactPlan &C) {
  if (P.n_bins < 2 || W > 65535 || H > 65535) return false;
  const long long K = P.n_bins - 1, Gp = W / 32 + 1;
  int tall = 0;
  for (int f = 0; f < P.n_fields; ++f) tall = std::max(tall, std::min(2 * P.ry[f] + 1, H));
  C.shift = group_shift((int)K);
  C.wide = 31LL * tall > 65535;
  const long long KL = 1LL << C.shift, groups = (K + KL - 1) >> C.shift;
  const long long recs = groups * Gp * (H + 1) * KL, slots = Gp * K * (H + 1);
  if (recs >= (1LL << 31) || slots >= (1LL << 31)) return false;  // 32-bit indices in the lookup
  C.rec_bytes = sizeof(uint2) * (size_t)recs;
  C.row_bytes = sizeof(uint16_t) * (size_t)(groups * Gp * H * KL);
  C.vec_bytes = (size_t)slots * 32 * (C.wide ? 4 : 2);
  return true;
}

int compact_row_blocks(int H, int K) {
  const int sh = group_shift(K);
  return (H + kRowWarps - 1) / kRowWarps * ((K + (1 << sh) - 1) >> sh);
}

int compact_col_units(int W, int K) {
  const int sh = group_shift(K);
  return (W / 32 + 1) * ((K + (1 << sh) - 1) >> sh);
}

int launch_compact_build(const Job *jobs, int njobs, int row_blocks, int col_blocks, int tall, int K, bool wide,
                         cudaStream_t s) {
  switch (group_shift(K)) {
    case 2: return launch_build<4>(jobs, njobs, row_blocks, col_blocks, tall, K, wide, s);
    case 3: return launch_build<8>(jobs, njobs, row_blocks, col_blocks, tall, K, wide, s);
    case 4: return launch_build<16>(jobs, njobs, row_blocks, col_blocks, tall, K, wide, s);
    case 5: return launch_build<32>(jobs, njobs, row_blocks, col_blocks, tall, K, wide, s);
    default: return launch_build<64>(jobs, njobs, row_blocks, col_blocks, tall, K, wide, s);
  }
}

int compact_look_blocks(int W, int H, int rows) {
  return (W + kLookCols - 1) / kLookCols * ((H + rows - 1) / rows);
}

template <class BT, bool kPlain, int kSmall, int kDt, int kMode>
static void launch_look(const DevParams &P, const LookPack &L, int blocks, cudaStream_t s) {
  switch (P.n_fields) {
#define TM_LOOK(nf)                                                                                            \
  case nf: k_lookup_compact<nf, BT, kPlain, kSmall, kDt, kMode><<<blocks, kLookCols, 0, s>>>(P, L); break;
    TM_LOOK(1) TM_LOOK(2) TM_LOOK(3) TM_LOOK(4) TM_LOOK(5) TM_LOOK(6) TM_LOOK(7) TM_LOOK(8)
#undef TM_LOOK
  }
}

template <class BT, int kSmall>
static void launch_look_dtype(const DevParams &P, const LookPack &L, int blocks, int dtype, cudaStream_t s) {
  if (dtype == kF32) launch_look<BT, true, kSmall, kF32, kOut>(P, L, blocks, s);
  else if (dtype == kF16) launch_look<BT, true, kSmall, kF16, kOut>(P, L, blocks, s);
  else launch_look<BT, true, kSmall, -1, kOut>(P, L, blocks, s);
}

int launch_lookup_compact(const DevParams &P, const Job *jobs, int njobs, int blocks, int rows, bool wide,
                          bool plain, bool keep, bool counts_only, int dtype, cudaStream_t s) {
  const bool general =
      !plain || !P.fast || (P.flags & kFlagAreaLit) || (keep && (wide || !P.small_win || dtype != kF32));
  LookPack L{};
  L.n = njobs;
  L.rows = rows;
  for (int i = 0; i < njobs; ++i) {
    const Job &J = jobs[i];
    L.j[i] = {J.in, J.out, J.bins, J.c_rec, J.c_vec, reinterpret_cast<const longlong2 *>(J.s1),
              reinterpret_cast<unsigned *>(J.cnt), J.mom, J.dbg, J.cnt_off[1] / 4, J.qbits, J.c_shift,
              J.b0[kStLook], 0};
  }
  if (counts_only && keep) {
    launch_look<uint16_t, true, 1, -1, kCountsMom>(P, L, blocks, s);
  } else if (counts_only) {
    if (wide) launch_look<uint32_t, true, -1, -1, kCountsOnly>(P, L, blocks, s);
    else launch_look<uint16_t, true, -1, -1, kCountsOnly>(P, L, blocks, s);
  } else if (general) {
    if (wide) launch_look<uint32_t, false, -1, -1, kOut>(P, L, blocks, s);
    else launch_look<uint16_t, false, -1, -1, kOut>(P, L, blocks, s);
  } else if (keep) {
    launch_look<uint16_t, true, 1, kF32, kOutKeep>(P, L, blocks, s);
  } else if (wide) {
    if (P.small_win) launch_look_dtype<uint32_t, 1>(P, L, blocks, dtype, s);
    else launch_look_dtype<uint32_t, 0>(P, L, blocks, dtype, s);
  } else {
    if (P.small_win) launch_look_dtype<uint16_t, 1>(P, L, blocks, dtype, s);
    else launch_look_dtype<uint16_t, 0>(P, L, blocks, dtype, s);
  }
  return 1;
}

}  // namespace tmk
