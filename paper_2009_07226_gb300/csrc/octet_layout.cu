// Octet layouts (described with OctLayout): the packed form of a matrix that
// the tensor-core products of 16-bit slices read.
//
// Built from the CSR of the plan in four passes over its column ids, one CTA
// per block of kOctRows rows:
//   1. the block's footprint (8-column groups) counted in a shared bitmap;
//   2. the footprint listed, ordered and cut into stages, and every entry's
//      position in it (stage * capacity + place in the stage);
//   3. per stage and octet, the distinct columns counted (a warp per octet,
//      its bitmaps in shared memory), hence the chunks;
//   4. the chunks filled: every entry finds its column's rank among the
//      octet's columns of the stage (popcounts of the bitmap) and from it its
//      chunk and place.
// A row may hold one column twice in a row (rays along a grid line, whose
// pixel flips by rounding): the later entry gets a column of its own.
#include <algorithm>

#include "xct_internal.cuh"

namespace xct {
namespace {

constexpr int kWinGroups = 1 << 18;               // groups per footprint window
constexpr int kWinWords = kWinGroups / 32;
constexpr int kThreads = 32 * kOcts;              // a warp per octet
constexpr int kWordsPerThread = (kWinWords + kThreads - 1) / kThreads;
constexpr int kStageWindow = 64;                  // stages whose bitmaps are held at once

inline unsigned grid_for(int64_t n, int threads, int64_t cap = 0x7fffffffLL) {
  int64_t b = (n + threads - 1) / threads;
  return (unsigned)(b < 1 ? 1 : (b > cap ? cap : b));
}

__device__ void block_entries(const CsrView& m, int64_t* e0, int64_t* e1) {
  const int64_t r0 = (int64_t)blockIdx.x * kOctRows;
  const int64_t r1 = min(r0 + kOctRows, m.nrows);
  *e0 = m.rowptr[r0];
  *e1 = m.rowptr[r1];
}

// smallest and largest column of the block's entries (lo_hi[1] < 0: none)
__device__ void column_range(const CsrView& m, int64_t e0, int64_t e1, int32_t* lo_hi) {
  int32_t lo = INT32_MAX, hi = -1;
  for (int64_t e = e0 + threadIdx.x; e < e1; e += blockDim.x) {
    const int32_t c = m.col[e];
    lo = min(lo, c);
    hi = max(hi, c);
  }
  lo = __reduce_min_sync(0xffffffffu, lo);
  hi = __reduce_max_sync(0xffffffffu, hi);
  if (threadIdx.x == 0) {
    lo_hi[0] = INT32_MAX;
    lo_hi[1] = -1;
  }
  __syncthreads();
  if ((threadIdx.x & 31) == 0) {
    atomicMin(&lo_hi[0], lo);
    atomicMax(&lo_hi[1], hi);
  }
  __syncthreads();
}

// words [0, nw) of the bitmap: the groups of window [g0, g0 + kWinGroups)
// that the block's entries touch
__device__ void mark_groups(const CsrView& m, int64_t e0, int64_t e1, int64_t g0, int nw, uint32_t* bm) {
  for (int i = threadIdx.x; i < nw; i += blockDim.x) bm[i] = 0u;
  __syncthreads();
  for (int64_t e = e0 + threadIdx.x; e < e1; e += blockDim.x) {
    const int64_t g = (m.col[e] >> 3) - g0;
    if (g >= 0 && g < kWinGroups) {
      const uint32_t bit = 1u << (g & 31);
      if (!(bm[g >> 5] & bit)) atomicOr(&bm[g >> 5], bit);
    }
  }
  __syncthreads();
}

// words of the bitmap that a window reaching up to group `last` uses
__device__ int window_words(int64_t g0, int64_t last) {
  const int64_t n = min((int64_t)kWinGroups, last - g0 + 1);
  return (int)((n + 31) >> 5);
}

__global__ void __launch_bounds__(kThreads) oct_fp_count_kernel(CsrView m, int64_t* fp_groups) {
  extern __shared__ uint32_t bm[];
  __shared__ int32_t lo_hi[2];
  __shared__ int total;
  int64_t e0, e1;
  block_entries(m, &e0, &e1);
  if (threadIdx.x == 0) total = 0;
  column_range(m, e0, e1, lo_hi);
  const int64_t first = lo_hi[0] >> 3, last = lo_hi[1] >> 3;
  for (int64_t g0 = first; lo_hi[1] >= 0 && g0 <= last; g0 += kWinGroups) {
    const int nw = window_words(g0, last);
    mark_groups(m, e0, e1, g0, nw, bm);
    int c = 0;
    for (int i = threadIdx.x; i < nw; i += blockDim.x) c += __popc(bm[i]);
    c = __reduce_add_sync(0xffffffffu, c);
    if ((threadIdx.x & 31) == 0 && c) atomicAdd(&total, c);
    __syncthreads();
  }
  __syncthreads();
  if (threadIdx.x == 0) fp_groups[blockIdx.x] = total;
}

// the footprint's groups in ascending order, and every entry's position in
// the block's footprint (8 positions per group)
__global__ void __launch_bounds__(kThreads) oct_fp_fill_kernel(CsrView m, const int64_t* fp_off,
                                                               int32_t* groups, int32_t* epos) {
  extern __shared__ uint32_t bm[];
  int32_t* pre = reinterpret_cast<int32_t*>(bm + kWinWords);   // groups before each word
  __shared__ int32_t lo_hi[2];
  __shared__ int32_t wtot[kThreads / 32];
  int64_t e0, e1;
  block_entries(m, &e0, &e1);
  column_range(m, e0, e1, lo_hi);
  if (lo_hi[1] < 0) return;
  const int64_t first = lo_hi[0] >> 3, last = lo_hi[1] >> 3;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int32_t base = 0;
  for (int64_t g0 = first; g0 <= last; g0 += kWinGroups) {
    const int nw = window_words(g0, last);
    mark_groups(m, e0, e1, g0, nw, bm);
    // exclusive scan of the words' counts: thread t owns kWordsPerThread words
    const int i0 = threadIdx.x * kWordsPerThread, i1 = min(i0 + kWordsPerThread, nw);
    int32_t local = 0;
    for (int i = i0; i < i1; ++i) local += __popc(bm[i]);
    int32_t inc = local;
    for (int o = 1; o < 32; o <<= 1) {
      const int32_t u = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += u;
    }
    if (lane == 31) wtot[warp] = inc;
    __syncthreads();
    int32_t run = base + inc - local, all = 0;
    for (int w = 0; w < kThreads / 32; ++w) {
      if (w < warp) run += wtot[w];
      all += wtot[w];
    }
    for (int i = i0; i < i1; ++i) {
      pre[i] = run;
      run += __popc(bm[i]);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < nw; i += blockDim.x) {
      uint32_t bits = bm[i];
      int32_t p = pre[i];
      while (bits) {
        const int b = __ffs(bits) - 1;
        bits &= bits - 1;
        groups[fp_off[blockIdx.x] + p++] = (int32_t)(g0 + i * 32 + b);
      }
    }
    for (int64_t e = e0 + threadIdx.x; e < e1; e += blockDim.x) {
      const int32_t c = m.col[e];
      const int64_t g = (c >> 3) - g0;
      if (g >= 0 && g < kWinGroups) {
        const uint32_t below = bm[g >> 5] & ((1u << (g & 31)) - 1u);
        epos[e] = (pre[g >> 5] + __popc(below)) * 8 + (c & 7);
      }
    }
    base += all;
    __syncthreads();
  }
}

// The row of octet place p (0 .. 7 of octet o) of block b, or -1 past the matrix.
__device__ __forceinline__ int64_t octet_row(int b, int o, int r, int angle_rows, int64_t nrows) {
  const int64_t row = (int64_t)b * kOctRows + (o >> 3) * 64 + oct_row((o & 7) * 8 + r, angle_rows);
  return row < nrows ? row : -1;
}

// Orders a block's groups so that a stage, a piece of the list, holds work for
// all of the block's rows: for rays by the place of the group's tile along
// the block's (middle) ray, for pixels by its angle tile.  In ascending ids a
// stage is a square patch of the footprint, which some of the block's rays
// miss: the busiest warp of a stage had twice the average's columns (512^2 x
// 768: 1.5 to 1.9 times, and 1.1 to 1.2 in this order).  512^2 x 768, 64
// slices: xct_project 0.78 -> 0.73 ms, xct_backproject 0.73 -> 0.69; 1536^2 x
// 1024, 32 slices: 7.0 -> 6.6.  A tile's groups stay together, and so do most
// runs.  A group that reaches past the matrix's columns comes last, where the
// descriptor expects it.
//
// A stage ends at `cap` rows, or before its chunks could pass kStageChunks (a
// group's weight is its columns over the block's octets; an octet's last chunk
// may be partly filled): near the rotation centre the same pixels meet many
// rays, and stages of equal rows sized the buffers for 1.5 to 1.9 times the
// average stage, at 384 rows at most.  With stages of up to 512 rows cut this
// way, and chunks leaving L2 first (spmm_mma.cu): 512^2 x 768, 64 slices 0.73 ->
// 0.69 and 0.69 -> 0.65 ms, 8 slices 0.35 -> 0.31; 1536^2 x 1024, 32 slices 6.6
// -> 5.8 and 5.8 -> 4.2 ms.
constexpr int kOrderMax = 8192;   // groups of a block that are ordered (else ids ascend)
constexpr int kStageColumns = (kStageChunks - kOcts) * 16;
// Cuts a list of groups into stages: add(i, weight of the list's i-th group)
// returns the group's place, stage * groups of a stage + place in the stage.
struct StageCut {
  int32_t* cut;   // first group of every stage
  int gps;
  int st = -1, in = 0;
  uint32_t cols = 0;
  __device__ uint32_t add(int i, uint32_t weight) {
    if (st < 0 || in == gps || cols + weight > (uint32_t)kStageColumns) {
      cut[++st] = i;
      in = 0;
      cols = 0;
    }
    cols += weight;
    return (uint32_t)(st * gps + in++);
  }
};
// shared memory for blocks of up to n groups (a power of two)
constexpr size_t order_smem(int n) { return (size_t)n * (kOcts + 4); }
__global__ void __launch_bounds__(kThreads) oct_order_kernel(CsrView m, FootprintOrder o, int cap, int nmax,
                                                             const int64_t* fp_off, int32_t* groups,
                                                             int32_t* epos, int32_t* cut, int64_t* nst) {
  extern __shared__ uint32_t sm[];
  const int b = blockIdx.x, warp = threadIdx.x >> 5, lane = threadIdx.x & 31, gps = cap / 8;
  const int64_t f0 = fp_off[b];
  const int64_t nf = fp_off[b + 1] - f0;
  int64_t e0, e1;
  block_entries(m, &e0, &e1);
  if (nf > nmax && nf <= 5 * nmax) {
    // ids ascend; a group's weight is its entries (at least its columns)
    for (int i = threadIdx.x; i < nf; i += blockDim.x) sm[i] = 0u;
    __syncthreads();
    for (int64_t e = e0 + threadIdx.x; e < e1; e += blockDim.x) atomicAdd(&sm[epos[e] >> 3], 1u);
    __syncthreads();
    if (threadIdx.x == 0) {
      StageCut c{cut + f0, gps};
      for (int g = 0; g < (int)nf; ++g) sm[g] = c.add(g, sm[g]);
      nst[b] = c.st + 1;
    }
    __syncthreads();
    for (int64_t e = e0 + threadIdx.x; e < e1; e += blockDim.x) {
      const int32_t p = epos[e];
      epos[e] = (int32_t)(sm[p >> 3] * 8 + (p & 7));
    }
    return;
  }
  if (nf == 0 || nf > nmax) {
    const int64_t ns = (nf + gps - 1) / gps;
    for (int64_t k = threadIdx.x; k < ns; k += blockDim.x) cut[f0 + k] = (int32_t)(k * gps);
    if (threadIdx.x == 0) nst[b] = ns;
    return;
  }
  const int n = (int)nf;
  uint32_t* weight = sm;              // [nmax]
  uint32_t* bits = sm + nmax;         // [octet][nmax / 4]: 8 columns of a group
  uint32_t* key = bits;               // [nmax], after the bits
  uint32_t* place = bits + nmax;      // [nmax]
  for (int i = threadIdx.x; i < nmax * (kOcts / 4 + 1); i += blockDim.x) sm[i] = 0u;
  __syncthreads();
  uint32_t* own = bits + warp * (nmax / 4);
  for (int r = 0; r < 8; ++r) {
    const int64_t row = octet_row(b, warp, r, o.rays, m.nrows);
    if (row < 0) continue;
    const int64_t r0 = m.rowptr[row], r1 = m.rowptr[row + 1];
    for (int64_t e = r0 + lane; e < r1; e += 32) {
      const int32_t p = epos[e];
      if (e > r0 && epos[e - 1] == p) {
        atomicAdd(&weight[p >> 3], 1u);   // a repeated entry has a column of its own
      } else {
        const uint32_t bit = 1u << (p & 31);
        if (!(own[p >> 5] & bit)) atomicOr(&own[p >> 5], bit);
      }
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    uint32_t c = 0;
    for (int w = 0; w < kOcts; ++w) c += __popc(bits[w * (nmax / 4) + (i >> 2)] >> (8 * (i & 3)) & 0xffu);
    weight[i] += c;
  }
  __syncthreads();
  int n2 = 2;
  while (n2 < n) n2 *= 2;
  const int64_t mid = min((int64_t)b * kOctRows + kOctRows / 2, m.nrows - 1);
  const int k_mid = o.rays ? o.row_inv[mid] / o.nd : 0;
  const float dx = o.rays ? -(float)o.cs[2 * k_mid + 1] : 0.0f, dy = o.rays ? (float)o.cs[2 * k_mid] : 0.0f;
  for (int i = threadIdx.x; i < n2; i += blockDim.x) {
    uint32_t k = 0xffffffffu;
    if (i < n) {
      const int64_t g = groups[f0 + i];
      if ((g + 1) * 8 <= m.ncols) {
        const int32_t id = o.col_inv[g * 8];
        int at;
        if (o.rays) {
          const int ix = id % o.n / o.tile * o.tile, iy = id / o.n / o.tile * o.tile;
          at = (int)floorf((float)ix * dx + (float)iy * dy) + 2 * o.n;
        } else {
          at = id / o.nd / o.tile;
        }
        k = (uint32_t)min(max(at, 0), (1 << 19) - 2) << 13 | (uint32_t)i;
      } else {
        k = 0xffffe000u | (uint32_t)i;
      }
    }
    key[i] = k;
  }
  __syncthreads();
  // bitonic sort
  for (int span = 2; span <= n2; span *= 2)
    for (int d = span / 2; d > 0; d /= 2) {
      for (int i = threadIdx.x; i < n2 / 2; i += blockDim.x) {
        const int lo = (i / d) * 2 * d + i % d, hi = lo + d;
        const uint32_t u = key[lo], v = key[hi];
        if ((u > v) == ((lo & span) == 0)) {
          key[lo] = v;
          key[hi] = u;
        }
      }
      __syncthreads();
    }
  if (threadIdx.x == 0) {
    StageCut c{cut + f0, gps};
    for (int i = 0; i < n; ++i) {
      const int g = key[i] & (kOrderMax - 1);
      place[g] = c.add(i, weight[g]);
    }
    nst[b] = c.st + 1;
  }
  // the list itself, in place: read, then written
  int32_t mine[kOrderMax / kThreads];
#pragma unroll
  for (int j = 0; j < kOrderMax / kThreads; ++j) {
    const int i = threadIdx.x + j * kThreads;
    if (i < n) mine[j] = groups[f0 + (key[i] & (kOrderMax - 1))];
  }
  __syncthreads();
#pragma unroll
  for (int j = 0; j < kOrderMax / kThreads; ++j) {
    const int i = threadIdx.x + j * kThreads;
    if (i < n) groups[f0 + i] = mine[j];
  }
  for (int64_t e = e0 + threadIdx.x; e < e1; e += kThreads) {
    const int32_t p = epos[e];
    epos[e] = (int32_t)(place[p >> 3] * 8 + (p & 7));
  }
}

__global__ void oct_max_kernel(const int64_t* v, int32_t n, unsigned long long* out) {
  const int32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) atomicMax(out, (unsigned long long)v[i]);
}

// the groups of stage k of the block whose groups are g[0 .. n), cut at cut[]
__device__ __forceinline__ const int32_t* stage_groups(const int32_t* g, const int32_t* cut, int64_t k, int64_t ns,
                                                       int64_t n, int* count) {
  const int32_t at = cut[k];
  *count = (int)((k + 1 < ns ? cut[k + 1] : n) - at);
  return g + at;
}

// An octet's distinct columns in a stage as a bitmap over the stage's
// positions (`words` = cap / 32 words), plus `dups` repeated entries.
// rank: the columns ordered by residue mod 8, then position.
struct OctCols {
  const uint32_t* bm;
  int words;
  __device__ int count() const {
    int n = 0;
    for (int w = 0; w < words; ++w) n += __popc(bm[w]);
    return n;
  }
  __device__ int rank(int pos) const {
    const int r = pos & 7, wp = pos >> 5;
    const uint32_t res = 0x01010101u << r, lower = 0x01010101u * ((1u << r) - 1u);
    int n = 0;
    for (int w = 0; w < words; ++w) {
      const uint32_t b = bm[w];
      n += __popc(b & lower);
      if (w < wp) n += __popc(b & res);
    }
    return n + __popc(bm[wp] & res & ((1u << (pos & 31)) - 1u));
  }
};

// place of the j-th column among an octet's g8 groups of 8 columns: columns
// of one residue go to different groups
__device__ __forceinline__ int oct_place(int j, int g8) { return (j % g8) * 8 + j / g8; }

// Marks the octet's columns of stages [s0, s0 + kStageWindow) in the warp's
// bitmaps and counts the repeated entries per stage.
__device__ void mark_octet(const CsrView& m, const int32_t* epos, int b, int o, int angle_rows, int s0,
                           int cap, uint32_t* bm, int* dups) {
  const int lane = threadIdx.x & 31, words = cap >> 5;
  for (int i = lane; i < kStageWindow * words; i += 32) bm[i] = 0u;
  for (int i = lane; i < kStageWindow; i += 32) dups[i] = 0;
  __syncwarp();
  for (int r = 0; r < 8; ++r) {
    const int64_t row = octet_row(b, o, r, angle_rows, m.nrows);
    if (row < 0) continue;
    const int64_t e0 = m.rowptr[row], e1 = m.rowptr[row + 1];
    for (int64_t e = e0 + lane; e < e1; e += 32) {
      const int32_t p = epos[e];
      const int st = p / cap - s0;
      if (st < 0 || st >= kStageWindow) continue;
      if (e > e0 && epos[e - 1] == p) {
        atomicAdd(&dups[st], 1);
      } else {
        const int q = p % cap;
        uint32_t* w = &bm[st * words + (q >> 5)];
        const uint32_t bit = 1u << (q & 31);
        if (!(*w & bit)) atomicOr(w, bit);
      }
    }
  }
  __syncwarp();
}

__device__ __forceinline__ size_t warp_words(int cap) { return (size_t)kStageWindow * (cap >> 5); }

// chunks of every (stage, octet)
__global__ void __launch_bounds__(kThreads) oct_count_kernel(CsrView m, const int32_t* epos,
                                                             const int64_t* blk_stage, int cap, int angle_rows,
                                                             int32_t* nch) {
  extern __shared__ uint32_t sm[];
  __shared__ int dups[kOcts][kStageWindow];
  const int b = blockIdx.x, o = threadIdx.x >> 5, lane = threadIdx.x & 31, words = cap >> 5;
  uint32_t* bm = sm + o * warp_words(cap);
  const int64_t sb = blk_stage[b];
  const int ns = (int)(blk_stage[b + 1] - sb);
  for (int s0 = 0; s0 < ns; s0 += kStageWindow) {
    mark_octet(m, epos, b, o, angle_rows, s0, cap, bm, dups[o]);
    for (int st = lane; st < min(kStageWindow, ns - s0); st += 32) {
      const OctCols c{bm + st * words, words};
      nch[(sb + s0 + st) * kOcts + o] = (c.count() + dups[o][st] + 15) / 16;
    }
    __syncwarp();
  }
}

// chunks of every stage, and the largest stage
__global__ void oct_stage_chunks_kernel(const int32_t* nch, int64_t nstages, int32_t* total,
                                        unsigned long long* emax) {
  int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (s >= nstages) return;
  int32_t n = 0;
  for (int o = 0; o < kOcts; ++o) n += nch[s * kOcts + o];
  total[s] = n;
  atomicMax(emax, (unsigned long long)n);
}

// runs of the stage's groups (consecutive groups join)
__device__ __forceinline__ bool run_starts(const int32_t* g, int i) { return i == 0 || g[i] != g[i - 1] + 1; }

__global__ void oct_run_count_kernel(const int64_t* blk_stage, const int64_t* fp_off, const int64_t* fp_groups,
                                     const int32_t* groups, const int32_t* cut, int* run_max) {
  const int b = blockIdx.x;
  for (int64_t s = blk_stage[b] + threadIdx.x; s < blk_stage[b + 1]; s += blockDim.x) {
    int n;
    const int32_t* g = stage_groups(groups + fp_off[b], cut + fp_off[b], s - blk_stage[b],
                                    blk_stage[b + 1] - blk_stage[b], fp_groups[b], &n);
    int r = 0;
    for (int i = 0; i < n; ++i) r += run_starts(g, i);
    atomicMax(run_max, r + 1);
  }
}

__global__ void oct_desc_kernel(const int64_t* blk_stage, const int64_t* fp_off, const int64_t* fp_groups,
                                const int32_t* groups, const int32_t* cut, const int32_t* nch, const int64_t* c0,
                                int64_t ncols, int run_stride, int64_t desc_bytes, unsigned char* desc,
                                uint2* chunks) {
  const int b = blockIdx.x;
  for (int64_t s = blk_stage[b] + threadIdx.x; s < blk_stage[b + 1]; s += blockDim.x) {
    int n;
    const int32_t* g = stage_groups(groups + fp_off[b], cut + fp_off[b], s - blk_stage[b],
                                    blk_stage[b + 1] - blk_stage[b], fp_groups[b], &n);
    OctStageHead h;
    h.c0 = c0[s];
    h.nch = (uint32_t)(c0[s + 1] - c0[s]);
    uint32_t at = 0;
    for (int o = 0; o <= kOcts; ++o) {
      h.ofs[o] = (uint16_t)at;
      if (o < kOcts) at += nch[s * kOcts + o];
    }
    int2* runs = reinterpret_cast<int2*>(desc + s * desc_bytes + sizeof(OctStageHead));
    int r = 0;
    for (int i = 0; i < n; ++i)
      if (run_starts(g, i)) runs[r++] = make_int2(g[i] * 8, i * 8);
    // the last group may reach past the matrix's columns
    const int64_t over = n > 0 ? ((int64_t)g[n - 1] + 1) * 8 - ncols : 0;
    h.np = (uint16_t)(n * 8 - (over > 0 ? over : 0));
    chunks[s] = make_uint2((uint32_t)h.c0, h.nch);
    h.nr = (uint16_t)(r + 1);
    for (; r < run_stride; ++r) runs[r] = make_int2(-1, (int)h.np);
    *reinterpret_cast<OctStageHead*>(desc + s * desc_bytes) = h;
  }
}

template <bool HALF>
__device__ __forceinline__ uint16_t stored16(double v) {
  return HALF ? __half_as_ushort(__double2half(__dmul_rn(v, 32768.0)))
              : __bfloat16_as_ushort(__double2bfloat16(v));
}

// values and positions of every chunk (`ent` starts zeroed)
template <bool HALF>
__global__ void __launch_bounds__(kThreads) oct_fill_kernel(CsrView m, const int32_t* epos,
                                                            const int64_t* blk_stage, int cap, int angle_rows,
                                                            const unsigned char* desc, int64_t desc_bytes,
                                                            unsigned char* ent) {
  extern __shared__ uint32_t sm[];
  __shared__ int dups[kOcts][kStageWindow];
  __shared__ int ucols[kOcts][kStageWindow];
  const int b = blockIdx.x, o = threadIdx.x >> 5, lane = threadIdx.x & 31, words = cap >> 5;
  uint32_t* bm = sm + o * warp_words(cap);
  const int64_t sb = blk_stage[b];
  const int ns = (int)(blk_stage[b + 1] - sb);
  auto head = [&](int st) -> const OctStageHead& {
    return *reinterpret_cast<const OctStageHead*>(desc + (sb + st) * desc_bytes);
  };
  for (int s0 = 0; s0 < ns; s0 += kStageWindow) {
    mark_octet(m, epos, b, o, angle_rows, s0, cap, bm, dups[o]);
    const int n = min(kStageWindow, ns - s0);
    for (int st = lane; st < n; st += 32) ucols[o][st] = OctCols{bm + st * words, words}.count();
    for (int st = lane; st < kStageWindow; st += 32) dups[o][st] = 0;   // now: repeated entries placed
    __syncwarp();
    // positions: every used column's, in its place
    for (int i = lane; i < n * words; i += 32) {
      const int st = i / words, w = i % words;
      uint32_t bits = bm[i];
      if (!bits) continue;
      const OctStageHead& h = head(s0 + st);
      const int f = h.ofs[o], g8 = 2 * (h.ofs[o + 1] - f);
      uint16_t* pos = reinterpret_cast<uint16_t*>(ent + h.c0 * kChunkBytes + h.nch * 256u + f * 32u);
      const OctCols c{bm + st * words, words};
      while (bits) {
        const int q = w * 32 + __ffs(bits) - 1;
        bits &= bits - 1;
        pos[oct_place(c.rank(q), g8)] = (uint16_t)q;
      }
    }
    // values
    for (int r = 0; r < 8; ++r) {
      const int64_t row = octet_row(b, o, r, angle_rows, m.nrows);
      if (row < 0) continue;
      const int64_t e0 = m.rowptr[row], e1 = m.rowptr[row + 1];
      for (int64_t eb = e0; eb < e1; eb += 32) {
        const int64_t e = eb + lane;
        int st = -1, q = 0;
        bool dup = false;
        if (e < e1) {
          const int32_t p = epos[e];
          st = p / cap - s0;
          q = p % cap;
          if (st >= kStageWindow) st = -1;
          dup = st >= 0 && e > e0 && epos[e - 1] == p;
        }
        // repeated entries take their columns in the order of the row
        int dr = 0;
        for (uint32_t left = __ballot_sync(0xffffffffu, dup); left; left &= left - 1) {
          if (lane == __ffs(left) - 1) dr = dups[o][st]++;
          __syncwarp();
        }
        if (st < 0) continue;
        const OctStageHead& h = head(s0 + st);
        const int f = h.ofs[o], g8 = 2 * (h.ofs[o + 1] - f);
        const OctCols c{bm + st * words, words};
        const int place = oct_place(dup ? ucols[o][st] + dr : c.rank(q), g8);
        const int k = place & 15;
        unsigned char* base = ent + h.c0 * kChunkBytes;
        reinterpret_cast<uint16_t*>(base + (f + (place >> 4)) * 256u + (r * 4 + ((k & 7) >> 1)) * 8u)
            [(k >> 3) * 2 + (k & 1)] = stored16<HALF>(m.val[e]);
        if (dup) reinterpret_cast<uint16_t*>(base + h.nch * 256u + f * 32u)[place] = (uint16_t)q;
      }
    }
    __syncwarp();
    // unused places repeat the first column of their group of 8, or of the
    // octet where the group is empty: a position whose row is staged
    for (int st = lane; st < n; st += 32) {
      const OctStageHead& h = head(s0 + st);
      const int f = h.ofs[o], g8 = 2 * (h.ofs[o + 1] - f), u = ucols[o][st] + dups[o][st];
      uint16_t* pos = reinterpret_cast<uint16_t*>(ent + h.c0 * kChunkBytes + h.nch * 256u + f * 32u);
      for (int j = u; j < g8 * 8; ++j) pos[oct_place(j, g8)] = pos[j % g8 < u ? (j % g8) * 8 : 0];
    }
    __syncwarp();
  }
}

}  // namespace

xct_status build_oct_layout(const CsrView& m, xct_dtype storage, const FootprintOrder& order, OctLayout& L,
                            Arena& keep, bool* fits, cudaStream_t s) {
  *fits = false;
  L = OctLayout{};
  L.nrows = m.nrows;
  L.ncols = m.ncols;
  L.angle_rows = order.rays;
  L.nblocks = (int32_t)((m.nrows + kOctRows - 1) / kOctRows);
  const int32_t nb = L.nblocks;
  int64_t nnz = 0;
  XCT_TRY_CUDA(cudaMemcpyAsync(&nnz, m.rowptr + m.nrows, sizeof(int64_t), cudaMemcpyDeviceToHost, s));
  XCT_TRY_CUDA(cudaStreamSynchronize(s));
  Arena tmp(s);
  int64_t *fp_groups, *fp_off, *nst;
  int32_t *groups, *epos, *cut;
  unsigned long long *most, most_h = 0;   // groups of the block with most
  XCT_TRY(tmp.get(&most, 1));
  XCT_TRY_CUDA(cudaMemsetAsync(most, 0, sizeof(*most), s));
  XCT_TRY(tmp.get(&fp_groups, nb));
  XCT_TRY(tmp.get(&fp_off, nb + 1));
  XCT_TRY(tmp.get(&nst, nb));
  XCT_TRY(tmp.get(&epos, nnz));
  const int count_smem = kWinWords * 4, fill_smem = kWinWords * 8;
  XCT_TRY(allow_all_smem<oct_fp_fill_kernel>());
  XCT_TRY(allow_all_smem<oct_order_kernel>());
  XCT_TRY(allow_all_smem<oct_count_kernel>());
  XCT_TRY(allow_all_smem<oct_fill_kernel<true>>());
  XCT_TRY(allow_all_smem<oct_fill_kernel<false>>());
  oct_fp_count_kernel<<<nb, kThreads, count_smem, s>>>(m, fp_groups);
  count_launch();
  XCT_TRY(exclusive_scan_i64(fp_groups, fp_off, nb, s));
  oct_max_kernel<<<grid_for(nb, 256), 256, 0, s>>>(fp_groups, nb, most);
  count_launch();
  XCT_TRY_CUDA(cudaMemcpyAsync(&most_h, most, sizeof(most_h), cudaMemcpyDeviceToHost, s));
  int64_t ngroups = 0;
  XCT_TRY_CUDA(cudaMemcpyAsync(&ngroups, fp_off + nb, sizeof(int64_t), cudaMemcpyDeviceToHost, s));
  XCT_TRY_CUDA(cudaStreamSynchronize(s));
  XCT_TRY(tmp.get(&groups, ngroups));
  XCT_TRY(tmp.get(&cut, ngroups));
  int nmax = 64;
  while (nmax < (int64_t)most_h && nmax < kOrderMax) nmax *= 2;
  // stage capacity: the first at which two stage buffers of 128-byte rows
  // fit a CTA
  for (int cap = kOctCap; cap >= 64; cap -= 64) {
    Arena own(s, true), part(s);
    L.cap = cap;
    const int bm_smem = kOcts * kStageWindow * cap / 8;
    oct_fp_fill_kernel<<<nb, kThreads, fill_smem, s>>>(m, fp_off, groups, epos);
    oct_order_kernel<<<nb, kThreads, order_smem(nmax), s>>>(m, order, cap, nmax, fp_off, groups, epos, cut, nst);
    count_launch(2);
    XCT_TRY(own.get(&L.blk_stage, nb + 1));
    XCT_TRY(exclusive_scan_i64(nst, L.blk_stage, nb, s));
    XCT_TRY_CUDA(cudaMemcpyAsync(&L.nstages, L.blk_stage + nb, sizeof(int64_t), cudaMemcpyDeviceToHost, s));
    XCT_TRY_CUDA(cudaStreamSynchronize(s));
    int32_t *nch, *total;
    int64_t* c0;
    unsigned long long* emax;
    int* run_max;
    XCT_TRY(part.get(&nch, L.nstages * kOcts));
    XCT_TRY(part.get(&total, L.nstages));
    XCT_TRY(part.get(&c0, L.nstages + 1));
    XCT_TRY(part.get(&emax, 1));
    XCT_TRY(part.get(&run_max, 1));
    XCT_TRY_CUDA(cudaMemsetAsync(emax, 0, sizeof(unsigned long long), s));
    XCT_TRY_CUDA(cudaMemsetAsync(run_max, 0, sizeof(int), s));
    oct_count_kernel<<<nb, kThreads, bm_smem, s>>>(m, epos, L.blk_stage, cap, L.angle_rows, nch);
    oct_stage_chunks_kernel<<<grid_for(L.nstages, 256), 256, 0, s>>>(nch, L.nstages, total, emax);
    oct_run_count_kernel<<<nb, 64, 0, s>>>(L.blk_stage, fp_off, fp_groups, groups, cut, run_max);
    count_launch(3);
    XCT_TRY(exclusive_scan_i32(total, c0, L.nstages, s));
    unsigned long long emax_h = 0;
    int run_max_h = 0;
    XCT_TRY_CUDA(cudaMemcpyAsync(&L.nchunks, c0 + L.nstages, sizeof(int64_t), cudaMemcpyDeviceToHost, s));
    XCT_TRY_CUDA(cudaMemcpyAsync(&emax_h, emax, sizeof(emax_h), cudaMemcpyDeviceToHost, s));
    XCT_TRY_CUDA(cudaMemcpyAsync(&run_max_h, run_max, sizeof(int), cudaMemcpyDeviceToHost, s));
    XCT_TRY_CUDA(cudaStreamSynchronize(s));
    L.emax = (int64_t)emax_h;
    const int run_stride = (run_max_h + 2) & ~1;
    L.desc_bytes = (int64_t)sizeof(OctStageHead) + 8 * run_stride;
    if (!oct_stage_fits(cap, L.emax, L.desc_bytes) || L.emax > 65535 || L.nchunks > 0xffffffffll) continue;
    XCT_TRY(own.get(&L.desc, (size_t)L.nstages * L.desc_bytes));
    XCT_TRY(own.get(&L.chunks, (size_t)L.nstages));
    XCT_TRY(own.get(&L.ent, (size_t)L.nchunks * kChunkBytes));
    oct_desc_kernel<<<nb, 64, 0, s>>>(L.blk_stage, fp_off, fp_groups, groups, cut, nch, c0, m.ncols,
                                      run_stride, L.desc_bytes, L.desc, L.chunks);
    XCT_TRY_CUDA(cudaMemsetAsync(L.ent, 0, (size_t)L.nchunks * kChunkBytes, s));
    if (half_values(storage)) {
      oct_fill_kernel<true><<<nb, kThreads, bm_smem, s>>>(m, epos, L.blk_stage, cap, L.angle_rows, L.desc,
                                                          L.desc_bytes, L.ent);
    } else {
      oct_fill_kernel<false><<<nb, kThreads, bm_smem, s>>>(m, epos, L.blk_stage, cap, L.angle_rows, L.desc,
                                                           L.desc_bytes, L.ent);
    }
    count_launch(2);
    XCT_TRY_CUDA(cudaGetLastError());
    XCT_TRY_CUDA(cudaStreamSynchronize(s));
    L.bytes = L.nchunks * kChunkBytes + L.nstages * (L.desc_bytes + 8) + (int64_t)(nb + 1) * 8;
    own.move_to(keep);
    *fits = true;
    return XCT_OK;
  }
  L = OctLayout{};
  return XCT_OK;
}

}  // namespace xct
