// Vector kernels around the products: layout conversion between the caller's
// slice-major natural order and the internal [tile][ordered row][slice]
// layout, and the CGLS vector updates and FP64 scalars (Eq. 1 with R = 0,
// CGLS form with one initial back projection, per-slice scalars).
#include <algorithm>
#include <type_traits>

#include "ff.cuh"
#include "xct_internal.cuh"
#include "xct_vec.cuh"

namespace xct {
namespace {

// Layout conversion: a block takes conv_rows(ST) ordered rows of a slice tile,
// a thread one row (its natural id read once) and every 256 / rows-th slice;
// the slices are transposed in shared memory and the internal layout is read
// and written 16 bytes at a time.  Maxima go through registers, a warp's
// reduction and shared memory to one global atomic a block and slice, left
// out where the slice already holds as much.  Bound by memory (8 bytes an
// element); 512^2 x 768, 64 slices: rays in 132 -> 80 us, pixels out 51 -> 24
// us.
constexpr int kConvThreads = 256;
__host__ __device__ constexpr int conv_rows(int st) { return st >= 32 ? 64 : st >= 8 ? 128 : 256; }

// natural [S][rows] -> internal [ntiles][rows][ST]; slices >= S are zero.
// Optionally accumulates max |v| per slice into max_bits (float bits).
template <int ST>
__global__ void __launch_bounds__(kConvThreads) to_internal_kernel(
    const float* __restrict__ nat, float* __restrict__ out, const int32_t* __restrict__ inv,
    int64_t rows, int S, uint32_t* __restrict__ max_bits) {
  constexpr int R = conv_rows(ST), V = 4;
  __shared__ float buf[ST][R + 1];
  __shared__ uint32_t smax[ST];
  const int64_t h0 = (int64_t)blockIdx.x * R;
  const int t = blockIdx.y, live = min(ST, S - t * ST);
  const int nr = (int)min((int64_t)R, rows - h0);
  const int r = threadIdx.x % R;
  allow_next();
  wait_previous();
  nat = after_wait(nat);
  const float* src = nat + (size_t)t * ST * rows + (r < nr ? inv[h0 + r] : 0);
  if (threadIdx.x < ST) smax[threadIdx.x] = 0u;
  __syncthreads();
#pragma unroll 8
  for (int sl = threadIdx.x / R; sl < ST; sl += kConvThreads / R) {
    const float v = r < nr && sl < live ? src[(size_t)sl * rows] : 0.0f;
    buf[sl][r] = v;
    if (max_bits) {
      const uint32_t m = __reduce_max_sync(0xffffffffu, __float_as_uint(fabsf(v)));
      if ((threadIdx.x & 31) == 0 && m) atomicMax(&smax[sl], m);
    }
  }
  __syncthreads();
  float* dst = out + ((size_t)t * rows + h0) * ST;
  for (int i = threadIdx.x; i < nr * (ST / V); i += kConvThreads) {
    const int row = i / (ST / V), sl = i % (ST / V) * V;
    reinterpret_cast<float4*>(dst)[i] = make_float4(buf[sl][row], buf[sl + 1][row], buf[sl + 2][row], buf[sl + 3][row]);
  }
  if (max_bits && threadIdx.x < ST) {
    const uint32_t m = smax[threadIdx.x];
    uint32_t* to = max_bits + t * ST + threadIdx.x;
    if (m > __ldcg(to)) atomicMax(to, m);
  }
}

template <int ST>
__global__ void __launch_bounds__(kConvThreads) to_natural_kernel(
    const float* __restrict__ in, float* __restrict__ nat, const int32_t* __restrict__ inv,
    int64_t rows, int S) {
  constexpr int R = conv_rows(ST), V = 4;
  __shared__ float buf[ST][R + 1];
  const int64_t h0 = (int64_t)blockIdx.x * R;
  const int t = blockIdx.y, live = min(ST, S - t * ST);
  const int nr = (int)min((int64_t)R, rows - h0);
  allow_next();
  wait_previous();
  in = after_wait(in);
  const float* src = in + ((size_t)t * rows + h0) * ST;
#pragma unroll 4
  for (int i = threadIdx.x; i < nr * (ST / V); i += kConvThreads) {
    const int row = i / (ST / V), sl = i % (ST / V) * V;
    if (sl >= live) continue;
    const float4 v = reinterpret_cast<const float4*>(src)[i];
    buf[sl][row] = v.x;
    buf[sl + 1][row] = v.y;
    buf[sl + 2][row] = v.z;
    buf[sl + 3][row] = v.w;
  }
  __syncthreads();
  const int r = threadIdx.x % R;
  if (r >= nr) return;
  float* dst = nat + (size_t)t * ST * rows + inv[h0 + r];
#pragma unroll 8
  for (int sl = threadIdx.x / R; sl < live; sl += kConvThreads / R) dst[(size_t)sl * rows] = buf[sl][r];
}

// ---------------------------------------------------------------------------
// CGLS vector updates.  Grid (kVecBlocks, ntiles); a thread visits elements
// i = tid*W + k*stride of its tile; stride is a multiple of st, so each thread
// always touches the same W slices and keeps their sums in registers.
// Per-block partial sums are reduced in a fixed order (deterministic).
// ---------------------------------------------------------------------------

// part[W], pmax[W] per thread -> per-slice block totals.  Threads `per` = st /
// W apart hold the same slices: lanes by shuffles, then the warps in order
// through shared memory (one thread adding 256 pairs per slice took most of
// a small vector's update: 20 -> 4 us a kernel at 128^2 x 180, one slice).
template <int W>
__device__ void block_slice_sums(FF* part, uint32_t* pmax, int st, int tile,
                                 double* out_part, uint32_t* out_max, int nbx) {
  __shared__ FF sd[kVecThreads / 32][64];
  __shared__ uint32_t sm[kVecThreads / 32][64];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int per = st / W;
  for (int o = 16; o >= per; o >>= 1)
#pragma unroll
    for (int w = 0; w < W; ++w) {
      if (part) part[w] = ff_add(part[w], ff_shfl_xor(part[w], o));
      if (pmax) pmax[w] = max(pmax[w], __shfl_xor_sync(0xffffffffu, pmax[w], o));
    }
  if (lane < per)
#pragma unroll
    for (int w = 0; w < W; ++w) {
      sd[warp][lane * W + w] = part ? part[w] : FF{0.0f, 0.0f};
      sm[warp][lane * W + w] = pmax ? pmax[w] : 0u;
    }
  __syncthreads();
  for (int sl = threadIdx.x; sl < st; sl += blockDim.x) {
    FF acc = sd[0][sl];
    uint32_t mx = sm[0][sl];
    for (int k = 1; k < kVecThreads / 32; ++k) {
      acc = ff_add(acc, sd[k][sl]);
      mx = max(mx, sm[k][sl]);
    }
    const int gs = tile * st + sl;
    if (out_part) out_part[(size_t)gs * nbx + blockIdx.x] = ff_to_double(acc);
    if (out_max && mx) atomicMax(&out_max[gs], mx);
  }
  __syncthreads();
}

// W consecutive floats (one 16-byte access for W = 4: element offsets are
// multiples of 4 and every tile starts on a 16-byte boundary)
template <int W>
__device__ __forceinline__ void ldw(const float* p, float (&v)[W]) {
  if constexpr (W == 4) {
    const float4 t = *reinterpret_cast<const float4*>(p);
    v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
  } else {
#pragma unroll
    for (int w = 0; w < W; ++w) v[w] = p[w];
  }
}
template <int W>
__device__ __forceinline__ void stw(float* p, const float (&v)[W]) {
  if constexpr (W == 4) {
    *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
  } else {
#pragma unroll
    for (int w = 0; w < W; ++w) p[w] = v[w];
  }
}

// x += alpha p (image); r -= alpha q (sinogram); max |r|, ||r||^2 partials
template <int W>
__global__ void __launch_bounds__(kVecThreads) update_xr_kernel(
    float* __restrict__ x, const float* __restrict__ p, int64_t npix_len,
    float* __restrict__ r, const float* __restrict__ q, int64_t nray_len, int st,
    const double* __restrict__ alpha, uint32_t* __restrict__ max_r, double* __restrict__ rpart) {
  allow_next();
  wait_previous();
  x = after_wait(x);
  p = after_wait(p);
  r = after_wait(r);
  q = after_wait(q);
  alpha = after_wait(alpha);
  const int tile = blockIdx.y;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x * W;
  const int64_t start = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) * W;
  const int sl0 = (int)(start % st);
  float a[W];
#pragma unroll
  for (int w = 0; w < W; ++w) a[w] = (float)alpha[tile * st + sl0 + w];
  float* xt = x + (size_t)tile * npix_len;
  const float* pt = p + (size_t)tile * npix_len;
  for (int64_t i = start; i < npix_len; i += stride) {
    float xv[W], pv[W];
    ldw<W>(xt + i, xv);
    ldw<W>(pt + i, pv);
#pragma unroll
    for (int w = 0; w < W; ++w) xv[w] = fmaf(a[w], pv[w], xv[w]);
    stw<W>(xt + i, xv);
  }
  float* rt = r + (size_t)tile * nray_len;
  const float* qt = q + (size_t)tile * nray_len;
  FF ss[W];
  uint32_t mx[W];
#pragma unroll
  for (int w = 0; w < W; ++w) { ss[w] = FF{0.0f, 0.0f}; mx[w] = 0u; }
  for (int64_t i = start; i < nray_len; i += stride) {
    float rv[W], qv[W];
    ldw<W>(rt + i, rv);
    ldw<W>(qt + i, qv);
#pragma unroll
    for (int w = 0; w < W; ++w) {
      rv[w] = fmaf(-a[w], qv[w], rv[w]);
      ss[w] = ff_add(ss[w], ff_sq(rv[w]));
      mx[w] = max(mx[w], __float_as_uint(fabsf(rv[w])));
    }
    stw<W>(rt + i, rv);
  }
  block_slice_sums<W>(ss, mx, st, tile, rpart, max_r, gridDim.x);
}

// p = s + beta p; max |p|
template <int W>
__global__ void __launch_bounds__(kVecThreads) update_p_kernel(
    float* __restrict__ p, const float* __restrict__ s, int64_t npix_len, int st,
    const double* __restrict__ beta, uint32_t* __restrict__ max_p) {
  allow_next();
  wait_previous();
  p = after_wait(p);
  s = after_wait(s);
  beta = after_wait(beta);
  const int tile = blockIdx.y;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x * W;
  const int64_t start = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) * W;
  const int sl0 = (int)(start % st);
  float bt[W];
  uint32_t mx[W];
#pragma unroll
  for (int w = 0; w < W; ++w) { bt[w] = (float)beta[tile * st + sl0 + w]; mx[w] = 0u; }
  float* ptile = p + (size_t)tile * npix_len;
  const float* stile = s + (size_t)tile * npix_len;
  for (int64_t i = start; i < npix_len; i += stride) {
    float pv[W], sv[W];
    ldw<W>(ptile + i, pv);
    ldw<W>(stile + i, sv);
#pragma unroll
    for (int w = 0; w < W; ++w) {
      pv[w] = fmaf(bt[w], pv[w], sv[w]);
      mx[w] = max(mx[w], __float_as_uint(fabsf(pv[w])));
    }
    stw<W>(ptile + i, pv);
  }
  block_slice_sums<W>(nullptr, mx, st, tile, nullptr, max_p, gridDim.x);
}

// r = r - q (x0 start) with max |r|; ||r||^2 partials of r (a = 0: only sums)
template <int W>
__global__ void __launch_bounds__(kVecThreads) residual_kernel(
    float* __restrict__ r, const float* __restrict__ q, int64_t nray_len, int st,
    uint32_t* __restrict__ max_r, double* __restrict__ rpart) {
  allow_next();
  wait_previous();
  r = after_wait(r);
  q = after_wait(q);
  const int tile = blockIdx.y;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x * W;
  const int64_t start = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) * W;
  float* rt = r + (size_t)tile * nray_len;
  const float* qt = q ? q + (size_t)tile * nray_len : nullptr;
  FF ss[W];
  uint32_t mx[W];
#pragma unroll
  for (int w = 0; w < W; ++w) { ss[w] = FF{0.0f, 0.0f}; mx[w] = 0u; }
  for (int64_t i = start; i < nray_len; i += stride) {
    float rv[W];
    ldw<W>(rt + i, rv);
    if (qt) {
      float qv[W];
      ldw<W>(qt + i, qv);
#pragma unroll
      for (int w = 0; w < W; ++w) rv[w] = rv[w] - qv[w];
      stw<W>(rt + i, rv);
    }
#pragma unroll
    for (int w = 0; w < W; ++w) {
      ss[w] = ff_add(ss[w], ff_sq(rv[w]));
      mx[w] = max(mx[w], __float_as_uint(fabsf(rv[w])));
    }
  }
  block_slice_sums<W>(ss, mx, st, tile, rpart, max_r, gridDim.x);
}

// r = q - y (data-fit residual of the regularised reconstruction); max |r|,
// ||r||^2 partials
template <int W>
__global__ void __launch_bounds__(kVecThreads) sub_kernel(const float* __restrict__ q,
                                                          const float* __restrict__ y,
                                                          float* __restrict__ r, int64_t len, int st,
                                                          uint32_t* __restrict__ max_r,
                                                          double* __restrict__ rpart) {
  allow_next();
  wait_previous();
  q = after_wait(q);
  y = after_wait(y);
  const int tile = blockIdx.y;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x * W;
  const int64_t start = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) * W;
  const float* qt = q + (size_t)tile * len;
  const float* yt = y + (size_t)tile * len;
  float* rt = r + (size_t)tile * len;
  FF ss[W];
  uint32_t mx[W];
#pragma unroll
  for (int w = 0; w < W; ++w) { ss[w] = FF{0.0f, 0.0f}; mx[w] = 0u; }
  for (int64_t i = start; i < len; i += stride) {
    float qv[W], yv[W], rv[W];
    ldw<W>(qt + i, qv);
    ldw<W>(yt + i, yv);
#pragma unroll
    for (int w = 0; w < W; ++w) {
      rv[w] = qv[w] - yv[w];
      ss[w] = ff_add(ss[w], ff_sq(rv[w]));
      mx[w] = max(mx[w], __float_as_uint(fabsf(rv[w])));
    }
    stw<W>(rt + i, rv);
  }
  block_slice_sums<W>(ss, mx, st, tile, rpart, max_r, gridDim.x);
}

// The same on natural vectors (one slice a row of the grid, no maxima): a
// block takes whole pieces of 8 values a thread, and the partials past the
// grid's blocks are zero.  Bound by memory; 1024 x 720 x 16 slices: 59 us with
// sub_kernel (under 3 values a thread, each block's sum for them) -> 24.
constexpr int kFlat = 8;
__global__ void __launch_bounds__(kVecThreads) sub_flat_kernel(const float* __restrict__ q,
                                                               const float* __restrict__ y,
                                                               float* __restrict__ r, int64_t len,
                                                               double* __restrict__ rpart) {
  const float* qt = q + (size_t)blockIdx.y * len;
  const float* yt = y + (size_t)blockIdx.y * len;
  float* rt = r + (size_t)blockIdx.y * len;
  FF ss[1] = {{0.0f, 0.0f}};
  for (int64_t b = blockIdx.x * (int64_t)(kVecThreads * kFlat); b < len;
       b += gridDim.x * (int64_t)(kVecThreads * kFlat)) {
    float v[kFlat];
#pragma unroll
    for (int k = 0; k < kFlat; ++k) {
      const int64_t i = b + k * kVecThreads + threadIdx.x;
      v[k] = i < len ? qt[i] - yt[i] : 0.0f;
    }
#pragma unroll
    for (int k = 0; k < kFlat; ++k) {
      const int64_t i = b + k * kVecThreads + threadIdx.x;
      if (i < len) rt[i] = v[k];
      ss[0] = ff_add(ss[0], ff_sq(v[k]));
    }
  }
  block_slice_sums<1>(ss, nullptr, 1, blockIdx.y, rpart, nullptr, kVecBlocks);
  for (int k = blockIdx.x + gridDim.x * (threadIdx.x + 1); k < kVecBlocks; k += gridDim.x * kVecThreads)
    rpart[(size_t)blockIdx.y * kVecBlocks + k] = 0.0;
}

// loss = sum over slices s < S of 0.5 ||r_s||^2 + tv[s]  (one block)
__global__ void loss_kernel(const double* __restrict__ rpart, int nbr, const double* __restrict__ tv,
                            int S, double* __restrict__ out) {
  __shared__ double sh[kVecThreads];
  double part[8] = {};   // independent: loads and adds overlap (16 slices: 24 -> 9 us)
  int k = threadIdx.x;
  for (; k + 7 * kVecThreads < S * nbr; k += 8 * kVecThreads)
#pragma unroll
    for (int j = 0; j < 8; ++j) part[j] += 0.5 * rpart[k + j * kVecThreads];
  for (; k < S * nbr; k += kVecThreads) part[0] += 0.5 * rpart[k];
  double a = ((part[0] + part[1]) + (part[2] + part[3])) + ((part[4] + part[5]) + (part[6] + part[7]));
  for (int i = threadIdx.x; i < S; i += blockDim.x) a += tv[i];
  sh[threadIdx.x] = a;
  __syncthreads();
  for (int o = blockDim.x / 2; o > 0; o >>= 1) {
    if ((int)threadIdx.x < o) sh[threadIdx.x] += sh[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) *out = sh[0];
}

// ---------------------------------------------------------------------------
// scalars: one block per slice, fixed-order tree reduction of partials
// ---------------------------------------------------------------------------

// sums of N arrays of n[k] partials each, in thread 0; the arrays' loads and
// additions overlap, and below 32 values the tree goes on in a warp's
// registers (the same additions as through shared memory, without five of its
// eight barriers; a 128^2 solve of 5 iterations: 395 -> 386 us)
template <int N>
__device__ __forceinline__ void block_reduce_fixed(const double* const (&part)[N], const int (&n)[N],
                                                   double (&sum)[N]) {
  __shared__ double sh[N][kVecThreads];
#pragma unroll
  for (int k = 0; k < N; ++k) {
    // four independent accumulators per thread (loads and adds overlap),
    // combined in a fixed order
    double a0 = 0.0, a1 = 0.0, a2 = 0.0, a3 = 0.0;
    const int step = blockDim.x;
    int i = threadIdx.x;
    for (; i + 3 * step < n[k]; i += 4 * step) {
      a0 += part[k][i];
      a1 += part[k][i + step];
      a2 += part[k][i + 2 * step];
      a3 += part[k][i + 3 * step];
    }
    for (; i < n[k]; i += step) a0 += part[k][i];
    sh[k][threadIdx.x] = (a0 + a1) + (a2 + a3);
  }
  __syncthreads();
  for (int o = kVecThreads / 2; o >= 32; o >>= 1) {
    if ((int)threadIdx.x < o)
#pragma unroll
      for (int k = 0; k < N; ++k) sh[k][threadIdx.x] += sh[k][threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x < 32)
#pragma unroll
    for (int k = 0; k < N; ++k) {
      double v = sh[k][threadIdx.x];
      for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
      sum[k] = v;
    }
}

// after the initial back projection: gamma = ||s||^2, log[0]
__global__ void __launch_bounds__(kVecThreads) cgls_init_kernel(
    const double* gpart, int nbg, const double* rpart, int nbr, CglsScalars sc, double* log,
    int S_pad) {
  allow_next();
  wait_previous();
  const int gs = blockIdx.x;
  double sums[2];
  block_reduce_fixed<2>({gpart + (size_t)gs * nbg, rpart + (size_t)gs * nbr}, {nbg, nbr}, sums);
  const double g = sums[0], rr = sums[1];
  if (threadIdx.x == 0) {
    sc.gamma[gs] = g;
    const int act = g > 0.0;
    sc.active[gs] = act;
    sc.active0[gs] = act;
    sc.beta[gs] = 0.0;
    sc.max_p[gs] = 0u;
    if (log) {
      log[(size_t)gs * 2] = sqrt(rr);
      log[(size_t)gs * 2 + 1] = sqrt(g);
    }
  }
}

// delta = ||q||^2; alpha = gamma / delta (0 for a stopped slice)
__global__ void __launch_bounds__(kVecThreads) cgls_alpha_kernel(const double* dpart, int nbd,
                                                                 CglsScalars sc) {
  allow_next();
  wait_previous();
  const int gs = blockIdx.x;
  double sums[1];
  block_reduce_fixed<1>({dpart + (size_t)gs * nbd}, {nbd}, sums);
  const double d = sums[0];
  if (threadIdx.x == 0) {
    int act = sc.active[gs] && d > 0.0;
    sc.active[gs] = act;
    sc.alpha[gs] = act ? sc.gamma[gs] / d : 0.0;
    sc.max_r[gs] = 0u;
  }
}

// gamma' = ||s||^2; beta = gamma'/gamma; log[k]
__global__ void __launch_bounds__(kVecThreads) cgls_beta_kernel(const double* gpart, int nbg,
                                                                const double* rpart, int nbr,
                                                                CglsScalars sc, double* log_k) {
  allow_next();
  wait_previous();
  const int gs = blockIdx.x;
  double sums[2];
  block_reduce_fixed<2>({gpart + (size_t)gs * nbg, rpart + (size_t)gs * nbr}, {nbg, nbr}, sums);
  const double g = sums[0], rr = sums[1];
  if (threadIdx.x == 0) {
    const int act = sc.active[gs];
    sc.beta[gs] = act ? g / sc.gamma[gs] : 0.0;
    if (act) sc.gamma[gs] = g;
    sc.active[gs] = act && g > 0.0;
    sc.max_p[gs] = 0u;
    if (log_k) {
      log_k[(size_t)gs * 2] = sqrt(rr);
      log_k[(size_t)gs * 2 + 1] = sqrt(g);
    }
  }
}

// resume from a saved state: gamma and the activity flags of the first S
// slices (padding slices inactive), log[0] from the residual partials
__global__ void __launch_bounds__(kVecThreads) cgls_restore_kernel(
    const double* gamma_in, const int32_t* active_in, int S, const double* rpart, int nbr,
    CglsScalars sc, double* log) {
  const int gs = blockIdx.x;
  double sums[1];
  block_reduce_fixed<1>({rpart + (size_t)gs * nbr}, {nbr}, sums);
  const double rr = sums[0];
  if (threadIdx.x == 0) {
    const double g = gs < S ? gamma_in[gs] : 0.0;
    const int act = gs < S ? active_in[gs] : 0;
    sc.gamma[gs] = g;
    sc.active[gs] = act;
    sc.active0[gs] = act;
    sc.beta[gs] = 0.0;
    if (log) {
      log[(size_t)gs * 2] = sqrt(rr);
      log[(size_t)gs * 2 + 1] = sqrt(g);
    }
  }
}

// save: gamma and the activity flags of the first S slices, and the header
__global__ void cgls_save_kernel(const CglsScalars sc, int S, CglsStateHeader hdr,
                                 CglsStateHeader* hdr_out, double* gamma_out, int32_t* active_out) {
  for (int s = threadIdx.x; s < S; s += blockDim.x) {
    gamma_out[s] = sc.gamma[s];
    active_out[s] = sc.active[s];
  }
  if (threadIdx.x == 0) *hdr_out = hdr;
}

// f(integral constant of the tile width; pick_slices_per_tile gives none below 4)
template <class F>
xct_status by_width(int st, F f) {
  switch (st) {
    case 4: XCT_TRY_CUDA(f(std::integral_constant<int, 4>())); break;
    case 8: XCT_TRY_CUDA(f(std::integral_constant<int, 8>())); break;
    case 16: XCT_TRY_CUDA(f(std::integral_constant<int, 16>())); break;
    case 32: XCT_TRY_CUDA(f(std::integral_constant<int, 32>())); break;
    case 64: XCT_TRY_CUDA(f(std::integral_constant<int, 64>())); break;
    default: return XCT_ERR_UNSUPPORTED;
  }
  count_launch();
  return XCT_OK;
}

}  // namespace

xct_status to_internal(const float* nat, float* in, const int32_t* inv_order, int64_t rows, int S,
                       int st, int ntiles, uint32_t* max_bits, cudaStream_t s) {
  return by_width(st, [&](auto w) {
    constexpr int ST = decltype(w)::value, R = conv_rows(ST);
    return launch_early(to_internal_kernel<ST>, dim3((unsigned)((rows + R - 1) / R), (unsigned)ntiles), kConvThreads, 0, s,
                        nat, in, inv_order, rows, S, max_bits);
  });
}

xct_status to_natural(const float* in, float* nat, const int32_t* inv_order, int64_t rows, int S,
                      int st, int ntiles, cudaStream_t s) {
  return by_width(st, [&](auto w) {
    constexpr int ST = decltype(w)::value, R = conv_rows(ST);
    return launch_early(to_natural_kernel<ST>, dim3((unsigned)((rows + R - 1) / R), (unsigned)ntiles), kConvThreads, 0, s,
                        in, nat, inv_order, rows, S);
  });
}

#define XCT_VEC_LAUNCH(KERNEL, BLOCKS, ...)                                           \
  do {                                                                                \
    dim3 grid_((unsigned)(BLOCKS), (unsigned)ntiles);                                         \
    if (st % 4 == 0) XCT_TRY_CUDA(launch_early(KERNEL<4>, grid_, kVecThreads, 0, s, __VA_ARGS__)); \
    else XCT_TRY_CUDA(launch_early(KERNEL<1>, grid_, kVecThreads, 0, s, __VA_ARGS__)); \
    count_launch();                                                                   \
  } while (0)

int vec_blocks(int64_t rows, int st) {
  const int64_t per = (int64_t)kVecThreads * (st % 4 == 0 ? 4 : 1);
  return (int)std::min<int64_t>(std::max<int64_t>((rows * st + per - 1) / per, 1), kVecBlocks);
}

xct_status cgls_update_xr(float* x, const float* p, int64_t npix, float* r, const float* q,
                          int64_t nray, int st, int ntiles, const CglsScalars& sc, double* rpart,
                          int nblk, cudaStream_t s) {
  XCT_VEC_LAUNCH(update_xr_kernel, nblk, x, p, npix * st, r, q, nray * st, st, sc.alpha, sc.max_r, rpart);
  return XCT_OK;
}

xct_status cgls_update_p(float* p, const float* sv, int64_t npix, int st, int ntiles,
                         const CglsScalars& sc, cudaStream_t s) {
  XCT_VEC_LAUNCH(update_p_kernel, vec_blocks(npix, st), p, sv, npix * st, st, sc.beta, sc.max_p);
  return XCT_OK;
}

xct_status cgls_residual(float* r, const float* q, int64_t nray, int st, int ntiles,
                         uint32_t* max_r, double* rpart, int nblk, cudaStream_t s) {
  XCT_VEC_LAUNCH(residual_kernel, nblk, r, q, nray * st, st, max_r, rpart);
  return XCT_OK;
}

xct_status vec_sub_sumsq(const float* q, const float* y, float* r, int64_t rows, int st,
                         int ntiles, uint32_t* max_r, double* rpart, cudaStream_t s) {
  if (st == 1 && !max_r) {
    const int64_t per = (int64_t)kVecThreads * kFlat;
    const dim3 grid((unsigned)std::min<int64_t>(std::max<int64_t>((rows + per - 1) / per, 1), kVecBlocks),
                    (unsigned)ntiles);
    sub_flat_kernel<<<grid, kVecThreads, 0, s>>>(q, y, r, rows, rpart);
    count_launch();
    XCT_TRY_CUDA(cudaGetLastError());
    return XCT_OK;
  }
  XCT_VEC_LAUNCH(sub_kernel, kVecBlocks, q, y, r, rows * st, st, max_r, rpart);
  return XCT_OK;
}

xct_status vec_loss(const double* rpart, const double* tv, int S, double* out, cudaStream_t s) {
  loss_kernel<<<1, kVecThreads, 0, s>>>(rpart, kVecBlocks, tv, S, out);
  count_launch();
  XCT_TRY_CUDA(cudaGetLastError());
  return XCT_OK;
}

xct_status cgls_init_scalars(const double* gpart, int nbg, const double* rpart, int nbr,
                             const CglsScalars& sc, double* log, int S_pad, cudaStream_t s) {
  XCT_TRY_CUDA(launch_early(cgls_init_kernel, S_pad, kVecThreads, 0, s, gpart, nbg, rpart, nbr, sc, log, S_pad));
  count_launch();
  return XCT_OK;
}

xct_status cgls_alpha(const double* dpart, int nbd, const CglsScalars& sc, int S_pad,
                      cudaStream_t s) {
  XCT_TRY_CUDA(launch_early(cgls_alpha_kernel, S_pad, kVecThreads, 0, s, dpart, nbd, sc));
  count_launch();
  return XCT_OK;
}

xct_status cgls_beta(const double* gpart, int nbg, const double* rpart, int nbr,
                     const CglsScalars& sc, double* log_k, int S_pad, cudaStream_t s) {
  XCT_TRY_CUDA(launch_early(cgls_beta_kernel, S_pad, kVecThreads, 0, s, gpart, nbg, rpart, nbr, sc, log_k));
  count_launch();
  return XCT_OK;
}

xct_status cgls_restore(const double* gamma_in, const int32_t* active_in, int S,
                        const double* rpart, int nbr, const CglsScalars& sc, double* log, int S_pad,
                        cudaStream_t s) {
  cgls_restore_kernel<<<S_pad, kVecThreads, 0, s>>>(gamma_in, active_in, S, rpart, nbr, sc,
                                                     log);
  count_launch();
  XCT_TRY_CUDA(cudaGetLastError());
  return XCT_OK;
}

xct_status cgls_save(const CglsScalars& sc, int S, const CglsStateHeader& hdr,
                     CglsStateHeader* hdr_out, double* gamma_out, int32_t* active_out,
                     cudaStream_t s) {
  cgls_save_kernel<<<1, 256, 0, s>>>(sc, S, hdr, hdr_out, gamma_out, active_out);
  count_launch();
  XCT_TRY_CUDA(cudaGetLastError());
  return XCT_OK;
}

}  // namespace xct
