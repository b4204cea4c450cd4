// Internal declarations of libxct.so (not part of the C-ABI).
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>
#include <map>
#include <vector>

#include <nvtx3/nvToolsExt.h>

#include "xct.h"

namespace xct {

// ---------------------------------------------------------------------------
// errors, allocation, launch accounting
// ---------------------------------------------------------------------------

void set_error(const char* fmt, ...);
// limit of the bounded waits inside the persistent kernels (xct_set_wait_limit)
uint64_t wait_limit_ns();
constexpr int kMaxDevices = 64;   // per-device caches of launch attributes
extern std::atomic<int64_t> g_launches;
inline void count_launch(int64_t k = 1) { g_launches.fetch_add(k, std::memory_order_relaxed); }

// Launches that overlap their predecessor's tail.  A kernel launched with
// launch_early may start once every block of the kernel before it on the
// stream has called allow_next (or ended); it calls wait_previous before it
// touches memory that other kernels write, and only constants of the plan
// before that.  The predecessor's results are visible after the wait, and a
// kernel that allows its successor waits itself, so order along the stream is
// kept.  (Solves of one 128^2 slice are a chain of 40 kernels of 2 to 15 us.)
__device__ __forceinline__ void allow_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void wait_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// the pointer as a new value, made after the wait: loads through a __restrict__
// parameter might otherwise be moved ahead of it
template <class T>
__device__ __forceinline__ T* after_wait(T* p) {
  asm volatile("" : "+l"(p) : : "memory");
  return p;
}
template <class... P, class... A>
cudaError_t launch_early(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, A&&... args) {
  cudaLaunchConfig_t c{};
  c.gridDim = grid;
  c.blockDim = block;
  c.dynamicSmemBytes = smem;
  c.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  c.attrs = at;
  c.numAttrs = 1;
  return cudaLaunchKernelEx(&c, kernel, static_cast<P>(args)...);
}

// Device allocation through the configured allocator (by default
// stream-ordered: working memory from the library's pool, memory that a plan
// keeps from the device's default pool).  Returns nullptr and sets the error
// message on failure.
void* dalloc(size_t bytes, cudaStream_t s, bool keep = false);
// a plan was made (1) or released (-1) on the device
void scratch_plans(int device, int change);
void dfree(void* p, size_t bytes, cudaStream_t s);

// An NVTX range for the duration of an entry point (a no-op unless a
// profiler is attached), so traces show the library's calls by name.
struct Trace {
  explicit Trace(const char* name) { nvtxRangePushA(name); }
  ~Trace() { nvtxRangePop(); }
  Trace(const Trace&) = delete;
  Trace& operator=(const Trace&) = delete;
};

// The fixed working array of xct_project_noalloc (noalloc.cu): resolve its
// device address on `device` (made current for the call, then restored), so
// that the array is resident there before the first call that relies on it.
xct_status noalloc_reserve(int device);

// (a failure is reported here: the runtime's record of it goes too, or the next
// check of that record, here or in another library, would report it again)
#define XCT_TRY_CUDA(call)                                                   \
  do {                                                                       \
    cudaError_t e_ = (call);                                                 \
    if (e_ != cudaSuccess) {                                                 \
      cudaGetLastError();                                                    \
      ::xct::set_error("%s failed: %s (%s:%d)", #call, cudaGetErrorString(e_), \
                       __FILE__, __LINE__);                                  \
      return XCT_ERR_CUDA;                                                   \
    }                                                                        \
  } while (0)

#define XCT_TRY(expr)                  \
  do {                                 \
    xct_status st_ = (expr);           \
    if (st_ != XCT_OK) return st_;     \
  } while (0)

// Lets blocks of a kernel ask for all the dynamic shared memory that a block
// may have, once per device.  (The limit belongs to the kernel, not to a
// launch: set to the size of each launch, one host thread could lower it
// between another's setting and launch.)
template <auto* Kernel>
xct_status allow_all_smem() {
  static std::atomic<bool> done[kMaxDevices];
  int dev = 0;
  XCT_TRY_CUDA(cudaGetDevice(&dev));
  const bool known = dev >= 0 && dev < kMaxDevices;
  if (known && done[dev].load()) return XCT_OK;
  cudaFuncAttributes at;
  int most = 0;
  XCT_TRY_CUDA(cudaFuncGetAttributes(&at, Kernel));
  XCT_TRY_CUDA(cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
  XCT_TRY_CUDA(cudaFuncSetAttribute(Kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    most - (int)at.sharedSizeBytes));
  if (known) done[dev].store(true);
  return XCT_OK;
}

// A set of device allocations released together (in reverse order).
struct Arena {
  struct Item { void* p; size_t n; };
  std::vector<Item> items;
  cudaStream_t stream = nullptr;
  bool keep = false;           // a plan's own memory
  explicit Arena(cudaStream_t s = nullptr, bool keep_ = false) : stream(s), keep(keep_) {}
  Arena(const Arena&) = delete;
  Arena& operator=(const Arena&) = delete;
  ~Arena() { release(); }
  template <class T>
  xct_status get(T** out, size_t count) {
    size_t bytes = count * sizeof(T);
    if (bytes == 0) bytes = 256;
    void* p = dalloc(bytes, stream, keep);
    if (!p) { *out = nullptr; return XCT_ERR_OOM; }
    items.push_back({p, bytes});
    *out = static_cast<T*>(p);
    return XCT_OK;
  }
  void release() {
    for (size_t i = items.size(); i-- > 0;) dfree(items[i].p, items[i].n, stream);
    items.clear();
  }
  // hand ownership of all items to another arena
  void move_to(Arena& other) {
    for (auto& it : items) other.items.push_back(it);
    items.clear();
  }
};

// storage forms: 16-bit matrix values; 16-bit (normalised) staged slices;
// binary16 (rather than bfloat16) values
inline bool matrix16(xct_dtype t) { return t != XCT_F32; }
inline bool stages16(xct_dtype t) { return t == XCT_F16 || t == XCT_BF16; }
inline bool half_values(xct_dtype t) { return t == XCT_F16 || t == XCT_F16A; }
inline bool valid_storage(int t) { return t >= XCT_F32 && t <= XCT_BF16A; }

// ---------------------------------------------------------------------------
// kernel layout of one matrix (A or A^T)
// ---------------------------------------------------------------------------

constexpr int kRowsPerBlock = 64;              // rows of one thread block
constexpr int kQuads = kRowsPerBlock / 4;      // 4-row groups per block

// Packed entries name their staged row by its byte offset at 128 bytes per
// row (position * 128): a tile with PIXB-byte staged rows finds the row at
// offset >> log2(128 / PIXB), one shift-add per entry.  16-bit entries hold
// {value bits (low 16), offset (high 16)}, FP32 entries {offset (low 32),
// value bits (high 32)}.  The offset of the zero slot (position cap) must fit
// in 16 bits.
constexpr int kEntryRowBytes = 128;
constexpr int kMaxStageCap = 65535 / kEntryRowBytes - 1;
// wide-stage layouts for few slices: 16-byte rows addressed at 16 bytes per
// row (up to 4094 rows a stage), entries streamed from global memory by the
// consumers instead of staged
constexpr int kWideRowBytes = 16;
// stage capacities (rows) of the wide layouts of A and A^T: 1524 rows of A
// (24 KB, four CTAs still fit an SM) measured 5% faster projections than
// 1016; for A^T 1016 measured best (762 and 1270 slower)
constexpr int kWideCapA = 1524;
constexpr int kWideCapAT = 1016;
constexpr int kWideGap = 16;
// log2(128 / pixb) for staged rows of pixb = 2 .. 128 bytes
__host__ __device__ constexpr int entry_shift(int pixb) {
  return pixb >= 128 ? 0 : pixb == 64 ? 1 : pixb == 32 ? 2 : pixb == 16 ? 3 : pixb == 8 ? 4
       : pixb == 4 ? 5 : 6;
}

// One (stage, quad) segment: the entries of 4 consecutive rows interleaved in
// chunks of 4 entries; `off` counts entries from the start of `ent`.
struct __align__(16) Seg {
  int64_t off;
  uint16_t cnt[4];
};

// A stage descriptor: what the persistent product's producer needs about
// one stage, stored at a fixed stride so that its address follows from the
// stage index alone and one bulk copy, requested several stages ahead, brings
// it in: the head, the stage's kQuads segment headers, then its run list
// padded to the layout's longest one with closing pairs.
struct __align__(16) StageDescHead {
  int64_t e0;          // first packed slot of the stage
  uint32_t slots;      // packed slots of the stage
  uint16_t np;         // staged rows
  uint16_t nr;         // run-list pairs (even)
};
inline int64_t stage_desc_bytes(int64_t run_stride) {
  return (int64_t)sizeof(StageDescHead) + kQuads * 16 + 8 * run_stride;
}

// Octet layout of one matrix for products of 16-bit slices on the tensor
// cores (spmm_mma.cu, built by octet_layout.cu).  A block is kOctRows
// consecutive rows; its input footprint is a list of aligned groups of 8
// columns, cut into stages of at most `cap` staged rows, a staged row's
// position being congruent to its column mod 8.  A block's rows form octets
// of 8 rows (for A 2 bins x 4 angles, for A^T 4 x 2 pixels of a tile), and
// an octet's entries in a stage form dense chunks: 16 columns (the distinct
// columns of the octet, 16 at a time) by 8 rows of 16-bit values.
//
// Chunk bytes: a stage's chunks are stored octet after octet as
// [chunk][lane][8 bytes] values (256 bytes a chunk: lane 4 n + t holds rows
// n of columns 2t, 2t + 1, 2t + 8, 2t + 9, the B fragment of an
// mma.m16n8k16), then [chunk][16] positions of 2 bytes.  Within a chunk the
// columns 0-7 and 8-15 have positions that are distinct mod 8 where the
// counts allow, so that the 8 row reads of one ldmatrix phase fall in
// distinct banks.  Unused columns carry value 0 and repeat a used position.
constexpr int kOctRows = 128;
constexpr int kOcts = kOctRows / 8;
// Row of a 64-row group at place p (octet p / 8) of the octet order.  A full
// tile of rays is numbered bin * 8 + angle: an octet takes 2 bins x 4 angles,
// the bin fastest; a full tile of pixels (2 x 2 groups) in its own order.
__host__ __device__ __forceinline__ int oct_row(int p, int angle_rows) {
  if (!angle_rows) return p;
  return (p & 48) | (p & 8) >> 1 | (p & 6) >> 1 | (p & 1) << 3;
}
constexpr int kChunkBytes = 256 + 32;
// first stage capacity tried, and the chunks of a stage at which it ends early
// (136: with 512 rows, two buffers of 128-byte rows, three of 64-byte ones and
// four of 32-byte ones fit a CTA).  A stage's fixed costs want large stages:
// projection of 8 slices at 512^2 x 768 0.35 ms with 384 rows, 0.46 with 256.
constexpr int kStageChunks = 136;
constexpr int kOctCap = 512;
// A stage's descriptor: this head, the first chunk of every octet (kOcts + 1
// numbers), padded to 16 bytes, then the runs of its staged rows as (first
// column, first position) pairs and closing pairs (-1, positions).
struct __align__(16) OctStageHead {
  int64_t c0;          // first chunk of the stage
  uint32_t nch;        // chunks of the stage
  uint16_t np;         // staged rows copied (columns past the matrix left out)
  uint16_t nr;         // run-list pairs, closing pair included
  uint16_t ofs[kOcts + 1];
};

struct OctLayout {
  int64_t nrows = 0, ncols = 0;
  int32_t nblocks = 0;
  int32_t cap = 0;             // staged rows of a stage, a multiple of 64
  int32_t angle_rows = 0;      // 1: rows are rays (see oct_row)
  int64_t nstages = 0, nchunks = 0;
  int64_t emax = 0;            // chunks of the largest stage
  int64_t* blk_stage = nullptr;   // [nblocks + 1]
  uint2* chunks = nullptr;        // [nstages] first chunk, chunks
  unsigned char* desc = nullptr;  // [nstages] descriptors of desc_bytes each
  int64_t desc_bytes = 0;
  unsigned char* ent = nullptr;   // chunk bytes, stage after stage
  int64_t bytes = 0;
};

struct Layout {
  int64_t nrows = 0, ncols = 0;
  int32_t nblocks = 0;
  int32_t cap = 0;             // staged vectors per stage (the zero slot is `cap`)
  int32_t ebytes = 0;          // 4: {u16 index, 16-bit value}; 8: {u32 index, f32}
  int64_t nstages = 0;
  int64_t nslots = 0;          // stored entries including padding
  int64_t footprint = 0;       // staged vectors over all stages
  int64_t fp_max = 0;          // staged vectors of the block with most
  int64_t* blk_stage = nullptr;   // [nblocks + 1] stage ranges of the blocks
  int64_t* stage_pix = nullptr;   // [nstages + 1] offsets into pix
  int32_t* stage_np = nullptr;    // [nstages] staged rows of each stage
  int32_t* pix = nullptr;         // staged input row ids, stage by stage
  Seg* seg = nullptr;             // [nstages * kQuads]
  void* ent = nullptr;            // packed entries
  int64_t* stage_ent = nullptr;   // [nstages + 1] first slot of each stage's entries
  int64_t emax_slots = 0;         // largest stage, in slots
  // contiguous runs of each stage's staged rows (see run_fill_kernel)
  int64_t* stage_run = nullptr;   // [nstages + 1] offsets into runs (even)
  int2* runs = nullptr;           // (first row id, first position) pairs
  int64_t nruns = 0;              // pairs over all stages
  int64_t run_max = 0;            // largest stage list, in pairs
  unsigned char* desc = nullptr;  // [nstages] stage descriptors of desc_bytes each
  int64_t desc_bytes = 0;
  // bytes per staged row in the entries' offsets (kEntryRowBytes, or 16 for
  // a wide-stage layout whose offsets address 16-byte rows directly)
  int32_t unit = kEntryRowBytes;
  // the wide-stage layout of the same matrix for 16-byte staged rows (built
  // with XCT_PLAN_FEW_SLICES), used in place of this one for such tiles
  const Layout* wide = nullptr;
  // the paired layout of the same matrix for 128-byte rows of 16-bit slices
  // (built with XCT_PLAN_PAIRED_ROWS), used in place of this one for such
  // tiles; `pair` marks a paired layout itself (its stages, staged rows and
  // runs are those of the plain layout, its segments and 8-byte slots its own)
  const Layout* paired = nullptr;
  bool pair = false;
  // the octet layout of the same matrix (see octets_for)
  const OctLayout* oct = nullptr;
  int64_t gathers = 0;         // paired: distinct columns of the pairs over all stages
                               // (the staged-row reads of one tile, padding aside)
  int64_t bytes = 0;
};

// Paired layout (XCT_PLAN_PAIRED_ROWS).  Rows 2p and 2p + 1 of a quad form
// pair p.  A pair's entries in a stage are split into shared slots, one per
// column both rows cross ({offset << 16 | value of row 2p, offset << 16 |
// value of row 2p + 1}), and split slots, one column of each row ({offset0 <<
// 16 | value0, offset1 << 16 | value1}, the zero slot with value 0 where one
// row has no entry left).  Two lanes of a pair take alternate slots (a chunk
// is 2 slots).  A (stage, quad) segment holds the shared region, then the
// split region; each region is a sequence of groups of kPairUA (shared) or
// kPairUB (split) chunks, and in a group the kPair* slots of each (pair, lane)
// are contiguous: slot u of lane e of pair p in group g of the shared region
// lies at g * 4 * kPairUA + (2 p + e) * kPairUA + u.  Seg::cnt holds the
// chunk counts {shared of pair 0, split of pair 0, shared of pair 1, split
// of pair 1}; each region has as many groups as its longer pair needs.
constexpr int kPairUA = 4;
constexpr int kPairUB = 2;

// Shared memory of one pipeline buffer (staged rows of `pixb` bytes, the
// stage's packed entries, its segment headers and header) with its share of
// the stage-descriptor slots (four slots over two buffers) -- see
// spmm_pipe.cu.
inline size_t pipe_buffer_bytes(const Layout& L, int pixb) {
  size_t x = ((size_t)(L.cap + 1) * pixb + 127) / 128 * 128;
  size_t e = ((size_t)L.emax_slots * L.ebytes + 127) / 128 * 128;
  size_t d = ((size_t)L.desc_bytes + 127) / 128 * 128;
  return x + e + 2 * d + 128 * 2 + 256;
}
#ifndef XCT_PIPE_BUFS
#define XCT_PIPE_BUFS 2
#endif
// stage buffers of a pipeline CTA (the producer fills up to kPipeBufs - 1
// stages ahead of the consumers)
constexpr int kPipeBufs = XCT_PIPE_BUFS;
static_assert(kPipeBufs == 2 || kPipeBufs == 3, "pipeline buffers");
// stage buffers and CTAs per SM of the pipeline with 16-byte staged rows
#ifndef XCT_PIPE_BUFS16
#define XCT_PIPE_BUFS16 2
#endif
#ifndef XCT_PIPE_MINB16
#define XCT_PIPE_MINB16 4
#endif
constexpr int kPipeBufs16 = XCT_PIPE_BUFS16;
constexpr int kPipeMinb16 = XCT_PIPE_MINB16;
// shared memory one pipeline CTA with 128-byte staged rows may use for its
// buffers (two such CTAs share an SM; the rest of a CTA's 113 KB goes to the
// barriers and run lists)
constexpr size_t kPipeSmemLimit = 110 * 1024;
// first stage capacity tried for each entry size (reduced until the buffers
// fit in kPipeSmemLimit)
constexpr int kPipeCap16 = kPipeBufs == 2 ? 280 : 184;
constexpr int kPipeCap32 = kPipeBufs == 2 ? 200 : 132;

struct Plan {
  xct_geometry g{};
  std::vector<double> cs;       // host angle table [M][2]
  xct_dtype storage = XCT_F32;
  uint32_t flags = 0;
  int device = 0;
  int64_t nray = 0, npix = 0, nnz = 0;
  int32_t* pix_order = nullptr;  // natural pixel -> ordered id
  int32_t* pix_inv = nullptr;    // ordered id -> natural pixel
  int32_t* ray_order = nullptr;
  int32_t* ray_inv = nullptr;
  Layout la, lat;
  Layout law, latw;              // wide-stage layouts (XCT_PLAN_FEW_SLICES)
  Layout lap, latp;              // paired layouts (XCT_PLAN_PAIRED_ROWS)
  OctLayout oa, oat;             // octet layouts (16-bit slices)
  int32_t mat_scale_exp = 0;     // k: stored value = RN(l * 2^k)
  int* err = nullptr;            // device flag: a bounded wait in a kernel ran out
  // kept FP64 matrices (ordered ids), only with XCT_PLAN_KEEP_F64
  int64_t* a_rowptr = nullptr; int32_t* a_col = nullptr; double* a_val = nullptr;
  int64_t* t_rowptr = nullptr; int32_t* t_col = nullptr; double* t_val = nullptr;
  Arena mem{nullptr, true};      // everything above lives here, but for
  Arena oct_mem{nullptr, true};  // the octet layouts (see OctUse)
  int oct_users = 0;             // products being enqueued on them
  bool oct_pinned = false;       // a captured graph refers to them
  xct_stats stats{};
  std::map<int, int> tile_choice;  // measured slice-tile width per slice count
};

// a matrix in ordered ids, as traced or transposed (FP64 values)
struct CsrView {
  const int64_t* rowptr;
  const int32_t* col;
  const double* val;
  int64_t nrows, ncols;
};
// How a block's footprint is ordered in an octet layout (see
// oct_order_kernel): the matrix's rows are rays (A) or pixels (A^T), with
// their and the columns' natural ids.
struct FootprintOrder {
  bool rays;
  const int32_t *row_inv, *col_inv;   // ordered -> natural ids
  const double* cs;                   // device [angles][2]
  int n, nd, tile;
};
// the octet layout of a matrix (octet_layout.cu); *fits is false, and
// nothing kept, when its stage buffers would not fit a product's CTA
xct_status build_oct_layout(const CsrView& m, xct_dtype storage, const FootprintOrder& order, OctLayout& L,
                            Arena& keep, bool* fits, cudaStream_t s);

// The octet layout that a product of the plan's matrix (or its transpose)
// between natural vectors runs on, for slice tiles of st; nullptr: it runs on
// the row layouts (FP32 slices; 8-slice tiles of a plan with wide-stage
// layouts, which stream fewer bytes: 0.20 - 0.23 ms against 0.31 at 512^2 x
// 768; a matrix whose octet layout did not fit, or a plan that asked for
// none).  On small grids too: 32^2 to 384^2, 1 to 100 binary16 slices, 21 to
// 587 us against 24 to 1189 on rows, but for 29 against 27 us for projections
// of up to 8 slices at 128^2, where both take one wave of blocks.  Products
// inside solves, and those whose FP64 cost is reported, stay on the row
// layouts: they keep each row's order of summation, so that logged residual
// norms and costs do not move.
inline const OctLayout* octets_for(const Plan& p, bool transposed, int st) {
  const Layout& L = transposed ? p.lat : p.la;
  return stages16(p.storage) && !(st == 8 && L.wide) ? L.oct : nullptr;
}

// A product's hold on the octet layout that it runs on, while it is enqueued
// (null: there is none).  When device memory runs out, the layouts of plans
// that no product is being enqueued on, and that no captured graph refers to,
// are given up (api.cu): solves and plans that would fit without them do.
class OctUse {
 public:
  OctUse(Plan& p, bool transposed, int st, cudaStream_t s);
  ~OctUse();
  OctUse(const OctUse&) = delete;
  OctUse& operator=(const OctUse&) = delete;
  explicit operator bool() const { return layout_ != nullptr; }
  const OctLayout& operator*() const { return *layout_; }

 private:
  Plan& plan_;
  const OctLayout* layout_;
};
// a plan whose octet layouts may be given up; before it is released, no more
void octets_may_go(Plan& p);
void octets_stay(Plan& p);
// in this thread, memory that runs out takes no other plan's octet layouts
struct KeepOctets {
  KeepOctets();
  ~KeepOctets();
};

// plan building (plan.cu)
xct_status build_plan(Plan& p, cudaStream_t s);
// y = A x without the stored matrix: every ray walked again (plan.cu)
xct_status matfree_project(const Plan& p, const double* cs_dev, const float* x, float* y, int S,
                           cudaStream_t s);
// x = A^T y without the stored matrix: pixel-driven, lengths from each
// pixel's boundary planes, equal to the stored values (plan.cu)
xct_status matfree_backproject(const Plan& p, const double* cs_dev, const float* y, float* x, int S,
                               cudaStream_t s);
// the double-precision form (f64.cu): products and CGLS on the kept FP64
// matrices, natural-layout device vectors; f64_cgls writes log [iters+1][S][2]
// (device, nullable) and whether any slice was active after the start
xct_status f64_apply(Plan& p, bool transposed, const double* in, double* out, int S,
                     cudaStream_t s);
xct_status f64_cgls(Plan& p, const double* y, double* x, int S, int iters, bool x0, double* log,
                    int* any_active, cudaStream_t s);
xct_status export_matrix(Plan& p, int what, int64_t* rowptr, int32_t* col,
                         double* val, int64_t* nnz);

// device exclusive scans (scan.cu): out[i] = sum_{j<i} in[j], out[n] = total
xct_status exclusive_scan_i32(const int32_t* in, int64_t* out, int64_t n, cudaStream_t s);
xct_status exclusive_scan_i64(const int64_t* in, int64_t* out, int64_t n, cudaStream_t s);

// ---------------------------------------------------------------------------
// products (spmm.cu) on the internal vector layout [tile][rows][st] float32
// ---------------------------------------------------------------------------

struct SpmmArgs {
  const Layout* L;
  const float* x;          // input [ntiles][L->ncols][st]
  float* y;                // output [ntiles][L->nrows][st]
  int st;                  // slices per tile
  int ntiles;
  xct_dtype storage;
  int mat_scale_exp;
  const uint32_t* in_max;  // per slice max |x| bits (16-bit storage) [ntiles*st]
  double* dot_partial;     // nullable: [ntiles*st][nblocks] sum of y^2 per block
  uint16_t* staged16;      // 16-bit storage: scratch [ntiles][L->ncols][st] for the
                           // normalised 16-bit copy of x (unused for FP32)
  int* work;               // scratch: one work counter (persistent form)
  int* err;                // device flag set to 1 if a bounded wait ran out
  bool work_zeroed = false;   // the work counter is zero already
};
// The layout a product runs on: the matrix's wide-stage layout, where the
// plan built one, for 16-byte staged rows of 16-bit slices; its paired
// layout, where the plan built one, for 128-byte staged rows of 16-bit
// slices; else its own.
inline SpmmArgs on_product_layout(SpmmArgs a) {
  if (a.L->wide && stages16(a.storage) && a.st * 2 == kWideRowBytes) a.L = a.L->wide;
  else if (a.L->paired && stages16(a.storage) && a.st * 2 == kEntryRowBytes) a.L = a.L->paired;
  return a;
}
// byte offset of the 16-byte chunk c of a 16-bit staged row of `rowb` bytes
// as octet products read it: chunks are permuted within the row by the
// row's id (congruent to its staged position mod 8), so that the same chunk
// of 8 rows of distinct ids mod 8 lies in 8 distinct 16-byte bank groups
__host__ __device__ constexpr int oct_swz_shift(int rowb) { return rowb >= 128 ? 0 : rowb == 64 ? 1 : 2; }
__host__ __device__ constexpr int oct_swz_mask(int rowb) { return rowb >= 128 ? 7 : rowb / 16 - 1; }
xct_status spmm(const SpmmArgs& a, cudaStream_t s);   // = spmm_stage + spmm_run
// 16-bit storage: the normalised 16-bit copy of the input (no-op for FP32)
xct_status spmm_stage(const SpmmArgs& a, cudaStream_t s);
// the product kernel itself
xct_status spmm_run(const SpmmArgs& a, cudaStream_t s);
// the persistent warp-specialised form (spmm_pipe.cu); false if it does not
// apply to this layout / tile width (the caller then uses the staged form)
bool spmm_pipe_applies(const SpmmArgs& a);
xct_status spmm_pipe(const SpmmArgs& a, cudaStream_t s);
// the direct form for a product of few blocks and 16-byte rows (spmm_pipe.cu)
bool spmm_direct_applies(const SpmmArgs& a);
xct_status spmm_direct(const SpmmArgs& a, cudaStream_t s);
// several products (same storage type, 128-byte rows) in one persistent
// launch sharing one work counter (list[0].work) -- the batched solver
constexpr int kMaxPipeProducts = 8;
bool spmm_pipe_multi_applies(const SpmmArgs* list, int count);
xct_status spmm_pipe_multi(const SpmmArgs* list, int count, cudaStream_t s);
// A product of 16-bit slices on an octet layout (spmm_mma.cu), between
// natural-layout device vectors.
struct OctProduct {
  const float* x;          // [S][ncols]
  float* y;                // [S][nrows]
  int S, st;               // slices, slices per tile
  const int32_t *col_inv, *row_inv;   // ordered -> natural ids
  int mat_scale_exp;
  uint32_t* in_max;        // scratch [ntiles * st]
  uint16_t* staged;        // scratch [ntiles][ncols][st]
  int* work;               // scratch: a work counter
  int* err;                // device flag set to 1 if a bounded wait ran out
};
// = oct_stage (reads x: maxima, staged rows) + oct_run (writes y)
xct_status oct_product(const OctLayout& L, const OctProduct& p, xct_dtype storage, cudaStream_t s);
xct_status oct_stage(const OctLayout& L, const OctProduct& p, xct_dtype storage, cudaStream_t s);
xct_status oct_run(const OctLayout& L, const OctProduct& p, xct_dtype storage, cudaStream_t s);
bool oct_stage_fits(int cap, int64_t emax, int64_t desc_bytes);
// number of per-slice partial sums spmm() writes for dot_partial (per slice):
// one per block of rows
int spmm_dot_count(const SpmmArgs& a);
bool spmm_supported(xct_dtype storage, int st);
int pick_slices_per_tile(xct_dtype storage, int S);

// regularisation (tv.cu)
xct_status tv_launch(const float* x, int n, int S, double eps, double weight, float* grad,
                     bool accumulate, double* partial, double* value_dev, cudaStream_t s);
int tv_partials(int n);
xct_status adam_launch(float* x, const float* g, float* m, float* v, int64_t count, double lr,
                       double beta1, double beta2, double eps, int step, cudaStream_t s);

// vector kernels (vec.cu)
xct_status to_internal(const float* nat, float* in, const int32_t* inv_order,
                       int64_t rows, int S, int st, int ntiles, uint32_t* max_bits,
                       cudaStream_t s);
xct_status to_natural(const float* in, float* nat, const int32_t* inv_order,
                      int64_t rows, int S, int st, int ntiles, cudaStream_t s);

}  // namespace xct

// The opaque handle of the C-ABI is the plan itself.
struct xct_plan_s : public xct::Plan {};
