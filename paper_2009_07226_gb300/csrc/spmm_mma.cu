// Products of 16-bit slices on the tensor cores (octet layouts, OctLayout).
//
// An octet of 8 neighbouring rows crosses few distinct columns of a stage
// (2 bins x 4 angles of A: a third of the octet's rows on average hold each
// of them), so its entries are stored as dense 16-column x 8-row chunks and a
// chunk times ST slices is ST / 16 mma.m16n8k16 instructions: slices as the
// MMA's rows, the octet's rows as its columns, FP32 accumulators.  The staged
// rows that a chunk names are gathered from shared memory by ldmatrix with
// transposition, 8 arbitrary rows per phase; row chunks are permuted by the
// row's id (stage_natural_kernel) and the plan gives a phase's rows distinct
// ids mod 8, so a phase is conflict-free.
//
// A persistent CTA per SM: a scheduler warp walks the stages and requests
// their descriptors, copy warps stream each stage (one bulk copy per run of
// staged rows and one for the stage's chunks) into a ring of stage buffers,
// 16 consumer warps take one octet each and write its rows in the caller's
// layout.
//
// What bounds it (512^2 x 768 x 512, binary16): with 64 slices shared memory,
// where a chunk's 16 gathered rows (2048 bytes) and its values and positions
// (288) take 19 wavefronts of 128 bytes, 0.37 ms of the product for its 6.2 M
// chunks, and the copies write the stages: 0.68 ms per xct_project, 0.65 per
// xct_backproject, 0.05 to 0.07 of them staging, against 1.45 / 1.41 on the
// paired row layouts (spmm_pipe.cu) with their conversions; 32 slices 0.40 /
// 0.38, 16 slices 0.33 / 0.32 and 8 slices 0.31 / 0.30 (the FMA kernels alone
// 0.77 / 0.76, 0.49 / 0.50 and 0.45 / 0.43), there close to the chunks' stream
// from device memory (1.8 GB, 0.27 ms).  At 1536^2 x 1024, 32 slices, the
// stream of 32 GB takes 4.8 ms of the 5.8 at the measured copy bandwidth.
// tcgen05 would want 64 or more rows an operand tile, where only a tenth of the
// cells are entries: more bytes from device memory than the sparse form needs.
#include <algorithm>
#include <atomic>
#include <type_traits>

#include "pipe.cuh"
#include "xct_internal.cuh"

namespace xct {
namespace {

constexpr int kMmaWarps = kOcts;                 // consumer warps
constexpr int kMaxBufs = 4;                      // stage buffers, a copy warp for each
constexpr int kSlots = 2 * kMaxBufs;             // stage descriptors in flight
// of a tile width: with 32 and 64 slices no more than 3 fit (2 with 64 on a
// large grid), and 20 warps may use 96 registers where 21 may use 80
constexpr int max_bufs(int st) { return st >= 32 ? 3 : kMaxBufs; }
constexpr int mma_threads(int st) { return (kMmaWarps + 1 + max_bufs(st)) * 32; }
constexpr size_t kMmaSmem = 227 * 1024;          // of one CTA per SM
constexpr uint32_t kHdrBytes = 16 * kMmaWarps;   // stage header: 16 bytes for every consumer warp
constexpr uint32_t kFirst = 1, kLast = 2, kEnd = 4, kReal = 8;   // of its block; no more work; has entries

struct MmaArgs {
  const int64_t* blk_stage;
  const uint2* chunks;
  const unsigned char* desc;
  int64_t desc_bytes;
  const unsigned char* ent;
  int64_t nrows, ncols;
  int nblocks, nwork, angle_rows, pairs, S;
  const unsigned char* xs;   // staged rows [tile][ncols][ROWB bytes]
  float* y;                  // natural [S][nrows]
  const int32_t* row_inv;    // row -> natural id
  const uint32_t* in_max;
  int mat_scale_exp;
  int nbufs;
  uint32_t xbytes, ebytes, dbytes;   // region sizes (128-byte multiples)
  int* work;
  int* err;
  uint64_t wait_ns;
};

// d = a b (no accumulation)
__device__ __forceinline__ void mma_16816(float (&d)[4], const uint32_t (&a)[4], uint2 b, __half) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%10,%10,%10,%10};"
      : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b.x), "r"(b.y), "f"(0.0f));
}
__device__ __forceinline__ void mma_16816(float (&d)[4], const uint32_t (&a)[4], uint2 b, __nv_bfloat16) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%10,%10,%10,%10};"
      : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b.x), "r"(b.y), "f"(0.0f));
}
__device__ __forceinline__ void ldsm_x4_t(uint32_t (&r)[4], uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr)
               : "memory");
}
__device__ __forceinline__ void ldsm_x2_t(uint32_t& r0, uint32_t& r1, uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0,%1}, [%2];"
               : "=r"(r0), "=r"(r1)
               : "r"(addr)
               : "memory");
}
__device__ __forceinline__ uint32_t lds_u16(uint32_t addr) {
  uint16_t v;
  asm volatile("ld.shared.u16 %0, [%1];" : "=h"(v) : "r"(addr) : "memory");
  return v;
}
__device__ __forceinline__ uint2 lds_v2(uint32_t addr) {
  uint2 v;
  asm volatile("ld.shared.v2.u32 {%0,%1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(addr) : "memory");
  return v;
}
__device__ __forceinline__ float to_f32(uint32_t bits, __half) {
  return __half2float(__ushort_as_half((unsigned short)bits));
}
__device__ __forceinline__ float to_f32(uint32_t bits, __nv_bfloat16) { return __uint_as_float(bits << 16); }

// a wait by a whole warp: the same answer in every lane
__device__ __forceinline__ bool warp_wait(uint64_t* bar, uint32_t parity, uint64_t limit_ns) {
  return __all_sync(0xffffffffu, mbar_wait(bar, parity, limit_ns));
}
// acc += d, two sums in one instruction, each rounded to nearest.  The MMA
// truncates as it adds to its accumulator (a bias that grows with the number
// of chunks), so chunks are summed here instead.
__device__ __forceinline__ void add2(float* acc, const float* d) {
  const float2 s = __fadd2_rn(make_float2(acc[0], acc[1]), make_float2(d[0], d[1]));
  acc[0] = s.x;
  acc[1] = s.y;
}
// sum = or += a chunk times MT * 16 slices
template <bool FIRST, class TX, int MT>
__device__ __forceinline__ void chunk_times(float (&sum)[MT][4], const uint32_t (&x)[MT][4], uint2 w) {
#pragma unroll
  for (int i = 0; i < MT; ++i) {
    if constexpr (FIRST) {
      mma_16816(sum[i], x[i], w, TX());
    } else {
      float d[4];
      mma_16816(d, x[i], w, TX());
      add2(sum[i], d);
      add2(sum[i] + 2, d + 2);
    }
  }
}
// to += what
template <int MT>
__device__ __forceinline__ void add_sums(float (&to)[MT][4], const float (&what)[MT][4]) {
#pragma unroll
  for (int i = 0; i < MT; ++i) {
    add2(to[i], what[i]);
    add2(to[i] + 2, what[i] + 2);
  }
}
// acc + low += d, low taking what acc's rounding loses (two-sum, Knuth)
__device__ __forceinline__ void add_exact(float& acc, float& low, float d) {
  const float s = __fadd_rn(acc, d), v = __fsub_rn(s, acc);
  low = __fadd_rn(low, __fadd_rn(__fsub_rn(acc, __fsub_rn(s, v)), __fsub_rn(d, v)));
  acc = s;
}

template <class TX, int ST>
__global__ void __launch_bounds__(mma_threads(ST), 1) spmm_mma_kernel(MmaArgs a) {
  constexpr int ROWB = 2 * ST;                        // bytes of a staged row
  constexpr int MT = ST < 16 ? 1 : ST / 16;           // MMAs per chunk
  constexpr int HN = ST < 16 ? 1 : 2;                 // 8-slice halves of an MMA's rows in use
  constexpr int SH = oct_swz_shift(ROWB), MASK = oct_swz_mask(ROWB);
  extern __shared__ __align__(128) unsigned char smem[];
  const int NB = a.nbufs;
  const uint32_t bufbytes = a.xbytes + a.ebytes + kHdrBytes;
  // [stage buffers][descriptor slots][barriers][stage identities]
  unsigned char* dslots = smem + NB * bufbytes;
  uint64_t* full = reinterpret_cast<uint64_t*>(dslots + kSlots * a.dbytes);
  uint64_t* empty = full + kMaxBufs;
  uint64_t* dbar = empty + kMaxBufs;
  uint64_t* dfree = dbar + kSlots;
  int2* ident = reinterpret_cast<int2*>(dfree + kSlots);
  auto xbuf = [&](int b) { return smem + b * bufbytes; };
  auto ebuf = [&](int b) { return smem + b * bufbytes + a.xbytes; };
  auto wbuf = [&](int b) { return reinterpret_cast<uint4*>(smem + b * bufbytes + a.xbytes + a.ebytes); };

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (tid == 0) {
    for (int b = 0; b < NB; ++b) {
      mbar_init(&full[b], 1);
      mbar_init(&empty[b], kMmaWarps);
    }
    for (int k = 0; k < kSlots; ++k) {
      mbar_init(&dbar[k], 1);
      mbar_init(&dfree[k], 1);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();

  if (warp == kMmaWarps) {
    // ----------------------------- scheduler ----------------------------
    // Walks the stages of the CTA's blocks (claimed from the work counter,
    // the next one while the current one is walked), and for every stage
    // writes its identity (work item, flags), requests its descriptor into a
    // ring of slots and a prefetch of its chunks, which come from device
    // memory, into L2.
    uint32_t it = 0;
    bool ok = true;
    auto emit = [&](int w, uint32_t flags, int64_t st, uint32_t c0, uint32_t nch) {
      const int ds = (int)(it % kSlots);
      if (!warp_wait(&dfree[ds], ((it / kSlots) & 1) ^ 1, a.wait_ns)) return false;
      if (lane == 0) {
        ident[ds] = make_int2(w, (int)flags);
        if (flags & kReal) {
          asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
          mbar_arrive_tx(&dbar[ds], (uint32_t)a.desc_bytes);
          bulk_g2s(dslots + (size_t)ds * a.dbytes, a.desc + (size_t)st * a.desc_bytes, (uint32_t)a.desc_bytes,
                   &dbar[ds]);
          if (nch) bulk_prefetch_l2(a.ent + (size_t)c0 * kChunkBytes, nch * (uint32_t)kChunkBytes);
        } else {
          mbar_arrive(&dbar[ds]);
        }
      }
      ++it;
      return true;
    };
    int next = 0;
    if (lane == 0) next = atomicAdd(a.work, 1);
    while (ok) {
      const int w = __shfl_sync(0xffffffffu, next, 0);
      if (w >= a.nwork) break;
      const int64_t s0 = a.blk_stage[w % a.nblocks], s1 = a.blk_stage[w % a.nblocks + 1];
      if (lane == 0) next = atomicAdd(a.work, 1);
      const int nst = (int)(s1 - s0);
      if (nst == 0) ok = emit(w, kFirst | kLast, 0, 0, 0);
      uint2 ck = make_uint2(0u, 0u);   // lane j: first chunk and chunks of stage (k & ~31) + j
      for (int k = 0; k < nst && ok; ++k) {
        if ((k & 31) == 0 && k + lane < nst) ck = __ldg(a.chunks + s0 + k + lane);
        const uint32_t c0 = __shfl_sync(0xffffffffu, ck.x, k & 31), nch = __shfl_sync(0xffffffffu, ck.y, k & 31);
        ok = emit(w, kReal | (k == 0 ? kFirst : 0u) | (k == nst - 1 ? kLast : 0u), s0 + k, c0, nch);
      }
    }
    // the end, once for every copy warp (only the first tells the consumers)
    for (int k = 0; k < NB && ok; ++k) ok = emit(k, kEnd, 0, 0, 0);
    // The descriptors requested land before the CTA's shared memory goes
    // away, here too when every request was accepted: work that fits the
    // slots is emitted without a wait, and a copy warp may have given up on
    // its descriptor since.  (A slot's earlier requests were read before it
    // was free for the last one.)
    if (!ok && lane == 0) atomicExch(a.err, 1);
    for (uint32_t j = it > (uint32_t)kSlots ? it - kSlots : 0; j < it; ++j)
      mbar_wait(&dbar[j % kSlots], (j / kSlots) & 1, kDrainNs);
    return;
  }
  if (warp > kMmaWarps) {
    // ---------------------------- copy warps ----------------------------
    // Copy warp c fills buffer c, with stages c, c + NB, ...: one warp's chain
    // of waits, header and copy issues takes longer (about 0.7 us) than the
    // consumers need for a stage, so the buffers' stages are set up at the
    // same time, all but the copies before the buffer is free.  (A buffer has
    // one filler: with another assignment a warp could test the buffer's
    // barrier two phases early, where the parity looks the same.  A
    // descriptor slot is safe with 2 NB <= kSlots: stage it - 2 NB was
    // released by the consumers before this warp filled stage it - NB.)
    const int buf = warp - kMmaWarps - 1;
    if (buf >= NB) return;
    uint32_t use = 0;
    for (uint32_t it = (uint32_t)buf;; it += NB, ++use) {
      const int ds = (int)(it % kSlots);
      bool ok = warp_wait(&dbar[ds], (it / kSlots) & 1, a.wait_ns);
      const int2 id = ident[ds];
      if (ok && (id.y & kEnd) && id.x > 0) {
        // the copies of this warp's last stage land first: consumers that
        // gave up do not wait for them
        if (use > 0) mbar_wait(&full[buf], (use - 1) & 1, kDrainNs);
        return;
      }
      const bool real = ok && (id.y & kReal) != 0;
      const unsigned char* dd = dslots + (size_t)ds * a.dbytes;
      const OctStageHead& dh = *reinterpret_cast<const OctStageHead*>(dd);
      const int2* rl = reinterpret_cast<const int2*>(dd + sizeof(OctStageHead));
      const uint32_t eb = real ? dh.nch * (uint32_t)kChunkBytes : 0u;
      const uint32_t xb = real ? dh.np * (uint32_t)ROWB : 0u;
      const int nruns = real ? (int)dh.nr - 1 : 0;
      const unsigned char* src = a.ent + (real ? (size_t)dh.c0 * kChunkBytes : 0);
      const unsigned char* xt = a.xs + (size_t)(real ? id.x / a.nblocks : 0) * a.ncols * ROWB;
      int2 run = make_int2(0, 0);
      uint32_t len = 0;
      if (lane < nruns) {
        run = rl[lane];
        len = (uint32_t)(rl[lane + 1].y - run.y) * ROWB;
      }
      // for consumer warp w: {first chunk << 16 | chunks of its octet, chunks
      // of the stage, work item, flags}
      uint4 word = make_uint4(0u, real ? dh.nch : 0u, (uint32_t)id.x, (uint32_t)id.y);
      if (real && lane < kOcts) word.x = (uint32_t)dh.ofs[lane] << 16 | (uint32_t)(dh.ofs[lane + 1] - dh.ofs[lane]);
      ok = ok && warp_wait(&empty[buf], (use & 1) ^ 1, a.wait_ns);
      if (!ok) {
        // let the copies of this warp's last stage land
        if (lane == 0) atomicExch(a.err, 1);
        if (use > 0) mbar_wait(&full[buf], (use - 1) & 1, kDrainNs);
        return;
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      if (lane == 0 && real) {
        mbar_expect_tx(&full[buf], xb + eb);
        // chunks are read once, staged rows by many blocks: without the hint
        // the chunks pushed them out of L2 (1536^2 x 1024: 16 slices 5.56 ->
        // 5.10 ms, 32 slices 7.68 -> 7.11; 512^2 x 768, 64 slices: 1%)
        if (eb) bulk_g2s_once(ebuf(buf), src, eb, &full[buf]);
      }
      __syncwarp();
      unsigned char* xd = xbuf(buf);
      if (len) bulk_g2s(xd + (size_t)run.y * ROWB, xt + (size_t)run.x * ROWB, len, &full[buf]);
      for (int k = lane + 32; k < nruns; k += 32) {
        const int2 r = rl[k];
        bulk_g2s(xd + (size_t)r.y * ROWB, xt + (size_t)r.x * ROWB, (uint32_t)(rl[k + 1].y - r.y) * ROWB, &full[buf]);
      }
      if (lane < kOcts) wbuf(buf)[lane] = word;
      __syncwarp();
      if (lane == 0) {
        mbar_arrive(&full[buf]);   // the phase's single arrival; publishes the header
        mbar_arrive(&dfree[ds]);
      }
      if (id.y & kEnd) return;   // (the stage before was consumed: the buffer was free)
    }
  }

  // ------------------------------ consumers ------------------------------
  // lane 4 g + t: slices 16 i + g and 16 i + 8 + g of octet rows 2 t, 2 t + 1
  const int g = lane >> 2, t = lane & 3;
  // the row of a chunk whose address this lane gives to ldmatrix, and the
  // 8-slice half it reads of it
  const int lk = ST < 16 ? (lane & 15) : (lane & 7) + ((lane >> 4) << 3);
  const uint32_t lh = ST < 16 ? 0u : (uint32_t)(lane >> 3) & 1u;
  // A row's 50 to 150 chunks added one after the other err more than the row
  // layouts, whose rows several lanes share, with 8 and 64 slices.  There the
  // chunks of a stage are summed first, then the stages: for 8 slices with
  // what their rounding loses, for 64 bfloat16 ones into two sums in turn.
  // Error of sums of positive terms at 400^2 x 300, in 10^-9 of the sum (rms;
  // rows, one level, as here): 8 slices binary16 86, 162, 34, bfloat16 45, 138,
  // 27; 64 slices 159, 162, 70 and 74, 138, 47; 16 and 32 slices, in one level,
  // 306, 162 and 177, 138.  512^2 x 768: 8 slices 0.308 -> 0.311 ms, 64 slices
  // binary16 0.685 -> 0.680, bfloat16 0.685 -> 0.704 (scales formed at a
  // block's end, out of the loop's registers: 64 slices 0.697 -> 0.680).
  constexpr bool EXACT = ST == 8, TWO = ST == 64;
  constexpr int NA = TWO && std::is_same<TX, __nv_bfloat16>::value ? 2 : 1;
  float acc[NA][MT][4];
  float low[EXACT ? 4 : 1];
  bool second = false;   // the sum that takes the next stage
  bool finite = true;
  int buf = 0;
  uint32_t use = 0;
  for (;;) {
    if (!warp_wait(&full[buf], use & 1, a.wait_ns)) {
      if (lane == 0) atomicExch(a.err, 1);
      return;
    }
    const uint4 word = wbuf(buf)[warp];
    if (word.w & kEnd) break;
    if (word.w & kFirst) {
      const uint32_t* im = a.in_max + (word.z / (uint32_t)a.nblocks) * ST;
      uint32_t big = 0;
      second = false;
#pragma unroll
      for (int i = 0; i < MT; ++i)
#pragma unroll
        for (int q = 0; q < HN; ++q) {
          const uint32_t mb = __ldg(im + 16 * i + 8 * q + g);
          // (or is so small, at most 2^-128, that its scale is infinite)
          big |= mb >= 0x7f800000u || mb - 1u < 0x00200000u;
        }
      finite = !__any_sync(0xffffffffu, big != 0u);
#pragma unroll
      for (int i = 0; i < MT; ++i)
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
          for (int k = 0; k < NA; ++k) acc[k][i][q] = 0.0f;
      if constexpr (EXACT)
#pragma unroll
        for (int q = 0; q < 4; ++q) low[q] = 0.0f;
    }
    if (word.x & 0xffffu) {
      const int c0 = (int)(word.x >> 16), n = (int)(word.x & 0xffffu);
      const uint32_t xb = su32(xbuf(buf));
      const uint32_t eb = su32(ebuf(buf));
      const uint32_t pb = eb + word.y * 256u;
      auto row_addr = [&](uint32_t pos) {
        return xb + pos * ROWB + ((lh ^ ((pos >> SH) & MASK)) << 4);
      };
      if (finite) {
        float own[MT][4] = {};
        float (&part)[MT][4] = EXACT || TWO ? own : acc[0];   // takes the stage's chunks
        uint32_t pa = pb + c0 * 32 + lk * 2, wa = eb + c0 * 256 + lane * 8;
        auto gather = [&](uint32_t (&x)[MT][4], uint32_t pos) {
          const uint32_t ad = row_addr(pos);
          if constexpr (ST >= 16) {
#pragma unroll
            for (int i = 0; i < MT; ++i) ldsm_x4_t(x[i], ad ^ (uint32_t)(i << 5));
          } else {
            ldsm_x2_t(x[0][0], x[0][2], ad);
            x[0][1] = x[0][3] = 0u;
          }
        };
        // U chunks at a time, the next U chunks' positions and values loaded
        // while they are multiplied (512^2 x 768 x 512, projection: 64
        // slices 0.701 ms with U = 1, 0.720 with 2; 32 slices 0.412, 0.416;
        // 16 slices 0.362, 0.361, 0.352 with 3)
        constexpr int U = MT >= 2 ? 1 : 3;
        uint32_t p[U];
        uint2 w[U];
        auto fetch = [&](int left) {
#pragma unroll
          for (int u = 0; u < U; ++u)
            if (left > u) {
              p[u] = lds_u16(pa + u * 32u);
              w[u] = lds_v2(wa + u * 256u);
            }
          pa += U * 32u;
          wa += U * 256u;
        };
        fetch(n);
        int left = n;
        if constexpr (TWO) {   // the first chunk: no sum to add it to
          uint32_t x[MT][4];
          gather(x, p[0]);
          const uint2 wc = w[0];
          fetch(--left);
          chunk_times<true, TX>(part, x, wc);
        }
        for (; left >= U; left -= U) {
          uint32_t x[U][MT][4];
          uint2 wc[U];
#pragma unroll
          for (int u = 0; u < U; ++u) {
            gather(x[u], p[u]);
            wc[u] = w[u];
          }
          fetch(left - U);
#pragma unroll
          for (int u = 0; u < U; ++u) chunk_times<false, TX>(part, x[u], wc[u]);
        }
#pragma unroll
        for (int u = 0; u < U - 1; ++u)
          if (u < left) {
            uint32_t x[MT][4];
            gather(x, p[u]);
            chunk_times<false, TX>(part, x, w[u]);
          }
        if constexpr (EXACT) {
#pragma unroll
          for (int q = 0; q < 4; ++q) add_exact(acc[0][0][q], low[q], part[0][q]);
        } else if constexpr (TWO) {
          if (NA > 1 && second)
            add_sums(acc[NA - 1], part);
          else
            add_sums(acc[0], part);
          second = !second;
        }
      } else {
        // a slice of this tile is staged with infinities or NaN: 0 times it in a
        // chunk's unused cells would reach rows that do not cross it, so the
        // entries are taken one by one
        for (int c = c0; c < c0 + n; ++c)
          for (int k = 0; k < 16; ++k) {
            const uint32_t pos = lds_u16(pb + c * 32 + k * 2);
            const uint32_t wk = eb + c * 256 + ((k & 7) >> 1) * 8 + ((k >> 3) * 2 + (k & 1)) * 2;
            const uint32_t w0 = lds_u16(wk + (2 * t) * 32), w1 = lds_u16(wk + (2 * t + 1) * 32);
#pragma unroll
            for (int i = 0; i < MT; ++i)
#pragma unroll
              for (int q = 0; q < HN; ++q) {
                const float xv = to_f32(
                    lds_u16(xb + pos * ROWB + (((uint32_t)(2 * i + q) ^ ((pos >> SH) & MASK)) << 4) + g * 2), TX());
                if (w0 & 0x7fffu) acc[0][i][2 * q] = fmaf(to_f32(w0, TX()), xv, acc[0][i][2 * q]);
                if (w1 & 0x7fffu) acc[0][i][2 * q + 1] = fmaf(to_f32(w1, TX()), xv, acc[0][i][2 * q + 1]);
              }
          }
      }
    }
    __syncwarp();
    if (lane == 0) mbar_arrive(&empty[buf]);
    if (word.w & kLast) {
      if constexpr (EXACT) {
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[0][0][q] += low[q];
      } else if constexpr (NA > 1) {
        add_sums(acc[0], acc[NA - 1]);
      }
      // ---- epilogue of a block: de-normalise, write to the natural layout
      // (the lane's two rows are neighbouring bins or pixels of a full tile)
      const int tile = (int)(word.z / (uint32_t)a.nblocks), b = (int)(word.z % (uint32_t)a.nblocks);
      const int p = (warp & 7) * 8 + 2 * t;
      const int64_t base = (int64_t)b * kOctRows + (warp >> 3) * 64;
      const int64_t r0 = base + oct_row(p, a.angle_rows), r1 = base + oct_row(p + 1, a.angle_rows);
      const bool v0 = r0 < a.nrows, v1 = r1 < a.nrows;
      const int64_t n0 = v0 ? __ldg(a.row_inv + r0) : 0, n1 = v1 ? __ldg(a.row_inv + r1) : 0;
      const bool two = a.pairs && v0 && v1 && n1 == n0 + 1 && (n0 & 1) == 0;
#pragma unroll
      for (int i = 0; i < MT; ++i)
#pragma unroll
        for (int q = 0; q < HN; ++q) {
          const int sl = tile * ST + 16 * i + 8 * q + g;
          if (sl >= a.S) continue;
          float* dst = a.y + (size_t)sl * a.nrows;
          const uint32_t mb = __ldg(a.in_max + tile * ST + 16 * i + 8 * q + g);
          const float scale = ldexpf(1.0f, ceil_log2_exp_p(__uint_as_float(mb)) - a.mat_scale_exp);
          const float u = acc[0][i][2 * q] * scale, v = acc[0][i][2 * q + 1] * scale;
          if (two) {
            *reinterpret_cast<float2*>(dst + n0) = make_float2(u, v);
          } else {
            if (v0) dst[n0] = u;
            if (v1) dst[n1] = v;
          }
        }
    }
    if (++buf == NB) {
      buf = 0;
      ++use;
    }
  }
}

size_t align128(size_t n) { return (n + 127) / 128 * 128; }

// shared memory besides the stage buffers
size_t fixed_smem(size_t dbytes) {
  return kSlots * dbytes + 8 * (2 * kMaxBufs + 2 * kSlots) + 8 * kSlots + 128;
}

// stage buffers that fit a CTA, at most `most`
int buffers(size_t xbytes, size_t ebytes, size_t dbytes, int most) {
  const size_t fixed = fixed_smem(dbytes);
  if (fixed >= kMmaSmem) return 0;
  const size_t n = (kMmaSmem - fixed) / (xbytes + ebytes + kHdrBytes);
  return n < (size_t)most ? (int)n : most;
}

// ---------------------------------------------------------------------------
// staging: natural FP32 vectors -> normalised 16-bit rows as ldmatrix reads
// them, with no FP32 copy in the ordered layout between
// ---------------------------------------------------------------------------

// max |x| of every slice (float bits)
__global__ void __launch_bounds__(256) slice_max_kernel(const float* __restrict__ x, int64_t len,
                                                        int S, uint32_t* __restrict__ out) {
  const int64_t i0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, step = (int64_t)gridDim.x * blockDim.x;
  for (int s = blockIdx.y; s < S; s += gridDim.y) {
    const float* p = x + (size_t)s * len;
    uint32_t m = 0;
    int64_t i = i0;
    if ((reinterpret_cast<uintptr_t>(p) & 15) == 0) {
      const int64_t n4 = len >> 2;
      for (; i < n4; i += step) {
        const float4 v = __ldg(reinterpret_cast<const float4*>(p) + i);
        m = max(max(m, max(__float_as_uint(fabsf(v.x)), __float_as_uint(fabsf(v.y)))),
                max(__float_as_uint(fabsf(v.z)), __float_as_uint(fabsf(v.w))));
      }
      i = (n4 << 2) + i0;
    }
    for (; i < len; i += step) m = max(m, __float_as_uint(fabsf(p[i])));
    m = __reduce_max_sync(0xffffffffu, m);
    if ((threadIdx.x & 31) == 0 && m) atomicMax(out + s, m);
  }
}

__device__ __forceinline__ uint32_t round16(float v, __half) { return __half_as_ushort(__float2half_rn(v)); }
__device__ __forceinline__ uint32_t round16(float v, __nv_bfloat16) {
  return __bfloat16_as_ushort(__float2bfloat16_rn(v));
}

// kStageRows ordered rows of one slice tile per block: read with the rows
// fastest (a Hilbert tile's rows are short contiguous pieces of the natural
// layout), transposed in shared memory, written as whole staged rows.  Bound
// by memory: 6 bytes an element; the FP32 source was read once before, for
// the maxima, and comes largely from L2.
constexpr int kStageRows = 64;
template <class TX, int ST>
__global__ void __launch_bounds__(256) stage_natural_kernel(const float* __restrict__ nat,
                                                            const int32_t* __restrict__ inv, int64_t rows, int S,
                                                            const uint32_t* __restrict__ in_max,
                                                            unsigned char* __restrict__ out) {
  __shared__ float buf[ST][kStageRows + 1];
  __shared__ float isc[ST];
  const int64_t h0 = (int64_t)blockIdx.x * kStageRows;
  const int s0 = blockIdx.y * ST;
  const int r = threadIdx.x % kStageRows;
  const bool in = h0 + r < rows;
  const int64_t id = in ? inv[h0 + r] : 0;
  for (int i = threadIdx.x; i < ST; i += 256)
    isc[i] = ldexpf(1.0f, -ceil_log2_exp_p(__uint_as_float(in_max[s0 + i])));
#pragma unroll 8
  for (int sl = threadIdx.x / kStageRows; sl < ST; sl += 256 / kStageRows)
    buf[sl][r] = in && s0 + sl < S ? nat[(size_t)(s0 + sl) * rows + id] : 0.0f;
  __syncthreads();
  constexpr int C = ST / 8;   // 16-byte chunks of a row
  constexpr int SH = oct_swz_shift(2 * ST), MASK = oct_swz_mask(2 * ST);
  uint4* dst = reinterpret_cast<uint4*>(out + ((size_t)blockIdx.y * rows + h0) * (2 * ST));
  for (int i = threadIdx.x; i < kStageRows * C; i += 256) {
    const int row = i / C, c = i % C;
    if (h0 + row >= rows) break;
    uint32_t w[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int sl = c * 8 + 2 * j;
      w[j] = round16(buf[sl][row] * isc[sl], TX()) | round16(buf[sl + 1][row] * isc[sl + 1], TX()) << 16;
    }
    dst[row * C + (c ^ (((uint32_t)(h0 + row) >> SH) & MASK))] = make_uint4(w[0], w[1], w[2], w[3]);
  }
}

template <class TX, int ST>
xct_status launch_stage(const OctLayout& L, const OctProduct& p, cudaStream_t st) {
  const int ntiles = (p.S + ST - 1) / ST;
  if (L.ncols == 0) return XCT_OK;
  XCT_TRY_CUDA(cudaMemsetAsync(p.in_max, 0, sizeof(uint32_t) * ntiles * ST, st));
  const int64_t mb = (L.ncols + 256 * 16 - 1) / (256 * 16);
  const dim3 mgrid((unsigned)std::min<int64_t>(mb, 64), (unsigned)std::min(p.S, 65535));
  slice_max_kernel<<<mgrid, 256, 0, st>>>(p.x, L.ncols, p.S, p.in_max);
  const dim3 sgrid((unsigned)((L.ncols + kStageRows - 1) / kStageRows), (unsigned)ntiles);
  stage_natural_kernel<TX, ST><<<sgrid, 256, 0, st>>>(p.x, p.col_inv, L.ncols, p.S, p.in_max,
                                                      reinterpret_cast<unsigned char*>(p.staged));
  count_launch(2);
  XCT_TRY_CUDA(cudaGetLastError());
  return XCT_OK;
}

template <class TX, int ST>
xct_status launch_mma(const OctLayout& L, const OctProduct& p, cudaStream_t st) {
  const int ntiles = (p.S + ST - 1) / ST;
  if (L.nblocks == 0) return XCT_OK;
  XCT_TRY_CUDA(cudaMemsetAsync(p.work, 0, sizeof(int), st));
  MmaArgs a{};
  a.blk_stage = L.blk_stage;
  a.chunks = L.chunks;
  a.desc = L.desc;
  a.desc_bytes = L.desc_bytes;
  a.ent = L.ent;
  a.nrows = L.nrows;
  a.ncols = L.ncols;
  a.nblocks = L.nblocks;
  a.nwork = L.nblocks * ntiles;
  a.angle_rows = L.angle_rows;
  a.pairs = (reinterpret_cast<uintptr_t>(p.y) & 7) == 0 && L.nrows % 2 == 0;
  a.S = p.S;
  a.xs = reinterpret_cast<const unsigned char*>(p.staged);
  a.y = p.y;
  a.row_inv = p.row_inv;
  a.in_max = p.in_max;
  a.mat_scale_exp = p.mat_scale_exp;
  a.work = p.work;
  a.err = p.err;
  a.wait_ns = wait_limit_ns();
  a.xbytes = (uint32_t)align128((size_t)L.cap * 2 * ST);
  a.ebytes = (uint32_t)align128((size_t)L.emax * kChunkBytes);
  a.dbytes = (uint32_t)align128((size_t)L.desc_bytes);
  a.nbufs = buffers(a.xbytes, a.ebytes, a.dbytes, max_bufs(ST));
  const size_t smem = fixed_smem(a.dbytes) + a.nbufs * (size_t)(a.xbytes + a.ebytes + kHdrBytes);
  int dev = 0, sms = 0;
  XCT_TRY_CUDA(cudaGetDevice(&dev));
  XCT_TRY_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  static std::atomic<bool> configured[kMaxDevices];
  if (dev < 0 || dev >= kMaxDevices || !configured[dev].load()) {
    XCT_TRY_CUDA(cudaFuncSetAttribute(spmm_mma_kernel<TX, ST>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)kMmaSmem));
    if (dev >= 0 && dev < kMaxDevices) configured[dev].store(true);
  }
  spmm_mma_kernel<TX, ST><<<a.nwork < sms ? a.nwork : sms, mma_threads(ST), smem, st>>>(a);
  count_launch();
  XCT_TRY_CUDA(cudaGetLastError());
  return XCT_OK;
}

// f(TX(), integral constant of the tile width)
template <class F>
xct_status by_tile(xct_dtype storage, int st, F f) {
  const bool h = storage == XCT_F16;
#define XCT_TILE(N) \
  case N: return h ? f(__half(), std::integral_constant<int, N>()) : f(__nv_bfloat16(), std::integral_constant<int, N>())
  switch (st) {
    XCT_TILE(8);
    XCT_TILE(16);
    XCT_TILE(32);
    XCT_TILE(64);
    default:
      set_error("octet product: unsupported tile width %d", st);
      return XCT_ERR_UNSUPPORTED;
  }
#undef XCT_TILE
}

}  // namespace

bool oct_stage_fits(int cap, int64_t emax, int64_t desc_bytes) {
  return buffers(align128((size_t)cap * 128), align128((size_t)emax * kChunkBytes), align128((size_t)desc_bytes), 2) >= 2;
}

xct_status oct_stage(const OctLayout& L, const OctProduct& p, xct_dtype storage, cudaStream_t s) {
  return by_tile(storage, p.st, [&](auto tx, auto n) { return launch_stage<decltype(tx), decltype(n)::value>(L, p, s); });
}

xct_status oct_run(const OctLayout& L, const OctProduct& p, xct_dtype storage, cudaStream_t s) {
  return by_tile(storage, p.st, [&](auto tx, auto n) { return launch_mma<decltype(tx), decltype(n)::value>(L, p, s); });
}

xct_status oct_product(const OctLayout& L, const OctProduct& p, xct_dtype storage, cudaStream_t s) {
  XCT_TRY(oct_stage(L, p, storage, s));
  return oct_run(L, p, storage, s);
}

}  // namespace xct
