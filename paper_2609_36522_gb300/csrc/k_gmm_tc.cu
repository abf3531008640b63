// Mixture denoiser on the tensor cores (tcgen05), three kernels:
//
//   k_gmm_dots_tc   partial dot products x . mu_k over a CTA's share of the
//                   columns, accumulated in TMEM
//   k_gmm_resp      a CTA per row: the partials summed, logits, max-subtracted
//                   softmax -> responsibilities R [row][component]
//   k_gmm_out_tc    eps = a x - a sqrt(a) R M, tiles of 128 columns x up to
//                   128 rows
//
// fp32 accuracy from shorter operands: every value is split in three bfloat16
// parts, which hold it exactly, and the products of parts down to 2^-26 of a
// product are added up in fp32.
//
// What bounds it: at 118 rows of 4x128x128 and 64 components a call reads the
// rows twice and the means twice and writes eps once, 126 MB (19 us at the copy
// rate, less for what the 126 MB L2 still holds). The two contractions are 1
// GFLOP each, in bfloat16 six to eight times that, 3 to 5 us on all SMs, so both large
// kernels are one CTA per SM that keeps copies in flight while the tensor core
// works: asynchronous copies into a ring of shared-memory stages, warps that
// split what has landed, one thread that issues a stage's MMAs as soon as it is
// full, mbarriers (tcgen05.commit) that free it again. Loads into registers
// cost the loop their latency wherever the value was moved. A
// row block belongs to a group of CTAs, so any row count fills the SMs about
// evenly; a CTA's partial sums of a row block have a place of their own, and R's
// kernel adds them in CTA order, so a result is reproducible bit for bit. The
// means are read as they lie: no image of them is kept.
//
// Every wait is bounded. A wait that runs out records kDevTimeout, the thread
// stops waiting, runs on with in-bounds accesses only, and eps is written as
// NaN.
#include <cmath>

#include "pa_bulk.cuh"
#include "pa_gmm_tc.h"
#include "pa_internal.h"
#include "pa_tcgen05.cuh"

namespace pa {
namespace {

constexpr int kRows = 128;       // rows of a row block: at most an MMA's N / 2
constexpr int kMaxCtas = 160;    // CTAs of the dot products at most (one per SM)
constexpr int kUnit = 32;        // columns of a piece of the dot products

// The CTAs that the dot products of up to max_rows rows keep busy, `limit` at most.
inline int dots_ctas(int64_t D, int max_rows, int limit) {
  const int64_t pieces = ((int64_t)max_rows + kRows - 1) / kRows * ((D + kUnit - 1) / kUnit);
  return pieces < limit ? (int)pieces : limit;
}

// components as stored: R rows and partial sums are padded to this many
__host__ __device__ inline int kpad(int K) { return K <= 16 ? 16 : K <= 32 ? 32 : K <= 64 ? 64 : 128; }

// How `blocks` row blocks of `units` column pieces each are shared by `grid`
// CTAs: up to `grid` blocks, each block has a group of neighbouring CTAs, which
// take its pieces in turn, so that at any time a group reads one contiguous
// stretch of every row (contiguous ranges per CTA measured the same); more
// blocks than CTAs, a CTA takes whole blocks in turn. A slot holds the sums of one CTA and block.
// (Rows that fit this GPU's memory make fewer than 2^31 pieces.)
struct Share {
  int blocks, units, grid;
  __device__ Share(int b, int u, int g) : blocks(b), units(u), grid(g) {}
  __device__ bool grouped() const { return blocks <= grid; }
  // the first CTA of a block's group; how many of the group have a piece
  // (32-bit: up to 160 CTAs and, where groups exist, as many blocks)
  __device__ int first(int blk) const { return (int)((uint32_t)(blk * grid + blocks - 1) / (uint32_t)blocks); }
  __device__ int members(int blk) const { return grouped() ? min(first(blk + 1) - first(blk), units) : 1; }
  // CTA `cta`'s first block (blocks or more: none), the step to its next one,
  // its first piece of a block and the step to its next one
  __device__ int block(int cta) const { return grouped() ? (int)((uint32_t)(cta * blocks) / (uint32_t)grid) : cta; }
  __device__ int block_step() const { return grouped() ? blocks : grid; }
  __device__ int unit(int cta, int blk) const { return grouped() ? cta - first(blk) : 0; }
  __device__ int unit_step(int blk) const { return grouped() ? first(blk + 1) - first(blk) : 1; }
  __device__ int slot(int blk, int member) const { return grouped() ? first(blk) + member : blk; }
};

// Eight values as three bfloat16 parts each, v = a + b + c exactly (8 + 8 + 8
// bits): 16 bytes per part, a half of a core-matrix pair's row.
struct Parts {
  uint4 a, b, c;
};
__device__ __forceinline__ uint32_t split2(float& x, float& y) {  // leaves what the part does not hold
  uint32_t p;
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(p) : "f"(y), "f"(x));
  x -= __uint_as_float(p << 16);
  y -= __uint_as_float(p & 0xffff0000u);
  return p;
}
__device__ __forceinline__ Parts split8(float4 u, float4 v) {
  Parts r;
  r.a = make_uint4(split2(u.x, u.y), split2(u.z, u.w), split2(v.x, v.y), split2(v.z, v.w));
  r.b = make_uint4(split2(u.x, u.y), split2(u.z, u.w), split2(v.x, v.y), split2(v.z, v.w));
  r.c = make_uint4(split2(u.x, u.y), split2(u.z, u.w), split2(v.x, v.y), split2(v.z, v.w));
  return r;
}

// Bounded wait (about a second) without a suspend-time hint: these barriers
// complete every few hundred nanoseconds. After a failure a thread no longer
// waits.
__device__ __forceinline__ void wait_or_fail(uint64_t* bar, uint32_t parity, bool* bad, int32_t* status) {
  if (*bad || mbar_test(bar, parity)) return;
  const long long t0 = clock64();
  while (!mbar_try(bar, parity)) {
    if (clock64() - t0 > 2000000000ll) {
      *bad = true;
      atomicCAS(status, 0, kDevTimeout);
      return;
    }
  }
}
__device__ __forceinline__ void named_sync(int id, int threads) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

// ---------------------------------------------------------------------------
// Dot products. A unit is kUnit columns of a row block. Every value is held
// exactly, as three bfloat16 parts a + b + c. The MMA's A operand is the means (M
// = 128 rows: parts a and b of 64 components, then part c above rows of zeros;
// for more than 64 components a part of 128), its B operand the rows (N: the
// block's rows, rounded up to 16; parts a and b together, or one part). So TMEM
// lane = component, column = row, and a row block of few rows costs few
// columns. Operand rows past the counts hold whatever was there: they only
// reach accumulators that nobody reads. The products a a have accumulators of
// their own; a b, b a, a c, c a, b b (and b c up to 64 components) go to others
// and are added once per chunk; the rest is below 2^-26 of a product.
// The tensor core's running fp32 sum drops bits as it grows (with one
// accumulator over all of a CTA's columns the dot products were off by five
// times as much), so it runs over kDtChunk units only, in two accumulators used
// in turn, and the converter warps add the finished chunk into registers,
// rounding to nearest, while the next is multiplied.
// (Two tf32 parts per value, 8 bytes of an operand stage in place of 6 and as
// much time of the tensor core, lost a bit of one value in four: error of the
// responsibilities against 64 bits, for rows of noise and small means, relative
// to the same with fp32 multiply-adds, 1.42 at 16 components and 1500 rows of
// 16384 columns, 1.15 at 64 components and 100 rows, 1.19 at 128 and 130 rows
// of 6000; 0.97, 0.93 and 1.01 so. A call at 118 rows of 4x128x128 and 64
// components takes 40.6 us, 41.4 with tf32 parts.)
//
// Warps: four loaders issue 16-byte asynchronous copies (cp.async) of a unit's
// rows and means into a ring of raw stages, already in core-matrix order;
// sixteen converters, in two groups that take units in turn, write a raw
// stage's parts into an operand stage; one thread issues the MMAs.
// A copy takes a microsecond and more, an operand stage's turn (split, MMAs)
// less: with raw values in rings of their own up to five units are on their
// way (four stages that held a unit from its copy to its MMAs: 20 us a call).
constexpr int kDtConvWarps = 16;
constexpr int kDtGroupWarps = kDtConvWarps / 2;
constexpr int kDtConv = kDtConvWarps * 32;
constexpr int kDtLoadWarps = 4;
constexpr int kDtLoad = kDtLoadWarps * 32;
constexpr int kDtThreads = kDtConv + kDtLoad + 32;
constexpr int kDtChunk = 2;                   // units per accumulator
constexpr int kDtFold = 8;                    // chunks per running sum (see the sums' part of the kernel)
constexpr uint32_t kDtTmem = 512;             // two accumulators of up to 256 columns

__host__ __device__ constexpr int dt_mu_rows(bool two) { return two ? 128 : 64; }
__host__ __device__ constexpr int dt_raw_floats(bool two) { return (kRows + dt_mu_rows(two)) * kUnit; }
__host__ __device__ constexpr int dt_raws(bool two) { return two ? 3 : 5; }
constexpr int kDtStages = 2;                  // operand stages: three parts of 2 bytes
constexpr int kDtPart = kUnit * 2;            // bytes of a row's part
// the rows' parts, the means' parts, up to 64 components 64 rows of zeros
__host__ __device__ constexpr int dt_stage_bytes(bool two) {
  return (3 * kRows + 3 * dt_mu_rows(two) + (two ? 0 : 64)) * kDtPart;
}
__host__ inline size_t dt_smem(bool two) {
  return (size_t)dt_raws(two) * dt_raw_floats(two) * sizeof(float) + (size_t)kDtStages * dt_stage_bytes(two);
}

__device__ __forceinline__ void copy1(uint32_t dst, const float* src, bool there) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(src), "r"(there ? 4 : 0) : "memory");
}
// Asynchronous copy of four columns of a row, zeros past its end (`left`
// columns remain): one 16-byte copy, or four of 4 bytes.
// (A copy of zeros reads nothing; `any` is an address that may be read.)
template <bool VEC>
__device__ __forceinline__ void copy4(uint32_t dst, const float* src, const float* any, int left) {
  if constexpr (VEC) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(left > 0 ? src : any),
                 "r"(left > 0 ? 16 : 0)
                 : "memory");
  } else {
#pragma unroll
    for (int k = 0; k < 4; ++k) copy1(dst + 4 * k, left > k ? src + k : any, left > k);
  }
}
// The mbarrier receives this thread's arrival when its copies so far have landed.
__device__ __forceinline__ void copies_arrive(uint64_t* bar) {
  asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void copies_drain() { asm volatile("cp.async.wait_all;" ::: "memory"); }

template <bool TWO, bool VEC>
__global__ void __launch_bounds__(kDtThreads, 1) k_gmm_dots_tc(const float* __restrict__ X, const float* __restrict__ mu,
                                                              const int32_t* __restrict__ n_rows_dev, int K, int64_t D,
                                                              int max_rows, float* __restrict__ part, int slots,
                                                              int32_t* status) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  constexpr int kMuRows = dt_mu_rows(TWO), kRaws = dt_raws(TWO), kRawFloats = dt_raw_floats(TWO);
  // the means in an operand stage and the distance of their parts, in bytes
  constexpr int kMu = 3 * kRows * kDtPart, kMuPart = kMuRows * kDtPart;
  __shared__ __align__(8) uint64_t raw[kRaws], rfree[kRaws], full[kDtStages], empty[kDtStages], done[2], afree[2];
  __shared__ uint32_t s_taddr;
  unsigned char* stage0 = smem_raw;
  float* raw0 = reinterpret_cast<float*>(stage0 + kDtStages * dt_stage_bytes(TWO));
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if constexpr (!TWO) {  // the rows below part c
    for (int q = tid; q < kDtStages * 64 * kDtPart / 16; q += kDtThreads) {
      const int s = q / (64 * kDtPart / 16);
      reinterpret_cast<uint4*>(stage0 + s * dt_stage_bytes(TWO) + kMu + 3 * kMuPart)[q % (64 * kDtPart / 16)] =
          make_uint4(0, 0, 0, 0);
    }
    fence_proxy_async_smem();
  }
  if (tid == 0) {
    for (int s = 0; s < kRaws; ++s) {
      mbar_init(&raw[s], kDtLoad);
      mbar_init(&rfree[s], kDtGroupWarps);
    }
    for (int s = 0; s < kDtStages; ++s) {
      mbar_init(&full[s], kDtGroupWarps);
      mbar_init(&empty[s], 1);
    }
    for (int d = 0; d < 2; ++d) {
      mbar_init(&done[d], 1);
      mbar_init(&afree[d], kDtConvWarps);
    }
    fence_barrier_init();
  }
  if (warp == 0) {
    tmem_alloc(&s_taddr, kDtTmem);
    tc_fence_before_sync();
  }
  __syncthreads();
  tc_fence_after_sync();
  const uint32_t taddr = s_taddr;
  const int KP = kpad(K), cta = blockIdx.x, units = (int)((D + kUnit - 1) / kUnit);
  // a loader thread's rows, columns and places in a stage: a warp step covers 8
  // rows x 16 columns, lanes 8q .. 8q + 7 fill one 128-byte core matrix, eight
  // 64-byte row pieces are read
  const int lw = warp - kDtConvWarps, c4 = (lw & 1) * 16 + (lane >> 3) * 4, rl = (lw >> 1) * 8 + (lane & 7);
  constexpr int kStep = kDtLoadWarps / 2 * 8;  // rows from one of a thread's rows to the next
  const uint32_t off = (uint32_t)(((rl >> 3) * (kUnit / 4) + (c4 >> 2)) * 32 + (rl & 7) * 4) * 4u;
  const bool loader = warp >= kDtConvWarps && warp < kDtConvWarps + kDtLoadWarps;
  auto copy_mu = [&](uint32_t s, int64_t c0) {
    const uint32_t dst = smem_u32(raw0 + s * kRawFloats + kRows * kUnit) + off;  // behind the rows
    const float* pm = mu + (int64_t)rl * D + c0 + c4;
    const int l = (int)min(D - c0 - c4, (int64_t)4);
#pragma unroll
    for (int q = 0; q < kMuRows / kStep; ++q)
      if (rl + q * kStep < K) copy4<VEC>(dst + q * kStep * kUnit * 4, pm + (int64_t)(q * kStep) * D, mu, l);
  };
  // with one row block the first units are known, and the means do not change:
  // their copies go out before the dependency wait
  const bool early = max_rows <= kRows;
  if (early && loader)
    for (int w = 0; w < kRaws; ++w)
      if (cta + w * (int)gridDim.x < units) copy_mu((uint32_t)w, (int64_t)(cta + w * (int)gridDim.x) * kUnit);
  pdl_wait();     // the rows and their count come from the kernel just before
  pdl_trigger();  // the successor may now run its prologue
  const int n_rows = min(*n_rows_dev, max_rows);
  const Share sh((n_rows + kRows - 1) / kRows, units, gridDim.x);
  bool bad = false;
  uint32_t v = 0;   // units so far: the stage and its phase
  uint32_t ck = 0;  // chunks so far: the accumulator and its phase
  for (int blk = n_rows > 0 ? sh.block(cta) : 0; blk < sh.blocks; blk += sh.block_step()) {
    const int u0 = sh.unit(cta, blk), ustep = sh.unit_step(blk);
    const int n = u0 < sh.units ? (sh.units - u0 + ustep - 1) / ustep : 0;  // this CTA's units of the block
    if (n == 0) continue;
    const int nc = (n + kDtChunk - 1) / kDtChunk;
    const int r0 = blk * kRows, nr = min(kRows, n_rows - r0);
    const int Nb = (nr + 15) & ~15;
    if (warp < kDtConvWarps) {
      const int group = warp / kDtGroupWarps, gt = tid & (kDtGroupWarps * 32 - 1);
      // this warp's share of the sums: lanes 32 q .. + 31 (q = warp & 3), rows rb .. rb + 31
      const int q4 = warp & 3, rb = (warp >> 2) * 32;
      const uint32_t tl = taddr + ((uint32_t)(32 * q4) << 16) + (uint32_t)rb;
      float acc[32];
#pragma unroll
      for (int i = 0; i < 32; ++i) acc[i] = 0.f;
      // a chunk's two sums first, so that the running sum is rounded once
      auto add = [&](uint32_t col) {
#pragma unroll
        for (int h = 0; h < 32; h += 8) {
          if (rb + h < Nb) {
            float t[8], u[8];
            tmem_ld8x2(tl + col + h, tl + col + (uint32_t)Nb + h, t, u);
#pragma unroll
            for (int i = 0; i < 8; ++i) acc[h + i] += t[i] + u[i];
          }
        }
      };
      // TMEM lane = component; up to 64 components lane 64 + k holds the products
      // with the means' part b
      // A CTA's share of a block can be hundreds of units long (K 16, D 65536, 600
      // rows: 68), and one fp32 sum over all of its chunks is then off by more than
      // fp32 multiply-adds are: every kDtFold chunks the running sum goes to memory
      // and starts again.
      auto fold = [&](bool more) {
        const int k = 32 * q4 + lane, rows = k < KP ? nr - rb : 0;
        float* o = part + ((int64_t)rb * slots + sh.slot(blk, u0)) * KP + k;
#pragma unroll
        for (int i = 0; i < 32; ++i, o += (int64_t)slots * KP) {
          if (i < rows) {
            if (more)
              atomicAdd(o, acc[i]);  // this thread's alone: an addition that nothing waits for
            else
              *o = acc[i];
          }
          acc[i] = 0.f;
        }
      };
      int taken = 0;  // chunks of this block added so far
      auto take_until = [&](int c1) {
        for (; taken < c1; ++taken) {  // the chunk is complete: add it, hand its accumulator back
          const uint32_t c = ck + (uint32_t)taken;
          wait_or_fail(&done[c & 1u], (c >> 1) & 1u, &bad, status);
          __syncwarp();
          tc_fence_after_sync();
          add((c & 1u) * 256u);
          tc_fence_before_sync();
          __syncwarp();
          if (lane == 0) mbar_arrive(&afree[c & 1u]);
          if ((TWO || q4 < 2) && taken % kDtFold == kDtFold - 1 && taken + 1 < nc) fold(taken >= kDtFold);
        }
      };
      for (int w = group; w < n; w += 2) {
        const uint32_t u = v + w, rs = u % kRaws, s = u % kDtStages;
        // the values in storage order: consecutive threads, consecutive 16 bytes
        constexpr int kGroup = kDtGroupWarps * 32, kX = kRows * kUnit / 4 / kGroup, kM = kMuRows * kUnit / 4 / kGroup;
        const int rr = (gt >> 6) * 8 + (gt & 7);  // this thread's first row; the next is kGroup / 8 rows on
        // its place in a part: 8 columns of 8 rows to a core matrix, 4 to a thread
        const int at = (gt >> 6) * (8 * kDtPart) + ((gt >> 4) & 3) * 128 + (gt & 7) * 16 + ((gt >> 3) & 1) * 8;
        constexpr int kNext = kGroup / 8 * kDtPart;
        auto put = [&](unsigned char* to, float4 f, int part) {
#pragma unroll
          for (int p = 0; p < 3; ++p, to += part) {
            const uint32_t lo = split2(f.x, f.y), hi = split2(f.z, f.w);
            *reinterpret_cast<uint2*>(to) = make_uint2(lo, hi);
          }
        };
        float4 val[kX + kM];
        wait_or_fail(&raw[rs], (u / kRaws) & 1u, &bad, status);
        const float4* from = reinterpret_cast<const float4*>(raw0 + rs * kRawFloats) + gt;
#pragma unroll
        for (int i = 0; i < kX + kM; ++i) val[i] = from[i * kGroup];
        __syncwarp();
        if (lane == 0) mbar_arrive(&rfree[rs]);
        if (u >= kDtStages) wait_or_fail(&empty[s], (u / kDtStages - 1) & 1u, &bad, status);
        unsigned char* xs = stage0 + s * dt_stage_bytes(TWO) + at;
        unsigned char* ms = xs + kMu;
#pragma unroll
        for (int i = 0; i < kX; ++i)
          if (rr + i * (kGroup / 8) < nr) put(xs + i * kNext, val[i], Nb * kDtPart);
#pragma unroll
        for (int i = 0; i < kM; ++i)
          if (rr + i * (kGroup / 8) < K) put(ms + i * kNext, val[kX + i], kMuPart);
        fence_proxy_async_smem();  // the tensor core reads what the threads wrote
        __syncwarp();
        if (lane == 0) mbar_arrive(&full[s]);
        // chunks whose units come before this one: their MMAs wait for no later unit
        take_until(w / kDtChunk);
      }
      take_until(nc);
      // [kRows][64]: every MMA that reads the stages is complete (and the zeros lie behind)
      float* sc = reinterpret_cast<float*>(stage0);
      static_assert(TWO || kRows * 64 * (int)sizeof(float) <= kMu + 3 * kMuPart, "the zeros stay");
      if constexpr (!TWO) {
        if (q4 >= 2) {
#pragma unroll
          for (int i = 0; i < 32; ++i) sc[(rb + i) * 64 + (q4 - 2) * 32 + lane] = acc[i];
        }
        named_sync(1, kDtConv);
      }
      if (TWO || q4 < 2) {
        if constexpr (!TWO) {
#pragma unroll
          for (int i = 0; i < 32; ++i) acc[i] += sc[(rb + i) * 64 + 32 * q4 + lane];
        }
        fold(nc > kDtFold);
      }
      tc_fence_before_sync();
    } else if (loader) {
      const int64_t cstep = (int64_t)ustep * kUnit;
      const float* px = X + (int64_t)(r0 + rl) * D + (int64_t)u0 * kUnit + c4;
      for (int w = 0; w < n; ++w, px += cstep) {
        const uint32_t s = (v + w) % kRaws, use = (v + w) / kRaws;
        if (use > 0) wait_or_fail(&rfree[s], (use - 1) & 1u, &bad, status);
        const uint32_t dst = smem_u32(raw0 + s * kRawFloats) + off;
        const int64_t c0 = (int64_t)u0 * kUnit + w * cstep;
        const int l = (int)min(D - c0 - c4, (int64_t)4);
#pragma unroll
        for (int q = 0; q < kRows / kStep; ++q)
          if (rl + q * kStep < nr) copy4<VEC>(dst + q * kStep * kUnit * 4, px + (int64_t)(q * kStep) * D, mu, l);
        if (!early || use > 0) copy_mu(s, c0);
        copies_arrive(&raw[s]);
      }
    } else if (lane == 0) {
      const uint32_t idesc = tc_idesc_bf16(128, 2 * Nb), idesc1 = tc_idesc_bf16(128, Nb);
      constexpr uint32_t sbo = (kUnit / 8) * 128;  // next 8-row group
      uint32_t c = ck;
      for (int w = 0; w < n; ++w) {
        const uint32_t s = (v + w) % kDtStages;
        const bool first = w % kDtChunk == 0;
        if (first && c >= 2) wait_or_fail(&afree[c & 1u], ((c >> 1) - 1) & 1u, &bad, status);
        wait_or_fail(&full[s], ((v + w) / kDtStages) & 1u, &bad, status);
        tc_fence_after_sync();
        const uint32_t xs = smem_u32(stage0 + s * dt_stage_bytes(TWO)), ms = xs + kMu;
        const uint32_t sum = taddr + (c & 1u) * 256u, small = sum + (uint32_t)Nb;
#pragma unroll
        for (int ks = 0; ks < kUnit / 16; ++ks) {
          const uint32_t ko = (uint32_t)ks * 256;  // two core matrices along the columns per step
          uint64_t m[3], x[3];
#pragma unroll
          for (int i = 0; i < 3; ++i) {
            m[i] = tc_smem_desc(ms + i * kMuPart + ko, 128, sbo);
            x[i] = tc_smem_desc(xs + (uint32_t)(i * Nb * kDtPart) + ko, 128, sbo);
          }
          tc_mma_f16(sum, m[0], x[0], idesc, !first || ks > 0 ? 1u : 0u);  // the rows' parts a and b
          tc_mma_f16(small, m[0], x[2], idesc1, 1u);
          if constexpr (TWO) {
            tc_mma_f16(small, m[1], x[1], idesc1, 1u);
            tc_mma_f16(small, m[1], x[0], idesc1, 1u);
          }
          tc_mma_f16(small, m[2], x[0], idesc1, 1u);
        }
        tc_commit(&empty[s]);
        if (w % kDtChunk == kDtChunk - 1 || w == n - 1) {
          tc_commit(&done[c & 1u]);
          ++c;
        }
      }
    }
    v += (uint32_t)n;
    ck += (uint32_t)nc;
    __syncthreads();  // the accumulators are read and the stages free for the next block
    tc_fence_after_sync();
  }
  if (warp >= kDtConvWarps) copies_drain();
  __syncthreads();
  __syncwarp();
  if (warp == 0) tmem_dealloc(taddr, kDtTmem);
}

// ---------------------------------------------------------------------------
// Responsibilities, a CTA per row: the CTAs' partial dot products of the row's
// block summed in CTA order (each thread a fixed share, as an error-free pair,
// so that the number of CTAs costs no precision), logits, softmax, and the
// row's two scalars for the output.
constexpr int kRespThreads = 512;
constexpr int kBatch = 20;       // partial sums in flight per thread: 152 of them at 64 components in one trip
constexpr int kRespGrid = 4096;  // rows beyond it are taken in turn

template <int KP>
__global__ void __launch_bounds__(kRespThreads) k_gmm_resp(const float* __restrict__ part, int slots, int dots_grid,
                                                           const float* __restrict__ coef, int T,
                                                           const int32_t* __restrict__ miss_bt,
                                                           const float* __restrict__ mnorm,
                                                           const int32_t* __restrict__ n_rows_dev, int K, int64_t D,
                                                           int max_rows, float* __restrict__ resp,
                                                           float* __restrict__ rcoef) {
  constexpr int kGroups = kRespThreads / KP, kPer = (KP + 31) / 32;
  __shared__ float2 s_sum[kGroups][KP];
  const int tid = threadIdx.x, lane = tid & 31;
  const int n_rows = min(*n_rows_dev, max_rows);  // written two kernels back, as the rows' timesteps
  const int k = tid % KP, grp = tid / KP;
  float mn[kPer] = {};
  if (tid < 32)
#pragma unroll
    for (int u = 0; u < kPer; ++u)
      if (lane + 32 * u < K) mn[u] = mnorm[lane + 32 * u];
  bool waited = false;
  for (int r = blockIdx.x; r < n_rows; r += gridDim.x) {
    const int i = miss_bt[2 * r + 1];
    const float sa = coef[i], q = coef[T + i], c = coef[2 * T + i];
    const Share sh((n_rows + kRows - 1) / kRows, (int)((D + kUnit - 1) / kUnit), dots_grid);
    const int blk = r / kRows, members = sh.members(blk);
    if (!waited) {
      pdl_wait();     // the dot products come from the kernel just before
      pdl_trigger();  // the successor may now run its prologue
      waited = true;
    }
    const float* p = part + ((int64_t)(r - blk * kRows) * slots + sh.slot(blk, 0)) * KP + k;
    float hi = 0.f, lo = 0.f;
    for (int s = grp; s < members; s += kBatch * kGroups) {
      float v[kBatch];  // kBatch loads in flight
#pragma unroll
      for (int u = 0; u < kBatch; ++u) {
        v[u] = 0.f;
        if (s + u * kGroups < members) v[u] = __ldcg(p + (int64_t)(s + u * kGroups) * KP);
      }
#pragma unroll
      for (int u = 0; u < kBatch; ++u) {  // TwoSum
        const float t = __fadd_rn(hi, v[u]), bb = __fsub_rn(t, hi);
        lo = __fadd_rn(lo, __fadd_rn(__fsub_rn(hi, __fsub_rn(t, bb)), __fsub_rn(v[u], bb)));
        hi = t;
      }
    }
    s_sum[grp][k] = make_float2(hi, lo);
    __syncthreads();
    if (tid < 32) {
      float l[kPer], mx = -INFINITY;
#pragma unroll
      for (int u = 0; u < kPer; ++u) {
        const int kk = lane + 32 * u;
        l[u] = -INFINITY;
        if (kk < K) {
          float h = 0.f, e = 0.f;
#pragma unroll
          for (int g = 0; g < kGroups; ++g) {
            const float2 v = s_sum[g][kk];
            const float t = __fadd_rn(h, v.x), bb = __fsub_rn(t, h);
            e = __fadd_rn(e, __fadd_rn(__fadd_rn(__fsub_rn(h, __fsub_rn(t, bb)), __fsub_rn(v.x, bb)), v.y));
            h = t;
          }
          const float dot = h + e;
          l[u] = (2.f * sa * dot - sa * sa * mn[u]) * q;
        }
        mx = fmaxf(mx, l[u]);
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
      float sum = 0.f;
#pragma unroll
      for (int u = 0; u < kPer; ++u) {
        l[u] = lane + 32 * u < K ? expf(l[u] - mx) : 0.f;
        sum += l[u];
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
      const float inv = 1.f / sum;
#pragma unroll
      for (int u = 0; u < kPer; ++u)
        if (lane + 32 * u < KP) resp[(int64_t)r * KP + lane + 32 * u] = l[u] * inv;  // zero for k >= K
      if (lane == 0) {
        rcoef[2 * r] = c;
        rcoef[2 * r + 1] = c * sa;
      }
    }
    __syncthreads();
  }
  if (!waited) pdl_wait();  // every CTA passes the dependency wait before it exits
}

// ---------------------------------------------------------------------------
// Output. A tile is 128 columns of D x the rows of a row block. The MMA's A
// operand is the means' transpose (M = 128 columns, K-major over the
// components), its B operand the responsibilities (N = the block's rows,
// rounded up to 16), so TMEM lane = column: a warp's loads of x and stores of
// eps are 128 adjacent bytes of one row, whatever D and the alignment. Four
// warps (a thread per column) copy the means of a stage of up to 32 components
// asynchronously, row by row, one stage ahead, and split and transpose the
// stage that has landed; a thread of a warp of its own issues the MMAs; sixteen
// output warps keep 32 rows of x per thread in flight and finish the tile from
// TMEM. Two operand stages and two accumulators: tile t + 1 is multiplied while
// tile t is written.
// Both operands are held exactly, as three bfloat16 parts, and an accumulator
// is two: the products of the first parts, and the five next larger products
// (the three left out are below 2^-26 of the value); the output adds the two
// with one rounding. Where one component carries all of the weight, as in most
// rows, the contraction is then exact, as it is with fp32 multiply-adds. (Two
// tf32 parts and one accumulator, as many MMAs and 8 bytes of shared memory per
// value in place of 6: rms error of eps against 64 bits 6.07e-8 at 92
// components, 360 rows of 2688 columns, 5.11e-8 so, 5.12e-8 with fp32
// multiply-adds; a call at 118 rows of 4x128x128 and 64 components 48.4 us, 43.4
// so.)
constexpr int kOtTile = 128;
constexpr int kOtOutWarps = 16;
constexpr int kOtOut = kOtOutWarps * 32;
constexpr int kOtConv = kOtTile;
constexpr int kOtThreads = kOtOut + kOtConv + 32;
constexpr uint32_t kOtSmall = 2 * kRows;  // TMEM columns of the small products' accumulators
constexpr uint32_t kOtTmem = 4 * kRows;

template <int KP>
struct OtShape {
  static constexpr int KH = KP < 32 ? KP : 32;     // components per stage
  static constexpr int NH = KP / KH;               // stages per tile
  static constexpr int kRespPart = kRows * KP * 2;        // bytes of a part of the responsibilities
  static constexpr int kMeanPart = kOtTile * KH * 2;      // ... of a stage's means
  static constexpr int kRawFloats = kOtTile * KH;         // [component][column], as they lie in memory
  static constexpr int NST = 2;                    // operand stages
  static constexpr int NRAW = KP > 64 ? 3 : 4;     // raw stages: all but one are in flight
  static constexpr size_t smem() {
    return (size_t)3 * kRespPart + (size_t)NST * 3 * kMeanPart + (size_t)NRAW * kRawFloats * sizeof(float);
  }
};

template <int KP>
__global__ void __launch_bounds__(kOtThreads, 1) k_gmm_out_tc(const float* __restrict__ X, const float* __restrict__ mu,
                                                             const float* __restrict__ resp,
                                                             const float* __restrict__ rcoef,
                                                             const int32_t* __restrict__ n_rows_dev, int K, int64_t D,
                                                             int max_rows, float* __restrict__ eps, int32_t* status) {
  using Sh = OtShape<KP>;
  constexpr int KH = Sh::KH, NH = Sh::NH, NST = Sh::NST, NRAW = Sh::NRAW;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  __shared__ __align__(8) uint64_t full[NST], empty[NST], dfull[2], dfree[2];
  __shared__ uint32_t s_taddr;
  __shared__ __align__(16) float2 s_c[kRows];
  unsigned char* R = smem_raw;
  unsigned char* stage0 = R + 3 * Sh::kRespPart;
  float* raw0 = reinterpret_cast<float*>(stage0 + NST * 3 * Sh::kMeanPart);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (tid == 0) {
    for (int s = 0; s < NST; ++s) {
      mbar_init(&full[s], kOtConv / 32);
      mbar_init(&empty[s], 1);
    }
    for (int s = 0; s < 2; ++s) {
      mbar_init(&dfull[s], 1);
      mbar_init(&dfree[s], kOtOutWarps);
    }
    fence_barrier_init();
  }
  if (warp == 0) {
    tmem_alloc(&s_taddr, kOtTmem);
    tc_fence_before_sync();
  }
  __syncthreads();
  tc_fence_after_sync();
  const uint32_t taddr = s_taddr;
  const int n_rows = min(*n_rows_dev, max_rows);  // written three kernels back, as the rows
  const int tpb = (int)((D + kOtTile - 1) / kOtTile);  // tiles per row block
  const Share sh((n_rows + kRows - 1) / kRows, tpb, gridDim.x);
  const int cta = blockIdx.x;
  const bool out_warp = warp < kOtOutWarps, conv_warp = !out_warp && warp < kOtOutWarps + kOtConv / 32;
  // converters: the raw copies of stage h of tile t, zeros for components and
  // columns that are not there; each thread copies and later reads its own
  // column (16-byte copies shared by the threads measured 25 against 20 us)
  const int lt = tid - kOtOut;
  auto copy_means = [&](int t, int h, uint32_t slot) {
    const int64_t col = (int64_t)t * kOtTile + lt;
    const uint32_t dst = smem_u32(raw0 + slot * Sh::kRawFloats + lt);
    const float* p = mu + (int64_t)h * KH * D + col;
    const int lim = col < D ? K - h * KH : 0;
#pragma unroll 8
    for (int k = 0; k < KH; ++k, p += D) copy1(dst + k * kOtTile * 4, k < lim ? p : mu, k < lim);
  };
  auto group_end = [] { asm volatile("cp.async.commit_group;" ::: "memory"); };
  // output warps: lane = column of quarter q, rows [32 (warp / 4), + 32) of the block
  const int q = warp & 3, row0 = (warp >> 2) * 32;
  float buf[32];  // a thread's column of x, one tile ahead
  auto fetch_rows = [&](int j, int blk, int t) {
    const int64_t col = (int64_t)t * kOtTile + 32 * q + lane;
    const int r0 = blk * kRows + row0 + 16 * j;
    const int lim = col < D ? min(kRows - row0 - 16 * j, n_rows - r0) : 0;
    const float* p = X + (int64_t)r0 * D + col;
#pragma unroll
    for (int i = 0; i < 16; ++i, p += D)
      if (i < lim) buf[16 * j + i] = __ldg(p);
  };
  // the means do not change and the rows were written three kernels back: the
  // first block's loads go out before the dependency wait
  auto begin_block = [&](int blk) {
    const int t = sh.unit(cta, blk), step = sh.unit_step(blk);
    if (t >= tpb) return;
    if (conv_warp) {
#pragma unroll
      for (int w = 0; w < NRAW - 1; ++w) {
        if (t + w / NH * step < tpb) copy_means(t + w / NH * step, w % NH, (uint32_t)w);
        group_end();
      }
    } else if (out_warp) {
      fetch_rows(0, blk, t);
      fetch_rows(1, blk, t);
    }
  };
  const int blk0 = n_rows > 0 ? sh.block(cta) : sh.blocks;
  if (blk0 < sh.blocks) begin_block(blk0);
  pdl_wait();     // the responsibilities and the row scalars come from the kernel just before
  pdl_trigger();  // the successor may now run its prologue
  bool bad = __ldcg(status) != 0;  // a dot-product wait ran out: the sums are incomplete
  uint32_t su = 0;   // operand stages used so far
  uint32_t tu = 0;   // tiles so far
  for (int blk = blk0; blk < sh.blocks; blk += sh.block_step()) {
    const int t0 = sh.unit(cta, blk), ustep = sh.unit_step(blk);
    const int n = t0 < tpb ? (tpb - t0 + ustep - 1) / ustep : 0;  // this CTA's tiles of the row block
    if (n == 0) continue;
    if (blk != blk0) begin_block(blk);
    const int r0 = blk * kRows, nr = min(kRows, n_rows - r0);
    const int nb = (nr + 15) & ~15;
    // the block's responsibilities, split, in core-matrix order (a warp step: 8
    // rows x 16 components, a lane 4 of them: 8 bytes of a core matrix's row)
    constexpr int kWarps = kOtThreads / 32, kSteps = kRows / 8 * (KP / 16), kBatch = kSteps < 4 * kWarps ? (kSteps + kWarps - 1) / kWarps : 4;
    for (int it0 = warp; it0 < (nb >> 3) * (KP / 16); it0 += kBatch * kWarps) {
      float4 v[kBatch];
#pragma unroll
      for (int i = 0; i < kBatch; ++i) {
        const int it = it0 + i * kWarps, r = (it / (KP / 16)) * 8 + (lane & 7), kq = (it % (KP / 16)) * 4 + (lane >> 3);
        v[i] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (r < nr) v[i] = __ldcg(reinterpret_cast<const float4*>(resp + (int64_t)(r0 + r) * KP + kq * 4));
      }
#pragma unroll
      for (int i = 0; i < kBatch; ++i) {
        const int it = it0 + i * kWarps, r = (it / (KP / 16)) * 8 + (lane & 7), kq = (it % (KP / 16)) * 4 + (lane >> 3);
        if (r >= nb) break;
        unsigned char* o = R + ((r >> 3) * (KP / 8) + (kq >> 1)) * 128 + (r & 7) * 16 + (kq & 1) * 8;
#pragma unroll
        for (int part = 0; part < 3; ++part) {
          const uint32_t p0 = split2(v[i].x, v[i].y), p1 = split2(v[i].z, v[i].w);
          *reinterpret_cast<uint2*>(o + part * Sh::kRespPart) = make_uint2(p0, p1);
        }
      }
    }
    for (int r = tid; r < nr; r += kOtThreads) s_c[r] = make_float2(rcoef[2 * (r0 + r)], rcoef[2 * (r0 + r) + 1]);
    fence_proxy_async_smem();
    __syncthreads();
    if (conv_warp) {
      for (int w = 0; w < n * NH; ++w) {
        const uint32_t u = su + (uint32_t)w, s = u % NST, use = u / NST;
        asm volatile("cp.async.wait_group %0;" ::"n"(NRAW - 2) : "memory");  // this stage's copies have landed
        const int nx = w + NRAW - 1;  // the raw stage read last is free for the copies of this one
        if (nx < n * NH) copy_means(t0 + nx / NH * ustep, nx % NH, (uint32_t)nx % NRAW);
        group_end();
        if (use > 0) wait_or_fail(&empty[s], (use - 1) & 1u, &bad, status);
        const float* rw = raw0 + (uint32_t)w % NRAW * Sh::kRawFloats + lt;
        unsigned char* as = stage0 + s * 3 * Sh::kMeanPart + (lt >> 3) * (KH / 8) * 128 + (lt & 7) * 16;
#pragma unroll
        for (int k8 = 0; k8 < KH / 8; ++k8) {
          const float* c = rw + 8 * k8 * kOtTile;
          const Parts h = split8(make_float4(c[0], c[kOtTile], c[2 * kOtTile], c[3 * kOtTile]),
                                 make_float4(c[4 * kOtTile], c[5 * kOtTile], c[6 * kOtTile], c[7 * kOtTile]));
          *reinterpret_cast<uint4*>(as + k8 * 128) = h.a;
          *reinterpret_cast<uint4*>(as + k8 * 128 + Sh::kMeanPart) = h.b;
          *reinterpret_cast<uint4*>(as + k8 * 128 + 2 * Sh::kMeanPart) = h.c;
        }
        fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) mbar_arrive(&full[s]);
      }
    } else if (out_warp) {
      for (int w = 0; w < n; ++w) {
        const uint32_t tile = tu + (uint32_t)w, d = tile & 1u;
        const int64_t col = (int64_t)(t0 + w * ustep) * kOtTile + 32 * q + lane;
        wait_or_fail(&dfull[d], (tile >> 1) & 1u, &bad, status);
        tc_fence_after_sync();
        bad = __any_sync(0xffffffffu, bad);
        const uint32_t tl = taddr + d * kRows + ((uint32_t)(32 * q) << 16);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const int rb = row0 + 8 * j;
          float acc[8], small[8];
          if (rb < nb) {
            tmem_ld8(tl + (uint32_t)rb, acc);
            tmem_ld8(tl + kOtSmall + (uint32_t)rb, small);
#pragma unroll
            for (int i = 0; i < 8; ++i) acc[i] += small[i];
          }
          if (j == 3) {  // the accumulator is read: the tile after the next may overwrite it
            tc_fence_before_sync();
            __syncwarp();
            if (lane == 0) mbar_arrive(&dfree[d]);
          }
          const int lim = col < D ? nr - rb : 0;
          float* er = eps + (int64_t)(r0 + rb) * D + col;
          if (lim >= 8 && !bad) {
#pragma unroll
            for (int i = 0; i < 8; i += 2, er += 2 * D) {
              const float4 c = *reinterpret_cast<const float4*>(&s_c[rb + i]);  // two rows' scalars
              er[0] = c.x * buf[8 * j + i] - c.y * acc[i];
              er[D] = c.z * buf[8 * j + i + 1] - c.w * acc[i + 1];
            }
          } else {
#pragma unroll
            for (int i = 0; i < 8; ++i, er += D)
              if (i < lim) *er = bad ? __int_as_float(0x7fc00000) : s_c[rb + i].x * buf[8 * j + i] - s_c[rb + i].y * acc[i];
          }
          if (w + 1 < n && (j & 1)) fetch_rows(j >> 1, blk, t0 + (w + 1) * ustep);
        }
      }
    } else {
      if (lane == 0) {
        const uint32_t idesc = tc_idesc_bf16(128, nb);
        constexpr uint32_t asbo = (KH / 8) * 128, bsbo = (KP / 8) * 128;  // next 8-row group
        for (int w = 0; w < n * NH; ++w) {
          const uint32_t u = su + (uint32_t)w, s = u % NST, tile = tu + (uint32_t)(w / NH), d = tile & 1u;
          if (w % NH == 0 && tile >= 2) wait_or_fail(&dfree[d], ((tile >> 1) - 1) & 1u, &bad, status);
          wait_or_fail(&full[s], (u / NST) & 1u, &bad, status);
          tc_fence_after_sync();
          const uint32_t a = smem_u32(stage0 + s * 3 * Sh::kMeanPart), b = smem_u32(R) + (uint32_t)(w % NH) * (KH / 8) * 128;
          const uint32_t acc = taddr + d * kRows, small = acc + kOtSmall;
#pragma unroll
          for (int ks = 0; ks < KH / 16; ++ks) {
            uint64_t ad[3], bd[3];
#pragma unroll
            for (int i = 0; i < 3; ++i) {
              ad[i] = tc_smem_desc(a + i * Sh::kMeanPart + (uint32_t)ks * 256, 128, asbo);
              bd[i] = tc_smem_desc(b + i * Sh::kRespPart + (uint32_t)ks * 256, 128, bsbo);
            }
            const uint32_t more = w % NH > 0 || ks > 0 ? 1u : 0u;
            tc_mma_f16(acc, ad[0], bd[0], idesc, more);
            tc_mma_f16(small, ad[2], bd[0], idesc, more);  // the smallest first
            tc_mma_f16(small, ad[1], bd[1], idesc, 1u);
            tc_mma_f16(small, ad[0], bd[2], idesc, 1u);
            tc_mma_f16(small, ad[1], bd[0], idesc, 1u);
            tc_mma_f16(small, ad[0], bd[1], idesc, 1u);
          }
          tc_commit(&empty[s]);
          if (w % NH == NH - 1) tc_commit(&dfull[d]);
        }
      }
    }
    tu += (uint32_t)n;
    su += (uint32_t)(n * NH);
    __syncthreads();  // every MMA that reads this block's responsibilities is complete (its tile was written)
  }
  copies_drain();
  tc_fence_after_sync();
  __syncthreads();
  __syncwarp();
  if (warp == 0) tmem_dealloc(taddr, kOtTmem);
}

template <int KP>
cudaError_t out_setup() {
  return allow_smem(reinterpret_cast<const void*>(k_gmm_out_tc<KP>), OtShape<KP>::smem());
}

// CTAs of the two large kernels: one per SM
cudaError_t sm_count(int* out) {
  static int nsm[64] = {};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  int n = dev >= 0 && dev < 64 ? nsm[dev] : 0;
  if (n == 0) {
    e = cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    if (dev >= 0 && dev < 64) nsm[dev] = n;
  }
  *out = n < kMaxCtas ? n : kMaxCtas;
  return cudaSuccess;
}

template <int KP>
cudaError_t launch_tail(const GmmTcArgs& a, const GmmTcLayout& L, int dots_grid, int grid, cudaStream_t st) {
  const float* part = reinterpret_cast<const float*>(a.ws + L.part);
  float* resp = reinterpret_cast<float*>(a.ws + L.resp);
  float* rcoef = reinterpret_cast<float*>(a.ws + L.rcoef);
  cudaError_t e = launch_ex(k_gmm_resp<KP>, dim3(a.max_rows < kRespGrid ? a.max_rows : kRespGrid), dim3(kRespThreads), 0,
                            st, 0, part, L.slots, dots_grid, a.coef, a.T, a.miss_bt, a.mnorm, a.n_rows, a.K, a.D, a.max_rows, resp,
                            rcoef);
  if (e != cudaSuccess) return e;
  return launch_ex(k_gmm_out_tc<KP>, dim3(grid), dim3(kOtThreads), OtShape<KP>::smem(), st, 0, a.X, a.mu,
                   (const float*)resp, (const float*)rcoef, a.n_rows, a.K, a.D, a.max_rows, a.eps, a.status);
}

}  // namespace

GmmTcLayout gmm_tc_layout(int K, int64_t D, int max_rows) {
  GmmTcLayout L{};
  size_t o = 0;
  auto take = [&](size_t bytes) { size_t at = o; o = align_up(o + bytes, kAlign); return at; };
  const size_t blocks = ((size_t)max_rows + kRows - 1) / kRows;
  const size_t ctas = (size_t)dots_ctas(D, max_rows, kMaxCtas);
  L.slots = (int)(ctas > blocks ? ctas : blocks);
  // [row of a block][CTA, or block where there are more][component]
  L.part = take((size_t)(max_rows < kRows ? max_rows : kRows) * L.slots * kpad(K) * sizeof(float));
  L.resp = take((size_t)max_rows * kpad(K) * sizeof(float));
  L.rcoef = take((size_t)2 * max_rows * sizeof(float));
  L.total = o;
  return L;
}

cudaError_t gmm_tc_setup(int K, bool* ok) {
  *ok = false;
  int dev = 0, major = 0, optin = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (e != cudaSuccess) return e;
  const bool two = K > 64;
  if (major != 10 || OtShape<128>::smem() + 4096 > (size_t)optin || dt_smem(two) + 1024 > (size_t)optin) return e;
  auto dots = two ? k_gmm_dots_tc<true, true> : k_gmm_dots_tc<false, true>;
  auto dots1 = two ? k_gmm_dots_tc<true, false> : k_gmm_dots_tc<false, false>;
  e = allow_smem(reinterpret_cast<const void*>(dots), dt_smem(two));
  if (e == cudaSuccess) e = allow_smem(reinterpret_cast<const void*>(dots1), dt_smem(two));
  if (e == cudaSuccess) {
    const int KP = kpad(K);
    e = KP == 16 ? out_setup<16>() : KP == 32 ? out_setup<32>() : KP == 64 ? out_setup<64>() : out_setup<128>();
  }
  *ok = e == cudaSuccess;
  return e;
}

cudaError_t gmm_tc_launch(const GmmTcArgs& a, cudaStream_t st) {
  int grid = 0;
  cudaError_t e = sm_count(&grid);
  if (e != cudaSuccess) return e;
  const int dots_grid = dots_ctas(a.D, a.max_rows, grid);
  const GmmTcLayout L = gmm_tc_layout(a.K, a.D, a.max_rows);
  // 16-byte loads of the rows and the means where all of them are aligned
  const bool vec = a.D % 4 == 0 && ((reinterpret_cast<uintptr_t>(a.X) | reinterpret_cast<uintptr_t>(a.mu)) & 15) == 0;
  const bool two = a.K > 64;
  auto dots = two ? (vec ? k_gmm_dots_tc<true, true> : k_gmm_dots_tc<true, false>)
                  : (vec ? k_gmm_dots_tc<false, true> : k_gmm_dots_tc<false, false>);
  e = launch_ex(dots, dim3(dots_grid), dim3(kDtThreads), dt_smem(two), st, 0, a.X, a.mu, a.n_rows, a.K, a.D, a.max_rows,
                reinterpret_cast<float*>(a.ws + L.part), L.slots, a.status);
  if (e != cudaSuccess) return e;
  switch (kpad(a.K)) {
    case 16: return launch_tail<16>(a, L, dots_grid, grid, st);
    case 32: return launch_tail<32>(a, L, dots_grid, grid, st);
    case 64: return launch_tail<64>(a, L, dots_grid, grid, st);
    default: return launch_tail<128>(a, L, dots_grid, grid, st);
  }
}

}  // namespace pa
