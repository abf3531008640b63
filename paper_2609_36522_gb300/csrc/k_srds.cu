// Parareal (SRDS-style) DDIM sampling with ParaAnya's output cache on every
// network evaluation (Sec. 2.1: Parareal-based samplers; Sec. 2.2: the cache
// applies to the coarse and fine evaluations, the Parareal update unchanged).
//
// Blocks of s = ceil(sqrt(T)) sampling steps, N = ceil(T / s) blocks; block n
// covers indices [n s, e_n), e_n = min((n + 1) s, T). Fine solver F_n: the
// DDIM steps of block n. Coarse solver G_n: one DDIM jump from alpha-bar(n s)
// to alpha-bar(e_n) with eps at (u, n s).
//   iteration 0   U_0 = x_init, U_{n+1} = G_n(U_n)                 (coarse stages)
//   iteration k   F_n(U_n^{k-1}) for all n                         (s fine stages)
//                 U_{n+1}^k = G_n(U_n^k) + F_n(U_n^{k-1}) - G_n(U_n^{k-1})  (N coarse stages)
//                 err = max_n (1/D) ||U_n^k - U_n^{k-1}||^2 <= tol => converged (Eq. 2 on the
//                 block boundaries); a converged trajectory is frozen; Parareal is exact at k = N.
// Every evaluation stage: cache distance of each live row against its index's
// entry (Eq. 4), hit iff entry && delta < tau_cache (Eq. 5), misses compacted
// trajectory-major and gathered for the denoiser (k_srds_plan_gather); then
// the step (k_srds_apply) takes eps from the batch (miss, updating the entry,
// Eq. 7) or from the cache (hit, Eq. 6). The distances of a stage's rows are
// summed by the previous stage's k_srds_apply, which produced those rows, into
// fp64 accumulators, one set per stage parity, while the new values are in
// registers. The rows of an iteration's first fine stage are the boundaries
// U_n, whose distances the coarse stages' own hit tests have already summed;
// they are kept per block (dist0). The Eq. 2 partials of a boundary come from
// the coarse stage that overwrites it, which also starts the next fine sweep
// (Y_n <- U_n) where it has just read F_n: no separate pass over the
// boundaries at the end of an iteration.
//
// Data (rows of D): U [B][N+1] boundaries; Y [B][N] fine states (F after the
// sweep); G [B][N] coarse results; Xh [B][T] and Eh [B][T] the cache; batch_x
// [B*N][D] fp32. The trajectory states U, Y, G, Xh are pairs of fp32 values,
// an unevaluated sum hi + lo of about 48 bits, a row being D hi parts and then
// D lo parts: a sample passes through about T steps plus N corrections, one
// rounding each, and single fp32 states drift by ~1e-5 of the latent scale over
// T = 100 (measured). Eh is fp32: the denoiser sees fp32 rows and returns fp32
// eps.
//
// What bounds it: a coarse stage has B rows and is a latency chain; a fine
// stage moves 24 to 44 bytes per value (x in and out, eps, the next entry's
// xhat, a miss's entry and batch row). Pairs and not fp64: this GPU's fp64 unit
// takes two operations per clock and SM, and the six per value of a fine step,
// with the fp64 shuffles of its sums, were what the stage waited for (25 us of
// a 42 us stage at 8 trajectories of 16,384 values); about 50 fp32 operations
// in their place take 2. The hi parts alone are what the denoiser's batch
// needs, so the gather reads half a row. Every thread takes four values with
// all of its loads issued before the first store, the ones that earlier stages
// wrote before the dependency wait.
#include <cmath>
#include <string>
#include <vector>

#include "../../include/paraanya.h"
#include "pa_internal.h"
#include "pa_pair.h"

namespace pa {
void set_error(const std::string& msg);  // pa_solver.cpp
}

namespace {

using pa::Pair;
using pa::pair_add;
using pa::pair_mul;
using pa::pair_or;
using pa::pair_sub;
using pa::pair_sub_full;
using pa::pair_value;

constexpr int kSThreads = 256;
constexpr int kSCols = 4;            // values per thread: 16 bytes of a row's high and of its low half
constexpr int kSChunk = kSThreads * kSCols;  // columns per apply CTA
constexpr int kSMaxRows = 2048;      // B * N

enum StageKind : int32_t { kCoarseInit = 0, kFine = 1, kCoarse = 2 };

struct SCtl {
  int32_t n_miss, n_active, iter, status;
  long long nfe, hits;
};

struct SDev {
  int T, B, N, s, nstrip;
  int64_t D;
  float* U;           // pairs: row pitch 2 D
  float* Y;
  float* G;
  float* Xh;
  float* Eh;
  int32_t* has;      // [B][T]
  float* batch_x;    // [B*N][D]
  int32_t* miss_bt;  // [B*N][2]
  int32_t* rank;     // [B*N]: miss rank, -1 hit, -2 not live
  double* part;      // [B*N][nstrip] Eq. 2 partials of the block boundaries, one per apply CTA
  double* dist0;     // [B*N] Eq. 4 sums of the next fine sweep's first rows (Y_n = U_n)
  double* sacc;      // [2][B*N] x kAccStride: Eq. 4 sums of the next stage's rows, set = stage number mod 2
  int32_t* active;   // [B]
  int32_t* iters;    // [B]
  float* err_log;    // [N][B]
  const float2* cm1;  // [T] single steps: c_i - 1, a pair like the states
  const float2* e1;   // [T]
  const float2* cjm1; // [N] block jumps: c - 1
  const float2* ej;   // [N]
  SCtl* ctl;
  double tol, cache_thresh;
  double thr_d;      // cache_thresh * D, the bound on a distance's undivided sum
};

struct Stage {
  int32_t kind, j, n, iter;  // fine: j; coarse: n
};

__device__ __forceinline__ int stage_rows(const SDev& d, const Stage& st) {
  return st.kind == kFine ? d.B * d.N : d.B;
}

// Row r of a stage: trajectory b, sampling index i, its input row; false if
// the row takes no part (frozen trajectory, or past the end of a short block).
__device__ __forceinline__ bool row_info(const SDev& d, const Stage& st, int r, int& b, int& n, int& i,
                                         float*& x) {
  if (st.kind == kFine) {
    b = r / d.N;
    n = r % d.N;
    i = n * d.s + st.j;
    const int end = min((n + 1) * d.s, d.T);
    x = d.Y + ((int64_t)b * d.N + n) * 2 * d.D;
    return d.active[b] && i < end;
  }
  b = r;
  n = st.n;
  i = n * d.s;
  x = d.U + ((int64_t)b * (d.N + 1) + n) * 2 * d.D;
  return d.active[b] != 0;
}

// A CTA's partial of an Eq. 4 sum (non-negative) as it enters the fp64
// accumulator that CTAs add into in arrival order: rounded up to a multiple of
// 2^-32, so every partial sum below 2^21 is exactly representable (2^21 / 2^-32
// = 2^53) and the accumulated sum is the same whatever the order; above 2^21
// the mean distance is at least 2^21 / D, far beyond any tau_cache.
__device__ __forceinline__ double quantize_sum(double v) {
  return ceil(v * 4294967296.0) * (1.0 / 4294967296.0);
}

// The sum over a warp (in every lane): a butterfly of pairs, beside one of
// plain values for a sum that is not finite.
__device__ __forceinline__ double warp_sum(Pair v) {
  float plain = v.h;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    v = pair_add(v, Pair{__shfl_xor_sync(0xffffffffu, v.h, o), __shfl_xor_sync(0xffffffffu, v.l, o)});
    plain += __shfl_xor_sync(0xffffffffu, plain, o);
  }
  return pair_value(pair_or(v, plain));
}

// The CTA's sums of v (if with_v) and w (if with_w) in a fixed order, valid in
// thread 0: pairs within a warp, fp64 over the warps.
__device__ __forceinline__ double2 block_sum2(Pair v, bool with_v, Pair w, bool with_w, double2* s_w) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const double sv = with_v ? warp_sum(v) : 0.0, sw = with_w ? warp_sum(w) : 0.0;
  if (lane == 0) s_w[warp] = make_double2(sv, sw);
  __syncthreads();
  double2 t = make_double2(0.0, 0.0);
  if (warp == 0) {
    static_assert(kSThreads / 32 == 8, "three halvings");
    t = s_w[lane & 7];
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) {
      if (with_v) t.x += __shfl_xor_sync(0xffffffffu, t.x, o);
      if (with_w) t.y += __shfl_xor_sync(0xffffffffu, t.y, o);
    }
  }
  return t;
}

// A thread's kSCols values of a row piece of kSChunk columns: adjacent ones
// (VEC: D % 4 == 0, 16-byte accesses), or every kSThreads-th one, so that a
// warp still touches adjacent columns. Columns past D are left alone.
template <bool VEC>
struct Piece {
  int64_t c;  // first column
  int n;      // of kSCols columns, how many lie inside the row
  __device__ Piece(int64_t base, int64_t D) {
    if constexpr (VEC) {
      c = base + (int64_t)threadIdx.x * kSCols;
      n = c < D ? kSCols : 0;
    } else {
      c = base + threadIdx.x;
      n = c < D ? (int)min((int64_t)kSCols, (D - c + kSThreads - 1) / kSThreads) : 0;
    }
  }
  __device__ void load(const float* row, float (&v)[kSCols]) const {
    if constexpr (VEC) {
      if (n) {
        const float4 a = *reinterpret_cast<const float4*>(row + c);
        v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
      }
    } else {
#pragma unroll
      for (int k = 0; k < kSCols; ++k)
        if (k < n) v[k] = row[c + (int64_t)k * kSThreads];
    }
  }
  // a row of pairs: D hi parts, then D lo parts
  __device__ void load(const float* row, int64_t D, Pair (&v)[kSCols]) const {
    float h[kSCols] = {}, l[kSCols] = {};
    load(row, h);
    load(row + D, l);
#pragma unroll
    for (int k = 0; k < kSCols; ++k) v[k] = Pair{h[k], l[k]};
  }
  __device__ void store(float* row, int64_t D, const Pair (&v)[kSCols]) const {
    store(row, {v[0].h, v[1].h, v[2].h, v[3].h});
    store(row + D, {v[0].l, v[1].l, v[2].l, v[3].l});
  }
  __device__ void store(float* row, const float (&v)[kSCols]) const {
    if constexpr (VEC) {
      if (n) *reinterpret_cast<float4*>(row + c) = make_float4(v[0], v[1], v[2], v[3]);
    } else {
#pragma unroll
      for (int k = 0; k < kSCols; ++k)
        if (k < n) row[c + (int64_t)k * kSThreads] = v[k];
    }
  }
};

// One stage's plan and batch, one launch. Every CTA takes the stage's
// decision over its rows (at most 2048) with all of its warps, one 32-row chunk
// per warp at a time: a live row with an entry hits iff its distance sum / D <
// tau_cache (Eq. 5); misses get ranks in row order (trajectory-major) from the
// chunks' ballots and one scan of their miss counts. The
// same inputs give the same plan in every CTA; CTA (0, 0) publishes it (ranks,
// miss list, counters) and clears the distance set the coming apply adds into
// (and, in an iteration's first coarse stage, the blocks' dist0).
// Then every CTA copies (the hi parts, the rows rounded to fp32) its column range of the batch row whose rank is its
// blockIdx.y, if that row holds a miss, kSUnroll pieces at a time with all
// loads before the stores.
constexpr int kSUnroll = 4;

template <bool VEC>
__global__ void __launch_bounds__(kSThreads) k_srds_plan_gather(SDev d, Stage st, int set) {
  pa::pdl_wait();     // everything read here comes from earlier kernels
  pa::pdl_trigger();  // the successor may now be scheduled
  constexpr int kChunks = kSMaxRows / 32, kWarps = kSThreads / 32;
  __shared__ int s_total, s_row;
  __shared__ unsigned s_mm[kChunks], s_hm[kChunks];  // miss / hit bits of each 32-row chunk
  __shared__ int s_base[kChunks];                     // misses before each chunk
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const bool publish = blockIdx.x == 0 && blockIdx.y == 0;
  const int rows = stage_rows(d, st);
  const int R = d.B * d.N;
  const int nchunk = (rows + 31) / 32;
  // 1. hit/miss of every row, one warp per chunk; a row's trajectory flag, entry
  //    flag and distance sum are read together
  for (int c = warp; c < nchunk; c += kWarps) {
    const int r = c * 32 + lane;
    bool live = false, hit = false;
    if (r < rows) {
      int b, n, i;
      float* x;
      live = row_info(d, st, r, b, n, i, x);
      const bool has = i < d.T && d.has[(int64_t)b * d.T + i];
      // the first fine rows are the boundaries: their sums were kept per block
      const double sv = st.kind == kFine && st.j == 0 ? d.dist0[r] : d.sacc[((size_t)set * R + r) * pa::kAccStride];
      hit = live && has && sv < d.thr_d;
    }
    const unsigned mm = __ballot_sync(0xffffffffu, live && !hit), hm = __ballot_sync(0xffffffffu, hit);
    if (lane == 0) {
      s_mm[c] = mm;
      s_hm[c] = hm;
    }
  }
  __syncthreads();
  // 2. each chunk's first rank (exclusive scan of the chunk miss counts, two
  //    chunks per lane), the totals, the counters
  if (warp == 0) {
    const int c0 = 2 * lane, c1 = 2 * lane + 1;
    const int n0 = c0 < nchunk ? __popc(s_mm[c0]) : 0, n1 = c1 < nchunk ? __popc(s_mm[c1]) : 0;
    int incl = n0 + n1;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += v;
    }
    const int excl = incl - (n0 + n1);
    if (c0 < nchunk) s_base[c0] = excl;
    if (c1 < nchunk) s_base[c1] = excl + n0;
    const int hits = __reduce_add_sync(0xffffffffu, (c0 < nchunk ? __popc(s_hm[c0]) : 0) +
                                                        (c1 < nchunk ? __popc(s_hm[c1]) : 0));
    const int total = __shfl_sync(0xffffffffu, incl, 31);
    if (lane == 0) {
      s_total = total;
      s_row = -1;
      if (publish) {
        d.ctl->n_miss = total;
        d.ctl->nfe += total;
        d.ctl->hits += hits;
      }
    }
    if (publish)
      for (int q = lane; q < R; q += 32) {
        d.sacc[((size_t)(set ^ 1) * R + q) * pa::kAccStride] = 0.0;
        if (st.kind != kFine && st.n == 0) d.dist0[q] = 0.0;
      }
  }
  __syncthreads();
  // 3. ranks in row order; the row of this CTA's rank
  for (int c = warp; c < nchunk; c += kWarps) {
    const int r = c * 32 + lane;
    if (r >= rows) continue;
    const unsigned mm = s_mm[c];
    const bool miss = (mm >> lane) & 1u;
    const int rank = s_base[c] + __popc(mm & ((1u << lane) - 1u));
    if (miss && rank == (int)blockIdx.y) s_row = r;  // one row holds each rank
    if (publish) {
      d.rank[r] = miss ? rank : (((s_hm[c] >> lane) & 1u) ? -1 : -2);
      if (miss) {
        int b, n, i;
        float* x;
        row_info(d, st, r, b, n, i, x);
        d.miss_bt[2 * rank] = b;
        d.miss_bt[2 * rank + 1] = i;
      }
    }
  }
  __syncthreads();
  const int m = blockIdx.y, r = s_row;
  if (m >= s_total || r < 0) return;
  int b, n, i;
  float* x;
  row_info(d, st, r, b, n, i, x);
  float* to = d.batch_x + (int64_t)m * d.D;
  const int64_t npiece = (d.D + kSChunk - 1) / kSChunk;
  for (int64_t q0 = blockIdx.x; q0 < npiece; q0 += (int64_t)gridDim.x * kSUnroll) {
    float v[kSUnroll][kSCols];
#pragma unroll
    for (int u = 0; u < kSUnroll; ++u) {
      const int64_t q = q0 + (int64_t)u * gridDim.x;
      if (q < npiece) Piece<VEC>(q * kSChunk, d.D).load(x, v[u]);
    }
#pragma unroll
    for (int u = 0; u < kSUnroll; ++u) {
      const int64_t q = q0 + (int64_t)u * gridDim.x;
      if (q < npiece) Piece<VEC>(q * kSChunk, d.D).store(to, v[u]);
    }
  }
}

// The step of every live row: eps from the batch (miss: the entry becomes
// (x, eps), Eq. 7) or the cache (hit, Eq. 6); then a fine step
// Y <- Y + (c_i - 1) Y + e_i eps, or a coarse jump g = x + (c - 1) x + e eps
// with U_{n+1} = g (iteration 0) or g + F_n - G_n (later), G_n <- g and, for
// the next fine sweep, Y_n <- x.
// The next stage's row that this row's value feeds also gets its Eq. 4
// distance here, added into set `nset`: a fine step feeds the next fine step
// of its block, a coarse block the next one. (The first coarse block's input
// U_0 never changes and equals its entry: its sum stays 0.) A coarse row's own
// distance is that of the next fine sweep's first row of its block too, zero
// once a miss has made the entry equal to the row (NaN if the row holds a
// NaN or an infinity, which is never a hit); it goes to dist0.
// grid: a CTA per kSChunk columns x rows. What earlier stages wrote (x, F, G,
// the old boundary, the next entry's xhat, flags) is read before the
// dependency wait; only the plan and eps, written by the two kernels before,
// are read after it.
template <bool VEC>
__global__ void __launch_bounds__(kSThreads) k_srds_apply(SDev d, Stage st, const float* __restrict__ beps,
                                                         int nset) {
  __shared__ double2 s_w[kSThreads / 32];
  const int r = blockIdx.y;
  int b, n, i;
  float* x;
  const bool live = row_info(d, st, r, b, n, i, x);
  if (!live) {  // every CTA passes the dependency wait before it exits
    pa::pdl_wait();
    return;
  }
  const bool fine = st.kind == kFine, corr = st.kind == kCoarse;
  const Piece<VEC> pc((int64_t)blockIdx.x * kSChunk, d.D);
  const int64_t e_off = ((int64_t)b * d.T + i) * d.D;
  const float2 cm1 = fine ? d.cm1[i] : d.cjm1[n];
  const float2 ec = fine ? d.e1[i] : d.ej[n];
  float* Un1 = d.U + ((int64_t)b * (d.N + 1) + n + 1) * 2 * d.D;
  float* Gn = d.G + ((int64_t)b * d.N + n) * 2 * d.D;
  float* Yn = d.Y + ((int64_t)b * d.N + n) * 2 * d.D;
  // the next stage's row fed by this one, if any: its row index and timestep
  int nrow = -1, i1 = 0;
  if (fine) {
    if (st.j + 1 < d.s && i + 1 < min((n + 1) * d.s, d.T)) { nrow = r; i1 = i + 1; }
  } else if (n + 1 < d.N) {
    nrow = b; i1 = (n + 1) * d.s;
  }
  const bool nhas = nrow >= 0 && d.has[(int64_t)b * d.T + i1] != 0;
  Pair xv[kSCols] = {}, xh1[kSCols] = {}, fv[kSCols] = {}, gv[kSCols] = {}, uv[kSCols] = {};
  pc.load(x, d.D, xv);
  if (nhas) pc.load(d.Xh + ((int64_t)b * d.T + i1) * 2 * d.D, d.D, xh1);
  if (corr) {
    pc.load(Yn, d.D, fv);
    pc.load(Gn, d.D, gv);
    pc.load(Un1, d.D, uv);
  }
  float ev[kSCols] = {};
  // a coarse stage is a chain of round trips: its entry is fetched before the
  // plan is known (a fine stage would pay the bytes of every miss's)
  if (!fine) pc.load(d.Eh + e_off, ev);
  pa::pdl_wait();     // the plan and the batch's eps come from the kernels just before
  pa::pdl_trigger();  // the successor may now be scheduled
  const int rk = d.rank[r];
  if (rk >= 0) {
    pc.load(beps + (int64_t)rk * d.D, ev);
  } else if (fine) {
    pc.load(d.Eh + e_off, ev);
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    if (rk >= 0) d.has[(int64_t)b * d.T + i] = 1;
    if (!fine && rk < 0)
      atomicAdd(d.dist0 + (int64_t)b * d.N + n, d.sacc[((size_t)(nset ^ 1) * d.B * d.N + r) * pa::kAccStride]);
  }
  Pair nv[kSCols], g[kSCols], err = {0.f, 0.f}, dist = {0.f, 0.f};
  float perr = 0.f, pdist = 0.f;  // the plain sums: what is left where the pairs are not finite
#pragma unroll
  for (int k = 0; k < kSCols; ++k) {
    const Pair dr = pair_add(pair_mul(Pair{cm1.x, cm1.y}, xv[k]), pair_mul(Pair{ec.x, ec.y}, ev[k]));
    g[k] = pair_or(pair_add(xv[k], dr), xv[k].h + fmaf(cm1.x, xv[k].h, ec.x * ev[k]));
    nv[k] = corr ? pair_or(pair_add(g[k], pair_sub_full(fv[k], gv[k])), g[k].h + (fv[k].h - gv[k].h)) : g[k];
    if (k < pc.n) {
      if (nhas) {
        const Pair df = pair_sub(nv[k], xh1[k]);
        dist = pair_add(dist, df.h < 0.f ? Pair{-df.h, -df.l} : df);
        pdist += fabsf(nv[k].h - xh1[k].h);
      }
      if (corr) {
        const Pair df = pair_sub(nv[k], uv[k]);
        err = pair_add(err, pair_mul(df, df));
        const float q = nv[k].h - uv[k].h;
        perr = fmaf(q, q, perr);
      }
    }
  }
  if (rk >= 0) {
    pc.store(d.Xh + ((int64_t)b * d.T + i) * 2 * d.D, d.D, xv);
    pc.store(d.Eh + e_off, ev);
    if (!fine) {
      float z = 0.f;
#pragma unroll
      for (int k = 0; k < kSCols; ++k) z += xv[k].h - xv[k].h;
      if (!(z == 0.f)) atomicAdd(d.dist0 + (int64_t)b * d.N + n, (double)z);
    }
  }
  if (fine) {
    pc.store(x, d.D, g);
  } else {
    pc.store(Un1, d.D, nv);
    pc.store(Gn, d.D, g);
    pc.store(Yn, d.D, xv);
  }
  if (nhas || corr) {
    const double2 t = block_sum2(pair_or(err, perr), corr, pair_or(dist, pdist), nhas, s_w);
    if (threadIdx.x == 0) {
      if (corr) d.part[((int64_t)b * d.N + n) * d.nstrip + blockIdx.x] = t.x;
      if (nhas) atomicAdd(d.sacc + ((size_t)nset * d.B * d.N + nrow) * pa::kAccStride, quantize_sum(t.y));
    }
  }
}

// The larger value, NaN if one is (fmax drops it): a trajectory with a NaN
// boundary has not converged.
__device__ __forceinline__ double nan_max(double a, double b) { return b > a || b != b ? b : a; }

// Convergence of every trajectory after iteration `iter` (one CTA, a warp per
// trajectory at a time, a lane per boundary): the boundaries' Eq. 2 sums from
// the apply CTAs' partials in order, then their maximum.
constexpr int kSFinishThreads = 512;

__global__ void __launch_bounds__(kSFinishThreads) k_srds_finish(SDev d, int iter, cudaGraphConditionalHandle next,
                                                                 int has_next) {
  pa::pdl_wait();     // everything read here comes from earlier kernels
  pa::pdl_trigger();  // the successor may now be scheduled
  __shared__ int s_act;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (threadIdx.x == 0) s_act = 0;
  __syncthreads();
  for (int b = warp; b < d.B; b += kSFinishThreads / 32) {
    if (!d.active[b]) continue;
    bool more = true;
    if (iter > 0) {
      double err = 0.0;
      for (int n = lane; n < d.N; n += 32) {
        const double* pt = d.part + ((int64_t)b * d.N + n) * d.nstrip;
        double sum = 0.0;
#pragma unroll 16
        for (int k = 0; k < d.nstrip; ++k) sum += pt[k];
        err = nan_max(err, sum);
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) err = nan_max(err, __shfl_xor_sync(0xffffffffu, err, o));
      err /= (double)d.D;  // one division: the fp64 unit takes two operations per clock
      more = !(err <= d.tol || iter >= d.N);
      if (lane == 0) {
        d.iters[b] = iter;
        d.err_log[(int64_t)(iter - 1) * d.B + b] = (float)err;
        if (!more) d.active[b] = 0;
      }
    }
    if (more && lane == 0) atomicAdd(&s_act, 1);
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    d.ctl->n_active = s_act;
    d.ctl->iter = iter;
    // inside a captured generation: the next iteration's IF node runs only
    // while a trajectory is still active
    if (has_next) cudaGraphSetConditional(next, s_act > 0 ? 1u : 0u);
  }
}

// The start of a generation: the fp32 rows of x_init (pitch D) widened into
// U_0, every flag, sum and counter cleared (grid x trajectories).
__global__ void __launch_bounds__(kSThreads) k_srds_init(SDev d, const float* __restrict__ src) {
  pa::pdl_wait();     // everything read here comes from earlier kernels
  pa::pdl_trigger();  // the successor may now be scheduled
  const int b = blockIdx.y;
  float* to = d.U + (int64_t)b * (d.N + 1) * 2 * d.D;
  const int64_t first = (int64_t)blockIdx.x * kSThreads + threadIdx.x, step = (int64_t)gridDim.x * kSThreads;
  for (int64_t c = first; c < d.D; c += step) {
    to[c] = src[(int64_t)b * d.D + c];
    to[d.D + c] = 0.f;
  }
  for (int64_t q = first; q < d.T; q += step) d.has[(int64_t)b * d.T + q] = 0;
  for (int64_t q = first; q < d.N; q += step) {
    const int64_t r = (int64_t)b * d.N + q, R = (int64_t)d.B * d.N;
    d.dist0[r] = 0.0;
    d.sacc[r * pa::kAccStride] = 0.0;
    d.sacc[(R + r) * pa::kAccStride] = 0.0;
  }
  if (first == 0) {
    d.active[b] = 1;
    d.iters[b] = 0;
    if (b == 0) {
      SCtl c{};
      c.n_active = d.B;
      *d.ctl = c;
    }
  }
}

__global__ void k_srds_store(SDev d, float* __restrict__ dst, int slot) {
  pa::pdl_wait();     // everything read here comes from earlier kernels
  pa::pdl_trigger();  // the successor may now be scheduled
  const int b = blockIdx.y;
  const float* from = d.U + ((int64_t)b * (d.N + 1) + slot) * 2 * d.D;  // the hi parts: rounded to fp32
  for (int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; c < d.D; c += (int64_t)gridDim.x * blockDim.x)
    dst[(int64_t)b * d.D + c] = from[c];
}

struct SLayout {
  size_t U, Y, G, Xh, Eh, has, batch_x, miss_bt, rank, part, dist0, sacc, active, iters, err_log, coef, ctl, total;
};

SLayout s_layout(int T, int64_t D, int B, int N, int nstrip) {
  SLayout L{};
  size_t o = 0;
  auto take = [&](size_t bytes) { size_t at = o; o = pa::align_up(o + bytes, pa::kAlign); return at; };
  const size_t row = (size_t)D * sizeof(float), row2 = 2 * row;  // rows of pairs
  L.U = take((size_t)B * (N + 1) * row2);
  L.Y = take((size_t)B * N * row2);
  L.G = take((size_t)B * N * row2);
  L.Xh = take((size_t)B * T * row2);
  L.Eh = take((size_t)B * T * row);
  L.has = take((size_t)B * T * sizeof(int32_t));
  L.batch_x = take((size_t)B * N * row);
  L.miss_bt = take((size_t)B * N * 2 * sizeof(int32_t));
  L.rank = take((size_t)B * N * sizeof(int32_t));
  L.part = take((size_t)B * N * nstrip * sizeof(double));
  L.dist0 = take((size_t)B * N * sizeof(double));
  L.sacc = take((size_t)2 * B * N * pa::kAccStride * sizeof(double));  // one 128-byte line per sum
  L.active = take((size_t)B * sizeof(int32_t));
  L.iters = take((size_t)B * sizeof(int32_t));
  L.err_log = take((size_t)N * B * sizeof(float));
  L.coef = take((size_t)(2 * T + 2 * N) * sizeof(float2));
  L.ctl = take(sizeof(SCtl));
  L.total = o;
  return L;
}

void s_blocks(int T, int* s, int* N) {
  int v = 1;
  while (v * v < T) ++v;
  *s = v;
  *N = (T + v - 1) / v;
}

}  // namespace

struct pa_srds {
  SDev d;
  SLayout L;
  char* ws;
  cudaStream_t st;
  int phase;      // -1 created, 0 ready for a step, 1 stepped (waiting for eps), 2 done
  int iter;       // current iteration (0 = coarse initialisation)
  int stage;      // index within the iteration: fine stages first (iter >= 1), then coarse
  int64_t g;      // stages since pa_srds_init: the distance set of stage g is g mod 2
  int dev, nsm;   // the device current at pa_srds_create, its SMs
  int64_t launches;
  SCtl* host_ctl;
  // a whole generation captured as one CUDA graph (pa_srds_loop_*): a chain
  // of IF nodes, one per Parareal iteration, each body that iteration's
  // stages; iteration i's finishing kernel sets the condition of i + 1
  cudaGraph_t loop_graph;
  cudaGraphExec_t loop_exec;
  std::vector<cudaGraphConditionalHandle> loop_cond;  // one per iteration 0..N
  cudaGraphNode_t loop_last;  // the IF node of the iteration being captured
  bool loop_capturing;
  int64_t loop_launches0;
};

namespace {

pa_status s_fail(const std::string& m, pa_status code) {
  pa::set_error(m);
  return code;
}

// Forget the captured generation graph.
void s_drop_loop(pa_srds* h) {
  if (h->loop_exec) cudaGraphExecDestroy(h->loop_exec);
  if (h->loop_graph) cudaGraphDestroy(h->loop_graph);  // and the bodies its IF nodes own
  h->loop_exec = nullptr;
  h->loop_graph = nullptr;
  h->loop_cond.clear();
  h->loop_last = nullptr;
}

// Append the IF node of iteration it to the chain and point the capture of
// the sampler's stream at its body.
cudaError_t s_open_iteration(pa_srds* h, int it) {
  cudaGraphNodeParams np = {};
  np.type = cudaGraphNodeTypeConditional;
  np.conditional.handle = h->loop_cond[it];
  np.conditional.type = cudaGraphCondTypeIf;
  np.conditional.size = 1;
  cudaGraphNode_t node = nullptr;
  const cudaGraphNode_t dep = h->loop_last;
  cudaError_t e = cudaGraphAddNode(&node, h->loop_graph, dep ? &dep : nullptr, nullptr, dep ? 1 : 0, &np);
  if (e != cudaSuccess) return e;
  h->loop_last = node;
  // relaxed: calls this thread makes meanwhile on other work must not
  // invalidate the capture
  return cudaStreamBeginCaptureToGraph(h->st, np.conditional.phGraph_out[0], nullptr, nullptr, 0,
                                       cudaStreamCaptureModeRelaxed);
}

// Let go of a generation graph whose capture the runtime invalidated,
// without destroying it: destroying such a graph crashed the host process
// inside the CUDA runtime. The graph leaks; the handle can capture again.
void s_forget_loop(pa_srds* h) {
  h->loop_exec = nullptr;
  h->loop_graph = nullptr;
  h->loop_cond.clear();
  h->loop_last = nullptr;
}

// Whether the sampler's kernels may take [batch][D] values where they lie: in
// this device's memory, outside the workspace or in batch_x, which the kernels
// that start and end a generation do not touch otherwise.
bool s_in_place(const pa_srds* h, const float* x) {
  const SLayout& L = h->L;
  const size_t n = (size_t)h->d.B * h->d.D * sizeof(float);
  return pa::on_device(x, h->dev) && pa::apart(x, n, h->ws, L.batch_x) &&
         pa::apart(x, n, h->ws + L.miss_bt, L.total - L.miss_bt);
}

Stage current_stage(const pa_srds* h) {
  Stage st{};
  st.iter = h->iter;
  const int nfine = h->iter == 0 ? 0 : h->d.s;
  if (h->stage < nfine) {
    st.kind = kFine;
    st.j = h->stage;
  } else {
    st.kind = h->iter == 0 ? kCoarseInit : kCoarse;
    st.n = h->stage - nfine;
  }
  return st;
}

cudaError_t s_sync_ctl(pa_srds* h) {
  cudaError_t e = cudaMemcpyAsync(h->host_ctl, h->d.ctl, sizeof(SCtl), cudaMemcpyDeviceToHost, h->st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(h->st);
  return e;
}

}  // namespace

extern "C" size_t pa_srds_workspace_bytes(int T, int64_t D, int batch) {
  if (T < 1 || T > 100000 || D < 1 || batch < 1 || batch > pa::kMaxBatch) return 0;
  int s, N;
  s_blocks(T, &s, &N);
  if ((int64_t)batch * N > kSMaxRows) return 0;
  return s_layout(T, D, batch, N, (int)((D + kSChunk - 1) / kSChunk)).total;
}

extern "C" pa_status pa_srds_create(pa_srds** out, int T, const int64_t* latent_shape, int ndim,
                                    const double* alphas_cumprod, double tol, double cache_thresh, int batch,
                                    void* workspace_dev, size_t workspace_bytes, void* stream) {
  if (!out) return s_fail("pa_srds_create: out is NULL", PA_ERR_ARG);
  *out = nullptr;
  if (T < 1 || T > 100000 || !latent_shape || ndim < 1 || ndim > 8 || !alphas_cumprod || batch < 1 ||
      batch > pa::kMaxBatch || !(tol >= 0.0) || !(cache_thresh >= 0.0))
    return s_fail("pa_srds_create: bad size, pointer or threshold", PA_ERR_ARG);
  int64_t D = 1;
  for (int k = 0; k < ndim; ++k) {
    if (latent_shape[k] < 1) return s_fail("pa_srds_create: latent_shape entries must be >= 1", PA_ERR_ARG);
    D *= latent_shape[k];
  }
  for (int i = 0; i <= T; ++i) {
    const double a = alphas_cumprod[i];
    if (!(a > 0.0 && a <= 1.0)) return s_fail("pa_srds_create: alphas_cumprod must be in (0, 1]", PA_ERR_ARG);
  }
  int s, N;
  s_blocks(T, &s, &N);
  if ((int64_t)batch * N > kSMaxRows) return s_fail("pa_srds_create: batch * blocks exceeds 2048", PA_ERR_ARG);
  const int nstrip = (int)((D + kSChunk - 1) / kSChunk);
  const SLayout L = s_layout(T, D, batch, N, nstrip);
  if (!workspace_dev || (reinterpret_cast<uintptr_t>(workspace_dev) % pa::kAlign) != 0 || workspace_bytes < L.total)
    return s_fail("pa_srds_create: workspace NULL, not 256-byte aligned, or smaller than pa_srds_workspace_bytes()",
                  PA_ERR_WORKSPACE);
  pa_srds* h = new pa_srds{};
  h->L = L;
  h->ws = static_cast<char*>(workspace_dev);
  h->st = static_cast<cudaStream_t>(stream);
  h->phase = -1;
  char* w = h->ws;
  SDev& d = h->d;
  d.T = T; d.B = batch; d.N = N; d.s = s; d.nstrip = nstrip; d.D = D;
  d.U = reinterpret_cast<float*>(w + L.U);
  d.Y = reinterpret_cast<float*>(w + L.Y);
  d.G = reinterpret_cast<float*>(w + L.G);
  d.Xh = reinterpret_cast<float*>(w + L.Xh);
  d.Eh = reinterpret_cast<float*>(w + L.Eh);
  d.has = reinterpret_cast<int32_t*>(w + L.has);
  d.batch_x = reinterpret_cast<float*>(w + L.batch_x);
  d.miss_bt = reinterpret_cast<int32_t*>(w + L.miss_bt);
  d.rank = reinterpret_cast<int32_t*>(w + L.rank);
  d.part = reinterpret_cast<double*>(w + L.part);
  d.dist0 = reinterpret_cast<double*>(w + L.dist0);
  d.sacc = reinterpret_cast<double*>(w + L.sacc);
  d.active = reinterpret_cast<int32_t*>(w + L.active);
  d.iters = reinterpret_cast<int32_t*>(w + L.iters);
  d.err_log = reinterpret_cast<float*>(w + L.err_log);
  float2* coef = reinterpret_cast<float2*>(w + L.coef);
  d.cm1 = coef;
  d.e1 = coef + T;
  d.cjm1 = coef + 2 * T;
  d.ej = coef + 2 * T + N;
  d.ctl = reinterpret_cast<SCtl*>(w + L.ctl);
  d.tol = tol;
  d.cache_thresh = cache_thresh;
  d.thr_d = cache_thresh * (double)D;
  // DDIM (eta = 0) jump from a to a2: x + (c - 1) x + e eps with c = sqrt(a2 / a),
  // e = sqrt(1 - a2) - sqrt(a2 (1 - a) / a); c - 1 formed without cancellation.
  // Each coefficient is handed over as a pair.
  auto pair = [](double v) {
    const float h = (float)v;
    return make_float2(h, (float)(v - (double)h));
  };
  auto jump = [&pair](double a, double a2, float2* cm1, float2* e) {
    const double r = a2 / a, c = std::sqrt(r);
    *cm1 = pair((r - 1.0) / (c + 1.0));
    *e = pair(std::sqrt(1.0 - a2) - std::sqrt(a2) * std::sqrt(1.0 - a) / std::sqrt(a));
  };
  std::vector<float2> hc(2 * (size_t)T + 2 * (size_t)N);
  for (int i = 0; i < T; ++i) jump(alphas_cumprod[i], alphas_cumprod[i + 1], &hc[i], &hc[T + i]);
  for (int n = 0; n < N; ++n) {
    const int a0 = n * s, a1 = (n + 1) * s < T ? (n + 1) * s : T;
    jump(alphas_cumprod[a0], alphas_cumprod[a1], &hc[2 * T + n], &hc[2 * T + N + n]);
  }
  cudaError_t e = cudaGetDevice(&h->dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&h->nsm, cudaDevAttrMultiProcessorCount, h->dev);
  if (e == cudaSuccess) e = cudaHostAlloc(reinterpret_cast<void**>(&h->host_ctl), sizeof(SCtl), cudaHostAllocDefault);
  if (e == cudaSuccess) e = cudaMemcpyAsync(coef, hc.data(), hc.size() * sizeof(float2), cudaMemcpyHostToDevice, h->st);
  if (e == cudaSuccess) e = cudaMemsetAsync(d.ctl, 0, sizeof(SCtl), h->st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(h->st);
  if (e != cudaSuccess) {
    if (h->host_ctl) cudaFreeHost(h->host_ctl);
    delete h;
    return s_fail(std::string("pa_srds_create: ") + cudaGetErrorString(e), PA_ERR_CUDA);
  }
  *out = h;
  return PA_OK;
}

extern "C" pa_status pa_srds_init(pa_srds* h, const float* x_init) {
  if (!h || !x_init) return s_fail("pa_srds_init: NULL argument", PA_ERR_ARG);
  if (h->loop_capturing) return s_fail("pa_srds_init: a generation is being captured", PA_ERR_STATE);
  const SDev& d = h->d;
  // x_init is widened into U_0 from where it lies, or staged in batch_x first
  const bool here = s_in_place(h, x_init);
  cudaError_t e = cudaSuccess;
  if (!here) e = cudaMemcpyAsync(d.batch_x, x_init, (size_t)d.B * d.D * sizeof(float), cudaMemcpyDefault, h->st);
  if (e != cudaSuccess) return s_fail(std::string("pa_srds_init: ") + cudaGetErrorString(e), PA_ERR_CUDA);
  e = pa::launch_ex(k_srds_init, dim3(32, d.B), dim3(kSThreads), 0, h->st, 0, d, here ? x_init : (const float*)d.batch_x);
  h->launches += 1;
  if (e != cudaSuccess) return s_fail(std::string("pa_srds_init: ") + cudaGetErrorString(e), PA_ERR_CUDA);
  h->iter = 0;
  h->stage = 0;
  h->g = 0;
  h->phase = 0;
  return PA_OK;
}

extern "C" pa_status pa_srds_step_async(pa_srds* h, const float** batch_x, const int32_t** miss_bt,
                                        const int32_t** n_miss_dev) {
  if (!h) return s_fail("pa_srds_step_async: NULL handle", PA_ERR_ARG);
  if (h->phase == 2) return PA_DONE;
  if (h->phase != 0) return s_fail("pa_srds_step_async: call order (pa_srds_init, then step / submit)", PA_ERR_STATE);
  const SDev& d = h->d;
  const Stage st = current_stage(h);
  const int rows = st.kind == kFine ? d.B * d.N : d.B;
  // every CTA plans: about two CTAs per SM in all, each copying its part of a row's high half
  int gx = d.nstrip;
  const int gcap = (2 * h->nsm + rows - 1) / rows;
  if (gx > gcap) gx = gcap;
  if (gx > 32) gx = 32;
  if (gx < 1) gx = 1;
  const cudaError_t e = pa::launch_ex(d.D % kSCols == 0 ? k_srds_plan_gather<true> : k_srds_plan_gather<false>,
                                      dim3(gx, rows), dim3(kSThreads), 0, h->st, 0, d, st, (int)(h->g & 1));
  h->launches += 1;
  if (e != cudaSuccess) return s_fail(std::string("pa_srds_step_async: ") + cudaGetErrorString(e), PA_ERR_CUDA);
  if (batch_x) *batch_x = d.batch_x;
  if (miss_bt) *miss_bt = d.miss_bt;
  if (n_miss_dev) *n_miss_dev = &d.ctl->n_miss;
  h->phase = 1;
  return PA_OK;
}

extern "C" pa_status pa_srds_step(pa_srds* h, int* n_miss, const float** batch_x, const int32_t** miss_bt) {
  if (!h || !n_miss) return s_fail("pa_srds_step: NULL argument", PA_ERR_ARG);
  if (h->loop_capturing)
    return s_fail("pa_srds_step: synchronises; inside a capture use pa_srds_step_async", PA_ERR_STATE);
  if (h->phase == 2) return PA_DONE;
  if (h->phase == 0 && h->stage == 0 && h->iter > 0) {  // a new iteration: anything left to refine?
    cudaError_t e = s_sync_ctl(h);
    if (e != cudaSuccess) return s_fail(std::string("pa_srds_step: ") + cudaGetErrorString(e), PA_ERR_CUDA);
    if (h->host_ctl->status != 0) return s_fail("pa_srds_step: device-side failure", PA_ERR_DEVICE);
    if (h->host_ctl->n_active == 0) {
      h->phase = 2;
      return PA_DONE;
    }
  }
  pa_status r = pa_srds_step_async(h, batch_x, miss_bt, nullptr);
  if (r != PA_OK) return r;
  const cudaError_t e = s_sync_ctl(h);
  if (e != cudaSuccess) return s_fail(std::string("pa_srds_step: ") + cudaGetErrorString(e), PA_ERR_CUDA);
  *n_miss = h->host_ctl->n_miss;
  return PA_OK;
}

extern "C" const int32_t* pa_srds_n_miss_dev(const pa_srds* h) { return h ? &h->d.ctl->n_miss : nullptr; }

extern "C" pa_status pa_srds_submit_eps(pa_srds* h, const float* batch_eps) {
  if (!h || !batch_eps) return s_fail("pa_srds_submit_eps: NULL argument", PA_ERR_ARG);
  if (h->phase != 1) return s_fail("pa_srds_submit_eps: no step to complete", PA_ERR_STATE);
  const SDev& d = h->d;
  const Stage st = current_stage(h);
  const int rows = st.kind == kFine ? d.B * d.N : d.B;
  const int nset = (int)((h->g + 1) & 1);  // the next stage's distance set
  // 16-byte accesses need whole groups of four columns and aligned eps rows
  const bool vec = d.D % kSCols == 0 && (reinterpret_cast<uintptr_t>(batch_eps) & 15) == 0;
  cudaError_t e = pa::launch_ex(vec ? k_srds_apply<true> : k_srds_apply<false>, dim3(d.nstrip, rows), dim3(kSThreads),
                                0, h->st, 0, d, st, batch_eps, nset);
  h->launches++;
  const int nstages = (h->iter == 0 ? 0 : d.s) + d.N;
  if (++h->stage == nstages) {  // the iteration is complete
    const bool next = h->loop_capturing && h->iter + 1 <= d.N;  // captured: set the next IF node's condition
    if (e == cudaSuccess)
      e = pa::launch_ex(k_srds_finish, dim3(1), dim3(kSFinishThreads), 0, h->st, 0, d, h->iter,
                        next ? h->loop_cond[h->iter + 1] : (cudaGraphConditionalHandle)0, next ? 1 : 0);
    h->launches += 1;
    h->stage = 0;
    h->iter++;
    if (h->loop_capturing) {  // the iteration's body is complete: close it, open the next one's
      cudaGraph_t body = nullptr;
      const cudaError_t ec = cudaStreamEndCapture(h->st, &body);
      if (e == cudaSuccess) e = ec;
      if (e == cudaSuccess && h->iter <= d.N) e = s_open_iteration(h, h->iter);
      if (e != cudaSuccess) {  // nothing ran; the capture is closed and dropped
        (void)cudaGetLastError();
        h->loop_capturing = false;
        if (ec != cudaSuccess)
          s_forget_loop(h);  // an invalidated capture: destroy nothing
        else
          s_drop_loop(h);
        h->phase = -1;  // pa_srds_init must follow
        return s_fail(std::string("pa_srds_submit_eps: capture: ") + cudaGetErrorString(e), PA_ERR_CUDA);
      }
    }
  }
  h->g++;
  if (e != cudaSuccess) return s_fail(std::string("pa_srds_submit_eps: ") + cudaGetErrorString(e), PA_ERR_CUDA);
  h->phase = (h->iter > d.N) ? 2 : 0;
  return PA_OK;
}

extern "C" pa_status pa_srds_poll(pa_srds* h, int* n_active) {
  if (!h) return s_fail("pa_srds_poll: NULL handle", PA_ERR_ARG);
  if (h->loop_capturing) return s_fail("pa_srds_poll: synchronises; not inside a capture", PA_ERR_STATE);
  const cudaError_t e = s_sync_ctl(h);
  if (e != cudaSuccess) return s_fail(std::string("pa_srds_poll: ") + cudaGetErrorString(e), PA_ERR_CUDA);
  const int act = h->host_ctl->n_active;
  if (n_active) *n_active = act;
  if (act == 0 && h->phase == 0) h->phase = 2;
  return act == 0 ? PA_DONE : PA_OK;
}

extern "C" pa_status pa_srds_result(pa_srds* h, float* x_out) {
  if (!h || !x_out) return s_fail("pa_srds_result: NULL argument", PA_ERR_ARG);
  if (h->loop_capturing) return s_fail("pa_srds_result: synchronises; not inside a capture", PA_ERR_STATE);
  if (h->phase != 2) return s_fail("pa_srds_result: not finished", PA_ERR_STATE);
  const SDev& d = h->d;
  // U_N narrowed to fp32 where it is wanted, or in batch_x (free once sampling
  // is done) and then copied out
  const bool here = s_in_place(h, x_out);
  cudaError_t e = pa::launch_ex(k_srds_store, dim3(32, d.B), dim3(256), 0, h->st, 0, d, here ? x_out : d.batch_x, d.N);
  h->launches++;
  if (e == cudaSuccess && !here)
    e = cudaMemcpyAsync(x_out, d.batch_x, (size_t)d.B * d.D * sizeof(float), cudaMemcpyDefault, h->st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(h->st);
  if (e != cudaSuccess) return s_fail(std::string("pa_srds_result: ") + cudaGetErrorString(e), PA_ERR_CUDA);
  return PA_OK;
}

extern "C" pa_status pa_srds_loop_capture_begin(pa_srds* h) {
  if (!h) return s_fail("pa_srds_loop_capture_begin: NULL handle", PA_ERR_ARG);
  if (h->loop_capturing) return s_fail("pa_srds_loop_capture_begin: a capture is already open", PA_ERR_STATE);
  if (h->phase != 0 || h->iter != 0 || h->stage != 0 || h->g != 0)
    return s_fail("pa_srds_loop_capture_begin: call right after pa_srds_init", PA_ERR_STATE);
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  cudaError_t e = cudaStreamIsCapturing(h->st, &cs);
  if (e != cudaSuccess) return s_fail(std::string("pa_srds_loop_capture_begin: ") + cudaGetErrorString(e), PA_ERR_CUDA);
  if (cs != cudaStreamCaptureStatusNone)
    return s_fail("pa_srds_loop_capture_begin: the stream is already being captured", PA_ERR_STATE);
  s_drop_loop(h);
  e = cudaGraphCreate(&h->loop_graph, 0);
  // iteration 0 (the coarse sweep) always runs; every later one only when the
  // previous one's finishing kernel found a trajectory still active
  h->loop_cond.assign((size_t)h->d.N + 1, 0);
  for (int i = 0; i <= h->d.N && e == cudaSuccess; ++i)
    e = cudaGraphConditionalHandleCreate(&h->loop_cond[i], h->loop_graph, i == 0 ? 1u : 0u,
                                         cudaGraphCondAssignDefault);
  if (e == cudaSuccess) e = s_open_iteration(h, 0);
  if (e != cudaSuccess) {
    (void)cudaGetLastError();
    s_drop_loop(h);
    return s_fail(std::string("pa_srds_loop_capture_begin: ") + cudaGetErrorString(e), PA_ERR_CUDA);
  }
  h->loop_capturing = true;
  h->loop_launches0 = h->launches;
  return PA_OK;
}

extern "C" pa_status pa_srds_loop_capture_end(pa_srds* h) {
  if (!h) return s_fail("pa_srds_loop_capture_end: NULL handle", PA_ERR_ARG);
  if (!h->loop_capturing) return s_fail("pa_srds_loop_capture_end: no capture is open", PA_ERR_STATE);
  h->loop_capturing = false;
  if (h->phase != 2) {  // a body is still open: close it, keep nothing
    cudaGraph_t body = nullptr;
    const cudaError_t ec = cudaStreamEndCapture(h->st, &body);
    (void)cudaGetLastError();
    if (ec != cudaSuccess)
      s_forget_loop(h);  // an invalidated capture: destroy nothing
    else
      s_drop_loop(h);
    h->phase = -1;  // pa_srds_init must follow
    return s_fail("pa_srds_loop_capture_end: issue every stage first (pa_srds_step_async until PA_DONE)",
                  PA_ERR_STATE);
  }
  const cudaError_t e = cudaGraphInstantiate(&h->loop_exec, h->loop_graph, 0);
  if (e != cudaSuccess) {
    (void)cudaGetLastError();
    s_drop_loop(h);
    h->phase = -1;
    return s_fail(std::string("pa_srds_loop_capture_end: ") + cudaGetErrorString(e), PA_ERR_CUDA);
  }
  // nothing ran: back to the state right after pa_srds_init
  h->iter = 0;
  h->stage = 0;
  h->g = 0;
  h->phase = 0;
  h->launches = h->loop_launches0;
  return PA_OK;
}

extern "C" pa_status pa_srds_loop_launch(pa_srds* h) {
  if (!h) return s_fail("pa_srds_loop_launch: NULL handle", PA_ERR_ARG);
  if (!h->loop_exec) return s_fail("pa_srds_loop_launch: nothing has been captured", PA_ERR_STATE);
  if (h->loop_capturing || h->phase != 0 || h->iter != 0 || h->stage != 0 || h->g != 0)
    return s_fail("pa_srds_loop_launch: call right after pa_srds_init", PA_ERR_STATE);
  const cudaError_t e = cudaGraphLaunch(h->loop_exec, h->st);
  if (e != cudaSuccess) return s_fail(std::string("pa_srds_loop_launch: ") + cudaGetErrorString(e), PA_ERR_CUDA);
  h->phase = 2;  // the graph runs the generation to its end
  h->iter = h->d.N + 1;
  return PA_OK;
}

extern "C" pa_status pa_srds_stats(pa_srds* h, pa_srds_stats_t* out) {
  if (!h || !out) return s_fail("pa_srds_stats: NULL argument", PA_ERR_ARG);
  if (h->loop_capturing) return s_fail("pa_srds_stats: synchronises; not inside a capture", PA_ERR_STATE);
  const cudaError_t e = s_sync_ctl(h);
  if (e != cudaSuccess) return s_fail(std::string("pa_srds_stats: ") + cudaGetErrorString(e), PA_ERR_CUDA);
  out->iters = h->host_ctl->iter;
  out->nfe = h->host_ctl->nfe;
  out->hits = h->host_ctl->hits;
  out->launches = h->launches;
  out->n_active = h->host_ctl->n_active;
  out->n_miss = h->host_ctl->n_miss;
  out->device_status = h->host_ctl->status;
  out->blocks = h->d.N;
  out->block_steps = h->d.s;
  return PA_OK;
}

extern "C" pa_status pa_srds_errors(pa_srds* h, float* err_out) {
  if (!h || !err_out) return s_fail("pa_srds_errors: NULL argument", PA_ERR_ARG);
  const cudaError_t e = cudaMemcpy(err_out, h->d.err_log, (size_t)h->d.N * h->d.B * sizeof(float),
                                   cudaMemcpyDeviceToHost);
  if (e != cudaSuccess) return s_fail(std::string("pa_srds_errors: ") + cudaGetErrorString(e), PA_ERR_CUDA);
  return PA_OK;
}

extern "C" void pa_srds_destroy(pa_srds* h) {
  if (!h) return;
  if (h->loop_capturing) {  // close the capture so that the stream stays usable
    cudaGraph_t g = nullptr;
    if (cudaStreamEndCapture(h->st, &g) != cudaSuccess) s_forget_loop(h);
    (void)cudaGetLastError();
  }
  s_drop_loop(h);
  if (h->host_ctl) cudaFreeHost(h->host_ctl);
  delete h;
}
