// Synthetic denoiser: posterior-mean noise of an isotropic Gaussian mixture,
// the seedable stand-in for the SD v1.5 UNet eps_theta (Sec. 3.2). Not part
// of ParaAnya; it produces the fresh eps of the misses (Eq. 6, miss branch).
//
//   v = a s^2 + 1 - a,   logit_k = (2 sqrt(a) x.mu_k - a ||mu_k||^2) / (2 v)
//   r = softmax(logit)   (the common -||x||^2 / (2 v) term cancels)
//   eps = sqrt(1 - a) / v * (x - sqrt(a) sum_k r_k mu_k)
//
// Three ways to compute it, chosen per handle (pa_gmm_create):
//   one kernel on thread-block clusters (k_gmm_cluster, form 2)
//   three persistent tensor-core kernels (k_gmm_tc.cu, form 1)
//   two CUDA-core kernels (form 0):
//   k_gmm_dots     dot products G = X M^T, split over column chunks of D
//                  (16-row tiles staged in shared memory, 4 rows x 8
//                  components per thread); each CTA adds its chunk sums, in
//                  fixed point, into int64 accumulators with integer atomics
//                  (exact: the order of arrival does not matter)
//   k_gmm_out      per 16-row block: logits and max-subtracted softmax of its
//                  rows from the accumulators, then eps = a x - a sqrt(a) R M
//                  over staged 16-row x 256-column tiles (4 x 4 outputs per
//                  thread)
// The accumulators come in two sets used in turn. A call's dot-product kernel
// reads the handle's epoch e, accumulates into set e mod 2, clears the other
// set (read by the previous call's output kernel, complete behind the dependency
// wait) and records e for the output kernel; the output kernel reads set e mod 2
// and advances the epoch. No kernel waits for another CTA, and the state lives on
// the device, so a captured CUDA graph replays correctly.
// The fixed point goes by the means (fixed_scale); a sum beyond it marks its
// accumulator, and the output kernel forms that dot product itself.
// Per-timestep scalars (sqrt(a), 1/(2v), sqrt(1-a)/v) are computed on the
// host in fp64 from alpha-bar and stored in fp32, so 1 - a never cancels in
// fp32. Reductions run in a fixed order: results are bitwise reproducible.
#include <cooperative_groups.h>

#include <cmath>
#include <cstdlib>
#include <cstring>
#include <string>
#include <vector>

#include "../../include/paraanya.h"
#include "pa_bulk.cuh"
#include "pa_gmm_tc.h"
#include "pa_internal.h"

namespace pa {
void set_error(const std::string& msg);  // pa_solver.cpp
}

namespace {

namespace cg = cooperative_groups;

using pa::pdl_trigger;
using pa::pdl_wait;
using pa::bulk_g2s;
using pa::fence_barrier_init;
using pa::mbar_arrive_expect_tx;
using pa::mbar_init;
using pa::mbar_wait_bounded;
using pa::smem_u32;

constexpr int kMaxK = 128;
constexpr int kThreads = 256;
constexpr int kDotRows = 16;     // rows per dots CTA (two per warp)
constexpr int kOutRows = 16;     // rows per output CTA
constexpr int kOutCols = 256;    // columns per output CTA (four per thread)
constexpr size_t kDotSmemBudget = 96 * 1024;
constexpr int kDotCtas = 480;    // CTAs that a dots launch should have: about three per SM

// The fixed point of the dot-product accumulators. Let 2^e be the root mean
// square of the largest mean, rounded down; rows are of the order of the means
// or of the unit noise, whichever is larger, so their products are of the order
// of 2^(e + max(e, 0)), and a unit is 2^-32 of that: at unit scale 2^-32. A chunk
// sum that leaves no room for `nchunk` of its size (2^59 units) is not added but
// marks the accumulator, a value that is not finite with the higher mark; the
// others' sums, below 2^59 in any order, move a mark by less than half of the
// distance to the next. So dot products of any size come out as in fp32: the
// output kernel forms a marked one from the row and the mean (up to kWideD
// columns: 16 rows of them take it 27 ms at 16 components; beyond, the row is
// NaN), and a row with a value that is not finite is NaN.
constexpr float kFixedRoom = 0x1p59f;
constexpr long long kMarkWide = 4ll << 60, kMarkNan = 6ll << 60;
constexpr int64_t kWideD = 1 << 18;
__device__ __forceinline__ int fixed_exponent(uint32_t norm_bits, int64_t D) {  // log2 of the units in 1
  const float ms = __uint_as_float(norm_bits) / (float)D;  // mean square
  if (!(ms > 0.f)) return 32;
  const int e = max(-40, min(40, ((int)(__float_as_uint(ms) >> 23) - 127) >> 1));
  return 32 - e - max(e, 0);
}
__device__ __forceinline__ float power_of_two(int e) { return __int_as_float((e + 127) << 23); }  // |e| <= 126

// Default form by sizes (pa_gmm_create). K components, D columns, a capacity of R
// rows; the figures are us per call on a batch filled to 4/5.
// Above 16 components the persistent tensor-core kernels (form 1) cost 12 us
// before they do anything, the CUDA-core kernels (form 0) 6, and those take time
// with K: form 1 from K D R = kTcWork on, above 64 components from kTcWideWork.
// Form 0 / 1: K 32, D 8192, R 64 (17e6) 10.5 / 13.7; K 32, D 16384, R 64 (34e6)
// 13.3 / 15.6; K 64, D 8192, R 128 (67e6) 20.1 / 16.5; K 64, D 65536, R 128
// (537e6) 145 / 41; K 90, D 8192, R 16 (12e6) 16.0 / 17.4; K 128, D 4096, R 64
// (34e6) 23.2 / 17.9; a generation at K 95, D 784, R 306 (23e6) 278 / 226.
// Up to 16 components the cluster kernel (form 2) is the shortest chain, but its
// time goes with the rows, eight to a cluster of 16 CTAs, however few columns
// they have: form 0 for many short rows. Form 0 / 2: K 8, D 4096, R 256 7.9 / 9.8,
// R 100 8.6 / 5.2; K 8, D 8192, R 256 10.2 / 10.8, R 400 14.7 / 16.9; K 16,
// D 16384, R 400 30.1 / 24.9; a generation at K 4, D 4224, R 256 815 / 910.
// Where the work is large form 1 wins here too: form 0 / 1 / 2 at K 16, D 16384,
// R 1000 (262e6) 63.1 / 56.4 / 58.6, R 1600 86.8 / 73.2 / 81.1; without the
// cluster kernel form 0 / 1 at K 16, D 40000, R 256 (164e6) 42.4 / 38.1, at K 8,
// R 1000 (320e6) 110 / 122, and with D % 4 != 0, where form 1 copies four bytes at
// a time, at K 16, D 40001, R 1000 170 / 188. Rows that form 0's fixed point does
// not hold (kWideD) take form 1 above 16 components.
constexpr int64_t kTcWork = 40 * 1000 * 1000;
constexpr int64_t kTcWideWork = 12 * 1000 * 1000;
constexpr int kManyRows = 200;        // many short rows: R >= kManyRows, D <= kShortRow,
constexpr int64_t kShortRow = 10000;  // and D <= kShortPerRow R
constexpr int64_t kShortPerRow = 25;
constexpr int64_t kTcFewWork = 250 * 1000 * 1000;   // up to 16 components, against form 2 ...
constexpr int kTcFewRows = 512;
constexpr int64_t kTcFewWork0 = 100 * 1000 * 1000;  // ... and against form 0
constexpr int kTcFewMinK = 9;

struct GmmLayout {
  size_t tc;        // scratch of the persistent tensor-core kernels
  size_t coef, mnorm, gacc, epoch, status, total;
  int nchunk;       // D-chunks of the CUDA-core dots kernel
  int chunk;        // columns per chunk
};

// Which accumulator set a call uses (see the file comment).
struct GmmEpoch {
  uint32_t epoch;   // advanced by the output kernel
  uint32_t cur;     // the epoch of the dot products just formed
  float scale;      // units of the fixed point in 1, and its inverse
  float unit;
  uint32_t norm;    // the largest ||mu_k||^2, as the bits of the fp32 value
  uint32_t norms;   // components whose norm is in it
};

size_t dots_smem_bytes(int K, int chunk) {
  // the staged tiles, later reused for the column-split sums
  int KG = 1;
  while (KG * 8 < K) KG <<= 1;
  const size_t tiles = (size_t)(kDotRows + K) * (chunk + 4) * sizeof(float);
  const size_t red = (size_t)(kThreads / (4 * KG) + 1) * kDotRows * K * sizeof(float);
  return tiles > red ? tiles : red;
}

int dots_chunk(int K, int64_t D, int max_rows) {
  // largest of 512/256/128/64 columns whose (rows + K) row segments fit the budget
  int c = 512;
  while (c > 64 && (size_t)(kDotRows + K) * (c + 4) * sizeof(float) > kDotSmemBudget) c /= 2;
  while (c > 64 && (int64_t)c >= 2 * D) c /= 2;
  // down to 128 while the launch has fewer CTAs than the SMs hold at a time, whose
  // copies and sums then overlap. A generation with 60, 120, 240 and 480 in place
  // of kDotCtas: 12810 columns, 50 rows, 16 components 110.8, 107.3, 102.7, 102.6
  // us; 3600 columns, 144 rows, 30 components 129, 127.5, 122.3, 122.2; 13860
  // columns, 150 rows, 12 components 152.0, 151.8, 152.0, 149.8
  const int64_t blocks = (max_rows + kDotRows - 1) / kDotRows;
  while (c > 128 && (D + c - 1) / c * blocks < kDotCtas) c /= 2;
  return c;
}

GmmLayout gmm_layout(int K, int64_t D, int max_rows, int T) {
  GmmLayout L{};
  size_t o = 0;
  auto take = [&](size_t bytes) { size_t at = o; o = pa::align_up(o + bytes, pa::kAlign); return at; };
  L.chunk = dots_chunk(K, D, max_rows);
  L.nchunk = (int)((D + L.chunk - 1) / L.chunk);
  L.coef = take((size_t)3 * T * sizeof(float));
  L.mnorm = take((size_t)K * sizeof(float));
  L.gacc = take((size_t)2 * max_rows * K * sizeof(long long));  // two sets, used in turn
  L.epoch = take(sizeof(GmmEpoch));
  L.status = take(sizeof(int32_t));
  L.tc = take(pa::gmm_tc_layout(K, D, max_rows).total);
  L.total = o;
  return L;
}

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// ||mu_k||^2, one CTA per component, fixed-order tree; the last one to finish
// takes the fixed point from the largest.
__global__ void __launch_bounds__(256) k_gmm_norms(const float* __restrict__ mu, int64_t D,
                                                   float* __restrict__ mnorm, GmmEpoch* ep) {
  __shared__ float s[8];
  const float* m = mu + (int64_t)blockIdx.x * D;
  float acc = 0.f;
  for (int64_t d = threadIdx.x; d < D; d += 256) acc = fmaf(m[d], m[d], acc);
  acc = warp_sum(acc);
  if ((threadIdx.x & 31) == 0) s[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    float t = 0.f;
    for (int w = 0; w < 8; ++w) t += s[w];
    mnorm[blockIdx.x] = t;
    if (t > 0.f) atomicMax(&ep->norm, __float_as_uint(t));  // the bits of positive values are in their order
    __threadfence();
    if (atomicAdd(&ep->norms, 1u) == gridDim.x - 1) {
      const int e = fixed_exponent(atomicMax(&ep->norm, 0u), D);
      ep->scale = power_of_two(e);
      ep->unit = power_of_two(-e);
    }
  }
}

// Stage `nrows` row segments [c0, c0 + ncol) of a row-major matrix with row
// length D into shared rows of stride `ld` floats: bulk copies counted on
// `bar`, issued by the lanes of warp 0 (after the caller announced the bytes),
// or, when `bulk` is false (rows that start on no 16-byte boundary), 4-byte
// asynchronous copies by every warp: no register waits for them, so a thread
// has all of its copies in flight together.
__device__ __forceinline__ void stage_rows(float* dst, int ld, const float* src, int64_t D, int64_t c0,
                                           int ncol, int nrows, bool bulk, uint64_t* bar) {
  if (bulk) {
    if (threadIdx.x < 32) {  // the lanes of warp 0 issue the rows in parallel
      const uint32_t seg = (uint32_t)ncol * sizeof(float);
      for (int r = threadIdx.x; r < nrows; r += 32)
        bulk_g2s(dst + (size_t)r * ld, src + (int64_t)r * D + c0, seg, bar);
    }
    return;
  }
  const int lane = threadIdx.x & 31;
  for (int r = threadIdx.x >> 5; r < nrows; r += blockDim.x >> 5) {
    const float* sr = src + (int64_t)r * D + c0;
    const uint32_t dr = smem_u32(dst + (size_t)r * ld);
    for (int c = lane; c < ncol; c += 32)
      asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dr + 4 * c), "l"(sr + c) : "memory");
  }
}

// Wait for the bulk copies of a single-phase kernel (without them, for the
// calling thread's own copies; the caller's barrier makes the others' visible).
// On a timeout: record it, let the copies already issued land (bounded), and
// report false.
__device__ __forceinline__ bool wait_staged(bool bulk, uint64_t* bar, int32_t* status) {
  if (!bulk) {
    asm volatile("cp.async.wait_all;" ::: "memory");
    return true;
  }
  if (mbar_wait_bounded(bar, 0, pa::kWaitLimit)) return true;
  atomicCAS(status, 0, pa::kDevTimeout);
  mbar_wait_bounded(bar, 0, pa::kDrainLimit);
  return false;
}

// The accumulator set of a dot-product kernel whose call has epoch e; all CTAs
// together (every CTA, also those without rows) clear the other set, and e is
// recorded for the output kernel. Only behind the dependency wait: the previous
// call's output kernel, which reads the other set and advances the epoch, may be
// the kernel just before.
__device__ __forceinline__ long long* begin_dots(long long* gacc2, GmmEpoch* ep, uint32_t e, int64_t set_size) {
  long long* other = gacc2 + (int64_t)((e + 1u) & 1u) * set_size;
  const int64_t cta = (int64_t)blockIdx.y * gridDim.x + blockIdx.x;
  const int64_t nthr = (int64_t)gridDim.x * gridDim.y * blockDim.x;
  for (int64_t q = cta * blockDim.x + threadIdx.x; q < set_size; q += nthr) other[q] = 0;
  if (cta == 0 && threadIdx.x == 0) ep->cur = e;
  return gacc2 + (int64_t)(e & 1u) * set_size;
}

// Dot products on the CUDA cores: a CTA stages 16 rows x `chunk` columns of
// X and the same columns of every mean, each thread accumulates a 4-row x
// 8-component block over a column split (register tiling: 12 shared loads per
// 32 FMAs), the column splits are summed in a fixed order through shared
// memory, and the chunk sums go into the accumulators (file comment).
__global__ void __launch_bounds__(kThreads) k_gmm_dots(const float* __restrict__ X,
                                                       const float* __restrict__ mu,
                                                       const int32_t* __restrict__ n_rows_dev,
                                                       int K, int64_t D, int chunk, float room, int max_rows,
                                                       bool bulk, long long* __restrict__ gacc2,
                                                       GmmEpoch* ep, int32_t* status) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  __shared__ __align__(8) uint64_t bar_m, bar_x;
  const int r0 = blockIdx.y * kDotRows;
  const int64_t c0 = (int64_t)blockIdx.x * chunk;
  const int ncol = (int)(((D - c0) < chunk) ? (D - c0) : chunk);
  const int ld = chunk + 4;  // padded row stride, keeps 16-byte alignment
  float* xs = reinterpret_cast<float*>(smem_raw);
  float* ms = xs + (size_t)kDotRows * ld;
  const int tid = threadIdx.x;
  if (tid == 0) {
    mbar_init(&bar_m, 1);
    mbar_init(&bar_x, 1);
    fence_barrier_init();
    if (bulk) mbar_arrive_expect_tx(&bar_m, (uint32_t)ncol * sizeof(float) * (uint32_t)K);
  }
  __syncthreads();
  stage_rows(ms, ld, mu, D, c0, ncol, K, bulk, &bar_m);  // the means do not depend on the predecessor
  pdl_wait();  // the rows and their count come from the kernel just before
  pdl_trigger();  // the successor may now run its prologue
  const int n_rows = min(*n_rows_dev, max_rows);
  const uint32_t epoch = ep->epoch;
  const float scale = ep->scale;
  const int nr = min(kDotRows, n_rows - r0);
  if (nr <= 0) {  // no rows for this CTA: the means copy lands before it exits
    begin_dots(gacc2, ep, epoch, (int64_t)max_rows * K);
    wait_staged(bulk, &bar_m, status);
    return;
  }
  for (int q = tid; q < (kDotRows - nr) * ld; q += kThreads) xs[(size_t)nr * ld + q] = 0.f;  // rows past nr
  if (tid == 0 && bulk) mbar_arrive_expect_tx(&bar_x, (uint32_t)ncol * sizeof(float) * (uint32_t)nr);
  __syncthreads();
  stage_rows(xs, ld, X + (int64_t)r0 * D, D, c0, ncol, nr, bulk, &bar_x);
  long long* gacc = begin_dots(gacc2, ep, epoch, (int64_t)max_rows * K);  // while the rows are on their way
  const bool ok_m = wait_staged(bulk, &bar_m, status);
  const bool ok = wait_staged(bulk, &bar_x, status) && ok_m;
  __syncthreads();
  if (!ok) return;

  // thread -> (column split tcs, component group tkg, row group trg)
  int KG = 1;
  while (KG * 8 < K) KG <<= 1;          // component groups of 8 (power of two)
  const int CS = kThreads / (4 * KG);   // column splits
  const int tcs = tid % CS, tkg = (tid / CS) % KG, trg = tid / (CS * KG);
  float acc[4][8];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int u = 0; u < 8; ++u) acc[i][u] = 0.f;
  for (int c = tcs; c < ncol; c += CS) {
    float xv[4], mv[8];
#pragma unroll
    for (int i = 0; i < 4; ++i) xv[i] = xs[(size_t)(trg * 4 + i) * ld + c];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int k = tkg + KG * u;  // interleaved: neighbouring groups read neighbouring rows
      mv[u] = (k < K) ? ms[(size_t)k * ld + c] : 0.f;
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int u = 0; u < 8; ++u) acc[i][u] = fmaf(xv[i], mv[u], acc[i][u]);
  }
  __syncthreads();  // the tiles are consumed: reuse their space for the split sums
  float* red = xs;  // [kDotRows * K][CS + 1]: split index fastest (conflict-free both ways)
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int k = tkg + KG * u;
      if (k < K) red[((size_t)(trg * 4 + i) * K + k) * (CS + 1) + tcs] = acc[i][u];
    }
  __syncthreads();
  for (int o = tid; o < nr * K; o += kThreads) {
    float a4[4] = {0.f, 0.f, 0.f, 0.f};
    const float* ro = red + (size_t)o * (CS + 1);
    int cs = 0;
    for (; cs + 3 < CS; cs += 4) {
      a4[0] += ro[cs];
      a4[1] += ro[cs + 1];
      a4[2] += ro[cs + 2];
      a4[3] += ro[cs + 3];
    }
    for (; cs < CS; ++cs) a4[0] += ro[cs];
    const float sum = (a4[0] + a4[1]) + (a4[2] + a4[3]);
    long long* acc_o = gacc + (int64_t)r0 * K + o;
    if (fabsf(sum * scale) < room)  // and not NaN
      atomicAdd(reinterpret_cast<unsigned long long*>(acc_o), static_cast<unsigned long long>(__float2ll_rn(sum * scale)));
    else
      atomicMax(acc_o, fabsf(sum) <= 3.402823466e38f ? kMarkWide : kMarkNan);
  }
}

// The logits of a row block whose dot products the fixed point did not hold (the
// value `wide` in s_r), by the whole CTA in a fixed order. Seldom: kept out of
// the output kernel's code.
__device__ __noinline__ void form_wide(const float* __restrict__ X, const float* __restrict__ mu,
                                       const float* __restrict__ mnorm, int K, int64_t D, int nr, float wide,
                                       const float* s_sa, const float* s_q, float* s_r, float* s_part) {
  const int tid = threadIdx.x;
  for (int q = 0; q < nr * K; ++q) {
    if (__float_as_uint(s_r[q]) != __float_as_uint(wide)) continue;  // the same for every thread
    const int rr = q / K, k = q % K;
    const float* xr = X + (int64_t)rr * D;
    const float* mk = mu + (int64_t)k * D;
    float dot = 0.f;
#pragma unroll 8
    for (int64_t c = tid; c < D; c += kThreads) dot = fmaf(xr[c], mk[c], dot);
    dot = warp_sum(dot);
    if ((tid & 31) == 0) s_part[tid >> 5] = dot;
    __syncthreads();
    if (tid == 0) {
      dot = 0.f;
      for (int w = 0; w < kThreads / 32; ++w) dot += s_part[w];
      const float sa = s_sa[rr];
      s_r[q] = (2.f * sa * dot - sa * sa * mnorm[k]) * s_q[rr];
    }
    __syncthreads();
  }
}

// Output kernel. First the 16 rows' responsibilities: the finished dot
// products (accumulator set of this call), the logits with ||mu_k||^2 and the
// per-timestep scalars, and the max-subtracted softmax, while the row and mean
// tiles are in flight. Then eps[r][c] = ac x[r][c] - ac sqrt(a) sum_k
// R[r][k] mu[k][c] over a 16-row x 256-column tile: each thread computes a
// 4-row x 4-column block (one 16-byte mean load and four broadcast
// responsibility loads per 16 FMAs).
__global__ void __launch_bounds__(kThreads) k_gmm_out(const float* __restrict__ X,
                                                      const float* __restrict__ mu,
                                                      const long long* __restrict__ gacc2,
                                                      GmmEpoch* ep, const float* __restrict__ coef, int T,
                                                      const int32_t* __restrict__ miss_bt,
                                                      const float* __restrict__ mnorm,
                                                      const int32_t* __restrict__ n_rows_dev,
                                                      int K, int64_t D, int max_rows, bool bulk, bool vec_out,
                                                      float* __restrict__ eps, int32_t* status) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  __shared__ __align__(8) uint64_t bar;
  __shared__ float s_r[kOutRows * kMaxK];
  __shared__ float s_c[kOutRows * 2];
  __shared__ float s_sa[kOutRows], s_q[kOutRows];
  __shared__ float s_part[kThreads / 32];
  const int n_rows = min(*n_rows_dev, max_rows);  // written two kernels back
  const int r0 = blockIdx.y * kOutRows;
  if (r0 >= n_rows) {  // every CTA passes the dependency wait before it exits
    pdl_wait();
    return;
  }
  const int nr = min(kOutRows, n_rows - r0);
  const int64_t c0 = (int64_t)blockIdx.x * kOutCols;
  const int ncol = (int)(((D - c0) < kOutCols) ? (D - c0) : kOutCols);
  float* ms = reinterpret_cast<float*>(smem_raw);   // [K][kOutCols]
  float* xs = ms + (size_t)K * kOutCols;            // [kOutRows][kOutCols]
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (tid == 0) {
    mbar_init(&bar, 1);
    fence_barrier_init();
    if (bulk) mbar_arrive_expect_tx(&bar, (uint32_t)ncol * sizeof(float) * (uint32_t)(nr + K));
  }
  __syncthreads();
  // the means and the rows (written two kernels back) do not depend on the predecessor
  stage_rows(ms, kOutCols, mu, D, c0, ncol, K, bulk, &bar);
  stage_rows(xs, kOutCols, X + (int64_t)r0 * D, D, c0, ncol, nr, bulk, &bar);
  for (int rr = tid; rr < nr; rr += kThreads) {
    const int i = miss_bt[2 * (r0 + rr) + 1];
    s_sa[rr] = coef[i];
    s_q[rr] = coef[T + i];
    s_c[2 * rr] = coef[2 * T + i];
    s_c[2 * rr + 1] = coef[2 * T + i] * coef[i];
  }
  pdl_wait();  // the dot products come from the kernel just before
  pdl_trigger();  // the successor may now run its prologue
  // both accumulator sets are read together with the set index and the
  // status word (one round trip): a dot-product kernel that timed out left
  // the sums incomplete
  const uint32_t cur = ep->cur;
  const float unit = ep->unit;
  const int dots_status = __ldcg(status);
  const int64_t set_size = (int64_t)max_rows * K;
  __syncthreads();
  const float nan = __int_as_float(0x7fc00000), wide = __int_as_float(0x7fc00001);  // a marked sum until it is formed
  bool any_wide = false;
  for (int q = tid; q < kOutRows * K; q += kThreads) {
    float l = 0.f;
    if (q < nr * K) {
      const int rr = q / K, k = q % K;
      const long long v0 = __ldcg(gacc2 + (int64_t)r0 * K + q);
      const long long v1 = __ldcg(gacc2 + set_size + (int64_t)r0 * K + q);
      const long long v = (cur & 1u) ? v1 : v0;
      if (v >= 3ll << 60) {
        const bool form = v < 5ll << 60 && D <= kWideD;
        l = form ? wide : nan;
        any_wide |= form;
      } else {
        const float dot = __ll2float_rn(v) * unit;  // exact scale
        const float sa = s_sa[rr];
        l = (2.f * sa * dot - sa * sa * mnorm[k]) * s_q[rr];
      }
    }
    s_r[q] = l;
  }
  if (__syncthreads_or(any_wide))
    form_wide(X + (int64_t)r0 * D, mu, mnorm, K, D, nr, wide, s_sa, s_q, s_r, s_part);
  // softmax per row: a half-warp per row when K <= 16 (two rows per warp and
  // pass), else a warp; the reductions are the same trees either way
  {
    const int width = K <= 16 ? 16 : 32, sub = lane / width, sl = lane % width;
    for (int rr0 = warp * (32 / width); rr0 < nr; rr0 += (kThreads / 32) * (32 / width)) {
      const int rr = rr0 + sub;
      const bool ok = rr < nr;
      float* l = s_r + (ok ? rr : 0) * K;
      float mx = -INFINITY;
      if (ok)
        for (int k = sl; k < K; k += width) mx = fmaxf(mx, l[k]);
      for (int o = width / 2; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
      float sum = 0.f;
      if (ok)
        for (int k = sl; k < K; k += width) sum += expf(l[k] - mx);
      for (int o = width / 2; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
      const float inv = 1.f / sum;
      __syncwarp();
      if (ok)
        for (int k = sl; k < K; k += width) l[k] = expf(l[k] - mx) * inv;
    }
  }
  if (blockIdx.x == 0 && blockIdx.y == 0 && tid == 0) ep->epoch = cur + 1u;  // the next call's set
  const bool ok = wait_staged(bulk, &bar, status);
  if (__syncthreads_or(!ok || dots_status != 0)) {
    // a bounded wait ran out here or in the dot products: the tile is written
    // as NaN, so the failure shows in the output as well as in the status word
    for (int q = tid; q < nr * ncol; q += kThreads)
      eps[(int64_t)(r0 + q / ncol) * D + c0 + q % ncol] = __int_as_float(0x7fc00000);
    return;
  }
  // kOutCols / 4 column groups of 4 x kThreads / (kOutCols / 4) row groups of 4
  static_assert(kThreads / (kOutCols / 4) * 4 == kOutRows, "the threads cover the tile's rows");
  const int cg = tid % (kOutCols / 4), rg = tid / (kOutCols / 4);
  const int cc = cg * 4;
  if (cc >= ncol) return;
  float acc[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;
  for (int k = 0; k < K; ++k) {
    const float4 m = *reinterpret_cast<const float4*>(ms + (size_t)k * kOutCols + cc);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float rk = s_r[(rg * 4 + i) * K + k];
      acc[i][0] = fmaf(rk, m.x, acc[i][0]);
      acc[i][1] = fmaf(rk, m.y, acc[i][1]);
      acc[i][2] = fmaf(rk, m.z, acc[i][2]);
      acc[i][3] = fmaf(rk, m.w, acc[i][3]);
    }
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int rr = rg * 4 + i;
    if (rr >= nr) break;
    const float ac = s_c[2 * rr], acs = s_c[2 * rr + 1];
    const float* xr = xs + (size_t)rr * kOutCols + cc;
    float* er = eps + (int64_t)(r0 + rr) * D + c0 + cc;
    if (vec_out && cc + 4 <= ncol) {
      const float4 x = *reinterpret_cast<const float4*>(xr);
      *reinterpret_cast<float4*>(er) = make_float4(ac * x.x - acs * acc[i][0], ac * x.y - acs * acc[i][1],
                                                   ac * x.z - acs * acc[i][2], ac * x.w - acs * acc[i][3]);
    } else {
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if (cc + j < ncol) er[j] = ac * xr[j] - acs * acc[i][j];
    }
  }
}

// ---------------------------------------------------------------------------
// Single-kernel form for up to 16 components (form 2): a thread-block cluster
// of CL CTAs takes a block of RB rows; CTA q of the cluster owns columns
// [q * chunk, (q + 1) * chunk) with chunk = D / CL. Each CTA stages its chunk of
// the means (before the dependency wait: the means do not change) and of the
// rows, forms the rows' partial dot products x . mu_k over its columns in
// registers (4 rows x 8 components per warp, packed fp32 pairs, 16-byte
// shared loads), and the CL partials are summed through distributed shared
// memory in rank order -- the same sums in every CTA of the cluster. Every CTA then
// takes the logits and the max-subtracted softmax of the block's rows and
// writes eps = a x - a sqrt(a) R M for its columns from the tiles it already
// holds: no second kernel, no global accumulators, nothing read twice. The
// cluster's barriers are hardware barriers; its CTAs are co-scheduled.
constexpr int kClThreads = 256;
constexpr int kClMaxK = 16;

// Per-timestep scalars are staged in shared memory where that is one load per
// thread: a short generation's call saves a round trip (T 16 at 4x8x8, 0.7 us per
// generation). A longer schedule's would not have landed when the rows do, 12 KB
// per CTA at T 1000; there a row's three scalars are fetched while the rows are
// on their way (a 1000-step generation of 4x64x64 with draws: 725 us with all of
// them staged before the means, 643 so; T 100, eight trajectories, 239 / 237).
constexpr int kClCoefT = kClThreads / 3;

template <int CL, int RB>
struct ClShape {
  static int ld(int chunk) { return chunk + 4; }  // padded row stride: the two half-warps' rows on other banks
  static size_t smem_bytes(int chunk) { return (size_t)(kClMaxK + RB) * ld(chunk) * sizeof(float); }
};

__device__ __forceinline__ void cluster_arrive_relaxed() {
  asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
}
// The address of this CTA's shared variable at `saddr` in the shared memory of
// cluster CTA `rank` (a shared::cluster address).
__device__ __forceinline__ uint32_t cluster_map(uint32_t saddr, int rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(saddr), "r"(rank));
  return r;
}
// A 4-byte store into a peer's shared memory that completes on the peer's
// mbarrier (both shared::cluster addresses): no round trip for the sender.
__device__ __forceinline__ void st_async_remote(uint32_t raddr, float v, uint32_t rbar) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];" ::"r"(raddr),
               "r"(__float_as_uint(v)), "r"(rbar)
               : "memory");
}
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }

template <int CL, int RB>
__global__ void __launch_bounds__(kClThreads, 2) k_gmm_cluster(const float* __restrict__ X, const float* __restrict__ mu,
                                                            const float* __restrict__ coef, int T,
                                                            const int32_t* __restrict__ miss_bt,
                                                            const float* __restrict__ mnorm,
                                                            const int32_t* __restrict__ n_rows_dev, int K, int64_t D,
                                                            int chunk, int max_rows, float* __restrict__ eps,
                                                            int32_t* status) {
  static_assert(RB == 8 && kClThreads == 256 && CL % 2 == 0,
                "8 warps: 2 row quads x 2 component octets x 2 column halves of the 8 x 16 block");
  extern __shared__ __align__(128) unsigned char smem_raw[];
  __shared__ __align__(8) uint64_t bar_m, bar_x, bar_p;
  __shared__ float s_all[CL][RB * kClMaxK];  // the partial dot products of every CTA, pushed by their owners
  __shared__ float s_half[2][RB * kClMaxK];  // this CTA's partials from each half of its columns
  __shared__ __align__(16) float s_rt[kClMaxK * RB];  // responsibilities [k][row]
  __shared__ float s_sa[RB], s_q[RB], s_c[RB], s_cs[RB];
  __shared__ float s_coef[3 * kClCoefT];
  __shared__ int s_bad;
  cg::cluster_group cluster = cg::this_cluster();
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int rank = (int)cluster.block_rank();
  const int ld = chunk + 4;
  const int64_t c0 = (int64_t)rank * chunk;
  float* ms = reinterpret_cast<float*>(smem_raw);  // [kClMaxK][ld], rows >= K zero
  float* xs = ms + (size_t)kClMaxK * ld;           // [RB][ld]
  // constants: ||mu_k||^2 of the component this thread takes in the softmax, and
  // one of the staged scalars
  const float mn = (tid < RB * kClMaxK && (tid & (kClMaxK - 1)) < K) ? mnorm[tid & (kClMaxK - 1)] : 0.f;
  const bool coef_staged = T <= kClCoefT;
  const float cv = coef_staged && tid < 3 * T ? coef[tid] : 0.f;
  // the means early: they do not depend on the predecessor, and how early they
  // are asked for is what the dependency wait can hide of them
  if (warp == 0) {
    if (lane == 0) {
      mbar_init(&bar_m, 1);
      mbar_init(&bar_x, 1);
      mbar_init(&bar_p, 1);
      fence_barrier_init();
      mbar_arrive_expect_tx(&bar_m, (uint32_t)chunk * sizeof(float) * (uint32_t)K);
      // every CTA of the cluster stores its RB x kClMaxK partials here
      mbar_arrive_expect_tx(&bar_p, (uint32_t)(CL * RB * kClMaxK * sizeof(float)));
      s_bad = 0;
    }
    __syncwarp();
    for (int k = lane; k < K; k += 32) bulk_g2s(ms + (size_t)k * ld, mu + (int64_t)k * D + c0, chunk * 4u, &bar_m);
  }
  for (int q = tid; q < (kClMaxK - K) * ld; q += kClThreads) ms[(size_t)K * ld + q] = 0.f;
  if (coef_staged && tid < 3 * T) s_coef[tid] = cv;
  __syncthreads();
  pdl_wait();     // the rows, their count and their timesteps come from the kernel just before
  pdl_trigger();  // the successor may now run its prologue
  const int n_rows = min(*n_rows_dev, max_rows);
  const int r0 = blockIdx.y * RB;
  const int nr = min(RB, n_rows - r0);
  if (nr <= 0) {  // the whole cluster has no rows (uniform): the means copy lands first
    if (!mbar_wait_bounded(&bar_m, 0, pa::kDrainLimit) && tid == 0) atomicCAS(status, 0, pa::kDevTimeout);
    return;
  }
  cluster_arrive_relaxed();  // this CTA runs: its peers may push into its shared memory after their wait
  // the row copies go out first: they need only the count, while each row's
  // coefficients wait for its timestep (one more trip to memory)
  if (warp == 0) {
    if (lane == 0) mbar_arrive_expect_tx(&bar_x, (uint32_t)chunk * sizeof(float) * (uint32_t)nr);
    __syncwarp();  // expect_tx precedes the copies
    for (int r = lane; r < nr; r += 32) bulk_g2s(xs + (size_t)r * ld, X + (int64_t)(r0 + r) * D + c0, chunk * 4u, &bar_x);
  }
  for (int q = tid; q < (RB - nr) * ld; q += kClThreads) xs[(size_t)nr * ld + q] = 0.f;  // rows past the count
  if (tid < nr) {
    const int i = miss_bt[2 * (r0 + tid) + 1];
    const float* cf = coef_staged ? s_coef : coef;
    const float sa = cf[i], q = cf[T + i], c = cf[2 * T + i];
    s_sa[tid] = sa;
    s_q[tid] = q;
    s_c[tid] = c;
    s_cs[tid] = c * sa;
  }
  // bounded waits; a CTA whose copies did not land keeps to the cluster's
  // barriers (its peers wait for it there) and writes NaN
  bool ok = mbar_wait_bounded(&bar_m, 0, pa::kWaitLimit);
  ok = mbar_wait_bounded(&bar_x, 0, pa::kWaitLimit) && ok;
  if (!ok) {
    if (tid == 0) atomicCAS(status, 0, pa::kDevTimeout);
    s_bad = 1;
    mbar_wait_bounded(&bar_m, 0, pa::kDrainLimit);
    mbar_wait_bounded(&bar_x, 0, pa::kDrainLimit);
  }
  __syncthreads();
  // partial dot products: warp w takes rows 4 (w & 1) .. + 3, components
  // 8 ((w >> 1) & 1) .. + 7 and half w >> 2 of the CTA's columns; lane l the
  // columns 4 l + 128 i of that half (16-byte shared loads, conflict-free),
  // accumulated in packed fp32 pairs (two columns per FMA): each loaded row
  // vector feeds 8 components and each mean vector 4 rows
  {
    const int rq = (warp & 1) * 4, ko = ((warp >> 1) & 1) * 8, half = warp >> 2;
    const int hb = ((chunk >> 2) >> 1) << 2;  // where the second half starts: a multiple of 4 columns
    const int cb = half ? hb : 0, ce = half ? chunk : hb;
    float2 a2[4][8];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int u = 0; u < 8; ++u) a2[i][u] = make_float2(0.f, 0.f);
#pragma unroll 2
    for (int c = cb + lane * 4; c < ce; c += 128) {
      float4 xv[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) xv[i] = *reinterpret_cast<const float4*>(xs + (size_t)(rq + i) * ld + c);
#pragma unroll
      for (int uh = 0; uh < 8; uh += 4) {
        float4 mv[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) mv[u] = *reinterpret_cast<const float4*>(ms + (size_t)(ko + uh + u) * ld + c);
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            float2& acc = a2[i][uh + u];
            acc = __ffma2_rn(make_float2(xv[i].x, xv[i].y), make_float2(mv[u].x, mv[u].y), acc);
            acc = __ffma2_rn(make_float2(xv[i].z, xv[i].w), make_float2(mv[u].z, mv[u].w), acc);
          }
      }
    }
    // the 32 sums (v = 8 i + u) over the 32 lanes by a halving exchange: at
    // offset o each lane keeps half of its values (the upper half if lane bit
    // o is set) and adds its partner's copy of them, so after offsets 16, 8,
    // 4, 2, 1 lane l holds value l summed over all lanes: 31 shuffles
    float a[32];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int u = 0; u < 8; ++u) a[i * 8 + u] = a2[i][u].x + a2[i][u].y;
#pragma unroll
    for (int o = 16, n = 16; o > 0; o >>= 1, n >>= 1) {
      const bool up = (lane & o) != 0;
#pragma unroll
      for (int v = 0; v < n; ++v) {
        const float send = up ? a[v] : a[v + n];
        const float keep = up ? a[v + n] : a[v];
        a[v] = keep + __shfl_xor_sync(0xffffffffu, send, o);
      }
    }
    s_half[half][(rq + (lane >> 3)) * kClMaxK + ko + (lane & 7)] = a[0];
  }
  __syncthreads();
  // this CTA's partial of (row, k) = idx: its two column halves, stored into
  // every CTA of the cluster (slot [this CTA's rank][idx] there), half of the
  // CTAs by each of the two threads that hold it, by asynchronous stores that
  // complete on the receiver's mbarrier: no round trip for the sender and no
  // cluster barrier; every CTA waits for its own barrier and then reads its
  // own shared memory only
  cluster_wait();  // every CTA of the cluster is running (its barrier initialised)
  {
    const int idx = tid & (RB * kClMaxK - 1);
    const float pv = s_half[0][idx] + s_half[1][idx];
    const uint32_t slot = smem_u32(&s_all[rank][idx]), bar = smem_u32(&bar_p);
    const int q0 = (tid >> 7) * (CL / 2);
#pragma unroll
    for (int q = 0; q < CL / 2; ++q) st_async_remote(cluster_map(slot, q0 + q), pv, cluster_map(bar, q0 + q));
  }
  if (!mbar_wait_bounded(&bar_p, 0, pa::kWaitLimit)) {  // every peer's partials have landed
    if (tid == 0) atomicCAS(status, 0, pa::kDevTimeout);
    s_bad = 1;
  }
  __syncthreads();
  // the complete dot products (the CL partials in rank order), the logits and
  // the max-subtracted softmax: thread t < 128 takes row t / 16, component
  // t % 16, so each row is a half-warp
  if (tid < RB * kClMaxK) {
    const int rr = tid >> 4, k = tid & 15;
    float dot = 0.f;
#pragma unroll
    for (int q = 0; q < CL; ++q) dot += s_all[q][tid];
    {
      const bool on = rr < nr && k < K;
      float l = -INFINITY;
      if (on) {
        const float sa = s_sa[rr];
        l = (2.f * sa * dot - sa * sa * mn) * s_q[rr];
      }
      float mx = l;
#pragma unroll
      for (int o = 8; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
      const float ex = on ? expf(l - mx) : 0.f;
      float sum = ex;
#pragma unroll
      for (int o = 8; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
      s_rt[k * RB + rr] = ex / sum;  // zero for k >= K
    }
  }
  __syncthreads();
  // eps = a x - a sqrt(a) sum_k R_k mu_k over this CTA's columns, four per thread
  const bool bad = s_bad != 0;
  for (int cq = tid * 4; cq < chunk; cq += kClThreads * 4) {
    float2 acc[RB][2];  // columns cq, cq+1 and cq+2, cq+3 of each row, packed fp32 pairs
#pragma unroll
    for (int r = 0; r < RB; ++r) acc[r][0] = acc[r][1] = make_float2(0.f, 0.f);
#pragma unroll 4
    for (int k = 0; k < K; ++k) {
      const float4 m = *reinterpret_cast<const float4*>(ms + (size_t)k * ld + cq);
      const float2 ml = make_float2(m.x, m.y), mh = make_float2(m.z, m.w);
#pragma unroll
      for (int r = 0; r < RB; r += 4) {
        const float4 v = *reinterpret_cast<const float4*>(s_rt + k * RB + r);  // responsibilities of 4 rows
        const float w4[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const float2 w2 = make_float2(w4[q], w4[q]);
          acc[r + q][0] = __ffma2_rn(w2, ml, acc[r + q][0]);
          acc[r + q][1] = __ffma2_rn(w2, mh, acc[r + q][1]);
        }
      }
    }
#pragma unroll
    for (int r = 0; r < RB; ++r) {
      if (r >= nr) break;
      const float4 x = *reinterpret_cast<const float4*>(xs + (size_t)r * ld + cq);
      const float ac = s_c[r], acs = s_cs[r];
      float4 o = make_float4(ac * x.x - acs * acc[r][0].x, ac * x.y - acs * acc[r][0].y, ac * x.z - acs * acc[r][1].x,
                             ac * x.w - acs * acc[r][1].y);
      if (bad) o = make_float4(__int_as_float(0x7fc00000), __int_as_float(0x7fc00000), __int_as_float(0x7fc00000),
                               __int_as_float(0x7fc00000));
      *reinterpret_cast<float4*>(eps + (int64_t)(r0 + r) * D + c0 + cq) = o;
    }
  }
}

}  // namespace

struct pa_gmm {
  int K, T, max_rows;
  int64_t D;
  const float* means;
  char* ws;
  GmmLayout L;
  cudaStream_t st;
  int64_t launches;
  bool per;     // the tensor-core kernels fit this device
  bool cl_ok;   // the single-kernel cluster form fits these sizes and this device
  int form;     // 0 CUDA cores, 1 tensor cores, 2 cluster form
};

namespace {
constexpr int kClSize = 16;   // CTAs per cluster (non-portable size, opted into)
constexpr int kClRows = 8;    // rows per cluster

// See the constants above. (`rows16`: the means' rows start on 16-byte boundaries.)
int default_form(const pa_gmm& g, bool rows16) {
  const double work = (double)g.K * (double)g.D * g.max_rows;
  if (g.K > kClMaxK) return g.per && (work >= (g.K > 64 ? kTcWideWork : kTcWork) || g.D > kWideD) ? 1 : 0;
  if (!g.cl_ok) return g.per && rows16 && g.K >= kTcFewMinK && work >= kTcFewWork0 ? 1 : 0;
  if (g.max_rows >= kManyRows && g.D <= kShortRow && g.D <= kShortPerRow * g.max_rows) return 0;
  return g.per && g.max_rows >= kTcFewRows && work >= kTcFewWork ? 1 : 2;
}
}  // namespace

extern "C" size_t pa_gmm_workspace_bytes(int K, int64_t D, int max_rows, int T) {
  if (K < 1 || K > kMaxK || D < 1 || max_rows < 1 || T < 1 || T > 100000) return 0;
  return gmm_layout(K, D, max_rows, T).total;
}

extern "C" pa_status pa_gmm_create(pa_gmm** out, int K, int64_t D, const float* means_dev,
                                   double std, const double* alphas_cumprod, int T,
                                   int max_rows, void* workspace_dev, size_t workspace_bytes,
                                   void* stream) {
  if (!out) { pa::set_error("pa_gmm_create: out is NULL"); return PA_ERR_ARG; }
  *out = nullptr;
  if (K < 1 || K > kMaxK) { pa::set_error("pa_gmm_create: K must be in [1, 128]"); return PA_ERR_ARG; }
  if (D < 1 || max_rows < 1 || T < 1 || T > 100000 || !means_dev || !alphas_cumprod ||
      !(std >= 0.0) || !std::isfinite(std)) {
    pa::set_error("pa_gmm_create: bad size, pointer or std");
    return PA_ERR_ARG;
  }
  for (int i = 0; i <= T; ++i) {
    const double a = alphas_cumprod[i];
    if (!(a > 0.0 && a <= 1.0)) { pa::set_error("pa_gmm_create: alphas_cumprod must be in (0, 1]"); return PA_ERR_ARG; }
  }
  GmmLayout L = gmm_layout(K, D, max_rows, T);
  if (!workspace_dev || (reinterpret_cast<uintptr_t>(workspace_dev) % pa::kAlign) != 0 ||
      workspace_bytes < L.total) {
    pa::set_error("pa_gmm_create: workspace NULL, not 256-byte aligned, or smaller than pa_gmm_workspace_bytes()");
    return PA_ERR_WORKSPACE;
  }
  pa_gmm* g = new pa_gmm{};
  g->K = K; g->T = T; g->max_rows = max_rows; g->D = D; g->means = means_dev;
  g->ws = static_cast<char*>(workspace_dev); g->L = L;
  g->st = static_cast<cudaStream_t>(stream);
  std::vector<float> coef(3 * (size_t)T);
  for (int i = 0; i < T; ++i) {
    const double a = alphas_cumprod[i];
    const double v = a * std * std + (1.0 - a);
    coef[i] = (float)std::sqrt(a);
    coef[T + i] = (float)(1.0 / (2.0 * v));
    coef[2 * T + i] = (float)(std::sqrt(1.0 - a) / v);
  }
  cudaError_t e = cudaMemcpyAsync(g->ws + L.coef, coef.data(), coef.size() * sizeof(float),
                                  cudaMemcpyHostToDevice, g->st);
  if (e == cudaSuccess) e = cudaMemsetAsync(g->ws + L.status, 0, sizeof(int32_t), g->st);
  if (e == cudaSuccess) e = cudaMemsetAsync(g->ws + L.epoch, 0, sizeof(GmmEpoch), g->st);
  if (e == cudaSuccess) e = cudaMemsetAsync(g->ws + L.gacc, 0, (size_t)2 * max_rows * K * sizeof(long long), g->st);
  if (e == cudaSuccess) {
    k_gmm_norms<<<K, 256, 0, g->st>>>(means_dev, D, reinterpret_cast<float*>(g->ws + L.mnorm),
                                      reinterpret_cast<GmmEpoch*>(g->ws + L.epoch));
    g->launches++;
    e = cudaGetLastError();
  }
  const size_t dots_smem = dots_smem_bytes(K, L.chunk);
  const size_t out_smem = (size_t)(K + kOutRows) * kOutCols * sizeof(float);
  if (e == cudaSuccess) e = pa::allow_smem(reinterpret_cast<const void*>(k_gmm_dots), dots_smem);
  if (e == cudaSuccess) e = pa::allow_smem(reinterpret_cast<const void*>(k_gmm_out), out_smem);
  int dev = 0, major = 0, optin = 0;
  if (e == cudaSuccess) e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  const bool rows16 = D % 4 == 0 && (reinterpret_cast<uintptr_t>(means_dev) & 15) == 0;
  g->per = false;
  if (e == cudaSuccess) e = pa::gmm_tc_setup(K, &g->per);
  // The single-kernel cluster form for K <= 16 when D splits into kClSize
  // 16-byte-aligned column chunks whose tiles fit in shared memory and a
  // cluster of kClSize CTAs can be resident.
  g->cl_ok = false;
  if (e == cudaSuccess && major == 10 && K <= kClMaxK && D % (4 * kClSize) == 0 && rows16) {
    const int chunk = (int)(D / kClSize);
    const size_t smem = ClShape<kClSize, kClRows>::smem_bytes(chunk);
    auto kern = k_gmm_cluster<kClSize, kClRows>;
    cudaFuncAttributes fa = {};
    e = cudaFuncGetAttributes(&fa, kern);
    if (e == cudaSuccess && smem + fa.sharedSizeBytes <= (size_t)optin) {
      e = pa::allow_smem(reinterpret_cast<const void*>(kern), smem);
      if (e == cudaSuccess) e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
      if (e == cudaSuccess) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(kClSize, 1, 1);
        cfg.blockDim = dim3(kClThreads);
        cfg.dynamicSmemBytes = smem;
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = kClSize;
        at[0].val.clusterDim.y = 1;
        at[0].val.clusterDim.z = 1;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        int nclusters = 0;
        e = cudaOccupancyMaxActiveClusters(&nclusters, kern, &cfg);
        g->cl_ok = e == cudaSuccess && nclusters > 0;
        if (e != cudaSuccess) {
          (void)cudaGetLastError();  // the size is not supported here: keep the other forms
          e = cudaSuccess;
        }
      }
    }
  }
  g->form = default_form(*g, rows16);
  if (e == cudaSuccess) e = cudaStreamSynchronize(g->st);
  if (e != cudaSuccess) {
    pa::set_error(std::string("pa_gmm_create: ") + cudaGetErrorString(e));
    delete g;
    return PA_ERR_CUDA;
  }
  *out = g;
  return PA_OK;
}

extern "C" pa_status pa_gmm_eps(pa_gmm* g, const float* batch_x_dev, const int32_t* miss_bt_dev,
                                const int32_t* n_rows_dev, float* batch_eps_dev) {
  if (!g || !batch_x_dev || !miss_bt_dev || !n_rows_dev || !batch_eps_dev) {
    pa::set_error("pa_gmm_eps: NULL argument");
    return PA_ERR_ARG;
  }
  const GmmLayout& L = g->L;
  const float* coef = reinterpret_cast<const float*>(g->ws + L.coef);
  const float* mnorm = reinterpret_cast<const float*>(g->ws + L.mnorm);
  long long* gacc2 = reinterpret_cast<long long*>(g->ws + L.gacc);
  GmmEpoch* ep = reinterpret_cast<GmmEpoch*>(g->ws + L.epoch);
  int32_t* status = reinterpret_cast<int32_t*>(g->ws + L.status);
  // bulk copies need 16-byte aligned rows: D % 4 == 0 and aligned base pointers
  const bool bulk = g->D % 4 == 0 && ((reinterpret_cast<uintptr_t>(batch_x_dev) |
                                       reinterpret_cast<uintptr_t>(g->means)) & 15) == 0;
  const bool vec_out = g->D % 4 == 0 && (reinterpret_cast<uintptr_t>(batch_eps_dev) & 15) == 0;
  const size_t out_smem = (size_t)(g->K + kOutRows) * kOutCols * sizeof(float);
  cudaError_t e;
  if (g->form == 1) {  // any D, any alignment
    const pa::GmmTcArgs a{batch_x_dev, g->means, coef, mnorm, miss_bt_dev, n_rows_dev, batch_eps_dev, g->ws + L.tc,
                          status, g->K, g->T, g->max_rows, g->D};
    e = pa::gmm_tc_launch(a, g->st);
    g->launches += pa::kGmmTcLaunches;
    if (e == cudaSuccess) e = cudaGetLastError();
    if (e != cudaSuccess) {
      pa::set_error(std::string("pa_gmm_eps: ") + cudaGetErrorString(e));
      return PA_ERR_CUDA;
    }
    return PA_OK;
  }
  if (g->form == 2 && bulk && vec_out) {  // one kernel: cluster of kClSize CTAs per kClRows rows
    const int chunk = (int)(g->D / kClSize);
    e = pa::launch_ex(k_gmm_cluster<kClSize, kClRows>, dim3(kClSize, (g->max_rows + kClRows - 1) / kClRows),
                      dim3(kClThreads), ClShape<kClSize, kClRows>::smem_bytes(chunk), g->st, kClSize,
                      batch_x_dev, g->means, coef, g->T, miss_bt_dev, mnorm, n_rows_dev, g->K, g->D, chunk,
                      g->max_rows, batch_eps_dev, status);
    g->launches += 1;
    if (e == cudaSuccess) e = cudaGetLastError();
    if (e != cudaSuccess) {
      pa::set_error(std::string("pa_gmm_eps: ") + cudaGetErrorString(e));
      return PA_ERR_CUDA;
    }
    return PA_OK;
  }
  e = pa::launch_ex(k_gmm_dots, dim3(L.nchunk, (g->max_rows + kDotRows - 1) / kDotRows), dim3(kThreads),
                    dots_smem_bytes(g->K, L.chunk), g->st, 0, batch_x_dev, g->means, n_rows_dev, g->K, g->D,
                    L.chunk, kFixedRoom / (float)L.nchunk, g->max_rows, bulk, gacc2, ep, status);
  if (e == cudaSuccess)
    e = pa::launch_ex(k_gmm_out,
                      dim3((unsigned)((g->D + kOutCols - 1) / kOutCols), (g->max_rows + kOutRows - 1) / kOutRows),
                      dim3(kThreads), out_smem, g->st, 0, batch_x_dev, g->means, (const long long*)gacc2, ep, coef,
                      g->T, miss_bt_dev, mnorm, n_rows_dev, g->K, g->D, g->max_rows, bulk, vec_out, batch_eps_dev,
                      status);
  g->launches += 2;
  if (e == cudaSuccess) e = cudaGetLastError();
  if (e != cudaSuccess) {
    pa::set_error(std::string("pa_gmm_eps: ") + cudaGetErrorString(e));
    return PA_ERR_CUDA;
  }
  return PA_OK;
}

extern "C" pa_status pa_gmm_check(pa_gmm* g) {
  if (!g) { pa::set_error("pa_gmm_check: NULL handle"); return PA_ERR_ARG; }
  int32_t st = 0;
  cudaError_t e = cudaMemcpyAsync(&st, g->ws + g->L.status, sizeof(st), cudaMemcpyDeviceToHost, g->st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(g->st);
  if (e != cudaSuccess) {
    pa::set_error(std::string("pa_gmm_check: ") + cudaGetErrorString(e));
    return PA_ERR_CUDA;
  }
  if (st == pa::kDevTimeout) { pa::set_error("pa_gmm_check: a bounded wait ran out"); return PA_ERR_TIMEOUT; }
  return PA_OK;
}

extern "C" int64_t pa_gmm_launches(const pa_gmm* g) { return g ? g->launches : -1; }

extern "C" pa_status pa_gmm_set_form(pa_gmm* g, int form) {
  if (!g) { pa::set_error("pa_gmm_set_form: NULL handle"); return PA_ERR_ARG; }
  if (form < 0 || form > 2) { pa::set_error("pa_gmm_set_form: form must be 0, 1 or 2"); return PA_ERR_ARG; }
  if (form == 1 && !g->per) {
    pa::set_error("pa_gmm_set_form: the tensor-core form needs an sm_100-family GPU and enough shared memory");
    return PA_ERR_ARG;
  }
  if (form == 2 && !g->cl_ok) {
    pa::set_error("pa_gmm_set_form: the cluster form needs K <= 16, D a multiple of 64, an sm_100-family GPU, "
                  "16-byte aligned means and enough shared memory");
    return PA_ERR_ARG;
  }
  g->form = form;
  return PA_OK;
}

extern "C" int pa_gmm_form(const pa_gmm* g) { return g ? g->form : -1; }

extern "C" void pa_gmm_destroy(pa_gmm* g) { delete g; }

// ---------------------------------------------------------------------------
// Allocation-free variant of pa_gmm_eps (no counterpart in the paper).
//
// Some callers cannot allocate device memory when they need the denoiser: a
// plugin that only receives buffers handed over by its host framework, a
// real-time loop that forbids cudaMalloc/cudaFree after start-up because an
// allocation may block, or code running where another allocator owns the
// device. pa_gmm_eps keeps its scratch (per-timestep coefficients, ||mu_k||^2,
// split-K partial dot products, responsibilities, a status word) in the
// workspace of a pa_gmm handle; pa_gmm_eps_noalloc keeps the same scratch in
// the fixed device array below and runs the same kernels on it.
constexpr size_t kNoAllocScratchBytes = (size_t)4 << 20;  // 4 MiB, held by every device that loads this library

// The fixed scratch. In host code `g_gmm_scratch` is only a stand-in name:
// its device address comes from cudaGetSymbolAddress, looked up on each call
// with the caller's device current.
static __device__ __align__(256) unsigned char g_gmm_scratch[kNoAllocScratchBytes];

namespace {

// Per-timestep scalars of the allocation-free path, formed on the device in
// fp64 from alpha-bar values that travel in the launch's own parameters (no
// host buffer, no host-to-device copy); the launch with i0 = 0 also stores the
// row count. Same expressions as pa_gmm_create's host loop, with no fused
// multiply-add, so the values round to fp32 alike.
constexpr int kNoAllocCoefChunk = 3000;  // alphas per launch: 24 KB of kernel parameters
struct AlphaChunk {
  int i0, n;
  double std;
  double a[kNoAllocCoefChunk];
};

__global__ void __launch_bounds__(256) k_noalloc_coef(AlphaChunk c, int T, int n_rows, float* __restrict__ coef,
                                                      int32_t* __restrict__ nrows_dev) {
  for (int u = threadIdx.x; u < c.n; u += blockDim.x) {
    const double a = c.a[u];
    const double v = __dadd_rn(__dmul_rn(__dmul_rn(a, c.std), c.std), 1.0 - a);
    coef[c.i0 + u] = (float)sqrt(a);
    coef[T + c.i0 + u] = (float)(1.0 / (2.0 * v));
    coef[2 * T + c.i0 + u] = (float)(sqrt(1.0 - a) / v);
  }
  if (c.i0 == 0 && threadIdx.x == 0) *nrows_dev = n_rows;
}

// Device address of g_gmm_scratch for the current device, looked up on every
// call (cheap, not a stream operation; a cached address could go stale if the
// device's context were torn down and the module reloaded elsewhere).
pa_status scratch_for_current_device(unsigned char** out) {
  void* p = nullptr;
  const cudaError_t e = cudaGetSymbolAddress(&p, g_gmm_scratch);
  if (e != cudaSuccess || !p) {
    pa::set_error(std::string("pa_gmm_eps_noalloc: cudaGetSymbolAddress: ") + cudaGetErrorString(e));
    return PA_ERR_CUDA;
  }
  *out = static_cast<unsigned char*>(p);
  return PA_OK;
}

}  // namespace

extern "C" pa_status pa_gmm_eps_noalloc(const float* means_dev, int K, int64_t D, double std,
                                        const double* alphas_cumprod, int T,
                                        const float* batch_x_dev, const int32_t* miss_bt_dev,
                                        int n_rows, float* batch_eps_dev, void* stream) {
  if (K < 1 || K > kMaxK || D < 1 || T < 1 || n_rows < 0 || !means_dev || !alphas_cumprod ||
      !batch_x_dev || !miss_bt_dev || !batch_eps_dev || !(std >= 0.0) || !std::isfinite(std)) {
    pa::set_error("pa_gmm_eps_noalloc: bad size, pointer or std");
    return PA_ERR_ARG;
  }
  for (int i = 0; i <= T; ++i) {
    const double a = alphas_cumprod[i];
    if (!(a > 0.0 && a <= 1.0)) {
      pa::set_error("pa_gmm_eps_noalloc: alphas_cumprod must be in (0, 1]");
      return PA_ERR_ARG;
    }
  }
  if (n_rows == 0) return PA_OK;
  // scratch layout: coef[3T] | mnorm[K] | gacc[2][n_rows][K] (int64) | epoch |
  //                 n_rows | status   (256-byte aligned pieces)
  const int chunk = dots_chunk(K, D, n_rows);
  const int nchunk = (int)((D + chunk - 1) / chunk);
  size_t o = 0;
  auto take = [&](size_t bytes) { size_t at = o; o = pa::align_up(o + bytes, pa::kAlign); return at; };
  const size_t o_coef = take((size_t)3 * T * sizeof(float));
  const size_t o_mnorm = take((size_t)K * sizeof(float));
  const size_t o_gacc = take((size_t)2 * n_rows * K * sizeof(long long));
  const size_t o_epoch = take(sizeof(GmmEpoch));
  const size_t o_n = take(sizeof(int32_t));
  const size_t o_status = take(sizeof(int32_t));
  if (o > kNoAllocScratchBytes) {
    pa::set_error("pa_gmm_eps_noalloc: these sizes need " + std::to_string(o) +
                  " bytes of scratch, more than the fixed 4 MiB (4194304 bytes); "
                  "use pa_gmm_create + pa_gmm_eps with a caller-allocated workspace");
    return PA_ERR_ARG;
  }
  unsigned char* scratch = nullptr;
  pa_status ps = scratch_for_current_device(&scratch);
  if (ps != PA_OK) return ps;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  float* coef = reinterpret_cast<float*>(scratch + o_coef);
  float* mnorm = reinterpret_cast<float*>(scratch + o_mnorm);
  long long* gacc2 = reinterpret_cast<long long*>(scratch + o_gacc);
  GmmEpoch* ep = reinterpret_cast<GmmEpoch*>(scratch + o_epoch);
  int32_t* nrows_dev = reinterpret_cast<int32_t*>(scratch + o_n);
  int32_t* status = reinterpret_cast<int32_t*>(scratch + o_status);

  // Per-timestep scalars and the row count: small launches whose parameters
  // carry the alphas (asynchronous, nothing on the host to outlive the call).
  cudaError_t e = cudaSuccess;
  {
    AlphaChunk c;
    c.std = std;
    for (int i0 = 0; i0 < T && e == cudaSuccess; i0 += kNoAllocCoefChunk) {
      c.i0 = i0;
      c.n = (T - i0) < kNoAllocCoefChunk ? (T - i0) : kNoAllocCoefChunk;
      for (int u = 0; u < c.n; ++u) c.a[u] = alphas_cumprod[i0 + u];
      k_noalloc_coef<<<1, 256, 0, st>>>(c, T, n_rows, coef, nrows_dev);
      e = cudaGetLastError();
    }
  }
  if (e == cudaSuccess) e = cudaMemsetAsync(status, 0, sizeof(int32_t), st);  // starts at zero every call
  if (e == cudaSuccess)  // the epoch and both accumulator sets start at zero every call too
    e = cudaMemsetAsync(ep, 0, sizeof(GmmEpoch), st);
  if (e == cudaSuccess) e = cudaMemsetAsync(gacc2, 0, (size_t)2 * n_rows * K * sizeof(long long), st);
  const size_t dots_smem = dots_smem_bytes(K, chunk);
  const size_t out_smem = (size_t)(K + kOutRows) * kOutCols * sizeof(float);
  if (e == cudaSuccess) e = pa::allow_smem(reinterpret_cast<const void*>(k_gmm_dots), dots_smem);
  if (e == cudaSuccess) e = pa::allow_smem(reinterpret_cast<const void*>(k_gmm_out), out_smem);
  if (e != cudaSuccess) {
    pa::set_error(std::string("pa_gmm_eps_noalloc: ") + cudaGetErrorString(e));
    return PA_ERR_CUDA;
  }
  const bool bulk = D % 4 == 0 && ((reinterpret_cast<uintptr_t>(batch_x_dev) |
                                    reinterpret_cast<uintptr_t>(means_dev)) & 15) == 0;
  k_gmm_norms<<<K, 256, 0, st>>>(means_dev, D, mnorm, ep);
  const bool vec_out = D % 4 == 0 && (reinterpret_cast<uintptr_t>(batch_eps_dev) & 15) == 0;
  k_gmm_dots<<<dim3(nchunk, (n_rows + kDotRows - 1) / kDotRows), kThreads, dots_smem, st>>>(
      batch_x_dev, means_dev, nrows_dev, K, D, chunk, kFixedRoom / (float)nchunk, n_rows, bulk, gacc2, ep, status);
  k_gmm_out<<<dim3((unsigned)((D + kOutCols - 1) / kOutCols), (n_rows + kOutRows - 1) / kOutRows), kThreads,
              out_smem, st>>>(batch_x_dev, means_dev, gacc2, ep, coef, T, miss_bt_dev, mnorm, nrows_dev, K, D,
                              n_rows, bulk, vec_out, batch_eps_dev, status);
  e = cudaGetLastError();
  if (e != cudaSuccess) {
    pa::set_error(std::string("pa_gmm_eps_noalloc: ") + cudaGetErrorString(e));
    return PA_ERR_CUDA;
  }
  return PA_OK;
}
