// Solver-step kernels for sm_103a: first-iteration plan, miss gather (a4),
// plain-load Picard update (a6-a9, a11) and the planning kernel that takes
// the decision after an update (a10, a2, a3) and gathers the next batch (a4).
//
// Data layout (fp32, one row = one timestep's latent of D floats):
//   X    [B][P+1][D]  state ring, state i lives in slot i mod (P+1)
//   Xhat [B][P][D]    cache inputs  xhat_i  (Eq. 3), slot i mod P
//   Ehat [B][P][D]    cache outputs ehat_i  (Eq. 3), slot i mod P
//   batch_x [B*P][D]  gathered latents of the misses, rank order
#include <type_traits>

#include "pa_decide.cuh"
#include "pa_internal.h"

namespace pa {
namespace {

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

__device__ __forceinline__ void set_status(Ctl* c, int code) {
  atomicCAS(&c->status, kDevOk, code);
}

// ---------------------------------------------------------------------------
// a4: batch_x[r] <- x_{miss[r]} for r < n_miss. A lazy state (i > e) reads
// state e, the value every new tail state was initialised to. Each thread
// moves kGatherUnroll vectors per row with all loads issued before the stores;
// 16 of them make a 4x64x64 row one CTA's work (100 planning CTAs at window
// 100: 25.9 against 26.3 us per iteration with quarter rows in 400 CTAs).
constexpr int kGatherThreads = 256;
constexpr int kGatherUnroll = 16;

// This CTA's part (blockIdx.x of gridDim.x) of a row of D values, to one
// place or two.
template <int VEC>
__device__ __forceinline__ void copy_part(int64_t D, const float* src, float* dst, float* dst2) {
  using T = typename std::conditional<VEC == 4, float4, float>::type;
  const int64_t nvec = D / VEC;
  const int64_t stride = (int64_t)gridDim.x * kGatherThreads;
  const int64_t base = (int64_t)blockIdx.x * kGatherThreads + threadIdx.x;
  const T* from = reinterpret_cast<const T*>(src);
  T* to = reinterpret_cast<T*>(dst);
  T* to2 = reinterpret_cast<T*>(dst2);
  for (int64_t v0 = base; v0 < nvec; v0 += stride * kGatherUnroll) {
    T buf[kGatherUnroll];
#pragma unroll
    for (int u = 0; u < kGatherUnroll; ++u) {
      const int64_t v = v0 + u * stride;
      if (v < nvec) buf[u] = __ldg(from + v);
    }
#pragma unroll
    for (int u = 0; u < kGatherUnroll; ++u) {
      const int64_t v = v0 + u * stride;
      if (v < nvec) {
        to[v] = buf[u];
        if (to2) to2[v] = buf[u];
      }
    }
  }
}

template <int VEC>
__device__ __forceinline__ void copy_row(const Dev& d, int b, int src_state, int r) {
  copy_part<VEC>(d.D, d.X + ((int64_t)b * (d.P + 1) + src_state % (d.P + 1)) * d.D, d.batch_x + (int64_t)r * d.D, nullptr);
}

// The sums of iteration par's decision (divided by D) for the host, and the
// accumulator set that the next iteration adds into cleared: CTA `cta` of `ctas`
// of kGatherThreads threads.
__device__ __forceinline__ void report_sums(const Dev& d, int par, int64_t cta = 0, int64_t ctas = 1) {
  const int npair = d.B * d.P;
  for (int64_t q = cta * kGatherThreads + threadIdx.x; q < npair; q += ctas * kGatherThreads) {
    const double* e = d.acc + ((size_t)(par * 2 + 0) * npair + q) * kAccStride;
    const double* dl = d.acc + ((size_t)(par * 2 + 1) * npair + q) * kAccStride;
    d.red_err[q] = (float)(__ldcg(e) * d.inv_d);
    d.red_del[q] = (float)(__ldcg(dl) * d.inv_d);
    d.acc[((size_t)((par ^ 1) * 2 + 0) * npair + q) * kAccStride] = 0.0;
    d.acc[((size_t)((par ^ 1) * 2 + 1) * npair + q) * kAccStride] = 0.0;
  }
}

// The gather of a plan already in memory (copy par), after the one-CTA planner.
// Its CTAs also report the sums that the plan was made from (set par ^ 1,
// divided by D) and clear the set that the planned iteration adds into: the
// divisions by D are fp64, which one SM of this GPU does two per clock of.
template <int VEC>
__global__ void __launch_bounds__(kGatherThreads) k_gather(Dev d, int par) {
  pdl_wait();  // everything read here comes from the kernel that planned
  pdl_trigger();  // the successor may now run its prologue
  report_sums(d, par ^ 1, (int64_t)blockIdx.y * gridDim.x + blockIdx.x, (int64_t)gridDim.x * gridDim.y);
  const int n = d.ctl->n_miss;
  const Traj* tr = d.traj + par * d.B;
  for (int r = blockIdx.y; r < n; r += gridDim.y) {
    const int b = d.miss_bt[2 * r], i = d.miss_bt[2 * r + 1];
    copy_row<VEC>(d, b, min(i, tr[b].e), r);
  }
}

// ---------------------------------------------------------------------------
// First iteration. x: x_init in device memory, which this kernel also copies
// into state 0; NULL: a copy has put it there. Every timestep of every first window enters for the first time, hence is a miss
// (Sec. 2.2); states 1..p are lazy copies of state 0 = x_init, so the frontier
// e starts at 0 and batch row r = b p0 + j is state 0 of trajectory b. One
// launch on the planning kernel's grid: each CTA copies its part of its batch
// rows; all
// CTAs together write the ranks and the miss list and clear both sets of the
// reduction accumulators (the entries that are added into, every
// kAccStride-th) and the fused step's barrier counter; CTA (0, 0) writes the
// trajectories, counters and the plan's counter copy 0.
template <int VEC>
__global__ void __launch_bounds__(kGatherThreads) k_init(Dev d, const float* __restrict__ x) {
  pdl_wait();  // the kernels and copies before are complete
  pdl_trigger();
  const int p0 = min(d.P, d.T);
  const int npair = d.B * d.P;
  const int64_t cta = (int64_t)blockIdx.y * gridDim.x + blockIdx.x;
  const int64_t step = (int64_t)gridDim.x * gridDim.y * kGatherThreads;
  for (int64_t q = cta * kGatherThreads + threadIdx.x; q < npair; q += step) {
    const int b = (int)(q / d.P), j = (int)(q % d.P);
    if (j < p0) {
      const int r = b * p0 + j;
      d.rank[q] = r;
      d.miss_bt[2 * r] = b;
      d.miss_bt[2 * r + 1] = j;
    } else {
      d.rank[q] = -1;
    }
  }
  for (int64_t q = cta * kGatherThreads + threadIdx.x; q < 4 * (int64_t)npair; q += step) {
    d.acc[q * kAccStride] = 0.0;  // [set][err, dist][B][P]
    if (d.taa) d.taa_acc[q * kAccStride] = 0.0;
  }
  if (cta == 0) {
    for (int b = threadIdx.x; b < d.B; b += blockDim.x) {
      Traj tr{};
      tr.t = 0; tr.p = p0; tr.e = 0; tr.done = 0; tr.m = p0; tr.h1 = 0;  // no entries yet: ne = nh = 0
      d.traj[b] = tr;  // copy 0: the plan of iteration 0
      if (d.adapt) d.tau[b] = d.cache_thresh;  // tau_cache starts at the configured value
    }
    if (threadIdx.x == 0) {
      *d.gbar = 0ull;
      Ctl c{};
      c.n_miss = d.B * p0;
      c.n_active = d.B;
      c.iter = 0;
      c.status = kDevOk;
      c.nfe = (long long)d.B * p0;
      c.hits = 0;
      *d.ctl = c;
      PlanCtr pc;
      pc.n_active = c.n_active;
      pc.iter = 0;
      pc.nfe = c.nfe;
      pc.hits = 0;
      d.pc[0] = pc;
    }
  }
  for (int r = blockIdx.y; r < d.B * p0; r += gridDim.y) {
    const int b = r / p0;
    float* state0 = d.X + (int64_t)b * (d.P + 1) * d.D;
    copy_part<VEC>(d.D, x ? x + (int64_t)b * d.D : state0, d.batch_x + (int64_t)r * d.D,
                   x && r == b * p0 ? state0 : nullptr);
  }
}

// The poll of a generation whose x_T goes to device memory, in one launch in
// place of two copies (the copy engine takes about 4 us for each, mostly
// between them): the states in the slot of t = T to out [B][D], the counters to
// pinned host memory.
template <int VEC>
__global__ void __launch_bounds__(kGatherThreads) k_poll(Dev d, float* __restrict__ out, Ctl* host) {
  pdl_wait();  // the counters and states come from the kernels before
  pdl_trigger();
  const int b = blockIdx.y;
  if (blockIdx.x == 0 && b == 0 && threadIdx.x == 0) {
    *host = *d.ctl;
    __threadfence_system();
  }
  copy_part<VEC>(d.D, d.X + ((int64_t)b * (d.P + 1) + d.T % (d.P + 1)) * d.D, out + (int64_t)b * d.D, nullptr);
}

// ---------------------------------------------------------------------------
// Plain-load Picard update. One CTA = one column chunk of one trajectory;
// each thread owns VEC adjacent columns and walks the window sequentially,
// which makes the window-axis prefix sum (Eq. 1) a register recurrence.
// Per window position j (timestep i = t + j):
//   eps_i  = batch_eps[rank] (miss) or ehat_i (hit)              Eq. 6
//   miss:  ehat_i <- eps_i, xhat_i <- x_i                         Eq. 7
//   d_i    = (c_i - 1) x_i + e_i eps_i (+ sigma_i z_i)            drift
//   x'_{i+1} = x_t + sum_{l<=j} d_{t+l}  (compensated)            Eq. 1
//   err_j  partial of sum (x'_{i+1} - x_{i+1})^2                  Eq. 2
//   del_j  partial of sum |x'_{i+1} - xhat_{i+1}| (next iteration) Eq. 4
// Partials are reduced per CTA in a fixed order and added into the
// iteration's fp64 accumulators (red_add); the planning kernel reads the sums.
template <int VEC>
struct V;
template <>
struct V<1> {
  float a[1];
};
template <>
struct V<4> {
  float a[4];
};

template <int VEC>
__device__ __forceinline__ V<VEC> ldv(const float* p) {
  V<VEC> r;
  if constexpr (VEC == 4) {
    float4 q = *reinterpret_cast<const float4*>(p);
    r.a[0] = q.x; r.a[1] = q.y; r.a[2] = q.z; r.a[3] = q.w;
  } else {
    r.a[0] = *p;
  }
  return r;
}

template <int VEC>
__device__ __forceinline__ void stv(float* p, const V<VEC>& v) {
  if constexpr (VEC == 4) {
    *reinterpret_cast<float4*>(p) = make_float4(v.a[0], v.a[1], v.a[2], v.a[3]);
  } else {
    *p = v.a[0];
  }
}

// A cache entry row (xhat or ehat) at element offset `off`: fp32, or bfloat16 when CB.
template <int VEC, bool CB>
__device__ __forceinline__ V<VEC> ld_entry(const float* base, int64_t off) {
  if constexpr (CB) {
    V<VEC> r;
    Bf16Row<VEC>::load(reinterpret_cast<const uint16_t*>(base) + off, r.a);
    return r;
  } else {
    return ldv<VEC>(base + off);
  }
}
template <int VEC, bool CB>
__device__ __forceinline__ void st_entry(float* base, int64_t off, const V<VEC>& v) {
  if constexpr (CB) {
    Bf16Row<VEC>::store(reinterpret_cast<uint16_t*>(base) + off, v.a);
  } else {
    stv<VEC>(base + off, v);
  }
}
template <int VEC, bool CB>
__device__ __forceinline__ V<VEC> as_entry(const V<VEC>& v) {
  if constexpr (CB) {
    V<VEC> r;
#pragma unroll
    for (int k = 0; k < VEC; ++k) r.a[k] = __bfloat162float(__float2bfloat16_rn(v.a[k]));
    return r;
  } else {
    return v;
  }
}

constexpr int kPlainThreads = 128;

template <int VEC, bool CB>
__global__ void __launch_bounds__(kPlainThreads) k_update_plain(Dev d, const float* __restrict__ beps, int par) {
  extern __shared__ float red[];  // [2][nwarps][P]
  const int b = blockIdx.y;
  pdl_wait();
  pdl_trigger();  // the successor may now run its prologue
  const Traj tr = d.traj[par * d.B + b];
  if (tr.p == 0) return;
  const int t = tr.t, p = tr.p, e = tr.e, P = d.P;
  const int64_t D = d.D;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  constexpr int nw = kPlainThreads / 32;
  const int64_t col = ((int64_t)blockIdx.x * kPlainThreads + threadIdx.x) * VEC;
  const bool live = col < D;
  float* Xb = d.X + (int64_t)b * (P + 1) * D + col;
  const int64_t cbase = (int64_t)b * P * D + col;  // element offset of this column in the cache rows
  const int32_t* rk = d.rank + b * P;
  const int n_miss = d.ctl->n_miss;

  V<VEC> xcur{}, acc{}, comp{}, xfill{};
  if (live) xcur = ldv<VEC>(Xb + (int64_t)(t % (P + 1)) * D);
  acc = xcur;
  xfill = xcur;  // state e when e == t
  for (int j = 0; j < p; ++j) {
    const int i = t + j;
    const int r = rk[j];
    if (r >= n_miss) set_status(d.ctl, kDevBadRank);
    const float cm1 = d.cm1[i], ec = d.ecoef[i];
    const float sg = d.noise ? d.sigma[i] : 0.f;
    const int slot = i % P;
    float ev = 0.f, dv = 0.f;
    if (live) {
      V<VEC> eps = (r >= 0) ? ldv<VEC>(beps + (int64_t)r * D + col)
                            : ld_entry<VEC, CB>(d.Ehat, cbase + (int64_t)slot * D);
      if (r >= 0) {
        st_entry<VEC, CB>(d.Ehat, cbase + (int64_t)slot * D, eps);
        st_entry<VEC, CB>(d.Xhat, cbase + (int64_t)slot * D, xcur);
      }
      V<VEC> xo;
      if (i + 1 <= e) {
        xo = ldv<VEC>(Xb + (int64_t)((i + 1) % (P + 1)) * D);
        if (i + 1 == e) xfill = xo;
      } else {
        xo = xfill;
      }
      V<VEC> zn{};
      if (d.noise) zn = ldv<VEC>(d.noise + ((int64_t)b * d.T + i) * D + col);  // the draw z_i
      V<VEC> xn;
#pragma unroll
      for (int v = 0; v < VEC; ++v) {
        const float dr = fmaf(sg, zn.a[v], cm1 * xcur.a[v] + ec * eps.a[v]);
        const float y = dr - comp.a[v];
        const float s = acc.a[v] + y;
        comp.a[v] = (s - acc.a[v]) - y;
        acc.a[v] = s;
        xn.a[v] = s;
        const float df = xn.a[v] - xo.a[v];
        ev += df * df;
      }
      stv<VEC>(Xb + (int64_t)((i + 1) % (P + 1)) * D, xn);
      if (j + 1 < p) {
        const int r1 = rk[j + 1];
        V<VEC> xh = (r1 >= 0) ? as_entry<VEC, CB>(xo) : ld_entry<VEC, CB>(d.Xhat, cbase + (int64_t)((i + 1) % P) * D);
#pragma unroll
        for (int v = 0; v < VEC; ++v) dv += fabsf(xn.a[v] - xh.a[v]);
      }
      xcur = xo;
    }
    ev = warp_sum(ev);
    dv = warp_sum(dv);
    if (lane == 0) {
      red[warp * P + j] = ev;
      red[(nw + warp) * P + j] = dv;
    }
  }
  __syncthreads();
  for (int j = threadIdx.x; j < p; j += kPlainThreads) {
    float se = 0.f, sd = 0.f;
#pragma unroll
    for (int w = 0; w < nw; ++w) {
      se += red[w * P + j];
      sd += red[(nw + w) * P + j];
    }
    red_add(d, par, 0, b * P + j, se);
    red_add(d, par, 1, b * P + j, sd);
  }
}

// ---------------------------------------------------------------------------
// Planning kernel (a10, a2, a3 after iteration k, then a4 of iteration k+1),
// one launch. The update kernel left complete fp64 sums of the Eq. 2 errors
// and Eq. 4 distances; every CTA reads them (B*P of each), compares them with tol
// D and tau_cache D (by their bits) and takes the whole decision in shared
// memory -- the same inputs and the same arithmetic give the same plan in every
// CTA -- then copies the column range blockIdx.x of batch rows blockIdx.y, blockIdx.y + gridDim.y, ... that hold
// a miss (one row per CTA unless the rows outnumber one wave of CTAs). A CTA of
// the last row also publishes the plan (copy par ^ 1 of the trajectories and
// counters, ranks, miss list, iteration log), one of the row before reports the
// reductions for the host and clears the accumulator set of iteration k+1: they
// seldom have a row to copy. Nobody waits for anybody: the other
// CTAs read copy par of the plan, which no CTA writes in this launch.
constexpr int kPlanThreads = 256;
static_assert(kPlanThreads == kGatherThreads, "report_sums");
constexpr int kPlanPerSm = 2;   // planning CTAs per SM (three: the launch bound makes the decision spill, slower)
constexpr int kFusedMaxPairs = 1024;  // B*P planned in every CTA at most; beyond, one CTA plans
// Beyond this many pairs one CTA plans and a separate gather follows unless
// tau_cache adapts (only the every-CTA planner forms the next tau). A generation
// with every CTA planning against one: windows of 100 at 4x64x64 with 500, 600,
// 800 and 1000 pairs 343 / 360, 401 / 413, 515 / 520 and 640 / 636 us, windows of
// 32 at 4x32x32 with 640 pairs 239 / 257.
constexpr int kFusedPreferPairs = 900;
static_assert(kFusedMaxPairs <= 32 * 32, "one miss mask per 32-position chunk, a lane each");

// The decision's inputs as bits in shared memory (one-CTA planner).
struct RedBits {
  const unsigned* conv_w;
  const unsigned* near_w;
  __device__ bool conv(int q) const { return (conv_w[q >> 5] >> (q & 31)) & 1u; }
  __device__ bool near(int q) const { return (near_w[q >> 5] >> (q & 31)) & 1u; }
};

// Division of positions q < 2^16 by P: ceil(2^32 / P) is formed before the
// dependency wait, each quotient is then one multiplication.
struct Div {
  uint32_t m;
  __device__ explicit Div(int P) : m(P == 1 ? 0u : 0xffffffffu / (uint32_t)P + 1u) {}
  __device__ int operator()(int q) const { return m ? (int)__umulhi((uint32_t)q, m) : q; }
};

// The decision over the grid: every CTA takes it whole, with all of its warps,
// from the bits that stage_decision_bits left (the rules are decide_par's, which
// takes it with one warp):
//  1. every warp advances all trajectories, lane b the b-th and (b + 32)-th:
//     a barrier less than one warp doing it for the others;
//  2. warp w forms the miss bits of the next windows' 32-position chunks w,
//     w + 8, ..., a trajectory's window by one shuffle of a packed word;
//  3. after one barrier every warp scans the chunks' miss counts (lane c: chunk
//     c), so ranks and rows need no further one.
// One warp walking the chunks took about 250 cycles for each.
struct GridPlan {
  unsigned mm;   // lane c: miss bits of chunk c
  int base;      // lane c: misses before chunk c
  int total;
};

__device__ __forceinline__ GridPlan decide_grid(const Dev& d, DecideShared& sh, Div div) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int B = d.B, P = d.P, T = d.T, N = B * P, nchunk = (N + 31) / 32;
  uint32_t packed[2] = {0u, 0u};
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    const int b = lane + 32 * k;
    if (b < B) {
      const int t = sh.t[b], p = sh.p[b];
      int stride = 0;
      if (p > 0) {
        int lead = 0;
        while (lead < p) {
          const unsigned w = bits32(sh.conv, b * P + lead);
          const int ones = w == 0xffffffffu ? 32 : __ffs(~w) - 1;
          lead += ones;
          if (ones < 32) break;
        }
        stride = min(p, 1 + min(lead, p));
      }
      const int tn = t + stride, pn = p > 0 ? min(P, T - tn) : 0, nh = p > 0 ? p - stride : 0;
      // window size (11 bits), positions with an entry (10), stride - 1 (10); B * P <= 1024
      packed[k] = (uint32_t)pn | (uint32_t)nh << 11 | (uint32_t)max(stride - 1, 0) << 21;
      if (warp == 0) {
        sh.tn[b] = tn;
        sh.pn[b] = pn;
        sh.en[b] = p > 0 ? t + p : sh.e[b];
        sh.stride[b] = stride;
        sh.nh[b] = nh;
        if (d.adapt) adapt_tau(d, sh, b, p, stride);
      }
    }
  }
  if (d.adapt) __syncthreads();  // the next hit test's bounds
  for (int c = warp; c < nchunk; c += kPlanThreads / 32) {
    const int q = c * 32 + lane;
    const int b = min(div(q), B - 1), jn = q - b * P;
    const uint32_t lo = __shfl_sync(0xffffffffu, packed[0], b & 31), hi = __shfl_sync(0xffffffffu, packed[1], b & 31);
    const uint32_t w = b < 32 ? lo : hi;
    const int pn = w & 0x7ff, nh = (w >> 11) & 0x3ff, back = w >> 21;  // stride - 1
    const bool win = q < N && jn < pn;
    bool hit = false;
    if (win && jn < nh) {
      const int qo = q + back;
      hit = d.adapt ? sum_lt(sh.del[qo], sh.thr[b]) : ((sh.near[qo >> 5] >> (qo & 31)) & 1u);
    }
    const unsigned wm = __ballot_sync(0xffffffffu, win), mm = __ballot_sync(0xffffffffu, win && !hit);
    if (lane == 0) {
      sh.cwin[c] = wm;
      sh.cmiss[c] = mm;
    }
  }
  __syncthreads();
  GridPlan g;
  g.mm = lane < nchunk ? sh.cmiss[lane] : 0u;
  const int cnt = __popc(g.mm);
  int incl = cnt;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int v = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += v;
  }
  g.base = incl - cnt;
  g.total = __shfl_sync(0xffffffffu, incl, 31);
  return g;
}

// The plan to memory, by one CTA: ranks and miss list (trajectory-major,
// ascending t), trajectories, counters and iteration log of the next iteration.
__device__ __forceinline__ void publish_plan(const Dev& d, DecideShared& sh, const GridPlan& g, int par, Div div) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int B = d.B, P = d.P, N = B * P, nchunk = (N + 31) / 32;
  for (int c = warp; c < nchunk; c += kPlanThreads / 32) {
    const int q = c * 32 + lane;
    const unsigned mm = __shfl_sync(0xffffffffu, g.mm, c);
    const int r = __shfl_sync(0xffffffffu, g.base, c) + __popc(mm & ((1u << lane) - 1u));
    if (q >= N) continue;
    if ((mm >> lane) & 1u) {
      const int b = div(q);
      d.rank[q] = r;
      d.miss_bt[2 * r] = b;
      d.miss_bt[2 * r + 1] = sh.tn[b] + (q - b * P);
    } else {
      d.rank[q] = -1;
    }
  }
  const int win = __reduce_add_sync(0xffffffffu, lane < nchunk ? __popc(sh.cwin[lane]) : 0);
  if (tid == 0) {
    int act = 0;
    for (int b = 0; b < B; ++b) act += (sh.pn[b] > 0);
    PlanCtr c;
    c.n_active = act;
    c.iter = sh.iter + 1;
    c.nfe = sh.nfe + g.total;
    c.hits = sh.hits + (win - g.total);
    d.pc[par ^ 1] = c;
    d.ctl->n_miss = g.total;
    d.ctl->n_active = act;
    d.ctl->iter = c.iter;
    d.ctl->nfe = c.nfe;
    d.ctl->hits = c.hits;
  }
  for (int b = tid; b < B; b += kPlanThreads) {
    publish_traj(d, sh, b, par);
    log_traj(d, sh, b);
  }
}

// The miss of batch row r < g.total: chunk c holds ranks base .. base +
// popc(mm) - 1, in bit order. Every lane of a warp calls it and gets the same
// answer; false if no chunk holds row r (never expected).
__device__ __forceinline__ bool row_miss(const DecideShared& ds, const GridPlan& g, int N, int P, Div div, int r,
                                         int* b, int* i) {
  const int lane = threadIdx.x & 31;
  const unsigned held = __ballot_sync(0xffffffffu, r >= g.base && r < g.base + __popc(g.mm));
  if (held == 0u) return false;
  const int c = __ffs(held) - 1;
  const unsigned m = __shfl_sync(0xffffffffu, g.mm, c);
  const int n = r - __shfl_sync(0xffffffffu, g.base, c);  // row r is the n-th miss of chunk c
  const unsigned at = __ballot_sync(0xffffffffu, ((m >> lane) & 1u) && __popc(m & ((1u << lane) - 1u)) == n);
  if (at == 0u) return false;
  const int q = c * 32 + __ffs(at) - 1;
  if (q >= N) return false;
  *b = div(q);
  *i = ds.tn[*b] + (q - *b * P);
  return true;
}

// COND: the planning kernel of the last iteration in a captured generation
// loop's body, which also sets the condition of the loop's node (set_plan_cond;
// in every iteration, or only as code not run, it cost each 0.5 us: the call
// makes the decision spill): go on while a trajectory is active, the
// device status is clean and fewer than lc.limit iterations have run (the
// window advances at least one step in each, so T of them always suffice, and
// the limit bounds the loop whatever the counters say).

template <int VEC, bool COND>
__global__ void __launch_bounds__(kPlanThreads, kPlanPerSm) k_plan_gather(Dev d, int par, LoopCond lc) {
  __shared__ DecideShared ds;
  // the last batch rows hold a miss only when everything misses: their CTAs
  // publish the plan and report the sums
  const bool publish = blockIdx.x == 0 && blockIdx.y == gridDim.y - 1;
  const bool report = blockIdx.x == gridDim.x - 1 && (int)blockIdx.y == max((int)gridDim.y - 2, 0);
  decide_load<kPlanThreads>(d, ds, par);
  const Div div(d.P);
  pdl_wait();  // the sums and the new states come from the update kernel
  pdl_trigger();  // the successor may now run its prologue
  stage_decision_bits(d, ds, par, -1, 1);
  __syncthreads();  // the decision's input bits and decide_load's state are staged
  const bool active = ds.active != 0;
  GridPlan g{0u, 0, 0};
  if (active) {
    g = decide_grid(d, ds, div);
    if (publish) publish_plan(d, ds, g, par, div);
  } else if (publish && threadIdx.x < 32) {
    carry_plan(d, par);
  }
  if constexpr (COND) {
    if (publish && threadIdx.x == 0) {
      int act = 0;
      if (active)
        for (int b = 0; b < d.B; ++b) act += ds.pn[b] > 0;
      const bool more = act > 0 && __ldcg(&d.ctl->status) == kDevOk && ds.iter + 1 < lc.limit;
      cudaGraphSetConditional(lc.handle, more ? 1u : 0u);
    }
  }
  for (int r = blockIdx.y; r < g.total; r += gridDim.y) {
    int b = 0, i = 0;
    if (!row_miss(ds, g, d.B * d.P, d.P, div, r, &b, &i)) {
      if (threadIdx.x == 0) set_status(d.ctl, kDevBadRank);
      continue;
    }
    copy_row<VEC>(d, b, min(i, ds.en[b]), r);
  }
  if (report) report_sums(d, par);
}

// One-CTA planner for B*P beyond kFusedPreferPairs (without adaptation) or
// kFusedMaxPairs; a separate gather follows. The sums are read once, all loads
// of a thread in flight together, and kept as the bits the decision needs: it
// looks at each position several times, and a trip to memory every time (1,600
// pairs) took 15 us a launch.
constexpr int kPlanOneThreads = 1024;
constexpr int kPlanOneWords = kMaxBatch * kMaxWindow / 32;

__global__ void __launch_bounds__(kPlanOneThreads) k_plan_one(Dev d, int par) {
  __shared__ DecideShared ds;
  __shared__ unsigned s_conv[kPlanOneWords], s_near[kPlanOneWords];
  const int npair = d.B * d.P, lane = threadIdx.x & 31;
  decide_load<kPlanOneThreads>(d, ds, par);
  pdl_wait();  // the sums come from the update kernel
  pdl_trigger();  // the successor may now run its prologue
  const double* acc_e = d.acc + (size_t)(par * 2 + 0) * npair * kAccStride;
  const double* acc_d = d.acc + (size_t)(par * 2 + 1) * npair * kAccStride;
  constexpr int kAhead = 4;
  for (int q0 = threadIdx.x; q0 - lane < npair; q0 += kAhead * kPlanOneThreads) {
    double e[kAhead], dl[kAhead];
#pragma unroll
    for (int u = 0; u < kAhead; ++u) {
      const int q = q0 + u * kPlanOneThreads;
      e[u] = dl[u] = 0.0;
      if (q < npair) {
        e[u] = __ldcg(acc_e + (size_t)q * kAccStride);
        dl[u] = __ldcg(acc_d + (size_t)q * kAccStride);
      }
    }
#pragma unroll
    for (int u = 0; u < kAhead; ++u) {
      const int q = q0 + u * kPlanOneThreads;
      const unsigned cm = __ballot_sync(0xffffffffu, q < npair && sum_le(e[u], d.tol_d));
      const unsigned nm = __ballot_sync(0xffffffffu, q < npair && sum_lt(dl[u], d.thr_d));
      if (lane == 0 && q < npair) {
        s_conv[q >> 5] = cm;
        s_near[q >> 5] = nm;
      }
    }
  }
  decide_run<kPlanOneThreads>(d, ds, RedBits{s_conv, s_near}, par, true);  // starts with a barrier
}

}  // namespace

namespace {
// No work: waits for its predecessor and lets its successor start, like the
// library's other kernels (programmatic dependent launch).
__global__ void k_gap() {
  pdl_wait();
  pdl_trigger();
}
}  // namespace

cudaError_t launch_gap(cudaStream_t st) { return launch_ex(k_gap, dim3(1), dim3(32), 0, st, 0); }

namespace {
dim3 gather_grid(const Dev& d) {
  const int rows = min(d.B * d.P, 65535);
  const int vec = (d.D % 4 == 0) ? 4 : 1;
  const int64_t nvec = d.D / vec;
  const int64_t want = (nvec + kGatherThreads * kGatherUnroll - 1) / (kGatherThreads * kGatherUnroll);
  return dim3((int)(want < 64 ? want : 64), rows);
}
}  // namespace

cudaError_t launch_gather(const Dev& d, int par, cudaStream_t st) {
  const dim3 g = gather_grid(d);
  if (d.D % 4 == 0) return launch_ex(k_gather<4>, g, dim3(kGatherThreads), 0, st, 0, d, par);
  return launch_ex(k_gather<1>, g, dim3(kGatherThreads), 0, st, 0, d, par);
}

namespace {
// The grid of a kernel whose CTA (x, y) copies part x of batch row y: as many
// parts per row as keep the grid within per_sm CTAs per SM (one wave), each
// part at least 1024 float4 columns; with more rows than one wave holds, one
// wave of whole-row CTAs, CTA y taking rows y, y + gridDim.y, ... An error
// only if the SM count cannot be read.
cudaError_t split_grid(const Dev& d, int per_sm, dim3* out) {
  static int nsm[64] = {};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev >= 0 && dev < 64 && nsm[dev] == 0) {
    e = cudaDeviceGetAttribute(&nsm[dev], cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
  }
  const int sms = (dev >= 0 && dev < 64 && nsm[dev] > 0) ? nsm[dev] : 148;
  dim3 g = gather_grid(d);
  const int64_t nvec = d.D / ((d.D % 4 == 0) ? 4 : 1);
  const int64_t cap = (nvec + kGatherThreads * 4 - 1) / (kGatherThreads * 4);
  int64_t gx = (int64_t)per_sm * sms / (int)g.y;
  if (gx > cap) gx = cap;
  if (gx > 64) gx = 64;
  g.x = gx < 1 ? 1 : (unsigned)gx;
  // more rows than one wave of CTAs: one wave, each CTA taking every
  // gridDim.y-th row (the planning kernel then plans once per CTA, not per row)
  if ((int64_t)g.y > (int64_t)per_sm * sms) g.y = (unsigned)(per_sm * sms);
  *out = g;
  return cudaSuccess;
}
}  // namespace

cudaError_t launch_init(const Dev& d, const float* x, cudaStream_t st) {
  dim3 g;
  const cudaError_t e = split_grid(d, kPlanPerSm, &g);
  if (e != cudaSuccess) return e;
  if (d.D % 4 == 0 && (reinterpret_cast<uintptr_t>(x) & 15) == 0)
    return launch_ex(k_init<4>, g, dim3(kGatherThreads), 0, st, 0, d, x);
  return launch_ex(k_init<1>, g, dim3(kGatherThreads), 0, st, 0, d, x);
}

cudaError_t launch_poll(const Dev& d, float* out, Ctl* host, cudaStream_t st) {
  const bool vec = d.D % 4 == 0 && (reinterpret_cast<uintptr_t>(out) & 15) == 0;
  const int64_t nvec = d.D / (vec ? 4 : 1), want = (nvec + kGatherThreads * 4 - 1) / (kGatherThreads * 4);
  const dim3 g((int)(want < 64 ? want : 64), d.B);
  if (vec) return launch_ex(k_poll<4>, g, dim3(kGatherThreads), 0, st, 0, d, out, host);
  return launch_ex(k_poll<1>, g, dim3(kGatherThreads), 0, st, 0, d, out, host);
}

cudaError_t set_plan_cond(cudaGraphNode_t node, const Dev& d, int par, LoopCond lc) {
  cudaKernelNodeParams kp = {};
  const cudaError_t e = cudaGraphKernelNodeGetParams(node, &kp);
  if (e != cudaSuccess) return e;
  Dev dev = d;
  void* args[] = {&dev, &par, &lc};
  kp.func = d.D % 4 == 0 ? reinterpret_cast<void*>(k_plan_gather<4, true>) : reinterpret_cast<void*>(k_plan_gather<1, true>);
  kp.kernelParams = args;
  kp.extra = nullptr;
  return cudaGraphKernelNodeSetParams(node, &kp);
}

cudaError_t launch_plan(const Dev& d, int par, cudaStream_t st, int* launches) {
  const LoopCond lc{};
  const int npair = d.B * d.P;
  if (npair <= kFusedPreferPairs || (d.adapt && npair <= kFusedMaxPairs)) {
    *launches = 1;
    // every CTA plans and copies a part of its batch row
    dim3 g;
    const cudaError_t e = split_grid(d, kPlanPerSm, &g);
    if (e != cudaSuccess) return e;
    if (d.D % 4 == 0) return launch_ex(k_plan_gather<4, false>, g, dim3(kPlanThreads), 0, st, 0, d, par, lc);
    return launch_ex(k_plan_gather<1, false>, g, dim3(kPlanThreads), 0, st, 0, d, par, lc);
  }
  *launches = 2;
  cudaError_t e = launch_ex(k_plan_one, dim3(1), dim3(kPlanOneThreads), 0, st, 0, d, par);
  if (e != cudaSuccess) return e;
  return launch_gather(d, par ^ 1, st);
}

cudaError_t launch_update_plain(const Dev& d, const float* batch_eps, int par, cudaStream_t st) {
  const size_t smem = (size_t)2 * (kPlainThreads / 32) * d.P * sizeof(float);
  // float4 rows need every row base 16-byte aligned: D % 4 == 0 and aligned
  // eps (and draws) pointers; the workspace arrays are 256-byte aligned
  const bool aligned = (reinterpret_cast<uintptr_t>(batch_eps) & 15) == 0 &&
                       (reinterpret_cast<uintptr_t>(d.noise) & 15) == 0;
  if (d.D % 4 == 0 && aligned) {
    const int nchunk = (int)((d.D + kPlainThreads * 4 - 1) / (kPlainThreads * 4));
    if (d.cache_bf16)
      return launch_ex(k_update_plain<4, true>, dim3(nchunk, d.B), dim3(kPlainThreads), smem, st, 0, d, batch_eps, par);
    return launch_ex(k_update_plain<4, false>, dim3(nchunk, d.B), dim3(kPlainThreads), smem, st, 0, d, batch_eps, par);
  }
  const int nchunk = (int)((d.D + kPlainThreads - 1) / kPlainThreads);
  if (d.cache_bf16)
    return launch_ex(k_update_plain<1, true>, dim3(nchunk, d.B), dim3(kPlainThreads), smem, st, 0, d, batch_eps, par);
  return launch_ex(k_update_plain<1, false>, dim3(nchunk, d.B), dim3(kPlainThreads), smem, st, 0, d, batch_eps, par);
}

}  // namespace pa
