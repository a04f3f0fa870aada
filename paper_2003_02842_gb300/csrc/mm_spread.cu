// mm_spread.cu -- stage (a) of the hot path: time rescaling and phase
// reduction to grid cells (Algorithm 4), returns (Algorithm 3 step F.3), the
// Nyquist cutoff (Algorithm 2) and the spreading of returns onto the
// oversampled grid (Eq. (12); Algorithms 8-10 step C) with the Gaussian (fast
// Gaussian gridding split, Eq. (17)), Kaiser-Bessel (Eq. (7)) or exponential
// of semicircle (Eq. (9)) kernel.
//
// Phase reduction. GB300 executes float64 at about 1/47 of the float32 rate
// (measured: 4.8e11 float64 FMAs per second over the chip), and a
// float32 cell coordinate loses the phase at large N. The cell coordinate
// u = (t - t0) M_r / span is therefore computed in exact 64-bit fixed point on
// the integer pipes: t_fix = trunc(t 2^F) is read off the float64 bit pattern,
// and u_fix = ((t_fix - t0_fix) S) >> sh = floor(u 2^40) comes from one
// 64 x 64 -> 128-bit product (S, sh fixed per call). b0 and the offset d in
// [0, 1) follow with 2^-40-cell resolution, finer than float64's own rounding
// of u. Returns delta = logp[h+1] - logp[h] use float64 on the FP64 path and
// an exact hi/lo float32 split of each log-price on the mixed path (about 47
// significant bits, so the cancellation in the difference costs nothing).
//
// Spreading design: one block owns a contiguous tile of grid cells of one
// asset and accumulates into shared memory. Because an asset's times are
// sorted, the events whose stencil reaches the tile form at most three index
// ranges (the tile plus its halo, and the halo's periodic images), found by a
// block-parallel search on the same integer u_fix the accumulation uses. No
// global atomics; every shared-memory write is checked against the tile, so
// malformed input cannot write out of bounds.
#include <math.h>

#include <algorithm>
#include <type_traits>

#include "mm_common.cuh"
#include "mm_spread_dev.cuh"

namespace mmgpu {

// ------------------------------------------------------------------ bounds
// Validates the CSR offsets, finds t_min / t_max (Algorithm 4) or takes the
// caller's window, fixes the time fixed-point format and writes the gate word
// (0 = proceed). Block g handles problem g of a batch (assets g*gsize ..
// (g+1)*gsize - 1; a single problem has one block with gsize = D). A block
// reads event times only after checking that its own offsets are
// non-decreasing and lie in [0, max_events], so a malformed offsets array
// anywhere leaves every read in bounds.
__global__ void k_bounds(const int64_t* __restrict__ off, const double* __restrict__ t, int D, int gsize,
                         int64_t max_events, double w0, double w1, int64_t Mr, Rescale* rs, int* status,
                         int* __restrict__ order, int* __restrict__ row_exp) {
  __shared__ double s_lo[8], s_hi[8];
  __shared__ int s_bad;
  pdl_wait();     // the previous call's kernels may still read the gate
  pdl_trigger();  // prep may be scheduled (it waits for this kernel)
  int* gate = status + 1;
  const int g = blockIdx.x;
  const int i0 = g * gsize, i1 = min(i0 + gsize, D);
  if (threadIdx.x == 0) s_bad = 0;
  __syncthreads();
  // 1) the offsets alone: non-decreasing from 0 up to at most max_events.
  //    Only when all of them hold is any event time read.
  int bad = 0;
  for (int i = i0 + threadIdx.x; i < i1; i += blockDim.x) {
    if (off[i + 1] < off[i]) bad = 1;
    if (row_exp) row_exp[i] = 0;  // the prep kernel raises it
  }
  if (threadIdx.x == 0 && (off[i0] < 0 || off[i1] > max_events || (g == 0 && off[0] != 0))) bad = 1;
  if (bad) atomicOr(&s_bad, 1);
  __syncthreads();
  if (s_bad) {
    if (threadIdx.x == 0) {
      atomicOr(status, ST_BAD_OFFSETS);
      rs[g].t0 = rs[g].t1 = 0.0;
      if (gridDim.x == 1) *gate = 1;
      else atomicOr(gate, 1);
    }
    return;
  }
  // 2) t_min / t_max from each asset's first and last event (Algorithm 4);
  //    the first asset's two times are loaded before the ranking below and
  //    used after it, so that the load latency overlaps the ranking
  const bool window = w1 > w0;
  double lo = INFINITY, hi = -INFINITY;
  int outwin = 0;
  double f0 = INFINITY, l0 = -INFINITY;
  bool has0 = false;
  {
    const int i = i0 + (int)threadIdx.x;
    if (i < i1) {
      const int64_t a = off[i], b = off[i + 1];
      if (b > a) {
        f0 = t[a];
        l0 = t[b - 1];
        has0 = true;
      }
    }
  }
  // the spreading tiles' dispatch order: assets ranked by event count,
  // heaviest first (ties by index), so that the longest tiles start first
  if (order) {  // uniform: a single problem, D <= kOrderMaxAssets
    __shared__ int s_cnt[kOrderMaxAssets];
    for (int i = threadIdx.x; i < D; i += blockDim.x) {
      const int64_t c = off[i + 1] - off[i];
      s_cnt[i] = (int)min(c, (int64_t)0x7fffffff);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < D; i += blockDim.x) {
      const int ci = s_cnt[i];
      int r = 0;
      for (int j = 0; j < D; ++j) {
        const int cj = s_cnt[j];
        r += (cj > ci || (cj == ci && j < i)) ? 1 : 0;
      }
      order[r] = i;
    }
  }
  if (has0) {
    lo = fmin(lo, f0);
    hi = fmax(hi, l0);
    if (window && (f0 < w0 || l0 > w1)) outwin = 1;
  }
  for (int i = i0 + (int)threadIdx.x + (int)blockDim.x; i < i1; i += blockDim.x) {
    const int64_t a = off[i], b = off[i + 1];
    if (b > a) {
      const double f = t[a], l = t[b - 1];
      lo = fmin(lo, f);
      hi = fmax(hi, l);
      if (window && (f < w0 || l > w1)) outwin = 1;
    }
  }
  if (outwin) atomicOr(&s_bad, 2);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    lo = fmin(lo, __shfl_xor_sync(0xffffffffu, lo, o));
    hi = fmax(hi, __shfl_xor_sync(0xffffffffu, hi, o));
  }
  if ((threadIdx.x & 31) == 0) {
    s_lo[threadIdx.x >> 5] = lo;
    s_hi[threadIdx.x >> 5] = hi;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < (int)(blockDim.x >> 5); ++w) {
      lo = fmin(lo, s_lo[w]);
      hi = fmax(hi, s_hi[w]);
    }
    s_lo[0] = lo;
    s_hi[0] = hi;
    const double t0 = window ? w0 : s_lo[0];
    const double t1 = window ? w1 : s_hi[0];
    int gt = 0;
    if (s_bad & 2) { atomicOr(status, ST_OUT_OF_WINDOW); gt = 1; }
    if (!gt && !(t1 > t0 && isfinite(t0) && isfinite(t1))) {
      // all assets empty, a single instant, or non-finite times
      if (s_hi[0] >= s_lo[0] || window || isnan(s_lo[0]) || isnan(s_hi[0])) atomicOr(status, ST_SPAN);
      gt = 1;
    }
    Rescale r{};
    r.t0 = t0;
    r.t1 = t1;
    if (!gt) {
      int ex;
      frexp(fmax(fabs(t0), fabs(t1)), &ex);  // max |t| < 2^ex
      r.F = 62 - (ex + 1);                   // |t_fix| < 2^61
      r.t0_fix = to_fix(t0, r.F);
      if (Mr > 0) {
        // the cell scale of this call's grid, once (float64 is slow here)
        const UScale us = make_uscale(r, Mr);
        r.S = us.S;
        r.sh = us.sh;
        r.scale_Mr = Mr;
      }
    }
    rs[g] = r;
    if (gridDim.x == 1) *gate = gt;  // one problem: this call's gate
    else if (gt) atomicOr(gate, 1);  // batched: cleared before the launch
  }
}

cudaError_t launch_bounds(const int64_t* off, const double* t, int D, int gsize, int64_t max_events, double w0,
                          double w1, int64_t Mr, Rescale* rs, int* status, int* order, int* row_exp,
                          cudaStream_t s) {
  const int G = (D + gsize - 1) / gsize;
  if (order && (G != 1 || D > kOrderMaxAssets)) return cudaErrorInvalidValue;
  if (G > 1) {
    cudaError_t e = cudaMemsetAsync(status + 1, 0, sizeof(int), s);  // the gate of this call
    if (e != cudaSuccess) return e;
  }
  // a warp is enough for a problem of at most 32 assets: 8192 problems of two
  // took 87 us with 256 threads and the cell scales (float64 divisions by one
  // thread) in every block, 13.6 us with a warp and the scales left to
  // k_group_scales
  const int nth = gsize <= 32 && !order ? 32 : 256;
  return launch_pdl(k_bounds, dim3(G), dim3(nth), 0, s, off, t, D, gsize, max_events, w0, w1, Mr, rs, status,
                    order, row_exp);
}

// Per-problem fixed-point cell scales for the grid size of this call.
__global__ void k_group_scales(const Rescale* __restrict__ rs, int G, int64_t Mr, const int* __restrict__ gate,
                               GroupScale* out) {
  const int g = blockIdx.x * blockDim.x + threadIdx.x;
  if (g >= G || *gate) return;
  const Rescale r = rs[g];
  GroupScale q;
  q.us = make_uscale(r, Mr);
  q.t0_fix = r.t0_fix;
  q.F = r.F;
  out[g] = q;
}

size_t group_scale_bytes() { return sizeof(GroupScale); }

cudaError_t launch_group_scales(const Rescale* rs, int G, int64_t Mr, GroupScale* out, const int* status,
                                cudaStream_t s) {
  k_group_scales<<<(G + 127) / 128, 128, 0, s>>>(rs, G, Mr, status + 1, out);
  return cudaGetLastError();
}

// ------------------------------------------------------------------ Nyquist
// Algorithm 2: per-asset smallest gap, then
// N = floor(span / (2 max_i gap_i)) = min_i floor(span / (2 gap_i)).
//
// Bound by the latency of one pass over the times: `splits` blocks (grid column)
// share an asset's gaps, 1024 a block where the chip has room, their minimum meets
// in gap[i] and the last block to arrive takes the maximum over the assets and the
// cutoff (a launch of its own before): 18 us in two launches before, 7.6 us now, for ten
// assets of some 12,500 events.
//
// gap[0 .. D) and the arrival counter gap[D] are zero between calls (the last block
// clears them). gap[i] holds the complement of the smallest gap's bits (positive
// doubles order like their bits), so that zero is "no gap seen"; a gap that is not
// positive counts as 0 and leaves its asset out.
constexpr int kGapThreads = 256;
constexpr int kGapPerBlock = 1024;

__global__ void __launch_bounds__(kGapThreads) k_min_gap(const int64_t* __restrict__ off,
                                                         const double* __restrict__ t, int D,
                                                         const Rescale* __restrict__ rs, const int* gate,
                                                         unsigned long long* gap, int* nyq, int* status) {
  __shared__ unsigned long long s_w[kGapThreads / 32];
  __shared__ bool s_last;
  pdl_wait();
  if (*gate) {  // uniform over the grid
    if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) *nyq = -1;
    return;
  }
  const int i = blockIdx.x;
  const int64_t a = off[i], b = off[i + 1];
  double g = INFINITY;
  int dup = 0;
  const int64_t step = (int64_t)gridDim.y * kGapThreads;
#pragma unroll 4
  for (int64_t h = a + (int64_t)blockIdx.y * kGapThreads + threadIdx.x; h + 1 < b; h += step) {
    const double d = t[h + 1] - t[h];
    if (!(d > 0)) dup = (d == 0) ? 1 : 2;
    g = fmin(g, d);
  }
  if (dup == 1) atomicOr(status, ST_DUPLICATE);
  if (dup == 2) atomicOr(status, ST_UNSORTED);
  // block maximum of the complements
  unsigned long long w = ~(unsigned long long)__double_as_longlong(g > 0 ? g : 0.0);
  auto warp_max = [](unsigned long long x) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x = max(x, __shfl_xor_sync(0xffffffffu, x, o));
    return x;
  };
  w = warp_max(w);
  if ((threadIdx.x & 31) == 0) s_w[threadIdx.x >> 5] = w;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int k = 1; k < kGapThreads / 32; ++k) w = max(w, s_w[k]);
    atomicMax(gap + i, w);
    __threadfence();
    s_last = atomicAdd(gap + D, 1ull) == (unsigned long long)gridDim.x * gridDim.y - 1;
    __threadfence();
  }
  __syncthreads();
  if (!s_last) return;
  // the last block: largest of the assets' smallest gaps, the words cleared
  const unsigned long long inf = (unsigned long long)__double_as_longlong(INFINITY);
  unsigned long long top = 0;
  for (int k = threadIdx.x; k < D; k += kGapThreads) {
    const unsigned long long q = ~__ldcg(gap + k);
    if (q < inf) top = max(top, q);
    gap[k] = 0;
  }
  top = warp_max(top);
  if ((threadIdx.x & 31) == 0) s_w[threadIdx.x >> 5] = top;
  __syncthreads();
  if (threadIdx.x == 0) {
    gap[D] = 0;
    for (int k = 1; k < kGapThreads / 32; ++k) top = max(top, s_w[k]);
    if (top == 0ull) {
      *nyq = -1;
      atomicOr(status, ST_CUTOFF);
    } else {
      const double v = floor((rs->t1 - rs->t0) / (2.0 * __longlong_as_double((long long)top)));
      *nyq = (v > 2147483647.0) ? 2147483647 : (int)v;
    }
  }
}

cudaError_t launch_min_gap(const int64_t* off, const double* t, int D, int64_t asset_events, const Rescale* rs,
                           unsigned long long* gap, int* nyq, int* status, cudaStream_t s) {
  // a block per kGapPerBlock events of an asset of the plan's mean size, eight
  // blocks an SM at most
  const int64_t want = (asset_events + kGapPerBlock - 1) / kGapPerBlock, room = std::max(1, 152 * 8 / D);
  const int splits = (int)std::max<int64_t>(1, std::min(want, room));
  return launch_pdl(k_min_gap, dim3(D, splits), dim3(kGapThreads), 0, s, off, t, D, rs, status + 1, gap, nyq, status);
}

constexpr int kSpreadThreads = 256;

// ------------------------------------------------------------------ prep
// Steps a0 / a1 of the hot path: for each event h, the rescaled cell
// coordinate in exact fixed point (Algorithm 4), split into the cell b0 and
// the offset d in [0, 1), and the return delta = logp[h+1] - logp[h]
// (Algorithm 3 step F.3), written once as a compact record (b0, d, delta) in
// event order. Since each asset's times are sorted, its records are sorted
// by cell: that order is the bin sort the spreading kernels search. The
// last event of an asset carries no return and its record is never read
// (it holds kNoCell or is left as it was).
//
// Bound by the integer pipe (51 % of its rate, and 70 % of the SMs' time at 1.03
// waves of the former 256-thread blocks): the cell and its offset of both paths come
// from one 64 x 64 -> 128-bit product (float32 offsets to 24 significant bits;
// a float-pair product took twice the instructions), the end of the asset is kept
// as a count instead of read for each event, a problem's scale is read once per
// asset of a thread, whole stretches come by 16-byte loads. 128 threads leave 56
// registers at nine blocks an SM, without the spills of 48. 9.2e6 events in 512
// problems: 146 -> 120 us; 100 assets of some 7,700: 16.4 -> 14.4 us.
//
// Each thread takes kPrepE consecutive events: it loads kPrepE + 1 times and
// log-prices, orders, checks and splits each value once (every value but the
// last serves two returns), and writes its records with vector stores.
constexpr int kPrepE = 4;
constexpr int kPrepThreads = 128;
// SPARE: a call for fewer assets than the plan's, whose grid by the plan's capacity
// would be mostly empty blocks (a server's requests: 34 -> 29.6 us each): two
// waves of blocks at most and a loop. Where the capacity is the call's own size the
// loop costs more than it gives (16.4 -> 19.2 us at 100 assets).
constexpr int64_t kPrepSpareBlocks = 152 * 9 * 2;

template <typename T> struct Rec4;
template <> struct Rec4<float> {
  static __device__ __forceinline__ void store(float* p, const float* v) {
    *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
  }
};
template <> struct Rec4<double> {
  static __device__ __forceinline__ void store(double* p, const double* v) {
    reinterpret_cast<double2*>(p)[0] = make_double2(v[0], v[1]);
    reinterpret_cast<double2*>(p)[1] = make_double2(v[2], v[3]);
  }
};

// z = d - 1/2 of a 40-bit offset as a float pair, exactly: 24 bits rounded into
// hi, the rest in lo (|lo| <= 2^-24), built with 1.5 2^23 instead of conversions.
__device__ __forceinline__ double offset_pair(unsigned long long frac) {
  const long long s = (long long)frac - (1ll << 39);
  const int hi = (int)((s + (1 << 16)) >> 17);
  const int lo = (int)(s - ((long long)hi << 17));
  const float zh = (__int_as_float(kRoundMagicBits + hi) - kRoundMagic) * 1.1920928955078125e-07f;      // 2^-23
  const float zl = (__int_as_float(kRoundMagicBits + lo) - kRoundMagic) * 9.094947017729282e-13f;       // 2^-40
  return __hiloint2double(__float_as_int(zh), __float_as_int(zl));
}

// PAIR (float64): the offset as the float pair of offset_pair in its 8 bytes, and
// each asset's largest exponent field of a return into row_exp (its grid row, in
// float pairs, is scaled by it).
template <typename T, bool PAIR, bool SPARE>
__global__ void __launch_bounds__(kPrepThreads, 9)
    k_prep(const int64_t* __restrict__ off, const double* __restrict__ t, const double* __restrict__ logp,
           const Rescale* __restrict__ rsp, const GroupScale* __restrict__ gsc, int gsize,
           const int* __restrict__ gate, int D, int64_t Mr, int* __restrict__ rb0, T* __restrict__ rd,
           T* __restrict__ rv, int* __restrict__ row_exp, int* status) {
  static_assert(kPrepE == 4, "records are stored as 4-vectors");
  __shared__ UScale s_us;
  __shared__ int s_flags;
  __shared__ int s_a0;
  // one round of loads: the gate, the event count and the call's rescaling
  // (with its cell scales when k_bounds knew the grid); then each thread's
  // event loads are in flight while warp 0 finds the block's asset. No event
  // is read before the gate (k_bounds' validation of the offsets) is known.
  pdl_wait();
  const int gated = *gate;
  const int64_t ntot = off[D];
  Rescale rs0{};
  if (!gsc) rs0 = *rsp;
  if (gated) return;  // uniform
  const bool scales = gsc || rs0.scale_Mr == Mr;  // uniform
  const bool vec = ((reinterpret_cast<uintptr_t>(t) | reinterpret_cast<uintptr_t>(logp)) & 15) == 0;
  for (int64_t hb = (int64_t)blockIdx.x * (kPrepThreads * kPrepE); hb < ntot;
       hb += (int64_t)gridDim.x * (kPrepThreads * kPrepE)) {
    const int64_t h0 = hb + (int64_t)threadIdx.x * kPrepE;
    double tv[kPrepE + 1], pv[kPrepE + 1];
    if (vec && h0 + kPrepE < ntot) {
      // 16-byte loads (h0 is a multiple of 4)
      const double2* t2 = reinterpret_cast<const double2*>(t + h0);
      const double2* p2 = reinterpret_cast<const double2*>(logp + h0);
      const double2 ta = __ldg(t2), tb = __ldg(t2 + 1), pa = __ldg(p2), pb = __ldg(p2 + 1);
      tv[0] = ta.x, tv[1] = ta.y, tv[2] = tb.x, tv[3] = tb.y, tv[4] = __ldg(t + h0 + 4);
      pv[0] = pa.x, pv[1] = pa.y, pv[2] = pb.x, pv[3] = pb.y, pv[4] = __ldg(logp + h0 + 4);
    } else {
#pragma unroll
      for (int j = 0; j <= kPrepE; ++j) {
        tv[j] = 0.0;
        pv[j] = 0.0;
        if (h0 + j < ntot) {
          tv[j] = t[h0 + j];
          pv[j] = logp[h0 + j];
        }
      }
    }
    if (threadIdx.x == 0) {
      if (!scales) s_us = make_uscale(rs0, Mr);  // (the same on each pass)
      s_flags = 0;
    }
    // asset of the block's first event (a 32-ary search by warp 0, a couple of
    // dependent loads), then each thread walks forward to its own events' assets
    if (threadIdx.x < 32) {
      // first index in [1, D] with off[idx] > hb (D when none): the asset is idx - 1
      const int lane = threadIdx.x;
      int64_t lo = 1, hi = D;
      for (int it = 0; it < 16 && hi > lo; ++it) {
        const int64_t len = hi - lo;
        const int64_t stride = (len + 31) / 32;
        const int64_t o = (int64_t)lane * stride;
        const bool below = o < len && off[lo + o] <= hb;
        const int cnt = __popc(__ballot_sync(0xffffffffu, below));
        if (cnt == 0) {
          hi = lo;
        } else {
          const int64_t nlo = lo + (int64_t)(cnt - 1) * stride + 1;
          const int64_t nhi = min(lo + (int64_t)cnt * stride, hi);
          lo = min(nlo, nhi);
          hi = nhi;
        }
      }
      if (lane == 0) s_a0 = (int)lo - 1;
    }
    __syncthreads();
    int flags = 0;
    int b0v[kPrepE];
    T dv[kPrepE], vv[kPrepE];
    int lo = s_a0;
    // events of asset lo from h0 on (a thread looks at five)
    auto left = [&](int a) {
      const int64_t r = off[a + 1] - h0;
      return r > kPrepE + 1 ? kPrepE + 2 : r < 0 ? 0 : (int)r;
    };
    int rem = left(lo);
    int cur = -1;  // asset of the scale in use (batched form)
    long long t0_fix = rs0.t0_fix;
    int F = rs0.F;
    UScale us{rs0.S, rs0.sh};
    if (!scales) us = s_us;
    int ex_asset = -1, ex_top = 0;  // PAIR: the asset of the thread's records so far and their largest exponent
    // per value, once: order key, finiteness and (float32 path) the exact hi + lo
    // split of the log-price
    long long key = order_key(tv[0]);
    bool fin_p = finite_bits(pv[0]);
    float ph = 0.f, pl = 0.f;
    if (sizeof(T) == 4) split_f64(pv[0], ph, pl);
#pragma unroll
    for (int j = 0; j < kPrepE; ++j) {
      const long long key0 = key;
      const bool fin_p0 = fin_p;
      const float ph0 = ph, pl0 = pl;
      key = order_key(tv[j + 1]);
      fin_p = finite_bits(pv[j + 1]);
      if (sizeof(T) == 4) split_f64(pv[j + 1], ph, pl);
      b0v[j] = kNoCell;
      dv[j] = (T)0;
      vv[j] = (T)0;
      while (j >= rem && lo + 1 < D) rem = left(++lo);
      if (!(j + 1 < rem)) continue;  // the asset's last event: no return
      // this event's problem: its fixed-point scale (batched form), kept while
      // the asset is the same, or the call's single one
      if (gsc && lo != cur) {
        const GroupScale q = gsc[lo / gsize];
        t0_fix = q.t0_fix;
        F = q.F;
        us = q.us;
        cur = lo;
      }
      if (!(key0 < key)) flags |= (key0 == key) ? ST_DUPLICATE : ST_UNSORTED;
      if (!(finite_bits(tv[j]) && fin_p0 && fin_p)) {
        flags |= ST_NONFINITE;
        continue;
      }
      const long long dt = to_fix(tv[j], F) - t0_fix;
      const unsigned long long uf = u_fix_of(dt, us);
      const int cb = (int)(uf >> kUFrac);
      const unsigned long long frac = uf & ((1ull << kUFrac) - 1);
      if (dt < 0 || cb > Mr || (cb == Mr && frac != 0ull)) {  // beyond the last cell's start
        flags |= ST_OUT_OF_WINDOW;
        continue;
      }
      b0v[j] = cb;
      if (PAIR) dv[j] = (T)offset_pair(frac);
      else dv[j] = frac_to<T>(frac);
      if (sizeof(T) == 8) vv[j] = (T)(pv[j + 1] - pv[j]);
      else vv[j] = (T)((ph - ph0) + (pl - pl0));
      if (PAIR) {
        if (lo != ex_asset && ex_asset >= 0) {
          atomicMax(row_exp + ex_asset, ex_top);
          ex_top = 0;
        }
        ex_asset = lo;
        ex_top = max(ex_top, (__double2hiint((double)vv[j]) >> 20) & 0x7FF);
      }
    }
    if (PAIR) {
      // one update a warp when its threads' last records are of one asset
      const int a0 = __shfl_sync(0xffffffffu, ex_asset, 0);
      if (__all_sync(0xffffffffu, ex_asset == a0)) {
        ex_top = __reduce_max_sync(0xffffffffu, ex_top);
        if ((threadIdx.x & 31) == 0 && a0 >= 0) atomicMax(row_exp + a0, ex_top);
      } else if (ex_asset >= 0) {
        atomicMax(row_exp + ex_asset, ex_top);
      }
    }
    if (h0 + kPrepE <= ntot) {
      // h0 is a multiple of 4 and the record arrays are the plan's own
      // (256-byte aligned) allocations: 16-byte vector stores
      *reinterpret_cast<int4*>(rb0 + h0) = make_int4(b0v[0], b0v[1], b0v[2], b0v[3]);
      Rec4<T>::store(rd + h0, dv);
      Rec4<T>::store(rv + h0, vv);
    } else {
#pragma unroll
      for (int j = 0; j < kPrepE; ++j) {
        if (h0 + j < ntot) {
          rb0[h0 + j] = b0v[j];
          rd[h0 + j] = dv[j];
          rv[h0 + j] = vv[j];
        }
      }
    }
    if (flags) atomicOr(&s_flags, flags);
    __syncthreads();
    if (threadIdx.x == 0 && s_flags) atomicOr(status, s_flags);
    if (!SPARE) break;
  }
  pdl_trigger();
}

template <typename T, bool PAIR>
static cudaError_t launch_prep_t(const int64_t* off, const double* t, const double* logp, const Rescale* rs,
                                 const GroupScale* gsc, int gsize, int D, int64_t Mr, int64_t max_events, bool spare,
                                 int* rb0, T* rd, T* rv, int* row_exp, int* status, cudaStream_t s) {
  if (max_events <= 0) return cudaSuccess;
  if ((((uintptr_t)rb0) | ((uintptr_t)rd) | ((uintptr_t)rv)) & 15) return cudaErrorMisalignedAddress;
  const int64_t per_block = (int64_t)kPrepThreads * kPrepE;
  int64_t blocks = (max_events + per_block - 1) / per_block;
  if (spare) blocks = std::min(blocks, kPrepSpareBlocks);
  return launch_pdl(spare ? k_prep<T, PAIR, true> : k_prep<T, PAIR, false>, dim3((unsigned)blocks),
                    dim3(kPrepThreads), 0, s, off, t, logp, rs, gsc, gsize, status + 1, D, Mr, rb0, rd, rv, row_exp,
                    status);
}

cudaError_t launch_prep_f32(const int64_t* off, const double* t, const double* logp, const Rescale* rs,
                            const GroupScale* gsc, int gsize, int D,
                            int64_t Mr, int64_t max_events, bool spare, int* rb0, void* rd, void* rv, int* status,
                            cudaStream_t s) {
  return launch_prep_t<float, false>(off, t, logp, rs, gsc, gsize, D, Mr, max_events, spare, rb0, (float*)rd, (float*)rv,
                                     nullptr, status, s);
}
cudaError_t launch_prep_f64(const int64_t* off, const double* t, const double* logp, const Rescale* rs,
                            const GroupScale* gsc, int gsize, int D,
                            int64_t Mr, int64_t max_events, bool spare, int* row_exp, int* rb0, void* rd, void* rv,
                            int* status, cudaStream_t s) {
  auto go = [&](auto fn) {
    return fn(off, t, logp, rs, gsc, gsize, D, Mr, max_events, spare, rb0, (double*)rd, (double*)rv, row_exp, status, s);
  };
  return row_exp ? go(launch_prep_t<double, true>) : go(launch_prep_t<double, false>);
}

// ------------------------------------------------------------------ spread
template <typename T> struct EvChunk { static constexpr int n = 1536; };  // 6 spreading blocks per SM

// Gather spreading (Eq. (12)): thread t owns cells c = t CPT .. t CPT + CPT-1
// of the tile and sums, in registers, delta_e phi(c - p_e - d_e) over the
// events with c - p_e in [klo, khi], a sliding window over the sorted
// positions of each event chunk (no atomics, deterministic).
template <typename T, int KERNEL, int CPT>
__global__ void __launch_bounds__(kSpreadThreads) k_spread_gather(const int64_t* __restrict__ off,
                                                                 const int* __restrict__ rb0,
                                                                 const T* __restrict__ rd, const T* __restrict__ rv,
                                                                 const int* __restrict__ gate, SpreadParams p,
                                                                 T* __restrict__ grid) {
  constexpr int EC = EvChunk<T>::n;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  int* ev_p = reinterpret_cast<int*>(smem_raw);
  T* ev_d = reinterpret_cast<T*>(smem_raw + EC * sizeof(int));
  T* ev_v = ev_d + EC;
  if (*gate) return;  // uniform: the whole block leaves
  const int a = blockIdx.y;
  const int64_t L = (int64_t)blockIdx.x * p.tile;
  const int Tlen = (int)min((int64_t)p.tile, p.Mr - L);
  TileRanges tr;
  tile_ranges(off, rb0, p, a, L, Tlen, tr);
  const int64_t ntot = tr.n2 + tr.n1 + tr.n0;
  const int c0 = threadIdx.x * CPT;
  T acc[CPT];
#pragma unroll
  for (int q = 0; q < CPT; ++q) acc[q] = (T)0;
  for (int64_t cs = 0; cs < ntot; cs += EC) {
    const int n = (int)min((int64_t)EC, ntot - cs);
    for (int i = threadIdx.x; i < n; i += kSpreadThreads) load_record<T>(rb0, rd, rv, p, tr, L, cs + i, ev_p[i], ev_d[i], ev_v[i]);
    __syncthreads();
    if (c0 < Tlen) {
      int lo = 0, hi = n;
      const int want = c0 - p.khi;
      while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (ev_p[mid] < want) lo = mid + 1;
        else hi = mid;
      }
#pragma unroll
      for (int q = 0; q < CPT; ++q) {
        const int c = c0 + q;
        while (lo < n && ev_p[lo] < c - p.khi) ++lo;
        T sum = (T)0;
        for (int e = lo; e < n; ++e) {
          const int k = c - ev_p[e];
          if (k < p.klo) break;
          sum += ev_v[e] * kernel_value<T, KERNEL>((T)k - ev_d[e], p);
        }
        acc[q] += sum;
      }
    }
    __syncthreads();
  }
  T* g = grid + (int64_t)a * p.Mr + L;
#pragma unroll
  for (int q = 0; q < CPT; ++q)
    if (c0 + q < Tlen) g[c0 + q] = acc[q];
}

// Scatter spreading (Eq. (12)): event records are staged per chunk in shared
// memory, then each thread adds one event's whole stencil into the shared-
// memory tile (at most KW points, unrolled; 32-bit indices). Lanes of a warp
// take consecutive events, so their cells rarely coincide.
template <typename T, int KERNEL, int KW>
__global__ void __launch_bounds__(kSpreadThreads) k_spread_scatter(const int64_t* __restrict__ off,
                                                                  const int* __restrict__ rb0,
                                                                  const T* __restrict__ rd, const T* __restrict__ rv,
                                                                  const int* __restrict__ gate, SpreadParams p,
                                                                  T* __restrict__ grid) {
  constexpr int EC = EvChunk<T>::n;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  int* ev_p = reinterpret_cast<int*>(smem_raw);
  T* ev_d = reinterpret_cast<T*>(smem_raw + EC * sizeof(int));
  T* ev_v = ev_d + EC;
  T* tile = ev_v + EC;
  if (*gate) return;  // uniform: the whole block leaves
  const int a = blockIdx.y;
  const int64_t L = (int64_t)blockIdx.x * p.tile;
  const int Tlen = (int)min((int64_t)p.tile, p.Mr - L);
  {
    float4* t4 = reinterpret_cast<float4*>(tile);
    const int n4 = (int)(((size_t)Tlen * sizeof(T) + 15) / 16);
    for (int c = threadIdx.x; c < n4; c += kSpreadThreads) t4[c] = make_float4(0.f, 0.f, 0.f, 0.f);
  }
  TileRanges tr;
  tile_ranges(off, rb0, p, a, L, Tlen, tr);
  const int64_t ntot = tr.n2 + tr.n1 + tr.n0;
  const int klo = p.klo, nk = p.khi - p.klo + 1;
  for (int64_t cs = 0; cs < ntot; cs += EC) {
    const int n = (int)min((int64_t)EC, ntot - cs);
    for (int i = threadIdx.x; i < n; i += kSpreadThreads) load_record<T>(rb0, rd, rv, p, tr, L, cs + i, ev_p[i], ev_d[i], ev_v[i]);
    __syncthreads();
    for (int e = threadIdx.x; e < n; e += kSpreadThreads) {
      const int pe = ev_p[e];
      const T de = ev_d[e], ve = ev_v[e];
      T x = (T)klo - de;
#pragma unroll
      for (int j = 0; j < KW; ++j) {
        if (j >= nk) break;
        const unsigned c = (unsigned)(pe + klo + j);
        if (c < (unsigned)Tlen) atomicAdd(tile + c, ve * kernel_value<T, KERNEL>(x, p));
        x += (T)1;
      }
    }
    __syncthreads();
  }
  T* g = grid + (int64_t)a * p.Mr + L;
  // rows of M_r (even) cells start 8-byte aligned; tiles are multiples of 4 cells
  if (((reinterpret_cast<uintptr_t>(g) & 15) == 0) && (Tlen * sizeof(T)) % 16 == 0) {
    const float4* t4 = reinterpret_cast<const float4*>(tile);
    float4* g4 = reinterpret_cast<float4*>(g);
    const int n4 = (int)((size_t)Tlen * sizeof(T) / 16);
    for (int c = threadIdx.x; c < n4; c += kSpreadThreads) g4[c] = t4[c];
  } else {
    for (int c = threadIdx.x; c < Tlen; c += kSpreadThreads) g[c] = tile[c];
  }
}

// Float32 scatter with polynomial taps and exact integer accumulation.
// Shared-memory float atomics run as compare-and-swap loops and 64-bit
// integer reductions are slower still (3.4x and 5.6x the time of an int32
// reduction on GB300), so each tap's product x = v phi 2^eh goes to two int32
// tiles by native int32 reductions: hi = round(x) and lo = round((x - hi) 2^k).
// Both sums are exact and independent of the order of the atomics; a cell
// holds (hi + lo 2^-k) 2^-eh with one quantum 2^-(eh + k) per tap.
//
// Scales (B = sum |v|, V = max |v| over the tile's n events, |phi| <= 1 + 1e-6):
//  * eh = min(29 - ex(B), 21 - ex(V)) with B < 2^ex(B), V < 2^ex(V): every
//    |x| < 2^21 (the rounding below needs |x| < 2^22) and a cell's hi sum is
//    below 2^29 (1 + 1e-6) + n/2 < 2^31;
//  * k = min(20, 30 - bitlen(n)): |lo| <= 2^(k-1) + 1 per tap, so a cell's lo
//    sum is below n (2^(k-1) + 1) < 2^30.
// The quantum per tap, 2^-(eh + k), is therefore at most
// max(B 2^-(28 + k), V 2^-(20 + k)): max(B 2^-48, V 2^-40) for tiles of up to
// 1023 events, and for larger tiles at most max(B n 2^-58, V n 2^-50)
// (2^-k < 2n 2^-30). Against float32 rounding of a tap's product (2^-24 of
// it) this is negligible up to about 2^20 events per tile.
//
// round(y) for |y| < 2^22 is taken as y + 1.5 2^23, whose float spacing is 1
// (one FMA, no conversion instruction; kRoundMagic).

// Threads of a polynomial-scatter block and records it stages at a time. A block is
// a chain of dependent latencies (offsets, search, records, barriers), which other
// blocks hide when there are many: 128 threads and eight blocks an SM from
// kPolyBlocksMany tiles up (512 replications of ten assets: 474 us against 609 us
// with 256 threads), 256 threads and six blocks down to kPolyBlocksSome (the block
// workload's 1000 tiles: 18.4 us against 20.7 us with 128), else 512 threads. 512 also
// where the assets' capacity gives a tile more than kPolyManyRecords (a busy day in
// the one tile of a low cutoff's grid): a thread then sums runs of several records
// of a cell before it reduces.
template <int NTH> struct PolyBlock;
template <> struct PolyBlock<128> { static constexpr int chunk = 896, per_sm = 8; };
template <> struct PolyBlock<256> { static constexpr int chunk = 1536, per_sm = 6; };
template <> struct PolyBlock<512> { static constexpr int chunk = 4096, per_sm = 2; };
// One block an SM fewer for wide stencils, whose dense tiles keep 24 sums or more a thread
// and spilled 130 bytes at 40 registers.
template <int NT, int NTH>
constexpr int kPolyPerSm = PolyBlock<NTH>::per_sm - (NT > 16 && NTH < 512 ? 1 : 0);
constexpr int64_t kPolyBlocksMany = 8 * 152 * 2;
constexpr int64_t kPolyBlocksSome = 2 * 152;
constexpr int kPolyManyRecords = 4096;

// Sparse tiles, one word per cell. When no stretch of 2 NP cells (a stencil)
// holds more than kOneRun records, a cell's sum is at most the largest sum W of
// |v| over kOneRun records in a row, not that of the tile: with x = v phi 2^e,
// e = 31 - ex(W kOneRoom), every cell's sum of the rounded x stays below 2^31 / kOneRoom
// times the taps' largest value (1 and their fit error, at most 0.05 at the loosest
// tolerance) + kOneRun / 2 < 2^31 in one int32, with a quantum of at most W 2^-30 1.07.
// The tile is taken so only where W is at most kOneEven times the largest run of every
// warp's records (32 in a row at a time): a tap is then off by at most 170 2^-31 of the
// mean |v| of a run nearby, 2^-24.4 of it rms, as the float32 product of a tap is, and a
// return that dwarfs the others does not cost them their digits (they keep two words;
// Brownian returns at Poisson times stay at about twice; the sum of |v| over the
// tile, reduced for this, cost 3 % of the kernel with 120 records a tile). Coefficients'
// float32 rounding is 1 to 3 % above that with two words (1.87e-7 and 1.84e-7 of a row at
// the block workload, beside a truncation of 3e-6; 2 to 4 % with a quantum of W 2^-29).
// One word halves the shared-memory reductions, which bound the taps, and the tile. With
// the shorter taps below, the guessed search and the block sizes above the block workload's
// spreading took 18.4 us (20.2 us with two words a cell in every tile), 500 stocks'
// day 128 us (143 us), 512 replications of ten assets 474 us (715 us).
constexpr int kOneRun = 20;
constexpr float kOneEven = 8.0f;
constexpr float kOneRoom = 1.0625f;

// Taps k and 1 - k of a record are phi(a - z) and phi(a + z), a = k - 1/2,
// z = d - 1/2: with tap k's polynomial E(z^2) + z O(z^2), tap 1 - k is
// E - z O, nine multiply-adds for two taps instead of sixteen. The ES and
// Kaiser-Bessel stencils have one tap more, -M_sp (zero for ES inside a cell).
struct PairTaps {
  float e[kPolyMaxTaps / 2][kPolyDeg / 2 + 1];
  float o[kPolyMaxTaps / 2][kPolyDeg / 2];
  float left[kPolyDeg + 1];
  int npair;
  int has_left;
};

template <int NP, int NTH>
__device__ __forceinline__ void spread_one_word(const int* ev_p, const float* ev_d, const float* ev_v, int n, int Tlen,
                                                const PairTaps& t, float scale, uint32_t tile_s) {
  constexpr int H = kPolyDeg / 2;
  for (int ei = threadIdx.x; ei < n; ei += NTH) {
    const int pe = ev_p[ei];
    if (pe == kNoCell) continue;
    const float z = ev_d[ei] - 0.5f, y = z * z;
    const float vs = ev_v[ei] * scale;
    const bool inside = pe >= NP && pe + NP < Tlen;  // every tap, -M_sp included
    const uint32_t at = tile_s + 4u * (uint32_t)pe;
#pragma unroll
    for (int q = 0; q < NP; ++q) {
      if (q >= t.npair) break;  // uniform; NP taps pairs in the exact instantiations
      float E = t.e[q][H], O = t.o[q][H - 1];
#pragma unroll
      for (int i = H - 1; i >= 0; --i) E = fmaf(E, y, t.e[q][i]);
#pragma unroll
      for (int i = H - 2; i >= 0; --i) O = fmaf(O, y, t.o[q][i]);
      const int xk = __float2int_rn(vs * fmaf(z, O, E));
      const int xm = __float2int_rn(vs * fmaf(-z, O, E));
      if (inside) {
        red_shared_add(at + 4 * (q + 1), xk);
        red_shared_add(at - 4 * q, xm);
      } else {
        if ((unsigned)(pe + q + 1) < (unsigned)Tlen) red_shared_add(at + 4 * (q + 1), xk);
        if ((unsigned)(pe - q) < (unsigned)Tlen) red_shared_add(at - 4 * q, xm);
      }
    }
    if (t.has_left && (unsigned)(pe - t.npair) < (unsigned)Tlen) {
      float w = t.left[kPolyDeg];
#pragma unroll
      for (int i = kPolyDeg - 1; i >= 0; --i) w = fmaf(w, z, t.left[i]);
      red_shared_add(at - 4 * t.npair, __float2int_rn(vs * w));
    }
  }
}

// Cells [s0, s0 + len) of a tile to the grid, cell c's value from get(c).
template <int NTH, class Get>
__device__ __forceinline__ void write_cells(const SpreadParams& p, float* __restrict__ grid, int a, int64_t L, int s0,
                                            int len, Get get) {
  if (p.perm_np > 0) {
    // the per-asset FFT's input order: complex point m = (L + c) / 2 goes to
    // its digit reversal (tiles and M_r are even, so cells pair up)
    float2* gz = reinterpret_cast<float2*>(grid + (int64_t)a * p.Mr);
    const int m0 = (int)((L + s0) >> 1);
    for (int c2 = threadIdx.x; c2 < (len >> 1); c2 += NTH) {
      int m = m0 + c2, pos = 0;
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        if (q < p.perm_np) {
          const int R = p.perm_rad[q];
          const int h = (int)__umulhi((unsigned)m, p.perm_magic[q]);
          pos += (m - h * R) * p.perm_stride[q];
          m = h;
        }
      }
      gz[pos] = make_float2(get(2 * c2), get(2 * c2 + 1));
    }
    return;
  }
  float* g = grid + (int64_t)a * p.Mr + L + s0;
  if (((reinterpret_cast<uintptr_t>(g) & 15) == 0) && (len & 3) == 0) {
    float4* g4 = reinterpret_cast<float4*>(g);
    for (int c = threadIdx.x; c < len / 4; c += NTH)
      g4[c] = make_float4(get(4 * c), get(4 * c + 1), get(4 * c + 2), get(4 * c + 3));
  } else {
    for (int c = threadIdx.x; c < len; c += NTH) g[c] = get(c);
  }
}

// One block per tile. `cells` int32 of shared memory: a sparse tile has one word
// per cell, a dense one (by the records themselves) is taken in parts of cells / 2
// with a hi and a lo word each. A part stages and evaluates the records that reach it,
// from its first on (every part going through all of the tile's: one asset of 40,000
// records among 99 of 2,000 on 40,500 cells 44.6 us, now 38.2; 25 of 500 assets with
// 100,000 on 57,600 cells 166 us, now 133).
template <int NT, int NP, int NTH>
__global__ void __launch_bounds__(NTH, kPolyPerSm<NT, NTH>) k_spread_poly(const int64_t* __restrict__ off,
                                                               const int* __restrict__ rb0,
                                                               const float* __restrict__ rd,
                                                               const float* __restrict__ rv,
                                                               const int* __restrict__ gate, SpreadParams p,
                                                               const __grid_constant__ KernelPoly poly,
                                                               const __grid_constant__ PairTaps taps, int cells,
                                                               int widths_first, float* __restrict__ grid) {
  constexpr int EC = PolyBlock<NTH>::chunk;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  int* ev_p = reinterpret_cast<int*>(smem_raw);
  float* ev_d = reinterpret_cast<float*>(smem_raw + EC * sizeof(int));
  float* ev_v = ev_d + EC;
  int* tile = reinterpret_cast<int*>(ev_v + EC);
  const uint32_t tile_s = (uint32_t)__cvta_generic_to_shared(tile);
  __shared__ float s_sum[NTH / 32], s_max[NTH / 32], s_run[NTH / 32];
  const int64_t L = (int64_t)blockIdx.x * p.tile;
  const int Tlen = (int)min((int64_t)p.tile, p.Mr - L);
  auto clear = [&] {
    for (int c = threadIdx.x; c < cells / 4; c += NTH) reinterpret_cast<int4*>(tile)[c] = make_int4(0, 0, 0, 0);
  };
  clear();
  pdl_wait();         // the records come from the prep kernel
  if (*gate) return;  // uniform: the whole block leaves
  const int a = p.order ? p.order[blockIdx.y] : (int)blockIdx.y;
  TileRanges tr;
  tile_ranges(off, rb0, p, a, L, Tlen, tr);
  const int64_t ntot = tr.n2 + tr.n1 + tr.n0;
  auto stage = [&](int64_t c0, int n) {
    for (int i = threadIdx.x; i < n; i += NTH)
      load_record<float>(rb0, rd, rv, p, tr, L, c0 + i, ev_p[i], ev_d[i], ev_v[i]);
  };
  // at most kOneRun records in any stencil's width, and the largest sum of |v| over that
  // many in a row (a shorter run at the end is part of one, or the tile has no longer one);
  // chunks overlap by a run, and the last one stays staged. Where the assets'
  // density makes dense tiles likely the widths are looked at first, so that such
  // a tile leaves before the sums, which cost half its taps (a barrier more: 1.5 us
  // of the block workload's spreading)
  bool sparse = Tlen <= cells;
  float run = 0.f;
  int64_t cs = 0;
  int n = 0;
  while (true) {
    n = (int)min((int64_t)EC, ntot - cs);
    stage(cs, n);
    __syncthreads();
    const bool last = cs + n == ntot;
    const int lim = last ? max(min(n, 1), n - kOneRun + 1) : n - kOneRun;
    if (widths_first) {
      for (int i = threadIdx.x; i + kOneRun < n; i += NTH)
        sparse = sparse && ev_p[i + kOneRun] - ev_p[i] > 2 * NP;
      sparse = __syncthreads_and(sparse);
      if (!sparse) break;
    }
    for (int i = threadIdx.x; i < lim; i += NTH) {
      if (i + kOneRun < n) sparse = sparse && ev_p[i + kOneRun] - ev_p[i] > 2 * NP;
      if (!sparse) break;  // the sums are not wanted
      float w = 0.f;
#pragma unroll
      for (int j = 0; j < kOneRun; ++j) w += i + j < n ? fabsf(ev_v[i + j]) : 0.f;
      run = fmaxf(run, w);
    }
    if (last) break;
    if (!__syncthreads_and(sparse)) {
      sparse = false;
      break;
    }
    cs += EC - kOneRun;
  }
  run = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(run)));  // not negative
  if ((threadIdx.x & 31) == 0) s_run[threadIdx.x >> 5] = run;
  sparse = __syncthreads_and(sparse);
  float low = INFINITY;  // the smallest of the warps' largest runs (of those that are not zero)
#pragma unroll
  for (int w = 0; w < NTH / 32; ++w) {
    const float r = s_run[w];
    run = sparse ? fmaxf(run, r) : 0.f;
    low = fminf(low, r > 0.f ? r : INFINITY);
  }
  const bool even = run <= kOneEven * low;
  // 2^e and 2^-e have to be normal floats
  if (sparse && even && run < 1.0e30f && (run > 1.0e-27f || run == 0.f)) {
    int ex = 0;
    if (run > 0.f) frexpf(run * kOneRoom, &ex);  // run kOneRoom < 2^ex
    const int e = 31 - ex;
    const float scale = __int_as_float((127 + e) << 23), inv = __int_as_float((127 - e) << 23);
    spread_one_word<NP, NTH>(ev_p, ev_d, ev_v, n, Tlen, taps, scale, tile_s);
    for (int64_t c0 = 0; c0 < cs; c0 += EC) {  // the records before the staged chunk
      __syncthreads();
      const int m = (int)min((int64_t)EC, cs - c0);
      stage(c0, m);
      __syncthreads();
      spread_one_word<NP, NTH>(ev_p, ev_d, ev_v, m, Tlen, taps, scale, tile_s);
    }
    __syncthreads();
    write_cells<NTH>(p, grid, a, L, 0, Tlen, [&](int c) { return (float)tile[c] * inv; });
    pdl_trigger();
    return;
  }
  // the tile's scales: sum and maximum of |v| over its records, those of the first
  // chunk from where they are staged
  const int first = cs == 0 ? n : 0;
  float part = 0.f, pmax = 0.f;
  for (int i = threadIdx.x; i < first; i += NTH) {
    part += fabsf(ev_v[i]);
    pmax = fmaxf(pmax, fabsf(ev_v[i]));
  }
  for (int64_t i = first + threadIdx.x; i < ntot; i += NTH) {
    int pp;
    float dd, vv;
    load_record<float>(rb0, rd, rv, p, tr, L, i, pp, dd, vv);
    part += fabsf(vv);
    pmax = fmaxf(pmax, fabsf(vv));
  }
  const TileScales ts = tile_scales<NTH>(part, pmax, ntot, s_sum, s_max);
  const float inv_h = ts.inv_h, inv_l = ts.inv_l;
  const int half = cells / 2 & ~3;
  // records of the staged chunk before `cell` (they are sorted)
  auto before = [&](int cell, int m) {
    int lo = 0, hi = m;
    while (lo < hi) {
      const int mid = (lo + hi) >> 1;
      if (ev_p[mid] < cell) lo = mid + 1;
      else hi = mid;
    }
    return lo;
  };
  int64_t from = 0;  // the part's first record
  for (int s0 = 0; s0 < Tlen; s0 += half) {
    const int len = min(half, Tlen - s0);
    const bool more = s0 + half < Tlen;  // another part follows
    int64_t next = ntot;
    if (s0 > 0) {
      __syncthreads();
      clear();
    }
    for (int64_t c0 = from; c0 < ntot; c0 += EC) {
      int m = (int)min((int64_t)EC, ntot - c0);
      if (c0 > 0 || s0 > 0 || first == 0) {  // else staged already
        __syncthreads();
        stage(c0, m);
      }
      __syncthreads();
      const int staged = m;
      if (more) {
        const int q = before(s0 + half - p.khi, staged);
        if (q < staged && next == ntot) next = c0 + q;
        m = before(s0 + half - p.klo, staged);
      }
      spread_chunk<NT, NTH>(ev_p, ev_d, ev_v, m, len, p.klo - s0, poly, ts, tile_s, tile_s + 4u * half, AllCells{});
      if (m < staged) break;  // uniform: the rest lies beyond the part
    }
    from = next;
    __syncthreads();
    write_cells<NTH>(p, grid, a, L, s0, len,
                     [&](int c) { return fmaf((float)tile[half + c], inv_l, (float)tile[c] * inv_h); });
  }
  pdl_trigger();
}

bool spread_poly_supported(int ntaps) {
  return ntaps == 9 || ntaps == 13 || ntaps == 14 || (ntaps >= 1 && ntaps <= kPolyMaxTaps);
}

cudaError_t launch_spread_poly(const int64_t* off, const int* rb0, const void* rd, const void* rv,
                               const SpreadParams& p, const KernelPoly& poly, float* grid, const int* status,
                               cudaStream_t s) {
  if (p.tile > spread_max_tile(false)) return cudaErrorInvalidValue;
  const int nt = p.khi - p.klo + 1;
  PairTaps taps{};
  taps.npair = p.khi;  // tap k = 1 .. M_sp pairs with 1 - k
  for (int k = 1; k <= p.khi; ++k) {
    const float* c = poly.c[k - p.klo];
    for (int i = 0; i <= kPolyDeg / 2; ++i) taps.e[k - 1][i] = c[2 * i];
    for (int i = 0; i < kPolyDeg / 2; ++i) taps.o[k - 1][i] = c[2 * i + 1];
  }
  if (p.klo == -p.khi) {
    for (int i = 0; i <= kPolyDeg; ++i) {
      taps.left[i] = poly.c[0][i];
      if (poly.c[0][i] != 0.0f) taps.has_left = 1;
    }
  }
  // staged records, then the tile: a word per cell, two while 4096 words hold
  // them (a small grid's only tile may be dense)
  const int tpad = (p.tile + 3) & ~3;
  const int cells = std::max({tpad, std::min(2 * tpad, 4096), 8});
  dim3 grd(p.ntiles, p.D);
  auto go = [&](auto fn, int nth, int chunk) -> cudaError_t {
    const size_t smem = (size_t)chunk * (sizeof(int) + 2 * sizeof(float)) + (size_t)cells * sizeof(int);
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    return launch_pdl(fn, grd, dim3(nth), smem, s, off, rb0, (const float*)rd, (const float*)rv,
                      (const int*)(status + 1), p, poly, taps, cells, p.dense, grid);
  };
  // tap counts without an instantiation: the next one up, padded with zero taps
  // (18 to 22 taps in the 32-tap one: 116 -> 156 us for 100 dense rows of 20,000 records)
  auto pick = [&](auto w) -> cudaError_t {
    constexpr int NTH = decltype(w)::value, EC = PolyBlock<NTH>::chunk;
    if (nt <= 9) return go(k_spread_poly<9, 4, NTH>, NTH, EC);
    if (nt <= 13) return go(k_spread_poly<13, 6, NTH>, NTH, EC);
    if (nt <= 14) return go(k_spread_poly<14, 7, NTH>, NTH, EC);
    if (nt <= 16) return go(k_spread_poly<16, 8, NTH>, NTH, EC);
    if (nt <= 24) return go(k_spread_poly<24, 12, NTH>, NTH, EC);
    if (nt <= 32) return go(k_spread_poly<32, 16, NTH>, NTH, EC);
    return cudaErrorInvalidValue;
  };
  const int64_t blocks = (int64_t)p.ntiles * p.D;
  if (p.asset_events > (int64_t)kPolyManyRecords * p.ntiles || blocks < kPolyBlocksSome)
    return pick(std::integral_constant<int, 512>{});
  if (blocks < kPolyBlocksMany) return pick(std::integral_constant<int, 256>{});
  return pick(std::integral_constant<int, 128>{});
}

// FP64 scatter in float pairs. The float64 pipe issues about two operations per
// clock and SM, a sixty-fourth of the float32 rate, so a stencil point of some
// sixty float64 operations (exponential and root, then a compare-and-swap loop
// in shared memory) set this stage's time: 1095 us on the block workload (766,162 records,
// 19 points each), 1250 us for 1024 small problems of three assets. Here a tap costs about
// 100 float32 operations instead: the even and odd polynomials of PairPoly (two
// taps each) by Horner's rule in float pairs h + l, the leading coefficients of
// which need one float only; the product with the return; and an accumulation
// that stays exact in three int32 words, as k_spread_poly's in two. Now 75 us and
// 97 us. The grid leaves as float pairs, which the FFT passes keep.
//
// Error: against the kernel in 64 bits a tap is off by at most 7e-15 of the peak
// (8e-16 rms; measured for the three kernels at tol 1e-12). With the FFT's rounding
// that is some 1e-14 of a coefficient before the deconvolution, whose largest factor
// decides where the path is taken (configure); tolerances below 1e-12 keep
// float64 throughout.
//
// Scales: V = max |v| < 2^exV over the tile's n records (from exponent fields:
// returns of any float64 magnitude), eh = 21 - exV - max(0, bitlen(n) - 9), so
// every |x| = |v phi 2^eh| < 2^21 and a cell's hi sum stays below 2^30. x = p + e
// (p the rounded leading product, |e| < 0.6): hi = round(p); the residues of hi
// and e, times 2^k, are rounded into mid (|mid| < 1.2 2^k + 2 a tap), their
// residues times 2^k into lo (likewise). k = min(20, 30 - bitlen(m)) for the m
// records of a staged chunk keeps a chunk's mid and lo sums below 2^31; between
// chunks lo carries into mid and mid into hi. The quantum is 2^-(eh + 2k) (V 2^-60
// for tiles of up to 511 records, V 2^-53 at 30,000), and no sum rounds.
// c + r y
__device__ __forceinline__ FloatPair pair_step(FloatPair r, FloatPair y, float ch, float cl) {
  const float p = __fmul_rn(r.h, y.h), e = __fmaf_rn(r.h, y.h, -p);
  const float s = __fadd_rn(ch, p), b = __fsub_rn(s, ch);
  const float t = __fadd_rn(__fsub_rn(ch, __fsub_rn(s, b)), __fsub_rn(p, b));
  return {s, __fadd_rn(__fmaf_rn(r.l, y.h, __fmaf_rn(r.h, y.l, cl)), __fadd_rn(e, t))};
}
__device__ __forceinline__ FloatPair pair_poly(const float* __restrict__ c, FloatPair y) {
  float top = c[2 * kPairWide + (kPairDeg - kPairWide)];
#pragma unroll
  for (int i = kPairDeg - 1; i >= kPairWide; --i) top = __fmaf_rn(top, y.h, c[kPairWide + i]);
  FloatPair r{top, 0.0f};
#pragma unroll
  for (int i = kPairWide - 1; i >= 0; --i) r = pair_step(r, y, c[i], c[kPairWide + i]);
  return r;
}

constexpr int kPairChunk = 1024;  // records staged per pass

struct Words {
  int hi, mid, lo;
};
// The three words of v w (v and w float pairs, |v w| < 2^21).
__device__ __forceinline__ Words tap_words(FloatPair v, FloatPair w, float K) {
  const float p = __fmul_rn(v.h, w.h);
  const float e = __fmaf_rn(v.h, w.l, __fmaf_rn(v.l, w.h, __fmaf_rn(v.h, w.h, -p)));
  const float th = __fadd_rn(p, kRoundMagic);
  const float r = __fsub_rn(p, __fsub_rn(th, kRoundMagic));
  const float tr = __fmaf_rn(r, K, kRoundMagic), te = __fmaf_rn(e, K, kRoundMagic);
  const float r2 = __fmaf_rn(r, K, -__fsub_rn(tr, kRoundMagic)), e2 = __fmaf_rn(e, K, -__fsub_rn(te, kRoundMagic));
  const float tl = __fmaf_rn(__fadd_rn(r2, e2), K, kRoundMagic);
  return {__float_as_int(th) - kRoundMagicBits,
          __float_as_int(tr) - kRoundMagicBits + (__float_as_int(te) - kRoundMagicBits),
          __float_as_int(tl) - kRoundMagicBits};
}

__global__ void __launch_bounds__(kSpreadThreads, 4) k_spread_pair(const int64_t* __restrict__ off,
                                                               const int* __restrict__ rb0,
                                                               const double* __restrict__ rd,
                                                               const double* __restrict__ rv,
                                                               const int* __restrict__ gate, SpreadParams p,
                                                               const __grid_constant__ PairPoly poly,
                                                               const int* __restrict__ row_exp,
                                                               FloatPair* __restrict__ grid) {
  constexpr int EC = kPairChunk;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  double* ev_d = reinterpret_cast<double*>(smem_raw);
  double* ev_v = ev_d + EC;
  int* ev_p = reinterpret_cast<int*>(ev_v + EC);
  const int tpad = (p.tile + 3) & ~3;
  int* tile = ev_p + EC;  // hi, mid and lo tiles
  const uint32_t tile_s = (uint32_t)__cvta_generic_to_shared(tile);
  __shared__ int s_max[kSpreadThreads / 32];
  const int64_t L = (int64_t)blockIdx.x * p.tile;
  const int Tlen = (int)min((int64_t)p.tile, p.Mr - L);
  for (int c = threadIdx.x; c < 3 * tpad / 4; c += kSpreadThreads)
    reinterpret_cast<int4*>(tile)[c] = make_int4(0, 0, 0, 0);
  pdl_wait();         // the records come from the prep kernel
  if (*gate) return;  // uniform: the whole block leaves
  const int a = p.order ? p.order[blockIdx.y] : (int)blockIdx.y;
  TileRanges tr;
  tile_ranges(off, rb0, p, a, L, Tlen, tr);
  const int64_t ntot = tr.n2 + tr.n1 + tr.n0;
  // the largest exponent field of the tile's returns (staged with the first
  // chunk when one chunk holds them all, else a pass over the returns)
  int top = 0;
  const int n_first = (int)min((int64_t)EC, ntot);
  for (int i = threadIdx.x; i < n_first; i += kSpreadThreads) {
    load_record<double>(rb0, rd, rv, p, tr, L, i, ev_p[i], ev_d[i], ev_v[i]);
    top = max(top, (__double2hiint(ev_v[i]) >> 20) & 0x7FF);
  }
  for (int64_t i = EC + threadIdx.x; i < ntot; i += kSpreadThreads) {
    int pp;
    double dd, vv;
    load_record<double>(rb0, rd, rv, p, tr, L, i, pp, dd, vv);
    top = max(top, (__double2hiint(vv) >> 20) & 0x7FF);
  }
  top = __reduce_max_sync(0xffffffffu, top);
  if ((threadIdx.x & 31) == 0) s_max[threadIdx.x >> 5] = top;
  __syncthreads();
#pragma unroll
  for (int w = 0; w < kSpreadThreads / 32; ++w) top = max(top, s_max[w]);
  const int bitlen = 64 - __clzll((long long)ntot);
  const int eh = 21 - (top - 1022) - max(0, bitlen - 9);
  const int kk = min(20, 30 - (32 - __clz(n_first)));
  const float K = __int_as_float((127 + kk) << 23);
  const bool left = poly.one_sided != 0;
  for (int64_t cs = 0; cs < ntot; cs += EC) {
    const int n = (int)min((int64_t)EC, ntot - cs);
    if (cs > 0) {
      __syncthreads();
      for (int c = threadIdx.x; c < Tlen; c += kSpreadThreads) {
        const int lo = tile[c + 2 * tpad], mid = tile[c + tpad] + (lo >> kk);
        tile[c + 2 * tpad] = lo & ((1 << kk) - 1);
        tile[c + tpad] = mid & ((1 << kk) - 1);
        tile[c] += mid >> kk;
      }
      for (int i = threadIdx.x; i < n; i += kSpreadThreads)
        load_record<double>(rb0, rd, rv, p, tr, L, cs + i, ev_p[i], ev_d[i], ev_v[i]);
    }
    __syncthreads();
    for (int e0 = threadIdx.x & ~31; e0 < n; e0 += kSpreadThreads) {
      const int e = e0 + (threadIdx.x & 31);
      const bool live = e < n && ev_p[e < n ? e : 0] != kNoCell;
      const int pe = live ? ev_p[e] : kNoCell;
      // a warp of records in one cell (dense tiles) adds its sum once
      const bool same = __all_sync(0xffffffffu, pe == __shfl_sync(0xffffffffu, pe, 0));
      if (same && pe == kNoCell) continue;  // uniform
      FloatPair z{0.0f, 0.0f}, v{0.0f, 0.0f};
      if (live) {
        const double zz = ev_d[e];
        z = {__int_as_float(__double2hiint(zz)), __int_as_float(__double2loint(zz))};
        // v 2^eh from the exponent field (a subnormal return's after 54 binary
        // places up); more than 2^1000 below V: zero
        long long b = __double_as_longlong(ev_v[e]);
        int ex = (int)((b >> 52) & 0x7FF), up = eh;
        if (ex == 0) {
          b = __double_as_longlong(ev_v[e] * 18014398509481984.0);  // 2^54
          ex = (int)((b >> 52) & 0x7FF);
          up = eh - 54;
        }
        if (ex > 0 && ex + up > 0) split_f64(__longlong_as_double(b + ((long long)up << 52)), v.h, v.l);
      }
      const float yh = __fmul_rn(z.h, z.h);
      const FloatPair y{yh, __fmaf_rn(z.l, z.l, __fmaf_rn(__fadd_rn(z.h, z.h), z.l, __fmaf_rn(z.h, z.h, -yh)))};
#pragma unroll 1
      for (int q = 0; q < poly.npair; ++q) {
        const FloatPair E = pair_poly(poly.c[q][0], y), O = pair_poly(poly.c[q][1], y);
        const float m = __fmul_rn(z.h, O.h);
        const float ml = __fmaf_rn(z.h, O.l, __fmaf_rn(z.l, O.h, __fmaf_rn(z.h, O.h, -m)));
#pragma unroll
        for (int side = 0; side < 2; ++side) {  // tap 1 - k, then k = q + 1
          if (side == 1 && left && q == poly.npair - 1) break;  // uniform
          const float mh = side ? -m : m, mlo = side ? -ml : ml;
          const float s = __fadd_rn(E.h, mh), bb = __fsub_rn(s, E.h);
          const float t = __fadd_rn(__fsub_rn(E.h, __fsub_rn(s, bb)), __fsub_rn(mh, bb));
          const FloatPair w{s, __fadd_rn(__fadd_rn(t, E.l), mlo)};
          Words x = tap_words(v, w, K);
          const unsigned c = (unsigned)(pe + (side ? q + 1 : -q));
          bool take = live && c < (unsigned)Tlen;
          if (same) {
            x.hi = __reduce_add_sync(0xffffffffu, x.hi);
            x.mid = __reduce_add_sync(0xffffffffu, x.mid);
            x.lo = __reduce_add_sync(0xffffffffu, x.lo);
            take = take && (threadIdx.x & 31) == 0;
          }
          if (take) {
            red_shared_add(tile_s + 4u * c, x.hi);
            red_shared_add(tile_s + 4u * (c + tpad), x.mid);
            red_shared_add(tile_s + 4u * (c + 2 * tpad), x.lo);
          }
        }
      }
    }
  }
  __syncthreads();
  // cells: (hi + (mid + lo 2^-k) 2^-k) 2^-eh as float pairs, scaled by the row's
  // largest exponent, from the exact integers: the leading 24 bits of A = hi 2^k +
  // mid, then the rest and lo
  FloatPair* g = grid + (int64_t)a * p.Mr + L;
  const int sa = -(eh + kk) - (row_exp[a] - 1022);  // returns of the row scaled below 1
  const bool plain = sa >= -80;
  const float unit = plain ? __int_as_float((127 + sa) << 23) : 1.0f;
  for (int c = threadIdx.x; c < Tlen; c += kSpreadThreads) {
    const long long A = ((long long)tile[c] << kk) + tile[c + tpad];
    const float below = (float)tile[c + 2 * tpad] * __int_as_float((127 - kk) << 23);
    const float h = (float)A;  // rounded to 24 bits: A - h is exact in 63 bits and has few left
    const float l = (float)(A - (long long)h) + below;
    if (plain) g[c] = FloatPair(h * unit, l * unit);
    else g[c] = FloatPair(ldexpf(h, sa), ldexpf(l, sa));
  }
}

cudaError_t launch_spread_pair(const int64_t* off, const int* rb0, const void* rd, const void* rv,
                               const SpreadParams& p, const PairPoly& poly, const int* row_exp, void* grid,
                               const int* status,
                               cudaStream_t s) {
  if (p.tile > spread_max_tile(true)) return cudaErrorInvalidValue;
  const size_t smem = (size_t)kPairChunk * (2 * sizeof(double) + sizeof(int)) + 3 * (((size_t)p.tile + 3) / 4 * 16);
  const cudaError_t e = cudaFuncSetAttribute(k_spread_pair, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  return launch_pdl(k_spread_pair, dim3(p.ntiles, p.D), dim3(kSpreadThreads), smem, s, off, rb0, (const double*)rd,
                    (const double*)rv, (const int*)(status + 1), p, poly, row_exp, (FloatPair*)grid);
}

template <typename T, int K>
static cudaError_t launch_variant(bool gather, int nk, dim3 grd, const int64_t* off, const int* rb0, const T* rd,
                                  const T* rv, const int* gate, const SpreadParams& p, T* grid, cudaStream_t s) {
  constexpr int CPT = sizeof(T) == 4 ? 16 : 8;
  const size_t ev_bytes = (size_t)EvChunk<T>::n * (sizeof(int) + 2 * sizeof(T));
  auto go = [&](auto fn, size_t smem) -> cudaError_t {
    if (smem > 48 * 1024) {
      cudaError_t r = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
      if (r != cudaSuccess) return r;
    }
    fn<<<grd, kSpreadThreads, smem, s>>>(off, rb0, rd, rv, gate, p, grid);
    return cudaGetLastError();
  };
  if (gather) return go(k_spread_gather<T, K, CPT>, ev_bytes);
  const size_t smem = ev_bytes + (size_t)p.tile * sizeof(T);
  if (nk <= 8) return go(k_spread_scatter<T, K, 8>, smem);
  if (nk <= 16) return go(k_spread_scatter<T, K, 16>, smem);
  if (nk <= 32) return go(k_spread_scatter<T, K, 32>, smem);
  return cudaErrorInvalidValue;
}

template <typename T>
static cudaError_t launch_spread_t(const int64_t* off, const int* rb0, const void* rd, const void* rv,
                                   const SpreadParams& p, T* grid, const int* status, cudaStream_t s) {
  constexpr int CPT = sizeof(T) == 4 ? 16 : 8;
  if (p.tile > kSpreadThreads * CPT) return cudaErrorInvalidValue;
  dim3 grd(p.ntiles, p.D);
  const int* gate = status + 1;
  const bool gather = p.algo == 1;
  const int nk = p.khi - p.klo + 1;
  const T* d = (const T*)rd;
  const T* v = (const T*)rv;
  switch (p.kernel) {
    case MM_KERNEL_GAUSS: return launch_variant<T, MM_KERNEL_GAUSS>(gather, nk, grd, off, rb0, d, v, gate, p, grid, s);
    case MM_KERNEL_KB: return launch_variant<T, MM_KERNEL_KB>(gather, nk, grd, off, rb0, d, v, gate, p, grid, s);
    case MM_KERNEL_ES: return launch_variant<T, MM_KERNEL_ES>(gather, nk, grd, off, rb0, d, v, gate, p, grid, s);
    default: return cudaErrorInvalidValue;
  }
}

int spread_max_tile(bool fp64) { return kSpreadThreads * (fp64 ? 8 : 16); }

cudaError_t launch_spread_f32(const int64_t* off, const int* rb0, const void* rd, const void* rv,
                              const SpreadParams& p, float* grid, const int* status, cudaStream_t s) {
  return launch_spread_t<float>(off, rb0, rd, rv, p, grid, status, s);
}
cudaError_t launch_spread_f64(const int64_t* off, const int* rb0, const void* rd, const void* rv,
                              const SpreadParams& p, double* grid, const int* status, cudaStream_t s) {
  return launch_spread_t<double>(off, rb0, rd, rv, p, grid, status, s);
}

}  // namespace mmgpu
