// mm_epps.cu -- the cutoff sweep of the batched form: for every problem of a
// batch (G problems of Dg assets each) and every cutoff N_j of an ascending
// list, the covariance and correlation of Algorithm 3 step C (Eqs. (2), (3))
// from ONE set of coefficients computed at N_max = max_j N_j.
//
// Prefix-weighted contraction. With the Hermitian half (the -k term of each
// pair k, -k folded into a factor 2 for k >= 1, no factor for k = 0) and
// Q_k = Re(F(k) F(k)^H) (a Dg x Dg matrix),
//   Dirichlet  Sigma(N) = (2 pi)^2 / (2N + 1) * P(N),
//   Fejer      Sigma(N) = (2 pi)^2 / ((N + 1) N) * sum_{k<=N} d_k (N - k) Q_k,
//   P(N) = sum_{k<=N} d_k Q_k,  d_0 = 1, d_k = 2.
// One pass over k accumulates, for each segment s = (e_{s-1}, e_s] of the
// cutoff list, S_s = sum d_k Q_k and T_s = sum d_k (e_s - k) Q_k; then
//   sum_{k<=N_j} d_k (N_j - k) Q_k = sum_{s<=j} ((N_j - e_s) S_s + T_s)
//                                  = A_j + sum_{s<=j} T_s,
//   A_j = A_{j-1} + (e_j - e_{j-1}) P_{j-1},  P_j = P_{j-1} + S_j,
// every cutoff from one contraction at N_max plus O(#cutoffs Dg^2) additions.
// All weights here are non-negative, so a diagonal entry is a sum of
// non-negative terms: the form P(N) - sum d_k k Q_k / N, which cancels when
// Q_0 dominates (a small total return at N = 1), is not used.
//
// A problem's modes are cut into work items on the host (epps_items), for warps
// of one CTA, or of S CTAs when there are fewer problems than the GPU wants:
//  * long items: up to chunk modes inside one segment. The lanes step through
//    the modes (coalesced loads of the Dg coefficients F_i(k)) adding the
//    Dg (Dg+1)/2 products into registers; one transposed shuffle reduction (each
//    step halves the sums a lane holds) leaves each lane its own sums to add
//    to the segment's in shared memory.
//  * short items: 32 modes that hold two segment ends or more, one mode a lane,
//    a segmented scan per pair of assets; the last lane of each segment adds.
// Accumulation is float32 within an item's segment; the prefix over the
// segments, the weights and the diagonal normalisation are float64. The FP64
// form (the comparator of the mixed one) runs the same sweep on complex128
// coefficients with float64 accumulation and float64 Sigma and R.
// Bound by the coefficients' reads when items are long, else by the reductions:
// a chunk of one segment with five shuffles per pair took 347 us at 512
// problems of 10 assets, 64 cutoffs to 14,399 (590 MB), and 232 us at 16
// problems on one CTA each; now 206 us and 73 us.
//
// Small problems (k_epps_small: float32, at most 4 assets and 511 modes, epps_small)
// take a warp each: one mode a lane, prefix sums over k by a warp scan in float pairs
// (48 bits, as the float64 pipe would bound it), for Fejer the prefix of the
// prefix (sum_{k<=N} (N - k) q_k = sum_{m<N} P(m)); the lane of a cutoff writes
// its Sigma and R. 8192 problems of two assets and 50 cutoffs:
// 690 -> 20 us.
#include <algorithm>
#include <vector>

#include "mm_common.cuh"

namespace mmgpu {

namespace {

constexpr int kEppsThreads = 256;

template <int DG>
struct Pairs {
  static constexpr int n = DG * (DG + 1) / 2;
};

template <typename T> struct Cx;
template <> struct Cx<float> { using type = float2; };
template <> struct Cx<double> { using type = double2; };

// Sums of v[0..N) over the lanes of a warp; lane l is left with the sums of
// indices start .. start + Left - 1 that lie below end.
template <int N, int BIT>
struct LaneSums {
  static constexpr int H = (N + 1) / 2;
  static constexpr int Left = LaneSums<H, BIT / 2>::Left;
  template <typename T>
  static __device__ __forceinline__ void run(T* v, int lane, int& start, int& end) {
    const bool up = (lane & BIT) != 0;
#pragma unroll
    for (int q = 0; q < H; ++q) {
      const T hi = q + H < N ? v[q + H] : (T)0;
      const T keep = up ? hi : v[q], send = up ? v[q] : hi;
      v[q] = keep + __shfl_xor_sync(0xffffffffu, send, BIT);
    }
    if (up) start += H;
    else end = min(end, start + H);
    LaneSums<H, BIT / 2>::run(v, lane, start, end);
  }
};
template <int N>
struct LaneSums<N, 0> {
  static constexpr int Left = N;
  template <typename T>
  static __device__ __forceinline__ void run(T*, int, int&, int&) {}
};
template <int N, typename T>
__device__ __forceinline__ void add_lane_sums(T* v, T* dst, int lane) {
  int start = 0, end = N;
  LaneSums<N, 16>::run(v, lane, start, end);
#pragma unroll
  for (int q = 0; q < LaneSums<N, 16>::Left; ++q)
    if (start + q < end) atomicAdd(dst + start + q, v[q]);
}

// 1 / sqrt(d) for the normalisation in T: float32 from the approximate
// reciprocal root and one Newton step in float64 (relative error 2^-41).
__device__ __forceinline__ float inv_root(double d, float) {
  const float f = (float)d;
  if (!(f > 1.0e-37f && f < 1.0e37f)) return (float)rsqrt(d);
  const double y = (double)rsqrtf(f);
  return (float)(y * fma(-0.5 * d, y * y, 1.5));
}
__device__ __forceinline__ double inv_root(double d, double) { return rsqrt(d); }

// Two CTAs an SM where the sums fit 128 registers a thread.
template <typename T, int DG, bool FEJER>
constexpr int kEppsPerSm = Pairs<DG>::n * (FEJER ? 2 : 1) * (int)(sizeof(T) / 4) <= 80 ? 2 : 1;

template <typename T, int DG, bool FEJER>
__global__ void __launch_bounds__(kEppsThreads, kEppsPerSm<T, DG, FEJER>) k_epps(const typename Cx<T>::type* __restrict__ coef, int ld,
                                                       const int* __restrict__ cut_g, int ncut,
                                                       const int2* __restrict__ items, int nitems,
                                                       T* __restrict__ part, int* __restrict__ arrived,
                                                       T* __restrict__ sigma, T* __restrict__ Rout,
                                                       const int* __restrict__ gate, int* status) {
  using C2 = typename Cx<T>::type;
  constexpr int NP = Pairs<DG>::n;
  constexpr int NS = FEJER ? 2 : 1;
  constexpr int NW = kEppsThreads / 32;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* sacc = reinterpret_cast<T*>(smem_raw);  // [NS][ncut][NP]
  double* ssig =
      reinterpret_cast<double*>(smem_raw + (((size_t)NS * ncut * NP * sizeof(T) + 15) & ~(size_t)15));  // [ncut][NP]
  __shared__ int scut[kMaxCutoffs];
  __shared__ double swt[kMaxCutoffs];                      // basis weight per cutoff
  __shared__ T sinv[kMaxCutoffs * DG];                     // 1 / sqrt(Sigma_aa(N_j))
  __shared__ int s_last;
  if (*gate) return;  // uniform
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int i = threadIdx.x; i < ncut; i += kEppsThreads) {
    const int c = cut_g[i];
    scut[i] = c;
    const double four_pi2 = 4.0 * kPi * kPi;
    swt[i] = FEJER ? four_pi2 / (((double)c + 1.0) * (double)c) : four_pi2 / (2.0 * (double)c + 1.0);
  }
  const int nacc = NS * ncut * NP;
  for (int i = threadIdx.x; i < nacc; i += kEppsThreads) sacc[i] = (T)0;
  __syncthreads();
  int zero_var = 0;
  const int g = blockIdx.x, S = gridDim.y;
  const C2* cg = coef + (size_t)g * DG * ld;
  // first segment whose end is at or beyond k
  auto segment_of = [&](int k) {
    int lo = 0, hi = ncut - 1;
    while (lo < hi) {
      const int mid = (lo + hi) >> 1;
      if (scut[mid] >= k) hi = mid;
      else lo = mid + 1;
    }
    return lo;
  };
  for (int it = blockIdx.y * NW + warp; it < nitems; it += S * NW) {
    const int2 item = __ldg(items + it);
    const int kb = item.x;
    C2 c[DG];
    if (item.y > 0) {
      const int ke = item.y;
      const int sj = segment_of(kb);  // the whole item
      const int es = scut[sj];        // the segment's end cutoff: weights e_s - k >= 0
      T acc[NP], acc1[FEJER ? NP : 1];
#pragma unroll
      for (int p = 0; p < NP; ++p) acc[p] = (T)0;
#pragma unroll
      for (int p = 0; p < (FEJER ? NP : 1); ++p) acc1[p] = (T)0;
      for (int k = kb + lane; k < ke; k += 32) {
#pragma unroll
        for (int i = 0; i < DG; ++i) c[i] = __ldg(cg + (size_t)i * ld + k);
        if (kb == 0 && k == 0) {  // d_0 = 1, d_k = 2: the items sum halves
#pragma unroll
          for (int i = 0; i < DG; ++i) {
            c[i].x *= (T)0.70710678118654752;
            c[i].y *= (T)0.70710678118654752;
          }
        }
        const T kf = (T)(es - k);
        int p = 0;
#pragma unroll
        for (int i = 0; i < DG; ++i)
#pragma unroll
          for (int j = i; j < DG; ++j, ++p) {
            if (FEJER) {
              const T q = fma(c[i].x, c[j].x, c[i].y * c[j].y);
              acc[p] += q;
              acc1[p] = fma(kf, q, acc1[p]);
            } else {
              acc[p] = fma(c[i].x, c[j].x, fma(c[i].y, c[j].y, acc[p]));
            }
          }
      }
      add_lane_sums<NP>(acc, sacc + sj * NP, lane);
      if (FEJER) add_lane_sums<NP>(acc1, sacc + (ncut + sj) * NP, lane);
    } else {
      const int ke = -item.y;
      const int k = kb + lane;
      const bool in = k < ke;
      const int sj = segment_of(min(k, ke - 1));
      const int first = max(kb, sj ? scut[sj - 1] + 1 : 0);  // first mode of the lane's segment in the item
      const int back = k - first;                            // lanes of the same segment before this one
      const bool last = in && (k == ke - 1 || k == scut[sj]);
#pragma unroll
      for (int i = 0; i < DG; ++i) {
        C2 v;
        v.x = v.y = (T)0;
        if (in) v = __ldg(cg + (size_t)i * ld + k);
        const T h = k == 0 ? (T)0.70710678118654752 : (T)1;
        c[i].x = v.x * h;
        c[i].y = v.y * h;
      }
      const T kf = (T)(scut[sj] - k);
      int p = 0;
#pragma unroll
      for (int i = 0; i < DG; ++i)
#pragma unroll
        for (int j = i; j < DG; ++j, ++p) {
          T q = fma(c[i].x, c[j].x, c[i].y * c[j].y);
          T w = FEJER ? kf * q : (T)0;
#pragma unroll
          for (int o = 1; o < 32; o <<= 1) {
            const T u = __shfl_up_sync(0xffffffffu, q, o);
            if (o <= back) q += u;
            if (FEJER) {
              const T x = __shfl_up_sync(0xffffffffu, w, o);
              if (o <= back) w += x;
            }
          }
          if (last) {
            atomicAdd(&sacc[sj * NP + p], q);
            if (FEJER) atomicAdd(&sacc[(ncut + sj) * NP + p], w);
          }
        }
    }
  }
  __syncthreads();
  if (S > 1) {
    // the problem's last CTA adds the S partial sums in order
    T* slot = part + (size_t)g * S * nacc;
    for (int i = threadIdx.x; i < nacc; i += kEppsThreads) slot[(size_t)blockIdx.y * nacc + i] = sacc[i];
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) s_last = atomicAdd(arrived + g, 1) == S - 1;
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    for (int i = threadIdx.x; i < nacc; i += kEppsThreads) {
      T v = (T)0;
      for (int y = 0; y < S; ++y) v += __ldcg(slot + (size_t)y * nacc + i);
      sacc[i] = v;
    }
    if (threadIdx.x == 0) arrived[g] = 0;
    __syncthreads();
  }
  // prefix over segments with the basis weights (float64), then the
  // diagonal normalisation: 1/sqrt(Sigma_aa) in float64 once per asset and
  // cutoff, the off-diagonal products in float32
  for (int p = threadIdx.x; p < NP; p += kEppsThreads) {
    double P = 0.0, A = 0.0, Ts = 0.0;
    for (int j = 0; j < ncut; ++j) {
      if (FEJER && j > 0) A += (double)(scut[j] - scut[j - 1]) * P;
      P += (double)sacc[j * NP + p];
      if (FEJER) Ts += (double)sacc[(ncut + j) * NP + p];
      ssig[j * NP + p] = 2.0 * (FEJER ? swt[j] * (A + Ts) : swt[j] * P);
    }
  }
  __syncthreads();
  for (int e = threadIdx.x; e < ncut * DG; e += kEppsThreads) {
    const int j = e / DG, a = e - j * DG;
    const double d = ssig[j * NP + a * DG - a * (a - 1) / 2];
    sinv[e] = d > 0.0 ? inv_root(d, (T)0) : (T)__longlong_as_double(0x7ff8000000000000ll);
    if (!(d > 0.0)) zero_var = 1;
  }
  __syncthreads();
  // Sigma and R for every cutoff, both triangles
  for (int e = threadIdx.x; e < ncut * DG * DG; e += kEppsThreads) {
    const int j = e / (DG * DG), r = e - j * DG * DG;
    const int a = r / DG, b = r - a * DG;
    const int lo = a < b ? a : b, hi = a < b ? b : a;
    const int p = lo * DG - lo * (lo - 1) / 2 + (hi - lo);  // index of pair (lo, hi)
    const T sv = (T)ssig[j * NP + p];
    const size_t o = ((size_t)g * ncut + j) * DG * DG + r;
    if (sigma) sigma[o] = sv;
    Rout[o] = a == b ? (sinv[j * DG + a] == sinv[j * DG + a] ? (T)1 : sinv[j * DG + a])
                     : sv * sinv[j * DG + a] * sinv[j * DG + b];
  }
  if (zero_var) atomicOr(status, ST_ZERO_VAR);
}

// ------------------------------------------------------------ small problems
constexpr int kSmallModes = 512;   // cutoffs below this
constexpr int kSmallAssets = 4;

// Float pairs h + l (|l| <= ulp(h) / 2): sum of two (Knuth's two-sum, then the
// low parts; relative error below 2^-46).
struct Pair2 {
  float h, l;
};
__device__ __forceinline__ Pair2 add2(Pair2 a, Pair2 b) {
  const float s = a.h + b.h;
  if (!(fabsf(s) <= 3.402823466e38f)) return {s, 0.f};  // infinite or NaN
  const float bb = s - a.h;
  const float e = (a.h - (s - bb)) + (b.h - bb) + (a.l + b.l);
  const float h = s + e;
  return {h, e - (h - s)};
}
__device__ __forceinline__ Pair2 shfl_up2(Pair2 v, int o) {
  return {__shfl_up_sync(0xffffffffu, v.h, o), __shfl_up_sync(0xffffffffu, v.l, o)};
}
__device__ __forceinline__ Pair2 scan2(Pair2 v, int lane) {
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const Pair2 u = shfl_up2(v, o);
    if (lane >= o) v = add2(u, v);
  }
  return v;
}

template <int DG, bool FEJER>
__global__ void __launch_bounds__(kEppsThreads) k_epps_small(const float2* __restrict__ coef, int ld,
                                                             const int* __restrict__ cut_g, int ncut, int G,
                                                             float* __restrict__ sigma, float* __restrict__ Rout,
                                                             const int* __restrict__ gate, int* status) {
  constexpr int NP = Pairs<DG>::n;
  __shared__ short s_of[kSmallModes];     // cutoff index of mode k, or -1
  __shared__ Pair2 s_w[kMaxCutoffs];      // weight of the cutoff
  if (*gate) return;  // uniform
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int i = threadIdx.x; i < kSmallModes; i += kEppsThreads) s_of[i] = -1;
  __syncthreads();
  for (int i = threadIdx.x; i < ncut; i += kEppsThreads) {
    const int c = cut_g[i];
    const double four_pi2 = 4.0 * kPi * kPi;
    const double w = FEJER ? four_pi2 / (((double)c + 1.0) * (double)c) : four_pi2 / (2.0 * (double)c + 1.0);
    s_of[c] = (short)i;
    s_w[i].h = (float)w;
    s_w[i].l = (float)(w - (double)s_w[i].h);
  }
  __syncthreads();
  const int N = ld - 1;
  int zero_var = 0;
  for (int g = blockIdx.x * (kEppsThreads / 32) + warp; g < G; g += gridDim.x * (kEppsThreads / 32)) {
    const float2* cg = coef + (size_t)g * DG * ld;
    Pair2 P[NP], A[FEJER ? NP : 1];  // sums over the modes before this step
#pragma unroll
    for (int p = 0; p < NP; ++p) P[p] = Pair2{0.f, 0.f};
#pragma unroll
    for (int p = 0; p < (FEJER ? NP : 1); ++p) A[p] = Pair2{0.f, 0.f};
    for (int kb = 0; kb <= N; kb += 32) {
      const int k = kb + lane;
      float2 c[DG];
#pragma unroll
      for (int i = 0; i < DG; ++i) c[i] = k <= N ? __ldg(cg + (size_t)i * ld + k) : make_float2(0.f, 0.f);
      const float d = k == 0 ? 1.f : 2.f;
      Pair2 val[NP];
      int p = 0;
#pragma unroll
      for (int i = 0; i < DG; ++i)
#pragma unroll
        for (int j = i; j < DG; ++j, ++p) {
          // d_k Re(F_i conj F_j) as one rounded product sum, then the scan
          const float q = d * fmaf(c[i].x, c[j].x, c[i].y * c[j].y);
          const Pair2 in = add2(scan2(Pair2{q, 0.f}, lane), P[p]);  // P(k)
          P[p] = Pair2{__shfl_sync(0xffffffffu, in.h, 31), __shfl_sync(0xffffffffu, in.l, 31)};
          if (FEJER) {
            const Pair2 run = add2(scan2(in, lane), A[p]);  // sum_{m <= k} P(m)
            const Pair2 prev = shfl_up2(run, 1);
            val[p] = lane ? prev : A[p];  // sum_{m < k} P(m)
            A[p] = Pair2{__shfl_sync(0xffffffffu, run.h, 31), __shfl_sync(0xffffffffu, run.l, 31)};
          } else {
            val[p] = in;
          }
        }
      const int j = k <= N ? s_of[k] : -1;
      if (j >= 0) {
        const Pair2 w = s_w[j];
        float sv[NP], inv[DG];
#pragma unroll
        for (int q = 0; q < NP; ++q)
          sv[q] = fabsf(val[q].h) <= 3.402823466e38f
                      ? fmaf(w.h, val[q].h, fmaf(w.h, val[q].l, w.l * val[q].h))
                      : w.h * val[q].h;
#pragma unroll
        for (int a = 0; a < DG; ++a) {
          const float x = sv[a * DG - a * (a - 1) / 2];
          if (x > 1.0e-37f && x < 1.0e37f) {
            const float y = rsqrtf(x);
            inv[a] = fmaf(0.5f * y, fmaf(-(x * y), y, 1.0f), y);
          } else {
            inv[a] = x > 0.f ? (float)rsqrt((double)x) : __int_as_float(0x7fc00000);
            if (!(x > 0.f)) zero_var = 1;
          }
        }
        const size_t o = ((size_t)g * ncut + j) * DG * DG;
        float sg[DG * DG], rr[DG * DG];
#pragma unroll
        for (int a = 0; a < DG; ++a)
#pragma unroll
          for (int b = 0; b < DG; ++b) {
            const int lo = a < b ? a : b, hi = a < b ? b : a;
            const float v = sv[lo * DG - lo * (lo - 1) / 2 + (hi - lo)];
            sg[a * DG + b] = v;
            rr[a * DG + b] = a == b ? (inv[a] == inv[a] ? 1.f : inv[a]) : v * inv[lo] * inv[hi];
          }
        // rows of DG^2 floats; even DG: whole 16-byte vectors of an aligned output
        const bool vec = DG % 2 == 0 && (((uintptr_t)Rout | (sigma ? (uintptr_t)sigma : 0)) & 15) == 0;
        if (vec) {
#pragma unroll
          for (int q = 0; q + 4 <= DG * DG; q += 4) {
            if (sigma) *reinterpret_cast<float4*>(sigma + o + q) = make_float4(sg[q], sg[q + 1], sg[q + 2], sg[q + 3]);
            *reinterpret_cast<float4*>(Rout + o + q) = make_float4(rr[q], rr[q + 1], rr[q + 2], rr[q + 3]);
          }
        } else {
#pragma unroll
          for (int q = 0; q < DG * DG; ++q) {
            if (sigma) sigma[o + q] = sg[q];
            Rout[o + q] = rr[q];
          }
        }
      }
    }
  }
  if (zero_var) atomicOr(status, ST_ZERO_VAR);
}

// A warp a problem is a chain of 32-mode steps, each a scan per pair of assets: 7 us
// to 250 us by its length, however few the problems. So it is taken for short chains,
// and for long ones from as many problems on as keep CTAs of the other form busy for
// longer. Steps times (pairs + 1), both forms measured at 1 to 4 assets, 20 to 511 modes
// and 4 to 8192 problems (us, a warp each against CTAs): 4 assets, 511 modes, 32 problems
// 74 against 15; 2 assets, 200 modes, 150 problems 25 against 14; 3 assets, 50 modes, 600
// problems 12 against 18; 2 assets, 350 modes, 2500 problems 30 against 41.
constexpr int kSmallShort = 12;      // chains that are always shorter
constexpr int kSmallLong = 128;      // and never
constexpr int kSmallPerStep = 28;    // problems per step between the two

bool epps_small(int Dg, int ld, int G) {
  if (Dg > kSmallAssets || ld > kSmallModes) return false;
  const int chain = (Dg * (Dg + 1) / 2 + 1) * ((ld + 31) / 32);
  return chain <= kSmallShort || (chain <= kSmallLong && G >= kSmallPerStep * chain);
}

template <typename T, int DG>
cudaError_t launch_dg(bool fejer, const EppsArgs& a, cudaStream_t s) {
  constexpr int NP = Pairs<DG>::n;
  const int* gate = a.status + 1;
  if constexpr (sizeof(T) == 4 && DG <= kSmallAssets) {
    if (epps_small(DG, a.ld, a.G)) {
      const int grid = std::min((a.G + 7) / 8, 6 * 152);
      auto small = [&](auto fn) {
        fn<<<grid, kEppsThreads, 0, s>>>((const float2*)a.coef, a.ld, a.cut, a.ncut, a.G, (float*)a.sigma,
                                         (float*)a.R, gate, a.status);
        return cudaGetLastError();
      };
      return fejer ? small(k_epps_small<DG, true>) : small(k_epps_small<DG, false>);
    }
  }
  const int NS = fejer ? 2 : 1;
  const size_t smem = (((size_t)NS * a.ncut * NP * sizeof(T) + 15) & ~(size_t)15) + (size_t)a.ncut * NP * 8;
  auto go = [&](auto fn) -> cudaError_t {
    // static + dynamic shared memory may pass 48 KB: always opt in
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    fn<<<dim3(a.G, a.splits), kEppsThreads, smem, s>>>((const typename Cx<T>::type*)a.coef, a.ld, a.cut, a.ncut,
                                                       (const int2*)a.items, a.nitems, (T*)a.part, a.arrived,
                                                       (T*)a.sigma, (T*)a.R, gate, a.status);
    return cudaGetLastError();
  };
  return fejer ? go(k_epps<T, DG, true>) : go(k_epps<T, DG, false>);
}

template <typename T>
cudaError_t launch_t(int Dg, bool fejer, const EppsArgs& a, cudaStream_t s) {
  switch (Dg) {
    case 1: return launch_dg<T, 1>(fejer, a, s);
    case 2: return launch_dg<T, 2>(fejer, a, s);
    case 3: return launch_dg<T, 3>(fejer, a, s);
    case 4: return launch_dg<T, 4>(fejer, a, s);
    case 5: return launch_dg<T, 5>(fejer, a, s);
    case 6: return launch_dg<T, 6>(fejer, a, s);
    case 7: return launch_dg<T, 7>(fejer, a, s);
    case 8: return launch_dg<T, 8>(fejer, a, s);
    case 9: return launch_dg<T, 9>(fejer, a, s);
    case 10: return launch_dg<T, 10>(fejer, a, s);
    case 11: return launch_dg<T, 11>(fejer, a, s);
    case 12: return launch_dg<T, 12>(fejer, a, s);
    default: return cudaErrorInvalidValue;
  }
}

// Two CTAs an SM.
constexpr int kEppsCtas = 2 * 152;

}  // namespace

int epps_max_assets() { return kMaxEppsAssets; }

// CTAs per problem: as many as fill the GPU twice over when there are fewer
// problems than CTAs (16 problems on one CTA each: 232 us; on 10 each,
// as many as its items feed: 73 us), no more than there are items for.
int epps_splits(int G, int nitems) {
  if (G >= kEppsCtas) return 1;
  return std::max(1, std::min(kEppsCtas / G, (nitems + kEppsThreads / 32 - 1) / (kEppsThreads / 32)));
}

size_t epps_part_bytes(int Dg, bool fp64, int G) {
  if (G >= kEppsCtas) return 0;
  return (size_t)kEppsCtas * 2 * kMaxCutoffs * (Dg * (Dg + 1) / 2) * (fp64 ? 8 : 4);
}

// The work items of a sweep (pairs k0, k1: modes k0 .. k1 - 1, -k1 for a short
// item): long chunks of 512 modes, 256 when the problems alone do not fill the
// GPU (more warps), and 32-mode short ones where two segments or more end.
std::vector<int> epps_items(const std::vector<int>& cut, int G) {
  const int chunk = G >= kEppsCtas ? 512 : 256;
  const int N = cut.back();
  std::vector<int> out;
  size_t seg = 0;
  for (int k = 0; k <= N;) {
    while (cut[seg] < k) ++seg;
    const int k1 = std::min(k + 32, N + 1);
    int end;
    if (cut[seg] < k1 - 1) {
      end = k1;
      out.push_back(k);
      out.push_back(-end);
    } else {
      end = std::min(k + chunk, cut[seg] + 1);
      out.push_back(k);
      out.push_back(end);
    }
    k = end;
  }
  return out;
}

size_t epps_items_max(int N_max) { return 2 * ((size_t)N_max / 32 + kMaxCutoffs + 2); }

cudaError_t launch_epps(int Dg, bool fejer, bool fp64, const EppsArgs& a, cudaStream_t s) {
  if (a.ncut < 1 || a.ncut > kMaxCutoffs || a.G < 1 || a.splits < 1) return cudaErrorInvalidValue;
  return fp64 ? launch_t<double>(Dg, fejer, a, s) : launch_t<float>(Dg, fejer, a, s);
}

}  // namespace mmgpu
