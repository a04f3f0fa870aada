// mm_pairwise.cu -- covariance with a cutoff per pair of assets and the
// repair to the nearest positive semi-definite matrix (Sec. 3.1: when each
// asset has its own cutoff, e.g. its own Nyquist cutoff in the arrival-time
// representation, each entry is a pairwise estimate, and neither basis then
// guarantees a positive semi-definite matrix).
//
// Sigma_ij is Eq. (2) (Dirichlet) or Eq. (3) (Fejer) at N_ij = min(N_i, N_j)
// from coefficients computed once at max_i N_i:
//   Dirichlet  (2 pi)^2 / (2N + 1)      * sum_{k<=N} d_k Re(F_i(k) conj F_j(k)),
//   Fejer      (2 pi)^2 / ((N + 1) N)   * sum_{k<=N} d_k (N - k) Re(F_i(k) conj F_j(k)),
// d_0 = 1, d_k = 2 (the -k half folded in); every weight is non-negative.
// A CTA takes a 16 x 16 tile of pairs (upper tiles) and every S-th chunk of 128
// modes, the two tiles' coefficient rows staged in shared memory; a thread owns
// one pair, sums a chunk in the coefficients' precision and adds it to a float64
// sum; the last CTA of a tile adds the S partial sums in order. Latency bound
// (staging, then dependent adds): with one CTA per tile, 28 CTAs at D = 100,
// N = 1e4 took 252 us; S filling the SMs takes 34 us.
//
// Repair: the matrix closest to Sigma in the Frobenius norm among the positive
// semi-definite ones is V max(Lambda, 0) V^T (Sigma = V Lambda V^T), the
// eigenvalue method the paper points to. The eigendecomposition is a cyclic
// Jacobi iteration: each step applies D/2 disjoint rotations (round-robin pairing), a
// sweep is D - 1 steps, and the sweeps stop when the off-diagonal norm is below
// 2 D eps of the matrix norm (eps of the working type: float64 for FP64 plans,
// float32 for the mixed precisions' float32 Sigma) or after kJacobiSweeps. GB300
// issues float64 at a small fraction of the float32 rate, so the mixed path
// works in float32.
#include <math.h>

#include <algorithm>

#include "mm_common.cuh"

namespace mmgpu {

namespace {

constexpr int kPT = 16;        // tile edge (pairs per tile: 16 x 16)
constexpr int kPChunk = 128;   // modes staged per chunk
constexpr int kPairwiseCtas = 4 * 152;  // CTAs k_pairwise aims at (33 KB of shared memory each in float32)
constexpr int kJacobiThreads = 1024;
constexpr int kJacobiSweeps = 40;
constexpr int kPsdMaxD = 158;      // the one-CTA iteration (at most kPsdRounds blocks a thread); in float64 the
constexpr int kPsdMaxD64 = 112;    // pipes of all SMs beat those of one beyond this
constexpr int kPsdRounds = 4;

__device__ __forceinline__ void tile_of(int p, int nt, int& I, int& J) {
  int i = 0;
  while (p >= nt - i) {
    p -= nt - i;
    ++i;
  }
  I = i;
  J = i + p;
}

template <typename T2>
__device__ __forceinline__ T2 zero2() {
  T2 z;
  z.x = 0;
  z.y = 0;
  return z;
}

template <typename T2, typename T, bool FEJER>
__global__ void __launch_bounds__(256) k_pairwise(const T2* __restrict__ F, int ld, const int* __restrict__ Nv,
                                                  int D, int nt, double* __restrict__ part, int* __restrict__ done,
                                                  double* __restrict__ sig) {
  __shared__ T2 a[kPT][kPChunk + 1], b[kPT][kPChunk + 1];
  __shared__ int s_nmax, s_last;
  int I, J;
  tile_of(blockIdx.x, nt, I, J);
  const int ti = threadIdx.x / kPT, tj = threadIdx.x % kPT;
  const int i = I * kPT + ti, j = J * kPT + tj;
  const bool valid = i < D && j < D && (I < J || ti <= tj);
  const int Nij = valid ? min(Nv[i], Nv[j]) : -1;
  if (threadIdx.x == 0) s_nmax = -1;
  __syncthreads();
  if (valid) atomicMax(&s_nmax, Nij);
  __syncthreads();
  const int nmax = s_nmax;  // the tile's largest pairwise cutoff
  double acc = 0.0;
  for (int k0 = blockIdx.y * kPChunk; k0 <= nmax; k0 += gridDim.y * kPChunk) {
    for (int e = threadIdx.x; e < kPT * kPChunk; e += blockDim.x) {
      const int r = e / kPChunk, c = e - r * kPChunk;
      const int k = k0 + c;
      const int ra = I * kPT + r, rb = J * kPT + r;
      a[r][c] = (k <= nmax && ra < D) ? F[(size_t)ra * ld + k] : zero2<T2>();
      b[r][c] = (k <= nmax && rb < D) ? F[(size_t)rb * ld + k] : zero2<T2>();
    }
    __syncthreads();
    T part_sum = 0;
    const int cend = min(kPChunk - 1, Nij - k0);  // last mode of this pair in the chunk
    for (int c = 0; c <= cend; ++c) {
      const int k = k0 + c;
      T w = k == 0 ? (T)1 : (T)2;
      if (FEJER) w *= (T)(Nij - k);
      part_sum += w * (a[ti][c].x * b[tj][c].x + a[ti][c].y * b[tj][c].y);
    }
    acc += (double)part_sum;
    __syncthreads();
  }
  if (gridDim.y > 1) {
    // partial sums of this split; the tile's last CTA adds all of them in order
    double* slot = part + (size_t)blockIdx.x * gridDim.y * 256;
    slot[(size_t)blockIdx.y * 256 + threadIdx.x] = acc;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) s_last = atomicAdd(done + blockIdx.x, 1) == (int)gridDim.y - 1;
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    acc = 0.0;
    for (int y = 0; y < (int)gridDim.y; ++y) acc += __ldcg(slot + (size_t)y * 256 + threadIdx.x);
    if (threadIdx.x == 0) done[blockIdx.x] = 0;
  }
  if (valid) {
    const double fp2 = 4.0 * kPi * kPi;
    const double v = acc * (FEJER ? fp2 / (((double)Nij + 1.0) * (double)Nij) : fp2 / (2.0 * Nij + 1.0));
    sig[(size_t)i * D + j] = v;
    sig[(size_t)j * D + i] = v;
  }
}

// The Jacobi iteration (Golub and Van Loan, the cyclic Jacobi algorithm with
// a parallel ordering): rotation (p, q) with tau = (a_qq - a_pp) / (2 a_pq),
// t = sign(tau) / (|tau| + sqrt(1 + tau^2)), c = 1 / sqrt(1 + t^2), s = t c
// zeroes a_pq in J^T A J, J = [[c, s], [-s, c]] on rows and columns p, q.
//
// V accumulates V J; when an eigenvalue is negative Sigma becomes
// V max(Lambda, 0) V^T.
//
// One CTA up to kPsdMaxD (kPsdMaxD64) assets. It is a serial chain of D - 1
// steps a sweep, so a step is kept short, with one barrier:
//  * a step's rotations, i = 0 .. nh-1 on players (u_i, v_i), split J^T A J into
//    independent 2 x 2 blocks (i, j), of which the upper triangle i <= j is
//    kept, by position: block e of a folded triangle at index e of four planes
//    (uu, uv, vu, vv), so a thread reads its own blocks at fixed places without
//    bank conflicts;
//  * the players move on by one rotation a step (u_i to i-1, v_i to i+1, around
//    the ends), so a block's four results go to four fixed places too, in the
//    other of two copies of the matrix, at a constant distance for neighbouring
//    threads;
//  * meanwhile the first warps work out the next step's rotations, each from the
//    three entries it needs of the matrix that the others are still writing.
// Shared-memory accesses and issue slots bound float32, the float64 pipe float64.
// The eigenvectors are not carried along: the rotations go to a log, and
// k_psd_vectors applies it to the rows of V, which are independent, a warp each
// over the whole GPU, when there is something to repair. Row and column passes
// over A and V in one CTA, with three barriers and 4-way conflicts, took 3709 us
// at D = 100 in float32 and 4328 us at D = 60 in float64; now 670 us and 1780 us
// (of it the vectors and the product 90 us and 125 us).
template <typename W>
struct __align__(2 * sizeof(W)) CosSin {
  W c, s;
};
struct PsdInfo {
  int neg;    // negative eigenvalues
  int steps;  // steps in the rotation log
};

// The rotation that zeroes a_pq. Any t gives a rotation when c = 1 / sqrt(1 + t^2)
// is exact, and a t off by a few 2^-22 leaves as much of a_pq, which the next
// sweep squares away: so t takes the approximate float32 operations. c does not:
// its rounding drifts V from orthogonality over the steps (one Newton step in
// place of the root and division raised the repaired matrix's float32 error 1.6
// times). In float64 two Newton steps, as small corrections, from the
// approximate reciprocal root reach rounding (relative error 2^-21, 2^-41).
__device__ __forceinline__ float tangent(float num, float den) {
  float tau = __fdividef(num, den);
  if (!(fabsf(tau) >= 0.0f)) tau = 0.0f;  // both underflow
  const float r = fmaf(tau, tau, 1.0f);
  return copysignf(__fdividef(1.0f, fminf(fabsf(tau) + r * rsqrtf(r), 1.0e37f)), tau);
}
__device__ __forceinline__ CosSin<float> rotation(float app, float aqq, float apq) {
  if (apq == 0.0f) return {1.0f, 0.0f};
  const float t = tangent(aqq - app, 2.0f * apq);
  const float x = fmaf(t, t, 1.0f);
  const float c = 1.0f / sqrtf(x);
  return {c, t * c};
}
__device__ __forceinline__ CosSin<double> rotation(double app, double aqq, double apq) {
  if (apq == 0.0) return {1.0, 0.0};
  const double t = (double)tangent((float)(aqq - app), (float)(2.0 * apq));
  const double x = fma(t, t, 1.0);
  double c = (double)rsqrtf((float)x);
  c = fma(0.5 * c, fma(-(x * c), c, 1.0), c);
  c = fma(0.5 * c, fma(-(x * c), c, 1.0), c);
  return {c, t * c};
}

// The folded triangle of blocks i <= j < nh: rows of nh + 1, row r holding
// i = r (nh - r blocks) and then i = nh - 1 - r.
__host__ __device__ __forceinline__ int fold(int i, int j, int nh) {
  return 2 * i <= nh - 1 ? i * (nh + 1) + (j - i) : (nh - 1 - i) * (nh + 1) + j + 1;
}
__host__ __device__ __forceinline__ int fold_size(int nh) { return (nh + 1) / 2 * (nh + 1); }
// false for the empty half of the middle row of an odd nh
__device__ __forceinline__ bool unfold(int e, int nh, int& i, int& j) {
  const int r = e / (nh + 1), x = e - r * (nh + 1);
  const bool first = x < nh - r;
  i = first ? r : nh - 1 - r;
  j = first ? r + x : x - 1;
  return first || 2 * r < nh - 1;
}
// Rotation and role (0: u, 1: v) of player (role, i) at the next step.
__device__ __forceinline__ void next_place(int nh, int& i, int& role) {
  if (role == 0) {
    if (i > 0) i -= 1;
    else if (nh > 1) i = 1, role = 1;
  } else if (i > 0) {
    if (i < nh - 1) i += 1;
    else role = 0;
  }
}
// Index in the four planes (each of P entries) of the entry between players
// (ra, i) and (rb, j).
__device__ __forceinline__ int entry_at(int nh, int P, int i, int ra, int j, int rb) {
  if (i > j || (i == j && ra > rb)) {
    int t = i;
    i = j;
    j = t;
    t = ra;
    ra = rb;
    rb = t;
  }
  return (2 * ra + rb) * P + fold(i, j, nh);
}

template <typename W>
__global__ void __launch_bounds__(kJacobiThreads) k_psd_jacobi(const double* __restrict__ sig, int D,
                                                               CosSin<W>* __restrict__ log, double* __restrict__ lam,
                                                               PsdInfo* info, int* clipped) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int m = (D + 1) & ~1;  // players of the round-robin (one idle when D is odd)
  const int nh = m / 2, P = fold_size(nh);
  CosSin<W>* rot = reinterpret_cast<CosSin<W>*>(smem_raw);  // this step's, then the next one's
  W* A = reinterpret_cast<W*>(rot + 2 * nh);                // two copies of four planes
  __shared__ double s_red[kJacobiThreads / 32];
  __shared__ int s_neg;
  const int tid = threadIdx.x, nth = (int)blockDim.x;
  auto block_red = [&](double v, bool max) -> double {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const double u = __shfl_xor_sync(0xffffffffu, v, o);
      v = max ? fmax(v, u) : v + u;
    }
    if ((tid & 31) == 0) s_red[tid >> 5] = v;
    __syncthreads();
    double t = s_red[0];
    for (int w = 1; w < (nth >> 5); ++w) t = max ? fmax(t, s_red[w]) : t + s_red[w];
    __syncthreads();
    return t;
  };
  // scale by a power of two (exact) to entries of at most 2
  double big = 0.0;
  for (int e = tid; e < D * D; e += nth) big = fmax(big, fabs(sig[e]));
  big = block_red(big, true);
  int ex = 0;
  if (big > 0.0 && big < INFINITY) ex = ilogb(big);
  const double down = ldexp(1.0, -ex), up = ldexp(1.0, ex);
  // players of rotation i at step 0: u_i = i, v_i = m - 1 - i
  double nrm = 0.0;
  for (int e = tid; e < 4 * P; e += nth) {
    const int plane = e / P;
    int i, j;
    W a = 0;
    if (unfold(e - plane * P, nh, i, j)) {
      const int r = (plane & 2) ? m - 1 - i : i, c = (plane & 1) ? m - 1 - j : j;
      if (r < D && c < D && !(i == j && plane == 2)) {
        a = (W)(sig[(size_t)min(r, c) * D + max(r, c)] * down);
        nrm += (r == c ? 1.0 : 2.0) * (double)a * (double)a;
      }
    }
    A[e] = a;
  }
  const double norm2 = block_red(nrm, false);
  // converged when the off-diagonal norm reaches the level rounding leaves in
  // a D x D rotation sequence, 2 D eps of the norm (eps of the working type)
  const double eps = sizeof(W) == 8 ? 1.1102230246251565e-16 : 5.9604644775390625e-8;
  const double rel2 = (2.0 * D * eps) * (2.0 * D * eps);

  // the first warps own the rotations, thread i < nh rotation i, the others the
  // blocks: kPsdRounds places of their blocks and of each block's four results
  const int rot_threads = (nh + 31) & ~31, nwt = nth - rot_threads;
  const int wt = tid - rot_threads;
  int src[kPsdRounds], bi[kPsdRounds], bj[kPsdRounds], dst[kPsdRounds][4];
  int n_uu = 0, n_vv = 0, n_uv = 0, r_uu = 0, r_vv = 0;  // a rotation thread's next entries: index, source
  int i_uu = 0, i_vv = 0;
#pragma unroll
  for (int q = 0; q < kPsdRounds; ++q) src[q] = -1;
  if (wt >= 0) {
#pragma unroll
    for (int q = 0; q < kPsdRounds; ++q) {
      const int e = wt + q * nwt;
      int i, j;
      if (e < P && unfold(e, nh, i, j)) {
        src[q] = e;
        bi[q] = i;
        bj[q] = j;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          int ni = i, nj = j, na = k >> 1, nb = k & 1;
          next_place(nh, ni, na);
          next_place(nh, nj, nb);
          dst[q][k] = entry_at(nh, P, ni, na, nj, nb);
        }
      }
    }
  } else if (tid < nh) {
    // the players of rotation tid at the next step: where they are now
    for (int i = 0; i < nh; ++i)
      for (int role = 0; role < 2; ++role) {
        int ni = i, nr = role;
        next_place(nh, ni, nr);
        if (ni == tid && nr == 0) i_uu = i, r_uu = role;
        if (ni == tid && nr == 1) i_vv = i, r_vv = role;
      }
    n_uu = fold(i_uu, i_uu, nh);
    n_vv = fold(i_vv, i_vv, nh);
    n_uv = fold(min(i_uu, i_vv), max(i_uu, i_vv), nh);
    const int e = fold(tid, tid, nh);
    const CosSin<W> cs = rotation(A[e], A[3 * P + e], A[P + e]);
    rot[tid] = cs;
    log[tid] = cs;
  }
  __syncthreads();
  // a result of a block under rotations R (rows) and S (columns)
  auto entry = [](W auu, W auv, W avu, W avv, CosSin<W> R, int a, CosSin<W> S, int b) -> W {
    const W x = a ? R.s : R.c, y = a ? R.c : -R.s;
    const W u = x * auu + y * avu, v = x * auv + y * avv;
    return (b ? S.s : S.c) * u + (b ? S.c : -S.s) * v;
  };
  int steps = 0;
  for (int sweep = 0; sweep < kJacobiSweeps; ++sweep) {
    W off = 0;
    for (int e = tid; e < P; e += nth) {
      const W* B = A + (steps & 1) * 4 * P + e;
      int i, j;
      if (unfold(e, nh, i, j)) off += B[P] * B[P] + (i == j ? (W)0 : B[0] * B[0] + B[2 * P] * B[2 * P] + B[3 * P] * B[3 * P]);
    }
    if (!(2.0 * block_red((double)off, false) > rel2 * norm2)) break;  // uniform
    for (int step = 0; step < m - 1; ++step, ++steps) {
      const W* __restrict__ B = A + (steps & 1) * 4 * P;
      W* __restrict__ C = A + ((steps & 1) ^ 1) * 4 * P;
      const CosSin<W>* cur = rot + (steps & 1) * nh;
      if (tid < nh) {
        const CosSin<W> R = cur[i_uu], S = cur[i_vv];
        const W* b = B + n_uu;
        const W aa = entry(b[0], b[P], b[P], b[3 * P], R, r_uu, R, r_uu);
        b = B + n_vv;
        const W bb = entry(b[0], b[P], b[P], b[3 * P], S, r_vv, S, r_vv);
        b = B + n_uv;
        W ab;
        if (i_uu == i_vv) ab = entry(b[0], b[P], b[P], b[3 * P], R, 0, R, 1);
        else if (i_uu < i_vv) ab = entry(b[0], b[P], b[2 * P], b[3 * P], R, r_uu, S, r_vv);
        else ab = entry(b[0], b[P], b[2 * P], b[3 * P], S, r_vv, R, r_uu);
        const CosSin<W> cs = rotation(aa, bb, ab);
        rot[((steps & 1) ^ 1) * nh + tid] = cs;
        log[(size_t)(steps + 1) * nh + tid] = cs;
      } else {
#pragma unroll
        for (int q = 0; q < kPsdRounds; ++q) {
          if (src[q] >= 0) {
            const CosSin<W> R = cur[bi[q]], S = cur[bj[q]];
            const W* b = B + src[q];
            const bool diag = bi[q] == bj[q];
            const W auu = b[0], auv = b[P], avu = diag ? auv : b[2 * P], avv = b[3 * P];
            // rows: J_i^T, then columns: J_j (with c and s: a common factor c_i c_j
            // after four multiply-adds with t rounds all four results alike, which
            // doubled the error)
            const W buu = R.c * auu - R.s * avu, buv = R.c * auv - R.s * avv;
            const W bvu = R.s * auu + R.c * avu, bvv = R.s * auv + R.c * avv;
            C[dst[q][0]] = S.c * buu - S.s * buv;
            C[dst[q][1]] = S.s * buu + S.c * buv;
            if (!diag) C[dst[q][2]] = S.c * bvu - S.s * bvv;  // a diagonal block's (v, u) is (u, v)
            C[dst[q][3]] = S.s * bvu + S.c * bvv;
          }
        }
      }
      __syncthreads();
    }
  }
  if (tid == 0) s_neg = 0;
  __syncthreads();
  for (int d = tid; d < D; d += nth) {
    // after whole sweeps the players are back where they started
    const bool v = d >= nh;
    const int i = v ? m - 1 - d : d;
    const double l = (double)A[((steps & 1) * 4 + (v ? 3 : 0)) * P + fold(i, i, nh)] * up;
    lam[d] = l;
    if (l < 0.0) atomicAdd(&s_neg, 1);
  }
  __syncthreads();
  if (tid == 0) {
    info->neg = s_neg;
    info->steps = steps;
    if (clipped) *clipped = s_neg;
  }
}

// Row x of V = J_1 J_2 ... J_n (block x): the unit row through the log's
// rotations; the next kLogAhead steps' rotations are loaded while the current
// ones are applied. Stored transposed (Vt[k][x] = V[x][k]) for k_psd_apply.
constexpr int kLogAhead = 4;
template <typename W, int NR>
__global__ void __launch_bounds__(32) k_psd_vectors(const CosSin<W>* __restrict__ log,
                                                    const PsdInfo* __restrict__ info, int D, W* __restrict__ Vt) {
  __shared__ W u[kPsdMaxD + 2];
  if (info->neg == 0) return;
  const int lane = threadIdx.x;
  const int m = (D + 1) & ~1, nh = m / 2;
  for (int i = lane; i < m; i += 32) u[i] = i == (int)blockIdx.x ? (W)1 : (W)0;
  __syncwarp();
  const int steps = info->steps;
  // players of this lane's rotations r = lane + 32 g at step 0
  int a[NR], b[NR];
#pragma unroll
  for (int g = 0; g < NR; ++g) {
    const int r = lane + 32 * g;
    a[g] = r % (m - 1);
    b[g] = r == 0 ? m - 1 : (2 * (m - 1) - r) % (m - 1);
  }
  CosSin<W> cur[kLogAhead][NR], nxt[kLogAhead][NR];
  auto fetch = [&](CosSin<W> (&d)[kLogAhead][NR], int t0) {
#pragma unroll
    for (int h = 0; h < kLogAhead; ++h)
#pragma unroll
      for (int g = 0; g < NR; ++g) {
        const int r = lane + 32 * g;
        if (t0 + h < steps && r < nh) d[h][g] = log[(size_t)(t0 + h) * nh + r];
      }
  };
  fetch(cur, 0);
  for (int t0 = 0; t0 < steps; t0 += kLogAhead) {
    fetch(nxt, t0 + kLogAhead);
#pragma unroll
    for (int h = 0; h < kLogAhead; ++h) {
      if (t0 + h < steps) {
        W up[NR], uq[NR];
#pragma unroll
        for (int g = 0; g < NR; ++g)
          if (lane + 32 * g < nh) {
            up[g] = u[a[g]];
            uq[g] = u[b[g]];
          }
#pragma unroll
        for (int g = 0; g < NR; ++g) {
          const int r = lane + 32 * g;
          if (r < nh) {
            const W c = cur[h][g].c, s = cur[h][g].s;
            u[a[g]] = c * up[g] - s * uq[g];
            u[b[g]] = s * up[g] + c * uq[g];
            a[g] = a[g] + 1 == m - 1 ? 0 : a[g] + 1;
            if (r > 0) b[g] = b[g] + 1 == m - 1 ? 0 : b[g] + 1;
          }
        }
        __syncwarp();
      }
    }
#pragma unroll
    for (int h = 0; h < kLogAhead; ++h)
#pragma unroll
      for (int g = 0; g < NR; ++g) cur[h][g] = nxt[h][g];
  }
  for (int i = lane; i < D; i += 32) Vt[(size_t)i * D + blockIdx.x] = u[i];
}

// V max(Lambda, 0) V^T, one thread per entry of the upper triangle.
template <typename W>
__global__ void __launch_bounds__(256) k_psd_apply(double* __restrict__ sig, const W* __restrict__ Vt,
                                                   const double* __restrict__ lam, const PsdInfo* __restrict__ info,
                                                   int D) {
  __shared__ W s_lam[kPsdMaxD];
  if (info->neg == 0) return;  // already positive semi-definite: Sigma unchanged
  for (int k = threadIdx.x; k < D; k += blockDim.x) s_lam[k] = lam[k] > 0.0 ? (W)lam[k] : (W)0;
  __syncthreads();
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= D * D) return;
  const int i = e / D, j = e - i * D;
  if (j < i) return;
  W v = 0;
#pragma unroll 16
  for (int k = 0; k < D; ++k) v += Vt[(size_t)k * D + i] * s_lam[k] * Vt[(size_t)k * D + j];
  sig[(size_t)i * D + j] = v;
  sig[(size_t)j * D + i] = v;
}

// The same cyclic Jacobi iteration over the whole GPU, for matrices larger
// than one CTA's shared memory holds: one CTA per SM under a cooperative
// launch (every CTA resident), A and V in global memory (read through L2).
// A round-robin step's rotations act on disjoint index pairs, so J^T A J
// splits into independent 2 x 2 blocks (rows p_i, q_i; columns p_j, q_j):
// after a grid barrier every CTA recomputes the step's D/2 rotations from
// A's current diagonal and pivot entries, and the threads of the grid update
// the blocks of A and the column pairs of V (each element written by one
// thread). One barrier per step, one reduction per sweep; every barrier wait
// is bounded (ST_TIMEOUT, and the CTA leaves).
struct GridSync {
  unsigned count;  // arrivals at the current barrier
  unsigned gen;    // barriers completed
  int neg;         // negative eigenvalues
  int pad;
  double red[3];   // [0] squared norm, [1], [2] off-diagonal sums of alternate sweeps
};

__device__ __forceinline__ uint64_t grid_timer_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// Grid-wide barrier for a cooperative launch; false when the wait timed out.
__device__ bool grid_barrier(GridSync* gs, unsigned nblocks, int* status) {
  __shared__ int s_ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    volatile unsigned* vgen = &gs->gen;
    const unsigned g = *vgen;
    __threadfence();
    int ok = 1;
    if (atomicAdd(&gs->count, 1u) == nblocks - 1) {
      atomicExch(&gs->count, 0u);
      __threadfence();
      atomicAdd(&gs->gen, 1u);
    } else {
      const uint64_t t0 = grid_timer_ns();
      while (*vgen == g) {
        if (grid_timer_ns() - t0 > kDefaultWaitNs) {
          ok = 0;
          atomicOr(status, ST_TIMEOUT);
          break;
        }
      }
    }
    __threadfence();
    s_ok = ok;
  }
  __syncthreads();
  return s_ok != 0;
}

constexpr int kGridJacobiThreads = 512;
constexpr int kGridMaxD = 4000;  // rotations of one step fit 48 KB of shared memory

template <typename W>
__global__ void __launch_bounds__(kGridJacobiThreads) k_psd_repair_grid(double* __restrict__ sig, W* __restrict__ A,
                                                                        W* __restrict__ V, int D, int* clipped,
                                                                        GridSync* gs, int* status) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int m = (D + 1) & ~1, nh = m / 2;
  W* rc = reinterpret_cast<W*>(smem_raw);
  W* rs = rc + nh;
  int* rp = reinterpret_cast<int*>(rs + nh);
  int* rq = rp + nh;
  __shared__ double s_red[kGridJacobiThreads / 32];
  const unsigned nb = gridDim.x;
  const int tid = threadIdx.x;
  const int64_t gtid = (int64_t)blockIdx.x * blockDim.x + tid, gnth = (int64_t)gridDim.x * blockDim.x;
  const int64_t DD = (int64_t)D * D;
  auto block_sum_to = [&](double v, double* dst) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if ((tid & 31) == 0) s_red[tid >> 5] = v;
    __syncthreads();
    if (tid == 0) {
      double t = 0.0;
      for (int w = 0; w < kGridJacobiThreads / 32; ++w) t += s_red[w];
      atomicAdd(dst, t);
    }
    __syncthreads();
  };
  double nrm = 0.0;
  for (int64_t e = gtid; e < DD; e += gnth) {
    const W a = (W)sig[e];
    A[e] = a;
    const int64_t r = e / D;
    V[e] = (r == e - r * D) ? (W)1 : (W)0;
    nrm += (double)a * (double)a;
  }
  block_sum_to(nrm, &gs->red[0]);
  if (!grid_barrier(gs, nb, status)) return;
  const double norm2 = __ldcg(&gs->red[0]);
  const double eps = sizeof(W) == 8 ? 1.1102230246251565e-16 : 5.9604644775390625e-8;
  const double rel2 = (2.0 * D * eps) * (2.0 * D * eps);
  for (int sweep = 0; sweep < kJacobiSweeps; ++sweep) {
    double* slot = &gs->red[1 + (sweep & 1)];
    double off = 0.0;
    for (int64_t e = gtid; e < DD; e += gnth) {
      const int64_t r = e / D;
      if (r != e - r * D) {
        const double a = (double)__ldcg(A + e);
        off += a * a;
      }
    }
    block_sum_to(off, slot);
    if (!grid_barrier(gs, nb, status)) return;
    const double off_all = __ldcg(slot);
    // the other slot was last read before this barrier: clear it for the next sweep
    if (blockIdx.x == 0 && tid == 0) gs->red[1 + ((sweep + 1) & 1)] = 0.0;
    if (!(off_all > rel2 * norm2)) break;  // uniform: every CTA read the same sum
    for (int step = 0; step < m - 1; ++step) {
      for (int i = tid; i < nh; i += blockDim.x) {
        int p, q;
        if (i == 0) {
          p = step;
          q = m - 1;
        } else {
          p = (step + i) % (m - 1);
          q = (step - i + (m - 1)) % (m - 1);
        }
        if (p > q) {
          const int x = p;
          p = q;
          q = x;
        }
        W c = 1, sn = 0;
        if (q < D) {
          const W apq = __ldcg(A + (int64_t)p * D + q);
          if (apq != (W)0) {
            const W tau = (__ldcg(A + (int64_t)q * D + q) - __ldcg(A + (int64_t)p * D + p)) / ((W)2 * apq);
            const W t = (tau >= (W)0 ? (W)1 : (W)-1) / (fabs(tau) + sqrt((W)1 + tau * tau));
            c = (W)1 / sqrt((W)1 + t * t);
            sn = t * c;
          }
        }
        rp[i] = p;
        rq[i] = q;
        rc[i] = c;
        rs[i] = sn;
      }
      __syncthreads();
      // A <- J^T A J by 2 x 2 blocks (rows of pair i, columns of pair j)
      const int64_t nblk = (int64_t)nh * nh;
      for (int64_t e = gtid; e < nblk; e += gnth) {
        const int i = (int)(e / nh), j = (int)(e - (int64_t)i * nh);
        const int pi = rp[i], qi = rq[i], pj = rp[j], qj = rq[j];
        const bool vi = qi < D, vj = qj < D;
        const W ci = rc[i], si = rs[i], cj = rc[j], sj = rs[j];
        const W app = __ldcg(A + (int64_t)pi * D + pj);
        const W apq = vj ? __ldcg(A + (int64_t)pi * D + qj) : (W)0;
        const W aqp = vi ? __ldcg(A + (int64_t)qi * D + pj) : (W)0;
        const W aqq = (vi && vj) ? __ldcg(A + (int64_t)qi * D + qj) : (W)0;
        // rows: J_i^T, then columns: J_j
        const W bpp = ci * app - si * aqp, bpq = ci * apq - si * aqq;
        const W bqp = si * app + ci * aqp, bqq = si * apq + ci * aqq;
        A[(int64_t)pi * D + pj] = cj * bpp - sj * bpq;
        if (vj) A[(int64_t)pi * D + qj] = sj * bpp + cj * bpq;
        if (vi) A[(int64_t)qi * D + pj] = cj * bqp - sj * bqq;
        if (vi && vj) A[(int64_t)qi * D + qj] = sj * bqp + cj * bqq;
      }
      // V <- V J by column pairs
      const int64_t nv = (int64_t)D * nh;
      for (int64_t e = gtid; e < nv; e += gnth) {
        const int x = (int)(e / nh), j = (int)(e - (int64_t)x * nh);
        const int pj = rp[j], qj = rq[j];
        if (qj >= D) continue;
        const W cj = rc[j], sj = rs[j];
        const W vp = __ldcg(V + (int64_t)x * D + pj), vq = __ldcg(V + (int64_t)x * D + qj);
        V[(int64_t)x * D + pj] = cj * vp - sj * vq;
        V[(int64_t)x * D + qj] = sj * vp + cj * vq;
      }
      if (!grid_barrier(gs, nb, status)) return;
    }
  }
  // eigenvalues: the diagonal, negatives clipped
  int neg = 0;
  for (int i = (int)gtid; i < D; i += (int)gnth)
    if (__ldcg(A + (int64_t)i * D + i) < (W)0) ++neg;
  if (neg) atomicAdd(&gs->neg, neg);
  if (!grid_barrier(gs, nb, status)) return;
  const int negs = *(volatile int*)&gs->neg;
  if (blockIdx.x == 0 && tid == 0 && clipped) *clipped = negs;
  if (negs == 0) return;  // already positive semi-definite: Sigma unchanged
  // the clipped eigenvalues in this CTA's shared memory (the rotation arrays
  // hold at least 8 D bytes)
  double* lam = reinterpret_cast<double*>(smem_raw);
  for (int k = tid; k < D; k += blockDim.x) {
    const double l = (double)__ldcg(A + (int64_t)k * D + k);
    lam[k] = l > 0.0 ? l : 0.0;
  }
  __syncthreads();
  const int64_t npairs = (int64_t)D * (D + 1) / 2;
  for (int64_t e = gtid; e < npairs; e += gnth) {
    // pair (i, j), i <= j, in row-major order of the upper triangle
    int i = (int)((sqrt(8.0 * (double)e + 1.0) - 1.0) * 0.5);
    while ((int64_t)(i + 1) * (i + 2) / 2 <= e) ++i;
    while ((int64_t)i * (i + 1) / 2 > e) --i;
    const int jj = (int)(e - (int64_t)i * (i + 1) / 2);  // 0..i
    const int r = jj, c = i;                             // r <= c
    double v = 0.0;
    for (int k = 0; k < D; ++k)
      if (lam[k] > 0.0) v += (double)__ldcg(V + (int64_t)r * D + k) * lam[k] * (double)__ldcg(V + (int64_t)c * D + k);
    sig[(int64_t)r * D + c] = v;
    sig[(int64_t)c * D + r] = v;
  }
}

// Sigma and R in the output precision: R_ij = Sigma_ij / sqrt(Sigma_ii Sigma_jj)
// (float64), R_ii = 1; a non-positive variance gives NaN and ST_ZERO_VAR.
template <typename T>
__global__ void k_pairwise_out(const double* __restrict__ sig, int D, T* __restrict__ sigma, T* __restrict__ R,
                               int* status) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= D * D) return;
  const int i = e / D, j = e - i * D;
  const double v = sig[e], a = sig[(size_t)i * D + i], b = sig[(size_t)j * D + j];
  if (sigma) sigma[e] = (T)v;
  double r;
  if (a > 0.0 && b > 0.0) {
    r = (i == j) ? 1.0 : v / (sqrt(a) * sqrt(b));
  } else {
    r = __longlong_as_double(0x7ff8000000000000ll);
    if (i == j) atomicOr(status, ST_ZERO_VAR);
  }
  R[e] = (T)r;
}

}  // namespace

}  // namespace mmgpu

namespace mmgpu {

int pairwise_psd_max_assets() { return kGridMaxD; }

static int pairwise_splits(int D, int ld) {
  const int nt = (D + kPT - 1) / kPT, tiles = nt * (nt + 1) / 2;
  return std::max(1, std::min((kPairwiseCtas + tiles - 1) / tiles, (ld + kPChunk - 1) / kPChunk));
}

size_t pairwise_part_bytes(int D) {
  const size_t nt = ((size_t)D + kPT - 1) / kPT, tiles = nt * (nt + 1) / 2;
  if (tiles >= (size_t)kPairwiseCtas) return 0;  // a CTA a tile
  return (tiles + kPairwiseCtas) * 256 * sizeof(double) + tiles * sizeof(int);
}

cudaError_t launch_pairwise(bool fp64, bool fejer, const void* coeffs, int ld, const int* Nv, int D,
                            void* part, double* sig, cudaStream_t s) {
  const int nt = (D + kPT - 1) / kPT, tiles = nt * (nt + 1) / 2;
  const dim3 grid(tiles, pairwise_splits(D, ld));
  // the tiles' arrival counters (zero between calls) after the partial sums
  double* pt = reinterpret_cast<double*>(part);
  int* done = reinterpret_cast<int*>(pt + ((size_t)tiles + kPairwiseCtas) * 256);
  if (fp64) {
    if (fejer) k_pairwise<double2, double, true><<<grid, 256, 0, s>>>((const double2*)coeffs, ld, Nv, D, nt, pt, done, sig);
    else k_pairwise<double2, double, false><<<grid, 256, 0, s>>>((const double2*)coeffs, ld, Nv, D, nt, pt, done, sig);
  } else {
    if (fejer) k_pairwise<float2, float, true><<<grid, 256, 0, s>>>((const float2*)coeffs, ld, Nv, D, nt, pt, done, sig);
    else k_pairwise<float2, float, false><<<grid, 256, 0, s>>>((const float2*)coeffs, ld, Nv, D, nt, pt, done, sig);
  }
  return cudaGetLastError();
}

static bool psd_one_cta(bool fp64, int D) { return D <= (fp64 ? kPsdMaxD64 : kPsdMaxD); }

// iteration, eigenvectors and product, or the cooperative kernel that does all
int psd_repair_launches(bool fp64, int D) { return psd_one_cta(fp64, D) ? 3 : 1; }

size_t psd_log_bytes(bool fp64, int D) {
  if (!psd_one_cta(fp64, D)) return 0;  // the multi-CTA iteration keeps none
  const size_t m = ((size_t)D + 1) & ~(size_t)1;
  return ((size_t)kJacobiSweeps * (m - 1) + 1) * (m / 2) * 2 * (fp64 ? 8 : 4);
}

template <typename W>
static cudaError_t launch_psd_one_cta(double* sig, double* A, W* V, int D, int* clipped, void* log, void* sync,
                                      cudaStream_t s) {
  const size_t m = ((size_t)D + 1) & ~(size_t)1;
  const int nh = (int)(m / 2);
  const size_t smem = 2 * (nh * sizeof(CosSin<W>) + 4 * (size_t)fold_size(nh) * sizeof(W));
  static_assert(((kPsdMaxD / 2 + 1) / 2) * (kPsdMaxD / 2 + 1) <= kPsdRounds * (kJacobiThreads - (kPsdMaxD / 2 + 31) / 32 * 32),
                "blocks per thread");
  auto* lg = reinterpret_cast<CosSin<W>*>(log);
  auto* info = reinterpret_cast<PsdInfo*>(sync);
  cudaError_t e = cudaFuncSetAttribute(k_psd_jacobi<W>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  // a thread per block where that many fit: barriers and sums over idle warps are
  // a tenth of the time at three assets
  const int threads = std::min(kJacobiThreads, ((nh + 31) & ~31) + ((fold_size(nh) + 31) & ~31));
  k_psd_jacobi<W><<<1, threads, smem, s>>>(sig, D, lg, A, info, clipped);
  switch ((m / 2 + 31) / 32) {
    case 1: k_psd_vectors<W, 1><<<D, 32, 0, s>>>(lg, info, D, V); break;
    case 2: k_psd_vectors<W, 2><<<D, 32, 0, s>>>(lg, info, D, V); break;
    default: k_psd_vectors<W, 3><<<D, 32, 0, s>>>(lg, info, D, V); break;
  }
  k_psd_apply<W><<<(D * D + 255) / 256, 256, 0, s>>>(sig, V, A, info, D);
  return cudaGetLastError();
}

cudaError_t launch_psd_repair(bool fp64, double* sig, double* A, double* V, int D, int* clipped, void* log,
                              void* sync, int* status, cudaStream_t s) {
  if (D > kGridMaxD) return cudaErrorInvalidValue;
  const size_t wb = fp64 ? 8 : 4;
  if (psd_one_cta(fp64, D)) {
    // A holds the eigenvalues, V the eigenvectors (transposed)
    if (fp64) return launch_psd_one_cta<double>(sig, A, V, D, clipped, log, sync, s);
    return launch_psd_one_cta<float>(sig, A, (float*)V, D, clipped, log, sync, s);
  }
  // the whole GPU: one CTA per SM, every CTA resident (cooperative launch)
  cudaError_t e = cudaMemsetAsync(sync, 0, sizeof(GridSync), s);
  if (e != cudaSuccess) return e;
  int dev = 0, sms = 0;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
  const int nh = ((D + 1) & ~1) / 2;
  const size_t smem = (size_t)nh * (2 * wb + 2 * sizeof(int));
  GridSync* gs = reinterpret_cast<GridSync*>(sync);
  auto launch = [&](auto kern, void* Aw, void* Vw) -> cudaError_t {
    int per_sm = 0;
    cudaError_t r = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kGridJacobiThreads, smem);
    if (r != cudaSuccess) return r;
    if (per_sm < 1) return cudaErrorInvalidConfiguration;
    void* args[] = {(void*)&sig, &Aw, &Vw, (void*)&D, (void*)&clipped, (void*)&gs, (void*)&status};
    return cudaLaunchCooperativeKernel((const void*)kern, dim3(sms), dim3(kGridJacobiThreads), args, smem, s);
  };
  if (fp64) return launch(k_psd_repair_grid<double>, (void*)A, (void*)V);
  return launch(k_psd_repair_grid<float>, (void*)A, (void*)V);
}

size_t psd_sync_bytes() { return sizeof(GridSync); }

cudaError_t launch_pairwise_out(bool fp64, const double* sig, int D, void* sigma, void* R, int* status,
                                cudaStream_t s) {
  const int n = D * D, grid = (n + 255) / 256;
  if (fp64) k_pairwise_out<double><<<grid, 256, 0, s>>>(sig, D, (double*)sigma, (double*)R, status);
  else k_pairwise_out<float><<<grid, 256, 0, s>>>(sig, D, (float*)sigma, (float*)R, status);
  return cudaGetLastError();
}

}  // namespace mmgpu
