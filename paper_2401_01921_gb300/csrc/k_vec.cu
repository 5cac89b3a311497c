// FP64 vector kernels: scaling, norms and the device-resident Lanczos loop.
//
// Sec. 9.3 of arXiv 2401.01921: Lanczos needs only the operator's action on a
// vector (a LinOp).  Everything except that action runs here, in FP64, with
// no host round trip inside the loop (so a whole solve can be captured in one
// CUDA graph):
//   alpha_j = <v_j, w>; w -= alpha_j v_j + beta_j v_{j-1} (three-term step);
//   c = V^T w, w -= V c   (one classical Gram-Schmidt pass against every
//   previous vector: full reorthogonalisation);
//   beta_{j+1} = ||w||; stop if beta_{j+1} < 1e-14 max(|alpha_i|, beta_i; i <= j);
//   v_{j+1} = w / beta_{j+1};
// then Sturm bisection on the tridiagonal T and inverse iteration for its
// eigenvector, and the Ritz vector V y.
// Reductions are deterministic: per-block partial sums with a fixed grid and
// a fixed-order tree (warp shuffles), then the partials in a fixed order.
#include <cooperative_groups.h>

#include "tnx_internal.h"

namespace {

constexpr int RT = 256;        // threads per reduction block
constexpr int RBLOCKS = 1216;  // 8 blocks per SM on 152 SMs
constexpr int LT = 256;        // threads per CTA of a Lanczos step

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  return v;
}

// block-wide sum, result valid in thread 0
__device__ double block_sum(double v, double* sh) {
  v = warp_sum(v);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (lane == 0) sh[wid] = v;
  __syncthreads();
  v = (threadIdx.x < (blockDim.x >> 5)) ? sh[threadIdx.x] : 0.0;
  if (wid == 0) v = warp_sum(v);
  __syncthreads();
  return v;
}

__device__ __forceinline__ bool stopped(const int32_t* state) { return *(volatile const int32_t*)(state + 1) != 0; }

// The words that the CTAs of a Lanczos step wait on, one per 128 bytes: barrier
// arrivals, norm arrivals, the decision (2 (j + 1), plus 1 with a pass).
__device__ __forceinline__ unsigned long long* step_words(const LanczosDev& L) {
  return (unsigned long long*)(L.state + 32);
}
constexpr int SW = 16;   // words apart: polls of one do not meet arrivals at another

// Reductions finish in the launch that produces their partial sums: every
// block publishes its partials, fences and counts itself in state[4]; the
// block that counts last (no block waits for another) reads all partials
// through L2, in a fixed order, so the result does not depend on which block
// that is, and resets the counter for the next launch.
__device__ bool last_block(int32_t* counter) {
  __shared__ int s_last;
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    s_last = atomicAdd(counter, 1) == (int)gridDim.x - 1;
  }
  __syncthreads();
  if (s_last) __threadfence();
  return s_last != 0;
}

__global__ void scale_kernel(double* x, int64_t n, double a) {
  tnx_grid_dependency();
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    x[i] *= a;
}

__global__ void add_scalar_kernel(double* x, int64_t n, double a) {
  tnx_grid_dependency();
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    x[i] += a;
}

// partial[b] = sum over this block's grid-stride share of x*y
__global__ void __launch_bounds__(RT) dot_partial_kernel(const double* __restrict__ x, const double* __restrict__ y,
                                                         int64_t n, double* partial, const int32_t* state) {
  tnx_grid_dependency();
  __shared__ double sh[32];
  if (state && stopped(state)) return;
  double acc = 0.0;
  for (int64_t i = (int64_t)blockIdx.x * RT + threadIdx.x; i < n; i += (int64_t)gridDim.x * RT)
    acc = fma(x[i], y[i], acc);
  acc = block_sum(acc, sh);
  if (threadIdx.x == 0) partial[blockIdx.x] = acc;
}

// mode 0: out = sum; mode 1: out = sqrt(sum)
__global__ void __launch_bounds__(RT) finalize_kernel(const double* partial, int np, double* out, int mode,
                                                      const int32_t* state) {
  tnx_grid_dependency();
  __shared__ double sh[32];
  if (state && stopped(state)) return;
  double acc = 0.0;
  for (int i = threadIdx.x; i < np; i += RT) acc += partial[i];
  acc = block_sum(acc, sh);
  if (threadIdx.x == 0) *out = mode ? sqrt(acc) : acc;
}

// ---------------------------------------------------------------- Lanczos
__global__ void lanczos_init_kernel(LanczosDev L, const double* v0) {
  tnx_grid_dependency();
  // V[0] = v0 / ||v0|| (norm already in L.scratch[0]); state reset
  const double inv = 1.0 / L.scratch[0];
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < L.n; i += (int64_t)gridDim.x * blockDim.x)
    L.V[i] = v0[i] * inv;
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    L.state[0] = 0;
    L.state[1] = 0;
    L.state[2] = 0;
    L.state[3] = 0;
    L.state[4] = 0;   // the last-block counter
    for (int q = 0; q < 3; ++q) step_words(L)[q * SW] = 0;
    L.beta[0] = 0.0;
    L.omega[0] = 1.0;   // <v_0, v_0>; the row before it is empty
  }
}

__global__ void set_slot_kernel(double** slot, double* p) {
  tnx_grid_dependency();
  *slot = p;
}

// beta_{j+1} = sqrt(sum of the nb norm partials); decide stop; record k; point
// the next apply's input slot at v_{j+1} (which the next kernel writes).  Run
// by one block of RT threads.
__device__ void beta_decide(const LanczosDev& L, int j, int nb, int last, double** next_slot) {
  __shared__ double sh[32];
  __shared__ double s_amax;
  double acc = 0.0;
  for (int b = threadIdx.x; b < nb; b += RT) acc += __ldcg(L.partial + b);
  if (threadIdx.x < 32) {
    double amax = 0.0;
    // the scale of T seen so far: max |alpha_i| and max beta_i (i <= j; beta_0 = 0)
    for (int i = threadIdx.x; i <= j; i += 32) amax = fmax(amax, fmax(fabs(L.alpha[i]), L.beta[i]));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) amax = fmax(amax, __shfl_xor_sync(0xffffffffu, amax, o));
    if (threadIdx.x == 0) s_amax = amax;
  }
  acc = block_sum(acc, sh);
  if (threadIdx.x == 0) {
    const double beta = sqrt(acc);
    L.beta[j + 1] = beta;
    L.scratch[3 * L.nmax + 3] = 1.0 / beta;   // for the normalising kernel
    L.state[0] = j + 1;
    if (last || beta < 1e-14 * s_amax) L.state[1] = 1;
    else *next_slot = L.V + (int64_t)(j + 1) * L.n;
  }
}

// Partial reorthogonalisation (Simon, Math. Comp. 42, 1984): omega_{j,k}
// estimates <v_j, v_k> through the recurrence that the Lanczos relation gives,
//   beta_{j+1} omega_{j+1,k} = beta_{k+1} omega_{j,k+1} + (alpha_k - alpha_j) omega_{j,k}
//                              + beta_k omega_{j,k-1} - beta_j omega_{j-1,k} + rounding,
// with the rounding term taken as sign(.) eps1 |T| (eps1 = sqrt(n) eps / 2, |T|
// bounded by max_i |alpha_i| + beta_i + beta_{i+1}) and omega_{j+1,j} =
// eps1 |T| / beta_{j+1}.  After the three-term step this kernel forms
// beta_{j+1} = |w| and the estimates of row j+1; the step takes a full
// Gram-Schmidt pass against v_0..v_j when the largest estimate exceeds
// tau (1e-10; a negative tau: every step), and so does the step after it (the error
// that v_j carries reaches v_{j+2} too); after a pass the estimates restart at eps1.
// Without a pass it also does what beta_decide does (beta_{j+1}, the stopping test, the
// next input slot); with one, the pass does.
constexpr int PRO_MAX = 514;   // rows of at most 500 steps + 2

// What a step waits for here is FP64 latency: an FP64 instruction takes its SM
// quarter 64 cycles however few lanes need it (a root ten of them, a division
// nine), so roots and divisions are taken once, by one warp, maxima of
// non-negative numbers are formed on their bit patterns, and eps1 comes from the
// host.
__device__ __forceinline__ unsigned long long bits_abs(double x) {
  return (unsigned long long)__double_as_longlong(x) & 0x7FFFFFFFFFFFFFFFull;
}
__device__ __forceinline__ unsigned long long warp_max(unsigned long long v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = max(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

// T and the estimates of rows j and j-1 in shared memory, read at the start of a step.
struct ProRows {
  double *al, *be, *om, *omp;   // alpha_k (k < j), beta_k (k <= j), omega_{j,k} (k <= j), omega_{j-1,k} (k < j)
};
__device__ __forceinline__ void pro_load(const LanczosDev& L, int j, const ProRows& r) {
  for (int k = threadIdx.x; k <= j; k += LT) {
    r.be[k] = L.beta[k];
    r.om[k] = L.omega[k];
    if (k < j) {
      r.al[k] = L.alpha[k];
      r.omp[k] = L.omega[L.nmax + 2 + k];
    }
  }
}

// max(|alpha_i|, beta_i) and max(|alpha_i| + beta_i + beta_{i+1}) over i <= j (alpha_j
// given, beta_{j+1} left out), as bit patterns; one warp.
__device__ __forceinline__ void tridiag_scale(const ProRows& r, int j, int lane, double aj,
                                              unsigned long long& amax, unsigned long long& an) {
  amax = an = 0;
  for (int i = lane; i <= j; i += 32) {
    const double a = fabs(i < j ? r.al[i] : aj), b = r.be[i];
    amax = max(amax, max(bits_abs(a), bits_abs(b)));
    an = max(an, bits_abs(a + b + (i < j ? r.be[i + 1] : 0.0)));
  }
  amax = warp_max(amax);
  an = warp_max(an);
}

// Before the norm is known: the part of each estimate that does not need it, into
// om_t[0 .. j), and the scales of T.  One block; `a` is alpha_j.
struct ProScales {
  unsigned long long amax, an;   // of tridiag_scale
};
__device__ void pro_prepare(const ProRows& r, int j, double a, double* om_t, ProScales* sc) {
  if ((int)threadIdx.x < 32) {
    unsigned long long amax, an;
    tridiag_scale(r, j, threadIdx.x, a, amax, an);
    if (threadIdx.x == 0) *sc = {amax, an};
  }
  const double bj = j > 0 ? r.be[j] : 0.0;
  for (int k = threadIdx.x; k < j; k += LT) {
    double t = r.be[k + 1] * r.om[k + 1] + (r.al[k] - a) * r.om[k] - bj * r.omp[k];
    if (k > 0) t += r.be[k] * r.om[k - 1];
    om_t[k] = t;
  }
}

// The decision of a step, by one block, from |w|^2 = acc and what pro_prepare left.
// Returns whether the step takes the pass; `word` (unless null) receives it for the
// other CTAs as soon as it is known.
__device__ bool pro_decide(const LanczosDev& L, int j, double acc, double a, double bj, int last, int forced,
                           double** next_slot, double tau, double eps1, double* om_t, const ProScales& sc,
                           unsigned long long* word) {
  __shared__ double s_b, s_inv;
  __shared__ unsigned long long s_mx[4];
  __shared__ int s_pass;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  // the root and the reciprocal root side by side, in two SM quarters
  if (threadIdx.x == 0) s_b = sqrt(acc);
  if (threadIdx.x == 32) s_inv = rsqrt(acc);
  __syncthreads();
  const double bn = s_b, inv = s_inv;
  // one warp per SM quarter covers the j + 1 estimates
  if (threadIdx.x < 128) {
    const double an = __longlong_as_double((long long)max(sc.an, bits_abs(fabs(a) + bj + bn)));
    const double round = eps1 * an;
    unsigned long long mx = 0;
    for (int k = threadIdx.x; k <= j; k += 128) {
      const double t = k < j ? om_t[k] : 0.0;
      const double e = k < j ? (t + copysign(round, t)) * inv : round * inv;
      om_t[k] = e;
      // beta_{j+1} = 0 or an overflowing estimate (its bit pattern lies above every
      // finite one's) counts as lost orthogonality
      mx = max(mx, bits_abs(e));
    }
    mx = warp_max(mx);
    if (lane == 0) s_mx[wid] = mx;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    const unsigned long long m = max(max(s_mx[0], s_mx[1]), max(s_mx[2], s_mx[3]));
    const int pass = forced || !(tau >= 0.0 && m <= bits_abs(tau));
    s_pass = pass;
    L.state[2] = pass;
    L.state[3] = pass && !forced;
    if (!pass) {
      L.beta[j + 1] = bn;
      L.scratch[3 * L.nmax + 3] = inv;   // for the normalising kernel
      L.state[0] = j + 1;
      if (last || bn < 1e-14 * __longlong_as_double((long long)sc.amax)) L.state[1] = 1;
      else *next_slot = L.V + (int64_t)(j + 1) * L.n;
    }
    if (word)
      asm volatile("st.release.gpu.u64 [%0], %1;" ::"l"(word), "l"(2ull * (j + 1) + (pass ? 1 : 0)) : "memory");
  }
  __syncthreads();
  return s_pass != 0;
}

// Row j of the estimates becomes row j-1, the new ones row j+1.
__device__ __forceinline__ void pro_shift(const LanczosDev& L, int j, bool pass, double eps1, const double* om_t,
                                          const double* om) {
  for (int k = threadIdx.x; k <= j; k += LT) {
    L.omega[L.nmax + 2 + k] = om[k];
    L.omega[k] = pass ? eps1 : om_t[k];
  }
  if (threadIdx.x == 0) L.omega[j + 1] = 1.0;
}

// ---------------------------------------------------------------- one step in one launch
// Waits among the CTAs of a step.  A cluster uses the hardware's cluster barrier.  A
// grid (cooperative: all CTAs resident, which the launch checks) counts arrivals in
// 64-bit words that only grow during a solve (lanczos_init_kernel zeroes them);
// every poll is bounded by the clock (about a second).
constexpr long long STEP_WAIT = 2000000000LL;
constexpr int STEP_CL = 8;   // CTAs of the cluster

__device__ bool poll_at_least(const unsigned long long* word, unsigned long long target) {
  const long long t0 = clock64();
  for (;;) {
    unsigned long long cur;
    asm volatile("ld.acquire.gpu.u64 %0, [%1];" : "=l"(cur) : "l"(word) : "memory");
    if (cur >= target) return true;
    if (clock64() - t0 > STEP_WAIT) return false;
  }
}

__device__ __forceinline__ unsigned long long arrive(unsigned long long* word) {
  unsigned long long old;
  asm volatile("atom.add.release.gpu.u64 %0, [%1], 1;" : "=l"(old) : "l"(word) : "memory");
  return old;
}

// Without ordering memory: that every CTA of the cluster has started is all it says.
__device__ __forceinline__ void cluster_arrive_started() {
  __syncwarp();
  asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_arrive() {
  __syncwarp();
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() {
  __syncwarp();
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// All CTAs; what thread 0 of each wrote before is visible to every thread after.
template <bool CLUSTER>
__device__ bool step_barrier(const LanczosDev& L) {
  if (CLUSTER) {
    cluster_arrive();
    cluster_wait();
    return true;
  }
  bool ok = true;
  if (threadIdx.x == 0) {
    // the count before this arrival lies in [k G, (k + 1) G) at barrier k of G CTAs
    const unsigned long long old = arrive(step_words(L));
    ok = poll_at_least(step_words(L), (old / gridDim.x + 1) * (unsigned long long)gridDim.x);
  }
  return __syncthreads_and(ok) != 0;
}

// Sum over the block, valid in warp 0's first eight lanes.
__device__ __forceinline__ double step_block_sum(double v, double* sh) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  v = warp_sum(v);
  if (lane == 0) sh[wid] = v;
  __syncthreads();
  if (wid == 0) {
    v = lane < LT / 32 ? sh[lane] : 0.0;
#pragma unroll
    for (int o = LT / 64; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  }
  return v;
}

// Leaves this CTA's partial (of step_block_sum) where every CTA's step_total finds it: in
// a cluster in the others' shared memory, else in part[].
template <bool CLUSTER>
__device__ __forceinline__ void step_publish(double v, double* part, double* s_part) {
  static_assert(LT / 32 >= STEP_CL, "lanes that hold the sum");
  if (CLUSTER) {
    if (threadIdx.x < STEP_CL)
      *cooperative_groups::this_cluster().map_shared_rank(s_part + blockIdx.x, threadIdx.x) = v;
  } else if (threadIdx.x == 0) {
    part[blockIdx.x] = v;
  }
}

// Sum of every CTA's partial, in the same order in every CTA; valid in all threads.
template <bool CLUSTER>
__device__ double step_total(const double* part, const double* s_part, double* sh) {
  if (CLUSTER) {   // every warp for itself
    double v = s_part[threadIdx.x & (STEP_CL - 1)];
#pragma unroll
    for (int o = STEP_CL / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
  }
  double v = 0.0;
  for (int b = threadIdx.x; b < (int)gridDim.x; b += LT) v += __ldcg(part + b);
  v = step_block_sum(v, sh);
  if (threadIdx.x == 0) sh[LT / 32] = v;
  __syncthreads();
  return sh[LT / 32];
}

// Dots of w against NG basis vectors from row g0 over this CTA's entries [c0, c1), left
// per thread in sh (NG fixed at compile time, so no FP64 instruction is issued for
// a vector that does not exist).
template <int NG>
__device__ __forceinline__ void multidot_group(const LanczosDev& L, int g0, int64_t c0, int64_t c1,
                                               double (*sh)[LT + 1]) {
  double acc[NG];
#pragma unroll
  for (int i = 0; i < NG; ++i) acc[i] = 0.0;
  for (int64_t x = c0 + threadIdx.x; x < c1; x += LT) {
    const double wx = L.w[x];
    double v[NG];
#pragma unroll
    for (int i = 0; i < NG; ++i) v[i] = L.V[(int64_t)(g0 + i) * L.n + x];
#pragma unroll
    for (int i = 0; i < NG; ++i) acc[i] = fma(v[i], wx, acc[i]);
  }
#pragma unroll
  for (int i = 0; i < NG; ++i) sh[i][threadIdx.x] = acc[i];
}

// Dots of this CTA's entries against V_0 .. V_{m-1} into out[i].
__device__ void block_multidot(const LanczosDev& L, int m, int64_t c0, int64_t c1, double (*sh)[LT + 1],
                               double* out) {
  for (int g0 = 0; g0 < m; g0 += 16) {
    const int ng = m - g0 < 16 ? m - g0 : 16;
    switch ((ng + 1) / 2) {
      case 1: ng == 1 ? multidot_group<1>(L, g0, c0, c1, sh) : multidot_group<2>(L, g0, c0, c1, sh); break;
      case 2: ng == 3 ? multidot_group<3>(L, g0, c0, c1, sh) : multidot_group<4>(L, g0, c0, c1, sh); break;
      case 3: ng == 5 ? multidot_group<5>(L, g0, c0, c1, sh) : multidot_group<6>(L, g0, c0, c1, sh); break;
      case 4: ng == 7 ? multidot_group<7>(L, g0, c0, c1, sh) : multidot_group<8>(L, g0, c0, c1, sh); break;
      case 5: ng == 9 ? multidot_group<9>(L, g0, c0, c1, sh) : multidot_group<10>(L, g0, c0, c1, sh); break;
      case 6: ng == 11 ? multidot_group<11>(L, g0, c0, c1, sh) : multidot_group<12>(L, g0, c0, c1, sh); break;
      case 7: ng == 13 ? multidot_group<13>(L, g0, c0, c1, sh) : multidot_group<14>(L, g0, c0, c1, sh); break;
      default: ng == 15 ? multidot_group<15>(L, g0, c0, c1, sh) : multidot_group<16>(L, g0, c0, c1, sh); break;
    }
    __syncthreads();
    // thread t sums every 16th entry of row t / 16, then its 16 partners combine
    const int row = threadIdx.x >> 4, part = threadIdx.x & 15;
    if (row < ng) {
      double v = 0.0;
#pragma unroll
      for (int q = 0; q < LT / 16; ++q) v += sh[row][part + 16 * q];
#pragma unroll
      for (int o = 8; o > 0; o >>= 1) v += __shfl_down_sync(0xffffu << (threadIdx.x & 16), v, o, 16);
      if (part == 0) out[g0 + row] = v;
    }
    __syncthreads();
  }
}

// A whole Lanczos step after w = H v_j, in one launch: alpha_j = <v_j, w>; the
// three-term step w <- (w - alpha_j v_j) - beta_j v_{j-1} (beta_0 = 0) with |w|^2; the
// decision above, by CTA 0 while the others wait for it; and, in a step that takes it,
// the Gram-Schmidt pass c = V^T w, w <- w - V c against v_0 .. v_j with the new
// norm, beta_{j+1} and the stopping test (by the CTA that finishes last).  Each CTA
// keeps to its own contiguous run of entries, so that only the partial sums cross
// CTAs, in regions of L.partial that no CTA can still be reading when they are
// rewritten.  The sums' order is fixed by the grid.
//
// Bound by latency up to some 10^5 entries and by FP64 issue above (4 fused
// multiply-adds per entry at 2 per clock and SM; a pass 2 (j + 1) + 1 more).  As four
// launches (the dots, the three-term step, and two that returned at once in a step
// without the pass) a step took 22, 27 and 50 us at 4096, 126780 and 1.46M entries;
// in one launch it takes 9.6, 12.5 and 25.5 (ncu, cold caches).
template <bool CLUSTER>
__global__ void __launch_bounds__(LT, 2) lanczos_step_kernel(LanczosDev L, int j, int last, double** next_slot,
                                                             double tau, double eps1, int32_t* status) {
  tnx_grid_dependency();
  __shared__ double sh_rows[16][LT + 1];
  __shared__ double s_v[PRO_MAX];   // estimates, then the pass's coefficients
  __shared__ double sh[32];
  __shared__ ProScales s_sc;
  __shared__ int s_ok, s_pass;
  __shared__ double s_part[2][STEP_CL];
  if (stopped(L.state)) return;   // all CTAs alike: what sets the flag waits for every CTA first
  // A CTA of the cluster may be written to (step_publish) once it is known to run; the wait
  // stands before the first such write, behind the loads.
  if (CLUSTER) cluster_arrive_started();
  const int nb = gridDim.x, tid = threadIdx.x;
  const int64_t chunk = ((L.n + nb - 1) / nb + 31) / 32 * 32;
  const int64_t c0 = min(L.n, chunk * blockIdx.x), c1 = min(L.n, c0 + chunk);
  const double* vj = L.V + (int64_t)j * L.n;
  const double* vp = L.V + (int64_t)(j > 0 ? j - 1 : 0) * L.n;
  double* part = L.partial;   // [nb] alpha (later the pass's norms), [nb] norms, [nb][j + 1] dots
  // a wait that ran out: the solve stops, with an eigenvalue that is not a number, and the
  // call that waits for it fails (the status word of its network)
  auto give_up = [&](int code) {
    if (tid == 0) {
      *(volatile int32_t*)status = code;   // host memory (any of the codes will do)
      L.alpha[j] = __longlong_as_double(0x7FF8000000000000ll);
      L.state[0] = j + 1;
      L.state[1] = 1;
    }
  };

  // Everything that does not depend on the sums is read at once: the first U entries
  // per thread of all three vectors (kept in registers), beta_j and, in CTA 0, T and the
  // estimates; a load that waits for a sum or a decision costs the step its latency.
  constexpr int U = 4;
  const ProRows rows = {&sh_rows[0][0], &sh_rows[0][0] + PRO_MAX, &sh_rows[0][0] + 2 * PRO_MAX,
                        &sh_rows[0][0] + 3 * PRO_MAX};
  static_assert(4 * PRO_MAX <= 16 * (LT + 1), "the rows lie where a pass keeps its products");
  const int64_t x0 = c0 + tid;
  double w0[U], v0[U], p0[U];
#pragma unroll
  for (int u = 0; u < U; ++u) {
    w0[u] = v0[u] = p0[u] = 0.0;
    if (x0 + u * LT < c1) {
      w0[u] = L.w[x0 + u * LT];
      v0[u] = vj[x0 + u * LT];
      p0[u] = vp[x0 + u * LT];
    }
  }
  const double b = j > 0 ? L.beta[j] : 0.0;
  int forced = 0;
  if (blockIdx.x == 0) {
    pro_load(L, j, rows);
    if (tid == 0) forced = L.state[3];
  }
  double acc = 0.0;
#pragma unroll
  for (int u = 0; u < U; ++u)
    if (x0 + u * LT < c1) acc = fma(w0[u], v0[u], acc);
  for (int64_t x = x0 + U * LT; x < c1; x += U * LT) {
    double w[U], v[U];
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (x + u * LT < c1) {
        w[u] = L.w[x + u * LT];
        v[u] = vj[x + u * LT];
      }
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (x + u * LT < c1) acc = fma(w[u], v[u], acc);
  }
  acc = step_block_sum(acc, sh);
  if (CLUSTER) cluster_wait();   // every CTA has started
  step_publish<CLUSTER>(acc, part, s_part[0]);
  if (!step_barrier<CLUSTER>(L)) return give_up(41);
  const double a = step_total<CLUSTER>(part, s_part[0], sh);
  __syncthreads();   // sh is reused

  double nrm = 0.0;
#pragma unroll
  for (int u = 0; u < U; ++u)
    if (x0 + u * LT < c1) {
      const double r = (w0[u] - a * v0[u]) - b * p0[u];
      L.w[x0 + u * LT] = r;
      nrm = fma(r, r, nrm);
    }
  for (int64_t x = x0 + U * LT; x < c1; x += U * LT) {
    double w[U], v[U], p[U];
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (x + u * LT < c1) {
        w[u] = L.w[x + u * LT];
        v[u] = vj[x + u * LT];
        p[u] = vp[x + u * LT];
      }
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (x + u * LT < c1) {
        const double r = (w[u] - a * v[u]) - b * p[u];
        L.w[x + u * LT] = r;
        nrm = fma(r, r, nrm);
      }
  }
  nrm = step_block_sum(nrm, sh);
  step_publish<CLUSTER>(nrm, part + nb, s_part[1]);

  bool pass;
  if (CLUSTER) {
    cluster_arrive();
    if (blockIdx.x == 0) {
      pro_prepare(rows, j, a, s_v, &s_sc);
      if (tid == 0) L.alpha[j] = a;
    }
    cluster_wait();
    if (blockIdx.x == 0) {
      __syncthreads();
      pass = pro_decide(L, j, step_total<CLUSTER>(part + nb, s_part[1], sh), a, b, last, forced, next_slot, tau, eps1, s_v, s_sc,
                        nullptr);
      if (tid < STEP_CL) *cooperative_groups::this_cluster().map_shared_rank(&s_pass, tid) = pass;
      cluster_arrive();
      pro_shift(L, j, pass, eps1, s_v, rows.om);
    } else {
      cluster_arrive();
    }
    cluster_wait();
    pass = s_pass != 0;
  } else {
    unsigned long long* words = step_words(L);
    if (tid == 0) arrive(words + SW);
    if (blockIdx.x == 0) {
      pro_prepare(rows, j, a, s_v, &s_sc);
      if (tid == 0) {
        L.alpha[j] = a;
        s_ok = poll_at_least(words + SW, (unsigned long long)(j + 1) * nb);
      }
      __syncthreads();
      if (!s_ok) return give_up(42);
      pass = pro_decide(L, j, step_total<CLUSTER>(part + nb, s_part[1], sh), a, b, last, forced, next_slot, tau, eps1, s_v, s_sc,
                        words + 2 * SW);
      pro_shift(L, j, pass, eps1, s_v, rows.om);
    } else {
      // nothing is left for these CTAs but to learn whether there is a pass
      if (tid == 0) {
        s_ok = poll_at_least(words + 2 * SW, 2ull * (j + 1));
        s_pass = (int)(*(volatile unsigned long long*)(words + 2 * SW) & 1);
      }
      __syncthreads();
      if (!s_ok) return give_up(43);
      pass = s_pass != 0;
    }
  }
  if (!pass) return;

  __syncthreads();   // the rows and estimates have been read
  const int m = j + 1;
  double* dots = part + 2 * nb;
  block_multidot(L, m, c0, c1, sh_rows, dots + (int64_t)blockIdx.x * m);
  __threadfence();   // the dots come from 16 threads, the barrier's arrival from one
  __syncthreads();
  if (!step_barrier<CLUSTER>(L)) return give_up(44);
  for (int i = tid >> 5; i < m; i += LT / 32) {
    double v = 0.0;
    for (int q = tid & 31; q < nb; q += 32) v += __ldcg(dots + (int64_t)q * m + i);
    v = warp_sum(v);
    if ((tid & 31) == 0) s_v[i] = v;
  }
  __syncthreads();
  nrm = 0.0;
  for (int64_t x = c0 + tid; x < c1; x += LT) {
    double w = L.w[x];
#pragma unroll 8
    for (int i = 0; i < m; ++i) w -= s_v[i] * L.V[(int64_t)i * L.n + x];
    L.w[x] = w;
    nrm = fma(w, w, nrm);
  }
  nrm = step_block_sum(nrm, sh);
  if (tid == 0) part[blockIdx.x] = nrm;
  if (last_block(L.state + 4)) {
    beta_decide(L, j, nb, last, next_slot);
    if (tid == 0) L.state[4] = 0;
  }
}

__global__ void lanczos_normalize_kernel(LanczosDev L, int j) {
  tnx_grid_dependency();
  if (stopped(L.state)) return;
  const double inv = L.scratch[3 * L.nmax + 3];   // 1 / beta_{j+1}, one FP64 division per step
  double* vn = L.V + (int64_t)(j + 1) * L.n;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < L.n; i += (int64_t)gridDim.x * blockDim.x)
    vn[i] = L.w[i] * inv;
}

// A key that orders doubles as integers (-0 and +0 share key 0), and back.
__device__ __forceinline__ long long dkey(double x) {
  const long long b = __double_as_longlong(x);
  return b >= 0 ? b : (long long)(0x8000000000000000ull - (unsigned long long)b);
}
__device__ __forceinline__ double dfromkey(long long key) {
  return __longlong_as_double(key >= 0 ? key : (long long)(0x8000000000000000ull - (unsigned long long)key));
}

// Doubles between lo and hi >= lo (unsigned: keys of both signs lie up to 2^64 apart).
__device__ __forceinline__ unsigned long long doubles_between(double lo, double hi) {
  return (unsigned long long)dkey(hi) - (unsigned long long)dkey(lo);
}

// Whether T - xI has an eigenvalue <= 0, i.e. whether its leading minors p_j are not
// all positive: p_{j+1} = (a_j - x) p_j - b_j^2 p_{j-1} (b2[j] = beta_j^2, b2[0] = 0).
// The pivots of the LDL^T factorisation are p_{j+1} / p_j, so this is Sturm's count
// >= 1 without a division per row (three FP64 instructions instead of twelve).
// The pair is rescaled by exponents when it leaves the middle of the range.
__device__ bool eigenvalue_below(const double* a, const double* b2, int k, double x) {
  double pm = 0.0, p = 1.0;
  for (int j = 0; j < k; ++j) {
    const double r = fma(a[j] - x, p, -(b2[j] * pm));
    pm = p;
    p = r;
    const int hi = __double2hiint(p);
    if (hi < 0 || (hi | __double2loint(p)) == 0) return true;   // negative, or zero (counted as negative)
    const int ex = hi >> 20;
    if (ex < 600 || (ex > 1450 && ex < 2047)) {
      const int sh = (ex < 600 ? 500 : -500) << 20, hm = __double2hiint(pm);
      p = __hiloint2double(hi + (ex > 0 ? sh : 0), __double2loint(p));
      const int em = (hm >> 20) + (sh >> 20);
      pm = hm >> 20 > 0 && em > 0 && em < 2047 ? __hiloint2double(hm + sh, __double2loint(pm)) : 0.0;
    }
  }
  return false;
}

// Lowest eigenvalue of T by multisection: each of the TT threads tests its own
// point of the current bracket, and the bracket shrinks to the one sub-interval
// where the test first holds (the same test as bisection, TT points per round),
// until at most TT doubles are left, which the threads test one by one: the
// result is the smallest double of the bracket for which the test holds, as
// bisection to adjacent doubles finds it.  Then inverse iteration (Thomas
// algorithm, 3 sweeps) for the eigenvector y, by one warp (its serial parts by all
// lanes alike).  beta[j] couples rows j-1 and j (beta[0] unused).  T is copied to
// shared memory first; the LU factors of T - shift I are the same in every sweep
// and computed once.  Four warps, one per SM quarter: more would queue for the
// quarters' FP64 units (an instruction takes one 64 cycles).  172 -> 54 us for
// 20 steps (with 256 threads and a division per row and point before).
constexpr int TD_MAX = 512;   // Lanczos steps are limited to 500
constexpr int TT = 128;

__global__ void __launch_bounds__(TT) tridiag_kernel(LanczosDev L) {
  tnx_grid_dependency();
  __shared__ double sa[TD_MAX], sb[TD_MAX], sb2[TD_MAX], sl[TD_MAX], sy[TD_MAX];
  __shared__ double s_x[TT];
  __shared__ long long s_key[2][TT / 32];
  __shared__ int s_first[TT / 32];
  const int k = L.state[0];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  for (int j = threadIdx.x; j < k; j += TT) {
    sa[j] = L.alpha[j];
    sb[j] = L.beta[j];
    sb2[j] = j > 0 ? sb[j] * sb[j] : 0.0;
  }
  __syncthreads();
  // Gershgorin bracket, compared as ordered integers
  long long klo = INT64_MAX, khi = INT64_MIN;
  for (int j = threadIdx.x; j < k; j += TT) {
    const double r = (j > 0 ? fabs(sb[j]) : 0.0) + (j + 1 < k ? fabs(sb[j + 1]) : 0.0);
    klo = min(klo, dkey(sa[j] - r));
    khi = max(khi, dkey(sa[j] + r));
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    klo = min(klo, __shfl_xor_sync(0xffffffffu, klo, o));
    khi = max(khi, __shfl_xor_sync(0xffffffffu, khi, o));
  }
  if (lane == 0) {
    s_key[0][wid] = klo;
    s_key[1][wid] = khi;
  }
  __syncthreads();
  for (int w = 0; w < TT / 32; ++w) {
    klo = min(klo, s_key[0][w]);
    khi = max(khi, s_key[1][w]);
  }
  double lo = dfromkey(klo), hi = dfromkey(khi);
  // index of the first thread whose test holds (TT: none); every thread gets it
  auto first = [&](bool holds) {
    const unsigned m = __ballot_sync(0xffffffffu, holds);
    if (lane == 0) s_first[wid] = m ? __ffs(m) - 1 + 32 * wid : TT;
    __syncthreads();
    int f = TT;
    for (int w = TT / 32 - 1; w >= 0; --w)
      if (s_first[w] < TT) f = s_first[w];
    __syncthreads();
    return f;
  };
  const double frac = (double)(threadIdx.x + 1) / (double)(TT + 1);
  for (int round = 0; round < 96 && doubles_between(lo, hi) > TT; ++round) {
    const double x = lo + (hi - lo) * frac;
    s_x[threadIdx.x] = x;
    const int f = first(dkey(x) > dkey(lo) && dkey(x) < dkey(hi) && eigenvalue_below(sa, sb2, k, x));
    const double nlo = f == 0 ? lo : s_x[f - 1], nhi = f == TT ? hi : s_x[f];
    __syncthreads();   // s_x is rewritten in the next round
    const bool same = nlo <= lo && nhi >= hi;
    if (nlo > lo) lo = nlo;
    if (nhi < hi) hi = nhi;
    if (same) break;
  }
  for (int it = 0; it < 200 && doubles_between(lo, hi) > TT; ++it) {   // what rounding left: plain halving
    const double mid = 0.5 * (lo + hi);
    if (mid <= lo || mid >= hi) break;
    if (eigenvalue_below(sa, sb2, k, mid)) hi = mid; else lo = mid;
  }
  const unsigned long long span = doubles_between(lo, hi);   // hi itself counts
  const int t = first((unsigned long long)threadIdx.x + 1 < span &&
                      eigenvalue_below(sa, sb2, k, dfromkey(dkey(lo) + threadIdx.x + 1)));
  if (wid != 0) return;
  const double lam = t < TT ? dfromkey(dkey(lo) + t + 1) : hi;
  if (lane == 0) *L.eval = lam;
  // LU of T - shift I (no pivoting): sl the multipliers, sb2 the pivots' reciprocals
  const double shift = lam - 1e-13 * fmax(1.0, fabs(lam));
  double inv = 0.0;
  for (int j = 0; j < k; ++j) {
    double piv = sa[j] - shift;
    if (j > 0) {
      const double l = sb[j] * inv;
      sl[j] = l;
      piv = fma(-l, sb[j], piv);
    }
    inv = 1.0 / (piv != 0.0 ? piv : 1e-300);
    sb2[j] = inv;
  }
  const double inv0 = 1.0 / sqrt((double)k);
  for (int j = lane; j < k; j += 32) sy[j] = inv0;
  __syncwarp();
  for (int sweep = 0; sweep < 3; ++sweep) {
    double y = sy[0];
    for (int j = 1; j < k; ++j) {
      y = fma(-sl[j], y, sy[j]);
      __syncwarp();
      sy[j] = y;
    }
    y = y * sb2[k - 1];
    __syncwarp();
    sy[k - 1] = y;
    for (int j = k - 2; j >= 0; --j) {
      y = fma(-sb[j + 1], y, sy[j]) * sb2[j];
      __syncwarp();
      sy[j] = y;
    }
    __syncwarp();
    double nrm = 0.0;
    for (int j = lane; j < k; j += 32) nrm = fma(sy[j], sy[j], nrm);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) nrm += __shfl_xor_sync(0xffffffffu, nrm, o);
    const double f = 1.0 / sqrt(nrm);
    for (int j = lane; j < k; j += 32) sy[j] *= f;
    __syncwarp();
  }
  int jm = 0;
  unsigned long long best = 0;
  for (int j = 0; j < k; ++j)
    if (bits_abs(sy[j]) > best) {
      best = bits_abs(sy[j]);
      jm = j;
    }
  const double sgn = sy[jm] < 0 ? -1.0 : 1.0;
  for (int j = lane; j < k; j += 32) L.y[j] = sgn * sy[j];
}

__global__ void __launch_bounds__(RT) ritz_kernel(LanczosDev L, double* out) {
  tnx_grid_dependency();
  __shared__ double c[512];
  const int k = L.state[0];
  for (int i = threadIdx.x; i < k; i += RT) c[i] = L.y[i];
  __syncthreads();
  for (int64_t x = (int64_t)blockIdx.x * RT + threadIdx.x; x < L.n; x += (int64_t)gridDim.x * RT) {
    double s = 0.0;
    for (int i = 0; i < k; ++i) s += c[i] * L.V[(int64_t)i * L.n + x];
    out[x] = s;
  }
}

int grid_for(int64_t n) {
  int64_t b = (n + RT - 1) / RT;
  return (int)(b < RBLOCKS ? (b < 1 ? 1 : b) : RBLOCKS);
}

}  // namespace

int tnx_reduce_blocks(int64_t n) { return grid_for(n); }

cudaError_t tnx_launch_scale(double* x, int64_t n, double alpha, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  {
    const cudaError_t le = tnx_launch(scale_kernel, dim3(grid_for(n)), dim3(RT), 0, st, x, n, alpha);
    if (le != cudaSuccess) return le;
  }
  tnx_note_launch(1);
  return cudaGetLastError();
}

cudaError_t tnx_launch_add_scalar(double* x, int64_t n, double alpha, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  {
    const cudaError_t le = tnx_launch(add_scalar_kernel, dim3(grid_for(n)), dim3(RT), 0, st, x, n, alpha);
    if (le != cudaSuccess) return le;
  }
  tnx_note_launch(1);
  return cudaGetLastError();
}

cudaError_t tnx_launch_norm2(const double* x, int64_t n, double* partial, double* out, cudaStream_t st) {
  const int nb = grid_for(n);
  {
    const cudaError_t le = tnx_launch(dot_partial_kernel, dim3(nb), dim3(RT), 0, st, x, x, n, partial, nullptr);
    if (le != cudaSuccess) return le;
  }
  tnx_note_launch(1);
  {
    const cudaError_t le = tnx_launch(finalize_kernel, dim3(1), dim3(RT), 0, st, partial, nb, out, 1, nullptr);
    if (le != cudaSuccess) return le;
  }
  tnx_note_launch(1);
  return cudaGetLastError();
}

cudaError_t tnx_launch_lanczos_init(const LanczosDev& L, const double* v0, cudaStream_t st) {
  const int nb = grid_for(L.n);
  {
    const cudaError_t le = tnx_launch(dot_partial_kernel, dim3(nb), dim3(RT), 0, st, v0, v0, L.n, L.partial, nullptr);
    if (le != cudaSuccess) return le;
  }
  tnx_note_launch(1);
  {
    const cudaError_t le = tnx_launch(finalize_kernel, dim3(1), dim3(RT), 0, st,
                                      L.partial, nb, L.scratch, 1, nullptr);
    if (le != cudaSuccess) return le;
  }
  tnx_note_launch(1);
  {
    const cudaError_t le = tnx_launch(lanczos_init_kernel, dim3(nb), dim3(RT), 0, st, L, v0);
    if (le != cudaSuccess) return le;
  }
  tnx_note_launch(1);
  return cudaGetLastError();
}

cudaError_t tnx_launch_lanczos_set_input(double** slot_ptr, const LanczosDev& L, int j, cudaStream_t st) {
  {
    const cudaError_t le = tnx_launch(set_slot_kernel, dim3(1), dim3(1), 0, st, slot_ptr, L.V + (int64_t)j * L.n);
    if (le != cudaSuccess) return le;
  }
  tnx_note_launch(1);
  return cudaGetLastError();
}

// The operator has been applied: L.w = H v_j.  One Lanczos step (without the
// final v_{j+1} = w / beta_{j+1} when `normalize` is false: the caller then
// fuses it with the next apply's relayout of the vector).
//
// Up to 20480 entries the step is one cluster of eight CTAs (barriers and partial sums
// stay among eight SMs, and its launch overlaps the end of the apply); above, where eight
// SMs' FP64 units would bound it, a resident grid of CTAs of 1024 entries, at most one
// per SM up to 4096 entries each, then two (more loads in flight).  Whole solves of 20
// steps, cluster | grid: 4096 entries 1033 | 1100 us, 16384 1179 | 1208, 25676 1538 |
// 1515, 37344 1117 | 1049, 126780 1661 | 1330; one | two CTAs per SM: 1.46M entries
// 5757 | 5676 us.
constexpr int64_t STEP_CLUSTER_MAX = 20480;

cudaError_t tnx_launch_lanczos_step(const LanczosDev& L, int j, double** next_slot, cudaStream_t st, bool normalize,
                                    bool always_pass, int32_t* status) {
  if (j + 2 > PRO_MAX) return cudaErrorInvalidValue;
  const double tau = always_pass ? -1.0 : 1e-10;
  const double eps1 = sqrt((double)L.n) * 0.5 * 2.220446049250313e-16;
  const int last = j == L.nmax - 1;
  const bool cluster = L.n <= STEP_CLUSTER_MAX;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute at[2];
  cfg.blockDim = dim3(LT);
  cfg.stream = st;
  cfg.attrs = at;
  if (cluster) {
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    at[1].id = cudaLaunchAttributeClusterDimension;
    at[1].val.clusterDim.x = STEP_CL;
    at[1].val.clusterDim.y = at[1].val.clusterDim.z = 1;
    cfg.numAttrs = 2;
    cfg.gridDim = dim3(STEP_CL);
  } else {
    int dev = 0, nsm = 0, per_sm = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, lanczos_step_kernel<false>, LT, 0);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) return cudaErrorNotSupported;
    const int64_t want = (L.n + 4 * LT - 1) / (4 * LT);
    int64_t nb = want <= nsm ? want : want <= 4 * (int64_t)nsm || per_sm < 2 ? nsm : 2 * (int64_t)nsm;
    if (nb > TNX_LANCZOS_BLOCKS) nb = TNX_LANCZOS_BLOCKS;
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
    cfg.numAttrs = 1;
    cfg.gridDim = dim3((unsigned)nb);
  }
  const cudaError_t le = cluster
      ? cudaLaunchKernelEx(&cfg, lanczos_step_kernel<true>, L, j, last, next_slot, tau, eps1, status)
      : cudaLaunchKernelEx(&cfg, lanczos_step_kernel<false>, L, j, last, next_slot, tau, eps1, status);
  if (le != cudaSuccess) return le;
  tnx_note_launch(1);
  if (normalize) {
    const cudaError_t e = tnx_launch(lanczos_normalize_kernel, dim3(grid_for(L.n)), dim3(RT), 0, st, L, j);
    if (e != cudaSuccess) return e;
    tnx_note_launch(1);
  }
  return cudaGetLastError();
}

cudaError_t tnx_launch_lanczos_finish(const LanczosDev& L, double* evec, cudaStream_t st) {
  {
    const cudaError_t le = tnx_launch(tridiag_kernel, dim3(1), dim3(TT), 0, st, L);
    if (le != cudaSuccess) return le;
  }
  tnx_note_launch(1);
  if (evec) {
    {
      const cudaError_t le = tnx_launch(ritz_kernel, dim3(grid_for(L.n)), dim3(RT), 0, st, L, evec);
      if (le != cudaSuccess) return le;
    }
    tnx_note_launch(1);
  }
  return cudaGetLastError();
}
