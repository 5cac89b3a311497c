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
// a fixed-order tree (warp shuffles), then one block summing the partials in
// a fixed order.
#include "tnx_internal.h"

namespace {

constexpr int RT = 256;        // threads per reduction block
constexpr int RBLOCKS = 1216;  // 8 blocks per SM on 152 SMs

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

// A gated launch of the Gram-Schmidt pass does nothing unless this step's
// decision asked for the pass.
__device__ __forceinline__ bool gated_off(const int32_t* state, int gate) {
  return gate && *(volatile const int32_t*)(state + 2) == 0;
}

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
    L.beta[0] = 0.0;
    L.omega[0] = 1.0;   // <v_0, v_0>; the row before it is empty
  }
}

__global__ void set_slot_kernel(double** slot, double* p) {
  tnx_grid_dependency();
  *slot = p;
}

// partial[b*m + i] = <V_i, w> over this block's contiguous chunk, i < m.  A
// grid of multidot_blocks(n) blocks keeps the number of partial sums (and so the
// FP64 additions of the reduction tree) bounded; each thread keeps NG <= 16
// running sums (NG fixed at compile time, so no FP64 instruction is issued for
// a vector that does not exist), w is read once per group of vectors, and the
// block reduction goes through shared memory: 16 rows of MD_T values, 8
// threads per row.  FP64 issue slots are scarce on this part, so the grid is
// only large enough to keep the loads in flight.
constexpr int MD_T = 128;
constexpr int MD_BLOCKS_MAX = 608;

// Blocks of the multidot kernel: about 416 vector entries per block (an
// L2-resident basis is bound by FP64 issue, where fewer partial sums help),
// at least 1; above one per SM rounded to a multiple of the SM count, at most 4 per
// SM (a basis in HBM needs the loads of that many blocks in flight).
int multidot_blocks(int64_t n) {
  int64_t b = n / 416;
  if (b < 1) b = 1;
  if (b > 152) b = (b + 151) / 152 * 152;
  if (b > MD_BLOCKS_MAX) b = MD_BLOCKS_MAX;
  return (int)b;
}

template <int NG>
__device__ __forceinline__ void multidot_group(const LanczosDev& L, int g0, int64_t c0, int64_t c1,
                                               double (*sh)[MD_T + 1]) {
  // g0 is the basis row of the group's first vector
  double acc[NG];
#pragma unroll
  for (int i = 0; i < NG; ++i) acc[i] = 0.0;
  // two entries per iteration: both rows' loads are in flight before the FMAs
  int64_t x = c0 + threadIdx.x;
  for (; x + MD_T < c1; x += 2 * MD_T) {
    const double w0 = L.w[x], w1 = L.w[x + MD_T];
    double v0[NG], v1[NG];
#pragma unroll
    for (int i = 0; i < NG; ++i) {
      v0[i] = L.V[(int64_t)(g0 + i) * L.n + x];
      v1[i] = L.V[(int64_t)(g0 + i) * L.n + x + MD_T];
    }
#pragma unroll
    for (int i = 0; i < NG; ++i) acc[i] = fma(v1[i], w1, fma(v0[i], w0, acc[i]));
  }
  if (x < c1) {
    const double wx = L.w[x];
#pragma unroll
    for (int i = 0; i < NG; ++i) acc[i] = fma(L.V[(int64_t)(g0 + i) * L.n + x], wx, acc[i]);
  }
#pragma unroll
  for (int i = 0; i < NG; ++i) sh[i][threadIdx.x] = acc[i];
}

// Dots of this block's chunk [c0, c1) against V_vb .. V_{vb+m-1} into partial[b*m + i].
__device__ void block_multidot(const LanczosDev& L, int m, int64_t c0, int64_t c1, double (*sh)[MD_T + 1],
                               int vb = 0) {
  for (int g0 = 0; g0 < m; g0 += 16) {
    const int ng = m - g0 < 16 ? m - g0 : 16;
    const int r0 = vb + g0;
    switch (ng) {
      case 1: multidot_group<1>(L, r0, c0, c1, sh); break;
      case 2: multidot_group<2>(L, r0, c0, c1, sh); break;
      case 3: multidot_group<3>(L, r0, c0, c1, sh); break;
      case 4: multidot_group<4>(L, r0, c0, c1, sh); break;
      case 5: multidot_group<5>(L, r0, c0, c1, sh); break;
      case 6: multidot_group<6>(L, r0, c0, c1, sh); break;
      case 7: multidot_group<7>(L, r0, c0, c1, sh); break;
      case 8: multidot_group<8>(L, r0, c0, c1, sh); break;
      case 9: multidot_group<9>(L, r0, c0, c1, sh); break;
      case 10: multidot_group<10>(L, r0, c0, c1, sh); break;
      case 11: multidot_group<11>(L, r0, c0, c1, sh); break;
      case 12: multidot_group<12>(L, r0, c0, c1, sh); break;
      case 13: multidot_group<13>(L, r0, c0, c1, sh); break;
      case 14: multidot_group<14>(L, r0, c0, c1, sh); break;
      case 15: multidot_group<15>(L, r0, c0, c1, sh); break;
      default: multidot_group<16>(L, r0, c0, c1, sh); break;
    }
    if (ng == 1) {   // a single vector: warp sums (the row sums below would chain 16 additions)
      const double v = warp_sum(sh[0][threadIdx.x]);
      __syncthreads();
      if ((threadIdx.x & 31) == 0) sh[0][threadIdx.x >> 5] = v;
      __syncthreads();
      if (threadIdx.x == 0)
        L.partial[(int64_t)blockIdx.x * m + g0] = (sh[0][0] + sh[0][1]) + (sh[0][2] + sh[0][3]);
      __syncthreads();
      continue;
    }
    __syncthreads();
    // thread t sums 16 consecutive entries of row t/8, then 8 partners combine
    const int row = threadIdx.x >> 3, part = threadIdx.x & 7;
    if (row < ng) {
      double v = 0.0;
#pragma unroll
      for (int q = 0; q < MD_T / 8; ++q) v += sh[row][part * (MD_T / 8) + q];
#pragma unroll
      for (int o = 4; o > 0; o >>= 1) v += __shfl_down_sync(0xffu << (threadIdx.x & 24), v, o, 8);
      if (part == 0) L.partial[(int64_t)blockIdx.x * m + g0 + row] = v;
    }
    __syncthreads();
  }
}

// coef[i] = sum_b partial[b*m + i] over the nb blocks of the launch (fixed
// order); the sum of row alpha_i (if >= 0) is also alpha_j = <v_j, H v_j>.
// Run by one block of any width.
__device__ void finalize_coefs(const LanczosDev& L, int m, int nb, int alpha_i, int alpha_j, double* sh) {
  for (int i = 0; i < m; ++i) {
    double acc = 0.0;
    for (int b = threadIdx.x; b < nb; b += blockDim.x) acc += __ldcg(L.partial + (int64_t)b * m + i);
    acc = nb > 32 ? block_sum(acc, sh) : warp_sum(acc);   // up to 32 partials lie in one warp
    if (threadIdx.x == 0) {
      L.coef[i] = acc;
      if (i == alpha_i) L.alpha[alpha_j] = acc;
    }
  }
}

// Dots of w against V_vb .. V_{vb+m-1}, the coefficients formed by the last block.
__global__ void __launch_bounds__(MD_T) multidot_kernel(LanczosDev L, int m, int vb, int gate, int alpha_i,
                                                        int alpha_j) {
  tnx_grid_dependency();
  __shared__ double sh[16][MD_T + 1];
  __shared__ double shr[32];
  if (stopped(L.state) || gated_off(L.state, gate)) return;
  const int64_t chunk = (L.n + gridDim.x - 1) / gridDim.x;
  const int64_t c0 = chunk * blockIdx.x, c1 = min(L.n, c0 + chunk);
  block_multidot(L, m, c0, c1, sh, vb);
  if (last_block(L.state + 4)) {
    finalize_coefs(L, m, gridDim.x, alpha_i, alpha_j, shr);
    if (threadIdx.x == 0) L.state[4] = 0;
  }
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

// w -= sum_i coef[i] V_i; with norm != 0 also partial[b] = sum of the new w^2
// over this block's grid-stride share (fixed order).
__global__ void __launch_bounds__(RT) gs_update_kernel(LanczosDev L, int m, int norm, int gate, int j, int last,
                                                        double** next_slot) {
  tnx_grid_dependency();
  __shared__ double c[512];
  __shared__ double sh[32];
  if (stopped(L.state) || gated_off(L.state, gate)) return;
  for (int i = threadIdx.x; i < m; i += RT) c[i] = L.coef[i];
  __syncthreads();
  double nrm = 0.0;
  // two entries per iteration (the second one stride later), so that the loads
  // of both are in flight together; each entry keeps its own subtraction order
  const int64_t stride = (int64_t)gridDim.x * RT;
  int64_t x = (int64_t)blockIdx.x * RT + threadIdx.x;
  for (; x + stride < L.n; x += 2 * stride) {
    double w0 = L.w[x], w1 = L.w[x + stride];
#pragma unroll 4
    for (int i = 0; i < m; ++i) {
      const double* vi = L.V + (int64_t)i * L.n;
      const double a0 = vi[x], a1 = vi[x + stride];
      w0 -= c[i] * a0;
      w1 -= c[i] * a1;
    }
    L.w[x] = w0;
    L.w[x + stride] = w1;
    nrm = fma(w0, w0, nrm);
    nrm = fma(w1, w1, nrm);
  }
  if (x < L.n) {
    double w = L.w[x];
#pragma unroll 8
    for (int i = 0; i < m; ++i) w -= c[i] * L.V[(int64_t)i * L.n + x];
    L.w[x] = w;
    nrm = fma(w, w, nrm);
  }
  if (norm) {
    nrm = block_sum(nrm, sh);
    if (threadIdx.x == 0) L.partial[blockIdx.x] = nrm;
    // the last block: beta_{j+1} and the stopping test of this step
    if (last_block(L.state + 4)) {
      beta_decide(L, j, gridDim.x, last, next_slot);
      if (threadIdx.x == 0) L.state[4] = 0;
    }
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
// tau (1e-10; a negative tau: every step), and so does the step after it (the error that v_j carries reaches
// v_{j+2} too); after a pass the estimates restart at eps1.  Without a pass
// it also does what beta_decide does (beta_{j+1}, the stopping
// test, the next input slot); with one, the gated launches after it do.
constexpr int PRO_MAX = 514;   // rows of at most 500 steps + 2

// What a step waits for here is FP64 latency: an FP64 instruction takes its SM
// quarter 64 cycles however few lanes need it (a root ten of them, a division
// nine), so roots and divisions are taken once, by one warp, maxima of
// non-negative numbers are formed on their bit patterns, and eps1 comes from the
// host.  Dense bond dimension 32 (4096 entries): the three-term launch 11.4 -> 9.0 us
// (ncu, cold caches).
__device__ __forceinline__ unsigned long long bits_abs(double x) {
  return (unsigned long long)__double_as_longlong(x) & 0x7FFFFFFFFFFFFFFFull;
}
__device__ __forceinline__ unsigned long long warp_max(unsigned long long v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = max(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

// max(|alpha_i|, beta_i) and max(|alpha_i| + beta_i + beta_{i+1}) over i <= j (beta_{j+1}
// left out), as bit patterns; one warp.
__device__ __forceinline__ void tridiag_scale(const LanczosDev& L, int j, int lane, unsigned long long& amax,
                                              unsigned long long& an) {
  amax = an = 0;
  for (int i = lane; i <= j; i += 32) {
    const double a = fabs(L.alpha[i]), b = L.beta[i];
    amax = max(amax, max(bits_abs(a), bits_abs(b)));
    an = max(an, bits_abs(a + b + (i < j ? L.beta[i + 1] : 0.0)));
  }
  amax = warp_max(amax);
  an = warp_max(an);
}

// Sum of the nb partials, in a fixed order; valid in thread 0.
__device__ double partial_sum(const double* partial, int nb, double* sh) {
  double acc = 0.0;
  for (int b = threadIdx.x; b < nb; b += RT) acc += __ldcg(partial + b);
  if (nb > 32) return block_sum(acc, sh);   // else the other warps hold zeros
  return warp_sum(acc);
}

// Run by one block of RT threads over the nb norm partials.
__device__ void pro_decide(const LanczosDev& L, int j, int nb, int last, double** next_slot, double tau,
                           double eps1) {
  __shared__ double sh[32];
  __shared__ double s_om[PRO_MAX];
  __shared__ double s_b, s_inv;
  __shared__ unsigned long long s_amax, s_an, s_mx[4];
  __shared__ int s_pass;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (wid == 1) {
    unsigned long long amax, an;
    tridiag_scale(L, j, lane, amax, an);
    if (lane == 0) {
      s_amax = amax;
      s_an = an;
    }
  }
  const double acc = partial_sum(L.partial, nb, sh);
  if (threadIdx.x == 0) {
    s_b = sqrt(acc);
    s_inv = 1.0 / s_b;
  }
  __syncthreads();
  const double bn = s_b, inv = s_inv;
  // one warp per SM quarter covers the j + 1 estimates
  if (threadIdx.x < 128) {
    const double* om = L.omega;                  // row j: k = 0..j
    const double* omp = L.omega + (L.nmax + 2);  // row j-1: k = 0..j-1
    const double aj = L.alpha[j], bj = j > 0 ? L.beta[j] : 0.0;
    const double an = __longlong_as_double((long long)max(s_an, bits_abs(fabs(aj) + bj + bn)));
    const double round = eps1 * an;
    unsigned long long mx = 0;
    for (int k = threadIdx.x; k <= j; k += 128) {
      double e;
      if (k < j) {
        double t = L.beta[k + 1] * om[k + 1] + (L.alpha[k] - aj) * om[k] - bj * omp[k];
        if (k > 0) t += L.beta[k] * om[k - 1];
        e = (t + copysign(round, t)) * inv;
      } else {
        e = round * inv;
      }
      s_om[k] = e;
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
    const int forced = L.state[3];
    const int pass = forced || !(tau >= 0.0 && m <= bits_abs(tau));
    s_pass = pass;
    L.state[2] = pass;
    L.state[3] = pass && !forced;
    if (!pass) {
      L.beta[j + 1] = bn;
      L.scratch[3 * L.nmax + 3] = inv;   // for the normalising kernel
      L.state[0] = j + 1;
      if (last || bn < 1e-14 * __longlong_as_double((long long)s_amax)) L.state[1] = 1;
      else *next_slot = L.V + (int64_t)(j + 1) * L.n;
    }
  }
  __syncthreads();
  // shift the rows: row j becomes row j-1, the new estimates row j+1
  double* cur = L.omega;
  double* prev = L.omega + (L.nmax + 2);
  for (int k = threadIdx.x; k <= j; k += RT) {
    prev[k] = cur[k];
    cur[k] = s_pass ? eps1 : s_om[k];
  }
  if (threadIdx.x == 0) cur[j + 1] = 1.0;
}

// The three-term step w <- (w - alpha_j v_j) - beta_j v_{j-1} (beta_0 = 0), with
// partial[b] = this block's share of the new |w|^2 (fixed order).
__global__ void __launch_bounds__(RT) three_term_norm_kernel(LanczosDev L, int j, int last, double** next_slot,
                                                              double tau, double eps1) {
  tnx_grid_dependency();
  __shared__ double sh[32];
  if (stopped(L.state)) return;
  const double a = L.alpha[j], b = j > 0 ? L.beta[j] : 0.0;
  const double* vj = L.V + (int64_t)j * L.n;
  const double* vp = L.V + (int64_t)(j > 0 ? j - 1 : 0) * L.n;
  double nrm = 0.0;
  const int64_t stride = (int64_t)gridDim.x * RT;
  int64_t x = (int64_t)blockIdx.x * RT + threadIdx.x;
  for (; x + stride < L.n; x += 2 * stride) {
    const double w0 = L.w[x], w1 = L.w[x + stride];
    const double a0 = vj[x], a1 = vj[x + stride];
    const double p0 = vp[x], p1 = vp[x + stride];
    const double u0 = (w0 - a * a0) - b * p0, u1 = (w1 - a * a1) - b * p1;
    L.w[x] = u0;
    L.w[x + stride] = u1;
    nrm = fma(u0, u0, nrm);
    nrm = fma(u1, u1, nrm);
  }
  if (x < L.n) {
    const double u = (L.w[x] - a * vj[x]) - b * vp[x];
    L.w[x] = u;
    nrm = fma(u, u, nrm);
  }
  nrm = block_sum(nrm, sh);
  if (threadIdx.x == 0) L.partial[blockIdx.x] = nrm;
  if (last_block(L.state + 4)) {
    pro_decide(L, j, gridDim.x, last, next_slot, tau, eps1);
    if (threadIdx.x == 0) L.state[4] = 0;
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
// fuses it with the next apply's relayout of the vector): alpha_j = <v_j, w>;
// the three-term step w <- w - alpha_j v_j - beta_j v_{j-1} with |w|; the
// orthogonality estimates, which decide whether this step takes a classical
// Gram-Schmidt pass c = V^T w, w <- w - V c against v_0..v_j (the gated
// launches: a step without the pass returns from them at once); then
// beta_{j+1}, the stopping test and v_{j+1} = w / beta_{j+1}.  FP64 work per
// entry: 3 fused multiply-adds, plus 2 (j + 1) + 1 in a step with the pass.
cudaError_t tnx_launch_lanczos_step(const LanczosDev& L, int j, double** next_slot, cudaStream_t st, bool normalize,
                                    bool always_pass) {
  if (j + 2 > PRO_MAX) return cudaErrorInvalidValue;
  const double tau = always_pass ? -1.0 : 1e-10;
  const int nb = grid_for(L.n);
  const int m = j + 1;
  const int mb = multidot_blocks(L.n);
  const int last = j == L.nmax - 1;
  {
    const cudaError_t le = tnx_launch(multidot_kernel, dim3(mb), dim3(MD_T), 0, st, L, 1, j, 0, 0, j);
    if (le != cudaSuccess) return le;
  }
  {
    const cudaError_t le = tnx_launch(three_term_norm_kernel, dim3(nb), dim3(RT), 0, st, L, j, last, next_slot, tau,
                                      sqrt((double)L.n) * 0.5 * 2.220446049250313e-16);
    if (le != cudaSuccess) return le;
  }
  {
    const cudaError_t le = tnx_launch(multidot_kernel, dim3(mb), dim3(MD_T), 0, st, L, m, 0, 1, -1, 0);
    if (le != cudaSuccess) return le;
  }
  {
    const cudaError_t le = tnx_launch(gs_update_kernel, dim3(nb), dim3(RT), 0, st, L, m, 1, 1, j, last, next_slot);
    if (le != cudaSuccess) return le;
  }
  tnx_note_launch(4);
  if (normalize) {
    {
      const cudaError_t le = tnx_launch(lanczos_normalize_kernel, dim3(nb), dim3(RT), 0, st, L, j);
      if (le != cudaSuccess) return le;
    }
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
