// Fused skinny contraction step: gather, FP64 product, scatter in one kernel.
//
// A contraction whose charge groups all have K <= 16 (the MPO step of the
// two-site H_eff, Sec. 11) is a small FP64 product between two relayouts: its
// operand A is gathered from the previous step's output blocks into the packed
// K-major matrix, and its output C is immediately relaid into the next step's
// packed operand.  Here one CTA takes a run of tiles of up to 128 rows (p, q) of one
// row block of A_g.  It lists the nonzeros of every column of the packed B_g (the
// MPO product is mostly zeros) and stages the columns' descriptors once, then per tile:
//   1. every A element of the tile is read from its source block through the
//      descriptor of its column (consecutive threads take consecutive q, the
//      source blocks' contiguous leg) one tile ahead, and put into the A rows in
//      shared memory;
//   2. two threads form each output row (even and odd columns), with the same FMA
//      chains as the unfused skinny kernel (bit-identical; a power-of-two first
//      coefficient is applied on the integer units, tnx_first_term);
//   3. every output element is stored through the descriptor of its column
//      straight into the next step's packed operand (consecutive threads take
//      consecutive p, that operand's contiguous leg), or the rows are written to
//      C_g when no next step reads them through descriptors.
// The packed A and the C rows never reach HBM when both ends are fused.  The
// descriptors are precomputed by the planner from the two relayouts' bands.
//
// Instruction issue bounds it: a charge group has only a few columns, so with one
// tile per CTA a thread formed 2.4 outputs on average and the warp issued 430
// instructions for them, mostly the lists, descriptors and index setup, which a
// run of tiles (tnx_fused_runs, tnx_network.cpp) shares: one apply of the Heisenberg
// H_eff (ncu, cold) at bond dimension 2048 75 -> 62 us, 4096 244 -> 188 us.
#include "tnx_internal.h"

namespace {

constexpr int FR = TNX_FUSED_ROWS; // a tile has FR rows at most, two threads per row
constexpr int FT = 2 * FR;         // threads
constexpr int FMAXN = 64;         // output columns (rows of B_g) at most
constexpr int FMAXK = 16;         // columns of A (ldK) at most
// the prologue's thread ranges: B nonzeros by threads [FR, FR + N), output
// column descriptors by [FR + FMAXN, FR + FMAXN + N), N <= FMAXN
static_assert(FR + 2 * FMAXN <= FT, "the fused tile needs FR >= 2 * FMAXN rows (threads for its prologue loads)");
static_assert((FR & (FR - 1)) == 0, "the fused tile row count must be a power of two");

struct FusedSmem {
  double s_v[FMAXN][FMAXK];       // nonzero B entries of each output column
  FusedCol s_sc[FMAXN];           // output column descriptors
  unsigned char s_k[FMAXN][FMAXK];
  int s_cnt[FMAXN];
  uint32_t s_p2[FMAXN];           // tnx_pow2_code of each column's first nonzero
};

// t / d for 0 <= t < FR and 1 <= d <= FR through m = ceil(2^16 / d): the estimate
// exceeds t / d by less than t / 2^16 < 1 / d.
__device__ __forceinline__ int small_magic(int d) { return (65536 + d - 1) / d; }
__device__ __forceinline__ int small_div(int t, int m) { return (t * m) >> 16; }

// RUN false: every run of the launch is one tile (nothing is read ahead).
template <bool RUN>
__global__ void __launch_bounds__(FT, RUN ? 5 : 6) fused_skinny_kernel(const GemmGroup* __restrict__ groups,
                                                          const FusedTile* __restrict__ tiles,
                                                          const FusedCol* __restrict__ cols, int kp, int np,
                                                          double* const* __restrict__ slots) {
  tnx_grid_dependency();
  extern __shared__ __align__(16) unsigned char dyn[];
  FusedSmem& S = *(FusedSmem*)dyn;
  double* sA = (double*)(dyn + sizeof(FusedSmem));   // [rows][kp]
  double* sC = sA + FR * kp;                         // [rows][np]
  FusedCol* s_gc = (FusedCol*)(sC + FR * np);        // RUN: [W] A column descriptors
  const FusedTile T = tiles[blockIdx.x];
  const int tid = threadIdx.x, half = tid / FR, t = tid & (FR - 1);
  const int W = T.W, N = T.N;
  // column descriptors: A's by threads [0, W), the output's by [FR + FMAXN, FR + FMAXN + N)
  if (RUN && tid < W) s_gc[tid] = cols[T.gcol + tid];
  if (tid >= FR + FMAXN && tid - FR - FMAXN < N && T.scol >= 0) S.s_sc[tid - FR - FMAXN] = cols[T.scol + tid - FR - FMAXN];
  // B nonzeros (threads [FR, FR + N))
  const GemmGroup g = groups[T.group];
  if (half == 1 && t < N) {
    const int K = g.K;
    const double* brow = slots[g.b_slot] + g.b_off + (int64_t)t * g.ldb;
    double b[FMAXK];
#pragma unroll
    for (int k = 0; k < FMAXK; ++k) b[k] = k < K ? brow[k] : 0.0;
    int c = 0;
#pragma unroll
    for (int k = 0; k < FMAXK; ++k) {
      if (b[k] != 0.0) {
        S.s_v[t][c] = b[k];
        S.s_k[t][c] = (unsigned char)k;
        ++c;
      }
    }
    S.s_cnt[t] = c;
    S.s_p2[t] = c ? tnx_pow2_code(S.s_v[t][0]) : 0u;
  }
  // the current tile: rows p in [p0, p0 + tp), q in [q0, q0 + tq)
  const int nQ = RUN ? (T.EQ + T.tQ - 1) / T.tQ : 1;
  const int mQ = RUN ? small_magic(T.tQ) : 0, mP = RUN ? small_magic(T.tP) : 0;
  int p0 = T.p0, q0 = T.q0, tp = T.eP, tq = T.eQ;
  auto over_q = [&](int r) { return !RUN ? r / tq : small_div(r, tq == T.tQ ? mQ : small_magic(tq)); };
  double v[FMAXK / 2];
  // this thread's entries of the tile's A: row t, q fastest; columns half, half + 2, ...
  auto fetch = [&](const FusedCol* gc) {
    if (t < tp * tq) {
      const int p = over_q(t), q = t - p * tq;
      const int P = p0 + p, Q = q0 + q;
#pragma unroll
      for (int j = 0; j < FMAXK / 2; ++j) {
        const int c = half + 2 * j;
        v[j] = 0.0;
        if (c < W) {
          const FusedCol d = gc[c];
          if (d.ptr) v[j] = __ldg(d.ptr + (int64_t)P * d.sP + (int64_t)Q * d.sQ);
        }
      }
    }
  };
  fetch(cols + T.gcol);   // beside the lists' and descriptors' own loads
  int pt = RUN ? T.t0 / nQ : 0, qt = RUN ? T.t0 - pt * nQ : 0;
  for (int i = 0; i < (RUN ? T.nt : 1); ++i) {
    const int rows = tp * tq;
    if (t < rows) {
#pragma unroll
      for (int j = 0; j < FMAXK / 2; ++j) {
        const int c = half + 2 * j;
        if (c < W) sA[t * kp + c] = v[j];
      }
    }
    __syncthreads();
    const int cp0 = p0, cq0 = q0, ctp = tp, ctq = tq;   // this tile, when p0 .. move on to the next
    if (RUN && i + 1 < T.nt) {
      if (++qt == nQ) {
        qt = 0;
        ++pt;
      }
      p0 = pt * T.tP;
      q0 = qt * T.tQ;
      tp = min(T.tP, T.EP - p0);
      tq = min(T.tQ, T.EQ - q0);
      fetch(s_gc);
    }
    if (t < rows) {
      const double* arow = sA + t * kp;
      double* crow = sC + t * np;
      for (int n = half; n < N; n += 2) {
        double acc = 0.0;
        const int c = S.s_cnt[n];
        if (c > 0) acc = tnx_first_term(arow[S.s_k[n][0]], S.s_v[n][0], S.s_p2[n]);
        for (int e = 1; e < c; ++e) acc = fma(arow[S.s_k[n][e]], S.s_v[n][e], acc);
        crow[n] = acc;
      }
    }
    __syncthreads();
    if (T.scol >= 0) {
      // scatter: p fastest (row r = p * tq + q in shared memory)
      if (t < rows) {
        const int q = !RUN ? t / ctp : small_div(t, ctp == T.tP ? mP : small_magic(ctp)), p = t - q * ctp;
        const int P = cp0 + p, Q = cq0 + q;
        const double* crow = sC + (p * ctq + q) * np;
        for (int c = half; c < N; c += 2) {
          const FusedCol d = S.s_sc[c];
          if (d.ptr) d.ptr[(int64_t)P * d.sP + (int64_t)Q * d.sQ] = crow[c];
        }
      }
    } else {
      // row (p, q) of the block is row row0 + p * EQ + q of C_g
      double* C = slots[g.c_slot] + g.c_off;
      for (int e = tid; e < rows * N; e += FT) {
        const int r = e / N, n = e - r * N;
        const int p = !RUN ? r / ctq : small_div(r, ctq == T.tQ ? mQ : small_magic(ctq)), q = r - p * ctq;
        const int64_t row = (int64_t)T.row0 + (int64_t)(cp0 + p) * T.EQ + cq0 + q;
        C[row * g.ldc + n] = sC[r * np + n];
      }
    }
    // the next tile's A rows are written behind this tile's products (the barrier
    // above), its C rows behind these reads of them (the next iteration's barriers)
  }
}

// The same step for small bands (charge blocks of a few rows), one warp per tile of at
// most FR rows.  A row belongs to one lane: it gathers the row's A elements into a column
// of the warp's shared memory that only it reads (the list of nonzeros picks elements by
// number), forms the outputs and stores them at once.  Lanes walk q, then p, of tiles at
// most 8 wide along q when the band allows it, so that 32-byte sectors are read whole
// along q and written whole along p without a transposing stage.
//
// A tile of 128 rows by 8 warps spends its time on the chain of loads before the
// product (tile, group and descriptors, B and A), whatever the number of rows, and an SM
// holds six; here it holds 28 chains.  Still bound by instruction issue and latency (about
// 1000 warp instructions a tile, 40% of the issue slots, FP64 pipe 30%).  48 Hubbard
// sites (75 thousand bands of 1 to 256 rows): 166 us for what took 178 (the instances
// with 32 rows per tile and more) and 135 (relayouts and skinny products of the others)
// before; the two MPO steps of one at bond dimension 601: 25 us for 41 (ncu, cold).
constexpr int FW = 4;   // warps per CTA, each on its own tile

__host__ __device__ constexpr size_t warp_smem(int kp, int np) {
  return ((size_t)kp * 32 * 8 + (size_t)np * kp * 9 + (size_t)(kp + np) * sizeof(FusedCol) + (size_t)np * 8 + 15) / 16 *
         16;
}

__global__ void __launch_bounds__(32 * FW, 8) fused_warp_kernel(const GemmGroup* __restrict__ groups,
                                                                const FusedTile* __restrict__ tiles, int ntiles,
                                                                const FusedCol* __restrict__ cols, int kp, int np,
                                                                double* const* __restrict__ slots) {
  tnx_grid_dependency();
  extern __shared__ __align__(16) unsigned char dyn[];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int ti = blockIdx.x * FW + wid;
  if (ti >= ntiles) return;
  unsigned char* base = dyn + (size_t)wid * warp_smem(kp, np);
  FusedCol* s_d = (FusedCol*)base;                        // [kp] of A, [np] of the output
  double* s_a = (double*)(s_d + kp + np) + lane;          // [kp][32]: this lane's column
  double* s_v = (double*)(s_d + kp + np) + kp * 32;       // [np][kp] nonzeros
  int* s_cnt = (int*)(s_v + np * kp);                     // [np]
  uint32_t* s_p2 = (uint32_t*)(s_cnt + np);               // [np]
  unsigned char* s_k = (unsigned char*)(s_p2 + np);       // [np][kp]
  const FusedTile T = tiles[ti];
  const int W = T.W, N = T.N;
  const GemmGroup g = groups[T.group];
  const int nd = T.scol >= 0 ? W + N : W;
  for (int i = lane; i < nd; i += 32) s_d[i < W ? i : kp + i - W] = cols[i < W ? T.gcol + i : T.scol + i - W];
  for (int n = lane; n < N; n += 32) {
    const double* brow = slots[g.b_slot] + g.b_off + (int64_t)n * g.ldb;
    int c = 0;
    for (int k0 = 0; k0 < g.K; k0 += 4) {
      double b[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) b[k] = k0 + k < g.K ? brow[k0 + k] : 0.0;
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        if (b[k] != 0.0) {
          s_v[n * kp + c] = b[k];
          s_k[n * kp + c] = (unsigned char)(k0 + k);
          ++c;
        }
      }
    }
    s_cnt[n] = c;
    s_p2[n] = c ? tnx_pow2_code(s_v[n * kp]) : 0u;
  }
  __syncwarp();
  double* C = T.scol >= 0 ? nullptr : slots[g.c_slot] + g.c_off;
  const int rows = T.eP * T.eQ, mq = small_magic(T.eQ);
  for (int r = lane; r < rows; r += 32) {
    const int p = small_div(r, mq), q = r - p * T.eQ;
    const int64_t P = T.p0 + p, Q = T.q0 + q;
    for (int c0 = 0; c0 < W; c0 += 4) {
      double v[4];
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        v[c] = 0.0;
        if (c0 + c < W) {
          const FusedCol d = s_d[c0 + c];
          if (d.ptr) v[c] = __ldg(d.ptr + P * d.sP + Q * d.sQ);
        }
      }
#pragma unroll
      for (int c = 0; c < 4; ++c)
        if (c0 + c < W) s_a[(c0 + c) * 32] = v[c];
    }
    for (int n = 0; n < N; ++n) {
      double acc = 0.0;
      const int c = s_cnt[n];
      const double* bv = s_v + n * kp;
      const unsigned char* bk = s_k + n * kp;
      if (c > 0) acc = tnx_first_term(s_a[bk[0] * 32], bv[0], s_p2[n]);
      for (int e = 1; e < c; ++e) acc = fma(s_a[bk[e] * 32], bv[e], acc);
      if (C) {
        C[((int64_t)T.row0 + P * T.EQ + Q) * g.ldc + n] = acc;
      } else {
        const FusedCol d = s_d[kp + n];
        if (d.ptr) d.ptr[P * d.sP + Q * d.sQ] = acc;
      }
    }
  }
}

}  // namespace

size_t tnx_fused_smem_bytes(int kp, int np) { return sizeof(FusedSmem) + (size_t)FR * (kp + np) * sizeof(double); }

namespace {
template <bool RUN>
cudaError_t launch_fused(const GemmGroup* groups, const FusedTile* tiles, int ntiles, const FusedCol* cols, int kp,
                         int np, double* const* slots, cudaStream_t st) {
  static int attr_dev = -1;   // the opt-in is per device
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (attr_dev != dev) {
    e = cudaFuncSetAttribute(fused_skinny_kernel<RUN>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)(tnx_fused_smem_bytes(FMAXK + 1, FMAXN + 1) + FMAXK * sizeof(FusedCol)));
    if (e != cudaSuccess) return e;
    attr_dev = dev;
  }
  const size_t smem = tnx_fused_smem_bytes(kp, np) + (RUN ? FMAXK * sizeof(FusedCol) : 0);
  return tnx_launch(fused_skinny_kernel<RUN>, dim3(ntiles), dim3(FT), smem, st, groups, tiles, cols, kp, np, slots);
}
cudaError_t launch_fused_warp(const GemmGroup* groups, const FusedTile* tiles, int ntiles, const FusedCol* cols, int kp,
                              int np, double* const* slots, cudaStream_t st) {
  static int attr_dev = -1;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (attr_dev != dev) {
    e = cudaFuncSetAttribute(fused_warp_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)(FW * warp_smem(FMAXK + 1, FMAXN + 1)));
    if (e != cudaSuccess) return e;
    attr_dev = dev;
  }
  return tnx_launch(fused_warp_kernel, dim3((ntiles + FW - 1) / FW), dim3(32 * FW), FW * warp_smem(kp, np), st, groups,
                    tiles, ntiles, cols, kp, np, slots);
}
}  // namespace

cudaError_t tnx_launch_fused_skinny(const GemmGroup* groups, const FusedTile* tiles, int ntiles, int run,
                                    const FusedCol* cols, int kp, int np, double* const* slots, cudaStream_t st) {
  if (ntiles <= 0) return cudaSuccess;
  if (kp < 1 || kp > FMAXK + 1 || np < 1 || np > FMAXN + 1) return cudaErrorInvalidValue;
  const cudaError_t le = run == 0  ? launch_fused_warp(groups, tiles, ntiles, cols, kp, np, slots, st)
                         : run > 1 ? launch_fused<true>(groups, tiles, ntiles, cols, kp, np, slots, st)
                                   : launch_fused<false>(groups, tiles, ntiles, cols, kp, np, slots, st);
  if (le != cudaSuccess) return le;
  tnx_note_launch(1);
  return cudaGetLastError();
}
