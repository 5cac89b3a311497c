// Fused skinny contraction step: gather, FP64 product, scatter in one kernel.
//
// A contraction whose charge groups all have K <= 16 (the MPO step of the
// two-site H_eff, Sec. 11) is a small FP64 product between two relayouts: its
// operand A is gathered from the previous step's output blocks into the packed
// K-major matrix, and its output C is immediately relaid into the next step's
// packed operand.  Here a CTA or a warp takes a tile of up to 128 rows (p, q) of one row
// block of A_g, lists the nonzeros of every column of the packed B_g (the MPO product is
// mostly zeros), reads every A element of the tile from its source block through
// the descriptor of its column, forms the output rows with the same FMA chains as the
// unfused skinny kernel (bit-identical; a power-of-two first coefficient is applied on
// the integer units, tnx_first_term), and stores every output element through the
// descriptor of its column straight into the next step's packed operand, or writes the
// rows to C_g when no next step reads them through descriptors.  The packed A and
// the C rows never reach HBM when both ends are fused.  The descriptors are precomputed by
// the planner from the two relayouts' bands.
//
// Which of the kernels takes a launch is decided by tnx_fused_tiles (tnx_network.cpp).
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

// One CTA per tile, two threads per row (even and odd columns): A goes to shared memory
// along q, the source blocks' contiguous leg, and the output leaves it along p, the next
// operand's.  For launches of few tiles, whose time is one tile's chain of loads and
// products: 186 tiles (Heisenberg at bond dimension 150) 7.3 us against 9.7 with the
// kernel below, 1372 tiles (512) 11.0 against 10.8 (ncu, cold).
__global__ void __launch_bounds__(FT, 6) fused_skinny_kernel(const GemmGroup* __restrict__ groups,
                                                             const FusedTile* __restrict__ tiles,
                                                             const FusedCol* __restrict__ cols, int kp, int np,
                                                             double* const* __restrict__ slots) {
  tnx_grid_dependency();
  extern __shared__ __align__(16) unsigned char dyn[];
  FusedSmem& S = *(FusedSmem*)dyn;
  double* sA = (double*)(dyn + sizeof(FusedSmem));   // [rows][kp]
  double* sC = sA + FR * kp;                         // [rows][np]
  const FusedTile T = tiles[blockIdx.x];
  const int tid = threadIdx.x, half = tid / FR, t = tid & (FR - 1);
  const int W = T.W, N = T.N, tq = T.eQ, tp = T.eP, rows = tp * tq;
  // output column descriptors (threads [FR + FMAXN, FR + FMAXN + N))
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
  // this thread's entries of A: row t, q fastest; columns half, half + 2, ...
  if (t < rows) {
    const int p = t / tq, q = t - p * tq;
    const int P = T.p0 + p, Q = T.q0 + q;
    double v[FMAXK / 2];   // all loads in flight before the first store
#pragma unroll
    for (int j = 0; j < FMAXK / 2; ++j) {
      const int c = half + 2 * j;
      v[j] = 0.0;
      if (c < W) {
        const FusedCol d = cols[T.gcol + c];
        if (d.ptr) v[j] = __ldg(d.ptr + (int64_t)P * d.sP + (int64_t)Q * d.sQ);
      }
    }
#pragma unroll
    for (int j = 0; j < FMAXK / 2; ++j) {
      const int c = half + 2 * j;
      if (c < W) sA[t * kp + c] = v[j];
    }
  }
  __syncthreads();
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
      const int q = t / tp, p = t - q * tp;
      const int P = T.p0 + p, Q = T.q0 + q;
      const double* crow = sC + (p * tq + q) * np;
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
      const int p = r / tq, q = r - p * tq;
      const int64_t row = (int64_t)T.row0 + (int64_t)(T.p0 + p) * T.EQ + T.q0 + q;
      C[row * g.ldc + n] = sC[r * np + n];
    }
  }
}

// The same step for many tiles, one warp per tile.  A row belongs to one lane (R rows to a
// lane at once): it gathers the row's A elements into columns of the warp's shared memory
// that only it reads (the list of nonzeros picks elements by number), forms the outputs and
// stores them at once.  Lanes walk q, then p, of tiles at most 8 wide along q when
// the band allows it, so that 32-byte sectors are read whole along q and written whole
// along p without a transposing stage, and no barrier.
//
// Bound by instruction issue and the latency of its loads (48 Hubbard sites: about 1000
// warp instructions a tile, 40% of the issue slots, FP64 pipe 30%).  A CTA per tile spent
// its time on the chain of loads before the product (tile, group and descriptors, B and
// A), six tiles to an SM; here an SM holds 28 or more.  Two rows per lane share the
// lists' and descriptors' reads where tiles are full (four took 156 us at 4096, one
// 168); bands of a few rows take one.  One apply (ncu, cold), with a CTA per tile ->
// now: Heisenberg at bond dimension 2048 75 -> 42 us, 4096 244 -> 136 (60 and 182 with
// runs of tiles to a CTA), environment step at 2048 50 -> 21; the two MPO steps of one
// Hubbard site at 601 41 -> 25; 48 Hubbard sites 178 us for the instances with 32 rows per
// tile and more and 135 for the relayouts and skinny products of the others -> 165 for
// all.
constexpr int FW = 4;   // warps per CTA, each on its own tile

__host__ __device__ constexpr size_t warp_smem(int kp, int np, int R) {
  return ((size_t)kp * 32 * R * 8 + (size_t)np * kp * 9 + (size_t)(kp + np) * sizeof(FusedCol) + (size_t)np * 8 + 15) / 16 *
         16;
}

template <int R>
__global__ void __launch_bounds__(32 * FW, 8) fused_warp_kernel(const GemmGroup* __restrict__ groups,
                                                                const FusedTile* __restrict__ tiles, int ntiles,
                                                                const FusedCol* __restrict__ cols, int kp, int np,
                                                                double* const* __restrict__ slots) {
  tnx_grid_dependency();
  extern __shared__ __align__(16) unsigned char dyn[];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int ti = blockIdx.x * FW + wid;
  if (ti >= ntiles) return;
  unsigned char* base = dyn + (size_t)wid * warp_smem(kp, np, R);
  FusedCol* s_d = (FusedCol*)base;                        // [kp] of A, [np] of the output
  double* s_a = (double*)(s_d + kp + np) + lane;          // [kp][R][32]: this lane's columns
  double* s_v = (double*)(s_d + kp + np) + kp * 32 * R;     // [np][kp] nonzeros
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
  for (int r = lane; r < rows; r += 32 * R) {
    int64_t P[R], Q[R];
#pragma unroll
    for (int i = 0; i < R; ++i) {
      const int x = min(r + 32 * i, rows - 1), p = small_div(x, mq);
      P[i] = T.p0 + p;
      Q[i] = T.q0 + x - p * T.eQ;
    }
    for (int c0 = 0; c0 < W; c0 += 4) {
      double v[4][R];
#pragma unroll
      for (int c = 0; c < 4; ++c) {
#pragma unroll
        for (int i = 0; i < R; ++i) v[c][i] = 0.0;
        if (c0 + c < W) {
          const FusedCol d = s_d[c0 + c];
          if (d.ptr) {
#pragma unroll
            for (int i = 0; i < R; ++i) v[c][i] = __ldg(d.ptr + P[i] * d.sP + Q[i] * d.sQ);
          }
        }
      }
#pragma unroll
      for (int c = 0; c < 4; ++c)
        if (c0 + c < W) {
#pragma unroll
          for (int i = 0; i < R; ++i) s_a[((c0 + c) * R + i) * 32] = v[c][i];
        }
    }
    for (int n = 0; n < N; ++n) {
      double acc[R];
#pragma unroll
      for (int i = 0; i < R; ++i) acc[i] = 0.0;
      const int c = s_cnt[n];
      const double* bv = s_v + n * kp;
      const unsigned char* bk = s_k + n * kp;
      if (c > 0) {
        const double* a = s_a + bk[0] * (32 * R);
        const double x = bv[0];
        const uint32_t code = s_p2[n];
#pragma unroll
        for (int i = 0; i < R; ++i) acc[i] = tnx_first_term(a[i * 32], x, code);
      }
      for (int e = 1; e < c; ++e) {
        const double* a = s_a + bk[e] * (32 * R);
        const double x = bv[e];
#pragma unroll
        for (int i = 0; i < R; ++i) acc[i] = fma(a[i * 32], x, acc[i]);
      }
      if (C) {
#pragma unroll
        for (int i = 0; i < R; ++i)
          if (r + 32 * i < rows) C[((int64_t)T.row0 + P[i] * T.EQ + Q[i]) * g.ldc + n] = acc[i];
      } else {
        const FusedCol d = s_d[kp + n];
        if (d.ptr) {
#pragma unroll
          for (int i = 0; i < R; ++i)
            if (r + 32 * i < rows) d.ptr[P[i] * d.sP + Q[i] * d.sQ] = acc[i];
        }
      }
    }
  }
}

}  // namespace

size_t tnx_fused_smem_bytes(int kp, int np) { return sizeof(FusedSmem) + (size_t)FR * (kp + np) * sizeof(double); }

namespace {
cudaError_t launch_fused(const GemmGroup* groups, const FusedTile* tiles, int ntiles, const FusedCol* cols, int kp,
                         int np, double* const* slots, cudaStream_t st) {
  static int attr_dev = -1;   // the opt-in is per device
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (attr_dev != dev) {
    e = cudaFuncSetAttribute(fused_skinny_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)tnx_fused_smem_bytes(FMAXK + 1, FMAXN + 1));
    if (e != cudaSuccess) return e;
    attr_dev = dev;
  }
  return tnx_launch(fused_skinny_kernel, dim3(ntiles), dim3(FT), tnx_fused_smem_bytes(kp, np), st, groups, tiles, cols,
                    kp, np, slots);
}

template <int R>
cudaError_t launch_fused_warp(const GemmGroup* groups, const FusedTile* tiles, int ntiles, const FusedCol* cols, int kp,
                              int np, double* const* slots, cudaStream_t st) {
  static int attr_dev = -1;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (attr_dev != dev) {
    e = cudaFuncSetAttribute(fused_warp_kernel<R>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)(FW * warp_smem(FMAXK + 1, FMAXN + 1, R)));
    if (e != cudaSuccess) return e;
    attr_dev = dev;
  }
  return tnx_launch(fused_warp_kernel<R>, dim3((ntiles + FW - 1) / FW), dim3(32 * FW), FW * warp_smem(kp, np, R), st,
                    groups, tiles, ntiles, cols, kp, np, slots);
}
}  // namespace

cudaError_t tnx_launch_fused_skinny(const GemmGroup* groups, const FusedTile* tiles, int ntiles, int lane_rows,
                                    const FusedCol* cols, int kp, int np, double* const* slots, cudaStream_t st) {
  if (ntiles <= 0) return cudaSuccess;
  if (kp < 1 || kp > FMAXK + 1 || np < 1 || np > FMAXN + 1) return cudaErrorInvalidValue;
  const cudaError_t le = lane_rows == 0   ? launch_fused(groups, tiles, ntiles, cols, kp, np, slots, st)
                         : lane_rows == 1 ? launch_fused_warp<1>(groups, tiles, ntiles, cols, kp, np, slots, st)
                                          : launch_fused_warp<2>(groups, tiles, ntiles, cols, kp, np, slots, st);
  if (le != cudaSuccess) return le;
  tnx_note_launch(1);
  return cudaGetLastError();
}
