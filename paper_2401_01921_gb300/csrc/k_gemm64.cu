// Grouped dense products for the fused charge sectors, native FP64.
//
// Sec. 7 / Sec. 10 of arXiv 2401.01921: after matching, each charge sector of
// a pairwise contraction is one dense matrix product (the paper hands these to
// BLAS / cuBLAS).  Here one launch covers every tile of every group:
// C_g[M,N] = A_g[M,K] * B_g[N,K]^T, operands K-major, C row-major.
//
// T x T output tile per CTA, K staged through shared memory in slices of BK, the
// next slice's entries read while the current one is multiplied.  What bounds it
// is FP64 issue (a warp instruction holds its SM quarter's unit for 64 cycles, so
// two multiply-adds per clock per SM), not memory, whatever the tile: even an 8 x 8
// tile reads only 16 entries per 64 multiply-adds.  Small tiles spread a product over
// the SMs and waste little on ragged edges, so FP64 runs on 8 x 8 (one column and row
// per thread) or 16 x 16 tiles (tnx_f64_edge, tnx_network.cpp, with the times of
// all sizes tried).  A product's terms are added in the order of k in every variant.
// 20-step FP64 Lanczos solve at bond dimension 150 (two products per step, K up to
// 150): 6.4 ms on 64 x 64 tiles, a handful of SMs busy; 1.24 ms now.
// The FP32 variant (operands rounded to FP32, FP32 FMAs, result widened) is
// the "single FP32" point of the precision sweep, always on 64 x 64 tiles.
#include "tnx_internal.h"

namespace {

// TX x TY threads, thread (tx, ty) takes rows ty + TY i, columns tx + TX j.
template <typename TC, int T, int TX, int TY, int BK>
__global__ void __launch_bounds__(TX* TY) gemm_kernel(const GemmGroup* __restrict__ groups,
                                                      const GemmTile* __restrict__ tiles,
                                                      double* const* __restrict__ slots) {
  tnx_grid_dependency();
  constexpr int NT = TX * TY, RI = T / TY, RJ = T / TX, LD = T * BK / NT;   // loads per thread, operand and slice
  __shared__ TC As[BK][T + 1];
  __shared__ TC Bs[BK][T + 1];
  const GemmTile tl = tiles[blockIdx.x];
  const GemmGroup g = groups[tl.group];
  const double* A = slots[g.a_slot] + g.a_off;
  const double* B = slots[g.b_slot] + g.b_off;
  double* C = slots[g.c_slot] + g.c_off;
  const int tx = threadIdx.x % TX, ty = threadIdx.x / TX;
  TC acc[RI][RJ];
#pragma unroll
  for (int i = 0; i < RI; ++i)
#pragma unroll
    for (int j = 0; j < RJ; ++j) acc[i][j] = 0;
  double ra[LD], rb[LD];
  auto fetch = [&](int k0) {   // T x BK of A and of B, k fastest
#pragma unroll
    for (int r = 0; r < LD; ++r) {
      const int idx = threadIdx.x + r * NT;
      const int row = idx / BK, gk = k0 + idx % BK;
      const int gm = tl.m0 + row, gn = tl.n0 + row;
      ra[r] = (gm < g.M && gk < g.K) ? A[(int64_t)gm * g.lda + gk] : 0.0;
      rb[r] = (gn < g.N && gk < g.K) ? B[(int64_t)gn * g.ldb + gk] : 0.0;
    }
  };
  fetch(0);
  for (int k0 = 0; k0 < g.K; k0 += BK) {
#pragma unroll
    for (int r = 0; r < LD; ++r) {
      const int idx = threadIdx.x + r * NT;
      As[idx % BK][idx / BK] = (TC)ra[r];
      Bs[idx % BK][idx / BK] = (TC)rb[r];
    }
    __syncthreads();
    if (k0 + BK < g.K) fetch(k0 + BK);
    const int kn = min(BK, g.K - k0);   // no multiply-adds for the padding of K
#pragma unroll 4
    for (int kk = 0; kk < kn; ++kk) {
      TC a[RI], b[RJ];
#pragma unroll
      for (int i = 0; i < RI; ++i) a[i] = As[kk][ty + TY * i];
#pragma unroll
      for (int j = 0; j < RJ; ++j) b[j] = Bs[kk][tx + TX * j];
#pragma unroll
      for (int i = 0; i < RI; ++i)
#pragma unroll
        for (int j = 0; j < RJ; ++j) acc[i][j] = fma(a[i], b[j], acc[i][j]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < RI; ++i) {
    const int gm = tl.m0 + ty + TY * i;
    if (gm >= g.M) continue;
#pragma unroll
    for (int j = 0; j < RJ; ++j) {
      const int gn = tl.n0 + tx + TX * j;
      if (gn < g.N) C[(int64_t)gm * g.ldc + gn] = (double)acc[i][j];
    }
  }
}

// Skinny products (K <= 16): a tile is up to 128 rows by `width` columns (the
// tile's pad0, 8 to 64); the 128 threads take one row each, or, for tiles of fewer
// rows, 2, 4, ... threads share a row and take every 2nd, 4th, ... column, so that
// all four SM quarters work.  The MPO-like operand B of these steps is small and
// mostly zeros (the two-site MPO product of the Heisenberg H_eff stores 30 nonzeros
// in 114 entries), and FP64 FMAs are the scarce resource of this part: each CTA
// first lists the nonzeros of every output column of its tile in shared memory (one
// thread per column, in k order), then every thread walks those lists against its
// row of A (staged in shared memory).  Skipping a zero term leaves an FMA chain
// unchanged, so the result equals the dense product bit for bit.  A dense B (the
// sectors with K <= 16 of an ordinary product) costs K FMA instructions per column
// and warp, 64 cycles each: 34 us for 64 columns, which narrower tiles spread over
// the SMs when there are few (tnx_skinny_tiles, tnx_network.cpp).
constexpr int SK_MAXK = 16;

__global__ void __launch_bounds__(128) gemm_skinny_kernel(const GemmGroup* __restrict__ groups,
                                                          const GemmTile* __restrict__ tiles,
                                                          double* const* __restrict__ slots) {
  tnx_grid_dependency();
  __shared__ double s_v[64][SK_MAXK];          // nonzero B entries of each output column
  __shared__ unsigned char s_k[64][SK_MAXK];   // their k
  __shared__ int s_cnt[64];
  __shared__ uint32_t s_p2[64];                // tnx_pow2_code of the first nonzero
  __shared__ double s_a[128][SK_MAXK + 1];     // the CTA's rows of A (padded: conflict-free)
  const GemmTile tl = tiles[blockIdx.x];
  const GemmGroup g = groups[tl.group];
  const double* A = slots[g.a_slot] + g.a_off;
  const double* B = slots[g.b_slot] + g.b_off;
  double* C = slots[g.c_slot] + g.c_off;
  const int nn = min(tl.pad0, g.N - tl.n0);
  const int K = g.K;
  if ((int)threadIdx.x < nn) {
    const double* brow = B + (int64_t)(tl.n0 + threadIdx.x) * g.ldb;
    int c = 0;
    for (int k = 0; k < K; ++k) {
      const double v = brow[k];
      if (v != 0.0) {
        s_v[threadIdx.x][c] = v;
        s_k[threadIdx.x][c] = (unsigned char)k;
        ++c;
      }
    }
    s_cnt[threadIdx.x] = c;
    s_p2[threadIdx.x] = c ? tnx_pow2_code(s_v[threadIdx.x][0]) : 0u;
  }
  // threads per row: the rows rounded up to a power of two fill the CTA
  const int rows = min(128, g.M - tl.m0);
  const int rp = rows > 1 ? 1 << (32 - __clz(rows - 1)) : 1;
  const int r = threadIdx.x & (rp - 1), sub = threadIdx.x / rp, step = 128 / rp;
  const int m = tl.m0 + r;
  if (sub == 0 && r < rows) {
    double a[SK_MAXK];
#pragma unroll
    for (int k = 0; k < SK_MAXK; ++k)
      if (k < K) a[k] = A[(int64_t)m * g.lda + k];
#pragma unroll
    for (int k = 0; k < SK_MAXK; ++k)
      if (k < K) s_a[r][k] = a[k];
  }
  __syncthreads();
  if (r >= rows) return;
  const double* arow = s_a[r];
  double* crow = C + (int64_t)m * g.ldc + tl.n0;
  for (int n = sub; n < nn; n += step) {
    double acc = 0.0;
    const int c = s_cnt[n];
    if (c > 0) acc = tnx_first_term(arow[s_k[n][0]], s_v[n][0], s_p2[n]);
    for (int e = 1; e < c; ++e) acc = fma(arow[s_k[n][e]], s_v[n][e], acc);
    crow[n] = acc;
  }
}

template <int T, int TX, int TY, int BK>
cudaError_t launch_f64(const GemmGroup* groups, const GemmTile* tiles, int ntiles, double* const* slots,
                       cudaStream_t st) {
  return tnx_launch(gemm_kernel<double, T, TX, TY, BK>, dim3(ntiles), dim3(TX * TY), 0, st, groups, tiles, slots);
}

}  // namespace

cudaError_t tnx_launch_gemm_skinny(const GemmGroup* groups, const GemmTile* tiles, int ntiles, double* const* slots,
                                   cudaStream_t st) {
  if (ntiles <= 0) return cudaSuccess;
  {
    const cudaError_t le = tnx_launch(gemm_skinny_kernel, dim3(ntiles), dim3(128), 0, st, groups, tiles, slots);
    if (le != cudaSuccess) return le;
  }
  tnx_note_launch(1);
  return cudaGetLastError();
}

cudaError_t tnx_launch_gemm_f64(const GemmGroup* groups, const GemmTile* tiles, int ntiles, int edge,
                                double* const* slots, cudaStream_t st) {
  if (ntiles <= 0) return cudaSuccess;
  cudaError_t le = cudaErrorInvalidValue;
  if (edge == 16) le = launch_f64<16, 16, 8, 32>(groups, tiles, ntiles, slots, st);
  else if (edge == 8) le = launch_f64<8, 8, 8, 32>(groups, tiles, ntiles, slots, st);
  if (le != cudaSuccess) return le;
  tnx_note_launch(1);
  return cudaGetLastError();
}

cudaError_t tnx_launch_gemm_f32(const GemmGroup* groups, const GemmTile* tiles, int ntiles,
                                double* const* slots, cudaStream_t st) {
  if (ntiles <= 0) return cudaSuccess;
  {
    const cudaError_t le =
        tnx_launch(gemm_kernel<float, 64, 16, 16, 16>, dim3(ntiles), dim3(256), 0, st, groups, tiles, slots);
    if (le != cudaSuccess) return le;
  }
  tnx_note_launch(1);
  return cudaGetLastError();
}
