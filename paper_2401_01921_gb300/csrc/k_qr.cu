// Column-pivoted Householder QR with the columns held in shared memory.
//
// The QR that preconditions the Jacobi sweeps (k_svd.cu) takes c dependent steps per
// charge block.  qr_coop_kernel reads and writes every column in L2 at every step,
// behind a grid barrier of all blocks: 7 us per step at c = 83, 18 us at c = 294.  Here a
// slot (one CTA, 8 warps) keeps up to 8 columns of one block for the whole
// factorisation, one per warp, and blocks do not wait for one another.  Step k:
//  1. every slot publishes its best remaining column (largest trailing norm, lowest
//     index on ties) with its reflector's scalars, and counts itself in;
//  2. behind the count of all slots of the block, each reads the offers, picks the
//     winner, and reads its column;
//  3. each warp applies the reflector to its column, which leaves the trailing norm
//     of the next step with it (summed from the updated entries); the winner's owner
//     stores its column: R above the diagonal, beta on it, the reflector below.
// The reflector is kept unscaled: u = x - beta e_0 with beta = -sign(x_0) |x|, H = I -
// kappa u u^T, kappa = 2 / u^T u = 1 / (|x|^2 + |x_0| |x|) (0 when x is zero below its
// first entry): two FP64 roots and divisions fewer on the path of a step than v = u / u_0 and
// its tau.  The sums over a warp run on the integer units (tnx_fp64.cuh).
// Offers alternate between two buffers: a slot overwrites step k's offer at step k + 2,
// behind the count of step k + 1, which every slot joins after reading step k's.
// All CTAs must be resident (a cooperative launch); waits are bounded as in k_jacobi.cu.
// Measured (ncu): bond dimension 200 (blocks of up to 83 columns) 0.58 -> 0.35 ms, 1024
// (up to 294) 5.5 -> 1.7 ms.
#include "tnx_fp64.cuh"
#include "tnx_internal.h"

namespace {

using namespace tnx_fp64;

constexpr int QW = 8;                                // columns (warps) per slot
constexpr long long QR_WAIT_LIMIT = 2000000000LL;    // clock cycles

struct QrShared {
  double nrm[QW], below[QW], x0[QW];   // trailing norm^2, its part below the first entry, the first entry
  int idx[QW];                         // column in the block; -1: none, or a pivot already
  QrOffer mine, won;
  int win;
};

__global__ void __launch_bounds__(32 * QW) qr_block_kernel(const SvdQr* __restrict__ qs,
                                                           const QbGroup* __restrict__ groups,
                                                           const int2* __restrict__ slots, int* status) {
  extern __shared__ __align__(16) unsigned char qr_dyn[];
  QrShared& S = *(QrShared*)qr_dyn;
  const int2 sl = slots[blockIdx.x];
  const SvdQr q = qs[sl.x];
  const QbGroup g = groups[sl.x];
  const int rp = (q.r + 31) & ~31;
  double* pv = (double*)(qr_dyn + (sizeof(QrShared) + 15) / 16 * 16);   // the pivot's reflector
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  double* a = pv + (int64_t)(1 + wid) * rp;                             // this warp's column
  const int col = sl.y * QW + wid;
  if (lane == 0) S.idx[wid] = col < q.c ? col : -1;
  if (col < q.c) {
    double s = 0.0;
    const double* x = q.X + (int64_t)col * q.r;
    for (int i = lane; i < rp; i += 32) {
      const double v = i < q.r ? x[i] : 0.0;
      a[i] = v;
      if (i > 0) s = fma(v, v, s);
    }
    s = warp_sum_double(s);
    __syncwarp();
    if (lane == 0) {
      S.below[wid] = s;
      S.x0[wid] = a[0];
      S.nrm[wid] = fma(a[0], a[0], s);
    }
  }
  for (int i = threadIdx.x; i < rp; i += 32 * QW) pv[i] = 0.0;
  __syncthreads();
  for (int k = 0; k < q.c; ++k) {
    // ---- this slot's offer: warp 0 its scalars, the others the column
    int best = -1;
    unsigned long long key = 0;
    for (int w = 0; w < QW; ++w) {
      const unsigned long long n = (unsigned long long)__double_as_longlong(S.nrm[w]);   // >= 0 (or NaN): ordered as bits
      if (S.idx[w] >= 0 && (best < 0 || n > key)) {
        best = w;
        key = n;
      }
    }
    QrOffer* offers = g.offers + (int64_t)(k & 1) * g.ns;
    double* column = g.columns + (int64_t)(k & 1) * g.ns * rp;
    if (wid == 0) {
      if (best >= 0) {
        const double m = S.nrm[best], x0 = S.x0[best];
        const double n = sqrt(m);
        if (lane == 0) {
          S.mine.nrm = m;
          S.mine.idx = S.idx[best];
          const bool flat = S.below[best] == 0.0;
          S.mine.beta = flat ? x0 : (x0 >= 0.0 ? -n : n);
          S.mine.u0 = flat ? 1.0 : x0 + (x0 >= 0.0 ? n : -n);
          const double d = fma(fabs(x0), n, m);   // at most 2 m
          double kappa = 1.0 / d;
          // half of it where d overflows; a norm that does leaves nothing finite behind it
          // (0 would leave the column as it is)
          if (!is_finite(d))
            kappa = is_finite(m) ? 0.5 / fma(0.5 * fabs(x0), n, 0.5 * m) : __longlong_as_double(0x7FF8000000000000ll);
          S.mine.kappa = flat ? 0.0 : kappa;
        }
      } else if (lane == 0) {
        S.mine.idx = -1;
      }
    } else if (best >= 0) {
      const double* src = pv + (int64_t)(1 + best) * rp;
      double* dst = column + (int64_t)sl.y * rp;
      for (int i = (k & ~31) + threadIdx.x - 32; i < q.r; i += 32 * (QW - 1)) __stcg(dst + i, src[i]);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      offers[sl.y] = S.mine;
      __threadfence();
      asm volatile("red.relaxed.gpu.global.add.u32 [%0], 1;" ::"l"(g.count) : "memory");
    }
    // ---- all offers of the block
    int ok = 1;
    if (threadIdx.x == 0) {
      const unsigned target = (unsigned)(k + 1) * (unsigned)g.ns;
      const long long t0 = clock64();
      for (unsigned it = 1;; ++it) {
        unsigned cur;
        asm volatile("ld.acquire.gpu.u32 %0, [%1];" : "=r"(cur) : "l"(g.count) : "memory");
        if (cur >= target) break;
        if ((it & 31u) != 0) continue;   // the error word and the clock every 32 polls
        if (*(volatile int*)status != 0) {
          ok = 0;
          break;
        }
        if (clock64() - t0 > QR_WAIT_LIMIT) {
          atomicExch(status, 1);
          ok = 0;
          break;
        }
      }
    }
    if (!__syncthreads_and(ok)) return;
    if (wid == 0) {
      // the largest norm, the lowest column on ties
      unsigned long long bk = 0;
      int bi = 0x7FFFFFFF, bs = -1;
      for (int s = lane; s < g.ns; s += 32) {
        const int idx = __ldcg(&offers[s].idx);
        const unsigned long long n = (unsigned long long)__double_as_longlong(__ldcg(&offers[s].nrm));
        if (idx >= 0 && (bs < 0 || n > bk || (n == bk && idx < bi))) {
          bk = n;
          bi = idx;
          bs = s;
        }
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long ok2 = __shfl_xor_sync(0xffffffffu, bk, o);
        const int oi = __shfl_xor_sync(0xffffffffu, bi, o), os = __shfl_xor_sync(0xffffffffu, bs, o);
        if (os >= 0 && (bs < 0 || ok2 > bk || (ok2 == bk && oi < bi))) {
          bk = ok2;
          bi = oi;
          bs = os;
        }
      }
      if (lane == 0) {
        S.win = bs;
        S.won.idx = bi;
        S.won.beta = __ldcg(&offers[bs].beta);
        S.won.u0 = __ldcg(&offers[bs].u0);
        S.won.kappa = __ldcg(&offers[bs].kappa);
      }
    }
    __syncthreads();
    const int win = S.win, pidx = S.won.idx;
    const double kappa = S.won.kappa, u0 = S.won.u0;
    {
      const double* src = column + (int64_t)win * rp;
      for (int i = (k & ~31) + threadIdx.x; i < q.r; i += 32 * QW) pv[i] = i < k ? 0.0 : (i == k ? u0 : __ldcg(src + i));
    }
    __syncthreads();
    // ---- the reflector on this warp's column
    const int mine = S.idx[wid];
    if (mine >= 0 && mine != pidx) {
      double w = 0.0;
      if (kappa != 0.0) {
#pragma unroll 4
        for (int i = (k & ~31) + lane; i < rp; i += 32) w = fma(pv[i], a[i], w);
        w = kappa * warp_sum_double(w);
      }
      double s = 0.0;
#pragma unroll 4
      for (int i = (k & ~31) + lane; i < rp; i += 32) {
        const double v = kappa != 0.0 ? fma(-w, pv[i], a[i]) : a[i];
        a[i] = v;
        if (i > k + 1) s = fma(v, v, s);
      }
      s = warp_sum_double(s);
      __syncwarp();
      if (lane == 0) {
        const double x0 = k + 1 < q.r ? a[k + 1] : 0.0;
        S.below[wid] = s;
        S.x0[wid] = x0;
        S.nrm[wid] = fma(x0, x0, s);
      }
    } else if (mine >= 0) {
      // the pivot's owner: R's column, the reflector below
      double* x = q.X + (int64_t)mine * q.r;
      for (int i = lane; i < q.r; i += 32) x[i] = i < k ? a[i] : (i == k ? S.won.beta : pv[i]);
      __syncwarp();
      if (lane == 0) {
        q.perm[k] = mine;
        q.tau[k] = kappa;
        q.u0[k] = u0;
        S.idx[wid] = -1;
      }
    }
    __syncthreads();
  }
}

size_t qr_bytes(int r) {
  return (sizeof(QrShared) + 15) / 16 * 16 + (size_t)(1 + QW) * (((size_t)r + 31) / 32 * 32) * sizeof(double);
}
constexpr size_t kQrSmemMax = 226 * 1024;

}  // namespace

int tnx_qr_block_columns(int maxr) { return qr_bytes(maxr) <= kQrSmemMax ? QW : 0; }

cudaError_t tnx_launch_qr_block(const SvdQr* qs, const QbGroup* groups, const int2* slots, int nslots, int maxr,
                                int* status, cudaStream_t st) {
  if (nslots <= 0) return cudaSuccess;
  const size_t smem = qr_bytes(maxr);
  int dev = 0, nsm = 0, per_sm = 0, coop = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(qr_block_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kQrSmemMax);
  if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, qr_block_kernel, 32 * QW, smem);
  if (e != cudaSuccess) return e;
  if (!coop || (int64_t)per_sm * nsm < nslots) return cudaErrorNotSupported;
  void* args[] = {(void*)&qs, (void*)&groups, (void*)&slots, (void*)&status};
  e = cudaLaunchCooperativeKernel((const void*)qr_block_kernel, dim3(nslots), dim3(32 * QW), args, smem, st);
  if (e != cudaSuccess) return e;
  tnx_note_launch(1);
  return cudaSuccess;
}
