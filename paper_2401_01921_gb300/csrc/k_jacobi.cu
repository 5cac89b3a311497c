// One-sided Jacobi sweeps on column blocks held in shared memory.
//
// The QR-preconditioned SVD (k_svd.cu) orthogonalises the c rows of R of every
// charge block by plane rotations, accumulated in J.  What bounds it on this
// part is FP64 issue: a warp instruction occupies its SM quarter's FP64 unit for
// 64 cycles, whether 32 lanes or one are active, independent or not (measured;
// a root is 10 such instructions, a division 9).  One rotation per trip through
// L2 and grid barrier, with the angle formed by every lane (jacobi_coop_kernel),
// costs about 6 us per round at c = 83 and 20 us at c = 294.  Here the vectors
// of a block are cut into nb blocks of at most w (4 or 8); a slot (one CTA: 8
// warps that move and rotate vectors, four that form angles) loads two of them
// with their rows of J, visits all pairs between them without leaving the SM,
// and writes them back:
//  * a sweep is nb - 1 rounds of nb / 2 disjoint slots (the round-robin order of
//    jacobi_round_kernel, over column blocks); the first round also visits the
//    pairs inside each block, so a sweep visits every pair once.  A round has w
//    steps of w disjoint pairs, one pair per warp, so the trips through L2 are
//    w times fewer;
//  * a slot waits for the two blocks it needs only (a version word per block),
//    and each charge block stops on its own;
//  * a rotation is applied in the scaled form of Gentleman's fast Givens
//    rotations: x_p <- x_p - a x_q, x_q <- x_q + b x_p with the cosines kept as a
//    factor per vector (D, folded into the vectors once a sweep): 2 FMAs per
//    entry pair instead of 2 products and 2 FMAs;
//  * the squared norms are carried from pair to pair, and summed again once a
//    sweep or when a rotation cancels most of one: a pair then costs one dot
//    product instead of three.  Its per-lane partial sums are added up as 64-bit
//    integers in units of 2^-54 of the largest (three 32-bit warp reductions), the
//    angle's tangent is formed in FP32 on mantissas with the exponents apart,
//    and thresholds compare such floats: none of that touches the FP64 units;
//  * what needs FP64 per pair (the cosine, factors, norms) is spread over four
//    warps on the four SM quarters, one lane per pair, and runs beside the other
//    warps' rotations and next dot products.
// Measured (the sweeps alone, wavefunctions of the U(1) Heisenberg chain with
// spectra over 12 decades): bond dimension 200 (blocks of up to 83 vectors) 4.6 ->
// 1.6 ms, 1024 (up to 294) 49 -> 13.5 ms.  At 294 the rotations' FP64 issue on the SMs
// that hold the largest blocks bounds a step, at 83 the chain dot, angle, rotation.
//
// The rotations, thresholds and stopping rule are those of k_svd.cu: a pair with
// g^2 <= 1e-30 |x_p|^2 |x_q|^2 is left alone (so is one with a norm that is zero,
// subnormal or not finite); a block stops after a sweep in which no pair
// exceeded tol^2.
//
// Waits: a slot's round needs slots of its block's previous round only, and every
// CTA runs its slots round by round, so with all CTAs resident (a cooperative
// launch) each wait ends; all are bounded (about a second of clock) all the
// same, and on expiry *status is set, every CTA leaves, and the kernels behind touch
// nothing.
#include "tnx_fp64.cuh"
#include "tnx_internal.h"

namespace {

using namespace tnx_fp64;

constexpr long long JB_WAIT_LIMIT = 2000000000LL;   // clock cycles
constexpr int W = 8;                                // warps that rotate: vectors per column block at most
constexpr int NH = 4;                               // angle warps
constexpr int JB_THREADS = 32 * (W + NH);

__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}

// Waits until *w0 >= target and *w1 >= target (one thread each); false on expiry
// or when another CTA gave up.
__device__ bool wait_words(const unsigned* w0, const unsigned* w1, unsigned target, int* status) {
  int ok = 1;
  if (threadIdx.x < 2) {
    const unsigned* w = threadIdx.x ? w1 : w0;
    const long long t0 = clock64();
    for (unsigned it = 1;; ++it) {
      unsigned cur;
      asm volatile("ld.acquire.gpu.u32 %0, [%1];" : "=r"(cur) : "l"(w) : "memory");
      if (cur >= target) break;
      if ((it & 31u) != 0) continue;   // the error word and the clock every 32 polls
      if (*(volatile int*)status != 0) {
        ok = 0;
        break;
      }
      if (clock64() - t0 > JB_WAIT_LIMIT) {
        atomicExch(status, 1);
        ok = 0;
        break;
      }
    }
  }
  return __syncthreads_and(ok) != 0;
}

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Named barriers: dot products done (rotating warps arrive, angle warps wait),
// coefficients ready (angle warps 0 and 1 arrive, rotating warps wait), rotating warps
// among themselves, angle warps among themselves.
enum { BAR_DOT = 1, BAR_COEF = 2, BAR_ROT = 3, BAR_ANGLE = 4 };
__device__ __forceinline__ void bar_sync(int id, int n) {
  __syncwarp();
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory");
}
__device__ __forceinline__ void bar_arrive(int id, int n) {
  __syncwarp();
  asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(n) : "memory");
}

__device__ __forceinline__ bool usable(double n) {   // positive, normal and finite
  const int hi = __double2hiint(n);
  return hi >= 0x00100000 && hi < 0x7FF00000;
}

// A number s m 2^e with m in [1, 4): a pair's dot product to about 22 bits, from
// the integer sum in units of 2^-k and the product of the two factors.
struct Rough {
  float m;
  int e;
  int s;      // sign bit (bit 31)
  bool zero;
};
__device__ __forceinline__ Rough rough_dot(long long v, int k, double dd) {
  Rough r;
  const unsigned long long u = (unsigned long long)(v < 0 ? -v : v);
  r.zero = u == 0;
  const int lz = r.zero ? 63 : __clzll((long long)u);
  r.s = (int)(v >> 32) & 0x80000000;
  const unsigned top = (unsigned)((u << lz) >> 40) & 0x7FFFFFu;   // 23 bits below the leading one
  r.m = __int_as_float(0x3F800000 | (int)top) * mant(dd);
  r.e = 63 - lz - k + expo(__double2hiint(dd)) - 1023;
  return r;
}

// 2^e as a float, e held to [-126, 120]
__device__ __forceinline__ float pow2f(int e) { return __int_as_float((127 + max(-126, min(e, 120))) << 23); }

// tan of the rotation angle, t = sign(z) / (|z| + sqrt(1 + z^2)) with z = df / (2 g),
// to about 21 bits: FP32 on the mantissas, the exponents carried apart (any range).
// |t| = t * 2^-sh.  A rotation by a slightly different angle is as orthogonal (its
// cosine is formed from this very t): it leaves 1e-6 of the pair's dot product
// instead of its rounding error, which the quadratic convergence hides.
struct Tan {
  float t;
  int sh, s;
};
__device__ __forceinline__ Tan rotation_tan(double df, const Rough& g) {
  const int hd = __double2hiint(df);
  const float md = mant(df);
  const int e = expo(hd) - 1023 - g.e - 1;   // |z| = md / g.m * 2^e
  Tan r;
  r.s = (hd ^ g.s) & 0x80000000;
  if (e > 60) {                              // t = 1 / (2 |z|)
    r.t = 0.5f * __fdividef(g.m, md);
    r.sh = e;
  } else {
    const float z = expo(hd) == 0 || e < -60 ? 0.0f : __fdividef(md, g.m) * pow2f(e);
    r.t = __fdividef(1.0f, z + sqrtf(fmaf(z, z, 1.0f)));
    r.sh = 0;
  }
  return r;
}
__device__ __forceinline__ double widen(const Tan& r) {   // exact; r.t is a normal float
  const int ft = __float_as_int(r.t), ex = ((ft >> 23) & 0xFF) - 127 + 1023 - r.sh;
  if (ex <= 0) return 0.0;
  return __hiloint2double(r.s | (ex << 20) | ((ft & 0x7FFFFF) >> 3), (int)((unsigned)ft << 29));
}

// g^2 / (a b) (0 below 2^-120, capped at 2^60), a and b usable
__device__ __forceinline__ float off_sq(const Rough& g, double a, double b) {
  const int e = 2 * g.e + 2046 - expo(__double2hiint(a)) - expo(__double2hiint(b));
  if (g.zero || e < -120) return 0.0f;
  return __fdividef(g.m * g.m, mant(a) * mant(b)) * pow2f(min(e, 60));
}

// What is left of a norm: (a - t g) / n0 for s = +1 (b: (b + t g) / n0 for s = -1), a and n0 usable.
__device__ __forceinline__ float norm_left(const Tan& t, const Rough& g, double a, double n0, float s) {
  const int e0 = expo(__double2hiint(n0)) - 1023;
  const float r0 = __fdividef(1.0f, mant(n0));
  const float q = mant(a) * r0 * pow2f(expo(__double2hiint(a)) - 1023 - e0);
  const float tg = t.t * g.m * r0 * pow2f(g.e - t.sh - e0);
  return q - ((t.s ^ g.s) < 0 ? -s : s) * tg;
}

// Local vector l < wm lies in the first column block of the slot, l >= wm in the
// second; pair tables are by pair (= rotating warp) of a step.
struct JbShared {
  double nrm[2 * W];           // squared norms
  double n0[2 * W];            // and what they were when last summed
  double d[2 * W], id[2 * W];  // scale factors and their reciprocals
  double fa[W], fb[W], dd[W];  // d_b / d_a, d_a / d_b, d_a d_b of the step's pairs
  double ca[W], cb[W];         // the step's coefficients
  // the step's pairs as its angles saw them: norms, factors, tangent, dot product, cosine
  double pa[W], pb[W], pda[W], pdb[W], pt[W], pg[W], pc[W];
  // the step's dot products, in units of 2^-sc; by step parity: angle warp 2 reads
  // them beside the next step's dot products
  long long dot[2][W];
  int sc[2][W];
  int act[W];                  // 0: leave the pair alone; 1: rotate; 2 / 3: and sum the norm of a / b again
  int any, big;
  unsigned done[TNX_JB_MAXSLOTS / 32];
};

// The pair w in step s: local vectors la, lb (la = -1: none).
__device__ __forceinline__ void step_pair(bool first, int w, int s, int wm, int nA, int nB, int& la, int& lb) {
  la = lb = -1;
  if (w >= wm) return;
  if (!first) {
    const int y = w + s < wm ? w + s : w + s - wm;
    if (w < nA && y < nB) {
      la = w;
      lb = wm + y;
    }
    return;
  }
  const int m = 2 * wm - 1;
  int x = w == 0 ? s : (s + w) % m, y = w == 0 ? m : (s - w + m) % m;
  if (x > y) {
    const int t = x;
    x = y;
    y = t;
  }
  if ((x < wm ? x < nA : x - wm < nB) && (y < wm ? y < nA : y - wm < nB)) {
    la = x;
    lb = y;
  }
}

__global__ void __launch_bounds__(JB_THREADS) jacobi_block_kernel(const JbGroup* __restrict__ groups,
                                                                  const int2* __restrict__ slots, int nslots,
                                                                  int max_sweeps, float tol2, int* __restrict__ met,
                                                                  unsigned* cnt, int* status, int* sweeps_out) {
  extern __shared__ __align__(16) unsigned char jb_dyn[];
  JbShared& S = *(JbShared*)jb_dyn;
  double* buf = (double*)(jb_dyn + (sizeof(JbShared) + 15) / 16 * 16);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  for (int i = threadIdx.x; i < TNX_JB_MAXSLOTS / 32; i += JB_THREADS) S.done[i] = 0;
  if (threadIdx.x == 0) S.big = 0;
  __syncthreads();
  bool ok = *(volatile int*)status == 0, more = true;   // an expired QR leaves nothing to sweep
  for (int it = 0; ok && more; ++it) {
    more = false;
    int mine = 0;
    for (int si = blockIdx.x; ok && si < nslots; si += gridDim.x, ++mine) {
      if (S.done[mine >> 5] >> (mine & 31) & 1u) continue;
      const int2 sl = slots[si];
      const JbGroup g = groups[sl.x];
      const int nr = g.nb - 1, sw = it / nr, k = it - sw * nr;
      const bool first = k == 0;
      if (first && sw > 0) {
        // every slot of the block has finished the sweep
        ok = wait_words(cnt + sl.x, cnt + sl.x, (unsigned)sw * (unsigned)(g.nb / 2), status);
        if (!ok) break;
        const int m = __ldcg(met + (int64_t)sl.x * max_sweeps + sw - 1);
        if (!m || sw == max_sweeps) {   // every slot of the block reads the same word
          if (threadIdx.x == 0) {
            S.done[mine >> 5] |= 1u << (mine & 31);
            if (sl.y == 0) atomicMax(sweeps_out, sw);
          }
          __syncthreads();
          continue;
        }
      }
      more = true;
      // ---- the two column blocks of this slot
      int p, q;
      if (sl.y == 0) {
        p = k;
        q = g.nb - 1;
      } else {
        p = (k + sl.y) % nr;
        q = (k - sl.y + nr) % nr;
      }
      if (p > q) {
        const int t = p;
        p = q;
        q = t;
      }
      const int p0 = (int)((int64_t)p * g.c / g.nb), nA = (int)((int64_t)(p + 1) * g.c / g.nb) - p0;
      const int q0 = (int)((int64_t)q * g.c / g.nb), nB = (int)((int64_t)(q + 1) * g.c / g.nb) - q0;
      const int ldp = (g.c + 31) & ~31, cs = 2 * ldp;   // a vector and its row of J, zero-padded to whole warps
      const int wm = g.wmax;
      // written back by the slots that held them in the previous round
      if (!first) {
        ok = wait_words(g.ver + p, g.ver + q, (unsigned)it, status);
        if (!ok) break;
      }
      if (wid < W) {
        // warp w loads vectors w of both blocks
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          if (wid < (h ? nB : nA)) {
            const int64_t row = (int64_t)((h ? q0 : p0) + wid) * g.ld;
            double* x = buf + (int64_t)(h ? wm + wid : wid) * cs;
            const uint32_t xs = (uint32_t)__cvta_generic_to_shared(x);
            for (int e = 2 * lane; e < g.ld; e += 64) {
              cp_async16(xs + 8 * e, g.X + row + e);
              cp_async16(xs + 8 * (ldp + e), g.J + row + e);
            }
            for (int e = g.ld + lane; e < ldp; e += 32) x[e] = x[ldp + e] = 0.0;
          }
        }
      } else if (wid == W && lane < 2 * wm) {
        const int i = lane < wm ? lane : lane - wm;
        if (i < (lane < wm ? nA : nB)) {
          const double* D = g.D + 4 * ((lane < wm ? p0 : q0) + i);
          S.d[lane] = __ldcg(D);
          S.id[lane] = __ldcg(D + 1);
          S.nrm[lane] = __ldcg(D + 2);
          S.n0[lane] = __ldcg(D + 3);
        }
        if (lane == 0) S.any = 0;
      }
      asm volatile("cp.async.wait_all;" ::: "memory");
      __syncthreads();
      if (wid < W) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int l = h ? wm + wid : wid;
          if (wid < (h ? nB : nA)) {
            double* x = buf + (int64_t)l * cs;
            const double d = S.d[l];
            // once a sweep (and when a factor has become small) the factors go
            // into the vectors; once a sweep the norms are summed
            const bool fold = d != 1.0 && (first || d < 1e-40);
            if (fold)
              for (int e = lane; e < cs; e += 32) x[e] *= d;
            double n = 0.0;
            if (first) {
              for (int e = lane; e < ldp; e += 32) n = fma(x[e], x[e], n);
              n = warp_sum(n);
            }
            __syncwarp();
            if (lane == 0) {
              if (first) S.nrm[l] = S.n0[l] = n;
              if (fold) {
                S.d[l] = S.id[l] = 1.0;
                S.any = 1;
              }
            }
          }
        }
      }
      __syncthreads();
      // ---- w steps of w disjoint pairs (first round of a sweep: all pairs of the two blocks)
      const int steps = first ? 2 * wm - 1 : wm;
      if (wid < W) {
        for (int s = 0; s < steps; ++s) {
          int la, lb;
          step_pair(first, wid, s, wm, nA, nB, la, lb);
          double* xa = buf + (int64_t)(la < 0 ? 0 : la) * cs;
          double* xb = buf + (int64_t)(la < 0 ? 0 : lb) * cs;
          if (la >= 0) {
            double g0 = 0.0, g1 = 0.0;
            int e = lane;
#pragma unroll 4
            for (; e + 32 < ldp; e += 64) {
              g0 = fma(xa[e], xb[e], g0);
              g1 = fma(xa[e + 32], xb[e + 32], g1);
            }
            if (e < ldp) g0 = fma(xa[e], xb[e], g0);
            int k2;
            const long long v = warp_sum_scaled(g0 + g1, k2);
            if (lane == 0) {
              S.dot[s & 1][wid] = v;
              S.sc[s & 1][wid] = k2;
            }
          }
          bar_arrive(BAR_DOT, JB_THREADS);
          bar_sync(BAR_COEF, 32 * (W + 2));
          const int act = la >= 0 ? S.act[wid] : 0;
          if (act) {
            const double ca = S.ca[wid], cb = S.cb[wid];
            // entries and rows of J lie back to back: one pass over both
#pragma unroll 4
            for (int e = lane; e < cs; e += 32) {
              const double u = xa[e], v = xb[e];
              xa[e] = fma(-ca, v, u);
              xb[e] = fma(cb, u, v);
            }
            if (act > 1) {
              const double* x = act == 2 ? xa : xb;
              double n = 0.0;
              for (int i = lane; i < ldp; i += 32) n = fma(x[i], x[i], n);
              n = warp_sum(n);
              if (lane == 0) {
                const double d = act == 2 ? S.pda[wid] : S.pdb[wid], t = S.pt[wid];
                S.nrm[act == 2 ? la : lb] = S.n0[act == 2 ? la : lb] = n * d * d / fma(t, t, 1.0);
              }
            }
          }
          bar_sync(BAR_ROT, 32 * W);
        }
      } else {
        const int h = wid - W;
        int la, lb;
        step_pair(first, lane, 0, wm, nA, nB, la, lb);
        for (int s = 0; s < steps; ++s) {
          // what does not depend on the dot products
          if (la >= 0) {
            if (h == 1) S.fa[lane] = S.d[lb] * S.id[la];
            if (h == 2) S.fb[lane] = S.d[la] * S.id[lb];
            if (h == 3) S.dd[lane] = S.d[la] * S.d[lb];
          }
          bar_sync(BAR_DOT, JB_THREADS);
          if (h <= 1) {
            // both form the angle: warp 0 the coefficients, warp 1 the decisions
            double t = 0.0;
            int act = 0;
            if (la >= 0) {
              const double a = S.nrm[la], b = S.nrm[lb], df = b - a;
              const Rough g = rough_dot(S.dot[s & 1][lane], S.sc[s & 1][lane], S.dd[lane]);
              const Tan r = rotation_tan(df, g);
              if (h == 0) {
                t = widen(r);
                S.ca[lane] = t * S.fa[lane];
                S.cb[lane] = t * S.fb[lane];
                S.pa[lane] = a;
                S.pb[lane] = b;
                S.pda[lane] = S.d[la];
                S.pdb[lane] = S.d[lb];
                S.pt[lane] = t;
              } else if (usable(a) && usable(b)) {
                const float o2 = off_sq(g, a, b);
                if (o2 > tol2) S.big = 1;
                if (o2 > 1e-30f) {
                  // a norm about to fall below 1/64 of its last sum is summed again
                  S.any = 1;
                  act = norm_left(r, g, a, S.n0[la], 1.0f) < 0.015625f
                            ? 2
                            : (norm_left(r, g, b, S.n0[lb], -1.0f) < 0.015625f ? 3 : 1);
                }
              }
            }
            if (h == 1 && lane < W) S.act[lane] = act;
            bar_arrive(BAR_COEF, 32 * (W + 2));
            if (h == 0 && la >= 0) S.pc[lane] = rsqrt(fma(t, t, 1.0));
          }
          bar_sync(BAR_ANGLE, 32 * NH);
          // beside the rotations: the new factors, their reciprocals, the new norms
          int act;
          if (h != 0 && lane < wm && (act = S.act[lane]) != 0) {
            const double c = S.pc[lane], t = S.pt[lane];
            if (h == 1) {
              // one Newton step each: the reciprocals stay within rounding of 1 / d
              const double ic = fma(t, t, 1.0) * c, ia = S.id[la] * ic, ib = S.id[lb] * ic;
              S.id[la] = fma(ia, fma(-(S.pda[lane] * c), ia, 1.0), ia);
              S.id[lb] = fma(ib, fma(-(S.pdb[lane] * c), ib, 1.0), ib);
            } else if (h == 2) {
              const double gm = shift_down((double)S.dot[s & 1][lane] * S.dd[lane], S.sc[s & 1][lane]);
              const double a = S.pa[lane], b = S.pb[lane], cc = c * c, g2 = gm + gm;
              if (act != 2) S.nrm[la] = fma(t, fma(t, b, -g2), a) * cc;
              if (act != 3) S.nrm[lb] = fma(t, fma(t, a, g2), b) * cc;
            } else {
              S.d[la] = S.pda[lane] * c;
              S.d[lb] = S.pdb[lane] * c;
            }
          }
          step_pair(first, lane, s + 1, wm, nA, nB, la, lb);
          bar_sync(BAR_ANGLE, 32 * NH);
        }
      }
      __syncthreads();
      // ---- write back (nothing changed: nothing to write)
      if (wid < W) {
        if (S.any) {
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            if (wid < (h ? nB : nA)) {
              const int64_t row = (int64_t)((h ? q0 : p0) + wid) * g.ld;
              const double* x = buf + (int64_t)(h ? wm + wid : wid) * cs;
              for (int e = 2 * lane; e < g.ld; e += 64) {
                *(double2*)(g.X + row + e) = *(const double2*)(x + e);
                *(double2*)(g.J + row + e) = *(const double2*)(x + ldp + e);
              }
            }
          }
        }
      } else if (wid == W && lane < 2 * wm) {
        const int i = lane < wm ? lane : lane - wm;
        if (i < (lane < wm ? nA : nB)) {
          double* D = g.D + 4 * ((lane < wm ? p0 : q0) + i);
          __stcg(D, S.d[lane]);
          __stcg(D + 1, S.id[lane]);
          __stcg(D + 2, S.nrm[lane]);
          __stcg(D + 3, S.n0[lane]);
        }
      }
      __syncthreads();
      if (threadIdx.x == 0) {
        // The flag is cleared by its reader: nothing orders this read before the other
        // warps' start on the CTA's next slot, whose first barrier orders the clear
        // before the angle warps set the flag again.
        if (S.big) __stcg(met + (int64_t)sl.x * max_sweeps + sw, 1);
        S.big = 0;
        __threadfence();   // one fence for the stores of the whole CTA, then plain flags
        asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" ::"l"(g.ver + p), "r"(it + 1) : "memory");
        asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" ::"l"(g.ver + q), "r"(it + 1) : "memory");
        if (k == nr - 1) asm volatile("red.relaxed.gpu.global.add.u32 [%0], 1;" ::"l"(cnt + sl.x) : "memory");
      }
    }
  }
}

size_t jb_bytes(int c, int w) {   // shared memory of a slot of two blocks of w vectors
  const size_t ldp = ((size_t)c + 31) / 32 * 32;
  return (sizeof(JbShared) + 15) / 16 * 16 + (size_t)2 * w * 2 * ldp * sizeof(double);
}

constexpr size_t kSmemMax = 226 * 1024;   // the 227 KB limit less the static shared memory

}  // namespace

// Vectors per column block: 8, or as many of 4, 2, 1 as fit shared memory (8 up to
// c = 896, 4 up to 1792, 2 up to 3584, 1 up to 7168).  8 against 4 in an SVD of
// Heisenberg wavefunctions: 3.3 against 3.4 ms at bond dimension 200 (blocks of up to 83
// vectors, SMs to spare: 4 spreads the FP64 work over twice the SMs but makes twice the
// trips through L2), 21.7 against 23.3 ms at 1024 (up to 294 vectors; 4 for the largest
// blocks only).  The narrow widths against jacobi_coop_kernel, SVD of one dense c x c
// block, ms: 1700 (4) 496 | 1057, 1900 (2) 1090 | 1366, 2600 (2) 2604 | 5045, 3400 (2)
// 5282 | 10021, 3700 (1) 14000 | 14869.
int tnx_jacobi_block_width(int c) {
  if (c < 2) return 0;
  int w = W;
  while (w > 0 && jb_bytes(c, w) > kSmemMax) w >>= 1;
  return w;
}

bool tnx_jacobi_block_fits(int64_t nslots, int nsm) { return nslots <= (int64_t)TNX_JB_MAXSLOTS * nsm; }

cudaError_t tnx_launch_jacobi_block(const JbGroup* groups, const JbGroup* host_groups, int ngroups, const int2* slots,
                                    int nslots, int max_sweeps, double tol, int* met, unsigned* cnt, int* status,
                                    int* sweeps_out, cudaStream_t st) {
  if (nslots <= 0) return cudaSuccess;
  size_t smem = 0;
  for (int i = 0; i < ngroups; ++i)
    if (host_groups[i].nb > 0) {
      if (host_groups[i].wmax > W) return cudaErrorInvalidValue;
      const size_t b = jb_bytes(host_groups[i].c, host_groups[i].wmax);
      if (b > smem) smem = b;
    }
  int dev = 0, nsm = 0, per_sm = 0, coop = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(jacobi_block_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemMax);
  if (e == cudaSuccess)
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, jacobi_block_kernel, JB_THREADS, smem);
  if (e != cudaSuccess) return e;
  if (!coop || per_sm < 1) return cudaErrorNotSupported;
  int grid = nsm * per_sm;
  if (grid > nslots) grid = nslots;
  // one slot per SM: shared memory that keeps a second CTA off (two on one SM
  // would share its FP64 units while others idle)
  if (nslots <= nsm && smem < kSmemMax / 2 + 1024) smem = kSmemMax / 2 + 1024;
  if ((nslots + grid - 1) / grid > TNX_JB_MAXSLOTS) return cudaErrorInvalidValue;   // tnx_jacobi_block_fits
  float tol2 = (float)(tol * tol);
  void* args[] = {(void*)&groups, (void*)&slots, (void*)&nslots, (void*)&max_sweeps, (void*)&tol2,
                  (void*)&met,    (void*)&cnt,   (void*)&status, (void*)&sweeps_out};
  e = cudaLaunchCooperativeKernel((const void*)jacobi_block_kernel, dim3(grid), dim3(JB_THREADS), args, smem, st);
  if (e != cudaSuccess) return e;
  tnx_note_launch(1);
  return cudaSuccess;
}
