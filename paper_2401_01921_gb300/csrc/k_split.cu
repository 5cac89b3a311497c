// Split-precision grouped GEMM on the tcgen05 tensor cores (sm_103a).
//
// The fused-sector products of a pairwise contraction (Sec. 7 of
// arXiv 2401.01921; the paper runs them as FP64 library GEMMs) are computed to
// FP64 accuracy from 16-bit tensor-core products with the error-free slicing
// of Ozaki, Ogita, Oishi and Rump (Numer. Algorithms 59, 2012):
//
//  * every row of A (and every column of B) gets a common power-of-two scale
//    2^(E+1) from the exponent E of its largest entry; an entry x becomes the
//    signed fixed-point integer v = round(x 2^(F-E-2)), |v| <= 2^(F-1),
//    F = n*beta, written in n balanced base-2^beta digits
//    v = sum_i d_i 2^(beta(n-1-i)), d_i in [-2^(beta-1), 2^(beta-1)]; each
//    digit is an integer, exact in BF16 or FP16;
//  * the product sum_k a_k b_k becomes sum over digit pairs (i, j); pairs with
//    the same level t = i + j share one FP32 accumulator in tensor memory; all
//    pairs with t <= n-1 are formed (terms below 2^-(beta n) are dropped); the
//    accumulators of consecutive levels sit in consecutive TMEM columns, so
//    one MMA of A slice i against the stacked B slices 0..n-1-i feeds all of
//    its levels at once;
//  * the K loop runs in chunks of KC = 640: with beta = 7 a level sums at
//    most n * KC * 64^2 < 2^24, so every FP32 accumulation is exact; after
//    each chunk the levels are read out of tensor memory and added, exactly,
//    into a 64-bit integer fixed-point accumulator
//    I = sum_t L_t 2^(beta(n-1-t));
//  * the result is rounded once: C = I * 2^(E_r + E_c + 2 - 2(F-1) + beta(n-1)).
// The only error is the rounding of each operand to F-1 bits below its
// row / column maximum and the dropped levels: about 2^-40 relative to
// max|row| * max|col| * K.
//
// Kernel layout: 128 x 64 output tiles, 10 warps per CTA: warp 0 issues the
// bulk copies (the TMA engine, cp.async.bulk) of pre-tiled slices into a
// 3-stage shared-memory ring, warp 1 issues tcgen05.mma (one elected lane),
// warps 2-9 (two per quarter of the TMEM lanes, each taking half of the
// tile's columns) drain tensor memory (tcgen05.ld) into the integer accumulators
// and write FP64.  Operands sit in global memory already in the canonical
// no-swizzle K-major core-matrix layout, so a stage is one contiguous copy.
// Every wait on an mbarrier is bounded (about a second of clock); a wait that
// runs out records an error code and the CTA winds down without hanging.
//
// The same kernel, instantiated with TF = true, is the one-pass TF32 variant:
// one "slice" per operand holding the entry scaled by its row (column) power of
// two and rounded to TF32 (10 explicit mantissa bits, nearest-even), 16 K
// values (64 bytes) per stage and row, tcgen05.mma.kind::tf32 with FP32
// accumulation per 640-long K chunk, chunks summed in FP64 by the epilogue.
#include <cooperative_groups.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "tnx_internal.h"

namespace {

constexpr int TM = 128;            // tile rows (A)
constexpr int TK = 32;             // K per stage
constexpr int KC = 640;            // K per exact chunk
constexpr int STAGES = 3;
constexpr int MAXN = 6;            // slices
constexpr int ATILE = TM * TK * 2; // bytes of one A slice tile (8 KB)
// tile columns (B rows): TNV = 64 (wide) or 32 (narrow); one B slice tile is TNV * TK * 2 bytes
constexpr long long WAIT_LIMIT = 2000000000LL;   // clock cycles (~1 s)
constexpr int EPI_WARPS = 8;       // epilogue warps: two per TMEM lane quarter, each takes half the columns
constexpr int SPLIT_THREADS = 32 * (2 + EPI_WARPS);

// ------------------------------------------------------------- PTX helpers
__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count));
}

__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

__device__ __forceinline__ bool mbar_try(uint64_t* bar, uint32_t phase) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(phase)
      : "memory");
  return ok != 0;
}

// bounded wait; returns false (and records `code`) if the limit runs out
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t phase, int32_t* status, int code,
                                          volatile int* abort_flag) {
  const long long t0 = clock64();
  while (!mbar_try(bar, phase)) {
    if (*abort_flag) return false;
    if (clock64() - t0 > WAIT_LIMIT) {
      *(volatile int32_t*)status = code;   // host memory (any of the codes will do)
      *abort_flag = 1;
      return false;
    }
  }
  return true;
}

__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(smem_u32(dst)),
      "l"(src), "r"(bytes), "r"(smem_u32(bar))
      : "memory");
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// shared-memory matrix descriptor: no swizzle, K-major, core matrices of
// 8 rows x 16 bytes; LBO = stride between core matrices along K (128 B),
// SBO = stride between 8-row groups (512 B for a 32-wide K tile).
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr) {
  uint64_t d = 0;
  d |= (uint64_t)((addr & 0x3FFFF) >> 4);
  d |= (uint64_t)(128 >> 4) << 16;
  d |= (uint64_t)(512 >> 4) << 32;
  d |= (uint64_t)1 << 46;   // descriptor version for tcgen05
  return d;                 // base offset 0, swizzle none
}

// instruction descriptor, kind::f16: D f32, A/B bf16 (1) or f16 (0), both K-major, M = 128, N = n
__device__ __forceinline__ uint32_t instr_desc(int f16, int n) {
  const uint32_t ab = f16 ? 0u : 1u;
  return (1u << 4) | (ab << 7) | (ab << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(TM >> 4) << 24);
}

// (value of a 64-bit integer) * 2^e rounded to nearest-even FP64, with integer
// operations only (the FP64 pipe of this part is slow); results below the
// normal range flush to zero.
__device__ __forceinline__ double i64_scaled_to_double(long long v, int e) {
  if (v == 0) return 0.0;
  const unsigned long long sign = v < 0 ? (1ull << 63) : 0ull;
  unsigned long long u = v < 0 ? (unsigned long long)(-v) : (unsigned long long)v;
  const int lz = __clzll(u);
  u <<= lz;                                   // leading one at bit 63
  unsigned long long mant = u >> 11;          // 53 bits
  const unsigned long long rem = u & 0x7FFull;
  if (rem > 0x400ull || (rem == 0x400ull && (mant & 1ull))) mant += 1;
  int ex = 63 - lz + e;
  if (mant >> 53) {
    mant >>= 1;
    ex += 1;
  }
  const int biased = ex + 1023;
  if (biased <= 0) return __longlong_as_double((long long)sign);
  if (biased >= 2047) return __longlong_as_double((long long)(sign | 0x7FF0000000000000ull));
  return __longlong_as_double((long long)(sign | ((unsigned long long)biased << 52) | (mant & 0xFFFFFFFFFFFFFull)));
}

// The same value through the hardware conversion: __ll2double_rn rounds v to
// 53 bits (nearest-even) and adding e to the exponent field is the exact
// scaling by 2^e while the result stays normal; outside that range the
// integer routine above decides.
__device__ __forceinline__ double i64_scaled_fast(long long v, int e) {
  if (v == 0) return 0.0;
  const long long bits = __double_as_longlong(__ll2double_rn(v));
  const int ex = (int)((bits >> 52) & 0x7FF) + e;
  if (ex >= 1 && ex <= 2046) return __longlong_as_double(bits + ((long long)e << 52));
  return i64_scaled_to_double(v, e);
}

// The same value and rounding on the integer units alone, |v| < 2^62: the leading one
// goes to bit 62, the low 10 bits are rounded off to nearest-even, and a carry out of
// the mantissa runs into the exponent.
__device__ __forceinline__ double i64_scaled_alu(long long v, int e) {
  const unsigned long long u = (unsigned long long)(v < 0 ? -v : v);
  const int lz = __clzll((long long)u);
  const int ex = 1086 - lz + e;   // biased exponent of the leading one
  if (v != 0 && (unsigned)(ex - 1) >= 2045u) return i64_scaled_to_double(v, e);
  const unsigned long long w = u << ((lz - 1) & 63);
  const unsigned long long m = (w + 0x1FFull + ((w >> 10) & 1ull)) >> 10;   // 2^52 .. 2^53
  const unsigned long long bits = ((unsigned long long)(unsigned)(ex - 1) << 52) + m;
  return v != 0 ? __longlong_as_double((long long)(bits | ((unsigned long long)v & (1ull << 63)))) : 0.0;
}

// kind::tf32: D f32, A/B tf32 (format 2), both K-major, M = 128, N = n
__device__ __forceinline__ uint32_t instr_desc_tf32(int n) {
  return (1u << 4) | (2u << 7) | (2u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(TM >> 4) << 24);
}

__device__ __forceinline__ void mma_tf32(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                         uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem_d),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}

__device__ __forceinline__ void mma_f16(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                        uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem_d),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}

__device__ __forceinline__ void mma_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
               : "memory");
}

__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t* r) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr));
}

__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// ------------------------------------------------------------ slicing
// 64 * (1 + 128 + ... + 128^5): added to a signed 42-bit value it makes every
// base-128 digit non-negative (digit i of the sum is digit i of v plus 64)
constexpr long long DIGIT_BIAS = 64LL * ((1LL << 42) - 1) / 127;

// The six digits of one entry, plus 64 each, as bytes: x[0] holds those of slices 5,
// 4, 3 (bytes 0, 1, 2), x[1] those of slices 2, 1, 0; byte 3 is the high byte of
// 128.0 in BF16 (1024.0 in FP16), so that a digit byte below it is the 16-bit float
// 128 + e (1024 + e), e <= 128.
struct DigitBytes {
  uint32_t x[2];
};
template <bool F16>
__device__ __forceinline__ DigitBytes digit_bytes(unsigned long long bits, int shift) {
  // |x| 2^(F-E-2) rounded half up is (t + 1) / 2 (whole part) with t = m53 >> (shift + 11),
  // shift = E_row - E >= 0, and with v that value signed, v + DIGIT_BIAS is the whole
  // part of half of (t or, for x < 0, its complement) + 1 + 2 DIGIT_BIAS.
  const uint32_t hi = (uint32_t)(bits >> 32);
  const int s = (hi & 0x7FF00000u) == 0 ? 63 : min(shift + 11, 63);   // zeros and subnormals: t = 0
  const unsigned long long m53 = (bits & 0xFFFFFFFFFFFFFull) | (1ull << 52);
  const unsigned long long sign = (unsigned long long)((long long)bits >> 63);
  const unsigned long long u2 = ((m53 >> s) ^ sign) + (unsigned long long)(2 * DIGIT_BIAS + 1);
  const uint32_t lo = (uint32_t)u2, up = (uint32_t)(u2 >> 22);
  const uint32_t top = F16 ? 0x64000000u : 0x43000000u;
  DigitBytes d;
  d.x[0] = ((lo >> 1) & 0x7Fu) | top;
  d.x[0] |= lo & 0x7F00u;
  d.x[0] |= (lo << 1) & 0x7F0000u;
  d.x[1] = (up & 0x7Fu) | top;
  d.x[1] |= (up << 1) & 0x7F00u;
  d.x[1] |= (up << 2) & 0xFF0000u;   // the top digit plus 64 reaches 128
  return d;
}

// Digits of slice i (0 = most significant) of two entries, less the 64, as a packed
// pair of 16-bit floats: 128 + e (1024 + e) less 192 (1088) is exact.
template <bool F16>
__device__ __forceinline__ uint32_t digit_pair(const DigitBytes& a, const DigitBytes& b, int i) {
  const int w = i < 3, byte = w ? 2 - i : 5 - i;
  const uint32_t p = __byte_perm(a.x[w], b.x[w], 0x7030u + 0x0400u + 0x0101u * (uint32_t)byte);
  if constexpr (F16) {
    const __half2 r = __hadd2(*(const __half2*)&p, __floats2half2_rn(-1088.0f, -1088.0f));
    return *(const uint32_t*)&r;
  } else {
    const __nv_bfloat162 r = __hadd2(*(const __nv_bfloat162*)&p, __floats2bfloat162_rn(-192.0f, -192.0f));
    return *(const uint32_t*)&r;
  }
}

// Slices of the packed operands, one CTA (8 warps) per work item.  Rows are
// taken in groups of 8 (rows past the operand's end in its last group give zero
// slices; the rows that pad it to whole tiles keep the zeros of the allocation); in a
// warp, lane = (row in group) * 4 + (8-column group).  A job gives each group
// SliceJob::wpg warps (1, 2, 4 or 8: more for longer rows), so an item is
// 8 / wpg groups; the warps of a group take every wpg-th 32-wide K tile, 8 entries
// per lane.  First the biased exponent of each row's largest |x| (over a lane's
// entries, then the lanes and the group's warps combine), stored for the GEMM
// epilogue; then the tiles are sliced, 16 bytes per slice per lane written in the
// tiled core-matrix layout the GEMM copies in.
// A warp keeps the entries of its first two tiles in registers between the two
// parts (all of them for K up to 512), and reads ahead by two tiles past that.
// With KX (K balancing), entry k counts as x * 2^(kx_sign * E_k), E_k the
// exponent of column k's largest entry in A: A's columns are scaled by 2^-E_k
// and B's rows by 2^E_k, exactly, so the product is unchanged while a row of
// A (column of B) whose entries scale differently along K keeps its bits.
// Only exponents move: the digits of x * 2^s are those of x with the
// effective exponent E + s.
// Instruction issue and load latency bound it.  Digits through byte permutes and
// packed 16-bit adds (33 instead of about 56 integer and FP32 instructions per entry)
// and one read of every entry instead of two: 47 -> 36 us for the last operand's 7.2M
// entries at bond dimension 2048 (ncu, cold), the vector mode 21.5 -> 16.4 us.
__device__ __forceinline__ int kx_shift(int raw, int sign) {
  return raw > 0 ? sign * (raw - 1023) : 0;   // raw: biased exponent, 0 for a zero column
}

// With VEC (vector mode, no K balancing) a row's entries come from the
// Lanczos vector through the row table, scaled by *inv, and the scaled values
// are written out as the next basis vector (VecSrc).
template <bool F16, bool KX, bool VEC>
__global__ void __launch_bounds__(256, 3) slice_rows_kernel(const SliceJob* __restrict__ jobs,
                                                            const int2* __restrict__ items, int64_t total,
                                                            double* const* __restrict__ slots, VecSrc vs) {
  static_assert(!(KX && VEC), "vector mode slices without K balancing");
  static_assert(MAXN * 7 == 42, "digit_bytes: 53 - 42 = 11 bits go with a shift of 0");
  tnx_grid_dependency();
  if constexpr (VEC) {
    if (*(volatile const int32_t*)(vs.state + 1) != 0) return;   // the solve has stopped
  }
  const double vinv = VEC ? *vs.inv : 1.0;
  __shared__ int s_max[8][8];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int r8 = lane >> 2, kq = lane & 3;
  for (int64_t w = blockIdx.x; w < total; w += gridDim.x) {
    const int2 item = items[w];   // (job, first 8-row group)
    const SliceJob& j = jobs[item.x];
    const int wpg = j.wpg;                        // uniform over the CTA
    const int sub = wid / wpg, wl = wid - sub * wpg;
    const int tile_rows = j.tile_rows, K = j.K;
    const int64_t ngroups = ((int64_t)j.rows + 7) / 8;
    const int64_t rg = (int64_t)item.y + sub;
    const int KT = (K + TK - 1) / TK;
    const int64_t row = rg * 8 + r8;
    const bool live = rg < ngroups && row < j.rows;
    int64_t voff = 0;   // vector mode: offset of the row's K entries in the vector
    const double* src;
    if constexpr (VEC) {
      voff = live ? vs.rowtab[j.src_off + row] : 0;
      src = vs.w + voff;
    } else {
      src = slots[j.src_slot] + j.src_off + row * j.ld;
    }
    const int32_t* kxp = KX ? (const int32_t*)slots[j.kx_slot] + j.kx_off : nullptr;
    // This lane's 8 entries of K tile kt (zeros past K).  Packed rows are whole
    // 32-byte units (ld a multiple of 4, bases 32-byte aligned).
    auto load = [&](int kt, unsigned long long (&x)[8], bool keep) {
      const int k = kt * TK + kq * 8;
#pragma unroll
      for (int e = 0; e < 8; ++e) x[e] = 0ull;
      if (!live || k >= K) return;
      if constexpr (VEC) {
#pragma unroll
        for (int e = 0; e < 8; ++e)
          if (k + e < K) {
            const double v = src[k + e] * vinv;
            if (keep) vs.vdst[voff + k + e] = v;
            x[e] = (unsigned long long)__double_as_longlong(v);
          }
      } else {
        const ulonglong2* p = (const ulonglong2*)(src + k);
#pragma unroll
        for (int h = 0; h < 4; ++h)
          if (k + 2 * h < K) {
            const ulonglong2 v = p[h];
            x[2 * h] = v.x;
            x[2 * h + 1] = k + 2 * h + 1 < K ? v.y : 0ull;
          }
      }
    };
    auto shifts = [&](int kt, int (&sh)[8]) {   // K balancing words: whole K tiles, 16-byte aligned
      if constexpr (KX) {
        const int4* p = (const int4*)(kxp + kt * TK + kq * 8);
        const int4 a = p[0], b = p[1];
        const int raw[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
#pragma unroll
        for (int e = 0; e < 8; ++e) sh[e] = kx_shift(raw[e], j.kx_sign);
      } else {
#pragma unroll
        for (int e = 0; e < 8; ++e) sh[e] = 0;
      }
    };
    constexpr int ZROW = KX ? -(1 << 20) : 0;   // no nonzero entry
    int mx = ZROW;
    auto scan = [&](int kt, const unsigned long long (&x)[8]) {   // the largest (effective) exponent field
      if (!live || kt >= KT) return;
      int sh[8];
      shifts(kt, sh);
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        const int eb = (int)((x[e] >> 52) & 0x7FF);
        if constexpr (KX) {
          if (eb != 0) mx = max(mx, eb + sh[e]);
        } else {
          mx = max(mx, eb);
        }
      }
    };
    unsigned long long x0[8], x1[8];
    load(wl, x0, true);
    load(wl + wpg, x1, true);
    scan(wl, x0);
    scan(wl + wpg, x1);
    for (int kt = wl + 2 * wpg; kt < KT; kt += wpg) {
      unsigned long long x2[8];
      load(kt, x2, false);
      scan(kt, x2);
    }
#pragma unroll
    for (int o = 1; o < 4; o <<= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if (wpg > 1) {
      if (kq == 0) s_max[wid][r8] = mx;
      __syncthreads();
      for (int q = sub * wpg; q < sub * wpg + wpg; ++q) mx = max(mx, s_max[q][r8]);
      __syncthreads();   // s_max is rewritten by the next item
    }
    if (rg >= ngroups) continue;   // a group past the job's last one
    const int eb_r = mx;
    if (live && kq == 0 && wl == 0) ((int32_t*)slots[j.exp_slot])[j.exp_off + row] = eb_r != ZROW ? eb_r : 0;
    const int64_t mt = row / tile_rows;
    const int rin = (int)(row % tile_rows);
    const int64_t tile_bytes = (int64_t)tile_rows * TK * 2;
    char* base = (char*)slots[j.dst_slot] + j.dst_off_bytes + (int64_t)(rin >> 3) * 512 + kq * 128 + (rin & 7) * 16;
    for (int kt = wl; kt < KT; kt += wpg) {
      int sh[8];
      shifts(kt, sh);
      uint32_t sl[MAXN][4];
#pragma unroll
      for (int e = 0; e < 8; e += 2) {
        const DigitBytes a = digit_bytes<F16>(x0[e], eb_r - (int)((x0[e] >> 52) & 0x7FF) - sh[e]);
        const DigitBytes c = digit_bytes<F16>(x0[e + 1], eb_r - (int)((x0[e + 1] >> 52) & 0x7FF) - sh[e + 1]);
#pragma unroll
        for (int i = 0; i < MAXN; ++i) sl[i][e >> 1] = digit_pair<F16>(a, c, i);
      }
      char* dst = base + (mt * KT + kt) * MAXN * tile_bytes;
#pragma unroll
      for (int i = 0; i < MAXN; ++i) *(uint4*)(dst + i * tile_bytes) = make_uint4(sl[i][0], sl[i][1], sl[i][2], sl[i][3]);
#pragma unroll
      for (int e = 0; e < 8; ++e) x0[e] = x1[e];
      if (kt + 2 * wpg < KT) load(kt + 2 * wpg, x1, true);
    }
  }
}

// Column maxima of the exponent fields of A: an item is 32 K indices (one per lane)
// and all rows (eight per warp and pass, loads in flight together).  Its CL CTAs, a
// cluster, share the rows; each combines its warps in its shared memory, and the
// first adds the others' maxima from there and stores one word per K index.  A maximum
// across unrelated CTAs wanted a launch that zeroes the words first (3 us per product);
// a single CTA per item is too slow for the 1280 rows of an environment update at
// bond dimension 2048 (19 us; 12 with the zeroing launch; 11 with clusters of 8).
constexpr int KEXP_T = 256, KEXP_CL = 8;
template <int CL>
__global__ void __launch_bounds__(KEXP_T) kexp_kernel(const KexpJob* __restrict__ jobs,
                                                      const int2* __restrict__ items, double* const* __restrict__ slots) {
  tnx_grid_dependency();
  constexpr int NW = KEXP_T / 32;
  __shared__ int s_mx[NW][32];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int rank = CL > 1 ? (int)(blockIdx.x % CL) : 0;
  const int2 it = items[blockIdx.x / CL];   // (job, first K index)
  const KexpJob& j = jobs[it.x];
  const int k = it.y + lane;
  int mx = 0;
  if (k < j.K) {
    const uint32_t* hi = (const uint32_t*)(slots[j.src_slot] + j.src_off + k) + 1;
    for (int r0 = rank * NW + wid; r0 < j.rows; r0 += 8 * NW * CL) {
      uint32_t h[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int r = r0 + NW * CL * u;
        h[u] = r < j.rows ? hi[2 * ((int64_t)r * j.ld)] : 0u;
      }
#pragma unroll
      for (int u = 0; u < 8; ++u) mx = max(mx, (int)((h[u] >> 20) & 0x7FFu));
    }
  }
  s_mx[wid][lane] = mx;
  __syncthreads();
  if (wid == 0) {
#pragma unroll
    for (int q = 1; q < NW; ++q) mx = max(mx, s_mx[q][lane]);
    if (CL > 1) s_mx[0][lane] = mx;
  }
  if constexpr (CL > 1) {
    auto cluster = cooperative_groups::this_cluster();
    cluster.sync();
    if (rank == 0 && wid == 0)
#pragma unroll
      for (int c = 1; c < CL; ++c) mx = max(mx, cluster.map_shared_rank(&s_mx[0][0], c)[lane]);
    cluster.sync();   // no CTA leaves while its maxima are read
  }
  if (rank == 0 && wid == 0 && k < j.K) ((int32_t*)slots[j.kx_slot])[j.kx_off + k] = mx;
}

// TF32 operands of the one-pass variant: one CTA (8 warps) per item of eight
// 8-row groups, one group per warp; lane = (row in group) * 4 + (4-column
// group).  A row is scaled by 2^-E (E: unbiased exponent of its largest |x|,
// stored for the epilogue like the split path's), rounded to 11 significant
// bits (nearest-even) straight from the FP64 bits, and written as FP32 words
// in the tiled core-matrix layout, 16 K values (64 bytes) per tile row.
// Entries more than 2^126 below their row maximum flush to zero.
__device__ __forceinline__ uint32_t tf32_word(unsigned long long bits, int eb_r) {
  const int eb = (int)((bits >> 52) & 0x7FF);
  const uint32_t sign = (uint32_t)(bits >> 63) << 31;
  if (eb == 0 || eb_r == 0) return sign;
  int ef = eb - eb_r + 127;
  unsigned long long keep = ((bits & 0xFFFFFFFFFFFFFull) | (1ull << 52)) >> 42;   // 11 bits
  const unsigned long long rem = bits & ((1ull << 42) - 1), half = 1ull << 41;
  if (rem > half || (rem == half && (keep & 1ull))) keep += 1;
  if (keep >> 11) {
    keep >>= 1;
    ef += 1;
  }
  if (ef <= 0) return sign;
  return sign | ((uint32_t)ef << 23) | ((uint32_t)(keep & 0x3FFull) << 13);
}

__global__ void __launch_bounds__(256) tf32_rows_kernel(const SliceJob* __restrict__ jobs,
                                                        const int2* __restrict__ items, int64_t total,
                                                        double* const* __restrict__ slots) {
  tnx_grid_dependency();
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int r8 = lane >> 2, kq = lane & 3;
  constexpr int TKF = 16;   // K values per tile row
  for (int64_t w = blockIdx.x; w < total; w += gridDim.x) {
    const int2 item = items[w];   // (job, first 8-row group)
    const SliceJob& j = jobs[item.x];
    const int64_t ngroups = ((int64_t)j.rows + j.tile_rows - 1) / j.tile_rows * (j.tile_rows / 8);
    const int64_t rg = (int64_t)item.y + wid;
    if (rg >= ngroups) continue;   // uniform over the warp
    const int64_t row = rg * 8 + r8;
    const bool live = row < j.rows;
    const double* src = slots[j.src_slot] + j.src_off + row * j.ld;
    unsigned long long mx = 0;
    if (live)
      for (int k = kq; k < j.K; k += 4) {
        const unsigned long long b = __double_as_longlong(src[k]) & 0x7FFFFFFFFFFFFFFFull;
        mx = b > mx ? b : mx;
      }
#pragma unroll
    for (int o = 1; o < 4; o <<= 1) {
      const unsigned long long v = __shfl_xor_sync(0xffffffffu, mx, o);
      mx = v > mx ? v : mx;
    }
    const int eb_r = (int)(mx >> 52);
    if (live && kq == 0) ((int32_t*)slots[j.exp_slot])[j.exp_off + row] = eb_r;
    const int KT = (j.K + TKF - 1) / TKF;
    const int tile_rows = j.tile_rows;
    const int64_t mt = row / tile_rows;
    const int rin = (int)(row % tile_rows);
    const int64_t tile_bytes = (int64_t)tile_rows * TKF * 4;
    char* base = (char*)slots[j.dst_slot] + j.dst_off_bytes;
    const int64_t inner = (int64_t)(rin >> 3) * 512 + kq * 128 + (rin & 7) * 16;
    for (int kt = 0; kt < KT; ++kt) {
      uint32_t o[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int k = kt * TKF + kq * 4 + e;
        const unsigned long long bits = (live && k < j.K) ? (unsigned long long)__double_as_longlong(src[k]) : 0ull;
        o[e] = tf32_word(bits, eb_r);
      }
      *(uint4*)(base + (mt * KT + kt) * tile_bytes + inner) = make_uint4(o[0], o[1], o[2], o[3]);
    }
  }
}

// --------------------------------------------------------- split GEMM
struct SplitShared {
  uint64_t full[STAGES], empty[STAGES];
  uint64_t accfull, accempty, done;
  uint32_t tmem_base;
  int abort_flag;
};

// Persistent over tiles: CTA b takes tiles b, b + gridDim.x, ... of the list
// (the host orders it longest-K first, or lays out a per-CTA schedule whose
// holes carry group -1).  Tensor memory and the barriers are set
// up once per CTA; the stage ring and the chunk hand-off between the MMA warp
// and the epilogue warps continue across tiles, so the producer streams the
// next tile's slices while the epilogue drains the current one.
template <int NS, int TNV, bool TF, int MODE>
__global__ void __launch_bounds__(SPLIT_THREADS, 1) split_gemm_kernel(const SplitGroup* __restrict__ groups,
                                                             const GemmTile* __restrict__ tiles, int ntiles, int beta,
                                                             int f16, double* const* __restrict__ slots,
                                                             int32_t* status) {
  tnx_grid_dependency();
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* ring = (unsigned char*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  constexpr int BTILE = TNV * TK * 2;
  constexpr int ECOLS = TNV / 2;     // tile columns per epilogue warp
  constexpr int STAGE_BYTES = NS * (ATILE + BTILE);
  SplitShared* sh = (SplitShared*)(ring + STAGES * STAGE_BYTES);
  double (*sh_stage)[4] = (double (*)[4])(ring + STAGES * STAGE_BYTES + ((sizeof(SplitShared) + 15) & ~(size_t)15));
  int* sh_ebc = (int*)(sh_stage + EPI_WARPS * 32);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  constexpr int TKE = TF ? 16 : TK;   // K values per stage (64 bytes per row either way)
  constexpr int KTPC = KC / TKE;      // K tiles per chunk
  static_assert(!TF || NS == 1, "the TF32 variant has one operand slice");

  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(&sh->full[s], 1);
      mbar_init(&sh->empty[s], 1);
    }
    mbar_init(&sh->accfull, 1);
    mbar_init(&sh->accempty, EPI_WARPS);
    mbar_init(&sh->done, 1);
    sh->abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(&sh->tmem_base)));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = sh->tmem_base;
  volatile int* abort_flag = &sh->abort_flag;

  if (warp == 0) {
    // ---------------- producer: bulk copies of pre-tiled slices
    if (lane == 0) {
      int g = 0;   // global K-tile counter of this CTA
      for (int ti = blockIdx.x; ti < ntiles && !*abort_flag; ti += gridDim.x) {
        const GemmTile tl = tiles[ti];
        if (tl.group < 0) continue;   // a hole of the per-CTA schedule
        const SplitGroup gr = groups[tl.group];
        const int KT = (gr.K + TKE - 1) / TKE;
        const char* Ab = (const char*)slots[gr.a_slot] + gr.a_off_bytes + ((int64_t)(tl.m0 / TM) * KT) * NS * ATILE;
        const char* Bb = (const char*)slots[gr.b_slot] + gr.b_off_bytes + ((int64_t)(tl.n0 / TNV) * KT) * NS * BTILE;
        for (int kt = 0; kt < KT; ++kt, ++g) {
          const int s = g % STAGES;
          const uint32_t ph = (uint32_t)(g / STAGES) & 1u;
          if (g >= STAGES && !mbar_wait(&sh->empty[s], ph ^ 1u, status, 11, abort_flag)) break;
          unsigned char* sa = ring + s * STAGE_BYTES;
          mbar_expect_tx(&sh->full[s], NS * (ATILE + BTILE));
          bulk_g2s(sa, Ab + (int64_t)kt * NS * ATILE, NS * ATILE, &sh->full[s]);
          bulk_g2s(sa + NS * ATILE, Bb + (int64_t)kt * NS * BTILE, NS * BTILE, &sh->full[s]);
        }
      }
      // never leave copies in flight: wait (bounded) for the last issued stages to land
      for (int q = (g > STAGES ? g - STAGES : 0); q < g; ++q) {
        const long long t0 = clock64();
        while (!mbar_try(&sh->full[q % STAGES], (uint32_t)(q / STAGES) & 1u) && clock64() - t0 < WAIT_LIMIT) {
        }
      }
    }
  } else if (warp == 1) {
    // ---------------- MMA issuer
    if (lane == 0) {
      int g = 0, chunk = 0;
      bool ok = true;
      for (int ti = blockIdx.x; ti < ntiles && ok; ti += gridDim.x) {
        const int tg = tiles[ti].group;
        if (tg < 0) continue;
        const SplitGroup gr = groups[tg];
        const int KT = (gr.K + TKE - 1) / TKE;
        for (int kt = 0; kt < KT; ++kt, ++g) {
          const int s = g % STAGES;
          const uint32_t ph = (uint32_t)(g / STAGES) & 1u;
          const bool first_in_chunk = (kt % KTPC) == 0;
          const bool last_in_chunk = ((kt + 1) % KTPC) == 0 || kt == KT - 1;
          if (first_in_chunk && chunk > 0 && !mbar_wait(&sh->accempty, (uint32_t)(chunk - 1) & 1u, status, 12, abort_flag)) {
            ok = false;
            break;
          }
          if (!mbar_wait(&sh->full[s], ph, status, 13, abort_flag)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t sa = smem_u32(ring + s * STAGE_BYTES);
          const uint32_t sb = sa + NS * ATILE;
          // A slice i meets the B slices j = 0 .. NS-1-i stacked along N (they are
          // consecutive TNV-row tiles, so the stack is one taller K-major operand);
          // its output columns are the accumulators of levels i .. NS-1, also
          // consecutive: one MMA (N <= 256, else two of half the stack) per A slice
          // and K step.  Halves because an MMA reads 4 KB of A and 32 bytes per
          // column of B while it computes for N / 2 cycles: below N = 128 it waits for
          // shared memory (128 bytes per cycle), as a remainder of 64 columns did.
          // A K step is 32 bytes of every row: 16 values of BF16/FP16, 8 of TF32.
#pragma unroll
          for (int ks = 0; ks < TK / 16; ++ks) {
#pragma unroll
            for (int i = 0; i < NS; ++i) {
              const uint64_t ad = smem_desc(sa + i * ATILE + ks * 256);
              const uint32_t acc = (first_in_chunk && ks == 0 && i == 0) ? 0u : 1u;
              const int cols = (NS - i) * TNV;
              const int n = cols <= 256 ? cols : cols / 2;
              static_assert(TNV % 32 == 0 && NS * TNV <= 512, "half a stack is a multiple of 16 columns, at most 256");
#pragma unroll
              for (int c0 = 0; c0 < cols; c0 += n) {
                const uint64_t bd = smem_desc(sb + c0 * (TK * 2) + ks * 256);
                if constexpr (TF) mma_tf32(tmem + (uint32_t)(i * TNV + c0), ad, bd, instr_desc_tf32(n), acc);
                else mma_f16(tmem + (uint32_t)(i * TNV + c0), ad, bd, instr_desc(f16, n), acc);
              }
            }
          }
          mma_commit(&sh->empty[s]);
          if (last_in_chunk) {
            mma_commit(&sh->accfull);
            ++chunk;
          }
        }
      }
      // all MMAs issued by this thread have completed before tensor memory is freed
      mma_commit(&sh->done);
      const long long t0 = clock64();
      while (!mbar_try(&sh->done, 0) && clock64() - t0 < WAIT_LIMIT) {
      }
    }
  } else {
    // ---------------- epilogue: warps 2..9; warp w reads TMEM lanes 32*(w%4) ..
    // (rows of the tile) and one half of the tile's columns
    const int sub = warp & 3;
    const int cb = ((warp - 2) >> 2) * ECOLS;
    int chunk = 0;
    bool ok = true;
    for (int ti = blockIdx.x; ti < ntiles && ok; ti += gridDim.x) {
      const GemmTile tl = tiles[ti];
      if (tl.group < 0) continue;
      const SplitGroup gr = groups[tl.group];
      const int KT = (gr.K + TKE - 1) / TKE;
      const int nchunks = (KT + KTPC - 1) / KTPC;
      const int row = tl.m0 + sub * 32 + lane;
      // This warp's part of the tile that exists: no columns when its rows don't.  Short
      // contractions are bound by this epilogue, not by the tensor cores (about 10 against
      // 9 thousand cycles a tile at bond dimension 2048), and small blocks leave most of a
      // tile empty: with the skip, two conversion units and the even MMAs the products of a
      // batch of 48 small sites went from 344 to 265 us, the two at 4096 from 570 to 545
      // us (ncu, cold); a solve at 2048 from 6106 to 6034 us.
      const int ncol = tl.m0 + sub * 32 < gr.M ? min(ECOLS, gr.N - tl.n0 - cb) : 0;
      // Row and column exponents are fetched before the first accumulator
      // wait, so their global-load latency hides behind the MMAs.
      double (*stg)[4] = sh_stage + (warp - 2) * 32;
      int* ebc_s = sh_ebc + (warp - 2) * ECOLS;
      const int eb_r = row < gr.M ? ((const int32_t*)slots[gr.ea_slot])[gr.ea_off + row] : 0;
      {
        const int32_t* eb_c = (const int32_t*)slots[gr.eb_slot] + gr.eb_off;
        const int col = tl.n0 + cb + lane;
        if (lane < ECOLS) ebc_s[lane] = col < gr.N ? eb_c[col] : 0;
      }
      long long acc[ECOLS];
      double accd[ECOLS];   // TF32: FP64 sum of the FP32 chunk sums
#pragma unroll
      for (int c = 0; c < ECOLS; ++c) {
        acc[c] = 0;
        accd[c] = 0.0;
      }
      for (int ch = 0; ch < nchunks; ++ch, ++chunk) {
        if (!mbar_wait(&sh->accfull, (uint32_t)chunk & 1u, status, 14, abort_flag)) {
          ok = false;
          break;
        }
        tc_fence_after();
        // all levels of 8 columns in flight at once, one wait per column group
#pragma unroll
        for (int cg = 0; cg < ECOLS / 8; ++cg) {
          if (cg * 8 >= ncol) break;
          uint32_t v[NS][8];
#pragma unroll
          for (int t = 0; t < NS; ++t)
            tmem_ld8(tmem + ((uint32_t)(sub * 32) << 16) + (uint32_t)(t * TNV + cb + cg * 8), v[t]);
          tmem_wait_ld();
#pragma unroll
          for (int c = 0; c < 8; ++c) {
            if constexpr (TF) {
              accd[cg * 8 + c] += (double)__uint_as_float(v[0][c]);
            } else if constexpr (MODE == 2) {
              // MODE 2: every tile of the launch has K <= 160, so each level sum is
              // below 6 * 160 * 64^2 < 2^22, where the FP32 -> int conversion is an
              // exact add of 1.5 * 2^23 on the full-rate ALU, and adjacent levels
              // combine in 32-bit integers before the 64-bit sum
              int d[NS];
#pragma unroll
              for (int t = 0; t < NS; ++t) d[t] = __float_as_int(__uint_as_float(v[t][c]) + 12582912.0f) - 0x4B400000;
              const int lo = d[5] + d[4] * 128, mid = d[3] + d[2] * 128, hi = d[1] + d[0] * 128;   // |.| < 2^30
              acc[cg * 8 + c] += ((long long)hi << 28) + ((long long)mid << 14) + (long long)lo;
            } else {
              // level 0 has one digit pair: |sum| <= 640 * 64^2 < 2^22, the exact add (above);
              // the conversion instruction runs at a quarter of that rate
              static_assert(KC * 64 * 64 < (1 << 22), "level 0 of a chunk");
              long long x = (long long)(__float_as_int(__uint_as_float(v[0][c]) + 12582912.0f) - 0x4B400000) *
                            (1LL << (7 * (NS - 1)));
#pragma unroll
              for (int t = 1; t < NS; ++t)
                x += (long long)__float2int_rn(__uint_as_float(v[t][c])) * (1LL << (7 * (NS - 1 - t)));
              acc[cg * 8 + c] += x;
            }
          }
        }
        tc_fence_before();
        if (lane == 0) mbar_arrive(&sh->accempty);
      }
      if (ok) {
        // Convert and write through a per-warp staging block of 32 rows x 4
        // columns, so each store instruction covers whole 32-byte sectors of
        // eight rows of C instead of one 8-byte word in each of 32 rows.
        // Column c of row r sits at position c ^ ((r >> 2) & 3), which keeps
        // the row-wise writes and the column-wise reads free of bank conflicts.
        __syncwarp();
        double* cbase = slots[gr.c_slot] + gr.c_off;
        // a folded output relayout: column descriptors, destination = the network's output
        // (MODE 1, the folded output relayout: an instantiation of its own, so the
        // plain store path keeps its registers)
        const FinalCol* fcol = MODE == 1 ? (const FinalCol*)slots[gr.fc_slot] + gr.fc_off : nullptr;
        double* obase = MODE == 1 ? slots[gr.out_slot] : nullptr;
        const int r0 = tl.m0 + sub * 32;
#pragma unroll
        for (int c4 = 0; c4 < ECOLS / 4; ++c4) {
          if (c4 * 4 >= ncol) break;
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            if constexpr (TF) {
              // operands were scaled by 2^-(E_r) and 2^-(E_c)
              stg[lane][c ^ ((lane >> 2) & 3)] = ldexp(accd[c4 * 4 + c], eb_r + ebc_s[c4 * 4 + c] - 2046);
            } else {
              const int e = eb_r + ebc_s[c4 * 4 + c] - 2044 - 2 * (NS * beta - 1) + beta * (NS - 1);
              // a conversion takes the FP64 unit 64 cycles: half of them run on the
              // integer units beside it
              stg[lane][c ^ ((lane >> 2) & 3)] =
                  c & 1 ? i64_scaled_alu(acc[c4 * 4 + c], e) : i64_scaled_fast(acc[c4 * 4 + c], e);
            }
          }
          __syncwarp();
          const int cc = lane & 3, col = tl.n0 + cb + c4 * 4 + cc;
          if constexpr (MODE == 1) {
            const FinalCol d = col < gr.N ? fcol[col] : FinalCol{-1, 0};
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              const int rr = q * 8 + (lane >> 2), r = r0 + rr;
              if (r < gr.M && d.off >= 0) obase[d.off + (int64_t)r * d.stride] = stg[rr][cc ^ ((rr >> 2) & 3)];
            }
          } else {
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              const int rr = q * 8 + (lane >> 2), r = r0 + rr;
              if (r < gr.M && col < gr.N) cbase[(int64_t)r * gr.ldc + col] = stg[rr][cc ^ ((rr >> 2) & 3)];
            }
          }
          __syncwarp();
        }
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem));
}

}  // namespace

cudaError_t tnx_launch_slices(const SliceJob* jobs, const int2* items, int64_t total_items, int nslice, int beta,
                              int f16, double* const* slots, cudaStream_t st, int use_kx) {
  if (total_items <= 0) return cudaSuccess;
  if (nslice != MAXN || beta != 7) return cudaErrorInvalidValue;   // the digit code is specialised
  int64_t blocks = total_items;
  if (blocks > 152 * 8) blocks = 152 * 8;
  {
    const dim3 g((int)blocks), b(256);
    const VecSrc none{nullptr, nullptr, nullptr, nullptr, nullptr};
    const cudaError_t le =
        f16 ? (use_kx ? tnx_launch(slice_rows_kernel<true, true, false>, g, b, 0, st, jobs, items, total_items, slots,
                                   none)
                      : tnx_launch(slice_rows_kernel<true, false, false>, g, b, 0, st, jobs, items, total_items,
                                   slots, none))
            : (use_kx ? tnx_launch(slice_rows_kernel<false, true, false>, g, b, 0, st, jobs, items, total_items,
                                   slots, none)
                      : tnx_launch(slice_rows_kernel<false, false, false>, g, b, 0, st, jobs, items, total_items,
                                   slots, none));
    if (le != cudaSuccess) return le;
  }
  tnx_note_launch(1);
  return cudaGetLastError();
}

cudaError_t tnx_launch_slices_vec(const SliceJob* jobs, const int2* items, int64_t total_items, int nslice, int beta,
                                  int f16, double* const* slots, const VecSrc& vs, cudaStream_t st) {
  if (total_items <= 0) return cudaSuccess;
  if (nslice != MAXN || beta != 7) return cudaErrorInvalidValue;   // the digit code is specialised
  if (!vs.rowtab || !vs.w || !vs.vdst || !vs.inv || !vs.state) return cudaErrorInvalidValue;
  int64_t blocks = total_items;
  if (blocks > 152 * 8) blocks = 152 * 8;
  {
    const dim3 g((int)blocks), b(256);
    const cudaError_t le =
        f16 ? tnx_launch(slice_rows_kernel<true, false, true>, g, b, 0, st, jobs, items, total_items, slots, vs)
            : tnx_launch(slice_rows_kernel<false, false, true>, g, b, 0, st, jobs, items, total_items, slots, vs);
    if (le != cudaSuccess) return le;
  }
  tnx_note_launch(1);
  return cudaGetLastError();
}

cudaError_t tnx_launch_kexp(const KexpJob* jobs, const int2* items, int64_t nitems, bool cluster,
                            double* const* slots, cudaStream_t st) {
  if (nitems <= 0) return cudaSuccess;
  if (nitems > INT32_MAX / KEXP_CL) return cudaErrorInvalidValue;
  cudaError_t le;
  if (!cluster) {
    le = tnx_launch(kexp_kernel<1>, dim3((int)nitems), dim3(KEXP_T), 0, st, jobs, items, slots);
  } else {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((int)nitems * KEXP_CL);
    cfg.blockDim = dim3(KEXP_T);
    cfg.stream = st;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    at[1].id = cudaLaunchAttributeClusterDimension;
    at[1].val.clusterDim.x = KEXP_CL;
    at[1].val.clusterDim.y = at[1].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 2;
    le = cudaLaunchKernelEx(&cfg, kexp_kernel<KEXP_CL>, jobs, items, slots);
  }
  if (le != cudaSuccess) return le;
  tnx_note_launch(1);
  return cudaGetLastError();
}

size_t tnx_split_smem_bytes(int nslice, int tn) {
  // alignment slack + stage ring + barriers + epilogue staging (32 rows x 4 doubles
  // per epilogue warp) + column exponents (tn / 2 per epilogue warp)
  return 1024 + (size_t)STAGES * nslice * (ATILE + (size_t)tn * TK * 2) + ((sizeof(SplitShared) + 15) & ~(size_t)15) +
         EPI_WARPS * 32 * 4 * sizeof(double) + EPI_WARPS * (tn / 2) * sizeof(int) + 64;
}

namespace {
template <int TNV, bool TF, int MODE>
cudaError_t launch_split_t(const SplitGroup* groups, const GemmTile* tiles, int ntiles, int beta, int f16,
                           double* const* slots, int32_t* status, cudaStream_t st, int grid) {
  constexpr int NS = TF ? 1 : MAXN;
  const size_t smem = tnx_split_smem_bytes(NS, TNV);
  static int attr_dev = -1;   // the opt-in is per device
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (attr_dev != dev) {
    e = cudaFuncSetAttribute(split_gemm_kernel<NS, TNV, TF, MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)smem);
    if (e != cudaSuccess) return e;
    attr_dev = dev;
  }
  return tnx_launch(split_gemm_kernel<NS, TNV, TF, MODE>, dim3(grid), dim3(SPLIT_THREADS), smem, st,
                    groups, tiles, ntiles, beta, f16, slots, status);
}

// mode: 0 plain stores, 1 folded output relayout, 2 plain stores with the
// short-K level combine (split BF16/FP16 only)
template <int TNV, bool TF>
cudaError_t launch_split(const SplitGroup* groups, const GemmTile* tiles, int ntiles, int beta, int f16,
                         double* const* slots, int32_t* status, cudaStream_t st, int grid, int mode) {
  if (mode == 1) return launch_split_t<TNV, TF, 1>(groups, tiles, ntiles, beta, f16, slots, status, st, grid);
  if constexpr (!TF) {
    if (mode == 2) return launch_split_t<TNV, TF, 2>(groups, tiles, ntiles, beta, f16, slots, status, st, grid);
  }
  return launch_split_t<TNV, TF, 0>(groups, tiles, ntiles, beta, f16, slots, status, st, grid);
}
}  // namespace

cudaError_t tnx_launch_gemm_split(const SplitGroup* groups, const GemmTile* tiles, int ntiles, int nslice, int beta,
                                  int f16, double* const* slots, int32_t* status, cudaStream_t st, int grid, int tn,
                                  int mode) {
  if (ntiles <= 0) return cudaSuccess;
  if (grid <= 0 || grid > ntiles) grid = ntiles;
  if (nslice != MAXN || beta != 7 || (tn != 32 && tn != 64)) return cudaErrorInvalidValue;
  const cudaError_t le =
      tn == 32 ? launch_split<32, false>(groups, tiles, ntiles, beta, f16, slots, status, st, grid, mode)
               : launch_split<64, false>(groups, tiles, ntiles, beta, f16, slots, status, st, grid, mode);
  if (le != cudaSuccess) return le;
  tnx_note_launch(1);
  return cudaGetLastError();
}

cudaError_t tnx_launch_tf32_rows(const SliceJob* jobs, const int2* items, int64_t total_items, double* const* slots,
                                 cudaStream_t st) {
  if (total_items <= 0) return cudaSuccess;
  int64_t blocks = total_items;
  if (blocks > 152 * 8) blocks = 152 * 8;
  const cudaError_t le = tnx_launch(tf32_rows_kernel, dim3((int)blocks), dim3(256), 0, st, jobs, items, total_items,
                                    slots);
  if (le != cudaSuccess) return le;
  tnx_note_launch(1);
  return cudaGetLastError();
}

cudaError_t tnx_launch_gemm_tf32(const SplitGroup* groups, const GemmTile* tiles, int ntiles, double* const* slots,
                                 int32_t* status, cudaStream_t st, int grid, int tn, int fold) {
  if (ntiles <= 0) return cudaSuccess;
  if (grid <= 0 || grid > ntiles) grid = ntiles;
  if (tn != 32 && tn != 64) return cudaErrorInvalidValue;
  const cudaError_t le = tn == 32 ? launch_split<32, true>(groups, tiles, ntiles, 0, 0, slots, status, st, grid, fold)
                                  : launch_split<64, true>(groups, tiles, ntiles, 0, 0, slots, status, st, grid, fold);
  if (le != cudaSuccess) return le;
  tnx_note_launch(1);
  return cudaGetLastError();
}
