// gemm_tc.cu -- C -= A B with FP64 operands on the tcgen05 tensor cores.
//
// The trailing updates of CALU / CAQR are the dense contractions of the
// method (Sec. 3: the Schur complement A22 -= L21 U12 and the compact-WY
// Q^T C).  On GB300 the FP64 pipe retires ~1.2 TFLOP/s while the bf16 tensor
// cores retire ~1.9 PFLOP/s, so the reduced-precision form of the update runs
// there:
//   * split: every row of A (every column of B) is scaled by a power of two,
//     2^-e with |x| < 2^e, and cut into S signed base-256 digits
//     t = sum_k d_k 2^(-8k), |d_1| <= 256, |d_k| <= 128 -- exact FP64 steps.
//     Digit k is stored in bf16 as d_k 2^(-8(k-1)), which bf16 holds exactly;
//   * tcgen05.mma (kind::f16, bf16 x bf16 -> FP32 in tensor memory) sums the
//     digit products d_k d'_l with k + l <= S + 1 for one 128 x 128 tile;
//     operand tiles arrive by TMA (cp.async.bulk.tensor, 128-byte swizzle);
//   * the epilogue reads the accumulator with tcgen05.ld and applies
//     C -= 2^(e_i + f_j - 16) acc in FP64.
// Fused mode: one FP32 accumulator with pre-scaled digits, accurate to about
// 2^-20 relative to max|row of A| max|column of B|; FP64 iterative refinement
// recovers the rest.  Exact mode: integer digits, one accumulator per digit
// diagonal; every diagonal sum is an integer below 2^24 (k <= 128), so the
// tensor cores' FP32 sums are exact and the only error is the dropped digits,
// 2^(-8 S) relative (7 digits: the FP64 level).
//   diagonal k + l = D, digits |d_1| <= 256, |d_k| <= 128, k = 128:
//   D = 2: 2^23, 3: 2^23, 4: 1.25 2^23, 5: 1.5 2^23, 6: 1.75 2^23, 7: 2^24,
//   D = 8: 2.25 2^23 per K block of 64 (so split by K block).
//
// Every wait on an mbarrier is bounded by a clock limit; on a timeout the CTA
// raises a status bit, waits (bounded) for its own copies and MMAs, frees its
// tensor memory and returns.
#include <cuda.h>
#include <cuda_bf16.h>

#include <climits>
#include <type_traits>

#include "ca_internal.cuh"
#include "device_once.cuh"

namespace cagb {

// --------------------------------------------------------------------------
// PTX wrappers
// --------------------------------------------------------------------------
__device__ __forceinline__ uint32_t smem_u32(const void *p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ void fence_mbar_init() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint64_t *bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
               : "memory");
}

// One lane of the (converged) warp.  The compiler knows that what runs under it
// is warp-uniform and keeps the operands of copies and MMAs in uniform
// registers.
__device__ __forceinline__ bool elect_one() {
  uint32_t p;
  asm volatile("{\n\t.reg .pred q;\n\telect.sync _|q, 0xffffffff;\n\tselp.u32 %0, 1, 0, q;\n\t}\n" : "=r"(p));
  return p != 0;
}

// Waits for the phase with parity `parity`; false after ~`limit` SM cycles.
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, uint32_t parity, long long limit) {
  const uint32_t addr = smem_u32(bar);
  const long long t0 = clock64();
  while (true) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}\n"
        : "=r"(done)
        : "r"(addr), "r"(parity)
        : "memory");
    if (done) return true;
    if (clock64() - t0 > limit) return false;
  }
}

__device__ __forceinline__ void tma_load_2d(void *dst, const CUtensorMap *map, uint64_t *bar, int x,
                                            int y) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], "
      "[%2];" ::"r"(smem_u32(dst)),
      "l"((uint64_t)map), "r"(smem_u32(bar)), "r"(x), "r"(y)
      : "memory");
}

__device__ __forceinline__ void tmem_alloc(uint32_t *dst, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(dst)),
               "r"(ncols)
               : "memory");
}
__device__ __forceinline__ void tmem_relinquish() {
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tc_fence_before() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}

__device__ __forceinline__ void tc_mma(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                       uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(d_tmem),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}

__device__ __forceinline__ void tc_commit(uint64_t *bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                   smem_u32(bar))
               : "memory");
}

// Thread i of the warp gets TMEM lane (lane base + i).
// 32 TMEM lanes x 4 consecutive 32-bit columns, without the wait
__device__ __forceinline__ void tmem_ld_32x4(uint32_t taddr, uint32_t (&r)[4]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(taddr));
}
// 32 TMEM lanes x 32 consecutive 32-bit columns, with the wait
__device__ __forceinline__ void tmem_ld_32x32(uint32_t taddr, uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];\n\t"
      "tcgen05.wait::ld.sync.aligned;"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]),
        "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]),
        "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]),
        "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr)
      : "memory");
}
// waits for the loads; every value passes through, so that no use of it moves up
__device__ __forceinline__ void tmem_ld_wait(uint32_t (&r)[8][4]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(r[0][0]), "+r"(r[0][1]), "+r"(r[0][2]), "+r"(r[0][3]), "+r"(r[1][0]), "+r"(r[1][1]),
                 "+r"(r[1][2]), "+r"(r[1][3]), "+r"(r[2][0]), "+r"(r[2][1]), "+r"(r[2][2]), "+r"(r[2][3]),
                 "+r"(r[3][0]), "+r"(r[3][1]), "+r"(r[3][2]), "+r"(r[3][3]), "+r"(r[4][0]), "+r"(r[4][1]),
                 "+r"(r[4][2]), "+r"(r[4][3]), "+r"(r[5][0]), "+r"(r[5][1]), "+r"(r[5][2]), "+r"(r[5][3])
               :
               : "memory");
  asm volatile(""
               : "+r"(r[6][0]), "+r"(r[6][1]), "+r"(r[6][2]), "+r"(r[6][3]), "+r"(r[7][0]), "+r"(r[7][1]),
                 "+r"(r[7][2]), "+r"(r[7][3])
               :
               : "memory");
}

__device__ __forceinline__ long long mad_wide(int a, int b, long long c) {
  long long r;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
  return r;
}

// Shared-memory matrix descriptor of a K-major operand written by TMA with a
// 128-byte swizzle (rows of 128 bytes, groups of 8 rows = 1024 bytes, layout
// type 2) or a 64-byte swizzle (rows of 64 bytes, groups of 8 = 512 bytes,
// layout type 4); sm_100 descriptor version.
__device__ __forceinline__ uint64_t sw_desc(uint32_t saddr, int swz) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr >> 4) & 0x3FFFu);
  d |= (uint64_t)1 << 16;                              // leading byte offset (unused, swizzled K-major)
  d |= (uint64_t)((swz == 2 ? 1024 : 512) >> 4) << 32;  // stride byte offset
  d |= (uint64_t)1 << 46;                              // version
  d |= (uint64_t)swz << 61;                            // layout type
  return d;
}

// Instruction descriptor, kind::f16: D = F32, A = B = BF16, both K-major.
__host__ __device__ constexpr uint32_t idesc_bf16_f32(int M, int N) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

// 2^k as a double for -1022 <= k <= 1023 (IEEE binary64 exponent field).
__device__ __forceinline__ double pow2i(int k) {
  k = k < -1022 ? -1022 : (k > 1023 ? 1023 : k);
  return __longlong_as_double((long long)(k + 1023) << 52);
}

// v * 2^e2 as a double, from the integer bits (round to nearest even) -- no
// FP64-pipe instruction; exact when |v| < 2^53.  The results here stay far
// inside the normal range.
__device__ __forceinline__ double i64_scaled_to_double(long long v, int e2) {
  if (v == 0) return 0.0;
  const unsigned long long sign = v < 0 ? (1ull << 63) : 0ull;
  unsigned long long u = v < 0 ? (unsigned long long)(-v) : (unsigned long long)v;
  const int nbits = 64 - __clzll((long long)u);  // significant bits
  int sh = nbits - 53;
  unsigned long long m;
  if (sh <= 0) {
    m = u << (-sh);
  } else {
    m = u >> sh;
    const unsigned long long rem = u & ((1ull << sh) - 1), half = 1ull << (sh - 1);
    if (rem > half || (rem == half && (m & 1ull))) ++m;
    if (m >> 53) {
      m >>= 1;
      ++sh;
    }
  }
  const long long E = 52 + sh + e2 + 1023;  // m in [2^52, 2^53)
  if (E >= 2047) return __longlong_as_double((long long)(sign | (0x7ffull << 52)));  // overflow: infinity
  if (E <= 0) {
    // subnormal or zero: m 2^(E - 1075) = (m >> (1 - E)) 2^-1074, rounded to
    // nearest even (a carry into bit 52 gives the smallest normal number)
    const int s2 = 1 - (int)E;
    if (s2 > 53) return __longlong_as_double((long long)sign);
    unsigned long long q = m >> s2;
    const unsigned long long rem = m & ((1ull << s2) - 1), half = 1ull << (s2 - 1);
    if (rem > half || (rem == half && (q & 1ull))) ++q;
    return __longlong_as_double((long long)(sign | q));
  }
  return __longlong_as_double((long long)(sign | ((unsigned long long)E << 52) | (m & ((1ull << 52) - 1))));
}

// (hi 2^16 + lo) 2^e2 as a double, rounded once to nearest even, |hi| < 2^60
// and |lo| < 2^40, without a branch and without the FP64 pipe (a conversion
// costs that pipe as much as an add): the sum is brought to 64 normalized bits
// with a sticky last one and rounded in integers.  slow: a sum of fewer than
// 17 bits or a result outside the normal range -- scaled_sum_slow then.
__device__ __forceinline__ double scaled_sum_rn(long long hi, long long lo, int e2, bool &slow) {
  hi += lo >> 16;                                  // floor: lo's low 16 bits stay non-negative
  unsigned long long w = (unsigned long long)(lo & 0xffff) << 48;  // bits below hi
  unsigned long long h = (unsigned long long)hi;
  const unsigned long long sign = h & (1ull << 63);
  const unsigned long long m0 = (unsigned long long)(hi >> 63);
  w = (w ^ m0) - m0;                               // two's complement of the pair when negative
  h = (h ^ m0) + (m0 && w == 0ull ? 1ull : 0ull);
  const int lz = __clzll((long long)(h | 1ull));   // >= 3
  unsigned long long n = (h << lz) | (w >> (64 - lz));
  n |= (w << lz) != 0ull;
  // n in [2^63, 2^64): value n 2^(e2 + 16 - lz), 53 bits kept
  const int E = 1023 + 63 + 16 - lz + e2;
  const bool zero = (h | w) == 0ull;
  slow = !zero && (h == 0ull || (unsigned)(E - 1) >= 2045u);
  unsigned long long m = n >> 11;
  const unsigned rem = (unsigned)n & 0x7ffu;
  m += (rem + (unsigned)(m & 1ull) > 0x400u) ? 1ull : 0ull;
  // a carry out of the 53 bits lands in the exponent
  return zero ? 0.0 : __longlong_as_double((long long)(sign | (((unsigned long long)(unsigned)(E - 1) << 52) + m)));
}

// hi 2^e2 by CUDA's correctly rounded conversion and an exponent add: cheaper
// where there are no low digits (4 digits, n = 4096: 149 against 151 us).
__device__ __forceinline__ double scaled_rn(long long hi, int e2, bool &slow) {
  const long long bits = __double_as_longlong(__ll2double_rn(hi));
  const int E = (int)((bits >> 52) & 0x7ff) + e2;
  slow = hi != 0 && (unsigned)(E - 1) >= 2046u;
  return hi == 0 ? 0.0 : __longlong_as_double(bits + ((long long)e2 << 52));
}

__device__ __noinline__ double scaled_sum_slow(long long hi, long long lo, int e2) {
  hi += lo >> 16;
  unsigned long long w = (unsigned long long)(lo & 0xffff) << 48, h = (unsigned long long)hi;
  const bool neg = hi < 0;
  if (neg) {
    w = 0ull - w;
    h = ~h + (w == 0ull);
  }
  double v;
  if (h == 0ull) {
    v = i64_scaled_to_double((long long)(w >> 48), e2);
  } else {
    const int lz = __clzll((long long)h);
    unsigned long long n = (h << lz) | (w >> (64 - lz));
    n |= (w << lz) != 0ull;
    v = i64_scaled_to_double((long long)(n >> 2) | (long long)((n & 3) != 0), e2 + 18 - lz);
  }
  return neg ? -v : v;
}

// Digits of x for the split: F = round(|x| 2^(8S - e)) (|x| < 2^e), as a
// signed integer with at most 8 S + 1 bits, from the FP64 bit pattern.
__device__ __forceinline__ long long fixed_point_digits(double x, int e, int S) {
  const unsigned long long bits = (unsigned long long)__double_as_longlong(x);
  const int E = (int)((bits >> 52) & 0x7ff);
  if (E == 0) return 0;  // zero or subnormal: below every digit
  const unsigned long long mant = (bits & ((1ull << 52) - 1)) | (1ull << 52);
  // |x| = mant 2^(E - 1075); F = mant 2^(E - 1075 + 8 S - e)
  const int sh = E - 1075 + 8 * S - e;
  unsigned long long F;
  if (sh >= 0) {
    F = mant << sh;  // |x| < 2^e keeps F < 2^(8S) <= 2^56
  } else if (sh > -64) {
    F = mant >> (-sh);
    const unsigned long long rem = mant & ((1ull << (-sh)) - 1), half = 1ull << (-sh - 1);
    if (rem > half || (rem == half && (F & 1ull))) ++F;
  } else {
    F = 0;
  }
  return (bits >> 63) ? -(long long)F : (long long)F;
}

constexpr int kTcBM = 128;
constexpr int kTcKpad = 64;                      // K is padded to a multiple of 64
constexpr long long kWaitLimit = 4000000000ll;   // ~2 s of SM clock
constexpr size_t kTcSmemBudget = 224 * 1024;
constexpr size_t kTcSmemHalf = 110 * 1024;  // per CTA when two share an SM

struct TcArgs {
  int kblocks, S, mpad, npad, bn;
  int bk, swz;   // K block (32 or 64 bf16) and its swizzle layout (4: 64 B, 2: 128 B)
  int exact;     // 1: one accumulator per digit diagonal (exact FP32 sums)
  int nstages;   // operand stages in shared memory (1 or 2)
  int tmem_cols;
  int nacc;      // TMEM accumulators (1, S, or 8 when the last of 7 diagonals is split)
  int nbatch;    // batch items (grid z)
  // valid rows / columns of item b: m_item[b] (or m, and m_last for the last item)
  int m, m_last, n, n_last;
  const int *m_item, *n_item;
  const int *ea, *eb;  // exponents, [item][mpad] and [item][npad]
  double *C;           // item b: C + b * sbc + coff[b], ld ldc
  int ldc;
  long long sbc;
  const int *coff;
  int sign;            // C -= sign * A B, sign = +1 or -1
  int *status;
  const int *skip;     // nonzero: a stage enqueued ahead that is not needed, do nothing
  int slices;          // operand slices per item: S digits, then the magnitudes when keep > 0
  float keep;          // TcGemm::keep
  int czero;           // TcGemm::czero
  unsigned *fp64;      // keep > 0: bit c of word [item][row / 32][column / 32]: these 32 rows of column c take FP64
  TcOperand A, B;
};

// Exponent mark of a vector that has no digits (TcGemm::keep).
constexpr int kExOdd = 1 << 20;

// Element (v, k) of item b of an operand, 0 outside its structure.
__device__ __forceinline__ double operand_at(const TcOperand &o, const double *X, int v, int k) {
  const int r = (o.trans ? k : v) + o.roff, q = o.trans ? v : k;
  if (o.shape == 0 || (o.shape == 1 && r > q) || (o.shape == 2 && r <= q))
    return X[(long long)v * o.sv + (long long)k * o.sk];
  return (o.shape == 1 && r == q) ? 1.0 : 0.0;
}
__device__ __forceinline__ const double *operand_item(const TcOperand &o, int b) {
  return o.X + (long long)b * o.sb + (o.off ? o.off[b] : 0);
}
__device__ __forceinline__ int operand_k(const TcOperand &o, int b, bool last) {
  return o.K_item ? o.K_item[b] : (last ? o.K_last : o.K);
}

// C -= sign A B in FP64 for the columns n0 + c, bit c of `cols`, of the rows
// r0 .. r0 + 31: what the digits cannot stand for.  A chain of multiply-adds
// over k, then one subtraction, as in gemm_fp64.cu (the same bits).  The whole
// CTA calls it; a warp takes every eighth column, a lane a row, so that the
// usual one or two columns cost one chain of K multiply-adds (64 clocks of the
// FP64 pipe each, 4 us) and not the 32 us of all 32 columns.  All of K is
// staged at once (sm: 2 x 128 x 33 doubles; K <= 128).
constexpr int kFpLd = 33;

__device__ __noinline__ void fp64_block(const TcArgs &a, int item, int r0, int n0, unsigned cols, int mv, int nvv,
                                        double *Cb, double *sm) {
  __shared__ int list[32];  // the columns
  const bool last = item == a.nbatch - 1;
  const int K = min(operand_k(a.A, item, last), operand_k(a.B, item, last));
  const double *X = operand_item(a.A, item), *Y = operand_item(a.B, item);
  double *As = sm, *Bs = sm + 128 * kFpLd;  // (k, row) and (k, place in the list)
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nf = __popc(cols);
  __syncthreads();  // the operands of an earlier call have been read
  if (tid < 32 && (cols >> tid & 1u)) list[__popc(cols & ((1u << tid) - 1u))] = tid;
  __syncthreads();
  // what A's structure leaves of k for these rows
  int klo = 0, khi = K;
  if (a.A.shape == 1) {
    if (a.A.trans)
      klo = max(0, r0 - a.A.roff);
    else
      khi = min(K, r0 + 32 + a.A.roff);
  } else if (a.A.shape == 2) {
    if (a.A.trans)
      khi = min(K, r0 + 32 - a.A.roff);
    else
      klo = max(0, r0 + a.A.roff);
  }
  const int kr = max(0, khi - klo);
#pragma unroll 8
  for (int e = tid; e < 32 * kr; e += 256) {  // along A's contiguous index
    const int v = a.A.sv == 1 ? e & 31 : e / kr, k = a.A.sv == 1 ? e >> 5 : e % kr;
    As[k * kFpLd + v] = r0 + v < mv ? operand_at(a.A, X, r0 + v, klo + k) : 0.0;
  }
#pragma unroll 4
  for (int e = tid; e < nf * kr; e += 256) {
    const int v = e / kr, k = e % kr, c = n0 + list[v];
    Bs[k * kFpLd + v] = c < nvv ? operand_at(a.B, Y, c, klo + k) : 0.0;
  }
  __syncthreads();
  const int nv = (nf - warp + 7) / 8;  // this warp's columns
  double acc[4] = {0.0, 0.0, 0.0, 0.0};
  for (int k = 0; k < kr; ++k) {
    const double x = As[k * kFpLd + lane];
#pragma unroll
    for (int v = 0; v < 4; ++v) {
      if (v >= nv) break;
      acc[v] = fma(x, Bs[k * kFpLd + warp + 8 * v], acc[v]);
    }
  }
#pragma unroll
  for (int v = 0; v < 4; ++v) {
    if (v >= nv) break;
    const int c = n0 + list[warp + 8 * v];
    if (r0 + lane >= mv || c >= nvv) continue;
    double *p = Cb + r0 + lane + (size_t)c * a.ldc;
    *p = a.sign > 0 ? *p - acc[v] : *p + acc[v];
  }
}

__device__ __forceinline__ unsigned *fp64_word_at(const TcArgs &a, int item, int mtile, int quad, int n0) {
  return a.fp64 + (((size_t)item * (a.mpad / kTcBM) + mtile) * 4 + quad) * (a.npad / 32) + n0 / 32;
}
__device__ __forceinline__ unsigned fp64_word(const TcArgs &a, int item, int mtile, int quad, int n0) {
  return a.keep > 0.0f ? *fp64_word_at(a, item, mtile, quad, n0) : 0u;
}

// Operand tiles for one K block: S boxes of A digits (128 x bk) then S boxes
// of B digits (bn x bk).
__host__ __device__ inline size_t tc_stage_bytes(int S, int bn, int bk) {
  return (size_t)S * (kTcBM + bn) * bk * 2;
}

__global__ void __launch_bounds__(256, 2)
    tc_gemm_kernel(const __grid_constant__ CUtensorMap mapA, const __grid_constant__ CUtensorMap mapB,
                   const __grid_constant__ TcArgs a) {
  extern __shared__ uint8_t smem_raw[];
  if (a.skip && *a.skip) return;  // before any barrier, copy or tensor-memory allocation
  uint8_t *base = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  const size_t stage_bytes = tc_stage_bytes(a.S, a.bn, a.bk);
  const int boxA = kTcBM * a.bk * 2;
  const int boxB = a.bn * a.bk * 2;
  uint64_t *full = (uint64_t *)(base + (size_t)a.nstages * stage_bytes);  // [2]
  uint64_t *empty = full + 2;                                            // [2]
  uint64_t *done = empty + 2;                                            // [1]
  uint32_t *tslot = (uint32_t *)(done + 1);
  volatile int *abort_flag = (volatile int *)(tslot + 1);
  const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;  // uniform
  const int m0 = blockIdx.x * kTcBM, n0 = blockIdx.y * a.bn;
  const int item = blockIdx.z;
  const bool last = item == a.nbatch - 1;
  const int mv = a.m_item ? a.m_item[item] : (last ? a.m_last : a.m);
  const int nvv = a.n_item ? a.n_item[item] : (last ? a.n_last : a.n);
  if (m0 >= mv || n0 >= nvv) return;  // an empty tile of a short batch item (uniform per CTA)
  __shared__ unsigned other_of[4];    // per 32 rows: the columns left to fp64_block
  if (threadIdx.x < 4) other_of[threadIdx.x] = fp64_word(a, item, blockIdx.x, threadIdx.x, n0);

  if (threadIdx.x == 0) {
    for (int i = 0; i < 2; ++i) {
      mbar_init(&full[i], 1);
      mbar_init(&empty[i], 1);
    }
    mbar_init(done, 1);
    *abort_flag = 0;
    fence_mbar_init();
  }
  if (warp == 0) {
    tmem_alloc(tslot, (uint32_t)a.tmem_cols);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tslot;
  int issued0 = 0, issued1 = 0;  // loads issued into stage 0 / 1

  if (warp == 0 && elect_one()) {
    // ---- producer: TMA loads of the digit tiles, one K block per stage ----
    for (int kb = 0; kb < a.kblocks; ++kb) {
      const int st = kb % a.nstages, round = kb / a.nstages;
      if (round > 0 && !mbar_wait(&empty[st], (round - 1) & 1, kWaitLimit)) {
        *abort_flag = 1;
        atomicOr(a.status, 2);
        break;
      }
      if (*abort_flag) break;
      uint8_t *sa = base + (size_t)st * stage_bytes;
      uint8_t *sb = sa + (size_t)a.S * boxA;
      mbar_expect_tx(&full[st], (uint32_t)stage_bytes);
      for (int s = 0; s < a.S; ++s) {
        tma_load_2d(sa + (size_t)s * boxA, &mapA, &full[st], kb * a.bk, (item * a.slices + s) * a.mpad + m0);
        tma_load_2d(sb + (size_t)s * boxB, &mapB, &full[st], kb * a.bk, (item * a.slices + s) * a.npad + n0);
      }
      if (st == 0)
        ++issued0;
      else
        ++issued1;
    }
  } else if (warp == 1 && elect_one()) {
    // ---- MMA issuer: digit products d_k d'_l with k + l <= S + 1 ----------
    // One thread issues, so the MMAs' count matters as much as their size: a
    // product of its own for each pair of digits (28 of 128 x 32 x 16 per K
    // step with 7 digits) took 121 clocks each; now S wide ones cover it.
    // n = 4096, K = 128: 7 digits 348 -> 268 us (448 TFLOP/s),
    // 5 digits 231 -> 190, 4 digits 143 -> 133.
    const uint32_t stepA = (uint32_t)boxA >> 4, stepB = (uint32_t)boxB >> 4;
    const int S = a.S, kst = a.bk / 16;
    const int khalf0 = (64 + a.bk - 1) / a.bk;  // first K block of the second 64-wide half
    const int wide = max(1, 256 / a.bn);        // digits of B that one MMA takes
    for (int kb = 0; kb < a.kblocks; ++kb) {
      const int st = kb % a.nstages;
      if (!mbar_wait(&full[st], (kb / a.nstages) & 1, kWaitLimit)) {
        *abort_flag = 1;
        atomicOr(a.status, 4);
        break;
      }
      tc_fence_after();
      const uint8_t *sa = base + (size_t)st * stage_bytes;
      const uint64_t ad0 = sw_desc(smem_u32(sa), a.swz);
      const uint64_t bd0 = sw_desc(smem_u32(sa + (size_t)S * boxA), a.swz);
      if (a.exact) {
        // Product d_ka d'_kq goes to the accumulator of its diagonal ka + kq.
        // The digits of B lie one after the other in shared memory and the
        // accumulators in tensor memory, so one MMA multiplies d_ka by as many
        // of B's digits as 256 columns hold.  With 7 digits over two halves of
        // K the last diagonal (7 products) has one accumulator per half, to
        // stay below 2^24: its product is issued alone in the second half.
        const bool second = a.nacc == 8 && kb >= khalf0;
        for (int ks = 0; ks < kst; ++ks) {  // +32 bytes of K per step
          uint64_t ad = ad0 + 2 * ks;
          for (int ka = 0; ka < S; ++ka) {
            const int nq = S - ka - (second ? 1 : 0);  // products in their own diagonal's accumulator
            const uint32_t more = kb > 0 || ka > 0 || ks > 0;  // 0: the accumulators hold nothing yet
            for (int kq = 0; kq < nq; kq += wide) {
              const int w = min(wide, nq - kq) * a.bn;
              tc_mma(tmem + (uint32_t)((ka + kq) * a.bn), ad, bd0 + (uint64_t)(kq * stepB + 2 * ks),
                     idesc_bf16_f32(kTcBM, w), more);
            }
            if (second)
              tc_mma(tmem + (uint32_t)(7 * a.bn), ad, bd0 + (uint64_t)(nq * stepB + 2 * ks),
                     idesc_bf16_f32(kTcBM, a.bn), kb > khalf0 || ka > 0 || ks > 0);
            ad += stepA;
          }
        }
      } else {
        const uint32_t idesc = idesc_bf16_f32(kTcBM, a.bn);
        uint64_t ad = ad0;
        for (int ka = 0; ka < S; ++ka) {
          uint64_t bd = bd0;
          for (int kq = 0; ka + kq < S; ++kq) {
            for (int ks = 0; ks < kst; ++ks)
              tc_mma(tmem, ad + 2 * ks, bd + 2 * ks, idesc, kb > 0 || ka > 0 || kq > 0 || ks > 0);
            bd += stepB;
          }
          ad += stepA;
        }
      }
      tc_commit(&empty[st]);  // the stage may be refilled once these MMAs are done
    }
    tc_commit(done);
  }
  __syncthreads();
  // ---- epilogue: C -= 2^(e_i + f_j - 16) sum_d 2^(-8 d) acc_d -------------
  bool ok = mbar_wait(done, 0, kWaitLimit) && (*abort_flag == 0);
  if (!ok && lane == 0) atomicOr(a.status, 8);
  tc_fence_after();
  const int nacc = a.nacc;
  if (ok) {
    // 8 warps: warp w reads TMEM lanes 32 (w % 4) .. + 31, column chunks
    // alternate between warps w and w + 4
    const int quad = warp & 3, half = warp >> 2;
    const int row = m0 + 32 * quad + lane;
    const bool rin = row < mv;
    const int er = rin ? a.ea[(size_t)item * a.mpad + row] : 0;
    const int *ebi = a.eb + (size_t)item * a.npad;
    double *Cb = a.C + (size_t)item * a.sbc + (a.coff ? a.coff[item] : 0);
    const unsigned other = other_of[quad];
    // exact mode: the digit diagonals D = 0 .. S-1 (weights 2^(-8 D)) are
    // integers below 2^24; combine them in integer arithmetic,
    //   T_hi = sum_{D <= 4} acc_D 2^(8 (4 - D)),  T_lo = sum_{D > 4} acc_D 2^(8 (6 - D)),
    // and round their sum to a double once.
    // Four columns per step; the next step's C and exponents are on their way
    // while this step's accumulators, all read at once, are combined.
    constexpr int kEp = 4;
    double cn[kEp];
    int en[kEp];
    auto fetch = [&](int c0) {
#pragma unroll
      for (int j = 0; j < kEp; ++j) {
        const int col = n0 + c0 + j;
        const bool ok_c = rin && c0 < a.bn && col < nvv;
        cn[j] = ok_c ? __ldcg(Cb + row + (size_t)col * a.ldc) : 0.0;
        en[j] = ok_c ? __ldg(ebi + col) : 0;
      }
    };
    fetch(half * kEp);
    for (int c0 = half * kEp; c0 < a.bn; c0 += 2 * kEp) {
      uint32_t r[8][kEp];
#pragma unroll
      for (int d = 0; d < 8; ++d) {
        r[d][0] = r[d][1] = r[d][2] = r[d][3] = 0u;
        if (d < nacc) tmem_ld_32x4(tmem + ((uint32_t)(32 * quad) << 16) + (uint32_t)(d * a.bn + c0), r[d]);
      }
      double cv[kEp];
      int ec[kEp];
#pragma unroll
      for (int j = 0; j < kEp; ++j) {
        cv[j] = cn[j];
        ec[j] = en[j];
      }
      fetch(c0 + 2 * kEp);
      tmem_ld_wait(r);
      // straight-line for all columns of the step (a branch per element would
      // run their long dependent chains one after the other)
      unsigned slow = 0;
      long long hi[kEp], lo[kEp];
#pragma unroll
      for (int j = 0; j < kEp; ++j) {
        const int sc = er + ec[j] - 16;  // C -= sign 2^sc value
        hi[j] = lo[j] = 0;
        if (a.exact) {
          // sum_D acc_D 2^(-8 D) = T_hi 2^(-32) + T_lo 2^(-48)
#pragma unroll
          for (int d = 0; d < 8; ++d) {
            const int q = a.sign * __float2int_rn(__uint_as_float(r[d][j]));  // 0 beyond the accumulators
            const int D = d < 7 ? d : 6;  // accumulator 7 is the second half of diagonal 6
            if (D <= 4)
              hi[j] = D == 0 ? (long long)q << 32 : mad_wide(q, 1 << (8 * (4 - D)), hi[j]);
            else
              lo[j] = mad_wide(q, 1 << (8 * (6 - D)), lo[j]);
          }
          bool sl;
          cv[j] -= nacc > 5 ? scaled_sum_rn(hi[j], lo[j], sc - 48, sl) : scaled_rn(hi[j], sc - 32, sl);
          slow |= sl ? 1u << j : 0u;
        } else {
          cv[j] = fma((double)(-a.sign * __uint_as_float(r[0][j])), pow2i(sc), cv[j]);
        }
      }
      if (slow) {
#pragma unroll
        for (int j = 0; j < kEp; ++j) {
          const int col = n0 + c0 + j;
          if (!((slow >> j) & 1u) || !rin || col >= nvv) continue;
          const int sc = er + ec[j] - 16;
          const double c = __ldcg(Cb + row + (size_t)col * a.ldc);
          cv[j] = c - scaled_sum_slow(hi[j], lo[j], sc - 48);
        }
      }
#pragma unroll
      for (int j = 0; j < kEp; ++j) {
        const int col = n0 + c0 + j;
        if (rin && col < nvv && !((other >> (c0 + j)) & 1u)) Cb[row + (size_t)col * a.ldc] = cv[j];
      }
    }
  }
  // every copy this CTA issued has landed before shared memory goes away
  // (the counts are the producer's)
  if (issued0 + issued1 > 0) {
    if (issued0 > 0) mbar_wait(&full[0], (issued0 - 1) & 1, kWaitLimit);
    if (issued1 > 0) mbar_wait(&full[1], (issued1 - 1) & 1, kWaitLimit);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) tmem_dealloc(tmem, (uint32_t)a.tmem_cols);
  // (the operand stages are free: every copy has landed, every MMA is done)
  for (int q = 0; q < 4; ++q)
    if (other_of[q])
      fp64_block(a, item, m0 + 32 * q, n0, other_of[q], mv, nvv,
                 a.C + (size_t)item * a.sbc + (a.coff ? a.coff[item] : 0), reinterpret_cast<double *>(base));
}

// --------------------------------------------------------------------------
// Where the digits may stand in for FP64 (TcGemm::keep).  The digits hold an
// operand to 2^-57 of its vector's 2^e > max, so an element's error is up to
// 2.5 K 2^-56 2^(e_i + f_j) (representation 2 K 2^-57, dropped products k + l
// >= 9 6 K 2^-58) however small the element is, while FP64 multiply-adds have
// the bound K 2^-53 (|C_ij| + sum_k |a_ik| |b_kj|).  The first is below the
// second where
//   |C_ij| + sum_k |a_ik| |b_kj| >= keep 2^(e_i + f_j),  keep = 2.5 / 8.
// This kernel checks that for every element: one bf16 MMA product of the
// operands' magnitudes (rounded down, relative to 2^e; a nonzero one is at
// least 2^-40) per 128 x 128 tile, C only where the sum alone does not reach
// keep.  A sum of zero means that every product is zero: no error.  Columns
// with an element that fails take FP64 in the 32 rows that hold it, which
// depends on nothing but those rows and that column: the result does not
// change with the way a matrix is cut into calls.  Non-finite vectors and
// those with values near the ends of the range (kExOdd) take it too.
// Bound by the chain load - MMA - read of a CTA, about 3 us: 2016 CTAs take 28
// us where the digits' split takes 300 and their product 540 (16 leaves, K =
// 128, 16128 columns); 127 us where most elements have to look at C.  The
// first form compared in FP64 and took four times as long.  With the FP64
// blocks: CALU + solve of n = 10240 113.3 -> 113.9 ms (no element fails),
// CAQR + solve of n = 6144 128.3 -> 131.6, CAQR of n = 16384 887 -> 906.
// --------------------------------------------------------------------------
constexpr int kChkN = 128;

__global__ void __launch_bounds__(256, 3)
    tc_check_kernel(const __grid_constant__ CUtensorMap mapA, const __grid_constant__ CUtensorMap mapB,
                    const __grid_constant__ TcArgs a) {
  extern __shared__ uint8_t smem_raw[];
  if (a.skip && *a.skip) return;
  uint8_t *base = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  __shared__ uint64_t bars[3];  // [0], [1]: a 64-wide half of K has arrived; [2]: the MMAs are done
  __shared__ uint32_t tslot;
  const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
  const int m0 = blockIdx.x * kTcBM, n0 = blockIdx.y * kChkN;
  const int item = blockIdx.z;
  const bool last = item == a.nbatch - 1;
  const int mv = a.m_item ? a.m_item[item] : (last ? a.m_last : a.m);
  const int nvv = a.n_item ? a.n_item[item] : (last ? a.n_last : a.n);
  if (m0 >= mv || n0 >= nvv) return;
  constexpr int boxA = kTcBM * 64 * 2, boxB = kChkN * 64 * 2;
  if (threadIdx.x == 0) {
    for (int i = 0; i < 3; ++i) mbar_init(&bars[i], 1);
    fence_mbar_init();
  }
  if (warp == 0) {
    tmem_alloc(&tslot, kChkN);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tslot;
  if (warp == 0 && elect_one()) {
    for (int kb = 0; kb < a.kblocks; ++kb) {  // at most two: all of K is resident
      uint8_t *sa = base + kb * (boxA + boxB);
      mbar_expect_tx(&bars[kb], boxA + boxB);
      tma_load_2d(sa, &mapA, &bars[kb], kb * 64, (item * a.slices + a.S) * a.mpad + m0);
      tma_load_2d(sa + boxA, &mapB, &bars[kb], kb * 64, (item * a.slices + a.S) * a.npad + n0);
    }
  } else if (warp == 1 && elect_one()) {
    for (int kb = 0; kb < a.kblocks; ++kb) {
      if (!mbar_wait(&bars[kb], 0, kWaitLimit)) {
        atomicOr(a.status, 4);
        break;
      }
      tc_fence_after();
      const uint8_t *sa = base + kb * (boxA + boxB);
      const uint64_t ad = sw_desc(smem_u32(sa), 2), bd = sw_desc(smem_u32(sa + boxA), 2);
      for (int ks = 0; ks < 4; ++ks)
        tc_mma(tmem, ad + 2 * ks, bd + 2 * ks, idesc_bf16_f32(kTcBM, kChkN), kb > 0 || ks > 0);
    }
    tc_commit(&bars[2]);
  }
  __syncthreads();
  bool ok = mbar_wait(&bars[2], 0, kWaitLimit);
  for (int kb = 0; kb < a.kblocks; ++kb) ok &= mbar_wait(&bars[kb], 0, kWaitLimit);  // its copies have landed
  if (!ok && lane == 0) atomicOr(a.status, 8);
  tc_fence_after();
  const int quad = warp & 3, half = warp >> 2;
  const int row = m0 + 32 * quad + lane;
  const bool rin = row < mv;
  const int er = rin ? a.ea[(size_t)item * a.mpad + row] : 0;
  const double *Cb = a.C + (size_t)item * a.sbc + (a.coff ? a.coff[item] : 0);
  for (int c0 = half * 64; c0 < half * 64 + 64 && n0 + c0 < nvv; c0 += 32) {
    uint32_t r[32];
    tmem_ld_32x32(tmem + ((uint32_t)(32 * quad) << 16) + (uint32_t)c0, r);
    const int mycol = n0 + c0 + lane;
    const int myec = mycol < nvv ? a.eb[(size_t)item * a.npad + mycol] : 0;
    unsigned fail = __ballot_sync(0xffffffffu, myec > kExOdd / 2);
    if (er > kExOdd / 2 || !ok) fail = 0xffffffffu;
    // FP32 and integers only: an FP64 instruction would hold the pipe for 64
    // clocks, and most of them for nothing
    unsigned low = 0;
#pragma unroll
    for (int c = 0; c < 32; ++c) {
      const float v = __uint_as_float(r[c]);
      low |= (v < a.keep && v != 0.0f) ? 1u << c : 0u;
    }
    low = rin ? low & ~fail : 0u;  // (padding columns have no magnitudes)
    if (a.czero) {  // no C to add
      fail |= low;
    } else if (__any_sync(0xffffffffu, low != 0u)) {
      constexpr int kAt = 16;  // loads of C in flight
#pragma unroll
      for (int c1 = 0; c1 < 32; c1 += kAt) {
        if (!__any_sync(0xffffffffu, (low >> c1 & 0xffffu) != 0u)) continue;
        unsigned long long cb[kAt];
#pragma unroll
        for (int j = 0; j < kAt; ++j)
          cb[j] = (low >> (c1 + j) & 1u) ? absbits(Cb[row + (size_t)(n0 + c0 + c1 + j) * a.ldc]) : 0ull;
#pragma unroll
        for (int j = 0; j < kAt; ++j) {
          const int ec = __shfl_sync(0xffffffffu, myec, c1 + j);
          // |C| 2^-(e_i + f_j) rounded down to a float's bits
          const int E = (int)(cb[j] >> 52), ef = E - 1023 + 127 - er - ec;
          const float f = E == 0 || ef <= 0 ? 0.0f
                          : ef >= 254      ? 1e38f
                                           : __uint_as_float(((unsigned)ef << 23) | (unsigned)(cb[j] >> 29 & 0x7fffffull));
          if ((low >> (c1 + j) & 1u) && (E == 0x7ff || !(__uint_as_float(r[c1 + j]) + f >= a.keep))) fail |= 1u << (c1 + j);
        }
      }
    }
    fail = __reduce_or_sync(0xffffffffu, rin ? fail : 0u);
    if (lane == 0) *fp64_word_at(a, item, blockIdx.x, quad, n0 + c0) = fail;
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) tmem_dealloc(tmem, kChkN);
}

// --------------------------------------------------------------------------
// split: the vectors of an operand (rows of A, columns of B) -> S bf16 digit
// slices, one warp per vector, K <= 256.  Item b, vector v, position k reads
// element (v, k) of the source: X[b * sb + off[b] + v * sv + k * sk], through
// the structure rule on (r, q) = (row, column) of the source:
// shape 0 dense, 1 unit lower (r > q stored, r == q is one, r < q zero),
// 2 upper (r <= q stored); (r, q) = (v + roff, k) or, transposed, (k + roff, v).
// Output: out[((b * slices + s) * vpad + v) * kpad + k], exponent ex[b * vpad + v];
// slices = S, with KEEP one more: the magnitudes |x| 2^-e rounded down.
// --------------------------------------------------------------------------
// One launch splits both operands: blocks from nblkA on work on B.
struct SplitSide {
  TcOperand o;
  int vpad;
  __nv_bfloat16 *out;
  int *ex;
  int ksign;           // KEEP: kexp is taken with this sign
};

template <bool KEEP, int S>
__global__ void __launch_bounds__(256, KEEP ? 4 : 1)
    split_kernel(const __grid_constant__ SplitSide sideA, const __grid_constant__ SplitSide sideB, int nblkA, int nbatch,
                 int kpad, int exact, const int *skip, const int *kexp) {
  if (skip && *skip) return;
  const bool second = (int)blockIdx.x >= nblkA;
  const SplitSide &d = second ? sideB : sideA;
  const TcOperand &o = d.o;
  const int vpad = d.vpad, ksign = d.ksign;
  __nv_bfloat16 *__restrict__ out = d.out;
  int *__restrict__ ex = d.ex;
  const int lane = threadIdx.x & 31;
  const int v = ((int)blockIdx.x - (second ? nblkA : 0)) * 8 + (threadIdx.x >> 5);
  const int b = blockIdx.y;
  if (v >= vpad) return;
  const bool last = b == nbatch - 1;
  const int nv = o.nv_item ? o.nv_item[b] : (last ? o.nv_last : o.nv);
  const int K = operand_k(o, b, last);
  const double *X = operand_item(o, b);
  constexpr int kPer = KEEP ? 4 : 8;  // K <= 128 (exact sums), 256
  constexpr int kSlices = S + (KEEP ? 1 : 0);
  double x[kPer];
  int sh[kPer];            // the element is taken times 2^sh
  unsigned long long mx = 0;
  int me = INT_MIN;        // largest exponent field + sh of a nonzero element
  unsigned odd = 0;
#pragma unroll
  for (int t = 0; t < kPer; ++t) {
    const int k = lane + 32 * t;
    double val = 0.0;
    if (v < nv && k < K) val = operand_at(o, X, v, k);
    x[t] = val;
    sh[t] = 0;
    if constexpr (KEEP) {
      const int E = (int)(__double2hiint(val) >> 20) & 0x7ff;
      const bool some = absbits(val) != 0ull;
      if (kexp && k < K) sh[t] = ksign * kexp[k];
      if (some) me = max(me, E + sh[t]);
      odd |= some && (unsigned)(E - 1) >= 0x7feu;  // not finite, or subnormal (the digits drop those)
    } else {
      const unsigned long long bits = absbits(val);
      mx = bits > mx ? bits : mx;
    }
  }
  int e = 0;  // |x| < 2^e, from the exponent field of the largest magnitude
  if constexpr (KEEP) {
    me = __reduce_max_sync(0xffffffffu, me);
    odd = __reduce_or_sync(0xffffffffu, odd);
    if (me != INT_MIN) {
      e = me - 1022;
      if (odd || e < -900 || e > 1000) {  // no digits: FP64
        e = kExOdd;
#pragma unroll
        for (int t = 0; t < kPer; ++t) x[t] = 0.0;
      }
    }
  } else {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
      const unsigned long long ot = __shfl_xor_sync(0xffffffffu, mx, off);
      mx = ot > mx ? ot : mx;
    }
    if (mx != 0) {
      const int E = (int)(mx >> 52);
      e = (E == 0) ? -1021 : E - 1022;
    }
  }
  if (lane == 0) ex[(long long)b * vpad + v] = e;
#pragma unroll
  for (int t = 0; t < kPer; ++t) {
    const int k = lane + 32 * t;
    if (k >= kpad) continue;
    // F = round(x 2^(8S - e)) = sum_s d_s 256^(S-1-s), balanced digits
    // d_s in [-128, 127] for s >= 1 and |d_0| <= 256: with 128 added at every
    // lower digit's place, the bytes of F are d_s + 128 and what is above them
    // is d_0.  A byte becomes a float by putting it into the mantissa of 2^23
    // (no conversion instruction).
    constexpr unsigned long long bias = 0x0080808080808080ull & ((1ull << (8 * (S - 1))) - 1);
    const unsigned long long F = (unsigned long long)fixed_point_digits(x[t], KEEP ? e - sh[t] : e, S) + bias;
#pragma unroll
    for (int s = 0; s < S; ++s) {
      const int sft = 8 * (S - 1 - s);
      const float d = s == 0 ? (float)(int)((long long)F >> sft)
                             : __uint_as_float(0x4b000000u | (unsigned)((F >> sft) & 255u)) - (8388608.0f + 128.0f);
      // stored value: d_s (exact mode) or d_s 2^(-8 s) (fused mode), exact in bf16
      // 2^(-8 s) as a float from its exponent field (s <= 7: a normal number)
      const float w = exact ? 1.0f : __int_as_float((127 - 8 * s) << 23);
      out[(((long long)b * kSlices + s) * vpad + v) * kpad + k] = __float2bfloat16_rn(d * w);
    }
    if constexpr (KEEP) {
      // exponent field and the first 7 bits of the mantissa, the exponent
      // moved from the double's bias to the bfloat's and by sh - e
      const int m = ((__double2hiint(x[t]) & 0x7fffffff) >> 13) + (sh[t] - e - (1023 - 127)) * 128;
      const unsigned mag = absbits(x[t]) == 0ull ? 0u : (unsigned)max(m, (127 - 40) * 128);
      out[(((long long)b * kSlices + S) * vpad + v) * kpad + k] = __ushort_as_bfloat16((unsigned short)mag);
    }
  }
}

// --------------------------------------------------------------------------
// host side
// --------------------------------------------------------------------------
static inline int rup(int x, int q) { return (x + q - 1) / q * q; }

typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                   const cuuint64_t *, const cuuint32_t *, const cuuint32_t *,
                                   CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion,
                                   CUtensorMapFloatOOBfill);

static EncodeTiledFn encode_fn() {
  static EncodeTiledFn fn = nullptr;
  static bool tried = false;
  if (!tried) {
    tried = true;
    void *p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
            cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = (EncodeTiledFn)p;
  }
  return fn;
}

static bool make_map(CUtensorMap *map, void *base, int kpad, int rows, int box_rows, int bk) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return false;
  cuuint64_t dims[2] = {(cuuint64_t)kpad, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)kpad * 2};
  cuuint32_t box[2] = {(cuuint32_t)bk, (cuuint32_t)box_rows};
  cuuint32_t estr[2] = {1, 1};
  return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, base, dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, bk == 64 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B,
            CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Accumulators: one (fused), one per digit diagonal (exact), and with 7
// digits over K > 64 the 7-product diagonal gets one per 64-wide half of K.
static int tc_nacc(int S, int exact, int kpad) {
  return exact ? ((S == 7 && kpad > 64) ? 8 : S) : 1;
}

static int pow2_at_least(int x) {
  int p = 32;
  while (p < x) p *= 2;
  return p;
}

struct TcCfg {
  int bn, bk, swz, nstages, tmem_cols;
  size_t smem;
};

// Tile width, K block and stages.  First choice: two CTAs of 8 warps per
// SM (each with at most 256 tensor-memory columns and half the shared
// memory), so that one CTA's epilogue -- the FP64 read-modify-write of its C
// tile -- overlaps the other's loads and MMAs; tiles at least 32 wide (5
// digits, n = 4096: 231 us with two CTAs of 32-wide tiles, 268 with one of 64;
// 7 digits 342 and 346; both with one MMA per pair of digits).
// Otherwise one CTA per SM: the widest tile whose accumulators fit in the
// 512 columns.  Then the deepest K-block pipeline that fits in shared memory
// (two stages overlap the loads of one K block with the MMAs of the
// previous one).
static bool tc_config(int S, int exact, int kpad, TcCfg &c) {
  const int nacc = tc_nacc(S, exact, kpad);
  {
    int bn2 = 128;
    while (bn2 > 32 && nacc * bn2 > 256) bn2 /= 2;
    if (nacc * bn2 <= 256) {
      const int opts2[3][2] = {{64, 2}, {32, 2}, {32, 1}};
      for (auto &o : opts2) {
        const int bk = o[0];
        int ns = o[1];
        const int kblocks = kpad / bk;
        if (ns > kblocks) ns = kblocks;
        const size_t smem = ns * tc_stage_bytes(S, bn2, bk) + 1024 + 256;
        if (smem <= kTcSmemHalf) {
          c = {bn2, bk, bk == 64 ? 2 : 4, ns, pow2_at_least(nacc * bn2), smem};
          return true;
        }
      }
    }
  }
  int bn = 128;
  while (bn > 32 && nacc * bn > 512) bn /= 2;
  if (nacc * bn > 512) return false;
  const int opts[4][2] = {{64, 2}, {32, 2}, {64, 1}, {32, 1}};
  for (auto &o : opts) {
    const int bk = o[0];
    int ns = o[1];
    const int kblocks = kpad / bk;
    if (ns > kblocks) ns = kblocks;
    const size_t smem = ns * tc_stage_bytes(S, bn, bk) + 1024 + 256;
    if (smem <= kTcSmemBudget) {
      c = {bn, bk, bk == 64 ? 2 : 4, ns, pow2_at_least(nacc * bn), smem};
      return true;
    }
  }
  return false;
}

size_t tc_gemm_ws_bytes_batched(int m, int n, int k, int S, int nbatch, bool keep) {
  const size_t mp = rup(m > 0 ? m : 1, kTcBM), np = rup(n > 0 ? n : 1, 128), kp = rup(k > 0 ? k : 1, kTcKpad);
  const size_t nb = nbatch > 0 ? nbatch : 1;
  const size_t ns = S + (keep ? 1 : 0);
  return align256(nb * ns * mp * kp * 2) + align256(nb * ns * np * kp * 2) + align256(nb * mp * 4) +
         align256(nb * np * 4) + (keep ? align256(nb * (mp / 32) * (np / 32) * 4) : 0) + 256;
}

size_t tc_gemm_ws_bytes(int m, int n, int k, int S) { return tc_gemm_ws_bytes_batched(m, n, k, S, 1); }

bool tc_gemm_supported(int k, int S, int exact) {
  if (k < 1 || k > 256 || S < 1 || S > 8) return false;
  if (exact && (S > 7 || k > 128)) return false;
  TcCfg c;
  return tc_config(S, exact, rup(k, kTcKpad), c);
}

cudaError_t gemm_tc(const TcGemm &g, void *ws, int *status, cudaStream_t st) {
  const int m = g.A.nv, n = g.B.nv, k = g.A.K > g.A.K_last ? g.A.K : g.A.K_last;
  if (m <= 0 || n <= 0 || k <= 0 || g.nbatch <= 0) return cudaSuccess;
  if (!tc_gemm_supported(k, g.S, g.exact)) return cudaErrorInvalidValue;
  const int S = g.S, exact = g.exact;
  const int mp = rup(m, kTcBM), np = rup(n, 128), kp = rup(k, kTcKpad);
  TcCfg cfg;
  if (!tc_config(S, exact, kp, cfg)) return cudaErrorInvalidValue;
  const int bn = cfg.bn;
  const bool keep = g.keep > 0.0f;
  if (keep && (bn != 32 || !exact || S != kTcF64Slices)) return cudaErrorInvalidValue;  // one word of columns per tile
  const size_t nb = g.nbatch, ns = S + (keep ? 1 : 0);
  char *p = (char *)(((uintptr_t)ws + 255) & ~(uintptr_t)255);
  __nv_bfloat16 *sa = (__nv_bfloat16 *)p;
  p += align256(nb * ns * mp * kp * 2);
  int *ea = (int *)p;
  p += align256(nb * mp * 4);
  __nv_bfloat16 *sb = (__nv_bfloat16 *)p;
  p += align256(nb * ns * np * kp * 2);
  int *eb = (int *)p;
  p += align256(nb * np * 4);
  {
    ProfScope ps(kClsSplit, st, 0.0);
    const SplitSide A = {g.A, mp, sa, ea, -1}, B = {g.B, np, sb, eb, 1};
    const int nblkA = g.reuse_a ? 0 : (mp + 7) / 8;
    const dim3 grid(nblkA + (np + 7) / 8, g.nbatch);
    auto run = [&](auto slices) {
      constexpr int kS = decltype(slices)::value;
      if (!keep)
        split_kernel<false, kS><<<grid, 256, 0, st>>>(A, B, nblkA, g.nbatch, kp, exact, g.skip, nullptr);
      else if constexpr (kS == kTcF64Slices)
        split_kernel<true, kS><<<grid, 256, 0, st>>>(A, B, nblkA, g.nbatch, kp, exact, g.skip, g.kexp);
    };
    switch (S) {
      case 1: run(std::integral_constant<int, 1>()); break;
      case 2: run(std::integral_constant<int, 2>()); break;
      case 3: run(std::integral_constant<int, 3>()); break;
      case 4: run(std::integral_constant<int, 4>()); break;
      case 5: run(std::integral_constant<int, 5>()); break;
      case 6: run(std::integral_constant<int, 6>()); break;
      case 7: run(std::integral_constant<int, 7>()); break;
      default: run(std::integral_constant<int, 8>()); break;
    }
  }
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  CUtensorMap ma, mb;
  if (!make_map(&ma, sa, kp, (int)(nb * ns * mp), kTcBM, cfg.bk) ||
      !make_map(&mb, sb, kp, (int)(nb * ns * np), bn, cfg.bk))
    return cudaErrorInvalidValue;
  TcArgs a;
  a.kblocks = kp / cfg.bk;
  a.S = S;
  a.mpad = mp;
  a.npad = np;
  a.bn = bn;
  a.bk = cfg.bk;
  a.swz = cfg.swz;
  a.exact = exact;
  a.nstages = cfg.nstages;
  a.nacc = tc_nacc(S, exact, kp);
  a.tmem_cols = cfg.tmem_cols;
  a.nbatch = g.nbatch;
  a.m = g.A.nv;
  a.m_last = g.A.nv_last;
  a.n = g.B.nv;
  a.n_last = g.B.nv_last;
  a.m_item = g.A.nv_item;
  a.n_item = g.B.nv_item;
  a.ea = ea;
  a.eb = eb;
  a.C = g.C;
  a.ldc = g.ldc;
  a.sbc = g.sbc;
  a.coff = g.coff;
  a.sign = g.sign > 0 ? 1 : -1;
  a.status = status;
  a.skip = g.skip;
  a.slices = (int)ns;
  a.keep = g.keep;
  a.czero = g.czero;
  a.fp64 = (unsigned *)p;
  a.A = g.A;
  a.B = g.B;
  const size_t smem = cfg.smem;
  static std::atomic<unsigned long long> init{0};
  e = once_per_device(init, [] {
    cudaError_t r = cudaFuncSetAttribute(tc_gemm_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)kTcSmemBudget);
    if (r != cudaSuccess) return r;
    return cudaFuncSetAttribute(tc_gemm_kernel, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
  });
  if (e != cudaSuccess) return e;
  if (keep) {
    CUtensorMap ca, cb;
    if (!make_map(&ca, sa, kp, (int)(nb * ns * mp), kTcBM, 64) || !make_map(&cb, sb, kp, (int)(nb * ns * np), kChkN, 64))
      return cudaErrorInvalidValue;
    constexpr int kHalfBytes = (kTcBM + kChkN) * 64 * 2;
    static std::atomic<unsigned long long> cinit{0};
    e = once_per_device(cinit, [] {
      return cudaFuncSetAttribute(tc_check_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 2 * kHalfBytes + 1024);
    });
    if (e != cudaSuccess) return e;
    TcArgs c = a;
    c.kblocks = kp / 64;
    ProfScope ps(kClsSplit, st, 0.0);
    tc_check_kernel<<<dim3(mp / kTcBM, np / kChkN, g.nbatch), 256, c.kblocks * kHalfBytes + 1024, st>>>(ca, cb, c);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  dim3 grid(mp / kTcBM, np / bn, g.nbatch);
  // bf16 tensor-core flops issued: S (S + 1) / 2 digit products
  ProfScope ps(kClsGemmTc, st, 2.0 * (double)mp * np * kp * (S * (S + 1) / 2) * nb);
  tc_gemm_kernel<<<grid, 256, smem, st>>>(ma, mb, a);
  return cudaGetLastError();
}

static TcGemm schur_gemm(int m, int n, int k, const double *A, int lda, const double *B, int ldb, double *C, int ldc,
                         int S, int exact, const int *skip) {
  TcGemm g = {};
  g.skip = skip;
  g.A.X = A;  // rows of A: element (i, k) at A[i + k lda]
  g.A.sv = 1;
  g.A.sk = lda;
  g.A.nv = g.A.nv_last = m;
  g.A.K = g.A.K_last = k;
  g.B.X = B;  // columns of B: element (j, k) at B[k + j ldb]
  g.B.sv = ldb;
  g.B.sk = 1;
  g.B.nv = g.B.nv_last = n;
  g.B.K = g.B.K_last = k;
  g.nbatch = 1;
  g.C = C;
  g.ldc = ldc;
  g.sign = 1.0;
  g.S = S;
  g.exact = exact;
  return g;
}

cudaError_t gemm_minus_tc(int m, int n, int k, const double *A, int lda, const double *B, int ldb, double *C,
                          int ldc, int S, int exact, void *ws, int *status, cudaStream_t st, const int *skip) {
  return gemm_tc(schur_gemm(m, n, k, A, lda, B, ldb, C, ldc, S, exact, skip), ws, status, st);
}

// --------------------------------------------------------------------------
// The FP64 Schur update on the tensor cores.  Seven digits of 8 bits hold
// every operand to 2^-57 of its vector's largest magnitude, the digit sums are
// exact and C is rounded once, so for operands of one scale the result is
// closer to the exact product than 128 FP64 multiply-adds: relative error
// 7e-17 against 3.8e-16 (256 x 256 x 128, N(0,1)), backward error of the whole
// CALU 5.6e-15 against 1.2e-14 (n = 2048, N(0,1)).  What the digits keep is
// relative to the largest magnitude of the row of A (column of B), so A's
// columns are first brought to one scale and B's rows scaled back (powers of
// two, column_exp_kernel), which undoes badly scaled rows of the matrix; and
// an element that is still small beside its row's and column's largest is
// found by tc_check_kernel and multiplied in FP64.
// CALU + solve of n = 10240, b = 128: 681 -> 186 ms (622 ms of FP64 GEMM
// became 120 ms here, most of it beside the next panel's tournament).
// --------------------------------------------------------------------------
// kexp[k]: exponent of the largest finite magnitude of column k of A (0 for a
// column without one); one CTA per column.
__global__ void __launch_bounds__(256) column_exp_kernel(int m, const double *__restrict__ A, int lda, int *kexp,
                                                         const int *skip) {
  if (skip && *skip) return;
  __shared__ int red[8];
  const double *a = A + (size_t)blockIdx.x * lda;
  int E = 0;
  for (int i = threadIdx.x; i < m; i += 256) {
    const int e = (int)(absbits(a[i]) >> 52);
    E = max(E, e == 0x7ff ? 0 : e);
  }
  E = __reduce_max_sync(0xffffffffu, E);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = E;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 0; w < 8; ++w) E = max(E, red[w]);
    kexp[blockIdx.x] = E == 0 ? 0 : E - 1023;
  }
}

size_t tc_f64_ws_bytes(int m, int n, int k) {
  return align256((size_t)k * 4) + 256 + tc_gemm_ws_bytes_batched(m, n, k, kTcF64Slices, 1, true);
}

// One 128 x 64 tile of digits costs about 15 us however little of it is used
// (three launches, 28 products); the FP64 kernel as much at 64 x 64 x 64.
// CALU of n = 600, b = 64 takes 4.25 ms with the line at 64 rows and columns,
// 4.45 with it at 128, and of n = 1024 7.9 against 8.2.
bool tc_f64_pays(int m, int n, int k) { return k >= 16 && k <= 128 && m >= 64 && n >= 64; }

cudaError_t gemm_minus_f64_tc(int m, int n, int k, const double *A, int lda, const double *B, int ldb, double *C,
                              int ldc, bool first, void *ws, int *status, cudaStream_t st, const int *skip) {
  char *p = (char *)(((uintptr_t)ws + 255) & ~(uintptr_t)255);
  int *kexp = (int *)p;
  TcGemm g = schur_gemm(m, n, k, A, lda, B, ldb, C, ldc, kTcF64Slices, 1, skip);
  g.keep = 2.5f / 8.0f;
  g.kexp = kexp;
  g.reuse_a = !first;
  if (first) {
    ProfScope ps(kClsSplit, st, 0.0);
    column_exp_kernel<<<k, 256, 0, st>>>(m, A, lda, kexp, skip);
  }
  return gemm_tc(g, p + align256((size_t)k * 4), status, st);
}

}  // namespace cagb
