// solve.cu -- triangular solves and row interchanges that consume the
// factors (PA = LU: swaps, unit-lower forward and upper back substitution;
// A = QR: back substitution with R after Q^T is applied through the tree).
//
// Blocked by kTb rows: for few right-hand sides one cooperative launch with
// one CTA per diagonal block, ordered by ready flags; otherwise the diagonal
// block is solved by one CTA in shared memory and the rows below (or above)
// are updated with the FP64 GEMM, one launch per block.
#include <atomic>

#include "ca_internal.cuh"
#include "device_once.cuh"

namespace cagb {

constexpr int kTb = 128;

// Row interchanges of LAPACK laswp (forward), one CTA per right-hand side;
// the column is staged in shared memory when it fits.
__global__ void __launch_bounds__(32) swap_rows_kernel(int n, const int *ipiv, double *B, int ldb,
                                                       int staged, const int *skip) {
  extern __shared__ __align__(16) double col[];
  if (skip && *skip) return;
  double *b = B + (size_t)blockIdx.x * ldb;
  const int lane = threadIdx.x;
  if (staged) {
    for (int i = lane; i < n; i += 32) col[i] = b[i];
    __syncwarp();
    if (lane == 0)
      for (int i = 0; i < n; ++i) {
        int p = ipiv[i] - 1;
        if (p != i) {
          double t = col[i];
          col[i] = col[p];
          col[p] = t;
        }
      }
    __syncwarp();
    for (int i = lane; i < n; i += 32) b[i] = col[i];
  } else if (lane == 0) {
    for (int i = 0; i < n; ++i) {
      int p = ipiv[i] - 1;
      if (p != i) {
        double t = b[i];
        b[i] = b[p];
        b[p] = t;
      }
    }
  }
}

cudaError_t getrs_swap(int n, int nrhs, const int *ipiv, double *B, int ldb, cudaStream_t st, const int *skip) {
  if (n <= 0 || nrhs <= 0) return cudaSuccess;
  static std::atomic<unsigned long long> init{0};
  cudaError_t e = once_per_device(init, [] {
    return cudaFuncSetAttribute(swap_rows_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
  });
  if (e != cudaSuccess) return e;
  int staged = ((size_t)n * 8 <= 200 * 1024) ? 1 : 0;
  ProfScope ps(kClsSolve, st, 0.0);
  swap_rows_kernel<<<nrhs, 32, staged ? (size_t)n * 8 : 0, st>>>(n, ipiv, B, ldb, staged, skip);
  return cudaGetLastError();
}

// Solve the nb x nb diagonal block T11 X = B1 in place (nb <= kTb) for all
// right-hand sides, one CTA per tile of 32 right-hand sides.
__global__ void __launch_bounds__(256) trsm_diag_kernel(int nb, int nrhs, const double *T, int ldt,
                                                        double *B, int ldb, int lower, int unit,
                                                        const int *skip) {
  extern __shared__ __align__(16) double tsm[];
  if (skip && *skip) return;
  double(*Ts)[kTb + 1] = reinterpret_cast<double(*)[kTb + 1]>(tsm);
  double(*Xs)[33] = reinterpret_cast<double(*)[33]>(tsm + kTb * (kTb + 1));
  const int tid = threadIdx.x;
  const int c0 = blockIdx.x * 32;
  const int nc = min(32, nrhs - c0);
  for (int idx = tid; idx < nb * nb; idx += 256) {
    int i = idx % nb, k = idx / nb;
    Ts[i][k] = T[i + (size_t)k * ldt];
  }
  for (int idx = tid; idx < nb * nc; idx += 256) {
    int i = idx % nb, c = idx / nb;
    Xs[i][c] = B[i + (size_t)(c0 + c) * ldb];
  }
  __syncthreads();
  // column-oriented substitution: finalize x_j, then update the rest
  for (int s = 0; s < nb; ++s) {
    const int j = lower ? s : nb - 1 - s;
    if (!unit) {
      const double d = Ts[j][j];
      for (int c = tid; c < nc; c += 256) Xs[j][c] = Xs[j][c] / d;
      __syncthreads();
    }
    const int lo = lower ? j + 1 : 0, hi = lower ? nb : j;
    const int nr = hi - lo;
    for (int idx = tid; idx < nr * nc; idx += 256) {
      int i = lo + idx % nr, c = idx / nr;
      Xs[i][c] = fma(-Ts[i][j], Xs[j][c], Xs[i][c]);
    }
    __syncthreads();
  }
  for (int idx = tid; idx < nb * nc; idx += 256) {
    int i = idx % nb, c = idx / nb;
    B[i + (size_t)(c0 + c) * ldb] = Xs[i][c];
  }
}

// ---------------------------------------------------------------------------
// One block (n <= kTb), few right-hand sides: substitution with a warp per
// right-hand side, its elements in registers (row lane + 32 t in x[t]), the
// triangle in shared memory; x_j goes round by a shuffle, no barrier after the
// load.  The operations on every element are trsm_diag_kernel's, in its order:
// a division per element, so that diagonals whose reciprocal is not a finite
// number are no special case, and the residual of substitution however
// ill-conditioned the triangle is (the product with an inverse has neither).
// Bound by the chain of n divisions (436 clocks) for U and multiply-adds for L.
// ---------------------------------------------------------------------------
template <bool LOWER, bool UNIT>
__global__ void __launch_bounds__(512) trsv_block_kernel(int n, int nrhs, const double *T, int ldt, double *B, int ldb,
                                                         const int *skip) {
  extern __shared__ __align__(16) double tsm[];  // T(i, j) at i + j (kTb + 1)
  if (skip && *skip) return;
  const int lane = threadIdx.x & 31;
  for (int idx = threadIdx.x; idx < n * n; idx += 512) {
    const int i = idx % n, j = idx / n;
    tsm[i + j * (kTb + 1)] = T[i + (size_t)j * ldt];
  }
  __syncthreads();
  for (int c = threadIdx.x >> 5; c < nrhs; c += 16) {
    double *b = B + (size_t)c * ldb;
    double x[4];
#pragma unroll
    for (int t = 0; t < 4; ++t) x[t] = lane + 32 * t < n ? b[lane + 32 * t] : 0.0;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int s = LOWER ? u : 3 - u;
#pragma unroll 1
      for (int q = 0; q < 32; ++q) {
        const int jl = LOWER ? q : 31 - q, j = 32 * s + jl;
        if (j >= n) continue;
        const double *tj = tsm + j * (kTb + 1);
        double xj = __shfl_sync(0xffffffffu, x[s], jl);
        if (!UNIT) xj = xj / tj[j];
        if (lane == jl) x[s] = xj;
#pragma unroll
        for (int v = 0; v < 4; ++v) {
          const int t = LOWER ? s + v : s - v, i = lane + 32 * t;
          if (t < 0 || t > 3) continue;
          if (LOWER ? i > j && i < n : i < j) x[t] = fma(-tj[i], xj, x[t]);
        }
      }
    }
#pragma unroll
    for (int t = 0; t < 4; ++t)
      if (lane + 32 * t < n) b[lane + 32 * t] = x[t];
  }
}

// ---------------------------------------------------------------------------
// Few right-hand sides, several blocks: one cooperative launch, one CTA per diagonal block,
// ordered by per-block ready flags instead of grid-wide barriers.
//   Phase 0: CTA c loads diagonal block c of T and inverts its four 32 x 32
//            diagonal sub-blocks, one warp each (one per SM sub-partition; a
//            lane per column, the column in registers).
//   Then CTA c takes the blocks it depends on in order (the ones before it
//   for L, after it for U): it waits until block j's solution is published
//   (flag j), subtracts T(c, j) x_j from its right-hand sides, and after the
//   last one solves T_cc x_c = b_c by sub-blocks, writes it to B and publishes
//   flag c.  (Inverting the whole 128 x 128 block took 0.85 ms of dependent
//   multiply-adds per triangle, whatever its order; the sub-blocks 16 us, and
//   the substitution over them as long as the product with the inverse did.)
//   The chain of dependent steps is one GEMV of a 128 x 128 block and one
//   small triangular multiply per block; the earlier GEMVs of a CTA overlap
//   with the chain.  The cooperative launch makes every CTA resident, as the
//   waits require; every wait is bounded (wait_limit cycles of SM clock,
//   about 2 s by default), after which the CTA ORs status_bit into *status
//   and leaves.  The flags live in the caller's workspace (SolveWs) and are
//   cleared before every launch.  withhold_blk >= 0 is a test hook: that
//   block never publishes its flag, so every wait on it runs out.
// Needs one CTA per diagonal block: n <= SMs * kTb.
// ---------------------------------------------------------------------------
constexpr int kCoopMaxRhs = 16;
constexpr int kMaxFlagBlocks = 1024;            // flag words of a solve workspace (covers any SM count here)
constexpr long long kSolveWaitLimit = 4000000000ll;

// Test hook state (host): the wait limit and the withheld block of the next
// dependency-ordered solves (kSolveWaitLimit and -1 unless a test set them).
static std::atomic<long long> g_wait_limit{kSolveWaitLimit};
static std::atomic<int> g_withhold{-1};

// ready flags: one byte per diagonal block (the workspace has room for 4 bytes
// per 128 rows, whichever block size a solve uses)
__device__ __forceinline__ int ld_acquire_gpu(const unsigned char *p) {
  unsigned short v;
  asm volatile("ld.acquire.gpu.global.u8 %0, [%1];" : "=h"(v) : "l"(p) : "memory");
  return v;
}

__device__ __forceinline__ void st_release_gpu(unsigned char *p) {
  asm volatile("st.release.gpu.global.u8 [%0], %1;" ::"l"(p), "h"((unsigned short)1) : "memory");
}

struct FlagArgs {
  unsigned char *flags;  // nblk ready flags, zero at launch
  int *status;           // gets status_bit when a wait gives up
  int status_bit;
  const int *skip;       // refinement: nonzero = the loop has stopped, do nothing
  long long wait_limit;  // cycles
  int withhold_blk;      // test hook (-1: off)
};

constexpr int kTs = 32;  // sub-block of a diagonal block

// Column `lane` of the inverse of the kTs x kTs triangle at Ti (ld kLdI,
// zeros outside it, a nonzero diagonal), by substitution on a unit vector.
template <bool LOWER, int kLdI>
__device__ __forceinline__ void invert_sub(double *Ti, bool unit, int lane) {
  double x[kTs];
#pragma unroll
  for (int i = 0; i < kTs; ++i) x[i] = (i == lane) ? 1.0 : 0.0;
  const double rd = unit ? 1.0 : 1.0 / Ti[lane + lane * kLdI];
#pragma unroll
  for (int s = 0; s < kTs; ++s) {
    const int k = LOWER ? s : kTs - 1 - s;
    const double r = __shfl_sync(0xffffffffu, rd, k);
    if (!unit) x[k] *= r;
#pragma unroll
    for (int i = 0; i < kTs; ++i)
      if (LOWER ? i > k : i < k) x[i] = fma(-Ti[i + k * kLdI], x[k], x[i]);
  }
  __syncwarp();
#pragma unroll
  for (int i = 0; i < kTs; ++i) Ti[i + lane * kLdI] = x[i];
}

template <bool LOWER, int kTb>
__global__ void __launch_bounds__(256, 1) trsv_flag_kernel(int n, int nrhs, const double *T, int ldt, double *B,
                                                           int ldb, int unit, FlagArgs fa) {
  extern __shared__ __align__(16) double csm[];
  constexpr bool lower = LOWER;
  constexpr int kLdI = kTb + 1;
  constexpr int kParts = 256 / kTb, kKp = kTb / kParts;  // threads per row of a block product, columns each
  double *Ti = csm;                          // the diagonal block, its sub-blocks inverted, ld kLdI
  double *sb = Ti + kTb * kLdI;                   // kTb x nrhs: my right-hand sides being reduced
  double *xj = sb + kTb * kCoopMaxRhs;       // kTb x nrhs: a published solution block
  double *part = xj + kTb * kCoopMaxRhs;     // kParts x kTb x nrhs: partial sums of the rows
  __shared__ int abort_flag;
  if (fa.skip && *fa.skip) return;
  unsigned char *flags = fa.flags;
  const int tid = threadIdx.x;
  const int nblk = (n + kTb - 1) / kTb;
  const int blk = blockIdx.x;
  if (blk >= nblk) return;
  const int r0 = blk * kTb, nb = min(kTb, n - r0);

  // ---- phase 0: my diagonal block (the identity beyond its rows) and the
  //      inverses of its diagonal sub-blocks ---------------------------------
  for (int idx = tid; idx < kTb * kTb; idx += blockDim.x) {
    const int i = idx % kTb, k = idx / kTb;
    const bool keep = i < nb && k < nb && (lower ? (i >= k) : (i <= k));
    Ti[i + k * kLdI] = keep ? T[(r0 + i) + (size_t)(r0 + k) * ldt] : (i == k ? 1.0 : 0.0);
  }
  for (int idx = tid; idx < kTb * nrhs; idx += blockDim.x) {
    const int k = idx % kTb, c = idx / kTb;
    sb[k + c * kTb] = k < nb ? B[(r0 + k) + (size_t)c * ldb] : 0.0;
  }
  __syncthreads();
  if ((tid >> 5) * kTs < nb && (tid >> 5) < kTb / kTs)
    invert_sub<LOWER, kLdI>(Ti + (tid >> 5) * kTs * (kLdI + 1), unit != 0, tid & 31);
  __syncthreads();

  // ---- the blocks this one depends on, in order ----------------------------
  const int ndep = lower ? blk : nblk - 1 - blk;
  const int r = tid & (kTb - 1), half = tid / kTb;  // row of my block, share of the columns
  for (int t = 0; t < ndep; ++t) {
    const int j = lower ? t : nblk - 1 - t;
    const int c0 = j * kTb, nbj = min(kTb, n - c0);
    // prefetch this thread's half row of T(blk, j) while waiting
    double trow[kKp];
    const int k0 = half * kKp;
#pragma unroll
    for (int k = 0; k < kKp; ++k)
      trow[k] = (r < nb && k0 + k < nbj) ? T[(r0 + r) + (size_t)(c0 + k0 + k) * ldt] : 0.0;
    if (tid == 0) {
      const long long tstart = clock64();
      int ok = 1;
      while (ld_acquire_gpu(flags + j) == 0) {
        if (clock64() - tstart > fa.wait_limit) {
          ok = 0;
          atomicOr(fa.status, fa.status_bit);  // the timeout record
          break;
        }
      }
      abort_flag = !ok;
    }
    __syncthreads();
    if (abort_flag) return;
    for (int idx = tid; idx < kTb * nrhs; idx += blockDim.x) {
      const int k = idx % kTb, c = idx / kTb;
      // zeros past a short block: the products there are with zeros of T, and
      // what shared memory holds may not be finite
      xj[k + c * kTb] = k < nbj ? __ldcg(B + (c0 + k) + (size_t)c * ldb) : 0.0;
    }
    __syncthreads();
    if (nrhs == 1) {  // one right-hand side: two independent partial sums (four take as long)
      double a2[2] = {0.0, 0.0};
#pragma unroll
      for (int k = 0; k < kKp; ++k) a2[k & 1] = fma(trow[k], xj[k0 + k], a2[k & 1]);
      part[half * kTb * kCoopMaxRhs + r] = a2[0] + a2[1];
    } else {
      double acc[kCoopMaxRhs];
#pragma unroll
      for (int c = 0; c < kCoopMaxRhs; ++c) acc[c] = 0.0;
#pragma unroll
      for (int k = 0; k < kKp; ++k) {
        const double tv = trow[k];
#pragma unroll
        for (int c = 0; c < kCoopMaxRhs; ++c)
          if (c < nrhs) acc[c] = fma(tv, xj[k0 + k + c * kTb], acc[c]);
      }
#pragma unroll
      for (int c = 0; c < kCoopMaxRhs; ++c)
        if (c < nrhs) part[half * kTb * kCoopMaxRhs + r + c * kTb] = acc[c];
    }
    __syncthreads();
    for (int idx = tid; idx < nb * nrhs; idx += blockDim.x) {
      const int i = idx % nb, c = idx / nb;
      double v = part[i + c * kTb];
#pragma unroll
      for (int h = 1; h < kParts; ++h) v += part[h * kTb * kCoopMaxRhs + i + c * kTb];
      sb[i + c * kTb] -= v;
    }
    __syncthreads();
  }

  // ---- T_blk x = b_blk by sub-blocks, published ----------------------------
  // x_s = (inverse of sub-block s) b_s: 8 threads per row; then the rows still
  // to come lose their part: kParts threads per row
  const int nsub = (nb + kTs - 1) / kTs;
  for (int t = 0; t < nsub; ++t) {
    const int s0 = (lower ? t : nsub - 1 - t) * kTs;
    {
      const int i = tid >> 3, k0 = 4 * (tid & 7);
      for (int c = 0; c < nrhs; ++c) {
        double acc = 0.0;
#pragma unroll
        for (int k = 0; k < 4; ++k) acc = fma(Ti[s0 + i + (s0 + k0 + k) * kLdI], sb[s0 + k0 + k + c * kTb], acc);
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        if ((tid & 7) == 0) {
          xj[i + c * kTs] = acc;
          if (s0 + i < nb) B[(r0 + s0 + i) + (size_t)c * ldb] = acc;
        }
      }
    }
    __syncthreads();
    if (t + 1 < nsub) {
      constexpr int kKs = kTs / kParts;
      const int i = tid / kParts, k0 = kKs * (tid % kParts);
      // whole warps (8 or 16 rows) are on one side of s0: no divergence at the shuffle
      if (i < nsub * kTs && (lower ? i >= s0 + kTs : i < s0)) {
        const unsigned m = __activemask();
        for (int c = 0; c < nrhs; ++c) {
          double a0 = 0.0, a1 = 0.0;
#pragma unroll
          for (int k = 0; k < kKs; k += 2) {
            a0 = fma(Ti[i + (s0 + k0 + k) * kLdI], xj[k0 + k + c * kTs], a0);
            a1 = fma(Ti[i + (s0 + k0 + k + 1) * kLdI], xj[k0 + k + 1 + c * kTs], a1);
          }
          a0 += a1;
#pragma unroll
          for (int o = kParts / 2; o > 0; o >>= 1) a0 += __shfl_xor_sync(m, a0, o);
          if (tid % kParts == 0) sb[i + c * kTb] -= a0;
        }
      }
      __syncthreads();
    }
  }
  __threadfence();
  __syncthreads();
  if (tid == 0 && blk != fa.withhold_blk) st_release_gpu(flags + blk);
}

// Solve workspace (caller memory): word 0 is the timeout record of the
// library's solves that use it, the ready flags start at word 32.
size_t solve_ws_bytes(int n) {
  const int nblk = (n + kTb - 1) / kTb;
  return align256((size_t)(32 + (nblk < 1 ? 1 : nblk)) * sizeof(int));
}

void solve_ws_carve(void *w, int n, SolveWs &s) {
  (void)n;
  s.status = (int *)w;
  s.flags = (unsigned char *)((int *)w + 32);
}

void solve_test_hook(long long wait_cycles, int withhold_blk) {
  g_wait_limit.store(wait_cycles > 0 ? wait_cycles : kSolveWaitLimit);
  g_withhold.store(withhold_blk);
}

// one CTA per SM, one diagonal block per CTA
static int coop_max_n() {
  int sms = 1;
  if (device_sm_count(&sms) != cudaSuccess) sms = 1;
  return (sms < kMaxFlagBlocks ? sms : kMaxFlagBlocks) * kTb;
}

template <int TB>
static cudaError_t trsm_left_flags(bool lower, bool unit, int n, int nrhs, const double *T, int ldt, double *B,
                                   int ldb, const SolveWs &ws, int *status, int status_bit, const int *skip,
                                   cudaStream_t st) {
  static std::atomic<unsigned long long> init{0};
  const size_t smem = ((size_t)TB * (TB + 1) + (2 + 256 / TB) * (size_t)TB * kCoopMaxRhs) * 8;
  cudaError_t e = once_per_device(init, [smem] {
    const cudaFuncAttribute a = cudaFuncAttributeMaxDynamicSharedMemorySize;
    const cudaError_t r = cudaFuncSetAttribute(trsv_flag_kernel<true, TB>, a, (int)smem);
    if (r != cudaSuccess) return r;
    return cudaFuncSetAttribute(trsv_flag_kernel<false, TB>, a, (int)smem);
  });
  if (e != cudaSuccess) return e;
  const int nblk = (n + TB - 1) / TB;
  if ((e = cudaMemsetAsync(ws.flags, 0, (size_t)nblk, st)) != cudaSuccess) return e;
  FlagArgs fa;
  fa.flags = ws.flags;
  fa.status = status;
  fa.status_bit = status_bit;
  fa.skip = skip;
  fa.wait_limit = g_wait_limit.load();
  fa.withhold_blk = g_withhold.load();
  if (fa.withhold_blk >= 0) fa.withhold_blk = lower ? 0 : nblk - 1;  // the block nothing else precedes
  int un = unit ? 1 : 0;
  void *args[] = {&n, &nrhs, (void *)&T, &ldt, &B, &ldb, &un, &fa};
  void *fn = lower ? (void *)trsv_flag_kernel<true, TB> : (void *)trsv_flag_kernel<false, TB>;
  ProfScope ps(kClsSolve, st, (double)n * n * nrhs);
  return cudaLaunchCooperativeKernel(fn, dim3(nblk), dim3(256), args, smem, st);
}

template <bool LOWER, bool UNIT>
static cudaError_t trsv_block(int n, int nrhs, const double *T, int ldt, double *B, int ldb, const int *skip,
                              cudaStream_t st) {
  static std::atomic<unsigned long long> init{0};
  cudaError_t e = once_per_device(init, [] {
    return cudaFuncSetAttribute(trsv_block_kernel<LOWER, UNIT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                kTb * (kTb + 1) * 8);
  });
  if (e != cudaSuccess) return e;
  ProfScope ps(kClsSolve, st, (double)n * n * nrhs);
  trsv_block_kernel<LOWER, UNIT><<<1, 512, (size_t)n * (kTb + 1) * 8, st>>>(n, nrhs, T, ldt, B, ldb, skip);
  return cudaGetLastError();
}

cudaError_t trsm_left(bool lower, bool unit, int n, int nrhs, const double *T, int ldt, double *B, int ldb,
                      const SolveWs &ws, int *status, int status_bit, const int *skip, cudaStream_t st) {
  if (n <= 0 || nrhs <= 0) return cudaSuccess;
  // up to 16 right-hand sides: one launch per triangle
  // Blocks of 64 rows while there is an SM for each: the chain is one block
  // product and one block solve per block on a single SM's FP64 pipe, so twice
  // the blocks of a quarter the work each (order 2048, 4 right-hand sides: 925
  // us a triangle before, 750 with blocks of 128, 440 with 64).
  if (nrhs <= kCoopMaxRhs && n <= kTb)
    return !lower ? (unit ? trsv_block<false, true> : trsv_block<false, false>)(n, nrhs, T, ldt, B, ldb, skip, st)
                  : (unit ? trsv_block<true, true> : trsv_block<true, false>)(n, nrhs, T, ldt, B, ldb, skip, st);
  if (nrhs <= kCoopMaxRhs && n <= coop_max_n()) {
    if (n <= coop_max_n() / 2)
      return trsm_left_flags<64>(lower, unit, n, nrhs, T, ldt, B, ldb, ws, status, status_bit, skip, st);
    return trsm_left_flags<kTb>(lower, unit, n, nrhs, T, ldt, B, ldb, ws, status, status_bit, skip, st);
  }
  const size_t smem = ((size_t)kTb * (kTb + 1) + (size_t)kTb * 33) * 8;
  static std::atomic<unsigned long long> init{0};
  cudaError_t e = once_per_device(init, [smem] {
    return cudaFuncSetAttribute(trsm_diag_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  });
  if (e != cudaSuccess) return e;
  const int nblk = (n + kTb - 1) / kTb;
  const dim3 g((nrhs + 31) / 32);
  for (int s = 0; s < nblk; ++s) {
    const int blk = lower ? s : nblk - 1 - s;
    const int r0 = blk * kTb;
    const int nb = min(kTb, n - r0);
    {
      ProfScope ps(kClsSolve, st, (double)nb * nb * nrhs);
      trsm_diag_kernel<<<g, 256, smem, st>>>(nb, nrhs, T + r0 + (size_t)r0 * ldt, ldt, B + r0, ldb,
                                             lower ? 1 : 0, unit ? 1 : 0, skip);
    }
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    if (lower) {
      const int rest = n - r0 - nb;
      e = gemm_minus_f64(rest, nrhs, nb, T + (r0 + nb) + (size_t)r0 * ldt, ldt, B + r0, ldb,
                         B + r0 + nb, ldb, st, skip);
    } else {
      e = gemm_minus_f64(r0, nrhs, nb, T + (size_t)r0 * ldt, ldt, B + r0, ldb, B, ldb, st, skip);
    }
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace cagb
