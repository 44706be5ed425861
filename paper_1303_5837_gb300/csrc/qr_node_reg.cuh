// qr_node_reg.cuh -- Householder QR of one tree node in the registers of a CTA
// of 256 threads (panel_qr_reg.cu, batched.cu).
#pragma once
#include "ca_internal.cuh"
#include "fp64_int.cuh"

namespace cagb {

constexpr int kRegThreads = 256;

template <int TC, int TS>
struct RegSmem {
  double xs[2][16 * TS];                 // x of the published column, by column parity
  double tau[16 * TC], scal[16 * TC];    // tau_q, s_q (1 when tau_q = 0)
  double Z[16 * TC * (16 * TC - 1) / 2];  // v_i^T v_j, i < j, at j (j - 1) / 2 + i
  double T[16 * TC * (16 * TC - 1) / 2];  // strict upper part of T, same packing
};

// The reflector of a column with diagonal alpha and sum of squares ss != 0
// below it: beta = -sign(alpha) ||(alpha, x)||, tau = (beta - alpha) / beta,
// s = 1 / (alpha - beta).  Three dependent FP64 instructions and integer work
// (about 470 clocks; a square root and two divisions take 2000).
static __device__ __noinline__ void reflector_lib(double alpha, double ss, double &beta, double &tau, double &s) {
  const double nrm = sqrt(fma(alpha, alpha, ss));
  beta = (alpha >= 0.0) ? -nrm : nrm;
  tau = (beta - alpha) / beta;
  s = 1.0 / (alpha - beta);
}
// The same three values bit for bit: square root and quotient by Markstein's
// final step (the exact residual of an approximation times its reciprocal,
// added to it), correctly rounded from approximations this close; the
// reciprocals correctly rounded in integers.
__device__ __forceinline__ void reflector_fixed(double alpha, double ss, double &beta, double &tau, double &s) {
  const double v = fma(alpha, alpha, ss);
  if (!int_range(v)) return reflector_lib(alpha, ss, beta, tau, s);
  const double y = rsqrt_near(v), q = v * y;
  const double nrm = fma(0.5 * y, fma(-q, q, v), q);
  const double be = (alpha >= 0.0) ? -nrm : nrm;
  const double num = be - alpha, rb = recip_exact_or_zero(be), rd = recip_exact_or_zero(-num);
  if (__double_as_longlong(rb) == 0 || __double_as_longlong(rd) == 0) return reflector_lib(alpha, ss, beta, tau, s);
  const double z = num * rb;
  beta = be;
  tau = fma(fma(-z, be, num), rb, z);
  s = rd;
}
// fixed: correctly rounded (panel_qr_fixed.cu)
__device__ __forceinline__ void reflector(double alpha, double ss, double &beta, double &tau, double &s,
                                          bool fixed = false) {
  if (fixed) return reflector_fixed(alpha, ss, beta, tau, s);
  const double v = fma(alpha, alpha, ss), a = fabs(alpha);
  if (int_range(v)) {
    const double y = rsqrt_near(v);
    const double nrm = v * y, d = a + nrm;
    tau = fma(a, y, 1.0);
    const double r = recip_near(d);
    const bool neg = __double_as_longlong(alpha) < 0 && a != 0.0;
    beta = neg ? nrm : -nrm;
    s = neg ? -r : r;
  } else {
    reflector_lib(alpha, ss, beta, tau, s);
  }
}
// Sum of e[t] over the 16 lanes of the half-warp by reduce-scatter: lane rg
// gets the sum of value t = sum_index<TC>(rg).
template <int TC>
__device__ __forceinline__ int sum_index(int rg) {
  constexpr int L = TC == 1 ? 0 : TC == 2 ? 1 : TC == 4 ? 2 : 3;
  return rg >> (4 - L);
}
template <int TC>
__device__ __forceinline__ int sum_lane(int t) {  // a lane that holds the sum of value t
  constexpr int L = TC == 1 ? 0 : TC == 2 ? 1 : TC == 4 ? 2 : 3;
  return t << (4 - L);
}
template <int TC>
__device__ __forceinline__ double half_sum_scatter(const double (&e)[TC], int rg) {
  constexpr int L = TC == 1 ? 0 : TC == 2 ? 1 : TC == 4 ? 2 : 3;
  double v[TC];
#pragma unroll
  for (int t = 0; t < TC; ++t) v[t] = e[t];
#pragma unroll
  for (int k = 0; k < L; ++k) {
    const int o = 8 >> k;
    const int h = TC >> (k + 1);
    const bool up = (rg & o) != 0;
#pragma unroll
    for (int i = 0; i < h; ++i) {
      const double keep = up ? v[i + h] : v[i];
      const double send = up ? v[i] : v[i + h];
      v[i] = keep + __shfl_xor_sync(0xffffffffu, send, o, 16);
    }
  }
#pragma unroll
  for (int k = L; k < 4; ++k) v[0] += __shfl_xor_sync(0xffffffffu, v[0], 8 >> k, 16);
  return v[0];
}

// Rows of a node that can be nonzero below the diagonal of column j (and so
// take part in its reflector): a leaf's rows below the diagonal; in a merge
// whose first child holds every diagonal row (c0 >= kmax) and whose other
// children have one height h, the other children's rows are kept in the
// order of their index t within the child (row t of every child, then row
// t + 1 ...), so the rows with t <= j -- the only ones of those children not
// structurally zero in column j -- come first, and the first child's rows
// below the diagonal are zero.  Row blocks [beg, end(j)) hold them all;
// skipping the others drops only exact zeros.  Other merges run dense.
template <bool MERGE>
struct NodeRows {
  int reord;  // 1: merge rows in the order above
  int beg;    // first block that can hold such rows
  int c0, nk, h, R;
  int fixed;  // correctly rounded reflectors (reflector_fixed)
  // leaves run every block (the zero rows of a short leaf cost nothing wrong)
  __device__ __forceinline__ int first() const { return MERGE ? beg : 0; }
  __device__ __forceinline__ int end(int j) const {
    if (!MERGE) return 1 << 20;
    const int p = reord ? c0 + nk * min(j + 1, h) : R;
    return (p + 15) >> 4;
  }
};

// Reflector of column jc = 16 U + jr, by the half-warp that holds it (cg =
// jr): beta = -sign(alpha) ||(alpha, x)||, tau = (beta - alpha) / beta,
// s = 1 / (alpha - beta); R(jc, jc) = beta; x published to xs.
template <int TC, int TS, int U, bool MERGE>
__device__ __forceinline__ void reflect(double (&A)[TS][TC], const NodeRows<MERGE> &nr, int rg, int jr, int jc,
                                        double *xs, double *tau, double *scal) {
  const unsigned hm = 0xffffu << (threadIdx.x & 16);
  const int se = nr.end(jc);
  double ss = 0.0;
#pragma unroll
  for (int s = U; s < TS; ++s) {
    if (s >= se) break;
    if (s < nr.first()) continue;
    if (s > U || rg > jr) ss = fma(A[s][U], A[s][U], ss);
  }
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) ss += __shfl_xor_sync(hm, ss, o, 16);
  const double alpha = __shfl_sync(hm, A[U][U], jr, 16);
  double t = 0.0, sc = 1.0;
  if (ss != 0.0) {
    double beta;
    reflector(alpha, ss, beta, t, sc, nr.fixed != 0);
    if (rg == jr) A[U][U] = beta;
  }
#pragma unroll
  for (int s = U; s < TS; ++s) {
    if (s >= se) break;
    if (s < nr.first()) continue;
    xs[16 * s + rg] = (s > U || rg > jr) ? A[s][U] : 0.0;
  }
  if (rg == 0) {
    tau[jc] = t;
    scal[jc] = sc;
  }
}

// A(:, q) -= v_j w_q for the thread's column t (q = cg + 16 t > j): row j
// takes w_q itself, rows below it x_i s_j w_q (x is zero at rows <= j).
template <int TC, int TS, int U>
__device__ __forceinline__ void update_col(double (&A)[TS][TC], const double (&x)[TS], int sb, int se, int t,
                                           double wt, double sw, bool row_j) {
#pragma unroll
  for (int s = U; s < TS; ++s) {
    if (s >= se) break;
    if (s < sb) continue;
    A[s][t] = fma(-x[s], sw, A[s][t]);
  }
  if (row_j) A[U][t] -= wt;
}

// Columns j = 16 U .. 16 U + 15 (those below kmax); row blocks [sb, se).
template <int TC, int TS, int U, bool MERGE>
__device__ __forceinline__ void qr_block(double (&A)[TS][TC], const NodeRows<MERGE> &nr, RegSmem<TC, TS> &sm,
                                         int rg, int cg, int kmax) {
  for (int jr = 0; jr < 16; ++jr) {
    const int j = 16 * U + jr;
    if (j >= kmax) return;
    __syncthreads();  // column j's x, tau_j and s_j are published
    const double tj = sm.tau[j], sj = sm.scal[j];
    const double *xb = sm.xs[j & 1];
    const int sb = nr.first(), se = nr.end(j);
    double x[TS];
#pragma unroll
    for (int s = 0; s < TS; ++s) x[s] = 0.0;
#pragma unroll
    for (int s = U; s < TS; ++s) {
      if (s >= se) break;
      if (s < sb) continue;
      x[s] = xb[16 * s + rg];
    }
    double w[TC], sw[TC];
#pragma unroll
    for (int t = 0; t < TC; ++t) w[t] = sw[t] = 0.0;
    if (tj != 0.0) {
      double e[TC];
#pragma unroll
      for (int t = 0; t < TC; ++t) {
        double acc = 0.0;
#pragma unroll
        for (int s = U; s < TS; ++s) {
          if (s >= se) break;
          if (s < sb) continue;
          acc = fma(x[s], A[s][t], acc);
        }
        e[t] = acc;
      }
      // what follows from a column's sum -- d_q, w_q and s_j w_q, or Z(q, j)
      // -- is computed on the lane that holds it, once for all TC columns
      const double sum = half_sum_scatter<TC>(e, rg);
      const int ts = sum_index<TC>(rg), qs = cg + 16 * ts;
      double ajq = 0.0;
#pragma unroll
      for (int t = 0; t < TC; ++t) {
        const double v = __shfl_sync(0xffffffffu, A[U][t], jr, 16);
        ajq = (t == ts) ? v : ajq;
      }
      const double d = fma(sj, sum, ajq);
      const double wq = qs > j ? tj * d : 0.0;
      const double swq = sj * wq;
      if (qs < j && rg == sum_lane<TC>(ts)) sm.Z[j * (j - 1) / 2 + qs] = sm.scal[qs] * d;
#pragma unroll
      for (int t = U; t < TC; ++t) {
        w[t] = __shfl_sync(0xffffffffu, wq, sum_lane<TC>(t), 16);
        sw[t] = __shfl_sync(0xffffffffu, swq, sum_lane<TC>(t), 16);
      }
    } else if (rg == 0) {
#pragma unroll
      for (int t = 0; t < TC; ++t) {
        const int q = cg + 16 * t;
        if (q < j) sm.Z[j * (j - 1) / 2 + q] = 0.0;
      }
    }
    const bool row_j = rg == jr;
    // the column after j first, then its reflector, then the other columns
    if (tj != 0.0 && cg > jr) update_col<TC, TS, U>(A, x, sb, se, U, w[U], sw[U], row_j);
    if (jr == 15) {
      if constexpr (U + 1 < TC) {
        if (tj != 0.0) update_col<TC, TS, U>(A, x, sb, se, U + 1, w[U + 1], sw[U + 1], row_j);
        if (j + 1 < kmax && cg == 0) reflect<TC, TS, U + 1, MERGE>(A, nr, rg, 0, j + 1, sm.xs[(j + 1) & 1], sm.tau, sm.scal);
#pragma unroll
        for (int t = U + 2; t < TC; ++t)
          if (tj != 0.0) update_col<TC, TS, U>(A, x, sb, se, t, w[t], sw[t], row_j);
      }
    } else {
      if (j + 1 < kmax && cg == jr + 1) reflect<TC, TS, U, MERGE>(A, nr, rg, jr + 1, j + 1, sm.xs[(j + 1) & 1], sm.tau, sm.scal);
#pragma unroll
      for (int t = U + 1; t < TC; ++t)
        if (tj != 0.0) update_col<TC, TS, U>(A, x, sb, se, t, w[t], sw[t], row_j);
    }
  }
}

template <int TC, int TS, int U, bool MERGE>
__device__ __forceinline__ void qr_blocks(double (&A)[TS][TC], const NodeRows<MERGE> &nr, RegSmem<TC, TS> &sm,
                                          int rg, int cg, int kmax) {
  if constexpr (U < TC) {
    qr_block<TC, TS, U, MERGE>(A, nr, sm, rg, cg, kmax);
    qr_blocks<TC, TS, U + 1, MERGE>(A, nr, sm, rg, cg, kmax);
  }
}

// The whole node: reflectors, v = s x below the diagonal, T (strict upper part
// in sm.T, diagonal in sm.tau).  Every thread of the CTA calls it.
template <int TC, int TS, bool MERGE>
__device__ __forceinline__ void qr_node(double (&A)[TS][TC], const NodeRows<MERGE> &nr, RegSmem<TC, TS> &sm, int kmax) {
  const int tid = threadIdx.x, lane = tid & 31;
  const int rg = lane & 15, cg = 2 * (tid >> 5) + (lane >> 4);
  if (kmax > 0 && cg == 0) reflect<TC, TS, 0, MERGE>(A, nr, rg, 0, 0, sm.xs[0], sm.tau, sm.scal);
  qr_blocks<TC, TS, 0, MERGE>(A, nr, sm, rg, cg, kmax);
  __syncthreads();  // every tau, s and Z entry is written

  // v = s x below the diagonal of every reflector column
#pragma unroll
  for (int t = 0; t < TC; ++t) {
    const int q = cg + 16 * t;
    if (q < kmax) {
      const double sq = sm.scal[q];
#pragma unroll
      for (int s = 0; s < TS; ++s)
        if (rg + 16 * s > q) A[s][t] *= sq;
    }
  }

  // ---- T (larft, forward columnwise): T(i, j) = -tau_j sum_{q=i}^{j-1} T(i, q) Z(q, j),
  //      T(j, j) = tau_j; four threads per row i, each over every fourth q
  const int i = tid >> 2, part = tid & 3;
  for (int j = 1; j < kmax; ++j) {
    const double tj = sm.tau[j];
    double acc = 0.0;
    if (i < j && tj != 0.0)
      for (int q = i + part; q < j; q += 4) {
        const double tiq = (q == i) ? sm.tau[i] : sm.T[q * (q - 1) / 2 + i];
        acc = fma(tiq, sm.Z[j * (j - 1) / 2 + q], acc);
      }
    acc += __shfl_xor_sync(0xffffffffu, acc, 1);
    acc += __shfl_xor_sync(0xffffffffu, acc, 2);
    if (i < j && part == 0) sm.T[j * (j - 1) / 2 + i] = (tj != 0.0) ? -tj * acc : 0.0;
    __syncthreads();  // column j of T is complete before column j + 1 reads it
  }
}

}  // namespace cagb
