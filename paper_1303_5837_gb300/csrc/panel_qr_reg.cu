// panel_qr_reg.cu -- TSQR tree nodes held in the registers of one CTA.
//
// A node of R <= 16 TS rows and bk <= 16 TC columns (a leaf of the panel, or
// the stacked R factors of a merge: Sec. 3.1) is factored by Householder QR
// with its tile in the registers of 256 threads: thread (rg, cg), rg = lane
// mod 16 and cg = 2 warp + lane / 16, holds rows rg + 16 s (s < TS) and
// columns cg + 16 t (t < TC).  A half-warp therefore holds every row of its
// TC columns, so the column sums of the method need no shared memory and no
// barrier: a few shuffles inside the half-warp.  Per column j, one barrier:
//   * the owner of column j (the half-warp with cg = j mod 16) has published
//     x = A(j+1:, j) (zeros at rows <= j), tau_j and s_j = 1 / (alpha - beta)
//     in shared memory (v_j = s_j x below the diagonal, 1 on it);
//   * every thread multiplies x with its columns over its rows and the
//     half-warp sums the products: d_q = A(j, q) + s_j x^T A(j+1:, q) for
//     every column q, so the work of a step is the same in every warp;
//   * q > j: A(j, q) -= tau_j d_q and A(i, q) -= x_i s_j tau_j d_q;
//   * q < j: d_q = x_q(j) + s_j x_q^T x, and Z(q, j) = v_q^T v_j = s_q d_q,
//     the dot products larft needs for T, from the same pass;
//   * the owner of column j + 1 updates that column first and derives its
//     reflector before its other columns (look-ahead), so the reflector's
//     square root and divisions overlap with the other warps' updates.
// The stored x of every column is scaled by s_q once, after the last column.
// On this part the FP64 pipe (2 multiply-adds per clock per SM) is the scarce
// resource; this layout keeps every warp's FP64 instructions full and
// balanced, where a shared-memory tile with column-per-thread dot products
// leaves half the warps idle once fewer than half the columns remain.
#include "ca_internal.cuh"
#include "cluster_copy.cuh"
#include "device_once.cuh"
#include "qr_node_reg.cuh"

namespace cagb {

namespace {

// Nodes of at most 128 rows, or 32 columns, leave room for two CTAs per SM,
// which hide each other's per-column barrier and reflector.
template <int TC, int TS>
constexpr int reg_min_blocks() {
  return TC * TS <= 32 ? 2 : 1;
}

template <int TC, int TS, bool MERGE>
__global__ void __launch_bounds__(kRegThreads, reg_min_blocks<TC, TS>()) tsqr_reg_kernel(TsqrNodeArgs a) {
  __shared__ RegSmem<TC, TS> sm;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int rg = lane & 15, cg = 2 * warp + (lane >> 4);
  const int node = blockIdx.x;
  const int bk = a.bk;

  // ---- node rows: a leaf's consecutive panel rows, or the children's R rows
  int R, r0 = 0, start = 0, cnt = 1, midx = 0;
  if (a.is_leaf) {
    r0 = node * a.leaf_rows;
    R = min(a.leaf_rows, a.mk - r0);
  } else {
    round_node(a.rd, node, start, cnt, midx);
    if (cnt == 1) {  // promotion: nothing to factor
      if (tid == 0) {
        a.top_out[node] = a.top_in[start];
        a.c_out[node] = a.c_in[start];
      }
      return;
    }
    R = 0;
    for (int ch = 0; ch < cnt; ++ch) R += a.c_in[start + ch];
  }
  const int kmax = min(R, bk);
  NodeRows<MERGE> nr;
  nr.R = R;
  nr.reord = 0;
  nr.beg = 0;
  nr.c0 = nr.nk = nr.h = 0;
  nr.fixed = a.fixed;
  if (!a.is_leaf) {
    const int c0 = a.c_in[start], h = a.c_in[start + 1];
    bool same = true;
    for (int ch = 2; ch < cnt; ++ch) same &= a.c_in[start + ch] == h;
    if (same && c0 >= kmax) {
      nr.reord = 1;
      nr.c0 = c0;
      nr.nk = cnt - 1;
      nr.h = h;
      nr.beg = c0 >> 4;
    }
  }
  // panel row of local row r and its first structurally nonzero column (a
  // merge row that is row t of its child's R is zero left of column t)
  auto row_info = [&](int r, int &prow, int &fz) {
    prow = -1;
    fz = 1 << 30;
    if (r >= R) return;
    if (a.is_leaf) {
      prow = r0 + r;
      fz = 0;
      return;
    }
    if (nr.reord && r >= nr.c0) {
      const int t = (r - nr.c0) / nr.nk, k = 1 + (r - nr.c0) % nr.nk;
      prow = a.top_in[start + k] + t;
      fz = t;
      return;
    }
    int off = 0;
    for (int ch = 0; ch < cnt; ++ch) {
      const int c = a.c_in[start + ch];
      if (r < off + c) {
        prow = a.top_in[start + ch] + (r - off);
        fz = r - off;
        return;
      }
      off += c;
    }
  };

  // ---- load: lanes of a half-warp read 16 consecutive rows of a column ----
  double A[TS][TC];
  bool bad = false;
#pragma unroll
  for (int s = 0; s < TS; ++s) {
    int prow, fz;
    row_info(rg + 16 * s, prow, fz);
#pragma unroll
    for (int t = 0; t < TC; ++t) {
      const int q = cg + 16 * t;
      double v = 0.0;
      if (prow >= 0 && q < bk && q >= fz) v = a.P[prow + (size_t)q * a.lda];
      bad |= not_finite(v);
      A[s][t] = v;
    }
  }
  if (bad && a.dev_info) atomicOr(a.dev_info + 1, CA_STATUS_NONFINITE);

  // ---- Householder QR, one barrier per column, and T -----------------------
  qr_node<TC, TS, MERGE>(A, nr, sm, kmax);
  {
    const int b = a.b;
    double *Tg = a.Tp + (size_t)(a.is_leaf ? node : a.nleaves + midx) * b * b;
    for (int idx = tid; idx < b * b; idx += kRegThreads) {
      const int i = idx % b, jj = idx / b;
      double v = 0.0;
      if (jj < kmax && i <= jj) v = (i == jj) ? sm.tau[jj] : sm.T[jj * (jj - 1) / 2 + i];
      Tg[idx] = v;
    }
  }

  // ---- write back: leaf in place; merge: R into the first child's rows, Y
  //      into the other children's rows (on and above their diagonal)
#pragma unroll
  for (int s = 0; s < TS; ++s) {
    int prow, fz;
    row_info(rg + 16 * s, prow, fz);
#pragma unroll
    for (int t = 0; t < TC; ++t) {
      const int q = cg + 16 * t;
      if (prow >= 0 && q < bk && q >= fz) a.P[prow + (size_t)q * a.lda] = A[s][t];
    }
  }
  if (tid == 0) {
    a.top_out[node] = a.is_leaf ? r0 : a.top_in[start];
    a.c_out[node] = kmax;
  }
}

template <int TC, int TS>
cudaError_t launch_reg(const TsqrNodeArgs &a, int nodes, cudaStream_t st) {
  if (a.is_leaf)
    tsqr_reg_kernel<TC, TS, false><<<nodes, kRegThreads, 0, st>>>(a);
  else
    tsqr_reg_kernel<TC, TS, true><<<nodes, kRegThreads, 0, st>>>(a);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Cluster form: a node of R <= 128 TS rows and bk <= 16 TC columns on 8 CTAs
// with the same thread layout (TC = 4 or 8 columns per thread).  A leaf's rows are
// split in contiguous chunks; a merge whose first child holds every diagonal
// row deals its rows round robin, the other children's rows in the order of
// their index within the child, so that the rows that can be nonzero in
// column j are the first ones of every CTA (NodeRows).  One exchange per
// column: every CTA sends the partial sums x_j^T A(:, q) of all columns (the
// sum of squares among them) and, from the CTA that holds it, row j; every
// CTA adds the 8 partials in rank order, derives the same reflector and w.
// They travel as bulk copies counted on the receiver's mbarrier (600 clocks;
// two cluster barriers and the reads of the peers' memory took 1500).  While
// they travel, column j - 1 of T is formed: half-warp hw of CTA `rank` owns
// row 8 hw + rank of T, in registers, so larft's recurrence needs no barrier
// and no pass of its own after the last column.
// Measured per node, before (two cluster barriers and a serial reflector per
// column; one CTA for 64 columns) and now: 1024 x 128 leaf rounds of CAQR 6144
// 2.47 -> 0.91 ms a launch on average, 256 x 128 nodes 1.43 -> 0.56 ms,
// 128 x 64 nodes 0.47 -> 0.21 ms.
// Both halves of a send buffer and of the receive buffers alternate by column
// parity: a CTA sends column j + 1 after it has received column j from all,
// whose senders had read every column j - 1 before they sent (the barrier in
// front of the copies) and had received this CTA's column j - 1.
// ---------------------------------------------------------------------------
constexpr int kCG = 8;    // CTAs per node

template <int TC, int TS>
struct alignas(16) CRegSmem {
  static constexpr int kCW = 16 * TC;  // columns of an exchanged row
  double in[2][kCG][kCW];      // received partial sums, by column parity and rank
  double row[2][kCW];          // received row j
  double out[2][2 * kCW];      // this CTA's partial sums and row j on their way out
  double xs[16 * TS];          // this CTA's part of x_j (zeros at rows <= j)
  double esum[kCW];            // x_j^T A(:, q) over the whole node
  double z[kCW];               // v_q^T v_j, q < j (zero from q = j on)
  double tau[kCW], scal[kCW];
  double beta;
  unsigned long long bar[2];   // column parity: sums and row have arrived
  int gave_up;                 // a CTA of the cluster gave up waiting
};

// What the column steps of one thread share.
template <int TC, int TS>
struct CNode {
  static constexpr int kCTC = TC, kCW = 16 * TC;
  CRegSmem<TC, TS> &sm;
  int rg, cg, warp, rank, kmax, bkw;  // bkw: columns sent (bk rounded up to 2)
  int cyc;                            // rows dealt round robin
  int c0, nk, h, R;                   // merge: first child's rows, other children, their height; node rows
  double A[TS][kCTC];
  double T[kCTC];                     // row 8 hw + rank of T, columns rg + 16 t
  bool dead;                          // a wait gave up; nothing is waited for any more
  int *status;
  long long limit;
  int nsend;                          // CTAs this one sends to: 8, or 0 after a give-up (test hook: always)

  __device__ __forceinline__ explicit CNode(CRegSmem<TC, TS> &s) : sm(s) {}
  __device__ __forceinline__ int node_row(int s) const {
    return cyc ? rank + kCG * (rg + 16 * s) : rank * 16 * TS + rg + 16 * s;
  }
  // row blocks [first(j), last(j)) of this CTA hold every nonzero of x_j
  __device__ __forceinline__ int first(int j) const {
    return cyc ? c0 / (16 * kCG) : max(0, (j + 1 - rank * 16 * TS) >> 4);
  }
  __device__ __forceinline__ int last(int j) const {
    const int end = cyc ? (c0 + nk * min(j + 1, h) + kCG - 1) / kCG : R - rank * 16 * TS;
    return min(TS, (end + 15) >> 4);
  }

  // column jt of T from z and tau (every thread; z is zero from jt on)
  __device__ __forceinline__ void t_column(int jt) {
    if (16 * warp > jt) return;  // rows past the diagonal (both rows of the warp)
    const double tj = sm.tau[jt];
    double acc = 0.0;
#pragma unroll
    for (int t = 0; t < kCTC; ++t)
      if (t >= warp && 16 * t < jt) acc = fma(T[t], sm.z[rg + 16 * t], acc);
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o, 16);
    const int i = 8 * cg + rank;
    const double v = i == jt ? tj : (i < jt && tj != 0.0) ? -tj * acc : 0.0;
#pragma unroll
    for (int t = 0; t < kCTC; ++t)
      if (rg + 16 * t == jt) T[t] = v;
  }

  // Columns j = 16 U .. 16 U + 15 below kmax.
  template <int U>
  __device__ __forceinline__ void block() {
    for (int jr = 0; jr < 16; ++jr) {
      const int j = 16 * U + jr;
      if (j >= kmax) return;
      const int q = j & 1;
      const int idx = cyc ? j / kCG : j % (16 * TS);  // row j within its CTA
      const bool row_j = (cyc ? j % kCG : j / (16 * TS)) == rank && (idx & 15) == rg;
      const int sj = idx >> 4;
      __syncthreads();  // x_j is staged
      const int sb = first(j), se = last(j);
      double x[TS];
#pragma unroll
      for (int s = 0; s < TS; ++s) x[s] = (s >= sb && s < se) ? sm.xs[rg + 16 * s] : 0.0;
      {
        double e[kCTC];
#pragma unroll
        for (int t = 0; t < kCTC; ++t) e[t] = 0.0;
#pragma unroll
        for (int s = 0; s < TS; ++s) {
          if (s < sb || s >= se) continue;
#pragma unroll
          for (int t = 0; t < kCTC; ++t) e[t] = fma(x[s], A[s][t], e[t]);
        }
        const double sum = half_sum_scatter<kCTC>(e, rg);
        const int ts = sum_index<kCTC>(rg);
        if (rg == sum_lane<kCTC>(ts)) sm.out[q][cg + 16 * ts] = sum;
      }
      if (row_j) {
#pragma unroll
        for (int s = 0; s < TS; ++s)
          if (s == sj) {
#pragma unroll
            for (int t = 0; t < kCTC; ++t) sm.out[q][kCW + cg + 16 * t] = A[s][t];
          }
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // the copies read what was just written
      __syncthreads();
      if ((int)threadIdx.x < nsend) {
        const unsigned bytes = 8u * bkw;
        bulk_to(sm.in[q][rank], sm.out[q], bytes, &sm.bar[q], threadIdx.x);
        if ((cyc ? j % kCG : j / (16 * TS)) == rank) bulk_to(sm.row[q], sm.out[q] + kCW, bytes, &sm.bar[q], threadIdx.x);
      }
      if (j > 0) t_column(j - 1);
      if (!dead && !bar_wait(&sm.bar[q], (j >> 1) & 1, limit)) {
        dead = true;
        nsend = 0;
      }
      if (threadIdx.x < kCW) {  // one warp per SM sub-partition adds the partials
        if (threadIdx.x == 0 && j + 2 < kmax && !dead) bar_expect(&sm.bar[q], 8u * bkw * (kCG + 1));
        double v = sm.in[q][0][threadIdx.x];
#pragma unroll
        for (int r = 1; r < kCG; ++r) v += sm.in[q][r][threadIdx.x];
        sm.esum[threadIdx.x] = v;
        if (warp == j >> 5) {
          const double ss = __shfl_sync(0xffffffffu, v, j & 31), alpha = sm.row[q][j];
          double t = 0.0, sc = 1.0, be = alpha;
          if (ss != 0.0) reflector(alpha, ss, be, t, sc);
          if ((threadIdx.x & 31) == 0) {
            sm.tau[j] = t;
            sm.scal[j] = sc;
            sm.beta = be;
          }
        }
      }
      __syncthreads();  // sums, tau_j and s_j; every partial and t_column's z has been read
      const double tj = sm.tau[j], sj_ = sm.scal[j];
      double w[kCTC], sw[kCTC];
      {
        const int ts = sum_index<kCTC>(rg), qs = cg + 16 * ts;
        const double d = fma(sj_, sm.esum[qs], sm.row[q][qs]);
        const double wq = (qs > j && tj != 0.0) ? tj * d : 0.0;
        const double swq = sj_ * wq;
        if (qs < j && rg == sum_lane<kCTC>(ts)) sm.z[qs] = sm.scal[qs] * d;
#pragma unroll
        for (int t = U; t < kCTC; ++t) {
          w[t] = __shfl_sync(0xffffffffu, wq, sum_lane<kCTC>(t), 16);
          sw[t] = __shfl_sync(0xffffffffu, swq, sum_lane<kCTC>(t), 16);
        }
      }
      // A(:, q) -= v_j w_q: rows below j x_i s_j w_q, row j itself w_q
      auto upd = [&](int t) {
        if (tj == 0.0) return;
#pragma unroll
        for (int s = 0; s < TS; ++s) {
          if (s < sb || s >= se) continue;
          A[s][t] = fma(-x[s], sw[t], A[s][t]);
        }
        if (row_j) {
#pragma unroll
          for (int s = 0; s < TS; ++s)
            if (s == sj) A[s][t] -= w[t];
        }
      };
      auto stage_next = [&](int t) {  // column j + 1 = cg + 16 t, held by this half-warp
#pragma unroll
        for (int s = 0; s < TS; ++s) sm.xs[rg + 16 * s] = node_row(s) > j + 1 ? A[s][t] : 0.0;
      };
      if (cg == jr && row_j) {
#pragma unroll
        for (int s = 0; s < TS; ++s)
          if (s == sj) A[s][U] = sm.beta;
      }
      const bool more = j + 1 < kmax;
      if (cg > jr) upd(U);
      if (jr == 15) {
        if constexpr (U + 1 < kCTC) {
          upd(U + 1);
          if (more && cg == 0) stage_next(U + 1);
#pragma unroll
          for (int t = U + 2; t < kCTC; ++t) upd(t);
        }
      } else {
        if (more && cg == jr + 1) stage_next(U);
#pragma unroll
        for (int t = U + 1; t < kCTC; ++t) upd(t);
      }
    }
  }
  template <int U>
  __device__ __forceinline__ void blocks() {
    if constexpr (U < kCTC) {
      block<U>();
      blocks<U + 1>();
    }
  }
};

template <int TC, int TS>
__global__ void __launch_bounds__(kRegThreads, 1) tsqr_creg_kernel(TsqrNodeArgs a) {
  cg::cluster_group cl = cg::this_cluster();
  const int rank = (int)cl.block_rank();
  const int node = blockIdx.x / kCG;
  constexpr int kCTC = TC, kCW = 16 * TC;
  __shared__ CRegSmem<TC, TS> sm;
  const int tid = threadIdx.x, lane = tid & 31;
  const int bk = a.bk;

  int R, r0 = 0, start = 0, cnt = 1, midx = 0;
  if (a.is_leaf) {
    r0 = node * a.leaf_rows;
    R = min(a.leaf_rows, a.mk - r0);
  } else {
    round_node(a.rd, node, start, cnt, midx);
    if (cnt == 1) {  // promotion: the whole cluster returns before any barrier
      if (rank == 0 && tid == 0) {
        a.top_out[node] = a.top_in[start];
        a.c_out[node] = a.c_in[start];
      }
      return;
    }
    R = 0;
    for (int ch = 0; ch < cnt; ++ch) R += a.c_in[start + ch];
  }
  CNode<TC, TS> nd(sm);
  nd.rg = lane & 15;
  nd.warp = tid >> 5;
  nd.cg = 2 * nd.warp + (lane >> 4);
  nd.rank = rank;
  nd.kmax = min(R, bk);
  nd.bkw = (bk + 1) & ~1;
  nd.R = R;
  nd.cyc = 0;
  nd.c0 = nd.nk = nd.h = 0;
  nd.dead = false;
  nd.status = a.dev_info ? a.dev_info + 1 : nullptr;
  nd.limit = a.wait_limit;
  nd.nsend = a.withhold && rank == kCG - 1 ? 0 : kCG;
  if (!a.is_leaf) {
    const int c0 = a.c_in[start], h = a.c_in[start + 1];
    bool same = true;
    for (int ch = 2; ch < cnt; ++ch) same &= a.c_in[start + ch] == h;
    if (same && c0 >= nd.kmax) {
      nd.cyc = 1;
      nd.c0 = c0;
      nd.nk = cnt - 1;
      nd.h = h;
    }
  }
  // panel row of node row r and its first structurally nonzero column
  auto row_info = [&](int r, int &prow, int &fz) {
    prow = -1;
    fz = 1 << 30;
    if (r >= R) return;
    if (a.is_leaf) {
      prow = r0 + r;
      fz = 0;
      return;
    }
    if (nd.cyc && r >= nd.c0) {
      const int t = (r - nd.c0) / nd.nk, k = 1 + (r - nd.c0) % nd.nk;
      prow = a.top_in[start + k] + t;
      fz = t;
      return;
    }
    int off = 0;
    for (int ch = 0; ch < cnt; ++ch) {
      const int c = a.c_in[start + ch];
      if (r < off + c) {
        prow = a.top_in[start + ch] + (r - off);
        fz = r - off;
        return;
      }
      off += c;
    }
  };

  bool bad = false;
#pragma unroll
  for (int s = 0; s < TS; ++s) {
    int prow, fz;
    row_info(nd.node_row(s), prow, fz);
#pragma unroll
    for (int t = 0; t < kCTC; ++t) {
      const int qc = nd.cg + 16 * t;
      double v = 0.0;
      if (prow >= 0 && qc < bk && qc >= fz) v = a.P[prow + (size_t)qc * a.lda];
      bad |= not_finite(v);
      nd.A[s][t] = v;
    }
  }
  if (bad && a.dev_info) atomicOr(a.dev_info + 1, CA_STATUS_NONFINITE);
#pragma unroll
  for (int t = 0; t < kCTC; ++t) nd.T[t] = 0.0;
  for (int i = tid; i < kCW; i += kRegThreads) sm.z[i] = 0.0;
  for (int i = tid; i < 2 * kCG * kCW; i += kRegThreads) (&sm.in[0][0][0])[i] = 0.0;  // columns from bk on
  for (int i = tid; i < 2 * kCW; i += kRegThreads) (&sm.row[0][0])[i] = 0.0;
  if (nd.cg == 0) {  // x_0
#pragma unroll
    for (int s = 0; s < TS; ++s) sm.xs[nd.rg + 16 * s] = nd.node_row(s) > 0 ? nd.A[s][0] : 0.0;
  }
  if (tid == 0) {
    for (int q = 0; q < 2; ++q)
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(&sm.bar[q])) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    for (int q = 0; q < 2; ++q)
      if (q < nd.kmax) bar_expect(&sm.bar[q], 8u * nd.bkw * (kCG + 1));
    sm.gave_up = 0;
  }
  // the zeros above come before the copies into the same buffers
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  cl.sync();  // every CTA's barriers are set up before anything is sent to them
  nd.template blocks<0>();
  tell_gave_up(cl, nd.dead, &sm.gave_up, nd.status);
  cl.sync();  // nothing is on its way to a CTA that has left; tau, scal and z are final
  if (cluster_gave_up(&sm.gave_up)) cl.sync();
  if (nd.kmax > 0) nd.t_column(nd.kmax - 1);

  // v = s x below the diagonal of every reflector column
#pragma unroll
  for (int t = 0; t < kCTC; ++t) {
    const int qc = nd.cg + 16 * t;
    if (qc < nd.kmax) {
      const double sq = sm.scal[qc];
#pragma unroll
      for (int s = 0; s < TS; ++s)
        if (nd.node_row(s) > qc) nd.A[s][t] *= sq;
    }
  }
  {
    const int b = a.b, i = 8 * nd.cg + rank;
    double *Tg = a.Tp + (size_t)(a.is_leaf ? node : a.nleaves + midx) * b * b;
    if (i < b) {
#pragma unroll
      for (int t = 0; t < kCTC; ++t) {
        const int qc = nd.rg + 16 * t;
        if (qc < b) Tg[i + (size_t)qc * b] = (i < nd.kmax && qc < nd.kmax && qc >= i) ? nd.T[t] : 0.0;
      }
      for (int qc = nd.rg + kCW; qc < b; qc += 16) Tg[i + (size_t)qc * b] = 0.0;  // a last panel narrower than b
    }
    constexpr int kTRows = 16 * kCG;  // one row of T per half-warp of the cluster
    if (rank == 0 && b > kTRows)      // b > 128 with at most 128 columns in the matrix: the rows past them
      for (size_t idx = tid; idx < (size_t)(b - kTRows) * b; idx += kRegThreads)
        Tg[kTRows + idx % (b - kTRows) + idx / (b - kTRows) * b] = 0.0;
  }
#pragma unroll
  for (int s = 0; s < TS; ++s) {
    int prow, fz;
    row_info(nd.node_row(s), prow, fz);
#pragma unroll
    for (int t = 0; t < kCTC; ++t) {
      const int qc = nd.cg + 16 * t;
      if (prow >= 0 && qc < bk && qc >= fz) a.P[prow + (size_t)qc * a.lda] = nd.A[s][t];
    }
  }
  if (rank == 0 && tid == 0) {
    a.top_out[node] = a.is_leaf ? r0 : a.top_in[start];
    a.c_out[node] = nd.kmax;
  }
}

template <int TC, int TS>
cudaError_t launch_creg(const TsqrNodeArgs &a, int nodes, cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(nodes * kCG);
  cfg.blockDim = dim3(kRegThreads);
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = kCG;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  TsqrNodeArgs args = a;
  args.wait_limit = panel_wait_limit();
  args.withhold = panel_withhold();
  return cudaLaunchKernelEx(&cfg, tsqr_creg_kernel<TC, TS>, args);
}

}  // namespace

bool tsqr_reg_fits(int rows, int bk) { return bk >= 1 && bk <= 64 && rows >= 1 && rows <= 256; }

// Cluster form: at most 128 columns and 1024 rows.  Nodes that fit one CTA run
// there while a round is small enough to finish sooner spread over 8 SMs each:
// TSQR of 1048576 x 64 takes 27.06 ms without it, 26.35 / 26.31 / 26.48 with
// up to 19 / 38 / 76 nodes; CAQR of 1024 x 1024 (8 nodes) 21.7 against 13.7 ms.
constexpr int kCregNodes = 38;

bool tsqr_creg_fits(int rows, int bk, int nodes) {
  if (bk < 1 || bk > 128 || rows < 1 || rows > 128 * kCG) return false;
  // (the shared-memory node sums x / (alpha - beta), this one x as it is, whose
  // products with a much smaller column may underflow: shapes that always had
  // the former keep it)
  if (bk > 64 && rows <= 128) return false;
  return !tsqr_reg_fits(rows, bk) || nodes <= kCregNodes;
}

cudaError_t launch_tsqr_creg(const TsqrNodeArgs &a, int nodes, int rows, cudaStream_t st) {
  if (a.bk > 64)
    return rows <= 32 * kCG   ? launch_creg<8, 2>(a, nodes, st)
           : rows <= 64 * kCG ? launch_creg<8, 4>(a, nodes, st)
                              : launch_creg<8, 8>(a, nodes, st);
  return rows <= 16 * kCG   ? launch_creg<4, 1>(a, nodes, st)
         : rows <= 32 * kCG ? launch_creg<4, 2>(a, nodes, st)
         : rows <= 64 * kCG ? launch_creg<4, 4>(a, nodes, st)
                            : launch_creg<4, 8>(a, nodes, st);
}

cudaError_t launch_tsqr_reg(const TsqrNodeArgs &a, int nodes, int rows, cudaStream_t st, bool *done) {
  *done = false;
  if (!tsqr_reg_fits(rows, a.bk)) return cudaSuccess;
  *done = true;
  if (a.bk <= 32) {
    if (rows <= 128) return launch_reg<2, 8>(a, nodes, st);
    return launch_reg<2, 16>(a, nodes, st);
  }
  if (rows <= 128) return launch_reg<4, 8>(a, nodes, st);
  return launch_reg<4, 16>(a, nodes, st);
}

// Test hook of the cluster nodes here and in panel_lu_reg.cu.
static std::atomic<long long> g_panel_wait{kPanelWait};
static std::atomic<int> g_panel_withhold{0};

long long panel_wait_limit() { return g_panel_wait.load(); }
int panel_withhold() { return g_panel_withhold.load(); }
void panel_test_hook(long long wait_cycles, int withhold) {
  g_panel_wait.store(wait_cycles > 0 ? wait_cycles : kPanelWait);
  g_panel_withhold.store(withhold);
}

}  // namespace cagb
