// lu_node.cuh -- what the tournament-node kernels (panel_lu.cu, panel_lu_reg.cu) share.
#pragma once
#include "ca_internal.cuh"

namespace cagb {

struct TsluNodeArgs {
  const double *P;  // panel (row 0 = first row of the panel), ld lda
  int lda, mk, bk;
  int leaf_rows;
  int is_leaf;      // nodes of this launch are the leaves
  int is_root;      // the single node of this launch is the root
  RoundDesc rd;     // merge round (when !is_leaf)
  const int *cand_in;
  const int *ncand_in;
  int *cand_out;
  int *ncand_out;
  int cand_ld;      // ints per node in the candidate buffers (= b)
  int rloc;         // rows per CTA
  // root outputs
  double *lu11;     // bk x bk, ld cand_ld
  int *perm_src, *perm_dst, *perm_cnt;
  int *ipiv_k;      // ipiv + kb
  int ipiv_base;    // kb
  const int *skip;  // nonzero: a stage enqueued ahead that is not needed, do nothing
  int *dev_info;    // [0] info, [1] status
  long long wait_limit;  // register nodes: SM clocks a wait may take
  int withhold;          // test hook: the last CTA of a cluster sends nothing
};

// register-resident nodes (panel_lu_reg.cu)
int tslu_reg_cluster(int R, int bk, int nodes, int *rloc);
cudaError_t launch_tslu_reg(const TsluNodeArgs &a, int nodes, int G, cudaStream_t st);

// The panel's swap sequence and net row permutation from the labels sel[0..bk)
// of the chosen rows in pivot order (one warp; work: 3 bk ints of shared
// memory).  LAPACK order: at step i, position i and the current position of
// the i-th chosen row are interchanged.
__device__ inline void lu_root_swaps(const TsluNodeArgs &a, const int *sel, int *work) {
  const int bk = a.bk;
  const int lane = threadIdx.x & 31;
  int *rev_top = work;          // position of top label x (>= 0) or -(slot + 1)
  int *top_c = work + bk;       // label at top position t
  int *far_c = work + 2 * bk;   // label at far position sel[s] (sel[s] >= bk)
  for (int t = lane; t < bk; t += 32) {
    rev_top[t] = t;
    top_c[t] = t;
    far_c[t] = sel[t];
  }
  __syncwarp();
  if (lane == 0)
  for (int i = 0; i < bk; ++i) {
    const int L = sel[i];
    int pp, fslot = -1;
    if (L < bk) {
      const int r = rev_top[L];
      if (r >= 0) {
        pp = r;
      } else {
        fslot = -r - 1;
        pp = sel[fslot];
      }
    } else {
      pp = L;
      fslot = i;
    }
    a.ipiv_k[i] = a.ipiv_base + pp + 1;
    if (pp == i) continue;
    const int Ci = top_c[i];
    top_c[i] = L;
    if (pp < bk) {
      top_c[pp] = Ci;
      rev_top[Ci] = pp;
    } else {
      far_c[fslot] = Ci;
      rev_top[Ci] = -(fslot + 1);
    }
    if (L < bk) rev_top[L] = i;
  }
  __syncwarp();
  int n = 0;
  auto add = [&](bool some, int dst, int src) {
    const unsigned m = __ballot_sync(0xffffffffu, some);
    if (some) {
      const int at = n + __popc(m & ((1u << lane) - 1u));
      a.perm_dst[at] = dst;
      a.perm_src[at] = src;
    }
    n += __popc(m);
  };
  for (int t0 = 0; t0 < bk; t0 += 32) {
    const int t = t0 + lane;
    const bool in = t < bk;
    const int c = in ? top_c[t] : 0, s = in ? sel[t] : 0, f = in ? far_c[t] : 0;
    add(in && c != t, t, c);
    add(in && s >= bk, s, f);
  }
  if (lane == 0) *a.perm_cnt = n;
}

}  // namespace cagb
