// panel_lu_reg.cu -- tournament nodes (GEPP of a leaf of the panel, or of the
// stacked candidate rows of a merge: Sec. 3.2) held in registers.
//
// A node's rows are split in contiguous chunks over the G CTAs of one cluster
// (G = 1, 2, 4, 8, 16).  TPR threads hold one row: thread `sub` of a row keeps the
// columns k TPR + sub, k < CPT, in registers.  Rows never move: every row
// carries the position it would have after the interchanges made so far (the
// rule "first maximum in the physically swapped order" needs it), and a row
// whose position is below the current column takes no further part.
// Per column j, from the published pivot row u and 1 / u_j:
//   * l = a_ij / u_j for every active row, column j + 1 updated first;
//   * every warp leaves its best (|a|, position) of column j + 1 in shared
//     memory, then runs most of the row update a_ik -= l u_k;
//   * after one CTA barrier every warp knows the CTA's best row; its warp
//     publishes the row, its key and its reciprocal once its own update is
//     done, while the others finish theirs.
// A node of one CTA waits for the row at a second CTA barrier.  In a cluster
// every CTA publishes its best row to all of them, and step j + 1 takes the
// best of the G rows: one exchange per column, no matter how many CTAs.  A row
// travels as one bulk copy per receiver, counted on its mbarrier: about 600
// clocks per exchange measured with 4 CTAs (the same row as 66 st.async stores
// of 16 bytes: 1000; two cluster barriers: 800 and the stores' flush).
// FP64 is the scarce resource here: a warp's multiply-add holds the FP64 pipe
// of its SM sub-partition for 64 clocks.  So everything but the update is kept
// off that pipe: keys compare as integers, rows are not swapped, the
// reciprocal is formed in integers, and warps whose rows are all chosen skip
// the update.
// The receive buffers are triple: a CTA publishes column j + 1 after it has
// received every row j; the sender of row j passed the CTA barrier of step
// j - 1, so all its warps are done with the rows j - 2 that the buffer held.
// Measured (single node, before: shared-memory cluster kernel): 1024 x 128
// 1310 -> 344 us, 512 x 128 520 -> 291 us, 128 x 64 200 -> 104 us, 96 x 96
// 362 -> 180 us; leaf and merge rounds of 1048576 x 64 12.9 -> 8.6 ms.
// The columns run in blocks of 4 TPR: register indices are constants inside a
// block, and after a block the registers move down by 4, so the code stays
// one block long and what is left of a row always starts at register 0.
// A waiter that sees a phase complete knows every warp of the cluster has
// passed its reads of the buffer two columns back: a warp publishes its key
// of column j + 1 after its last read of keys j and rows j - 1, the winner of
// column j + 1 exists only once every warp has published, and keys j + 2 are
// published only after row j + 1 has arrived.
#include <climits>

#include "ca_internal.cuh"
#include "cluster_copy.cuh"
#include "device_once.cuh"
#include "fp64_int.cuh"
#include "lu_node.cuh"

namespace cagb {

namespace {

struct alignas(16) Key {
  unsigned long long key;  // |a| bits
  int pos;
  int pad;
};

constexpr int kMaxG = 16;
constexpr int kMaxWarps = 16;

template <int TPR, int CPT, bool CL>
struct alignas(16) LuRegSmem {
  // a published row: its Key, 1 / pivot, a pad, then the threads' parts four
  // registers at a time (block, sub, 4)
  static constexpr int kRow = 4 + TPR * CPT;
  double u[CL ? 3 * kMaxG : 2][kRow];  // [column mod 3][rank] (one CTA: [column mod 2])
  double stage[CL ? 2 : 1][kRow];      // cluster: the CTA's row on its way out, by column parity
  Key keys[2][kMaxWarps];              // best of every warp of this CTA, by column parity
  unsigned long long bar[3];                  // cluster: the rows of a column have arrived
  int gave_up;                                // a CTA of the cluster gave up waiting
  int sel[128];                               // root, rank 0: labels of the chosen rows in pivot order
  int work[3 * 128];
};

// split barrier of the cluster (of the CTA when G = 1)
__device__ __forceinline__ void cl_arrive() {
  __syncwarp();
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cl_wait() {
  __syncwarp();
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// Largest key of the warp, smallest position among equal keys (on every lane).
__device__ __forceinline__ void warp_best(unsigned long long &key, int &pos) {
  const unsigned hi = (unsigned)(key >> 32);
  const unsigned mh = __reduce_max_sync(0xffffffffu, hi);
  const unsigned lo = hi == mh ? (unsigned)key : 0u;
  const unsigned ml = __reduce_max_sync(0xffffffffu, lo);
  const int p = (hi == mh && lo == ml) ? pos : INT_MAX;
  pos = __reduce_min_sync(0xffffffffu, p);
  key = ((unsigned long long)mh << 32) | ml;
}

// out of line, so that it is not computed beside the integer form every time
__device__ __noinline__ double recip_lib(double v) { return __drcp_rn(v); }

template <int TPR, int CPT, bool CL>
struct Node {
  cg::cluster_group cl;
  LuRegSmem<TPR, CPT, CL> &sm;
  int G, rank, nw, lane, warp, sub, kmax, kend;
  double a[CPT];
  int pos;  // position of the row after the interchanges so far; -1: no row
  bool dead = false;  // cluster: a wait gave up; nothing is waited for any more
  int *status;
  long long limit;
  int nsend;          // CTAs this one sends its rows to: G, or 0 after a give-up (test hook: always)

  __device__ __forceinline__ explicit Node(LuRegSmem<TPR, CPT, CL> &s) : cl(cg::this_cluster()), sm(s) {}

  // blocks of 4 registers per thread from column j's block to the row's end
  __device__ __forceinline__ int blocks(int j) const { return (kend + 3) / 4 - j / (4 * TPR); }

  static __device__ __forceinline__ unsigned row_bytes(int nb) { return 32u + 32u * TPR * nb; }

  __device__ __forceinline__ void expect(int j) {
    if (j < kmax) bar_expect(&sm.bar[j % 3], (unsigned)G * row_bytes(blocks(j)));
  }

  // this warp's best of column j
  __device__ __forceinline__ void post_key(int j, unsigned long long key, int p) {
    warp_best(key, p);
    if (lane == 0)
      *reinterpret_cast<uint4 *>(&sm.keys[j & 1][warp]) =
          make_uint4((unsigned)key, (unsigned)(key >> 32), (unsigned)p, 0u);
  }
  // the CTA's best of column j (after the barrier that follows post_key)
  __device__ __forceinline__ void best_of_cta(int j, unsigned long long &key, int &p) {
    key = 0;
    p = INT_MAX;
    if (lane < nw) {
      const uint4 e = *reinterpret_cast<const uint4 *>(&sm.keys[j & 1][lane]);
      key = ((unsigned long long)e.y << 32) | e.x;
      p = (int)e.z;
    }
    warp_best(key, p);
  }

  // Publishes the CTA's best row of column j: on the warp that holds it
  // (mine; `lead` holds its leading value v, r its reciprocal or 0), or, without a
  // candidate in this CTA, an empty key from warp 0.
  __device__ __forceinline__ void publish(int j, int nb, bool mine, bool lead, double v, double r,
                                          unsigned long long key, int p) {
    double *u = CL ? sm.stage[j & 1] : sm.u[j & 1];
    if (mine) {
#pragma unroll
      for (int c = 0; c < CPT / 4; ++c) {
        if (c >= nb) break;
        double2 *d = reinterpret_cast<double2 *>(u + 4 + 4 * (c * TPR + sub));
        d[0] = make_double2(a[4 * c], a[4 * c + 1]);
        d[1] = make_double2(a[4 * c + 2], a[4 * c + 3]);
      }
    }
    if (lead) {
      if (__double_as_longlong(r) == 0) r = recip_lib(v);  // an integer test: a compare of doubles is FP64 work
      u[2] = r;
    }
    if constexpr (CL) {
      if (lane == 0)
        *reinterpret_cast<uint4 *>(u) = make_uint4((unsigned)key, (unsigned)(key >> 32), (unsigned)p, 0u);
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // the copies read what was just written
      __syncwarp();
      const int b3 = j % 3;
      if (lane < nsend) bulk_to(sm.u[b3 * kMaxG + rank], u, row_bytes(nb), &sm.bar[b3], lane);
    }
  }

  // Waits for column j's rows; key and position of the pivot and its row.
  __device__ __forceinline__ const double *receive(int j, unsigned long long &key, int &p) {
    if constexpr (CL) {
      const int b3 = j % 3;
      if (!dead && !bar_wait(&sm.bar[b3], (j / 3) & 1, limit)) {
        dead = true;
        nsend = 0;
      }
      if (threadIdx.x == 0 && !dead) expect(j + 3);
      unsigned long long mk = 0;
      int mp = INT_MAX;
      if (lane < G) {
        const uint4 e = *reinterpret_cast<const uint4 *>(sm.u[b3 * kMaxG + lane]);
        mk = ((unsigned long long)e.y << 32) | e.x;
        mp = (int)e.z;
      }
      key = mk;
      p = mp;
      warp_best(key, p);
      const unsigned who = __ballot_sync(0xffffffffu, lane < G && mk == key && mp == p);
      return sm.u[b3 * kMaxG + (who ? __ffs(who) - 1 : 0)];
    } else {
      __syncthreads();
      return sm.u[j & 1];  // key and p are the CTA's best
    }
  }

  // a_ik -= l u_k for registers 4 C .. 4 C + 7 from K0 on; the second four
  // only when that block is left of the row's end
  template <int C, int K0>
  __device__ __forceinline__ void update8(const double *u, double l, int nb) {
    double2 w[4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if (4 * C + 2 * i < CPT) w[i] = *reinterpret_cast<const double2 *>(u + 4 * TPR * (C + (i >> 1)) + 2 * (i & 1));
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int k = 4 * C + 2 * i;
      if (k >= CPT) break;
      if (i == 2 && C + 1 >= nb) break;
      if (k >= K0) a[k] = fma(-l, w[i].x, a[k]);
      if (k + 1 >= K0) a[k + 1] = fma(-l, w[i].y, a[k + 1]);
    }
  }

  // State of the column loop.
  struct Run {
    int j, nb;               // column; blocks of 4 registers from the current one to the row's end
    unsigned long long key;  // the CTA's best of column j
    int p;
    bool early;              // every warp prepares its candidate's reciprocal
    double v, r;             // this thread's value of column j (where sub holds it), its reciprocal
    double aj;               // column j of this row
    int *info;               // root: where a zero column is recorded (or null)
    int ipiv_base;
    double *keep;            // root: this row's place for finished registers (or null)
  };

  // Columns of register Q of the current block; false after the last column.
  template <int Q>
  __device__ __forceinline__ bool group(Run &s) {
#pragma unroll 1
    for (int h = 0; h < TPR; ++h) {
      const int j = s.j, nb = s.nb;
      {
        const bool mine = s.key != 0ull && pos == s.p;
        if (__any_sync(0xffffffffu, mine) || (CL && s.key == 0ull && warp == 0)) {
          if (!s.early) s.r = recip_exact_or_zero(s.v);
          publish(j, nb, mine, mine && sub == h, s.v, s.r, s.key, s.p);
        }
      }
      const double *ur = receive(j, s.key, s.p);
      const double *u = ur + 4 + 4 * sub;  // register k at 4 TPR (k / 4) + k mod 4
      // a column without a non-zero candidate: nothing changes
      const bool zero = s.key == 0ull;
      if (!zero) pos = pos == s.p ? j : pos == j ? s.p : pos;
      const bool act = pos > j && !zero;
      double l = 0.0;
      if (act) {
        const double u0 = u[Q], u1 = Q < 3 ? u[Q + 1] : u[4 * TPR];
        l = s.aj * ur[2];
        if (sub == h) a[Q] = l;
        if (sub > h) a[Q] = fma(-l, u0, a[Q]);
        a[Q + 1] = fma(-l, u1, a[Q + 1]);
      }
      if (zero && s.info) atomicCAS(s.info, 0, s.ipiv_base + j + 1);
      const bool more = j + 1 < kmax;
      const bool wrap = h + 1 == TPR;
      const int sn = wrap ? 0 : h + 1;  // sub of column j + 1, in register Q or Q + 1
      s.v = wrap ? a[Q + 1] : a[Q];
      if (more) {
        const bool cand = pos > j && sub == sn;
        post_key(j + 1, cand ? absbits(s.v) : 0ull, cand ? pos : INT_MAX);
      }
      s.aj = TPR > 1 ? __shfl_sync(0xffffffffu, s.v, sn, TPR) : s.v;
      if (s.early) s.r = recip_exact_or_zero(s.v);
      if (act) {
#pragma unroll
        for (int k = Q + 2; k < 4; ++k) a[k] = fma(-l, u[k], a[k]);
        if (CPT > 12 && nb > 3) update8<3, 12>(u, l, nb);
        if (CPT > 20 && nb > 5) update8<5, 20>(u, l, nb);
        if (CPT > 28 && nb > 7) update8<7, 28>(u, l, nb);
      }
      if (more) {
        __syncthreads();
        best_of_cta(j + 1, s.key, s.p);
      }
      if (act && nb > 1) update8<1, (Q == 3 ? 5 : 4)>(u, l, nb);
      if (!more) {
        if (s.keep) *s.keep = a[Q];
        return false;
      }
      s.j = j + 1;
    }
    if (s.keep) {
      *s.keep = a[Q];
      s.keep += TPR;
    }
    return true;
  }

  // Every column.
  __device__ __forceinline__ void columns(Run &s) {
    s.j = 0;
    s.nb = blocks(0);
    s.v = a[0];
    s.r = recip_exact_or_zero(s.v);
    s.aj = TPR > 1 ? __shfl_sync(0xffffffffu, s.v, 0, TPR) : s.v;
    // few warps: every warp has its own candidate's reciprocal ready when the
    // best is known; many: one warp forms it then, and the others keep the
    // issue slots
    s.early = nw <= 4;
    const bool cand = pos >= 0 && sub == 0;
    post_key(0, cand ? absbits(s.v) : 0ull, cand ? pos : INT_MAX);
    __syncthreads();
    best_of_cta(0, s.key, s.p);
#pragma unroll 1
    while (group<0>(s) && group<1>(s) && group<2>(s) && group<3>(s)) {
#pragma unroll
      for (int k = 0; k + 4 < CPT; ++k) a[k] = a[k + 4];
      --s.nb;
    }
  }
};

// rows per CTA
template <int TPR, int CPT>
constexpr int lu_reg_rows() {
  return TPR * CPT > 64 ? 128 : TPR == 4 ? 64 : 256;
}

template <int TPR, int CPT, bool CL>
__global__ void __launch_bounds__(lu_reg_rows<TPR, CPT>() * TPR, CPT == 16 && TPR < 4 ? 2 : 1) tslu_reg_kernel(TsluNodeArgs a) {
  if (a.skip && *a.skip) return;  // every CTA of the cluster reads the same word
  __shared__ LuRegSmem<TPR, CPT, CL> sm;
  Node<TPR, CPT, CL> nd(sm);
  const int tid = threadIdx.x;
  nd.G = (int)nd.cl.num_blocks();
  nd.rank = (int)nd.cl.block_rank();
  nd.lane = tid & 31;
  nd.warp = tid >> 5;
  nd.nw = blockDim.x >> 5;
  nd.sub = tid & (TPR - 1);
  const int node = blockIdx.x / nd.G;
  const int bk = a.bk;
  const int row = tid / TPR;
  const int p = nd.rank * a.rloc + row;  // the row's position in the node

  // ---- node inputs: the row's label (panel row) --------------------------
  int R, lab = -1, start = 0, cnt = 1, midx = 0;
  if (a.is_leaf) {
    const int r0 = node * a.leaf_rows;
    R = min(a.leaf_rows, a.mk - r0);
    if (row < a.rloc && p < R) lab = r0 + p;
  } else {
    round_node(a.rd, node, start, cnt, midx);
    if (cnt == 1) {  // promotion: the candidate set passes through unchanged
      if (nd.rank == 0) {
        const int c = a.ncand_in[start];
        for (int i = tid; i < c; i += blockDim.x)
          a.cand_out[(size_t)node * a.cand_ld + i] = a.cand_in[(size_t)start * a.cand_ld + i];
        if (tid == 0) a.ncand_out[node] = c;
      }
      return;
    }
    R = 0;
    for (int ch = 0; ch < cnt; ++ch) {
      const int c = a.ncand_in[start + ch];
      if (row < a.rloc && p >= R && p < R + c) lab = a.cand_in[(size_t)(start + ch) * a.cand_ld + (p - R)];
      R += c;
    }
  }
  nd.kmax = min(R, bk);
  nd.kend = (bk + TPR - 1) / TPR;
  nd.pos = lab >= 0 ? p : -1;

  // ---- the row's original panel values ------------------------------------
  bool bad = false;
#pragma unroll
  for (int k = 0; k < CPT; ++k) {
    const int col = k * TPR + nd.sub;
    double v = 0.0;
    if (lab >= 0 && col < bk) v = a.P[lab + (size_t)col * a.lda];
    bad |= not_finite(v);
    nd.a[k] = v;
  }
  if (bad && a.dev_info) atomicOr(a.dev_info + 1, CA_STATUS_NONFINITE);

  // ---- column 0's pivot row, then every column ----------------------------
  nd.status = a.dev_info ? a.dev_info + 1 : nullptr;
  nd.limit = a.wait_limit;
  nd.nsend = a.withhold && nd.rank == nd.G - 1 ? 0 : nd.G;
  if constexpr (CL) {
    if (tid == 0) {
      for (int q = 0; q < 3; ++q)
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(&sm.bar[q])) : "memory");
      asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
      for (int q = 0; q < 3; ++q) nd.expect(q);
      sm.gave_up = 0;
    }
    cl_arrive();  // the barriers of every CTA are set up before anything is sent to them
    cl_wait();
  }
  extern __shared__ __align__(16) double keep[];  // root: rows x columns, odd row length
  const int ldk = (a.bk + TPR - 1) / TPR * TPR | 1;
  typename Node<TPR, CPT, CL>::Run run;
  run.info = (a.is_root && nd.rank == 0 && tid == 0) ? a.dev_info : nullptr;
  run.ipiv_base = a.ipiv_base;
  run.keep = a.is_root && lab >= 0 ? keep + (size_t)row * ldk + nd.sub : nullptr;
  nd.columns(run);

  // ---- outputs: labels in pivot order; root: L11 \ U11 of the chosen rows ---
  auto outputs = [&] {
    const bool chosen = nd.pos >= 0 && nd.pos < nd.kmax;
    if (chosen && nd.sub == 0) a.cand_out[(size_t)node * a.cand_ld + nd.pos] = lab;
    if (nd.rank == 0 && tid == 0) a.ncand_out[node] = nd.kmax;
    if (!a.is_root || !chosen) return;
    for (int col = nd.sub; col < bk; col += TPR) a.lu11[nd.pos + (size_t)col * a.cand_ld] = keep[(size_t)row * ldk + col];
    if (nd.sub == 0) *nd.cl.map_shared_rank(&sm.sel[nd.pos], 0) = lab;
  };
  outputs();
  if constexpr (CL) tell_gave_up(nd.cl, nd.dead, &sm.gave_up, nd.status);
  if (CL || a.is_root) {  // nothing is on its way to a CTA that has left; rank 0 holds every chosen label
    cl_arrive();
    cl_wait();
  }
  if constexpr (CL)
    if (cluster_gave_up(&sm.gave_up)) {
      // positions may be anything: the node's first rows stand in for the
      // choice (valid labels, each once; the status tells)
      nd.pos = lab >= 0 ? p : -1;
      outputs();
      cl_arrive();
      cl_wait();
    }
  if (!a.is_root) return;
  if (nd.rank == 0 && tid < 32) lu_root_swaps(a, sm.sel, sm.work);
}

constexpr int kKeepBytes = (128 * 129 > 256 * 65 ? 128 * 129 : 256 * 65) * 8;  // most dynamic shared memory (root)

// Whether the current device can place a cluster of kMaxG CTAs of this kernel
// (more than the portable 8, so it depends on the device and its partition),
// asked once per device, for the largest shape it is launched with.
template <int TPR, int CPT>
bool big_cluster_fits() {
  static std::atomic<unsigned long long> asked{0}, fits{0};
  const cudaError_t e = once_per_device(asked, [] {
    auto *fn = tslu_reg_kernel<TPR, CPT, true>;
    cudaError_t r = cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (r == cudaSuccess) r = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, kKeepBytes);
    int dev = 0, n = 0;
    if (r == cudaSuccess) r = cudaGetDevice(&dev);
    if (r == cudaSuccess) {
      cudaLaunchConfig_t cfg = {};
      cfg.gridDim = dim3(kMaxG);
      cfg.blockDim = dim3(lu_reg_rows<TPR, CPT>() * TPR);
      cfg.dynamicSmemBytes = kKeepBytes;
      cudaLaunchAttribute at[1];
      at[0].id = cudaLaunchAttributeClusterDimension;
      at[0].val.clusterDim.x = kMaxG;
      at[0].val.clusterDim.y = 1;
      at[0].val.clusterDim.z = 1;
      cfg.attrs = at;
      cfg.numAttrs = 1;
      if (cudaOccupancyMaxActiveClusters(&n, fn, &cfg) != cudaSuccess) {
        cudaGetLastError();  // a refusal is an answer, not a failure of the call that asks
        n = 0;
      }
      if (n > 0 && dev < kMaxDevices) fits.fetch_or(1ull << dev, std::memory_order_relaxed);
    }
    return r;
  });
  int dev = 0;
  return e == cudaSuccess && cudaGetDevice(&dev) == cudaSuccess && dev < kMaxDevices &&
         (fits.load(std::memory_order_relaxed) >> dev & 1ull);
}

bool big_cluster_fits(int bk, int rloc) {  // of the kernel that launch_tslu_reg takes
  if (bk <= 16) return big_cluster_fits<1, 16>();
  if (bk <= 32) return big_cluster_fits<2, 16>();
  if (bk <= 64) return rloc <= 64 ? big_cluster_fits<4, 16>() : big_cluster_fits<2, 32>();
  return big_cluster_fits<4, 32>();
}

template <int TPR, int CPT, bool CL>
cudaError_t launch_reg1(const TsluNodeArgs &a, int nodes, int G, cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(nodes * G);
  cfg.blockDim = dim3((a.rloc * TPR + 31) / 32 * 32);
  cfg.stream = st;
  if (a.is_root) {
    static std::atomic<unsigned long long> init{0};
    cudaError_t e = once_per_device(init, [] {
      return cudaFuncSetAttribute(tslu_reg_kernel<TPR, CPT, CL>, cudaFuncAttributeMaxDynamicSharedMemorySize, kKeepBytes);
    });
    if (e != cudaSuccess) return e;
    cfg.dynamicSmemBytes = (size_t)a.rloc * ((a.bk + TPR - 1) / TPR * TPR | 1) * 8;
  }
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = G;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  TsluNodeArgs args = a;
  args.wait_limit = panel_wait_limit();
  args.withhold = panel_withhold();
  return cudaLaunchKernelEx(&cfg, tslu_reg_kernel<TPR, CPT, CL>, args);
}

template <int TPR, int CPT>
cudaError_t launch_reg(const TsluNodeArgs &a, int nodes, int G, cudaStream_t st) {
  return G > 1 ? launch_reg1<TPR, CPT, true>(a, nodes, G, st) : launch_reg1<TPR, CPT, false>(a, nodes, G, st);
}

}  // namespace

static std::atomic<int> g_max_cluster{16};  // test hook

void tslu_test_max_cluster(int n) { g_max_cluster.store(n > 0 ? n : 16); }

// Cluster size of a node of R rows and bk columns (a round of `nodes`), and
// the rows per CTA; 0 when the rows do not fit the registers of 8 CTAs.  The
// smallest cluster that holds the rows, doubled while the round's CTAs still
// find an SM each and a CTA keeps at least kMinRows rows (128 x 64: 125 us on
// one CTA, 121 on 2, 104 on 4, 109 on 8; 256 x 64: 201, 150, 123, 109).
// Sixteen CTAs (beyond the portable cluster size, so never needed to hold the
// rows, and only where the device can place such clusters) for rounds that
// fill at most two thirds of the SMs (six nodes of 152): 1024 x 128
// 471 -> 344 us, 512 x 128 317 -> 291.  The result does not depend on G.
int tslu_reg_cluster(int R, int bk, int nodes, int *rloc) {
  if (bk < 1 || bk > 128 || R < 1) return 0;
  const int rmax = bk <= 64 ? 256 : 128;
  constexpr int kMinRows = 24;
  int sms = 0, G = 1;
  if (device_sm_count(&sms) != cudaSuccess) return 0;
  while (G < 8 && (R + G - 1) / G > rmax) G *= 2;
  if ((R + G - 1) / G > rmax) return 0;
  while (G < 8 && (long long)nodes * G * 2 <= sms && (R + 2 * G - 1) / (2 * G) >= kMinRows) G *= 2;
  if (G == 8 && (long long)nodes * kMaxG * 3 <= 2 * sms && (R + kMaxG - 1) / kMaxG >= kMinRows &&
      g_max_cluster.load() >= kMaxG && big_cluster_fits(bk, (R + kMaxG - 1) / kMaxG))
    G = kMaxG;
  *rloc = (R + G - 1) / G;
  return G;
}

cudaError_t launch_tslu_reg(const TsluNodeArgs &a, int nodes, int G, cudaStream_t st) {
  if (a.bk <= 16) return launch_reg<1, 16>(a, nodes, G, st);
  if (a.bk <= 32) return launch_reg<2, 16>(a, nodes, G, st);
  // up to 64 rows four threads share a row (128 x 64 on 4 CTAs 104 us, with two
  // threads 139); with more rows two (256 x 64 on one CTA 201 us): every warp
  // instruction that is not part of the update costs the FP64 pipe per warp
  if (a.bk <= 64) return a.rloc <= 64 ? launch_reg<4, 16>(a, nodes, G, st) : launch_reg<2, 32>(a, nodes, G, st);
  return launch_reg<4, 32>(a, nodes, G, st);
}

}  // namespace cagb
