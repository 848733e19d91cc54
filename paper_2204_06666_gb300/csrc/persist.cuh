// Device code of the persistent solver kernels (cg.cu, pcg.cu): a whole Krylov iteration, and then the next,
// inside one cooperative launch with one block per partition.
//
// A solver iteration as separate launches re-reads what the block that owns a partition has just had in hand:
// the direction is staged into shared memory for every product, q and r go through memory between the product
// and the updates, and every launch drains and refills the chip (tet 80^3, 512k rows: product 29 us, update 14
// us, direction 5 us cold, 44 us an iteration back to back from a graph, for 74 MB of matrix).  Here a block keeps
// its partition's slices of the vectors in shared memory from one iteration to the next, as many of them as fit,
// and the iteration's inner products double as the barriers that the data dependences need.  Scalars (a division
// is a dozen dependent FP64 operations, and FP64 operations of 32 warps queue for one unit) are one thread's work.
// Whole solves of (A + 0.1 mean diagonal) x = b to 1e-10, separate launches -> persistent, FP64 CG (40 to 66
// iterations): tet 20^3 0.96 -> 0.61 ms, 40^3 1.11 -> 0.76, 80^3 2.06 -> 1.56, 126^3 4.55 -> 4.19, elasticity 24^3 1.86 ->
// 1.34, 48^3 5.19 -> 4.90, 70^3 10.87 -> 10.75; elasticity 30^3 (81k rows, bound by 17 slices on four quarters of an SM)
// 2.54 both.  Mixed-precision PCG: tet 80^3 2.13 -> 1.53, elasticity 40^3 3.56 -> 2.90, 70^3 8.33 -> 7.70; FP64 PCG: tet 80^3 1.76 -> 1.25, elasticity 70^3 11.69 -> 11.45.  A third of the tet 80^3 iteration is still outside the product: FP64
// vector arithmetic (five FMAs a row, 4.4 us at the pipe's rate) and the three meetings.
#pragma once
#include "ehyb_core.cuh"

namespace ehyb {
namespace persist {

using namespace core;

constexpr int kMaxGrid = 160;      // blocks of a persistent launch (five partial sums per gathering lane)
constexpr uint64_t kMinLimitNs = 2000000000ull;  // least time limit of a wait for the other blocks
constexpr int kAborted = 2;

// One block's partial sum: the halves of a double, each beside the number of its round in an 8-byte word of its own, so
// that a reader sees for each half whether it is the one it waits for.
struct __align__(16) Slot {
  unsigned long long lo, hi;
};

// The memory the blocks meet in, all zero at launch.
struct Meeting {
  Slot slot[2][kMaxGrid];    // partial sums of the even and the odd rounds of sums
  int32_t summed, pad0[31];  // blocks that have published, over all rounds of sums
  int32_t arrived, pad1[31]; // arrivals at the plain rounds
};

struct SyncArgs {
  Meeting* m;
  int32_t* status;            // the plan's status word: EHYB_ERR_TIMEOUT when a wait ran out
  int32_t* done;              // set to kAborted with it, so that the host stops launching
  uint64_t limit_ns;
};

// Shared memory of a persistent block, out of the SM's 256 KB that the rest of L1 shares: the least of the sizes the
// hardware can set aside that holds `must` bytes (what the kernel cannot do without), less what the system and the
// kernel's own variables take; the vectors beyond it go there only as far as they fit.  The extra rows gather freshly
// written vectors through L1, so a vector kept in shared memory at L1's cost loses more than it saves: at elasticity
// 64^3 (41 KB a vector) the FP64 PCG took 23.1 ms a solve with five vectors in shared memory (215 KB), 9.5 with two
// (separate launches 9.8); scalar hexahedra 80^3 with BF16 G 3.0 and 1.9 ms (2.4).  0: more than 196 KB, where
// the separate launches are the faster form (tet 126^3, FP64 G, two vectors of 105 KB: 4.9 ms against 3.9).
inline size_t shared_budget(size_t must) {
  for (size_t kb : {100, 132, 164, 196})
    if (must + 3072 <= kb * 1024) return kb * 1024 - 3072;
  return 0;
}

// Rows of a partition up to which FP32 iterations run persistently.  Beyond, the FP32 products are short of bytes rather
// than of launches, and the vectors' passes of the separate launches are the faster ones (us an iteration, separate ->
// persistent: tet 102^3, 6,982 rows, CG 42.8 -> 39.5, mixed PCG 85.4 -> 79.9; tet 114^3, 9,747 rows, 50.8 -> 52.1 and
// 99.9 -> 106.8; tet 126^3 61.0 -> 65.3 and 127.1 -> 139.7; FP64 iterations gain there: CG 93.6 -> 85.4, PCG 203.7 -> 202.3).
constexpr int kMaxRows32 = 8192;

__device__ __forceinline__ void fence_acq_rel() { asm volatile("fence.acq_rel.gpu;" ::: "memory"); }

// a wait that has lasted: true when it must give up (its limit is over, or another block gave up)
struct Patience {
  uint64_t t0 = 0;
  int spins = 0;
  __device__ __forceinline__ bool over(const SyncArgs& g) {
    if ((++spins & 63) != 0) return false;
    const uint64_t t = globaltimer_ns();
    if (t0 == 0) t0 = t;
    return t - t0 > g.limit_ns || *(volatile int32_t*)g.status == kTimeoutCode;
  }
};
__device__ __forceinline__ void give_up(const SyncArgs& g) {
  atomicCAS(g.status, 0, kTimeoutCode);
  *(volatile int32_t*)g.done = kAborted;
}

// wait until all blocks have added `round` (1, 2, ...) times to the counter; false: gave up.  ACQUIRE: what they
// wrote before adding (with a release) is visible then.
template <bool ACQUIRE>
__device__ __forceinline__ bool wait_at(const SyncArgs& g, const int32_t* counter, int round) {
  const int target = round * (int)gridDim.x;
  Patience wait;
  for (;;) {
    int v;
    if (ACQUIRE) asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(counter) : "memory");
    else asm volatile("ld.relaxed.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(counter) : "memory");
    if (v >= target) return true;
    if (wait.over(g)) {
      give_up(g);
      return false;
    }
  }
}

// Sum over all threads of all blocks, which is a grid-wide barrier too, in two halves so that a block can work in
// between.  Every thread has put its term into red[threadIdx.x] and passed a __syncthreads; then, for the launch's
// sums number round = 1, 2, ...:
//   publish_sum (the block's first four warps): the block's sum into its slot, then one more on the counter;
//   gather_sum (warp 0): waits for the counter, then adds the slots, lane-strided, then an xor tree: every block
//     gets the same bits.  False when a wait ran out (every wait is bounded).
// With ORDER whatever a block wrote before it published is visible after the gather.  Without, no fence is paid
// for (one costs half a microsecond to a microsecond behind a product): the counter is only the sign that
// looking is worth while, the rounds in the slots tell whether a value is there.  Polling the one counter and
// reading the slots once beats polling the slots (152 blocks, nothing else to do: 1.9 against 3.5 to 4.9 us;
// many lines, written by stores and polled by all, against one atomic).  An FP64 instruction occupies its
// quarter of the SM for 64 cycles however few lanes need it, so the block's sum is spread over one warp in each
// quarter (eight adds, a tree, three adds), not a tree in every warp.  Two sets of slots take turns: a block
// writes round + 2 only after all published round + 1, hence have read `round`.
constexpr int kSumWarps = 4;
template <bool ORDER>
__device__ __forceinline__ void publish_sum(const SyncArgs& g, int round, double* red) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, bd = blockDim.x;
  const int sw = min(kSumWarps, bd >> 5);
  double v = red[tid];
  for (int i = tid + 32 * sw; i < bd; i += 32 * sw) v += red[i];
  for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(FULL, v, off);
  if (sw > 1) {  // every term has been read before the warps' sums take their place
    asm volatile("bar.sync 1, %0;" ::"r"(32 * sw) : "memory");
    if (lane == 0) red[warp] = v;
    asm volatile("bar.sync 1, %0;" ::"r"(32 * sw) : "memory");
    if (warp > 0) return;
    v = red[0] + red[1];
    if (sw > 2) v += sw > 3 ? red[2] + red[3] : red[2];
  }
  if (lane == 0) {
    const unsigned long long bits = (unsigned long long)__double_as_longlong(v), tag = (unsigned long long)round << 32;
    if (ORDER) fence_acq_rel();
    asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(&g.m->slot[round & 1][blockIdx.x]),
                 "l"(tag | (bits & 0xffffffffull)), "l"(tag | (bits >> 32))
                 : "memory");
    asm volatile("red.relaxed.gpu.global.add.s32 [%0], 1;" ::"l"(&g.m->summed) : "memory");
  }
}
template <bool ORDER>
__device__ __forceinline__ bool gather_sum(const SyncArgs& g, int round, double* sum) {
  const int lane = threadIdx.x, nb = gridDim.x;
  const bool ok = lane > 0 || wait_at<false>(g, &g.m->summed, round);
  if (!__all_sync(FULL, ok)) return false;
  const Slot* slot = g.m->slot[round & 1];
  unsigned long long lo[kMaxGrid / 32], hi[kMaxGrid / 32];
  Patience wait;
  for (;;) {
    bool all = true;
#pragma unroll
    for (int k = 0; k < kMaxGrid / 32; ++k) {
      lo[k] = hi[k] = 0;
      if (lane + 32 * k < nb)
        asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];"
                     : "=l"(lo[k]), "=l"(hi[k])
                     : "l"(slot + lane + 32 * k)
                     : "memory");
    }
#pragma unroll
    for (int k = 0; k < kMaxGrid / 32; ++k)
      if (lane + 32 * k < nb) all = all && (int)(lo[k] >> 32) == round && (int)(hi[k] >> 32) == round;
    if (__all_sync(FULL, all)) break;
    if (__any_sync(FULL, wait.over(g))) {
      if (lane == 0) give_up(g);
      return false;
    }
  }
  if (ORDER) fence_acq_rel();
  double s = 0.0;
#pragma unroll
  for (int k = 0; k < kMaxGrid / 32; ++k)
    s += __longlong_as_double((long long)((hi[k] << 32) | (lo[k] & 0xffffffffull)));
  for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(FULL, s, off);
  *sum = s;
  return true;
}

// Barrier without a value, in two halves: arrive (one thread, after a __syncthreads that follows the block's writes) and a
// wait that each warp makes when it first needs the other blocks' writes, usually long after all have arrived.
// round: 1, 2, ... within the launch.  seen: the last round this block knows to be complete, in shared memory.
__device__ __forceinline__ void arrive(const SyncArgs& g) {
  asm volatile("red.release.gpu.global.add.s32 [%0], 1;" ::"l"(&g.m->arrived) : "memory");
}
__device__ __forceinline__ bool wait_round(const SyncArgs& g, int round, int* seen) {
  int known;
  asm volatile("ld.acquire.cta.shared.s32 %0, [%1];" : "=r"(known) : "r"(smem_addr(seen)) : "memory");
  known = __shfl_sync(FULL, known, 0);
  if (known >= round) return true;
  if (known < 0) return false;  // another warp gave up
  const bool ok = __all_sync(FULL, wait_at<true>(g, &g.m->arrived, round));
  if ((threadIdx.x & 31) == 0) {
    const int now = ok ? round : -1;
    asm volatile("st.release.cta.shared.s32 [%0], %1;" ::"r"(smem_addr(seen)), "r"(now) : "memory");
  }
  __syncwarp();
  return ok;
}

// One product of a block: what run_slices needs of the plan, the partition and the vectors.  It lies in shared memory,
// and run_slices is a function of its own: a persistent kernel holds several loops that need every register, and
// what the compiler keeps in registers across them (parameters, addresses) it would have to spill, to come back
// from L2 each time since the barriers' fences empty L1.
template <typename V, typename X>
struct Product {
  const V *ell_val, *er_val;
  const uint16_t* ell_col;
  const int32_t *er_col, *slice_order;
  const int64_t *slice_pos, *er_slice_pos;
  const X* xg;              // x in memory, for the extra rows
  X *out, *mirror;          // out[m] = sum of the row; mirror (optional): the same in memory
  const int32_t* n2o;       // m = n2o[row] - pb (optional: m = row)
  const uint16_t* er_hcol;  // staged extra rows (else null): 16-bit columns into x staged at `halo`
  const int32_t* halo;
  const SliceMeta* tbl;     // slice table, or null: the metadata is read from memory
  int32_t *status, *stop, *seen;
  int64_t n_x;
  int32_t xs_off, lim;      // x in shared memory: byte offset of the slice (by local column), its elements
  int32_t xh_off, nh;       // staged extra rows: byte offset, columns
  int32_t rows, s0, s1, tpr_log2, pb, meta_cap, counter;
};

// thread 0 fills pr for partition p of the plan of `a` (tbl: room for its slice table, or null); all threads the table
template <typename V, typename X>
__device__ __forceinline__ void init_product(Product<V, X>* pr, const KArgs& a, const V* ev, const V* erv,
                                             const int32_t* ecol, int p, SliceMeta* tbl) {
  const int s0 = a.slice_ptr[p], ns = a.slice_ptr[p + 1] - s0;
  if (threadIdx.x == 0) {
    pr->ell_val = ev;
    pr->er_val = erv;
    pr->ell_col = a.ell_col;
    pr->er_col = ecol;
    pr->slice_order = a.slice_order;
    pr->slice_pos = a.slice_pos;
    pr->er_slice_pos = a.er_slice_pos;
    pr->mirror = nullptr;
    pr->n2o = nullptr;
    pr->er_hcol = nullptr;
    pr->nh = 0;
    pr->tbl = tbl;
    pr->status = a.status;
    pr->n_x = a.n_x;
    pr->pb = a.part_ptr[p];
    pr->rows = pr->lim = a.part_ptr[p + 1] - a.part_ptr[p];
    pr->s0 = s0;
    pr->s1 = s0 + ns;
    pr->tpr_log2 = a.tpr_log2;
    pr->meta_cap = a.meta_cap;
  }
  if (!tbl) return;
  for (int t = threadIdx.x; t < ns; t += blockDim.x) {
    const int sl = a.slice_order[s0 + t];
    SliceMeta m;
    m.pos = a.slice_pos[sl];
    m.w = (int)((a.slice_pos[sl + 1] - m.pos) >> 5);
    m.epos = a.er_slice_pos[sl];
    m.we = (int)((a.er_slice_pos[sl + 1] - m.epos) >> 5);
    m.s = sl;
    m.pad = 0;
    tbl[checked(t, a.meta_cap, a.status)] = m;
  }
}

// thread 0: pr reads its extra rows from x staged at the partition's columns (plan of D, numbering `cols`), at `off`
template <typename V, typename X>
__device__ __forceinline__ void use_halo(Product<V, X>* pr, const KArgs& a, const int32_t* cols, int p, int32_t off) {
  if (!a.er_hcol || off < 0) return;
  pr->er_hcol = a.er_hcol;
  pr->halo = cols + a.halo_ptr[p];
  pr->nh = (int)(a.halo_ptr[p + 1] - a.halo_ptr[p]);
  pr->xh_off = off;
}

// (G and G^T of the preconditioner.  Not the matrix's product: staging waits for the other blocks' direction at once,
// which the slabs otherwise hide; elasticity 40^3, mixed-precision solve: 2.80 ms gathered, 2.84 with G and G^T
// staged, 3.05 with A too; 60^3: 5.46, 5.32, 5.31.)
// stage x at the columns of the product's extra rows (when it does so), by all threads, before run_slices; the
// caller's next __syncthreads is inside
template <typename V, typename X>
__device__ __noinline__ void stage_halo(Product<V, X>* pr, const SyncArgs* sync, int round) {
  if (!pr->er_hcol) return;  // uniform over the block
  extern __shared__ __align__(16) unsigned char smem_raw[];
  X* const xh = reinterpret_cast<X*>(smem_raw + pr->xh_off);
  if (!wait_round(*sync, round, pr->seen)) *pr->stop = 1;
  const int nh = pr->nh, bd = blockDim.x;
  for (int j0 = threadIdx.x; j0 < nh; j0 += 4 * bd) {
    int c[4];
    X v[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) c[u] = j0 + u * bd < nh ? (int)checked((int64_t)pr->halo[j0 + u * bd], pr->n_x, pr->status) : 0;
#pragma unroll
    for (int u = 0; u < 4; ++u) v[u] = j0 + u * bd < nh ? load_x(pr->xg + c[u]) : X(0);
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (j0 + u * bd < nh) xh[j0 + u * bd] = v[u];
  }
  __syncthreads();
}

// All slices of the block's partition, claimed dynamically from pr->counter (blockDim.x / 32 on entry).  Before its
// first extra row a warp waits until round `round` of arrive() is complete (0: at once); a wait that ran out
// raises *pr->stop and ends the pass.
template <typename V, typename X, int KB, bool RUNS>
__device__ __noinline__ void run_slices(Product<V, X>* pr, const SyncArgs* sync, int round) {
  const int lane = threadIdx.x & 31;
  const V *ell_val = pr->ell_val, *er_val = pr->er_val;
  const uint16_t* ell_col = pr->ell_col;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const X* const xsl = reinterpret_cast<const X*>(smem_raw + pr->xs_off);
  const int s0 = pr->s0, s1 = pr->s1, lim = pr->lim;
  int32_t* const status = pr->status;
  auto meta = [&](int j, int& sj, int64_t& posj, int& wj, int64_t& eposj, int& wej) {
    if (const SliceMeta* tbl = pr->tbl) {
      const SliceMeta m = tbl[checked(j - s0, pr->meta_cap, status)];
      sj = m.s;
      posj = m.pos;
      wj = m.w;
      eposj = m.epos;
      wej = m.we;
      return;
    }
    sj = pr->slice_order[j];
    posj = pr->slice_pos[sj];
    wj = (int)((pr->slice_pos[sj + 1] - posj) >> 5);
    eposj = pr->er_slice_pos[sj];
    wej = (int)((pr->er_slice_pos[sj + 1] - eposj) >> 5);
  };
  int i = s0 + (threadIdx.x >> 5), s = s1;
  int64_t pos = 0, epos = 0;
  int w = 0, we = 0;
  if (i < s1) meta(i, s, pos, w, epos, we);
  while (i < s1) {
    int t = 0;
    if (lane == 0) t = atomicAdd(&pr->counter, 1);
    const int inxt = s0 + __shfl_sync(FULL, t, 0);
    int nxt = s1;
    int64_t npos = 0, nepos = 0;
    int nw = 0, nwe = 0;
    if (inxt < s1) meta(inxt, nxt, npos, nw, nepos, nwe);
    X acc;
    if constexpr (RUNS) acc = slab_dot_runs<V, X, KB>(ell_val + pos, ell_col + pos, lane, w, xsl, X(0), lim, status);
    else acc = slab_dot<V, X, KB>(ell_val + pos + lane, ell_col + pos + lane, w, xsl, X(0), lim, status);
    if (we > 0) {
      if (!wait_round(*sync, round, pr->seen)) {
        *pr->stop = 1;
        return;
      }
      const int32_t* ecol = pr->er_col;
      if constexpr (RUNS) {
        if (const uint16_t* hcol = pr->er_hcol) {
          const X* const xh = reinterpret_cast<const X*>(smem_raw + pr->xh_off);
          acc = slab_dot_runs<V, X, 16>(er_val + epos, hcol + epos, lane, we, xh, acc, pr->nh, status);
          goto summed;
        }
      }
      if constexpr (RUNS) acc = er_dot_runs<V, X>(er_val + epos, ecol + epos, lane, we, pr->xg, acc, pr->n_x, status);
      else acc = er_dot<V, X, KB>(er_val + epos + lane, ecol + epos + lane, we, pr->xg, acc, pr->n_x, status);
    }
  summed:
    const int lg = pr->tpr_log2, tpr = 1 << lg;
    for (int off = tpr >> 1; off > 0; off >>= 1) acc += __shfl_xor_sync(FULL, acc, off);
    const int row = (s - s0) * (32 >> lg) + (lane >> lg);
    if ((lane & (tpr - 1)) == 0 && row < pr->rows) {
      const int m = pr->n2o ? checked(pr->n2o[row] - pr->pb, pr->rows, status) : row;
      pr->out[m] = acc;
      if (pr->mirror) pr->mirror[m] = acc;
    }
    i = inxt;
    s = nxt;
    pos = npos;
    w = nw;
    epos = nepos;
    we = nwe;
  }
}

}  // namespace persist
}  // namespace ehyb
