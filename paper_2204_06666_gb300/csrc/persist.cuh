// Device code of the persistent solver kernels (cg.cu, pcg.cu): a whole Krylov iteration, and then the next, inside
// one cooperative launch with one block per partition.
//
// A solver iteration as separate launches re-reads what the block that owns a partition has just had in hand: the
// direction is staged into shared memory for every product, q and r go through memory between the product and the
// updates, and every launch drains and refills the chip (tet 80^3, 512k rows: product 29 us, update 14 us, direction
// 5 us cold, 44 us an iteration back to back from a graph, for 74 MB of matrix).  Here a block keeps its partition's
// slices of the vectors in shared memory from one iteration to the next, as many of them as fit, and the iteration's
// inner products double as the barriers that the data dependences need.  Scalars (a division is a dozen dependent
// FP64 operations, and FP64 operations of 32 warps queue for one unit) are one thread's work.
//
// The sums are added in the order of the separate launches, so both forms give the same bits; that costs a meeting
// more an iteration (r.r, below) and a serial chain over the block's warps (p.q: 32 dependent FP64 additions, 1.6 us):
// 35.1 us an iteration at tet 80^3, 31 with sums in the blocks' own order, 43 in separate launches.
// Whole solves of (A + 0.1 mean diagonal) x = b to 1e-10, separate launches -> persistent, FP64 CG (44 to 65
// iterations): tet 40^3 1.12 -> 0.79 ms, 80^3 2.10 -> 1.76, 126^3 4.63 -> 4.48, elasticity 24^3 2.11 -> 1.50, 40^3 3.88 ->
// 3.43, 64^3 9.32 -> 8.80.  FP32 CG (refinement): tet 40^3 1.61 -> 1.09, 101^3 3.25 -> 2.91, elasticity 64^3 7.88 -> 7.52.
// Mixed-precision PCG (1e-9): tet 80^3 1.77 -> 1.33, elasticity 40^3 3.55 -> 2.94, 64^3 7.32 -> 6.71; FP64 PCG: tet 80^3
// 1.74 -> 1.30, elasticity 64^3 9.88 -> 9.31.
#pragma once
#include <algorithm>

#include "ehyb_core.cuh"

namespace ehyb {
namespace persist {

using namespace core;

constexpr int kMaxGrid = 160;  // blocks of a persistent launch
// Least time limit (wait_timeout_ns) with which solvers iterate persistently: the others' work, or another process's
// time slice, may keep a block waiting for milliseconds.  Plans with a shorter one take the separate launches, which
// have no such waits.
constexpr uint64_t kMinLimitNs = 100000000ull;
constexpr int kAborted = 2;

// Grid of the vector kernels of the separate launches.  Their inner products add a vector's squares in the order of
// these threads, blocks and partials, and the persistent kernels add them in the same one: a solve's bits do not
// depend on the form its iterations take.
constexpr int kVecBlocks = 608;  // 4 per SM; 8 per SM measured slower
constexpr int kVecThreads = 256;
constexpr int kVecWarps = kVecThreads / 32;

// A partial sum: the halves of a double, each beside the number of its round in an 8-byte word of its own, so that a
// reader sees for each half whether it is the one it waits for.
struct __align__(16) Slot {
  unsigned long long lo, hi;
};

// The memory the blocks meet in, all zero at launch.
struct Meeting {
  Slot part[2][kMaxGrid];    // partitions' partial sums: p.q; t.t
  Slot vec[kVecBlocks];      // vector blocks' partial sums: r.r
  int32_t summed, pad0[31];  // blocks that have published, over all rounds of sums
  int32_t arrived, pad1[31]; // arrivals at the plain rounds
};

struct SyncArgs {
  Meeting* m;
  int32_t* status;            // the plan's status word: EHYB_ERR_TIMEOUT when a wait ran out
  int32_t* done;              // set to kAborted with it, so that the other blocks give up and the host stops launching
  uint64_t limit_ns;
};

// Shared memory of a persistent block, out of the SM's 256 KB that the rest of L1 shares: the least of the sizes the
// hardware can set aside that holds `must` bytes (what the kernel should not do without), less what the system and
// the kernel's own variables take; the vectors beyond it go there only as far as they fit.  The extra rows gather
// freshly written vectors through L1, so a vector kept in shared memory at L1's cost loses more than it saves: at
// elasticity 64^3 (41 KB a vector) the FP64 PCG took 23.1 ms a solve with five vectors in shared memory (215 KB), 9.5
// with two (separate launches 9.8); scalar hexahedra 80^3 with BF16 G 3.0 and 1.9 ms (2.4).  0: more than `most` KB,
// where the separate launches are the faster form: 196 for CG (ms a solve, separate -> persistent: tet 150^3 9.61 ->
// 8.48), 164 for PCG, which gathers two more vectors (FP64 G: tet 111^3, 160 KB, 3.00 -> 2.80, scalar hexahedra
// 115^3, 176 KB, 6.11 -> 6.89; FP32 G: tet 121^3, 156 KB, 3.25 -> 3.17, 126^3, 175 KB, 3.57 -> 3.61).
//
// The budget only decides what is placed.  What a kernel may be launched with is a property of its instantiation,
// shared by every plan and host thread, so it is always set to the device's limit: a smaller plan's budget set there
// would refuse the launch of a larger one that another thread is about to make.  (A launch's own size decides L1's
// share.)
constexpr int kMaxStatic = 2048;  // static shared memory of a persistent kernel
inline size_t shared_budget(size_t must, size_t most) {
  for (size_t kb : {100, 132, 164, 196})
    if (kb <= most && must + 3072 <= kb * 1024) return kb * 1024 - 3072;
  return 0;
}

// Rows of a partition up to which iterations on FP32 vectors run persistently.  Beyond, the FP32 products are short
// of bytes rather than of launches, and the vectors' passes of the separate launches are the faster ones.  Time of a
// solve, separate over persistent: CG (refinement), FP32 values, tet 107^3 (8,060 rows) 1.10, 120^3 (11,369) 1.04,
// scalar hexahedra 110^3 (8,757) 1.03, 120^3 0.99, elasticity 64^3 (5,174) 1.00, 76^3 (8,664) 1.09; BF16, tet 107^3
// 1.07, 120^3 1.02, scalar hexahedra 110^3 1.00, 120^3 0.98.  Where the separate product stages its extra rows and
// this one gathers them, BF16: elasticity 50^3 (2,468) 1.01, 54^3 (3,108) 1.00, 64^3 0.96.  Mixed PCG: tet 120^3
// 1.09, scalar hexahedra 120^3 1.04, elasticity 58^3 1.03.
constexpr int kMaxRowsF32 = 11500, kMaxRowsBf16 = 9000, kMaxRowsBf16Staged = 3000, kMaxRowsPcg32 = 11500;

// Whether a plan's partitions are even enough with the SMs: a block passes over its partition's vectors alone, where
// the separate launches spread them over the chip, so each row beyond the chip's share costs about 1.7 ns an
// iteration of FP64 CG against the 5 us or so that the launches cost.  `spare`: the rows beyond n / SMs up to which
// persistent iterations were the faster ones (ms a solve, separate -> persistent; FP64 CG: tet 37^3 in partitions of
// 3,000 rows 1.57 -> 1.48, of 6,000 2.11 -> 2.23, tet 60^3 in 6,000 2.28 -> 2.36, tet 90^3 in 8,000 3.03 -> 2.94, in
// 10,000 3.40 -> 3.55; FP32 CG: tet 37^3 in 4,500 2.36 -> 2.12, elasticity 24^3 in 3,000 3.45 -> 3.07, in 4,500 4.06
// -> 4.10; FP64 PCG with BF16 G: tet 60^3 in 6,000 1.78 -> 1.70, in 12,000 2.56 -> 2.87; the other PCG forms gained
// at every size).
inline bool even_enough(int max_rows, int64_t n, int sms, int spare) { return max_rows - n / sms <= spare; }
constexpr int kSpare64 = 3500, kSpare32 = 4000, kSparePcg = 4500;

// The meeting place of a launch, zeroed.  Test hook (inject_wait_fault 2 / 3): one arrival at the sums / the plain
// rounds never happens, so that the first wait there runs out.
inline cudaError_t clear_meeting(Meeting* m, int inject, cudaStream_t s) {
  cudaError_t e = cudaMemsetAsync(m, 0, sizeof(Meeting), s);
  if (e == cudaSuccess && inject >= 2)
    e = cudaMemsetAsync(inject == 2 ? &m->summed : &m->arrived, 0xff, sizeof(int32_t), s);
  return e;
}

// a wait that has lasted: true when it must give up (its limit is over, or another block gave up)
struct Patience {
  uint64_t t0 = 0;
  int spins = 0;
  __device__ __forceinline__ bool over(const SyncArgs& g) {
    if ((++spins & 63) != 0) return false;
    const uint64_t t = globaltimer_ns();
    if (t0 == 0) t0 = t;
    return t - t0 > g.limit_ns || *(volatile int32_t*)g.done == kAborted;
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

// Sums over the grid, each a grid-wide barrier too, in two halves so that a block can work in between.  The sums'
// number in the launch is `round` = 1, 2, ...  A block's partial sums (one for its partition, or one for each vector
// block it stands in for) go into slots with the round in them, and one more onto the counter; a gather waits for the
// counter, then adds the slots, lane-strided, then an xor tree: every block gets the same bits.  No fence is paid for
// (one costs half a microsecond to a microsecond behind a product): the counter is only the sign that looking is
// worth while, the rounds in the slots tell whether a value is there.  Polling the one counter and reading the slots
// once beats polling the slots (152 blocks, nothing else to do: 1.9 against 3.5 to 4.9 us; many lines, written by
// stores and polled by all, against one atomic).  A slot is written again an iteration later, when a sum of another
// kind has been gathered since, to which every block added after it had read the slot.
//
// An FP64 instruction occupies its quarter of the SM for 64 cycles however few lanes need it, so a block's lane trees
// are not made by every warp (five adds each, eight warps a quarter) but by one warp in each quarter for eight warps'
// terms at once (nine adds), from shared memory.  Terms lie there as they do in a warp, lane l of warp w at
// term_at(w, l): four threads that read a row, and the four rows beside it, touch all banks.
constexpr int kSumWarps = 4;
__device__ __forceinline__ int term_at(int w, int l) { return 32 * w + ((l + 4 * w) & 31); }

// sums[w] = the xor tree's sum of warp w's terms, w < count, by the block's first kSumWarps warps (all that there are)
__device__ __forceinline__ void tree_sums(const double* red, int count, double* sums) {
  const int tid = threadIdx.x, j = tid & 3, threads = min(32 * kSumWarps, (int)blockDim.x);
  for (int w0 = 0; w0 < count; w0 += threads / 4) {
    const int w = w0 + (tid >> 2);
    double a[4] = {0.0, 0.0, 0.0, 0.0};
    if (w < count)
#pragma unroll
      for (int k = 0; k < 4; ++k) a[k] = red[term_at(w, j + 4 * k)] + red[term_at(w, j + 4 * k + 16)];
    double v = (a[0] + a[2]) + (a[1] + a[3]);
    v += __shfl_xor_sync(FULL, v, 2);
    v += __shfl_xor_sync(FULL, v, 1);
    if (w < count && j == 0) sums[w] = v;
  }
}
__device__ __forceinline__ void sum_warps_sync() {
  const int threads = min(32 * kSumWarps, (int)blockDim.x);
  asm volatile("bar.sync 1, %0;" ::"r"(threads) : "memory");
}
__device__ __forceinline__ void put_slot(Slot* slot, int round, double v) {
  const unsigned long long bits = (unsigned long long)__double_as_longlong(v), tag = (unsigned long long)round << 32;
  asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(slot), "l"(tag | (bits & 0xffffffffull)),
               "l"(tag | (bits >> 32))
               : "memory");
}
__device__ __forceinline__ void count_published(const SyncArgs& g) {
  asm volatile("red.relaxed.gpu.global.add.s32 [%0], 1;" ::"l"(&g.m->summed) : "memory");
}

// The block's partial of a partition's sum, by its first kSumWarps warps, after a __syncthreads behind the terms of
// `warps` warps in red.  The order of the product's fused sum: a tree in each warp, then the warps one after the
// other.
static __device__ __noinline__ void publish_part(const SyncArgs& g, int round, int which, const double* red, int warps,
                                                double* sums) {
  tree_sums(red, warps, sums);
  sum_warps_sync();
  if (threadIdx.x == 0) {
    double v = 0.0;
    for (int w = 0; w < warps; ++w) v += sums[w];
    put_slot(&g.m->part[which][blockIdx.x], round, v);
    count_published(g);
  }
}

// (The helpers from here on are functions of their own that need few registers.  Inlined, or with five slots a lane in
// flight, they left the product's loop, which the same kernel calls, short of registers: 244 bytes of spills, 45.6 us
// an iteration at tet 80^3 instead of 35.1.)
//
// Sum of `count` slots, by all threads, valid in warp 0.  One thread watches the counter; the slots are then read by
// as many warps as there are, one slot a lane (vals: shared memory for them, the terms' place: the trees are done).
// A wait that ran out raises *stop (down before) and gives false.
static __device__ __noinline__ bool gather_sum(const SyncArgs& g, int round, const Slot* slot, int count, double* vals,
                                               int* stop, double* sum) {
  const int tid = threadIdx.x;
  volatile int* const over = stop;
  if (tid == 0 && !wait_at<false>(g, &g.m->summed, round)) *over = 1;
  __syncthreads();
  if (!*over) {
#pragma unroll 1
    for (int i = tid; i < count; i += blockDim.x) {
      Patience wait;
      unsigned long long lo, hi;
      for (;;) {
        asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(lo), "=l"(hi) : "l"(slot + i) : "memory");
        if ((int)(lo >> 32) == round && (int)(hi >> 32) == round) break;
        if (wait.over(g)) {
          give_up(g);
          *over = 1;
          break;
        }
      }
      vals[i] = __longlong_as_double((long long)((hi << 32) | (lo & 0xffffffffull)));
    }
  }
  __syncthreads();
  if (tid >= 32 || *over) return false;
  double s = 0.0;
  for (int i = tid; i < count; i += 32) s += vals[i];
  for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(FULL, s, off);
  *sum = s;
  return true;
}

// Terms of a partition's sum, in the order of the product's fused sum with `warps` warps: warp w's lanes take the
// rows of its slices w, w + warps, ... of the processing order.  load(row): the two factors.
template <typename P, typename F>
__device__ __forceinline__ void part_terms(const P& pr, int warps, double* red, F&& load) {
  constexpr int U = 4;  // rows a lane has in flight
  const int lane = threadIdx.x & 31, lg = pr.tpr_log2, s0 = pr.s0, ns = pr.s1 - s0, rows = pr.rows;
  const bool lead = (lane & ((1 << lg) - 1)) == 0;
  for (int w = threadIdx.x >> 5; w < warps; w += blockDim.x >> 5) {
    double acc = 0.0;
    for (int t0 = w; t0 < ns; t0 += U * warps) {
      int row[U];
      double2 v[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int t = t0 + u * warps;
        row[u] = rows;
        if (t < ns && lead) {
          const int sl = pr.tbl ? pr.tbl[checked(t, pr.meta_cap, pr.status)].s : pr.slice_order[s0 + t];
          row[u] = (sl - s0) * (32 >> lg) + (lane >> lg);
        }
      }
#pragma unroll
      for (int u = 0; u < U; ++u) v[u] = row[u] < rows ? load(row[u]) : make_double2(0.0, 0.0);
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (row[u] < rows) acc = fma(v[u].x, v[u].y, acc);
    }
    red[term_at(w, lane)] = acc;
  }
}

// 16 bytes of a vector that other blocks have written (ordered by a round), not through L1
__device__ __forceinline__ void load_vec(const double* p, double (&v)[2]) {
  asm volatile("ld.relaxed.gpu.global.v2.f64 {%0, %1}, [%2];" : "=d"(v[0]), "=d"(v[1]) : "l"(p) : "memory");
}
__device__ __forceinline__ void load_vec(const float* p, float (&v)[4]) {
  asm volatile("ld.relaxed.gpu.global.v4.f32 {%0, %1, %2, %3}, [%4];"
               : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3])
               : "l"(p)
               : "memory");
}
__device__ __forceinline__ void load_one(const double* p, double& v) {
  asm volatile("ld.relaxed.gpu.global.f64 %0, [%1];" : "=d"(v) : "l"(p) : "memory");
}
__device__ __forceinline__ void load_one(const float* p, float& v) {
  asm volatile("ld.relaxed.gpu.global.f32 %0, [%1];" : "=f"(v) : "l"(p) : "memory");
}

// shared memory of the terms, which a gather's values take too
inline size_t terms_bytes(int threads) { return sizeof(double) * (size_t)std::max(threads, kVecBlocks); }

// vector blocks whose terms are not all zero
template <typename X>
__host__ __device__ __forceinline__ int vec_blocks(int64_t n) {
  const int64_t nv = n / (16 / (int)sizeof(X)), b = (nv + kVecThreads - 1) / kVecThreads;
  return b < 1 ? 1 : b < kVecBlocks ? (int)b : kVecBlocks;
}

// The block's partials of r.r over the whole vector (16-byte aligned, in memory, written by all blocks and ordered by a
// round): the block stands in for the vector blocks blockIdx.x, blockIdx.x + gridDim.x, ... of an update launch and
// forms the sums that their threads, warps and blocks would.  All threads.
template <typename X>
__device__ __noinline__ void publish_vec(const SyncArgs& g, int round, const X* r, int n, double* red, double* sums) {
  constexpr unsigned NV = 16 / (unsigned)sizeof(X), kStride = kVecBlocks * kVecThreads;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
  const int active = vec_blocks<X>(n), chunk = max(1, warps / kVecWarps);  // vector blocks at a time
  const unsigned nv = (unsigned)n / NV;
  for (int first = blockIdx.x; first < active; first += chunk * gridDim.x) {
    for (int w = warp; w < chunk * kVecWarps; w += warps) {
      const int vb = first + (w / kVecWarps) * gridDim.x;
      double acc = 0.0;
      if (vb < active) {
        const unsigned v = (unsigned)vb * kVecThreads + 32 * (w % kVecWarps) + lane;
#pragma unroll 1
        for (unsigned j = v; j < nv; j += kStride) {
          X x[NV];
          load_vec(r + NV * (size_t)j, x);
#pragma unroll
          for (unsigned k = 0; k < NV; ++k) acc = fma((double)x[k], (double)x[k], acc);
        }
        if (v < (unsigned)n - nv * NV) {
          X x;
          load_one(r + (nv * NV + v), x);
          acc = fma((double)x, (double)x, acc);
        }
      }
      red[term_at(w, lane)] = acc;
    }
    __syncthreads();
    if (threadIdx.x < 32 * kSumWarps) {
      tree_sums(red, chunk * kVecWarps, sums);
      sum_warps_sync();
      const int vb = first + threadIdx.x * gridDim.x;
      if (threadIdx.x < chunk && vb < active) {
        double s = 0.0;
#pragma unroll
        for (int k = 0; k < kVecWarps; ++k) s += sums[kVecWarps * threadIdx.x + k];
        put_slot(&g.m->vec[vb], round, s);
      }
    }
    if (first + chunk * gridDim.x < active) __syncthreads();  // the terms have been read
  }
  __syncwarp();
  if (threadIdx.x == 0) count_published(g);
}

// Barrier without a value, in two halves: arrive (one thread, after a __syncthreads that follows the block's writes)
// and a wait that each warp makes when it first needs the other blocks' writes, usually long after all have arrived.
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

// the same by one thread for its whole block, which a __syncthreads has to follow
__device__ __forceinline__ bool wait_block(const SyncArgs& g, int round, int* seen) {
  const bool ok = wait_at<true>(g, &g.m->arrived, round);
  const int now = ok ? round : -1;
  asm volatile("st.release.cta.shared.s32 [%0], %1;" ::"r"(smem_addr(seen)), "r"(now) : "memory");
  return ok;
}

// Whether the product itself leaves the terms of p.q (run_slices, DOT): on low-precision values, and where a warp has
// hardly more than one slice (MAXT 512: at most 16 warps, one for each slice of the average partition).
template <typename V, int MAXT>
constexpr bool kDotInProduct = sizeof(V) < 8 || MAXT <= 512;

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
    for (int u = 0; u < 4; ++u)
      c[u] = j0 + u * bd < nh ? (int)checked((int64_t)pr->halo[j0 + u * bd], pr->n_x, pr->status) : 0;
#pragma unroll
    for (int u = 0; u < 4; ++u) v[u] = j0 + u * bd < nh ? load_x(pr->xg + c[u]) : X(0);
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (j0 + u * bd < nh) xh[j0 + u * bd] = v[u];
  }
  __syncthreads();
}

// All slices of the block's partition, claimed dynamically from pr->counter (blockDim.x / 32 on entry).  Before its
// first extra row a warp waits until round `round` of arrive() is complete (0: at once); a wait that ran out raises
// *pr->stop and ends the pass.
// STAGED: the extra rows' x may be staged (pr->er_hcol).
// DOT: the terms of out.x go to red, in the order of part_terms; the warps then take their slices in turn instead of
// claiming them.  Low-precision products gain by that (a pass over q and x less: elasticity 64^3 FP32 CG 102.9 ->
// 97.7 us an iteration), FP64 ones need the balance more (elasticity 40^3 CG 54.5 us an iteration with claims, 59.4
// without) unless a warp has one slice anyway (tet 40^3 FP64 CG 18.9 -> 18.2 us).
template <typename V, typename X, int KB, bool RUNS, bool STAGED, bool DOT>
__device__ __noinline__ void run_slices(Product<V, X>* pr, const SyncArgs* sync, int round, double* red = nullptr) {
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
  double dacc = 0.0;
  while (i < s1) {
    int inxt;
    if constexpr (DOT) {
      inxt = i + (int)(blockDim.x >> 5);
    } else {
      int t = 0;
      if (lane == 0) t = atomicAdd(&pr->counter, 1);
      inxt = s0 + __shfl_sync(FULL, t, 0);
    }
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
      if constexpr (RUNS && STAGED) {
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
      if constexpr (DOT) dacc = fma((double)acc, (double)xsl[row], dacc);
      else if (pr->mirror) pr->mirror[m] = acc;
    }
    i = inxt;
    s = nxt;
    pos = npos;
    w = nw;
    epos = nepos;
    we = nwe;
  }
  if constexpr (DOT) red[term_at(threadIdx.x >> 5, lane)] = dacc;
}

}  // namespace persist
}  // namespace ehyb
