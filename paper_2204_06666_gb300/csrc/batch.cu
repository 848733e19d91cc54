// Batched EHYB SpMV: many plans (matrices of uneven size) in one persistent launch.
//
// The work units are (plan, partition) tiles or, where a partition is a large share of the batch, equal shares
// of its slices (see kShare), sorted by their slot count, largest first (longest-processing-time order).  A
// grid of (SMs x resident blocks) blocks pulls units from one atomic counter and runs each with the same
// per-partition code as the single-plan kernel (core::partition_spmv), so every row is summed in exactly the
// same order as by ehyb_spmv: the batch result equals the per-plan results bit for bit.  Each unit stages its
// partition's slice of x straight from the caller's x through the plan's new_to_old (the permutation is fused
// into the loads, as in ehyb_spmv), so the batch is ONE launch.  The last block to leave resets the counter; a
// call only rewrites the table of x / y pointers when they change.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstring>
#include <new>
#include <vector>

#include "ehyb_core.cuh"
#include "plan_internal.h"

namespace ehyb {
namespace {

using namespace core;

struct BatchPlan {
  KArgs a;
  const double* ell_val;
  const double* er_val;
  const double* x;  // caller's x (original numbering)
  double* y;        // caller's y (original numbering)
  int64_t n;
  int32_t kbatch;   // the plan's batch depth (6 on wide slices, else 8)
};

// A partition worth more than 1 / kShare of a resident block's share of the batch is split into units that each take
// every nsub-th slice of its processing order (and stage the whole slice of x again, which costs about kStageCost
// slots a row, from L2).  With whole partitions as units, a batch with fewer large partitions than resident blocks
// took as long as its largest one: 24 matrices of 5k to 100k rows on 304 blocks, about 50 partitions of up to 640k
// entries, 272 us; 91 us in shares (launched directly under the previous grid's tail).  Plans with wide slices are
// not split (one block combines their partial sums). Nothing is split where the largest partition is less than kWhole
// of an SM's share: then the order alone balances the units, and the extra staging would only cost (64 matrices of 5k
// to 300k rows, 0.52 of a share: whole 315 us, in shares 337; the first 56 of them, 0.67 of a share: 280 and 263).
constexpr double kShare = 2.0;
constexpr double kWhole = 0.6;
constexpr int kStageCost = 2;

constexpr int kMaxThreads = 1024;  // block size: 512 when two or more blocks fit an SM, else 1024

// plans with wide slices, out of line: their code costs the other plans of the batch no registers
__device__ __noinline__ bool wide_partition(const BatchPlan& bp, int p, double* xs, BlockState& bs) {
  return partition_spmv<double, double, true, true, false, true, kBatch, false, false, false, true>(
      bp.a, bp.ell_val, bp.er_val, bp.x, bp.y, p, xs, bs);
}

// tiles: (plan, partition, share, shares).  WIDE: a plan of the batch has wide slices.  Batches without go without
// the call: it cost every batch a few registers' spills (64 matrices 317.9 -> 313.4 us, 32 of them 172 -> 160, 16 of
// them 112 -> 110).
template <bool WIDE>
__global__ void __launch_bounds__(kMaxThreads, 1) batch_kernel(const BatchPlan* __restrict__ plans,
                                                              const int4* __restrict__ tiles, int ntiles,
                                                              int* counters) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ BlockState bs;
  __shared__ int tile_s;
  if (threadIdx.x == 0) {
    bs.bar_ready = 0;
    bs.phase = 0;
  }
  pdl_launch_dependents();
  pdl_wait();  // launched with programmatic stream serialization: the previous grid's work is complete from here
  for (;;) {
    __syncthreads();  // the previous tile's reads of shared memory are complete
    if (threadIdx.x == 0) tile_s = atomicAdd(&counters[0], 1);
    __syncthreads();
    const int t = tile_s;
    if (t >= ntiles) break;
    const int4 tl = tiles[t];
    const BatchPlan& bp = plans[tl.x];
    double* xs = reinterpret_cast<double*>(smem_raw);
    const bool ok =
        WIDE && bp.a.wide_parts > 0 ? wide_partition(bp, tl.y, xs, bs)
        : bp.kbatch == 6
            ? partition_spmv<double, double, true, true, false, true, 6>(bp.a, bp.ell_val, bp.er_val, bp.x, bp.y,
                                                                         tl.y, xs, bs, tl.z, tl.w)
            : partition_spmv<double, double, true, true, false, true>(bp.a, bp.ell_val, bp.er_val, bp.x, bp.y, tl.y,
                                                                      xs, bs, tl.z, tl.w);
    if (!ok) break;
  }
  __syncthreads();
  if (threadIdx.x == 0) {  // the last block out resets the queue for the next launch
    __threadfence();
    if (atomicAdd(&counters[1], 1) == (int)gridDim.x - 1) {
      counters[0] = 0;
      counters[1] = 0;
      __threadfence();
    }
  }
}

}  // namespace
}  // namespace ehyb

using namespace ehyb;

struct ehyb_batch_s {
  int32_t count = 0;
  int device = -1;
  std::vector<ehyb_plan_t> plans;
  std::vector<BatchPlan> table;
  std::vector<const double*> xs;
  std::vector<double*> ys;
  void* arena = nullptr;
  BatchPlan* d_table = nullptr;
  int4* d_tiles = nullptr;
  int* d_counters = nullptr;
  int ntiles = 0, nunits = 0, grid = 0, threads = 512;  // partitions, work units
  size_t smem = 0;
  int64_t max_n = 0;
  void (*kernel)(const BatchPlan*, const int4*, int, int*) = nullptr;
  bool dirty = true;  // the pointers in `table` are not (known to be) on the device
};

#define CKB(call)                                                     \
  do {                                                                \
    cudaError_t e_ = (call);                                          \
    if (e_ != cudaSuccess) return cuda_error_status(e_, #call);       \
  } while (0)

static void batch_free(ehyb_batch_t b) {
  if (!b) return;
  if (b->arena) cudaFree(b->arena);
  delete b;
}

extern "C" ehyb_status_t ehyb_batch_create(int32_t count, const ehyb_plan_t* plans, ehyb_batch_t* out) {
  if (!out) return EHYB_ERR_INVALID_ARG;
  *out = nullptr;
  if (count < 1 || !plans) return EHYB_ERR_INVALID_ARG;
  ehyb_batch_s* b = new (std::nothrow) ehyb_batch_s();
  if (!b) return EHYB_ERR_OOM;
  b->count = count;
  struct Tile {
    int plan, part;
    int32_t slices, rows;
    int64_t slots;
    bool wide;
  };
  std::vector<Tile> parts;
  for (int i = 0; i < count; ++i) {
    ehyb_plan_t P = plans[i];
    if (!P) { batch_free(b); return EHYB_ERR_INVALID_ARG; }
    if (P->host_only || P->er_layout != 0) { batch_free(b); return EHYB_ERR_UNSUPPORTED; }
    if (b->device < 0) b->device = P->device;
    if (P->device != b->device) { batch_free(b); return EHYB_ERR_INVALID_ARG; }
    b->plans.push_back(P);
    BatchPlan bp;
    std::memset(&bp, 0, sizeof(bp));
    bp.a = make_kargs(P->dev);
    bp.ell_val = P->dev.ell_val;
    bp.er_val = P->dev.er_sval;
    bp.n = P->dev.n;
    bp.kbatch = P->dev.kbatch;
    b->table.push_back(bp);
    b->max_n = std::max(b->max_n, P->dev.n);
    b->smem = std::max(b->smem, ehyb_smem_bytes(P->dev, 8));
    const HostPlan& H = P->host;
    for (int32_t p = 0; p < H.nparts; ++p) {
      const int32_t s0 = H.slice_ptr[(size_t)p], s1 = H.slice_ptr[(size_t)p + 1];
      const int64_t c = (H.slice_pos[(size_t)s1] - H.slice_pos[(size_t)s0]) +
                        (H.er_slice_pos[(size_t)s1] - H.er_slice_pos[(size_t)s0]) + 32;
      parts.push_back({i, p, s1 - s0, H.part_ptr[(size_t)p + 1] - H.part_ptr[(size_t)p], c, P->dev.wide_parts > 0});
    }
  }
  b->ntiles = (int)parts.size();
  b->xs.assign((size_t)count, nullptr);
  b->ys.assign((size_t)count, nullptr);

  int cur = -1;
  cudaError_t e = cudaGetDevice(&cur);
  if (e != cudaSuccess || cur != b->device) { batch_free(b); return EHYB_ERR_INVALID_ARG; }
  int sms = 0, per_sm = 0, optin = 0;
  e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, b->device);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, b->device);
  bool wide = false;
  for (const Tile& t : parts) wide = wide || t.wide;
  b->kernel = wide ? batch_kernel<true> : batch_kernel<false>;
  // the device's limit for every batch: a smaller one set for this batch would refuse the launches of another
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(b->kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, optin - 1024);
  // 512 threads while two blocks fit an SM (one block's staging overlaps the other's slices), otherwise
  // one block of 1024 threads per SM (32 warps keep enough loads in flight)
  if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, b->kernel, 512, b->smem);
  if (e == cudaSuccess && per_sm < 2) {
    b->threads = kMaxThreads;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, b->kernel, kMaxThreads, b->smem);
  }
  if (e != cudaSuccess) { batch_free(b); return cuda_error_status(e, "batch launch setup"); }
  b->grid = sms * std::max(per_sm, 1);
  // units: a partition's slices in as many shares as keep its units near the target, each with at least one
  // slice for every warp; longest units first (stable, so ties keep plan / partition / share order)
  std::vector<int4> tiles;
  std::vector<int64_t> cost;
  {
    int64_t total = 0;
    int64_t largest = 0;
    for (const Tile& t : parts) {
      total += t.slots;
      largest = std::max(largest, t.slots);
    }
    const bool whole = (double)largest * sms < kWhole * (double)total;
    const double target = std::max(1.0, (double)total / ((double)b->grid * kShare));
    for (const Tile& t : parts) {
      const int64_t most = std::max<int64_t>(1, t.slices / (b->threads / 32));
      const int nsub = t.wide || whole ? 1 : (int)std::min<int64_t>(most, (int64_t)((double)t.slots / target + 0.999));
      for (int k = 0; k < std::max(nsub, 1); ++k) {
        tiles.push_back(make_int4(t.plan, t.part, k, std::max(nsub, 1)));
        cost.push_back(t.slots / std::max(nsub, 1) + kStageCost * (int64_t)t.rows);
      }
    }
  }
  std::vector<size_t> order(tiles.size());
  for (size_t k = 0; k < order.size(); ++k) order[k] = k;
  std::stable_sort(order.begin(), order.end(), [&](size_t u, size_t v) { return cost[u] > cost[v]; });
  std::vector<int4> sorted(tiles.size());
  for (size_t k = 0; k < order.size(); ++k) sorted[k] = tiles[order[k]];
  b->nunits = (int)sorted.size();

  const size_t t_bytes = ((size_t)count * sizeof(BatchPlan) + 255) & ~(size_t)255;
  const size_t l_bytes = ((size_t)std::max(b->nunits, 1) * sizeof(int4) + 255) & ~(size_t)255;
  // partial sums of the plans' wide slices: the batch's own, since a plan may be in it more than once
  size_t sums = 0;
  for (BatchPlan& bp : b->table) sums += (size_t)bp.a.wide_parts * 32 * sizeof(double);
  ehyb_status_t st = device_alloc(&b->arena, t_bytes + l_bytes + 256 + sums);
  if (st != EHYB_OK) { batch_free(b); return st; }
  b->d_table = (BatchPlan*)b->arena;
  b->d_tiles = (int4*)((char*)b->arena + t_bytes);
  b->d_counters = (int*)((char*)b->arena + t_bytes + l_bytes);
  double* ww = (double*)((char*)b->arena + t_bytes + l_bytes + 256);
  for (BatchPlan& bp : b->table) {
    bp.a.wide_ws = ww;
    ww += (size_t)bp.a.wide_parts * 32;
  }
  e = cudaMemcpy(b->d_table, b->table.data(), (size_t)count * sizeof(BatchPlan), cudaMemcpyHostToDevice);
  if (e == cudaSuccess && b->nunits)
    e = cudaMemcpy(b->d_tiles, sorted.data(), sorted.size() * sizeof(int4), cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMemset(b->d_counters, 0, 256);
  if (e != cudaSuccess) { batch_free(b); return cuda_error_status(e, "batch upload"); }
  *out = b;
  return EHYB_OK;
}

extern "C" ehyb_status_t ehyb_batch_spmv(ehyb_batch_t b, const double* const* xs, double* const* ys, void* stream) {
  if (!b || !xs || !ys) return EHYB_ERR_INVALID_ARG;
  cudaStream_t s = (cudaStream_t)stream;
  for (int i = 0; i < b->count; ++i)
    if (b->table[(size_t)i].n > 0 && (!xs[i] || !ys[i] || (const void*)xs[i] == (const void*)ys[i]))
      return EHYB_ERR_INVALID_ARG;
  // A captured call would only record the table's copy: later calls with the same pointers would launch without it, and
  // a replay after a call with other pointers would use those.
  cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
  CKB(cudaStreamIsCapturing(s, &capture));
  if (capture != cudaStreamCaptureStatusNone)
    return cuda_error_status(cudaErrorStreamCaptureUnsupported, "ehyb_batch_spmv on a capturing stream");
  for (int i = 0; i < b->count; ++i) {
    if (xs[i] != b->xs[(size_t)i] || ys[i] != b->ys[(size_t)i]) {
      b->xs[(size_t)i] = xs[i];
      b->ys[(size_t)i] = ys[i];
      b->table[(size_t)i].x = xs[i];
      b->table[(size_t)i].y = ys[i];
      b->dirty = true;
    }
  }
  if (b->dirty)
    CKB(cudaMemcpyAsync(b->d_table, b->table.data(), (size_t)b->count * sizeof(BatchPlan), cudaMemcpyHostToDevice, s));
  b->dirty = false;
  if (b->ntiles == 0) return EHYB_OK;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)b->grid);
  cfg.blockDim = dim3((unsigned)b->threads);
  cfg.dynamicSmemBytes = b->smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  CKB(cudaLaunchKernelEx(&cfg, b->kernel, (const BatchPlan*)b->d_table, (const int4*)b->d_tiles, b->nunits,
                         b->d_counters));
  return EHYB_OK;
}

extern "C" ehyb_status_t ehyb_batch_info(ehyb_batch_t b, int32_t* ntiles, int32_t* grid, int32_t* threads) {
  if (!b) return EHYB_ERR_INVALID_ARG;
  if (ntiles) *ntiles = b->ntiles;
  if (grid) *grid = b->grid;
  if (threads) *threads = b->threads;
  return EHYB_OK;
}

extern "C" ehyb_status_t ehyb_batch_destroy(ehyb_batch_t b) {
  if (!b) return EHYB_OK;
  cudaError_t e = cudaDeviceSynchronize();
  batch_free(b);
  return e == cudaSuccess ? EHYB_OK : cuda_error_status(e, "cudaDeviceSynchronize");
}
