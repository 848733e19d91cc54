// Conjugate gradients on an EHYB plan (the solver whose SpMV cost motivates the method, Sec. 6), and FP64 iterative
// refinement around an inner CG whose matrix values are stored in FP32 or BF16.
//
// All vectors live in the plan's numbering (b and x are permuted once in and once out).  One CG iteration is three
// kernels:
//   K1  q = A p on the EHYB kernel, with p . q accumulated in its epilogue (p_r is already in shared
//       memory): one partial per partition, reduced into one scalar by the last block to finish;
//   K2  alpha = (r.r) / (p.q) (once per block); x += alpha p; r -= alpha q; partial sums of the new r.r;
//       the last block reduces them, stores r.r(new) in the history, computes beta = r.r(new) / r.r(old),
//       advances the device iteration counter and raises `done` at convergence or at the limit;
//   K3  p = r + beta p.
// alpha and beta never leave the device.  Every reduction runs in a fixed order, so a solve is bit-reproducible.
// Once `done` is up the remaining kernels of a chunk return at once, so the iteration count is exact although the
// host looks at the flag only once per chunk.  A chunk of kChunk iterations is captured once into a CUDA graph and
// replayed.  A plan whose partitions are all resident at once (at most one per SM) runs its iterations inside one
// cooperative kernel instead (cg_persist_kernel), with the same bits, where that is the faster form: on Eq. 1's
// partitions up to about 3.6 M rows in FP64 (two vectors' worth of shared memory), 1.75 M with FP32 values, 1.37 M with
// BF16.
//
// Refinement (refine = 1: FP32 values, 2: BF16 values): outer FP64 residual r = b - A x on the FP64 plan, inner CG on
// the low-precision copy of the values with FP32 vectors, FP32 SpMV accumulation and FP64 dot products / alpha /
// beta, started from d = 0 on r / ||r||; x += ||r|| d in FP64.
#include <cuda_runtime.h>

#include <chrono>
#include <cmath>
#include <cstring>
#include <vector>

#include "persist.cuh"
#include "plan_internal.h"

namespace ehyb {

namespace {

using core::FULL;
constexpr int kVB = persist::kVecBlocks, kVT = persist::kVecThreads;  // vector kernels
constexpr int kChunk = 16;
constexpr double kFcgInnerRtol = 0.1;  // default inner tolerance of the flexible CG's preconditioning solve

}  // namespace

struct CgState {
  int32_t it, done, converged, arrive_dot;
  int32_t arrive_rr, max_iter, breakdown, pad;
  double tol2, pq, beta, grow_limit;
};

struct CgWork {
  int64_t n = 0;
  int32_t nparts = 0, hist_cap = 0;
  void* arena = nullptr;
  double *bp = nullptr, *xp = nullptr, *r = nullptr, *p = nullptr, *q = nullptr, *xs = nullptr;
  float *r32 = nullptr, *p32 = nullptr, *q32 = nullptr, *d32 = nullptr;
  double *part_a = nullptr, *part_b = nullptr, *pq_part = nullptr, *hist = nullptr;
  CgState* st = nullptr;
  persist::Meeting* meeting = nullptr;  // of the persistent kernel's blocks
  cudaStream_t cap = nullptr;
  cudaGraphExec_t g64 = nullptr, g32 = nullptr;
  int g32_lowp = 0;
};

void cg_work_free(CgWork* w) {
  if (!w) return;
  if (w->g64) cudaGraphExecDestroy(w->g64);
  if (w->g32) cudaGraphExecDestroy(w->g32);
  if (w->cap) cudaStreamDestroy(w->cap);
  if (w->arena) cudaFree(w->arena);
  delete w;
}

namespace {

// warp-level fixed-order sum of count partials (lane-strided, then an xor tree); every lane gets it
__device__ __forceinline__ double warp_sum(const double* part, int count) {
  const int lane = threadIdx.x & 31;
  double v = 0.0;
  for (int i = lane; i < count; i += 32) v += part[i];
  for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(FULL, v, off);
  return v;
}

// fixed-order block sum; result valid in thread 0
__device__ __forceinline__ double block_sum(double v) {
  __shared__ double ws[32];
  for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(FULL, v, off);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (lane == 0) ws[warp] = v;
  __syncthreads();
  double s = 0.0;
  if (threadIdx.x == 0)
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += ws[w];
  return s;
}

__device__ __forceinline__ int64_t gtid() { return (int64_t)blockIdx.x * blockDim.x + threadIdx.x; }
__device__ __forceinline__ int64_t gstride() { return (int64_t)gridDim.x * blockDim.x; }

// r = b - q, p = r; partials of r.r (part_a) and b.b (part_b)
__global__ void init64_kernel(int64_t n, const double* __restrict__ b, const double* __restrict__ q, double* r,
                              double* p, double* part_a, double* part_b) {
  double ra = 0.0, bb = 0.0;
  for (int64_t i = gtid(); i < n; i += gstride()) {
    const double bi = b[i], ri = bi - q[i];
    r[i] = ri;
    p[i] = ri;
    ra = fma(ri, ri, ra);
    bb = fma(bi, bi, bb);
  }
  const double s1 = block_sum(ra);
  __syncthreads();
  const double s2 = block_sum(bb);
  if (threadIdx.x == 0) { part_a[blockIdx.x] = s1; part_b[blockIdx.x] = s2; }
}

// inner start: r32 = scale * r64 (rounded to FP32), p32 = r32, d32 = 0; partials of r32.r32
__global__ void init32_kernel(int64_t n, const double* __restrict__ r64, double scale, float* r32, float* p32,
                              float* d32, double* part_a) {
  double ra = 0.0;
  for (int64_t i = gtid(); i < n; i += gstride()) {
    const float ri = (float)(r64[i] * scale);
    r32[i] = ri;
    p32[i] = ri;
    d32[i] = 0.0f;
    ra = fma((double)ri, (double)ri, ra);
  }
  const double s = block_sum(ra);
  if (threadIdx.x == 0) part_a[blockIdx.x] = s;
}

// single block: hist[0] = r.r, convergence threshold, counters
__global__ void init_finish_kernel(const double* part_a, int na, const double* part_b, int nb, double rtol2,
                                   int relative_to_r0, int max_iter, double* hist, CgState* st) {
  if (threadIdx.x >= 32) return;
  const double rr = warp_sum(part_a, na);
  const double bb = part_b ? warp_sum(part_b, nb) : 0.0;
  if (threadIdx.x == 0) {
    hist[0] = rr;
    st->tol2 = rtol2 * (relative_to_r0 ? rr : bb);
    st->grow_limit = 1e12 * rr;
    st->it = 0;
    st->arrive_dot = 0;
    st->arrive_rr = 0;
    st->breakdown = 0;
    st->max_iter = max_iter;
    st->converged = rr <= st->tol2 ? 1 : 0;
    st->done = (st->converged || max_iter <= 0) ? 1 : 0;
  }
}

template <typename T> struct Vec16;
template <> struct Vec16<double> { using type = double2; static constexpr int N = 2; };
template <> struct Vec16<float> { using type = float4; static constexpr int N = 4; };
template <typename T> __device__ __forceinline__ T& lane_of(typename Vec16<T>::type& v, int i) {
  return reinterpret_cast<T*>(&v)[i];
}

// K2: alpha = hist[it] / (p.q); x += alpha p; r -= alpha q; r.r(new) by the last block, which also
// stores it, computes beta and advances the iteration.  16-byte vector accesses (the workspace vectors
// are 256-byte aligned), scalar tail.  p.q <= 0 means the operator is not positive definite along p:
// the iteration stops with `breakdown` set and nothing updated.
template <typename T>
__global__ void update_kernel(int64_t n, T* __restrict__ x, const T* __restrict__ p, const T* __restrict__ q,
                              T* __restrict__ r,
                              double* hist, CgState* st, double* rr_part) {
  if (st->done) return;
  using V = typename Vec16<T>::type;
  constexpr int NV = Vec16<T>::N;
  __shared__ double alpha_s;
  __shared__ int last_s;
  if (threadIdx.x == 0) alpha_s = st->pq > 0.0 ? hist[st->it] / st->pq : 0.0;
  __syncthreads();
  if (!(alpha_s > 0.0) && hist[st->it] > 0.0) {
    if (blockIdx.x == 0 && threadIdx.x == 0) {
      st->breakdown = 1;
      st->done = 1;
    }
    return;
  }
  const T a = (T)alpha_s;
  double acc = 0.0;
  const int64_t nv = n / NV;
  for (int64_t j = gtid(); j < nv; j += gstride()) {
    V xv = reinterpret_cast<V*>(x)[j];
    const V pv = reinterpret_cast<const V*>(p)[j];
    const V qv = reinterpret_cast<const V*>(q)[j];
    V rv = reinterpret_cast<V*>(r)[j];
#pragma unroll
    for (int u = 0; u < NV; ++u) {
      V& xx = xv;
      lane_of<T>(xx, u) = fma(a, lane_of<T>(const_cast<V&>(pv), u), lane_of<T>(xx, u));
      const T ri = fma(-a, lane_of<T>(const_cast<V&>(qv), u), lane_of<T>(rv, u));
      lane_of<T>(rv, u) = ri;
      acc = fma((double)ri, (double)ri, acc);
    }
    reinterpret_cast<V*>(x)[j] = xv;
    reinterpret_cast<V*>(r)[j] = rv;
  }
  for (int64_t i = nv * NV + gtid(); i < n; i += gstride()) {
    x[i] = fma(a, p[i], x[i]);
    const T ri = fma(-a, q[i], r[i]);
    r[i] = ri;
    acc = fma((double)ri, (double)ri, acc);
  }
  const double s = block_sum(acc);
  if (threadIdx.x == 0) {
    rr_part[blockIdx.x] = s;
    __threadfence();
    last_s = atomicAdd(&st->arrive_rr, 1) == (int)gridDim.x - 1;  // every block has read st->it
  }
  __syncthreads();
  if (last_s && threadIdx.x < 32) {
    __threadfence();
    const double rrn = warp_sum(rr_part, (int)gridDim.x);
    if (threadIdx.x == 0) {
      const int k = st->it;
      hist[k + 1] = rrn;
      st->beta = rrn / hist[k];
      st->arrive_rr = 0;
      st->it = k + 1;
      if (rrn <= st->tol2) {
        st->converged = 1;
        st->done = 1;
      } else if (!(rrn <= st->grow_limit)) {  // non-finite or diverging: stop this inner iteration
        st->breakdown = 1;
        st->done = 1;
      } else if (k + 1 >= st->max_iter) {
        st->done = 1;
      }
    }
  }
}

// K3: p = r + beta p (force: run although `done` is up -- the residual-replacement driver completes the
// iteration whose update raised the flag)
template <typename T>
__global__ void pupdate_kernel(int64_t n, T* __restrict__ p, const T* __restrict__ r, const CgState* st,
                               int force = 0) {
  if (st->done && !force) return;
  if (st->breakdown) return;
  using V = typename Vec16<T>::type;
  constexpr int NV = Vec16<T>::N;
  const T b = (T)st->beta;
  const int64_t nv = n / NV;
  for (int64_t j = gtid(); j < nv; j += gstride()) {
    V pv = reinterpret_cast<V*>(p)[j];
    V rv = reinterpret_cast<const V*>(r)[j];
#pragma unroll
    for (int u = 0; u < NV; ++u) lane_of<T>(pv, u) = fma(b, lane_of<T>(pv, u), lane_of<T>(rv, u));
    reinterpret_cast<V*>(p)[j] = pv;
  }
  for (int64_t i = nv * NV + gtid(); i < n; i += gstride()) p[i] = fma(b, p[i], r[i]);
}

// r = b - q (FP64) with partials of r.r
__global__ void residual_kernel(int64_t n, const double* __restrict__ b, const double* __restrict__ q, double* r,
                                double* part) {
  double acc = 0.0;
  for (int64_t i = gtid(); i < n; i += gstride()) {
    const double ri = b[i] - q[i];
    if (r) r[i] = ri;
    acc = fma(ri, ri, acc);
  }
  const double s = block_sum(acc);
  if (threadIdx.x == 0) part[blockIdx.x] = s;
}

// partials of a.b
__global__ void dot_kernel(int64_t n, const double* __restrict__ a, const double* __restrict__ b, double* part) {
  double acc = 0.0;
  for (int64_t i = gtid(); i < n; i += gstride()) acc = fma(a[i], b[i], acc);
  const double s = block_sum(acc);
  if (threadIdx.x == 0) part[blockIdx.x] = s;
}

// x += scale * d (FP64 update of the refinement)
__global__ void correct_kernel(int64_t n, double* x, const float* __restrict__ d, double scale) {
  for (int64_t i = gtid(); i < n; i += gstride()) x[i] = fma(scale, (double)d[i], x[i]);
}

// residual replacement: p32 *= ratio; r32 = r64 * inv_scale (FP32); d32 = 0; partials of r32.r32
__global__ void replace_kernel(int64_t n, const double* __restrict__ r64, double inv_scale, float ratio, float* r32,
                               float* p32, float* d32, double* part_a) {
  double ra = 0.0;
  for (int64_t i = gtid(); i < n; i += gstride()) {
    const float ri = (float)(r64[i] * inv_scale);
    r32[i] = ri;
    p32[i] *= ratio;
    d32[i] = 0.0f;
    ra = fma((double)ri, (double)ri, ra);
  }
  const double s = block_sum(ra);
  if (threadIdx.x == 0) part_a[blockIdx.x] = s;
}

// after a replacement: hist[it] = r32.r32, new trigger delta2 * r32.r32, iterations continue
__global__ void replace_finish_kernel(const double* part_a, int na, double delta2, double* hist, CgState* st) {
  if (threadIdx.x >= 32) return;
  const double rr = warp_sum(part_a, na);
  if (threadIdx.x == 0) {
    hist[st->it] = rr;
    st->tol2 = delta2 * rr;
    st->grow_limit = 1e12 * rr;
    st->arrive_dot = 0;
    st->arrive_rr = 0;
    st->converged = 0;
    st->breakdown = 0;
    st->done = st->it >= st->max_iter ? 1 : 0;
  }
}

// ---- flexible CG (Notay's FCG with one kept direction), FP64 outer, low-precision inner CG as the variable
// preconditioner z = B_k(r)

// z = r (use_r: the inner solve gave nothing) or z = scale * d (FP32 -> FP64); partials of z.q
__global__ void fcg_z_kernel(int64_t n, int use_r, const double* __restrict__ r, const float* __restrict__ d,
                             double scale, double* __restrict__ z, const double* __restrict__ q, double* part) {
  double acc = 0.0;
  for (int64_t i = gtid(); i < n; i += gstride()) {
    const double zi = use_r ? r[i] : scale * (double)d[i];
    z[i] = zi;
    acc = fma(zi, q[i], acc);
  }
  const double s = block_sum(acc);
  if (threadIdx.x == 0) part[blockIdx.x] = s;
}

// p = z + beta p; partials of p.r
__global__ void fcg_dir_kernel(int64_t n, const double* __restrict__ z, double beta, double* __restrict__ p,
                               const double* __restrict__ r, double* part) {
  double acc = 0.0;
  for (int64_t i = gtid(); i < n; i += gstride()) {
    const double pi = fma(beta, p[i], z[i]);
    p[i] = pi;
    acc = fma(pi, r[i], acc);
  }
  const double s = block_sum(acc);
  if (threadIdx.x == 0) part[blockIdx.x] = s;
}

// x += alpha p; r -= alpha q; partials of r.r
__global__ void fcg_update_kernel(int64_t n, double alpha, const double* __restrict__ p, const double* __restrict__ q,
                                  double* __restrict__ x, double* __restrict__ r, double* part) {
  double acc = 0.0;
  for (int64_t i = gtid(); i < n; i += gstride()) {
    x[i] = fma(alpha, p[i], x[i]);
    const double ri = fma(-alpha, q[i], r[i]);
    r[i] = ri;
    acc = fma(ri, ri, acc);
  }
  const double s = block_sum(acc);
  if (threadIdx.x == 0) part[blockIdx.x] = s;
}

// ---- persistent iterations: up to max_steps CG iterations (K1, K2, K3 of the launches above, the same arithmetic
// per element and the same order of every sum) in one cooperative launch, block p owning partition p's rows.  p stays
// in shared memory (it is the product's slice of x) and is mirrored to memory for the other blocks' extra rows; q, r
// and x stay there too as far as they fit (in that order: q is written and read twice an iteration, r read and
// written, x likewise but by one pass).  The blocks meet four times an iteration: for p.q, for the new r, which is
// mirrored to memory too since r.r is summed in the order of K2's threads (x is updated while r travels), for r.r and
// for the new p, which a warp waits for only when it comes to its first extra row.
template <typename X>
struct CgPersist {
  X *x, *r, *p, *q;                 // global vectors, plan numbering
  int32_t q_off, r_off, x_off;      // byte offsets in dynamic shared memory; -1: the vector stays in global memory
  int32_t red_off, tbl_off;         // the block sum's terms; the slice table (-1: none)
  int32_t max_steps;
  CgState* st;
  double* hist;
  persist::SyncArgs sync;
};

// A block's state, in shared memory: thread 0's scalars (it alone divides and decides) and where the vectors are.
template <typename V, typename X>
struct CgBlock {
  double alpha, beta, rr, tol2, grow_limit;
  int it, max_iter, converged, breakdown, done, stop, seen, nh;
  const int32_t* halo;
  X *q, *r, *x, *p;  // p: the block's rows of p in memory
  X* rm;             // r's mirror in memory (null: r lies there)
  const X* r_all;    // r of all blocks in memory
  int n;
  persist::Product<V, X> prod;
  double* hist;
  int32_t red_off;
  double sums[32];
  persist::SyncArgs sync;
};

// p.q and alpha
template <bool DOT, typename V, typename X>
__device__ __noinline__ void cg_step_pq(CgBlock<V, X>& sh, int round) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const X* const ps = reinterpret_cast<const X*>(smem_raw);
  const int warps = blockDim.x >> 5;
  double* const red = reinterpret_cast<double*>(smem_raw + sh.red_off);
  if constexpr (!DOT) {
    const X* const q = sh.q;
    persist::part_terms(sh.prod, warps, red, [&](int i) { return make_double2((double)q[i], (double)ps[i]); });
    __syncthreads();
  }
  if (threadIdx.x < 32 * persist::kSumWarps) persist::publish_part(sh.sync, round, 0, red, warps, sh.sums);
  double pq;
  const bool ok = persist::gather_sum(sh.sync, round, sh.sync.m->part[0], gridDim.x, red, &sh.stop, &pq);
  if (threadIdx.x == 0) {
    sh.prod.counter = warps;  // for the next product
    const double rr = sh.rr, alpha = ok && pq > 0.0 ? rr / pq : 0.0;
    // A is not positive definite along p: nothing is updated
    if (ok && !(alpha > 0.0) && rr > 0.0) sh.breakdown = sh.done = sh.stop = 1;
    sh.alpha = alpha;
  }
  __syncthreads();
}

template <typename V, typename X>
__device__ __noinline__ void cg_step_update(CgBlock<V, X>& sh, int round, int r_round) {
  constexpr int U = 4;  // elements a thread has in flight
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const X* const ps = reinterpret_cast<const X*>(smem_raw);
  const int bd = blockDim.x, tid = threadIdx.x, rows = sh.prod.rows;
  const X al = (X)sh.alpha;
  {  // r -= alpha q
    const X* const q = sh.q;
    X *const r = sh.r, *const rm = sh.rm;
    for (int i0 = tid; i0 < rows; i0 += U * bd) {
      X qv[U], rv[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int i = i0 + u * bd;
        qv[u] = i < rows ? q[i] : X(0);
        rv[u] = i < rows ? r[i] : X(0);
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int i = i0 + u * bd;
        if (i < rows) {
          rv[u] = fma(-al, qv[u], rv[u]);
          r[i] = rv[u];
          if (rm) rm[i] = rv[u];
        }
      }
    }
  }
  __syncthreads();
  if (tid == 0) persist::arrive(sh.sync);
  {  // x += alpha p while r is on its way
    X* const x = sh.x;
    for (int i0 = tid; i0 < rows; i0 += U * bd) {
      X xv[U], pv[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int i = i0 + u * bd;
        xv[u] = i < rows ? x[i] : X(0);
        pv[u] = i < rows ? ps[i] : X(0);
      }
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (i0 + u * bd < rows) x[i0 + u * bd] = fma(al, pv[u], xv[u]);
    }
  }
  if (tid == 0 && !persist::wait_block(sh.sync, r_round, &sh.seen)) sh.stop = 1;
  __syncthreads();
  if (sh.stop) return;
  double* const red = reinterpret_cast<double*>(smem_raw + sh.red_off);
  persist::publish_vec(sh.sync, round, sh.r_all, sh.n, red, sh.sums);
  double rrn;
  if (persist::gather_sum(sh.sync, round, sh.sync.m->vec, persist::vec_blocks<X>(sh.n), red, &sh.stop, &rrn) &&
      tid == 0) {
    const int it = sh.it + 1;
    if (blockIdx.x == 0) sh.hist[it] = rrn;
    sh.beta = rrn / sh.rr;
    sh.rr = rrn;
    sh.it = it;
    if (rrn <= sh.tol2) sh.converged = sh.stop = 1;
    else if (!(rrn <= sh.grow_limit)) sh.breakdown = sh.stop = 1;  // non-finite or diverging
    else if (it >= sh.max_iter) sh.stop = 1;
    sh.done = sh.stop;
  }
  __syncthreads();
}

template <typename V, typename X>
__device__ __noinline__ void cg_step_direction(CgBlock<V, X>& sh) {
  constexpr int U = 4;  // elements a thread has in flight
  extern __shared__ __align__(16) unsigned char smem_raw[];
  X* const ps = reinterpret_cast<X*>(smem_raw);
  const int bd = blockDim.x;
  // p = r + beta p
  {
    const X be = (X)sh.beta;
    const X* const r = sh.r;
    X* const p = sh.p;
    const int rows = sh.prod.rows;
    const int tid = threadIdx.x;
    for (int i0 = tid; i0 < rows; i0 += U * bd) {
      X pv[U], rv[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int i = i0 + u * bd;
        pv[u] = i < rows ? ps[i] : X(0);
        rv[u] = i < rows ? r[i] : X(0);
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int i = i0 + u * bd;
        if (i < rows) {
          const X pi = fma(be, pv[u], rv[u]);
          ps[i] = pi;
          p[i] = pi;
        }
      }
    }
  }
}

// MAXT 512 for blocks that are no larger: 128 registers a thread, and with them deeper batches (KB)
template <typename V, typename X, int KB, bool RUNS, int MAXT>
__global__ void __launch_bounds__(MAXT, 1) cg_persist_kernel(core::KArgs a, const V* __restrict__ ell_val,
                                                             const V* __restrict__ er_val, CgPersist<X> c) {
  using namespace core;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ CgBlock<V, X> sh;
  static_assert(sizeof(sh) <= persist::kMaxStatic, "static shared memory");
  X* const ps = reinterpret_cast<X*>(smem_raw);
  const int bd = blockDim.x;
  if (c.st->done) return;  // uniform over the grid: nobody writes it before every block has met the others
  {
    const int tid = threadIdx.x, blk = blockIdx.x;
    const int pb = a.part_ptr[blk], rows = a.part_ptr[blk + 1] - pb;
    X* r = c.r_off >= 0 ? reinterpret_cast<X*>(smem_raw + c.r_off) : c.r + pb;
    X* x = c.x_off >= 0 ? reinterpret_cast<X*>(smem_raw + c.x_off) : c.x + pb;
    if (tid == 0) {
      const int it = c.st->it;
      sh.it = it;
      sh.max_iter = c.st->max_iter;
      sh.tol2 = c.st->tol2;
      sh.grow_limit = c.st->grow_limit;
      sh.rr = c.hist[it];
      sh.beta = 0.0;
      sh.converged = sh.breakdown = sh.done = sh.stop = sh.seen = 0;
      sh.q = c.q_off >= 0 ? reinterpret_cast<X*>(smem_raw + c.q_off) : c.q + pb;
      sh.r = r;
      sh.x = x;
      sh.p = c.p + pb;
      sh.rm = c.r_off >= 0 ? c.r + pb : nullptr;
      sh.r_all = c.r;
      sh.n = (int)a.n;
      sh.hist = c.hist;
      sh.red_off = c.red_off;
      sh.sync = c.sync;
      sh.nh = a.halo_ptr ? (int)(a.halo_ptr[blk + 1] - a.halo_ptr[blk]) : 0;
      sh.halo = a.halo_ptr ? a.halo_new + a.halo_ptr[blk] : nullptr;
    }
    persist::init_product(&sh.prod, a, ell_val, er_val, a.er_scol, blk,
                          c.tbl_off >= 0 ? reinterpret_cast<SliceMeta*>(smem_raw + c.tbl_off) : nullptr);
    if (tid == 0) {
      sh.prod.xs_off = 0;
      sh.prod.counter = bd >> 5;
      sh.prod.xg = c.p;
      sh.prod.out = sh.q;
      sh.prod.lim = rows + sh.nh;
      sh.prod.stop = &sh.stop;
      sh.prod.seen = &sh.seen;
    }
    for (int i = tid; i < rows; i += bd) {
      ps[checked(i, a.smem_elems, a.status)] = c.p[pb + i];
      if (c.r_off >= 0) r[i] = c.r[pb + i];
      if (c.x_off >= 0) x[i] = c.x[pb + i];
    }
  }
  __syncthreads();
  for (int step = 0; step < c.max_steps; ++step) {
    // rounds of the sums p.q and r.r, and rounds of arrivals with r and p: 2 step + 1 and 2 step + 2 each
    const int round = 2 * step + 1;
    // q = A p; p of the other blocks from round 2 step on (their p at launch: nothing to wait for)
    if (sh.nh > 0) {
      if (!persist::wait_round(sh.sync, 2 * step, &sh.seen)) sh.stop = 1;
      for (int j = threadIdx.x; j < sh.nh; j += bd)
        ps[checked(sh.prod.rows + j, a.smem_elems, a.status)] = load_x(c.p + checked(sh.halo[j], a.n, a.status));
      __syncthreads();
    }
    persist::run_slices<V, X, KB, RUNS, false, persist::kDotInProduct<V, MAXT>>(
        &sh.prod, &sh.sync, 2 * step, reinterpret_cast<double*>(smem_raw + sh.red_off));
    __syncthreads();
    if (sh.stop) break;
    cg_step_pq<persist::kDotInProduct<V, MAXT>>(sh, round);
    if (sh.stop) break;
    cg_step_update(sh, round + 1, round);
    if (sh.stop) break;
    cg_step_direction(sh);
    __syncthreads();
    if (threadIdx.x == 0) persist::arrive(sh.sync);
  }
  __syncthreads();
  {
    const X* const x = sh.x;
    const int rows = sh.prod.rows, pb = sh.prod.pb;
    if (c.x_off >= 0)
      for (int i = threadIdx.x; i < rows; i += bd) c.x[pb + i] = x[i];
  }
  // a launch that ran out of steps leaves with p updated; one that gave up has told the host already
  if (blockIdx.x == 0 && threadIdx.x == 0 && (sh.done || !sh.stop)) {
    c.st->it = sh.it;
    c.st->beta = sh.beta;
    c.st->converged = sh.converged;
    c.st->breakdown = sh.breakdown;
    c.st->done = sh.done;
  }
}

double now_s() {
  return std::chrono::duration<double>(std::chrono::steady_clock::now().time_since_epoch()).count();
}

#define CKC(call)                                                     \
  do {                                                                \
    cudaError_t e_ = (call);                                          \
    if (e_ != cudaSuccess) return cuda_error_status(e_, #call);       \
  } while (0)

ehyb_status_t work_get(ehyb_plan_t P, int hist_need, CgWork** out) {
  CgWork* w = P->cg;
  const int64_t n = P->dev.n;
  if (w && w->hist_cap >= hist_need) {
    *out = w;
    return EHYB_OK;
  }
  if (w) {
    CKC(cudaDeviceSynchronize());
    cg_work_free(w);
    P->cg = nullptr;
  }
  w = new CgWork();
  w->n = n;
  w->nparts = P->dev.nparts;
  w->hist_cap = hist_need < 1024 ? 1024 : hist_need;
  auto al = [](size_t b) { return (b + 255) & ~(size_t)255; };
  const size_t v64 = al((size_t)(n + 2) * 8), v32 = al((size_t)(n + 4) * 4);
  const size_t parts = al((size_t)kVB * 8), pq = al((size_t)(w->nparts + 1) * 8);
  const size_t hist = al((size_t)(w->hist_cap + 2) * 8), st = al(sizeof(CgState));
  const size_t meeting = al(sizeof(persist::Meeting));
  const size_t total = 6 * v64 + 4 * v32 + 2 * parts + pq + hist + st + meeting;
  ehyb_status_t s = device_alloc(&w->arena, total);
  if (s != EHYB_OK) {
    delete w;
    return s;
  }
  char* b = (char*)w->arena;
  w->bp = (double*)b; b += v64;
  w->xp = (double*)b; b += v64;
  w->r = (double*)b; b += v64;
  w->p = (double*)b; b += v64;
  w->q = (double*)b; b += v64;
  w->xs = (double*)b; b += v64;
  w->r32 = (float*)b; b += v32;
  w->p32 = (float*)b; b += v32;
  w->q32 = (float*)b; b += v32;
  w->d32 = (float*)b; b += v32;
  w->part_a = (double*)b; b += parts;
  w->part_b = (double*)b; b += parts;
  w->pq_part = (double*)b; b += pq;
  w->hist = (double*)b; b += hist;
  w->st = (CgState*)b; b += st;
  w->meeting = (persist::Meeting*)b;
  cudaError_t e = cudaStreamCreateWithFlags(&w->cap, cudaStreamNonBlocking);
  if (e != cudaSuccess) {
    cg_work_free(w);
    return cuda_error_status(e, "cg workspace");
  }
  P->cg = w;
  *out = w;
  return EHYB_OK;
}

// FP64 iterations (lowp == 0) or inner FP32-vector iterations (lowp = 1 / 2), kChunk of them
ehyb_status_t enqueue_chunk(ehyb_plan_t P, CgWork* w, int lowp, cudaStream_t s) {
  const DevPlan& D = P->dev;
  const int64_t n = D.n;
  for (int k = 0; k < kChunk; ++k) {
    DotOut dot{w->pq_part, &w->st->arrive_dot, &w->st->pq};
    if (lowp == 0) {
      CKC(launch_ehyb_f64(D, w->p, w->q, 0, s, &dot, &w->st->done));
      update_kernel<double><<<kVB, kVT, 0, s>>>(n, w->xp, w->p, w->q, w->r, w->hist, w->st, w->part_a);
      pupdate_kernel<double><<<kVB, kVT, 0, s>>>(n, w->p, w->r, w->st);
    } else {
      CKC(launch_ehyb_lowp(D, lowp, w->p32, w->q32, 0, s, &dot, &w->st->done));
      update_kernel<float><<<kVB, kVT, 0, s>>>(n, w->d32, w->p32, w->q32, w->r32, w->hist, w->st, w->part_a);
      pupdate_kernel<float><<<kVB, kVT, 0, s>>>(n, w->p32, w->r32, w->st);
    }
    CKC(cudaGetLastError());
  }
  return EHYB_OK;
}

// one chunk through the plan's cached CUDA graph (captured on first use)
ehyb_status_t run_chunk(ehyb_plan_t P, CgWork* w, int lowp, cudaStream_t s) {
  cudaGraphExec_t* g = lowp == 0 ? &w->g64 : &w->g32;
  if (lowp && w->g32 && w->g32_lowp != lowp) {
    cudaGraphExecDestroy(w->g32);
    w->g32 = nullptr;
  }
  if (!*g) {
    cudaGraph_t graph;
    CKC(cudaStreamBeginCapture(w->cap, cudaStreamCaptureModeThreadLocal));
    ehyb_status_t st = enqueue_chunk(P, w, lowp, w->cap);
    cudaError_t e = cudaStreamEndCapture(w->cap, &graph);
    if (st != EHYB_OK) return st;
    CKC(e);
    e = cudaGraphInstantiate(g, graph, 0);
    cudaGraphDestroy(graph);
    CKC(e);
    if (lowp) w->g32_lowp = lowp;
  }
  CKC(cudaGraphLaunch(*g, s));
  return EHYB_OK;
}

// One persistent launch of at most kPersistSteps iterations; *ran = false (and nothing launched) for a plan that
// needs the separate launches: more partitions than SMs (a block owns one partition, all blocks resident), a wide
// slice (its sums go through the plan's workspace), more shared memory than persist::shared_budget grants, more rows
// a partition than persist::even_enough or, with FP32 vectors, kMaxRowsF32 / kMaxRowsBf16(Staged) allow, a time
// limit below kMinLimitNs, the staging-fault test hook.
constexpr int kPersistSteps = 2000;  // bounds one launch to a fraction of a second

template <typename V, typename X, int KB, bool RUNS, int MAXT>
ehyb_status_t launch_persist(ehyb_plan_t P, const V* ev, const V* erv, CgPersist<X> c, cudaStream_t s, bool* ran) {
  const DevPlan& D = P->dev;
  auto kernel = cg_persist_kernel<V, X, KB, RUNS, MAXT>;
  core::KArgs a = core::make_kargs(D);
  if (RUNS) {
    a.ell_col = D.ell_col_low;
    a.er_scol = D.er_scol_low;
  }
  int optin = 0, resident = 0, sms = 0;
  CKC(cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, P->device));
  CKC(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, P->device));
  if (!persist::even_enough(D.max_part_rows, D.n, sms, sizeof(X) == 8 ? persist::kSpare64 : persist::kSpare32))
    return EHYB_OK;
  auto al = [](size_t b) { return (b + 15) & ~(size_t)15; };
  size_t smem = ehyb_smem_bytes(D, (int)sizeof(X));
  a.smem_elems = (int64_t)(smem / sizeof(X));
  const size_t tbl = al((size_t)D.max_part_slices * sizeof(core::SliceMeta));
  const size_t vec = al((size_t)D.max_part_rows * sizeof(X));
  // with the slice table where that fits (ms a solve, separate launches -> without it -> with: tet 133^3 5.57, 5.62,
  // 5.31; 140^3 6.18, 6.69, 6.25)
  const size_t must = smem + persist::terms_bytes(D.threads), with_table = persist::shared_budget(must + tbl, 196);
  const size_t budget = std::min((size_t)(optin - persist::kMaxStatic),
                                 with_table ? with_table : persist::shared_budget(must, 196));
  auto place = [&](size_t bytes) -> int32_t {
    if (smem + bytes > budget) return -1;
    const size_t o = smem;
    smem += bytes;
    return (int32_t)o;
  };
  c.red_off = place(persist::terms_bytes(D.threads));
  c.tbl_off = place(tbl);
  a.meta_cap = D.max_part_slices;
  if (c.red_off < 0) return EHYB_OK;
  c.q_off = place(vec);
  c.r_off = place(vec);
  c.x_off = place(vec);
  CKC(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, optin - persist::kMaxStatic));
  CKC(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&resident, kernel, D.threads, smem));
  *ran = D.nparts <= sms * resident && D.nparts <= persist::kMaxGrid;
  if (!*ran) return EHYB_OK;
  CKC(persist::clear_meeting(c.sync.m, D.inject_wait_fault, s));
  void* args[] = {&a, (void*)&ev, (void*)&erv, &c};
  CKC(cudaLaunchCooperativeKernel((const void*)kernel, dim3((unsigned)D.nparts), dim3((unsigned)D.threads), args, smem,
                                  s));
  return EHYB_OK;
}

ehyb_status_t run_persist(ehyb_plan_t P, CgWork* w, int lowp, cudaStream_t s, bool* ran) {
  const DevPlan& D = P->dev;
  *ran = false;
  if (D.wide_parts > 0 || D.inject_wait_fault == 1 || D.wait_timeout_ns < persist::kMinLimitNs ||
      D.nparts > persist::kMaxGrid)
    return EHYB_OK;
  const persist::SyncArgs sync{w->meeting, D.status, &w->st->done, D.wait_timeout_ns};
  if (lowp == 0) {
    const CgPersist<double> c{w->xp, w->r, w->p, w->q, -1, -1, -1, -1, -1, kPersistSteps, w->st, w->hist, sync};
    if (D.threads <= 512) return launch_persist<double, double, 16, false, 512>(P, D.ell_val, D.er_sval, c, s, ran);
    return D.kbatch == 6 ? launch_persist<double, double, 6, false, 1024>(P, D.ell_val, D.er_sval, c, s, ran)
                         : launch_persist<double, double, 8, false, 1024>(P, D.ell_val, D.er_sval, c, s, ran);
  }
  if (D.max_part_rows > (lowp == 1       ? persist::kMaxRowsF32
                         : D.er_hcol_low ? persist::kMaxRowsBf16Staged
                                         : persist::kMaxRowsBf16))
    return EHYB_OK;
  const CgPersist<float> c{w->d32, w->r32, w->p32, w->q32, -1, -1, -1, -1, -1, kPersistSteps, w->st, w->hist, sync};
  const bool runs = D.lowp_group == 4, half = D.threads <= 512;
  if (lowp == 1)
    return !runs  ? launch_persist<float, float, 12, false, 1024>(P, D.ell_val_f32, D.er_sval_f32, c, s, ran)
           : half ? launch_persist<float, float, 32, true, 512>(P, D.ell_val_f32, D.er_sval_f32, c, s, ran)
                  : launch_persist<float, float, 16, true, 1024>(P, D.ell_val_f32, D.er_sval_f32, c, s, ran);
  return !runs  ? launch_persist<uint16_t, float, 12, false, 1024>(P, D.ell_val_bf16, D.er_sval_bf16, c, s, ran)
         : half ? launch_persist<uint16_t, float, 32, true, 512>(P, D.ell_val_bf16, D.er_sval_bf16, c, s, ran)
                : launch_persist<uint16_t, float, 16, true, 1024>(P, D.ell_val_bf16, D.er_sval_bf16, c, s, ran);
}

ehyb_status_t read_state(CgWork* w, cudaStream_t s, CgState* out) {
  CKC(cudaMemcpyAsync(out, w->st, sizeof(CgState), cudaMemcpyDeviceToHost, s));
  CKC(cudaStreamSynchronize(s));
  return EHYB_OK;
}

ehyb_status_t sum_parts(CgWork* w, cudaStream_t s, double* out) {
  double h[kVB];
  CKC(cudaMemcpyAsync(h, w->part_a, sizeof(h), cudaMemcpyDeviceToHost, s));
  CKC(cudaStreamSynchronize(s));
  double t = 0.0;
  for (int i = 0; i < kVB; ++i) t += h[i];
  *out = t;
  return EHYB_OK;
}

ehyb_status_t cg_loop(ehyb_plan_t P, CgWork* w, int lowp, cudaStream_t s, int* iters, int* converged,
                      int* breakdown);

// Flexible CG (Notay, "Flexible conjugate gradients", SIAM J. Sci. Comput. 22, 2000; truncation to one
// direction) in FP64 on the plan's FP64 values, from the x_p, r of w (r = b - A x_p, ||r||^2 = rr): each
// step applies the variable preconditioner z = B_k(r) = ||r|| d, d from an inner CG on the low-precision
// values (FP32 vectors, stopped at inner_rtol or inner_max iterations), then
//   p = z + beta p with beta = -(z . q_prev) / (p_prev . q_prev) (A-orthogonal to the previous direction),
//   q = A p, alpha = (p . r) / (p . q), x += alpha p, r -= alpha q.
// The recursive residual decides; on its convergence the true FP64 residual is recomputed and, if it is
// still too large, the iteration restarts from it.  *iters counts inner iterations, *outer the steps.
ehyb_status_t fcg_solve(ehyb_plan_t P, CgWork* w, int lowp, cudaStream_t s, double bnorm, double rtol, int max_iter,
                        double inner_rtol, double& rr, int* iters, int* outer, int* converged, double* rel_out) {
  const DevPlan& D = P->dev;
  const int64_t n = D.n;
  const int inner_max = 500;
  double* z = w->xs;
  double pq_prev = 0.0;
  bool restart = true;
  ehyb_status_t st;
  int true_checks = 0;
  for (;;) {
    const double rel = std::sqrt(rr) / bnorm;
    *rel_out = rel;
    if (rel <= rtol || rr == 0.0) {
      // confirm on the true residual (the recursive one may have drifted)
      CKC(launch_ehyb_f64(D, w->xp, w->q, 0, s));
      residual_kernel<<<kVB, kVT, 0, s>>>(n, w->bp, w->q, w->r, w->part_a);
      if ((st = sum_parts(w, s, &rr)) != EHYB_OK) return st;
      *rel_out = std::sqrt(rr) / bnorm;
      if (*rel_out <= rtol || rr == 0.0 || ++true_checks > 3) {
        *converged = *rel_out <= rtol || rr == 0.0;
        return EHYB_OK;
      }
      restart = true;  // continue from the true residual with a fresh direction
    }
    if (*iters >= max_iter || !std::isfinite(rr)) return EHYB_OK;
    // z = B(r): inner CG on the low-precision values, from 0, on r / ||r||
    const double rn = std::sqrt(rr);
    init32_kernel<<<kVB, kVT, 0, s>>>(n, w->r, 1.0 / rn, w->r32, w->p32, w->d32, w->part_a);
    const int cap = std::min(inner_max, max_iter - *iters);
    init_finish_kernel<<<1, 32, 0, s>>>(w->part_a, kVB, nullptr, 0, inner_rtol * inner_rtol, 1, cap, w->hist, w->st);
    CKC(cudaGetLastError());
    int it_in = 0, conv_in = 0, brk = 0;
    if ((st = cg_loop(P, w, lowp, s, &it_in, &conv_in, &brk)) != EHYB_OK) return st;
    *iters += it_in;
    // a first-iteration breakdown leaves d = 0: take the unpreconditioned step z = r
    fcg_z_kernel<<<kVB, kVT, 0, s>>>(n, it_in == 0 ? 1 : 0, w->r, w->d32, rn, z, w->q, w->part_a);
    double zq = 0.0;
    if ((st = sum_parts(w, s, &zq)) != EHYB_OK) return st;
    const double beta = (restart || !(pq_prev > 0.0)) ? 0.0 : -zq / pq_prev;
    fcg_dir_kernel<<<kVB, kVT, 0, s>>>(n, z, beta, w->p, w->r, w->part_a);
    double pr = 0.0;
    if ((st = sum_parts(w, s, &pr)) != EHYB_OK) return st;
    DotOut dot{w->pq_part, &w->st->arrive_dot, &w->st->pq};
    CKC(cudaMemsetAsync(&w->st->arrive_dot, 0, sizeof(int32_t), s));
    CKC(launch_ehyb_f64(D, w->p, w->q, 0, s, &dot));
    double pq = 0.0;
    CKC(cudaMemcpyAsync(&pq, &w->st->pq, sizeof(double), cudaMemcpyDeviceToHost, s));
    CKC(cudaStreamSynchronize(s));
    ++*outer;
    if (!(pq > 0.0)) return EHYB_OK;  // A is not positive definite along p: stop (not converged)
    if (!(pr > 0.0)) {                 // not a descent direction: restart from z = B(r) alone
      if (restart) return EHYB_OK;
      restart = true;
      continue;
    }
    fcg_update_kernel<<<kVB, kVT, 0, s>>>(n, pr / pq, w->p, w->q, w->xp, w->r, w->part_a);
    if ((st = sum_parts(w, s, &rr)) != EHYB_OK) return st;
    pq_prev = pq;
    restart = false;
  }
}

// CG loop on the vectors of w (FP64 or inner FP32); returns iterations and convergence
ehyb_status_t cg_loop(ehyb_plan_t P, CgWork* w, int lowp, cudaStream_t s, int* iters, int* converged,
                      int* breakdown) {
  CgState h;
  bool persistent = true;
  for (;;) {
    ehyb_status_t st = EHYB_OK;
    if (persistent) st = run_persist(P, w, lowp, s, &persistent);
    if (st == EHYB_OK && !persistent) st = run_chunk(P, w, lowp, s);
    if (st != EHYB_OK) return st;
    if ((st = read_state(w, s, &h)) != EHYB_OK) return st;
    if (h.done == persist::kAborted) return EHYB_ERR_TIMEOUT;
    if (h.done) break;
  }
  *iters = h.it;
  *converged = h.converged;
  if (breakdown) *breakdown = h.breakdown;
  return EHYB_OK;
}

}  // namespace

}  // namespace ehyb

using namespace ehyb;

extern "C" ehyb_status_t ehyb_cg(ehyb_plan_t P, const double* b, double* x, double rtol, int32_t max_iter,
                                 int32_t refine, double inner_rtol, ehyb_cg_info_t* info, void* stream) {
  if (!P || !info) return EHYB_ERR_INVALID_ARG;
  std::memset(info, 0, sizeof(*info));
  if (P->host_only) return EHYB_ERR_UNSUPPORTED;
  if (refine < 0 || refine > 6 || !(rtol >= 0.0) || max_iter < 0) return EHYB_ERR_INVALID_ARG;
  const int lowp = refine == 0 ? 0 : (refine % 2 == 1) ? 1 : 2;
  if (refine && P->lowp != lowp) return EHYB_ERR_UNSUPPORTED;  // the plan lacks that value copy
  if (P->er_layout == 1) return EHYB_ERR_UNSUPPORTED;            // the fused dot needs every row final after its slice
  const int64_t n = P->dev.n;
  const double t0 = now_s();
  if (n == 0) {
    info->converged = 1;
    return EHYB_OK;
  }
  if (!b || !x) return EHYB_ERR_INVALID_ARG;
  cudaStream_t s = (cudaStream_t)stream;
  CgWork* w = nullptr;
  ehyb_status_t st = work_get(P, max_iter + 2, &w);
  if (st != EHYB_OK) return st;
  const DevPlan& D = P->dev;
  CKC(launch_permute_f64(D, 1, b, w->bp, s));
  CKC(launch_permute_f64(D, 1, x, w->xp, s));
  // ||b||
  dot_kernel<<<kVB, kVT, 0, s>>>(n, w->bp, w->bp, w->part_a);
  double bb = 0.0;
  if ((st = sum_parts(w, s, &bb)) != EHYB_OK) return st;
  const double bnorm = bb > 0.0 ? std::sqrt(bb) : 1.0;

  int converged = 0, iters = 0, outer = 0;
  // a stalled BF16 refinement (refine 2 / 4) hands its x and FP64 residual (w->r, rr_stall) to the flexible CG
  bool stalled = false;
  double rr_stall = 0.0;
  if (refine >= 5) {
    CKC(launch_ehyb_f64(D, w->xp, w->q, 0, s));
    residual_kernel<<<kVB, kVT, 0, s>>>(n, w->bp, w->q, w->r, w->part_a);
    double rr = 0.0;
    if ((st = sum_parts(w, s, &rr)) != EHYB_OK) return st;
    double rel = 0.0;
    const double irtol = inner_rtol > 0.0 ? inner_rtol : kFcgInnerRtol;
    if ((st = fcg_solve(P, w, lowp, s, bnorm, rtol, max_iter, irtol, rr, &iters, &outer, &converged, &rel)) != EHYB_OK)
      return st;
    info->relres_recursive = rel;
    info->flexible = 1;
  } else if (refine == 0) {
    CKC(launch_ehyb_f64(D, w->xp, w->q, 0, s));
    init64_kernel<<<kVB, kVT, 0, s>>>(n, w->bp, w->q, w->r, w->p, w->part_a, w->part_b);
    init_finish_kernel<<<1, 32, 0, s>>>(w->part_a, kVB, w->part_b, kVB, rtol * rtol, 0, max_iter, w->hist, w->st);
    CKC(cudaGetLastError());
    if ((st = cg_loop(P, w, 0, s, &iters, &converged, nullptr)) != EHYB_OK) return st;
    double rr_last = 0.0;
    CKC(cudaMemcpyAsync(&rr_last, w->hist + iters, sizeof(double), cudaMemcpyDeviceToHost, s));
    CKC(cudaStreamSynchronize(s));
    info->relres_recursive = std::sqrt(rr_last) / bnorm;
  } else if (refine >= 3) {
    // residual replacement: low-precision CG iterations that keep their search direction; whenever the
    // low-precision residual has dropped by `delta`, x += s d in FP64, the residual is recomputed in FP64
    // and the iteration continues on it (p rescaled, not restarted)
    const double delta = inner_rtol > 0.0 ? inner_rtol : 0.1;
    CKC(launch_ehyb_f64(D, w->xp, w->q, 0, s));
    residual_kernel<<<kVB, kVT, 0, s>>>(n, w->bp, w->q, w->r, w->part_a);
    double rr = 0.0;
    if ((st = sum_parts(w, s, &rr)) != EHYB_OK) return st;
    double scale = std::sqrt(rr);
    if (scale / bnorm <= rtol || rr == 0.0) {
      converged = 1;
    } else {
      init32_kernel<<<kVB, kVT, 0, s>>>(n, w->r, 1.0 / scale, w->r32, w->p32, w->d32, w->part_a);
      init_finish_kernel<<<1, 32, 0, s>>>(w->part_a, kVB, nullptr, 0, delta * delta, 1, max_iter, w->hist, w->st);
      CKC(cudaGetLastError());
      double prev_rr = rr;
      int rejections = 0;
      for (;;) {
        int it_in = 0, conv_in = 0, brk = 0;
        if ((st = cg_loop(P, w, lowp, s, &it_in, &conv_in, &brk)) != EHYB_OK) return st;
        iters = it_in;
        // the direction update of the iteration that raised the trigger was skipped with it
        if (conv_in) pupdate_kernel<float><<<kVB, kVT, 0, s>>>(n, w->p32, w->r32, w->st, 1);
        CKC(cudaMemcpyAsync(w->xs, w->xp, (size_t)n * 8, cudaMemcpyDeviceToDevice, s));
        correct_kernel<<<kVB, kVT, 0, s>>>(n, w->xp, w->d32, scale);
        CKC(launch_ehyb_f64(D, w->xp, w->q, 0, s));
        residual_kernel<<<kVB, kVT, 0, s>>>(n, w->bp, w->q, w->r, w->part_a);
        if ((st = sum_parts(w, s, &rr)) != EHYB_OK) return st;
        ++outer;
        bool rejected = false;
        if (!(rr < prev_rr)) {  // the correction did not help (or is not finite): undo it
          rejected = true;
          CKC(cudaMemcpyAsync(w->xp, w->xs, (size_t)n * 8, cudaMemcpyDeviceToDevice, s));
          CKC(launch_ehyb_f64(D, w->xp, w->q, 0, s));
          residual_kernel<<<kVB, kVT, 0, s>>>(n, w->bp, w->q, w->r, w->part_a);
          if ((st = sum_parts(w, s, &rr)) != EHYB_OK) return st;
        }
        const double rel = std::sqrt(rr) / bnorm;
        info->relres_recursive = rel;
        if (rel <= rtol) { converged = 1; break; }
        rejections = rejected ? rejections + 1 : 0;
        if (rejections >= 3 && std::isfinite(rr) && rr > 0.0) {
          stalled = true;
          rr_stall = rr;
        }
        if (iters >= max_iter || rr == 0.0 || !std::isfinite(rr) || rejections >= 3) break;
        const double ns = std::sqrt(rr);
        if (brk || rejected) {
          // lost positive definiteness along p, or no progress: restart the direction from the residual
          init32_kernel<<<kVB, kVT, 0, s>>>(n, w->r, 1.0 / ns, w->r32, w->p32, w->d32, w->part_a);
        } else {
          replace_kernel<<<kVB, kVT, 0, s>>>(n, w->r, 1.0 / ns, (float)(scale / ns), w->r32, w->p32, w->d32,
                                             w->part_a);
        }
        replace_finish_kernel<<<1, 32, 0, s>>>(w->part_a, kVB, delta * delta, w->hist, w->st);
        CKC(cudaGetLastError());
        scale = ns;
        prev_rr = rr;
      }
    }
  } else {
    // FP64 residual outside, FP32-vector CG on the low-precision values inside
    const double irtol = inner_rtol > 0.0 ? inner_rtol : (refine == 1 ? 1e-4 : 1e-2);
    const int outer_max = 60;
    double prev = 0.0;
    for (;;) {
      CKC(launch_ehyb_f64(D, w->xp, w->q, 0, s));
      residual_kernel<<<kVB, kVT, 0, s>>>(n, w->bp, w->q, w->r, w->part_a);
      double rr = 0.0;
      if ((st = sum_parts(w, s, &rr)) != EHYB_OK) return st;
      const double rel = std::sqrt(rr) / bnorm;
      info->relres_recursive = rel;
      if (rel <= rtol) { converged = 1; break; }
      if (iters < max_iter && std::isfinite(rr) && (outer >= outer_max || (outer > 0 && !(rel < prev)))) {
        stalled = true;
        rr_stall = rr;
      }
      if (outer >= outer_max || iters >= max_iter || (outer > 0 && !(rel < prev))) break;
      prev = rel;
      ++outer;
      const double rnorm = std::sqrt(rr);
      init32_kernel<<<kVB, kVT, 0, s>>>(n, w->r, 1.0 / rnorm, w->r32, w->p32, w->d32, w->part_a);
      init_finish_kernel<<<1, 32, 0, s>>>(w->part_a, kVB, nullptr, 0, irtol * irtol, 1, max_iter - iters, w->hist,
                                          w->st);
      CKC(cudaGetLastError());
      int it_in = 0, conv_in = 0;
      if ((st = cg_loop(P, w, lowp, s, &it_in, &conv_in, nullptr)) != EHYB_OK) return st;
      iters += it_in;
      correct_kernel<<<kVB, kVT, 0, s>>>(n, w->xp, w->d32, rnorm);
      CKC(cudaGetLastError());
    }
  }
  if (stalled && lowp == 2 && !converged && iters < max_iter) {
    // BF16 values and u_bf16 kappa(A) near or above 1: the refinement stalls; the flexible CG keeps the
    // BF16 solve as a preconditioner only and lets the FP64 outer iteration carry the accuracy
    double rel = 0.0;
    if ((st = fcg_solve(P, w, lowp, s, bnorm, rtol, max_iter, kFcgInnerRtol, rr_stall, &iters, &outer, &converged,
                        &rel)) != EHYB_OK)
      return st;
    info->relres_recursive = rel;
    info->flexible = 1;
  }
  // true residual in FP64, then x back to the original numbering
  CKC(launch_ehyb_f64(D, w->xp, w->q, 0, s));
  residual_kernel<<<kVB, kVT, 0, s>>>(n, w->bp, w->q, nullptr, w->part_a);
  double rr = 0.0;
  if ((st = sum_parts(w, s, &rr)) != EHYB_OK) return st;
  CKC(launch_permute_f64(D, 0, w->xp, x, s));
  CKC(cudaStreamSynchronize(s));
  info->iterations = iters;
  info->refinements = outer;
  info->relres = std::sqrt(rr) / bnorm;
  info->converged = converged;
  info->seconds = now_s() - t0;
  int32_t dev_status = 0;
  CKC(cudaMemcpy(&dev_status, P->dev.status, sizeof(int32_t), cudaMemcpyDeviceToHost));
  if (dev_status) return (ehyb_status_t)dev_status;
  return converged ? EHYB_OK : EHYB_ERR_NOT_CONVERGED;
}

extern "C" ehyb_status_t ehyb_cg_history(ehyb_plan_t P, double* hist, int32_t cap, int32_t* count) {
  if (!P || !count || (cap > 0 && !hist)) return EHYB_ERR_INVALID_ARG;
  *count = 0;
  if (!P->cg) return EHYB_OK;
  CgState h;
  CKC(cudaDeviceSynchronize());
  CKC(cudaMemcpy(&h, P->cg->st, sizeof(h), cudaMemcpyDeviceToHost));
  const int m = h.it + 1 < cap ? h.it + 1 : cap;
  if (m > 0) CKC(cudaMemcpy(hist, P->cg->hist, (size_t)m * sizeof(double), cudaMemcpyDeviceToHost));
  *count = m;
  return EHYB_OK;
}
