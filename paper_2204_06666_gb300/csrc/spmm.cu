// EHYB SpMM: Y = A X for k right-hand sides (X, Y row-major n x k, original numbering).
//
// FP64 SpMM on this part is bound by the FP64 FMA pipe k times over (k FMAs per 10-byte slab slot), so
// the plan's Eq. 1 partitions are kept (no re-partitioning for smaller slices, no extra ER) and the
// columns are processed in chunks of KC in {8, 4, 2, 1}: the largest KC whose KC-column slice of X fits
// one block's shared memory and divides k.  Each chunk is one launch with one block per partition that
// gathers its rows' KC columns of X through the permutation into shared memory (KC consecutive doubles of a
// row: whole 32-byte sectors from KC = 4 up), walks the slab and the sliced ER slots of its slices exactly like
// the SpMV (same slot order, so column j of Y equals ehyb_spmv of column j bit for bit) and writes KC outputs
// per row into Y[new_to_old[r]][c*KC + j].  Re-streaming the slab once per chunk costs far less time than
// the chunk's FMAs.
#include <cuda_runtime.h>

#include <algorithm>
#include <type_traits>

#include "ehyb_core.cuh"
#include "plan_internal.h"

namespace ehyb {
namespace {

using namespace core;

// KC columns of one row, 16 bytes at a time where the rows allow it (VEC: X and Y on 16 bytes, k and KC even)
template <int KC, bool VEC>
struct RowCols {
  double v[KC];
  __device__ __forceinline__ void ldg(const double* p) {
    if constexpr (VEC) {
#pragma unroll
      for (int j = 0; j < KC; j += 2) {
        const double2 d = load_x2(p + j);
        v[j] = d.x;
        v[j + 1] = d.y;
      }
    } else {
#pragma unroll
      for (int j = 0; j < KC; ++j) v[j] = load_x(p + j);
    }
  }
};

template <int KC, bool VEC>
__global__ void __launch_bounds__(512) spmm_kernel(KArgs a, const double* __restrict__ ell_val,
                                                   const double* __restrict__ er_val, const double* __restrict__ X,
                                                   double* __restrict__ Y, int k, int c0) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ BlockState bs;
  const int p = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarps = blockDim.x >> 5;
  const int pb = a.part_ptr[p], pe = a.part_ptr[p + 1];
  const int s0 = a.slice_ptr[p], s1 = a.slice_ptr[p + 1];
  double* xs = reinterpret_cast<double*>(smem_raw);
  if (tid == 0) bs.slice_counter = s0 + nwarps;
  pdl_launch_dependents();
  pdl_wait();
  const double* Xc = X + c0;  // this chunk's columns of row r: Xc[r * k + j]
  {
    // xs[(r - pb) * KC + j]: 8 elements (VEC: pairs) per thread in flight
    constexpr int W = VEC ? 2 : 1, N = 8, PR = KC / W;
    const int total = (pe - pb) * PR;
    for (int i0 = tid; i0 < total; i0 += N * blockDim.x) {
      int64_t src[N];
#pragma unroll
      for (int u = 0; u < N; ++u) {
        const int i = i0 + u * blockDim.x;
        src[u] = i < total ? (int64_t)checked(__ldg(a.new_to_old + pb + i / PR), a.n, a.status) * k + (i % PR) * W : -1;
      }
      double v[N * W];
#pragma unroll
      for (int u = 0; u < N; ++u) {
        if constexpr (VEC) {
          const double2 d = src[u] >= 0 ? load_x2(Xc + src[u]) : make_double2(0.0, 0.0);
          v[2 * u] = d.x;
          v[2 * u + 1] = d.y;
        } else {
          v[u] = src[u] >= 0 ? load_x(Xc + src[u]) : 0.0;
        }
      }
#pragma unroll
      for (int u = 0; u < N; ++u) {
        const int i = i0 + u * blockDim.x;
        if (i >= total) break;
        double* d = xs + checked(i * W, a.smem_elems - W + 1, a.status);
        if constexpr (VEC) *reinterpret_cast<double2*>(d) = make_double2(v[2 * u], v[2 * u + 1]);
        else *d = v[u];
      }
    }
  }
  __syncthreads();
  const int tpr = 1 << a.tpr_log2;
  const int sub = lane & (tpr - 1);
  const int rows_per_slice = 32 >> a.tpr_log2;

  int s = s0 + warp;
  while (s < s1) {
    double acc[KC];
#pragma unroll
    for (int j = 0; j < KC; ++j) acc[j] = 0.0;
    const int64_t pos = a.slice_pos[s];
    const int w = (int)((a.slice_pos[s + 1] - pos) >> 5);
    const double* vp = ell_val + pos + lane;
    const uint16_t* cp = a.ell_col + pos + lane;
    const int64_t epos = a.er_slice_pos[s];
    const int we = (int)((a.er_slice_pos[s + 1] - epos) >> 5);
    const double* evp = er_val + epos + lane;
    const int32_t* ecp = a.er_scol_old + epos + lane;
    // slab slots [k0, k1) into q[0..KC)
    auto slab = [&](int k0, int k1, double (&q)[KC]) {
      for (int kk = k0; kk < k1; ++kk) {
        const double v = __ldcs(vp + 32 * (int64_t)kk);
        const int c = checked((int)__ldcs(reinterpret_cast<const unsigned short*>(cp + 32 * (int64_t)kk)), pe - pb, a.status);
        const double* xr = xs + c * KC;
#pragma unroll
        for (int j = 0; j < KC; ++j) q[j] = fma(v, xr[j], q[j]);
      }
    };
    // N extra-row slots from kk on: their columns, then their rows of X, then the FMAs in slot order.  The loads of X
    // keep their order (load_x), so slot by slot each waited for its column and its row in turn; a small plan's few
    // warps cannot hide that, nor a long slice's chain (us, k = 2 / 3 / 8 / 16, slot by slot -> in batches: power-law
    // 12k rows 476 / 650 / 920 / 1840 -> 314 / 463 / 582 / 1163, elasticity 20^3 34.6 / 72.7 / 64.1 / 127 -> 31.3 /
    // 69.6 / 55.8 / 111, tet 40^3 13.1 / 25.8 / 22.0 / 44.5 -> 10.0 / 23.0 / 20.4 / 41.0).
    auto batch = [&](auto count, int kk, double (&q)[KC]) {
      constexpr int N = decltype(count)::value;
      double v[N];
      int64_t c[N];
      RowCols<KC, VEC> xr[N];
#pragma unroll
      for (int u = 0; u < N; ++u) {
        v[u] = __ldcs(evp + 32 * (int64_t)(kk + u));
        c[u] = (int64_t)checked(__ldcs(ecp + 32 * (int64_t)(kk + u)), a.n, a.status) * k;
      }
#pragma unroll
      for (int u = 0; u < N; ++u) xr[u].ldg(Xc + c[u]);
#pragma unroll
      for (int u = 0; u < N; ++u)
#pragma unroll
        for (int j = 0; j < KC; ++j) q[j] = fma(v[u], xr[u].v[j], q[j]);
    };
    // extra-row slots [k0, k1)
    auto extra = [&](int k0, int k1, double (&q)[KC]) {
      constexpr int N = KC == 8 ? 4 : KC == 4 ? 6 : KC == 2 ? 12 : 12;
      int kk = k0;
#pragma unroll 1
      for (; kk + N <= k1; kk += N) batch(std::integral_constant<int, N>(), kk, q);
      if constexpr (N > 4)
#pragma unroll 1
        for (; kk + 4 <= k1; kk += 4) batch(std::integral_constant<int, 4>(), kk, q);
      if (kk + 2 <= k1) {
        batch(std::integral_constant<int, 2>(), kk, q);
        kk += 2;
      }
      if (kk < k1) batch(std::integral_constant<int, 1>(), kk, q);
    };
    const int cap = a.wide_parts > 0 ? kWideCap : 0x7fffffff;
    slab(0, min(w, cap), acc);
    extra(0, min(we, cap), acc);
    if (w > cap || we > cap) {  // a wide slice's later chunks, summed as the SpMV sums them
      double t[KC];
#pragma unroll
      for (int j = 0; j < KC; ++j) t[j] = 0.0;
#pragma unroll 1
      for (int part = 0; part < 2; ++part)
#pragma unroll 1
        for (int k = kWideCap; k < (part ? we : w); k += kWideCap) {
          double q[KC];
#pragma unroll
          for (int j = 0; j < KC; ++j) q[j] = 0.0;
          if (part) extra(k, min(k + kWideCap, we), q);
          else slab(k, min(k + kWideCap, w), q);
#pragma unroll
          for (int j = 0; j < KC; ++j) t[j] += q[j];
        }
#pragma unroll
      for (int j = 0; j < KC; ++j) acc[j] += t[j];
    }
#pragma unroll
    for (int j = 0; j < KC; ++j)
      for (int off = tpr >> 1; off > 0; off >>= 1) acc[j] += __shfl_xor_sync(FULL, acc[j], off);
    const int row = pb + (s - s0) * rows_per_slice + (lane >> a.tpr_log2);
    if (sub == 0 && row < pe) {
      double* yr = Y + (int64_t)checked(a.new_to_old[row], a.n, a.status) * k + c0;
      if constexpr (VEC) {
#pragma unroll
        for (int j = 0; j < KC; j += 2) *reinterpret_cast<double2*>(yr + j) = make_double2(acc[j], acc[j + 1]);
      } else {
#pragma unroll
        for (int j = 0; j < KC; ++j) yr[j] = acc[j];
      }
    }
    int nxt = 0;
    if (lane == 0) nxt = atomicAdd(&bs.slice_counter, 1);
    s = __shfl_sync(FULL, nxt, 0);
  }
}

template <int KC, bool VEC>
cudaError_t launch_chunk(const DevPlan& D, int smem_max, const double* X, double* Y, int k, int c0, size_t smem,
                         cudaStream_t s) {
  cudaError_t e = cudaFuncSetAttribute(spmm_kernel<KC, VEC>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_max);
  if (e != cudaSuccess) return e;
  KArgs a = make_kargs(D);
  a.smem_elems = (int64_t)(smem / sizeof(double));
  // chunk after chunk overlaps the next one's launch with the tail of the one before (pdl_wait orders the data)
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)D.nparts);
  cfg.blockDim = dim3(512);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, spmm_kernel<KC, VEC>, a, D.ell_val, D.er_sval, X, Y, k, c0);
}

}  // namespace
}  // namespace ehyb

using namespace ehyb;

extern "C" ehyb_status_t ehyb_spmm(ehyb_plan_t P, int32_t k, const double* X, double* Y, void* stream) {
  if (!P || k < 1) return EHYB_ERR_INVALID_ARG;
  if (P->host_only || P->er_layout != 0) return EHYB_ERR_UNSUPPORTED;
  const DevPlan& D = P->dev;
  if (D.n == 0) return EHYB_OK;
  if (!X || !Y || (const void*)X == (const void*)Y) return EHYB_ERR_INVALID_ARG;
  int dev = 0, optin = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (e != cudaSuccess) return cuda_error_status(e, "device query");
  const size_t budget = (size_t)optin - 1024;
  int kc = 0;
  for (int c : {8, 4, 2, 1}) {
    const size_t need = ((size_t)(D.max_part_rows + 1) * c + 2) * 8;
    if (k % c == 0 && need <= budget) { kc = c; break; }
  }
  if (kc == 0) return EHYB_ERR_TOO_LARGE;
  const size_t need = ((((size_t)(D.max_part_rows + 1) * kc + 2) * 8) + 15) & ~(size_t)15;
  cudaStream_t s = (cudaStream_t)stream;
  const int smax = (int)budget;
  const bool vec = k % 2 == 0 && ((reinterpret_cast<uintptr_t>(X) | reinterpret_cast<uintptr_t>(Y)) & 15u) == 0;
  for (int c = 0; c < k / kc; ++c) {
    switch (kc) {
      case 8: e = vec ? launch_chunk<8, true>(D, smax, X, Y, k, c * kc, need, s) : launch_chunk<8, false>(D, smax, X, Y, k, c * kc, need, s); break;
      case 4: e = vec ? launch_chunk<4, true>(D, smax, X, Y, k, c * kc, need, s) : launch_chunk<4, false>(D, smax, X, Y, k, c * kc, need, s); break;
      case 2: e = vec ? launch_chunk<2, true>(D, smax, X, Y, k, c * kc, need, s) : launch_chunk<2, false>(D, smax, X, Y, k, c * kc, need, s); break;
      default: e = launch_chunk<1, false>(D, smax, X, Y, k, c * kc, need, s); break;
    }
    if (e != cudaSuccess) return cuda_error_status(e, "spmm launch");
  }
  return EHYB_OK;
}
