// The tuner network: a 3-layer perceptron 16 -> 64 -> 64 -> 4 (ReLU after the hidden layers, linear
// output), FP32, with hand-written forward, mean-squared-error backward and Adam kernels.  It is not in
// the paper: it is the learned-knob subsystem built around the method (it predicts the partition size
// of Eq. 1/2, the slab width cap and the lanes per row).
//
// Parameters are one flat array in this order (row-major): W1 (64x16), b1 (64), W2 (64x64), b2 (64),
// W3 (4x64), b3 (4) -- 5,508 floats.  A batch X is B x 16 row-major, targets T and outputs B x 4.
// Every reduction (over the batch for weight gradients, over the outputs for the loss) runs in a fixed
// order, so gradients and training runs are bit-reproducible.
//
// A step has less than a microsecond of arithmetic (43 MFLOP at 2,000 samples), so launches, dependent passes
// over small buffers and long serial sums are what it costs.  One thread per output element and one kernel
// per layer and direction took 395 us a step at 2,000 samples, 640 us of cold kernel time in the three weight
// gradients alone (a thread summed all samples one after the other).  Now the batch is cut into blocks of 16
// or more samples: a block keeps the whole network in shared memory and takes its samples through the
// forward pass, the loss and the backward pass, its weight gradients held in registers (a 4 x 4 tile of the
// 64 x 64 layer a thread); a second kernel sums the blocks' gradients.  Now 19 us a step at 2,000 samples, most
// of it the calls.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "ehyb_core.cuh"
#include "plan_internal.h"

namespace ehyb {
namespace {

using core::pdl_launch_dependents;
using core::pdl_wait;

constexpr int D0 = 16, D1 = 64, D2 = 64, D3 = 4;
constexpr int OW1 = 0, OB1 = OW1 + D1 * D0, OW2 = OB1 + D1, OB2 = OW2 + D2 * D1, OW3 = OB2 + D2, OB3 = OW3 + D3 * D2;
constexpr int NPARAM = OB3 + D3;
static_assert(NPARAM == 5508, "parameter count");

constexpr int kTS = 16;      // samples a block works on at a time (and the fewest a block is given)
constexpr int kMlpT = 256;   // threads: 64 units x 4 groups of 4 samples
constexpr int LX = D0 + 4;   // padded rows: every row starts on 16 bytes, and 8 lanes reading 16 bytes of 8
constexpr int LH = D1 + 4;   //   consecutive rows touch all banks once
constexpr int kWsPerSample = 2 * D1 + 2 * D2 + 3 * D3 + D2 + D1;  // floats of workspace the ABI asks for
constexpr int kPart = NPARAM + 4;  // one block's gradient, then its squared-error sum (a double as two words)
constexpr int kMaxBlocks = 1216;   // 8 per SM: bounds the second kernel's sums

struct MlpSmem {
  float w1[D1 * LX], w2[D2 * LH], w3[D3 * LH], b1[D1], b2[D2], b3[D3];
  float x[kTS * LX], h1[kTS * LH], h2[kTS * LH], d2[kTS * LH], d1[kTS * LH], dout[kTS * D3];
};
static_assert(sizeof(MlpSmem) <= 48 * 1024, "static shared memory");

__device__ __forceinline__ float4 ld4(const float* p) { return *reinterpret_cast<const float4*>(p); }

// h[b][o] = relu(bias[o] + sum_i W[o][i] in[b][i]) for this thread's unit o and 4 samples, inputs in order
template <int K, int LI>
__device__ __forceinline__ void dense_relu(const float* W, const float* bias, const float* in, int o, int b0,
                                           float* h) {
  float s[4];
#pragma unroll
  for (int u = 0; u < 4; ++u) s[u] = bias[o];
#pragma unroll 4
  for (int i = 0; i < K; i += 4) {
    const float4 w = ld4(W + o * LI + i);
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const float4 v = ld4(in + (b0 + u) * LI + i);
      s[u] = fmaf(w.w, v.w, fmaf(w.z, v.z, fmaf(w.y, v.y, fmaf(w.x, v.x, s[u]))));
    }
  }
#pragma unroll
  for (int u = 0; u < 4; ++u) h[(b0 + u) * LH + o] = s[u] < 0.0f ? 0.0f : s[u];
}

// One block's samples [blockIdx.x * per, ...): forward (BWD false: outputs to `out`), or forward, squared error
// against T and the gradient summed over the block's samples, to part + kPart * blockIdx.x; with `direct` (one
// block) the mean-squared-error loss and the gradient themselves.  Global reads are scalar: the caller's
// arrays are aligned to their element only.  No __restrict__ on what an earlier kernel of the stream may still
// be writing when this one becomes resident: such loads must not be moved across the wait.
template <bool BWD>
__global__ void __launch_bounds__(kMlpT) mlp_kernel(const float* P, const float* X, const float* T, int B, int per, float* part,
                                                    float* grad, float* loss, int direct) {
  __shared__ __align__(16) MlpSmem m;
  const int t = threadIdx.x;
  const int o = t & 63, b0 = (t >> 6) * 4;
  pdl_launch_dependents();
  pdl_wait();
  for (int i = t; i < D1 * D0; i += kMlpT) m.w1[(i / D0) * LX + i % D0] = P[OW1 + i];
  for (int i = t; i < D2 * D1; i += kMlpT) m.w2[(i / D1) * LH + i % D1] = P[OW2 + i];
  for (int i = t; i < D3 * D2; i += kMlpT) m.w3[(i / D2) * LH + i % D2] = P[OW3 + i];
  if (t < D1) m.b1[t] = P[OB1 + t];
  if (t < D2) m.b2[t] = P[OB2 + t];
  if (t < D3) m.b3[t] = P[OB3 + t];
  const int first = blockIdx.x * per, end = min(B, first + per);
  const float scale = (float)(B * (int64_t)D3);
  // this thread's sums: W2 rows 4 (t/16).. x columns 4 (t%16).., W1 row t/4 x columns 4 (t%4).., one W3, one bias
  float g2[4][4] = {}, g1[4] = {}, g3 = 0.0f, gb = 0.0f;
  double sq = 0.0;
  for (int s0 = first; s0 < end; s0 += kTS) {
    const int cnt = min(kTS, end - s0);
    __syncthreads();
    for (int i = t; i < kTS * D0; i += kMlpT)
      m.x[(i / D0) * LX + i % D0] = i / D0 < cnt ? X[(int64_t)s0 * D0 + i] : 0.0f;
    __syncthreads();
    dense_relu<D0, LX>(m.w1, m.b1, m.x, o, b0, m.h1);
    __syncthreads();
    dense_relu<D1, LH>(m.w2, m.b2, m.h1, o, b0, m.h2);
    __syncthreads();
    if (t < kTS * D3) {  // linear output of sample t / 4, unit t % 4
      const int b = t / D3, q = t % D3;
      float s = m.b3[q];
#pragma unroll 4
      for (int i = 0; i < D2; i += 4) {
        const float4 w = ld4(m.w3 + q * LH + i), v = ld4(m.h2 + b * LH + i);
        s = fmaf(w.w, v.w, fmaf(w.z, v.z, fmaf(w.y, v.y, fmaf(w.x, v.x, s))));
      }
      if (!BWD) {
        if (b < cnt) part[(int64_t)(s0 + b) * D3 + q] = s;
      } else if (b < cnt) {
        const float e = s - T[(int64_t)(s0 + b) * D3 + q];
        m.dout[t] = 2.0f * e / scale;
        sq += (double)(e * e);
      } else {
        m.dout[t] = 0.0f;
      }
    }
    if (!BWD) continue;
    __syncthreads();
    {  // back through layer 3 and the second ReLU
      float s[4] = {};
#pragma unroll
      for (int q = 0; q < D3; ++q)
#pragma unroll
        for (int u = 0; u < 4; ++u) s[u] = fmaf(m.dout[(b0 + u) * D3 + q], m.w3[q * LH + o], s[u]);
#pragma unroll
      for (int u = 0; u < 4; ++u) m.d2[(b0 + u) * LH + o] = m.h2[(b0 + u) * LH + o] > 0.0f ? s[u] : 0.0f;
    }
    __syncthreads();
    {  // back through layer 2 and the first ReLU
      float s[4] = {};
#pragma unroll 4
      for (int q = 0; q < D2; q += 4) {
        float4 d[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) d[u] = ld4(m.d2 + (b0 + u) * LH + q);
        const float w0 = m.w2[q * LH + o], w1 = m.w2[(q + 1) * LH + o], w2 = m.w2[(q + 2) * LH + o],
                    w3 = m.w2[(q + 3) * LH + o];
#pragma unroll
        for (int u = 0; u < 4; ++u)
          s[u] = fmaf(d[u].w, w3, fmaf(d[u].z, w2, fmaf(d[u].y, w1, fmaf(d[u].x, w0, s[u]))));
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) m.d1[(b0 + u) * LH + o] = m.h1[(b0 + u) * LH + o] > 0.0f ? s[u] : 0.0f;
    }
    __syncthreads();
    // weight gradients of the valid samples only (a padding sample's activations may not be finite)
#pragma unroll 2
    for (int b = 0; b < cnt; ++b) {
      const float4 d = ld4(m.d2 + b * LH + 4 * (t >> 4)), v = ld4(m.h1 + b * LH + 4 * (t & 15));
      const float dd[4] = {d.x, d.y, d.z, d.w}, vv[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
      for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int k = 0; k < 4; ++k) g2[u][k] = fmaf(dd[u], vv[k], g2[u][k]);
      const float e = m.d1[b * LH + (t >> 2)];
      const float4 xv = ld4(m.x + b * LX + 4 * (t & 3));
      g1[0] = fmaf(e, xv.x, g1[0]);
      g1[1] = fmaf(e, xv.y, g1[1]);
      g1[2] = fmaf(e, xv.z, g1[2]);
      g1[3] = fmaf(e, xv.w, g1[3]);
      g3 = fmaf(m.dout[b * D3 + (t >> 6)], m.h2[b * LH + o], g3);
      if (t < D1) gb += m.d1[b * LH + t];
      else if (t < D1 + D2) gb += m.d2[b * LH + t - D1];
      else if (t < D1 + D2 + D3) gb += m.dout[b * D3 + t - D1 - D2];
    }
  }
  if (!BWD) return;
  float* g = direct ? grad : part + (int64_t)blockIdx.x * kPart;
#pragma unroll
  for (int u = 0; u < 4; ++u)
#pragma unroll
    for (int k = 0; k < 4; ++k) g[OW2 + (4 * (t >> 4) + u) * D1 + 4 * (t & 15) + k] = g2[u][k];
#pragma unroll
  for (int k = 0; k < 4; ++k) g[OW1 + (t >> 2) * D0 + 4 * (t & 3) + k] = g1[k];
  g[OW3 + t] = g3;
  if (t < D1) g[OB1 + t] = gb;
  else if (t < D1 + D2) g[OB2 + t - D1] = gb;
  else if (t < D1 + D2 + D3) g[OB3 + t - D1 - D2] = gb;
  __shared__ double ws[2];
  if (t < kTS * D3) {
    for (int off = 16; off > 0; off >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, off);
    if ((t & 31) == 0) ws[t >> 5] = sq;
  }
  __syncthreads();
  if (t == 0) {
    const double s = ws[0] + ws[1];
    if (direct) {
      *loss = (float)(s / (double)((int64_t)B * D3));
    } else {
      g[NPARAM] = __int_as_float(__double2loint(s));
      g[NPARAM + 1] = __int_as_float(__double2hiint(s));
    }
  }
}

// gradient = sum of the blocks' partial gradients, loss = the mean of their squared errors.  32 parameters a
// block, eight warps each summing every eighth partial, then the eight sums in order; the last block takes
// the loss.
__global__ void __launch_bounds__(256) mlp_reduce(const float* part, int nb, int B, float* grad,
                                                  float* loss) {
  __shared__ float ws[8][32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  pdl_launch_dependents();
  pdl_wait();
  if (blockIdx.x == gridDim.x - 1) {
    if (warp) return;
    double s = 0.0;
    for (int b = lane; b < nb; b += 32) {
      const float* q = part + (int64_t)b * kPart + NPARAM;
      s += __hiloint2double(__float_as_int(q[1]), __float_as_int(q[0]));
    }
    for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
    if (lane == 0) *loss = (float)(s / (double)((int64_t)B * D3));
    return;
  }
  const int i = blockIdx.x * 32 + lane;
  float s = 0.0f;
  if (i < NPARAM) {
#pragma unroll 8
    for (int b = warp; b < nb; b += 8) s += part[(int64_t)b * kPart + i];
  }
  ws[warp][lane] = s;
  __syncthreads();
  if (warp == 0 && i < NPARAM) {
    float r = ws[0][lane];
#pragma unroll
    for (int w = 1; w < 8; ++w) r += ws[w][lane];
    grad[i] = r;
  }
}

__global__ void adam_kernel(float* p, float* m, float* v, const float* g, int count, float lr,
                            float b1, float b2, float eps, float c1, float c2) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  pdl_launch_dependents();
  pdl_wait();
  if (t >= count) return;
  const float gi = g[t];
  const float mi = b1 * m[t] + (1.0f - b1) * gi;
  const float vi = b2 * v[t] + (1.0f - b2) * gi * gi;
  m[t] = mi;
  v[t] = vi;
  p[t] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
}

inline int nblk(int64_t work) { return (int)((work + 255) / 256); }

// every launch carries the programmatic-stream-serialization attribute: a kernel's blocks become resident
// under the previous one's tail and wait there (pdl_wait) before they touch memory
template <typename... A>
cudaError_t launch(void (*k)(A...), int grid, int threads, cudaStream_t s, A... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3((unsigned)threads);
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k, args...);
}

}  // namespace
}  // namespace ehyb

using namespace ehyb;

extern "C" int32_t ehyb_mlp_param_count(void) { return NPARAM; }

extern "C" int64_t ehyb_mlp_workspace_bytes(int32_t batch) {
  if (batch < 0) return -1;
  return (int64_t)batch * kWsPerSample * (int64_t)sizeof(float);
}

extern "C" ehyb_status_t ehyb_mlp_forward(const float* params, const float* X, int32_t batch, float* out,
                                          void* workspace, void* stream) {
  if (!params || !X || !out || batch < 0 || (batch > 0 && !workspace)) return EHYB_ERR_INVALID_ARG;
  if (batch == 0) return EHYB_OK;
  // outputs in X's own memory: a block would write over samples that another has yet to read
  const uintptr_t x0 = reinterpret_cast<uintptr_t>(X), o0 = reinterpret_cast<uintptr_t>(out);
  const size_t xb = (size_t)batch * D0 * sizeof(float), ob = (size_t)batch * D3 * sizeof(float);
  if (x0 < o0 + ob && o0 < x0 + xb) {
    const cudaError_t e = cudaMemcpyAsync(workspace, X, xb, cudaMemcpyDeviceToDevice, (cudaStream_t)stream);
    if (e != cudaSuccess) return cuda_error_status(e, "mlp forward");
    X = (const float*)workspace;
  }
  const int per = (int)std::max<int64_t>(kTS, ((int64_t)batch + kMaxBlocks - 1) / kMaxBlocks);
  const int nb = (int)(((int64_t)batch + per - 1) / per);
  const cudaError_t e = launch(mlp_kernel<false>, nb, kMlpT, (cudaStream_t)stream, params, X, (const float*)nullptr,
                               (int)batch, per, out, (float*)nullptr, (float*)nullptr, 0);
  return e == cudaSuccess ? EHYB_OK : cuda_error_status(e, "mlp forward");
}

extern "C" ehyb_status_t ehyb_mlp_loss_grad(const float* params, const float* X, const float* T, int32_t batch,
                                            float* grad, float* loss, void* workspace, void* stream) {
  if (!params || !X || !T || !grad || !loss || batch <= 0 || !workspace) return EHYB_ERR_INVALID_ARG;
  cudaStream_t s = (cudaStream_t)stream;
  const int B = batch;
  // at least 16 samples a block, and no more blocks than partial gradients fit the caller's workspace
  const int64_t fit = (int64_t)B * kWsPerSample / kPart;
  const int64_t want = std::max<int64_t>(1, std::min<int64_t>({((int64_t)B + kTS - 1) / kTS, fit, kMaxBlocks}));
  const int per = (int)(((int64_t)B + want - 1) / want);
  const int nb = (int)(((int64_t)B + per - 1) / per);
  cudaError_t e = launch(mlp_kernel<true>, nb, kMlpT, s, params, X, T, B, per, (float*)workspace, grad, loss,
                         nb == 1 ? 1 : 0);
  if (e == cudaSuccess && nb > 1)
    e = launch(mlp_reduce, (NPARAM + 31) / 32 + 1, 256, s, (const float*)workspace, nb, B, grad, loss);
  return e == cudaSuccess ? EHYB_OK : cuda_error_status(e, "mlp backward");
}

extern "C" ehyb_status_t ehyb_mlp_adam(float* params, float* m, float* v, const float* grad, int32_t step, float lr,
                                       float beta1, float beta2, float eps, void* stream) {
  if (!params || !m || !v || !grad || step < 1) return EHYB_ERR_INVALID_ARG;
  const float c1 = 1.0f - powf(beta1, (float)step), c2 = 1.0f - powf(beta2, (float)step);
  const cudaError_t e = launch(adam_kernel, nblk(NPARAM), 256, (cudaStream_t)stream, params, m, v, grad, (int)NPARAM,
                               lr, beta1, beta2, eps, c1, c2);
  return e == cudaSuccess ? EHYB_OK : cuda_error_status(e, "mlp adam");
}
