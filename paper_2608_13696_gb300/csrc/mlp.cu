// The planner's network: 264 sketch features -> 64 -> 64 -> 4 outputs
// (log2 of the number of groups, and logits of the three group-by variants:
// CTA-private tables, one global table, partitioned).  Weights are stored in
// FP32 (the optimiser's master copy) with a BF16 copy used by the forward and
// backward passes; the BF16 operands are multiplied and accumulated in FP32
// (a BF16 x BF16 product is exact in FP32).  Inputs and hidden activations
// are rounded to BF16 where they enter a layer.  Hidden layers use ReLU.
//
// Loss per sample: (y0 - log2 ndv)^2 + cross-entropy(softmax(y1..y3), label),
// averaged over the batch.  The network is tiny (21,380 parameters), so the
// kernels are plain per-thread dot products; nothing here is a contraction
// worth tensor cores.
#include <cuda_bf16.h>

#include "mlp.cuh"

namespace rel {

namespace {

__device__ __forceinline__ float bf(float x) { return __bfloat162float(__float2bfloat16_rn(x)); }

__device__ __forceinline__ float wbf(const __nv_bfloat16* w, int i) {
  return __bfloat162float(w[i]);
}

// Every kernel here is latency: a few hundred dependent multiply-adds per
// output on weights that fit one SM.  A thread reading its own weight row from
// global memory, two bytes at a time, waited for each (forward 17 us, gradients
// 23 us on a batch of 256), so the weights and the batch's gradients now come
// to shared memory first, in whole words.  The order of every sum is that of
// the plain loop over k (or over the batch), so results do not depend on it.
constexpr int FW_SAMPLES = 4;                  // samples per CTA at a time
constexpr int FW_BLOCK = FW_SAMPLES * MLP_H;
// words (two weights) per staged row: odd, so that consecutive rows start on
// different banks
constexpr int FW_LD1 = MLP_IN / 2 + 1, FW_LD2 = MLP_H / 2 + 1;

// ROWS x COLS BF16 weights at w into dst, ld words a row (COLS / 2 of them
// used).  All of a thread's loads go out before the first store.
template <int ROWS, int COLS>
__device__ __forceinline__ void stage_rows(uint32_t* dst, int ld, const __nv_bfloat16* w) {
  constexpr int VEC = COLS / 8;  // 16-byte pieces per row
  constexpr int PER = (ROWS * VEC + FW_BLOCK - 1) / FW_BLOCK;
  if (((uintptr_t)w & 15) == 0) {
    uint4 v[PER];
#pragma unroll
    for (int q = 0; q < PER; ++q) {
      const int i = threadIdx.x + q * FW_BLOCK;
      if (i < ROWS * VEC) v[q] = __ldg((const uint4*)w + i);
    }
#pragma unroll
    for (int q = 0; q < PER; ++q) {
      const int i = threadIdx.x + q * FW_BLOCK;
      if (i >= ROWS * VEC) continue;
      uint32_t* d = dst + i / VEC * ld + i % VEC * 4;
      d[0] = v[q].x; d[1] = v[q].y; d[2] = v[q].z; d[3] = v[q].w;
    }
    return;
  }
  for (int i = threadIdx.x; i < ROWS * COLS / 2; i += FW_BLOCK) {  // any alignment
    const unsigned short* e = (const unsigned short*)(w + 2 * i);
    dst[i / (COLS / 2) * ld + i % (COLS / 2)] = (uint32_t)e[0] | (uint32_t)e[1] << 16;
  }
}
__device__ __forceinline__ float lo_bf(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float hi_bf(uint32_t w) { return __uint_as_float(w & 0xFFFF0000u); }

// sum_k w[k] * x[k] in the order of k
template <int K>
__device__ __forceinline__ float dot(const uint32_t* w, const float* x) {
  float z = 0.f;
#pragma unroll 12
  for (int k = 0; k < K / 2; ++k) {
    const uint32_t ww = w[k];
    const float2 xx = *(const float2*)(x + 2 * k);
    z = fmaf(lo_bf(ww), xx.x, z);
    z = fmaf(hi_bf(ww), xx.y, z);
  }
  return z;
}

__global__ void __launch_bounds__(FW_BLOCK) mlp_fwd_k(const __nv_bfloat16* __restrict__ wb,
                                                      const float* __restrict__ pf,
                                                      const float* __restrict__ x, int batch,
                                                      float* __restrict__ out,
                                                      float* __restrict__ acts) {
  __shared__ uint32_t w1[MLP_H * FW_LD1], w2[MLP_H * FW_LD2], w3[MLP_OUT * FW_LD2];
  __shared__ __align__(8) float xin[FW_SAMPLES][MLP_IN], h1[FW_SAMPLES][MLP_H], h2[FW_SAMPLES][MLP_H];
  stage_rows<MLP_H, MLP_IN>(w1, FW_LD1, wb + OFF_W1);
  stage_rows<MLP_H, MLP_H>(w2, FW_LD2, wb + OFF_W2);
  stage_rows<MLP_OUT, MLP_H>(w3, FW_LD2, wb + OFF_W3);
  const int q = threadIdx.x / MLP_H, j = threadIdx.x % MLP_H;
  const float b1 = pf[OFF_B1 + j], b2 = pf[OFF_B2 + j];
  for (int b0 = blockIdx.x * FW_SAMPLES; b0 < batch; b0 += gridDim.x * FW_SAMPLES) {
    const int b = b0 + q;
    const bool in = b < batch;
#pragma unroll
    for (int k = j; k < MLP_IN; k += MLP_H) xin[q][k] = in ? bf(x[(size_t)b * MLP_IN + k]) : 0.f;
    __syncthreads();
    float z = dot<MLP_IN>(w1 + j * FW_LD1, xin[q]) + b1;
    h1[q][j] = bf(z > 0.f ? z : 0.f);
    if (acts && in) acts[(size_t)b * ACT_STRIDE + j] = z;
    __syncthreads();
    z = dot<MLP_H>(w2 + j * FW_LD2, h1[q]) + b2;
    h2[q][j] = bf(z > 0.f ? z : 0.f);
    if (acts && in) acts[(size_t)b * ACT_STRIDE + MLP_H + j] = z;
    __syncthreads();
    if (j < MLP_OUT && in)
      out[(size_t)b * MLP_OUT + j] = dot<MLP_H>(w3 + j * FW_LD2, h2[q]) + pf[OFF_B3 + j];
    // the next samples' inputs are read by no one before the barrier after them
  }
}

// Output gradient of a sample (mean loss over the batch) and its loss.
__device__ __forceinline__ float out_grad(const float* y, float t, int lab, float inv_b, float* d) {
  const float e = y[0] - t;
  const float m = fmaxf(y[1], fmaxf(y[2], y[3]));
  const float s1 = expf(y[1] - m), s2 = expf(y[2] - m), s3 = expf(y[3] - m);
  const float sum = s1 + s2 + s3;
  const float p[3] = {s1 / sum, s2 / sum, s3 / sum};
  d[0] = 2.f * e * inv_b;
  for (int c = 0; c < 3; ++c) d[1 + c] = (p[c] - (c == lab ? 1.f : 0.f)) * inv_b;
  const float ce = logf(sum) + m - y[1 + lab];
  return (e * e + ce) * inv_b;
}

// Per-sample part of the backward pass: output gradient, then dz2, dz1
// (gradients at the hidden pre-activations).
__global__ void __launch_bounds__(FW_BLOCK) mlp_bwd_sample_k(
    const __nv_bfloat16* __restrict__ wb, const float* __restrict__ acts,
    const float* __restrict__ out, const float* __restrict__ t_ndv,
    const int32_t* __restrict__ t_var, int batch, float* __restrict__ dz) {
  __shared__ __align__(16) __nv_bfloat16 w2[MLP_H * MLP_H];
  __shared__ float dout[FW_SAMPLES][MLP_OUT], d2[FW_SAMPLES][MLP_H];
  stage_rows<MLP_H, MLP_H>((uint32_t*)w2, MLP_H / 2, wb + OFF_W2);
  const int q = threadIdx.x / MLP_H, j = threadIdx.x % MLP_H, b = blockIdx.x * FW_SAMPLES + q;
  const bool in = b < batch;
  if (j == 0 && in) {
    float d[MLP_OUT];
    out_grad(out + (size_t)b * MLP_OUT, t_ndv[b], t_var[b], 1.f / (float)batch, d);
    for (int c = 0; c < MLP_OUT; ++c) dz[(size_t)b * DZ_STRIDE + 2 * MLP_H + c] = dout[q][c] = d[c];
  }
  const float z2 = in ? acts[(size_t)b * ACT_STRIDE + MLP_H + j] : 0.f;
  const float z1 = in ? acts[(size_t)b * ACT_STRIDE + j] : 0.f;
  __syncthreads();
  // dh2[j] = sum_o W3[o][j] dout[o]; dz2 = dh2 where z2 > 0
  float g = 0.f;
#pragma unroll
  for (int o = 0; o < MLP_OUT; ++o) g = fmaf(wbf(wb, OFF_W3 + o * MLP_H + j), dout[q][o], g);
  const float g2 = z2 > 0.f ? g : 0.f;
  d2[q][j] = g2;
  if (in) dz[(size_t)b * DZ_STRIDE + MLP_H + j] = g2;
  __syncthreads();
  // dh1[j] = sum_i W2[i][j] dz2[i]; dz1 = dh1 where z1 > 0
  g = 0.f;
#pragma unroll 8
  for (int i = 0; i < MLP_H; ++i) g = fmaf(__bfloat162float(w2[i * MLP_H + j]), d2[q][i], g);
  if (in) dz[(size_t)b * DZ_STRIDE + j] = z1 > 0.f ? g : 0.f;
}

// Parameter gradients grad[j][k] = sum_b d[b][j] h[b][k], tiles of 64 rows j by
// PG_COLS columns k, the batch PG_STAGE samples at a time through shared
// memory: W1's tiles, then W2's, then one CTA for W3, the biases and the loss.
constexpr int PG_COLS = 4, PG_STAGE = 64, PG_BLOCK = 64 * PG_COLS;
constexpr int PG_W1 = MLP_IN / PG_COLS, PG_W2 = MLP_H / PG_COLS;
static_assert(MLP_IN % PG_COLS == 0 && MLP_H % PG_COLS == 0, "whole tiles");

__global__ void __launch_bounds__(PG_BLOCK) mlp_bwd_param_k(
    const float* __restrict__ x, const float* __restrict__ acts, const float* __restrict__ dz,
    const float* __restrict__ out, const float* __restrict__ t_ndv,
    const int32_t* __restrict__ t_var, int batch, float* __restrict__ grad,
    float* __restrict__ loss) {
  static_assert(PG_COLS == MLP_OUT && PG_BLOCK == PG_STAGE * PG_COLS, "one staged value per thread");
  __shared__ __align__(16) float d[PG_STAGE][MLP_H], h[PG_STAGE][PG_COLS];
  const int tile = blockIdx.x, tid = threadIdx.x, j = tid % 64, c = tid / 64;
  if (tile < PG_W1 + PG_W2) {
    const bool first = tile < PG_W1;
    const int k0 = (first ? tile : tile - PG_W1) * PG_COLS;
    float s = 0.f;
    for (int b0 = 0; b0 < batch; b0 += PG_STAGE) {
      const int nb = batch - b0 < PG_STAGE ? batch - b0 : PG_STAGE;
      __syncthreads();
      constexpr int VEC = MLP_H / 4, PER = PG_STAGE * VEC / PG_BLOCK;
      float4 v[PER];  // all loads of the stage in flight before the first store
      float hv = 0.f;
#pragma unroll
      for (int q = 0; q < PER; ++q) {
        const int b = (tid + q * PG_BLOCK) / VEC;
        if (b < nb)
          v[q] = *(const float4*)(dz + (size_t)(b0 + b) * DZ_STRIDE + (first ? 0 : MLP_H) +
                                  4 * ((tid + q * PG_BLOCK) % VEC));
      }
      if (tid / PG_COLS < nb) {
        const size_t b = b0 + tid / PG_COLS;
        const int k = k0 + tid % PG_COLS;
        hv = first ? x[b * MLP_IN + k] : acts[b * ACT_STRIDE + k];
        if (!first) hv = hv > 0.f ? hv : 0.f;
      }
#pragma unroll
      for (int q = 0; q < PER; ++q) {
        const int b = (tid + q * PG_BLOCK) / VEC;
        if (b < nb) ((float4*)d[b])[(tid + q * PG_BLOCK) % VEC] = v[q];
      }
      h[tid / PG_COLS][tid % PG_COLS] = bf(hv);
      __syncthreads();
#pragma unroll 8
      for (int b = 0; b < nb; ++b) s = fmaf(d[b][j], h[b][c], s);
    }
    grad[(first ? OFF_W1 + j * MLP_IN : OFF_W2 + j * MLP_H) + k0 + c] = s;
    return;
  }
  if (tile == PG_W1 + PG_W2) {  // W3[o][k]: dout[o] * h2[k]; one output per thread
    const int o = tid / MLP_H, k = tid % MLP_H;
    float s = 0.f;
    for (int b0 = 0; b0 < batch; b0 += PG_STAGE) {
      const int nb = batch - b0 < PG_STAGE ? batch - b0 : PG_STAGE;
      __syncthreads();
#pragma unroll 4
      for (int b = o; b < nb; b += MLP_OUT) {
        const float z2 = acts[(size_t)(b0 + b) * ACT_STRIDE + MLP_H + k];
        d[b][k] = bf(z2 > 0.f ? z2 : 0.f);
      }
      if (tid < nb * MLP_OUT) h[tid / MLP_OUT][tid % MLP_OUT] = dz[(size_t)(b0 + tid / MLP_OUT) * DZ_STRIDE + 2 * MLP_H + tid % MLP_OUT];
      __syncthreads();
#pragma unroll 8
      for (int b = 0; b < nb; ++b) s = fmaf(h[b][o], d[b][k], s);
    }
    grad[OFF_W3 + tid] = s;
    return;
  }
  // biases: sums of dz over the batch, in its order
  if (tid < 2 * MLP_H + MLP_OUT) {
    float s = 0.f;
#pragma unroll 32
    for (int b = 0; b < batch; ++b) s += dz[(size_t)b * DZ_STRIDE + tid];
    grad[tid < MLP_H ? OFF_B1 + tid : tid < 2 * MLP_H ? OFF_B2 + tid - MLP_H : OFF_B3 + tid - 2 * MLP_H] = s;
  } else {
    // the other threads: the loss
    const int lane = tid & 31, first = 2 * MLP_H + 32;  // whole warps from here on
    if (tid < first) return;
    float l = 0.f, dd[MLP_OUT];
    for (int b = tid - first; b < batch; b += PG_BLOCK - first)
      l += out_grad(out + (size_t)b * MLP_OUT, t_ndv[b], t_var[b], 1.f / (float)batch, dd);
#pragma unroll
    for (int o = 16; o; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
    if (lane == 0) d[0][tid >> 5] = l;
    asm volatile("bar.sync 1, %0;" ::"n"(PG_BLOCK - 2 * MLP_H - 32) : "memory");
    if (tid == first) {
      l = 0.f;
      for (int w = first / 32; w < PG_BLOCK / 32; ++w) l += d[0][w];
      *loss = l;
    }
  }
}

// AdamW (Loshchilov & Hutter 2019): decoupled weight decay on the weights
// (not the biases), bias-corrected moments; refreshes the BF16 copy.
__global__ void mlp_adamw_k(float* __restrict__ p, __nv_bfloat16* __restrict__ wb,
                            float* __restrict__ m, float* __restrict__ v,
                            const float* __restrict__ g, MlpAdamW h) {
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= MLP_PARAMS) return;
  const bool is_bias = (q >= OFF_B1 && q < OFF_W2) || (q >= OFF_B2 && q < OFF_W3) || q >= OFF_B3;
  const float gq = g[q];
  const float mq = h.beta1 * m[q] + (1.f - h.beta1) * gq;
  const float vq = h.beta2 * v[q] + (1.f - h.beta2) * gq * gq;
  m[q] = mq;
  v[q] = vq;
  const float mhat = mq / h.bc1, vhat = vq / h.bc2;
  float pq = p[q];
  if (!is_bias) pq -= h.lr * h.wd * pq;
  pq -= h.lr * mhat / (sqrtf(vhat) + h.eps);
  p[q] = pq;
  wb[q] = __float2bfloat16_rn(pq);
}

__global__ void mlp_round_k(const float* __restrict__ p, __nv_bfloat16* __restrict__ wb) {
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q < MLP_PARAMS) wb[q] = __float2bfloat16_rn(p[q]);
}

rel_status done(const char* what) {
  const cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? REL_OK : relhost::cuda_fail(e, what);
}

}  // namespace

rel_status mlp_round(const float* p, void* wb, cudaStream_t st) {
  relhost::launch_begin(relhost::K_MLP, st);
  mlp_round_k<<<(MLP_PARAMS + 255) / 256, 256, 0, st>>>(p, (__nv_bfloat16*)wb);
  relhost::launch_end(relhost::K_MLP, st);
  return done("launch(mlp round)");
}

rel_status mlp_forward(const void* wb, const float* p, const float* x, int batch, float* out,
                       float* acts, cudaStream_t st) {
  if (batch == 0) return REL_OK;
  relhost::launch_begin(relhost::K_MLP, st);
  const int grid = (batch + FW_SAMPLES - 1) / FW_SAMPLES, most = 4 * relhost::device_sms();
  mlp_fwd_k<<<grid < most ? grid : most, FW_BLOCK, 0, st>>>((const __nv_bfloat16*)wb, p, x, batch, out, acts);
  relhost::launch_end(relhost::K_MLP, st);
  return done("launch(mlp forward)");
}

rel_status mlp_backward(const void* wb, const float* x, const float* acts, const float* out,
                        const float* t_ndv, const int32_t* t_var, int batch, float* dz,
                        float* grad, float* loss, cudaStream_t st) {
  if (batch == 0) {
    cudaError_t e = cudaMemsetAsync(loss, 0, sizeof(float), st);
    if (e == cudaSuccess) e = cudaMemsetAsync(grad, 0, sizeof(float) * MLP_PARAMS, st);
    return e == cudaSuccess ? REL_OK : relhost::cuda_fail(e, "cudaMemsetAsync");
  }
  relhost::launch_begin(relhost::K_MLP, st);
  mlp_bwd_sample_k<<<(batch + FW_SAMPLES - 1) / FW_SAMPLES, FW_BLOCK, 0, st>>>(
      (const __nv_bfloat16*)wb, acts, out, t_ndv, t_var, batch, dz);
  relhost::launch_end(relhost::K_MLP, st);
  rel_status r = done("launch(mlp backward)");
  if (r) return r;
  relhost::launch_begin(relhost::K_MLP, st);
  mlp_bwd_param_k<<<PG_W1 + PG_W2 + 2, PG_BLOCK, 0, st>>>(x, acts, dz, out, t_ndv, t_var, batch, grad, loss);
  relhost::launch_end(relhost::K_MLP, st);
  return done("launch(mlp gradients)");
}

rel_status mlp_adamw(float* p, void* wb, float* m, float* v, const float* g, const MlpAdamW& h,
                     cudaStream_t st) {
  relhost::launch_begin(relhost::K_MLP, st);
  mlp_adamw_k<<<(MLP_PARAMS + 255) / 256, 256, 0, st>>>(p, (__nv_bfloat16*)wb, m, v, g, h);
  relhost::launch_end(relhost::K_MLP, st);
  return done("launch(mlp adamw)");
}

}  // namespace rel
