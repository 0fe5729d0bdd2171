// mlp.cu - the learned launch-configuration cost model: MLP 4 -> 64 -> 64 -> 64 -> 1.
//
// No counterpart in the paper (auto-tuning is named as future work, §8).
// FP32 FFMA kernels (the network is far too small for tensor cores to pay):
//   jacc_k_mlp_fwd_bwd  one CTA per chunk of 32 samples: parameters and the
//                       chunk's activations in shared memory, forward pass,
//                       squared-error loss and backward pass; writes the
//                       chunk's gradient to its own row of `partial`.
//   jacc_k_mlp_adam     sums the chunk gradients in fixed order (deterministic)
//                       and applies one Adam step with bias correction.
//   jacc_k_mlp_forward  predictions only.
//   jacc_k_mlp_pick     per query, the argmin of the predictions over the valid
//                       tile configurations and the gap to the second best.
// Parameter layout: W1[64][4] b1[64] W2[64][64] b2[64] W3[64][64] b3[64] W4[64] b4.
//
// One training step is two dependent kernels of a few microseconds, so what
// counts is the latency of one CTA's chain of small layers.  Activations sit
// in shared memory transposed, [unit][sample], and weights in rows padded to
// 68 floats; every product is a register tile fed by 16- and 8-byte shared
// loads (4 outputs x 2 samples of a layer, 4 x 4 entries of a weight
// gradient), where one output per load of both operands kept the FMA pipes
// at 12 %.  Every sum keeps its order: over a layer's inputs, over the
// chunk's samples, over the chunks.  The Adam kernel runs on one small CTA per
// 64 parameters and has 32 chunk gradients in flight per thread.  2000
// samples: 35 -> 15.5 us a step.
#include <cuda_runtime.h>

#include "../host/jacc_internal.h"
#include "mlp.h"

namespace {

constexpr int H = 64;
constexpr int NIN = 4;
constexpr int S = 32;   // samples per CTA
constexpr int NT = 256; // 8 warps
constexpr int LW = H + 4;  // weight row pitch
constexpr int LS = S + 4;  // activation row pitch
constexpr int OFF_W1 = 0, OFF_B1 = 256, OFF_W2 = 320, OFF_B2 = 4416, OFF_W3 = 4480, OFF_B3 = 8576, OFF_W4 = 8640,
              OFF_B4 = 8704;
constexpr int NADAM = 64;  // threads per Adam CTA

struct Smem {
  float w2[H][LW], w3[H][LW];
  float w1[H][NIN], b1[H], b2[H], b3[H], w4[H], b4[4];
  float xt[NIN][LS];                       // inputs, [feature][sample]
  float h1[H][LS], h2[H][LS], h3[H][LS];   // activations after the ReLU (positive where the pre-activation is)
  float d[H][LS], d2[H][LS];               // back-propagated dz
  float y[S], dy[S];
};

__device__ __forceinline__ float relu(float z) { return z > 0.f ? z : 0.f; }
__device__ __forceinline__ void griddep_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void griddep_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

__device__ __forceinline__ void copy16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}

// Requests the parameters into shared memory (every segment of the layout
// starts on a 16-byte boundary; b4 is one float).
__device__ __forceinline__ void load_params(Smem& sm, const float* __restrict__ P) {
  for (int j = threadIdx.x; j < H * H / 4; j += NT) {
    const int o = j / (H / 4), i = 4 * (j % (H / 4));
    copy16(&sm.w2[o][i], P + OFF_W2 + 4 * j);
    copy16(&sm.w3[o][i], P + OFF_W3 + 4 * j);
  }
  const int t = threadIdx.x;
  if (t < 64) copy16(&sm.w1[0][0] + 4 * t, P + OFF_W1 + 4 * t);
  else if (t < 80) copy16(sm.b1 + 4 * (t - 64), P + OFF_B1 + 4 * (t - 64));
  else if (t < 96) copy16(sm.b2 + 4 * (t - 80), P + OFF_B2 + 4 * (t - 80));
  else if (t < 112) copy16(sm.b3 + 4 * (t - 96), P + OFF_B3 + 4 * (t - 96));
  else if (t < 128) copy16(sm.w4 + 4 * (t - 112), P + OFF_W4 + 4 * (t - 112));
  else if (t == 128) sm.b4[0] = __ldcg(P + OFF_B4);
  asm volatile("cp.async.commit_group;\n\tcp.async.wait_group 0;" ::: "memory");
}

__device__ __forceinline__ void load_inputs(Smem& sm, const float* __restrict__ X, long long s0, int nvalid) {
  if (threadIdx.x < S * NIN) {
    const int s = threadIdx.x / NIN, i = threadIdx.x % NIN;
    sm.xt[i][s] = s < nvalid ? X[(s0 + s) * NIN + i] : 0.f;
  }
}

// ho[o][s] = relu(b[o] + sum_i W[o][i] hi[i][s]): a thread's tile is outputs
// og + 16 r and samples 2 sp, 2 sp + 1.
__device__ __forceinline__ void dense64(const float (&W)[H][LW], const float* b, const float (&hi)[H][LS],
                                        float (&ho)[H][LS]) {
  const int sp = threadIdx.x & 15, og = threadIdx.x >> 4;
  float a[4][2];
#pragma unroll
  for (int r = 0; r < 4; ++r) a[r][0] = a[r][1] = b[og + 16 * r];
#pragma unroll 4
  for (int i = 0; i < H; i += 4) {
    float4 w[4];
    float2 h[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) w[r] = *reinterpret_cast<const float4*>(&W[og + 16 * r][i]);
#pragma unroll
    for (int c = 0; c < 4; ++c) h[c] = *reinterpret_cast<const float2*>(&hi[i + c][2 * sp]);
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      a[r][0] = fmaf(w[r].w, h[3].x, fmaf(w[r].z, h[2].x, fmaf(w[r].y, h[1].x, fmaf(w[r].x, h[0].x, a[r][0]))));
      a[r][1] = fmaf(w[r].w, h[3].y, fmaf(w[r].z, h[2].y, fmaf(w[r].y, h[1].y, fmaf(w[r].x, h[0].y, a[r][1]))));
    }
  }
#pragma unroll
  for (int r = 0; r < 4; ++r)
    *reinterpret_cast<float2*>(&ho[og + 16 * r][2 * sp]) = make_float2(relu(a[r][0]), relu(a[r][1]));
}

// Inputs and parameters are in shared memory; leaves h1..h3 and y.
__device__ __forceinline__ void forward_chunk(Smem& sm) {
  {  // layer 1 (4 inputs)
    const int sp = threadIdx.x & 15, og = threadIdx.x >> 4;
    float2 x[NIN];
#pragma unroll
    for (int i = 0; i < NIN; ++i) x[i] = *reinterpret_cast<const float2*>(&sm.xt[i][2 * sp]);
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const int o = og + 16 * r;
      const float4 w = *reinterpret_cast<const float4*>(&sm.w1[o][0]);
      const float a0 = fmaf(w.w, x[3].x, fmaf(w.z, x[2].x, fmaf(w.y, x[1].x, fmaf(w.x, x[0].x, sm.b1[o]))));
      const float a1 = fmaf(w.w, x[3].y, fmaf(w.z, x[2].y, fmaf(w.y, x[1].y, fmaf(w.x, x[0].y, sm.b1[o]))));
      *reinterpret_cast<float2*>(&sm.h1[o][2 * sp]) = make_float2(relu(a0), relu(a1));
    }
  }
  __syncthreads();
  dense64(sm.w2, sm.b2, sm.h1, sm.h2);
  __syncthreads();
  dense64(sm.w3, sm.b3, sm.h2, sm.h3);
  __syncthreads();
  if (threadIdx.x < S) {
    float a = sm.b4[0];
#pragma unroll 16
    for (int i = 0; i < H; ++i) a = fmaf(sm.w4[i], sm.h3[i][threadIdx.x], a);
    sm.y[threadIdx.x] = a;
  }
}

// gW[o][i] = sum_s dz[o][s] h[i][s], a 4 x 4 tile per thread (o = og + 16 r,
// i = ig + 16 c); gb[o] = sum_s dz[o][s].
__device__ __forceinline__ void weight_grad(const float (&dz)[H][LS], const float (&h)[H][LS], float* gW, float* gb) {
  const int ig = threadIdx.x & 15, og = threadIdx.x >> 4;
  float a[4][4] = {};
#pragma unroll 2
  for (int s = 0; s < S; s += 4) {
    float4 d[4], x[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) d[r] = *reinterpret_cast<const float4*>(&dz[og + 16 * r][s]);
#pragma unroll
    for (int c = 0; c < 4; ++c) x[c] = *reinterpret_cast<const float4*>(&h[ig + 16 * c][s]);
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
      for (int c = 0; c < 4; ++c)
        a[r][c] = fmaf(d[r].w, x[c].w, fmaf(d[r].z, x[c].z, fmaf(d[r].y, x[c].y, fmaf(d[r].x, x[c].x, a[r][c]))));
  }
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int c = 0; c < 4; ++c) gW[(og + 16 * r) * H + ig + 16 * c] = a[r][c];
  if (threadIdx.x < H) {
    float b = 0.f;
#pragma unroll 8
    for (int s = 0; s < S; ++s) b += dz[threadIdx.x][s];
    gb[threadIdx.x] = b;
  }
}

// dzi[i][s] = (h[i][s] > 0) * sum_o W[o][i] dzo[o][s]: inputs 4 ig .. 4 ig + 3
// and samples 2 sp, 2 sp + 1.
__device__ __forceinline__ void back64(const float (&W)[H][LW], const float (&dzo)[H][LS], const float (&h)[H][LS],
                                       float (&dzi)[H][LS]) {
  const int sp = threadIdx.x & 15, ig = threadIdx.x >> 4;
  float a[4][2] = {};
#pragma unroll 8
  for (int o = 0; o < H; ++o) {
    const float4 w = *reinterpret_cast<const float4*>(&W[o][4 * ig]);
    const float2 g = *reinterpret_cast<const float2*>(&dzo[o][2 * sp]);
    a[0][0] = fmaf(w.x, g.x, a[0][0]);
    a[0][1] = fmaf(w.x, g.y, a[0][1]);
    a[1][0] = fmaf(w.y, g.x, a[1][0]);
    a[1][1] = fmaf(w.y, g.y, a[1][1]);
    a[2][0] = fmaf(w.z, g.x, a[2][0]);
    a[2][1] = fmaf(w.z, g.y, a[2][1]);
    a[3][0] = fmaf(w.w, g.x, a[3][0]);
    a[3][1] = fmaf(w.w, g.y, a[3][1]);
  }
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const float2 z = *reinterpret_cast<const float2*>(&h[4 * ig + r][2 * sp]);
    *reinterpret_cast<float2*>(&dzi[4 * ig + r][2 * sp]) =
        make_float2(z.x > 0.f ? a[r][0] : 0.f, z.y > 0.f ? a[r][1] : 0.f);
  }
}

__global__ void __launch_bounds__(NT) jacc_k_mlp_fwd_bwd(const float* __restrict__ P, const float* __restrict__ X,
                                                         const float* __restrict__ Y, int n, float* __restrict__ partial,
                                                         float* __restrict__ loss_partial, unsigned* step) {
  extern __shared__ __align__(16) unsigned char smraw[];
  Smem& sm = *reinterpret_cast<Smem*>(smraw);
  const long long s0 = (long long)blockIdx.x * S;
  const int nvalid = (int)((n - s0) < S ? (n - s0) : S);
  griddep_wait();
  griddep_launch();
  load_inputs(sm, X, s0, nvalid);
  if (step && blockIdx.x == 0 && threadIdx.x == 0) atomicAdd(step, 1u);  // Adam step counter for this step
  load_params(sm, P);
  __syncthreads();
  forward_chunk(sm);
  // loss and dL/dy (mean over all n samples), by the warp that holds y
  if (threadIdx.x < S) {
    const int lane = threadIdx.x;
    const float e = lane < nvalid ? sm.y[lane] - Y[s0 + lane] : 0.f;
    sm.dy[lane] = 2.f * e / (float)n;
    float l = e * e;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
    if (lane == 0) loss_partial[blockIdx.x] = l;
  }
  __syncthreads();
  float* g = partial + (long long)blockIdx.x * JACC_MLP_NPARAM;
  // dz3[o][s] = dy[s] W4[o] (h3 > 0)
  for (int t = threadIdx.x; t < S * H; t += NT) {
    const int o = t / S, s = t % S;
    sm.d[o][s] = sm.h3[o][s] > 0.f ? sm.dy[s] * sm.w4[o] : 0.f;
  }
  __syncthreads();
  back64(sm.w3, sm.d, sm.h2, sm.d2);  // dz2
  weight_grad(sm.d, sm.h2, g + OFF_W3, g + OFF_B3);
  if (threadIdx.x >= NT - H) {  // layer 4
    const int i = threadIdx.x - (NT - H);
    float a = 0.f;
#pragma unroll 8
    for (int s = 0; s < S; ++s) a = fmaf(sm.dy[s], sm.h3[i][s], a);
    g[OFF_W4 + i] = a;
    if (i == 0) {
      float b = 0.f;
      for (int s = 0; s < S; ++s) b += sm.dy[s];
      g[OFF_B4] = b;
    }
  }
  __syncthreads();
  back64(sm.w2, sm.d2, sm.h1, sm.d);  // dz1 (overwrites dz3, no longer needed)
  weight_grad(sm.d2, sm.h1, g + OFF_W2, g + OFF_B2);
  __syncthreads();
  {  // layer 1: one weight per thread
    const int o = threadIdx.x / NIN, i = threadIdx.x % NIN;
    float a = 0.f;
#pragma unroll
    for (int s = 0; s < S; s += 4) {
      const float4 d = *reinterpret_cast<const float4*>(&sm.d[o][s]);
      const float4 x = *reinterpret_cast<const float4*>(&sm.xt[i][s]);
      a = fmaf(d.w, x.w, fmaf(d.z, x.z, fmaf(d.y, x.y, fmaf(d.x, x.x, a))));
    }
    g[OFF_W1 + o * NIN + i] = a;
    if (threadIdx.x < H) {
      float b = 0.f;
#pragma unroll 8
      for (int s = 0; s < S; ++s) b += sm.d[threadIdx.x][s];
      g[OFF_B1 + threadIdx.x] = b;
    }
  }
}

// Sum of v[c * stride], c = 0 .. n-1, in that order, 32 loads in flight.
__device__ __forceinline__ float ordered_sum(const float* __restrict__ v, long long stride, int n) {
  float a = 0.f;
  int c = 0;
  for (; c + 32 <= n; c += 32) {
    float t[32];
#pragma unroll
    for (int q = 0; q < 32; ++q) t[q] = v[(c + q) * stride];
#pragma unroll
    for (int q = 0; q < 32; ++q) a += t[q];
  }
  float t[31];
#pragma unroll
  for (int q = 0; q < 31; ++q) t[q] = c + q < n ? v[(c + q) * stride] : 0.f;
#pragma unroll
  for (int q = 0; q < 31; ++q)
    if (c + q < n) a += t[q];
  return a;
}

// One thread per parameter: fixed-order sum of the chunk gradients, then Adam.
__global__ void __launch_bounds__(NADAM) jacc_k_mlp_adam(float* __restrict__ P, float* __restrict__ M,
                                                         float* __restrict__ V, const float* __restrict__ partial,
                                                         int nparts, const float* __restrict__ loss_partial, int n,
                                                         float* loss_out, const unsigned* step, float lr, float b1,
                                                         float b2, float eps, float* grad_out) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  griddep_wait();
  griddep_launch();
  if (loss_out && j == 0) *loss_out = ordered_sum(loss_partial, 1, nparts) / (float)n;
  if (j >= JACC_MLP_NPARAM) return;
  const float gsum = ordered_sum(partial + j, JACC_MLP_NPARAM, nparts);
  if (grad_out) grad_out[j] = gsum;
  if (!step) return;  // gradient only
  const float t = (float)(*step);
  const float m = b1 * M[j] + (1.f - b1) * gsum;
  const float v = b2 * V[j] + (1.f - b2) * gsum * gsum;
  M[j] = m;
  V[j] = v;
  const float mh = m / (1.f - powf(b1, t));
  const float vh = v / (1.f - powf(b2, t));
  P[j] = P[j] - lr * mh / (sqrtf(vh) + eps);
}

__global__ void __launch_bounds__(NT) jacc_k_mlp_forward(const float* __restrict__ P, const float* __restrict__ X, int n,
                                                         float* __restrict__ Yout) {
  extern __shared__ __align__(16) unsigned char smraw[];
  Smem& sm = *reinterpret_cast<Smem*>(smraw);
  const long long s0 = (long long)blockIdx.x * S;
  const int nvalid = (int)((n - s0) < S ? (n - s0) : S);
  load_inputs(sm, X, s0, nvalid);
  load_params(sm, P);
  __syncthreads();
  forward_chunk(sm);
  if (threadIdx.x < nvalid) Yout[s0 + threadIdx.x] = sm.y[threadIdx.x];
}

// Queries of JACC_NUM_TILES rows each: pick[q] = argmin over valid rows (ties
// to the lowest tile id), gap[q] = second-lowest valid prediction - lowest.
__global__ void jacc_k_mlp_pick(const float* __restrict__ pred, const int* __restrict__ valid, int nq, int ntile,
                                int* pick, float* gap) {
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= nq) return;
  float best = 3.4e38f, second = 3.4e38f;
  int bi = -1;
  for (int t = 0; t < ntile; ++t) {
    if (!valid[q * ntile + t]) continue;
    const float v = pred[q * ntile + t];
    if (v < best) {
      second = best;
      best = v;
      bi = t;
    } else if (v < second) {
      second = v;
    }
  }
  pick[q] = bi;
  gap[q] = (bi >= 0 && second < 3.0e38f) ? second - best : 3.4e38f;
}

}  // namespace

namespace jacc {

size_t mlp_smem_bytes() { return sizeof(Smem); }

cudaError_t mlp_setup() {
  cudaError_t e = cudaFuncSetAttribute(jacc_k_mlp_fwd_bwd, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(Smem));
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(jacc_k_mlp_forward, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(Smem));
}

int mlp_nparts(int n) { return (n + S - 1) / S; }

// Launches that may start while the previous kernel of the stream drains
// (each waits for it before it touches memory).
template <class... A, class... B>
static cudaError_t launch_pdl(void (*f)(A...), int grid, int block, size_t smem, cudaStream_t s, B... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3((unsigned)block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, f, static_cast<A>(args)...);
}

cudaError_t mlp_fwd_bwd(const float* P, const float* X, const float* Y, int n, float* partial, float* loss_partial,
                        unsigned* step, cudaStream_t s) {
  return launch_pdl(jacc_k_mlp_fwd_bwd, mlp_nparts(n), NT, sizeof(Smem), s, P, X, Y, n, partial, loss_partial, step);
}

cudaError_t mlp_adam(float* P, float* M, float* V, const float* partial, int nparts, const float* loss_partial, int n,
                     float* loss_out, const unsigned* step, float lr, float b1, float b2, float eps, float* grad_out,
                     cudaStream_t s) {
  return launch_pdl(jacc_k_mlp_adam, (JACC_MLP_NPARAM + NADAM - 1) / NADAM, NADAM, 0, s, P, M, V, partial, nparts,
                    loss_partial, n, loss_out, step, lr, b1, b2, eps, grad_out);
}

cudaError_t mlp_forward(const float* P, const float* X, int n, float* Y, cudaStream_t s) {
  jacc_k_mlp_forward<<<mlp_nparts(n), NT, sizeof(Smem), s>>>(P, X, n, Y);
  return cudaGetLastError();
}

cudaError_t mlp_pick(const float* pred, const int* valid, int nq, int ntile, int* pick, float* gap, cudaStream_t s) {
  jacc_k_mlp_pick<<<(nq + 127) / 128, 128, 0, s>>>(pred, valid, nq, ntile, pick, gap);
  return cudaGetLastError();
}

}  // namespace jacc
