// Training kernels of the eddy-viscosity network (include/fr.h, fr_mlp_*), FP32.
//
// Network (see fr_set_closure): x^ = (x - mean)/std, three GELU layers of 64, z = w4.h3 + b4,
// prediction softplus(z).  Loss = mean over the n samples of (softplus(z) - y)^2.  Backpropagation
// is written out layer by layer: deltas da_l = (W_{l+1}^T da_{l+1}) * gelu'(a_l), weight gradients
// sum da_l (x) h_{l-1} over the samples.
#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>

#include "fr.h"

namespace {

constexpr int NIN = 11, NH = 64;
// Offsets in the flat parameter vector.
constexpr int oW1 = 0, ob1 = oW1 + NH * NIN, oW2 = ob1 + NH, ob2 = oW2 + NH * NH, oW3 = ob2 + NH, ob3 = oW3 + NH * NH,
              ow4 = ob3 + NH, ob4 = ow4 + NH, NPAR = ob4 + 1;
static_assert(NPAR == FR_CLOSURE_NPARAMS, "parameter layout");
// Workspace the caller provides per sample (include/fr.h): the partial gradients of the blocks live there.
constexpr int WS = 6 * NH + 2;

__device__ __forceinline__ float gelu(float a) { return 0.5f * a * (1.f + erff(a * 0.70710678118654752f)); }
__device__ __forceinline__ float gelu_prime(float a) {
  return 0.5f * (1.f + erff(a * 0.70710678118654752f)) + a * 0.39894228040143268f * expf(-0.5f * a * a);
}
__device__ __forceinline__ float softplus(float z) { return fmaxf(z, 0.f) + log1pf(expf(-fabsf(z))); }
__device__ __forceinline__ float sigmoid(float z) { return 1.f / (1.f + expf(-z)); }

// One block of NT threads carries a tile of TS samples through the whole network, forward and (TRAIN)
// backward, with the weights and every activation of the tile in shared memory; it leaves the tile's
// parameter gradients in its own row of the partial sums, which k_reduce adds up.  Bound by FP32 issue and the
// latency of the eight dependent small products (a training pass of 4096 samples is 0.22 GFLOP, 3 us at the
// FP32 rate, on 128 blocks).  GB300, 4096 samples, loss and gradient: 2.07 ms with one kernel per layer
// and a thread per weight that read all samples in a chain; with this kernel and its reduction a loss,
// gradient and optimiser step together take 37 us.
// Tile: 32 samples fill 128 SMs at the pipeline's batch of 4096 (the one size it was measured at), and leave each block's partial row
// (NPAR + 1 floats) within the workspace of its own samples (32 WS).  Each thread owns 4 samples x 4
// neurons (stride 16), so four k-steps take 8 16-byte shared loads for 64 FMAs; rows are LD = 68 floats
// apart, so the 16 neuron rows a half-warp reads lie in different banks.
constexpr int TS = 32, NT = 128, LD = NH + 4;
constexpr int kPart = NPAR + 1;               // gradients, then the loss
constexpr int kMaxBlocks = 304;               // two per SM; further tiles are looped over

struct TileSmem {
  float W2[NH * LD], W3[NH * LD], W1[NH * 12], b1[NH], b2[NH], b3[NH], w4[NH], sc[2 * NIN], b4, pad;
  float x[TS * 12];
  float a[3][TS * LD], h[3][TS * LD];         // pre-activations (then deltas) and activations
  float dz[TS], r2[TS];
};

// out[s][j] = bias[j] + sum_k W[j][k] in[s][k], then its activation; 64 x 64 weights.
__device__ __forceinline__ void dense(const float *W, const float *bias, const float *in, float *a, float *h, int tj,
                                      int s0) {
  float acc[4][4];
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int q = 0; q < 4; ++q) acc[r][q] = bias[tj + 16 * r];
#pragma unroll 4
  for (int k = 0; k < NH; k += 4) {
    float4 w[4], x[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) w[r] = *reinterpret_cast<const float4 *>(W + (tj + 16 * r) * LD + k);
#pragma unroll
    for (int q = 0; q < 4; ++q) x[q] = *reinterpret_cast<const float4 *>(in + (s0 + q) * LD + k);
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
      for (int q = 0; q < 4; ++q)
        acc[r][q] = fmaf(w[r].w, x[q].w, fmaf(w[r].z, x[q].z, fmaf(w[r].y, x[q].y, fmaf(w[r].x, x[q].x, acc[r][q]))));
  }
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int o = (s0 + q) * LD + tj + 16 * r;
      a[o] = acc[r][q];
      h[o] = gelu(acc[r][q]);
    }
}

// Delta of a layer from the next one's, d[s][k] = gelu'(a[s][k]) sum_j W[j][k] dn[s][j], over a; this
// thread: 4 samples x 4 neighbouring neurons k0.
__device__ __forceinline__ void delta(const float *W, const float *dn, float *a, int k0, int s0) {
  float acc[4][4] = {};
#pragma unroll 2
  for (int j = 0; j < NH; j += 4) {
    float4 w[4], d[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) w[r] = *reinterpret_cast<const float4 *>(W + (j + r) * LD + k0);
#pragma unroll
    for (int q = 0; q < 4; ++q) d[q] = *reinterpret_cast<const float4 *>(dn + (s0 + q) * LD + j);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const float dq[4] = {d[q].x, d[q].y, d[q].z, d[q].w};
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        acc[q][0] = fmaf(w[r].x, dq[r], acc[q][0]);
        acc[q][1] = fmaf(w[r].y, dq[r], acc[q][1]);
        acc[q][2] = fmaf(w[r].z, dq[r], acc[q][2]);
        acc[q][3] = fmaf(w[r].w, dq[r], acc[q][3]);
      }
    }
  }
#pragma unroll
  for (int q = 0; q < 4; ++q)
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      float *p = a + (s0 + q) * LD + k0 + c;
      *p = acc[q][c] * gelu_prime(*p);
    }
}

// Sum over the tile's samples of d[s][j] h[s][k]: this thread the neurons j = tj + 16 r and eight k.
__device__ __forceinline__ void weight_grad(const float *d, const float *h, float *g, int tj, int k0, bool first) {
  float acc[4][8] = {};
#pragma unroll 4
  for (int s = 0; s < TS; ++s) {
    const float4 u = *reinterpret_cast<const float4 *>(h + s * LD + k0);
    const float4 v = *reinterpret_cast<const float4 *>(h + s * LD + k0 + 4);
    const float hv[8] = {u.x, u.y, u.z, u.w, v.x, v.y, v.z, v.w};
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const float dv = d[s * LD + tj + 16 * r];
#pragma unroll
      for (int c = 0; c < 8; ++c) acc[r][c] = fmaf(dv, hv[c], acc[r][c]);
    }
  }
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      float *p = g + (tj + 16 * r) * NH + k0 + c;
      *p = first ? acc[r][c] : *p + acc[r][c];
    }
}

template <bool TRAIN>
__global__ void __launch_bounds__(NT) k_tile(const float *__restrict__ P, const float *__restrict__ X,
                                             const float *__restrict__ sc, const float *__restrict__ y, int64_t n,
                                             float *__restrict__ pred, float *__restrict__ grad, float *__restrict__ loss,
                                             float *__restrict__ part) {
  extern __shared__ float4 smem4[];
  TileSmem &S = *reinterpret_cast<TileSmem *>(smem4);
  const int tid = threadIdx.x, tj = tid & 15, s0 = (tid >> 4) * 4;
  for (int i = tid; i < NH * NH; i += NT) {
    S.W2[(i >> 6) * LD + (i & 63)] = P[oW2 + i];
    S.W3[(i >> 6) * LD + (i & 63)] = P[oW3 + i];
  }
  for (int i = tid; i < NH * NIN; i += NT) S.W1[i / NIN * 12 + i % NIN] = P[oW1 + i];
  if (tid < NH) {
    S.b1[tid] = P[ob1 + tid];
    S.b2[tid] = P[ob2 + tid];
    S.b3[tid] = P[ob3 + tid];
    S.w4[tid] = P[ow4 + tid];
  }
  if (tid < 2 * NIN) S.sc[tid] = sc[tid];
  if (tid == 0) S.b4 = P[ob4];
  // One block alone writes the results themselves, several their partial rows.
  float *g = gridDim.x == 1 ? grad : part + (int64_t)blockIdx.x * kPart;
  float *gl = gridDim.x == 1 ? loss : g + NPAR;
  const int64_t tiles = (n + TS - 1) / TS;
  bool first = true;
  for (int64_t tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
    const int64_t base = tile * TS;
    const int cnt = (int)(n - base < TS ? n - base : TS);
    __syncthreads();
    for (int i = tid; i < TS * NIN; i += NT) {
      const int s = i / NIN, k = i % NIN;
      S.x[s * 12 + k] = s < cnt ? (X[(base + s) * NIN + k] - S.sc[k]) / S.sc[NIN + k] : 0.f;
    }
    __syncthreads();
    {
      float acc[4][4];
#pragma unroll
      for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[r][q] = S.b1[tj + 16 * r];
#pragma unroll
      for (int k = 0; k < NIN; ++k)
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          const float w = S.W1[(tj + 16 * r) * 12 + k];
#pragma unroll
          for (int q = 0; q < 4; ++q) acc[r][q] = fmaf(w, S.x[(s0 + q) * 12 + k], acc[r][q]);
        }
#pragma unroll
      for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int o = (s0 + q) * LD + tj + 16 * r;
          S.a[0][o] = acc[r][q];
          S.h[0][o] = gelu(acc[r][q]);
        }
    }
    __syncthreads();
    dense(S.W2, S.b2, S.h[0], S.a[1], S.h[1], tj, s0);
    __syncthreads();
    dense(S.W3, S.b3, S.h[1], S.a[2], S.h[2], tj, s0);
    __syncthreads();
    {
      // Output: four threads per sample.
      const int s = tid >> 2, c = tid & 3;
      float z = 0.f;
#pragma unroll
      for (int k = 0; k < NH / 4; ++k) z = fmaf(S.w4[c + 4 * k], S.h[2][s * LD + c + 4 * k], z);
      z += __shfl_xor_sync(0xffffffffu, z, 1);
      z += __shfl_xor_sync(0xffffffffu, z, 2);
      z += S.b4;
      if (c == 0) {
        const float sp = softplus(z);
        if (!TRAIN) {
          if (s < cnt) pred[base + s] = sp;
        } else {
          const float r = s < cnt ? sp - y[base + s] : 0.f;
          S.dz[s] = 2.f * r * sigmoid(z) / (float)n;
          S.r2[s] = r * r / (float)n;
        }
      }
    }
    if constexpr (TRAIN) {
      __syncthreads();
      const int k0 = tj * 4;
#pragma unroll
      for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          float *p = S.a[2] + (s0 + q) * LD + k0 + c;
          *p = S.dz[s0 + q] * S.w4[k0 + c] * gelu_prime(*p);
        }
      __syncthreads();
      delta(S.W3, S.a[2], S.a[1], k0, s0);
      __syncthreads();
      delta(S.W2, S.a[1], S.a[0], k0, s0);
      __syncthreads();
      weight_grad(S.a[2], S.h[1], g + oW3, tj, s0 * 2, first);
      weight_grad(S.a[1], S.h[0], g + oW2, tj, s0 * 2, first);
      for (int i = tid; i < NH * NIN; i += NT) {
        const int j = i / NIN, k = i % NIN;
        float v = 0.f;
#pragma unroll 8
        for (int s = 0; s < TS; ++s) v = fmaf(S.a[0][s * LD + j], S.x[s * 12 + k], v);
        g[oW1 + i] = first ? v : g[oW1 + i] + v;
      }
      // Biases, the output layer and the loss.
      const float *src[4] = {S.a[0], S.a[1], S.a[2], S.h[2]};
      const int off[4] = {ob1, ob2, ob3, ow4};
      for (int i = tid; i < 4 * NH; i += NT) {
        const int l = i >> 6, j = i & 63;
        float v = 0.f;
#pragma unroll 8
        for (int s = 0; s < TS; ++s) v += l == 3 ? S.dz[s] * src[3][s * LD + j] : src[l][s * LD + j];
        float *p = g + off[l] + j;
        *p = first ? v : *p + v;
      }
      if (tid < 2) {
        float v = 0.f;
        for (int s = 0; s < TS; ++s) v += tid ? S.r2[s] : S.dz[s];
        float *p = tid ? gl : g + ob4;
        *p = first ? v : *p + v;
      }
      first = false;
    }
  }
}

// grad and loss = sum of the blocks' partial rows: 32 parameters x 8 row groups per block.
__global__ void __launch_bounds__(256) k_reduce(const float *__restrict__ part, int rows, float *__restrict__ grad,
                                                float *__restrict__ loss) {
  __shared__ float s[8][33];
  const int c = threadIdx.x & 31, r0 = threadIdx.x >> 5, i = blockIdx.x * 32 + c;
  float v = 0.f;
  if (i < kPart)
#pragma unroll 8
    for (int r = r0; r < rows; r += 8) v += part[(int64_t)r * kPart + i];
  s[r0][c] = v;
  __syncthreads();
  if (r0 == 0 && i < kPart) {
#pragma unroll
    for (int r = 1; r < 8; ++r) v += s[r][c];
    if (i < NPAR)
      grad[i] = v;
    else
      *loss = v;
  }
}

__global__ void k_adam(float *__restrict__ P, const float *__restrict__ g, float *__restrict__ m, float *__restrict__ v,
                       int n, float lr, float b1, float b2, float eps, float c1, float c2) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const float mi = b1 * m[i] + (1.f - b1) * g[i];
  const float vi = b2 * v[i] + (1.f - b2) * g[i] * g[i];
  m[i] = mi;
  v[i] = vi;
  P[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
}

// Blocks of a pass: one per tile, at most kMaxBlocks, and in training no more partial rows than the
// caller's workspace holds.
template <bool TRAIN>
fr_status launch_tile(const float *P, const float *X, const float *sc, const float *y, int64_t n, float *pred,
                      float *grad, float *loss, float *work, cudaStream_t st) {
  if (cudaFuncSetAttribute(k_tile<TRAIN>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(TileSmem)) !=
      cudaSuccess)
    return FR_ECUDA;
  int64_t blocks = (n + TS - 1) / TS;
  if (blocks > kMaxBlocks) blocks = kMaxBlocks;
  if (TRAIN) {
    const int64_t rows = (n * WS + 1) / kPart;
    if (blocks > rows) blocks = rows > 0 ? rows : 1;
  }
  k_tile<TRAIN><<<(unsigned)blocks, NT, sizeof(TileSmem), st>>>(P, X, sc, y, n, pred, grad, loss, work);
  if (TRAIN && blocks > 1) k_reduce<<<(kPart + 31) / 32, 256, 0, st>>>(work, (int)blocks, grad, loss);
  return cudaGetLastError() == cudaSuccess ? FR_OK : FR_ECUDA;
}

}  // namespace

extern "C" int64_t fr_mlp_workspace_floats(int64_t n) { return n * WS + 1; }

extern "C" fr_status fr_mlp_forward(const float *params, const float *scales, const float *X, int64_t n, float *out,
                                    float *work, uintptr_t stream) {
  if (!params || !scales || !X || !out || !work || n < 1) return FR_EINVAL;
  return launch_tile<false>(params, X, scales, nullptr, n, out, nullptr, nullptr, work, (cudaStream_t)stream);
}

extern "C" fr_status fr_mlp_loss_grad(const float *params, const float *scales, const float *X, const float *y,
                                      int64_t n, float *grad, float *loss, float *work, uintptr_t stream) {
  if (!params || !scales || !X || !y || !grad || !loss || !work || n < 1) return FR_EINVAL;
  return launch_tile<true>(params, X, scales, y, n, nullptr, grad, loss, work, (cudaStream_t)stream);
}

extern "C" fr_status fr_mlp_adam(float *params, const float *grad, float *m, float *v, int32_t n_params, float lr,
                                 float beta1, float beta2, float eps, int32_t step, uintptr_t stream) {
  if (!params || !grad || !m || !v || n_params < 1 || step < 1) return FR_EINVAL;
  const float c1 = 1.f - powf(beta1, (float)step), c2 = 1.f - powf(beta2, (float)step);
  k_adam<<<(n_params + 255) / 256, 256, 0, (cudaStream_t)stream>>>(params, grad, m, v, n_params, lr, beta1, beta2, eps,
                                                                    c1, c2);
  return cudaGetLastError() == cudaSuccess ? FR_OK : FR_ECUDA;
}
