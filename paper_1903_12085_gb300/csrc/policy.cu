// policy.cu -- storage of the per-phase policy network and its FP32 training
// kernels (forward, backward, Adam).  The network and its features are defined
// in policy.cuh.
//
// Training objective (masked mean squared error): for sample b, taken in a
// phase that ran with arm a_b and cost t_b (log2 of the phase time per settled
// vertex), loss = (1/B) sum_b (y_b[a_b] - t_b)^2 where y_b is the network output.
//
// Backward pass in two kernels:
//   k_mlp_grad         a warp takes samples, two at a time, lane j as hidden
//                      unit j of both layers, with its weights and its share of
//                      the gradient in registers; each block adds its warps'
//                      gradients up and writes one partial gradient;
//   k_mlp_grad_reduce  sums the blocks' partial gradients.
// Both in a fixed order for a given batch size and GPU, so gradients are
// deterministic.
#include <mutex>

#include "internal.h"
#include "policy.cuh"

namespace sssp {
namespace {

constexpr int kMaxDevices = 64;
float* g_policy[kMaxDevices] = {nullptr};
std::mutex g_policy_mu;

__global__ void k_mlp_forward(const float* __restrict__ w, const float* __restrict__ x, uint32_t batch,
                              float* __restrict__ y) {
  __shared__ float sw[kPolWeights];
  for (int i = threadIdx.x; i < kPolWeights; i += blockDim.x) sw[i] = w[i];
  __syncthreads();
  // (64 bits: near 2^32 samples a 32-bit counter would wrap and never end)
  for (uint64_t b = blockIdx.x * blockDim.x + threadIdx.x; b < batch; b += gridDim.x * blockDim.x) {
    float h1[kPolHidden], h2[kPolHidden];
    for (int j = 0; j < kPolHidden; ++j) {
      float z = sw[kPolOffB1 + j];
      for (int i = 0; i < kPolFeat; ++i) z = fmaf(x[(size_t)b * kPolFeat + i], sw[kPolOffW1 + i * kPolHidden + j], z);
      h1[j] = fmaxf(z, 0.0f);
    }
    for (int j = 0; j < kPolHidden; ++j) {
      float z = sw[kPolOffB2 + j];
      for (int i = 0; i < kPolHidden; ++i) z = fmaf(h1[i], sw[kPolOffW2 + i * kPolHidden + j], z);
      h2[j] = fmaxf(z, 0.0f);
    }
    for (int a = 0; a < kPolArms; ++a) {
      float z = sw[kPolOffB3 + a];
      for (int i = 0; i < kPolHidden; ++i) z = fmaf(h2[i], sw[kPolOffW3 + i * kPolArms + a], z);
      y[(size_t)b * kPolArms + a] = z;
    }
  }
}

// Gradient row of a block: the kPolWeights weight gradients, then the loss.
constexpr int kGradRow = kPolWeights + 1;
constexpr int kGradWarps = 8;
constexpr int kGradTile = 8;  // samples a warp takes at a time
__host__ __device__ constexpr uint32_t grad_tiles(uint32_t batch) { return batch / kGradTile + (batch % kGradTile != 0); }
static_assert(grad_tiles(~0u) == 1u << 29 && grad_tiles(9) == 2 && grad_tiles(8) == 1, "no wrap-around");

// Gradient of the batch, one partial gradient per block.  Bound by the FP32
// pipes and the latency of a sample's chain (about 115 multiply-adds a lane and
// 24 broadcast loads of shared memory): 60,000 samples are 0.44 GFLOP, 6 us of
// the GPU's multiply-adds, and nothing of a sample leaves the SM.  (One thread
// a sample with its activations in local memory and 532 bytes of scratch per
// sample, reduced by 76 blocks striding over them, took 500 us on 60,000 samples: a
// training step 577 us, with this 55.)
__global__ void __launch_bounds__(32 * kGradWarps, 1)
k_mlp_grad(const float* __restrict__ w, const float* __restrict__ x, const float* __restrict__ target,
           const uint32_t* __restrict__ arm, uint32_t batch, float* __restrict__ partial) {
  __shared__ __align__(16) float s_x[kGradWarps][kGradTile][kPolFeat];
  __shared__ __align__(16) float s_h[kGradWarps][2][kPolHidden], s_g[kGradWarps][2][kPolHidden];
  __shared__ float s_grad[kGradWarps / 2][kGradRow];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const float inv_b = 1.0f / (float)batch;
  float w1[kPolFeat], w2c[kPolHidden], w2r[kPolHidden], w3[kPolArms], b3[kPolArms];
#pragma unroll
  for (int i = 0; i < kPolFeat; ++i) w1[i] = w[kPolOffW1 + i * kPolHidden + lane];
#pragma unroll
  for (int i = 0; i < kPolHidden; ++i) {
    w2c[i] = w[kPolOffW2 + i * kPolHidden + lane];
    w2r[i] = w[kPolOffW2 + lane * kPolHidden + i];
  }
#pragma unroll
  for (int a = 0; a < kPolArms; ++a) {
    w3[a] = w[kPolOffW3 + lane * kPolArms + a];
    b3[a] = w[kPolOffB3 + a];
  }
  const float b1 = w[kPolOffB1 + lane], b2 = w[kPolOffB2 + lane];
  float g1[kPolFeat] = {}, g2[kPolHidden] = {}, g3[kPolArms] = {}, gb1 = 0.0f, gb2 = 0.0f, gb3 = 0.0f, se = 0.0f;
  // tiles of consecutive samples, dealt to the blocks in turn (a small batch
  // spreads over the SMs)
  const uint32_t tiles = grad_tiles(batch);
  for (uint32_t tile = warp * gridDim.x + blockIdx.x; tile < tiles; tile += gridDim.x * kGradWarps) {
    const uint32_t s0 = tile * kGradTile;
    const int n = (int)min(batch - s0, (uint32_t)kGradTile);
    __syncwarp();
#pragma unroll
    for (int q = 0; q < kGradTile * kPolFeat / 32; ++q) {
      const int e = q * 32 + lane;
      (&s_x[warp][0][0])[e] = e < n * kPolFeat ? x[(size_t)s0 * kPolFeat + e] : 0.0f;
    }
    float my_t = 0.0f;
    uint32_t my_a = 0;
    if (lane < n) {
      my_t = target[s0 + lane];
      my_a = arm[s0 + lane];
      my_a = my_a < (uint32_t)kPolArms ? my_a : 0u;
    }
    __syncwarp();
    for (int s = 0; s < n; s += 2) {  // (an odd last sample's twin counts for nothing: its activations and error are zero)
      float h1[2], h2[2], g[2];
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        float z = b1;
#pragma unroll
        for (int i = 0; i < kPolFeat; ++i) z = fmaf(s_x[warp][s + u][i], w1[i], z);
        h1[u] = s + u < n ? fmaxf(z, 0.0f) : 0.0f;
        s_h[warp][u][lane] = h1[u];
      }
      __syncwarp();
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        float z = b2;
#pragma unroll
        for (int i = 0; i < kPolHidden; ++i) z = fmaf(s_h[warp][u][i], w2c[i], z);
        h2[u] = s + u < n ? fmaxf(z, 0.0f) : 0.0f;
      }
      float ya[2];
      uint32_t a[2];
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        a[u] = __shfl_sync(0xFFFFFFFFu, my_a, s + u);
        const float w3a = a[u] == 0 ? w3[0] : a[u] == 1 ? w3[1] : a[u] == 2 ? w3[2] : w3[3];
        ya[u] = h2[u] * w3a;
        g[u] = w3a;
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
        for (int u = 0; u < 2; ++u) ya[u] += __shfl_xor_sync(0xFFFFFFFFu, ya[u], o);
      }
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const float b3a = a[u] == 0 ? b3[0] : a[u] == 1 ? b3[1] : a[u] == 2 ? b3[2] : b3[3];
        const float err = s + u < n ? ya[u] + b3a - __shfl_sync(0xFFFFFFFFu, my_t, s + u) : 0.0f;
        const float dya = 2.0f * err * inv_b;  // d loss / d y_b[a]
        se = fmaf(err * inv_b, err, se);
        const float dz2 = h2[u] > 0.0f ? g[u] * dya : 0.0f;
        g[u] = dz2;
        s_g[warp][u][lane] = dz2;
        gb2 += dz2;
#pragma unroll
        for (int k = 0; k < kPolArms; ++k) g3[k] = fmaf(h2[u], a[u] == (uint32_t)k ? dya : 0.0f, g3[k]);
        if ((uint32_t)lane == a[u]) gb3 += dya;  // (lane k: output k)
      }
      __syncwarp();
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        float d = 0.0f;
#pragma unroll
        for (int i = 0; i < kPolHidden; ++i) {
          d = fmaf(w2r[i], s_g[warp][u][i], d);
          g2[i] = fmaf(s_h[warp][u][i], g[u], g2[i]);
        }
        const float dz1 = h1[u] > 0.0f ? d : 0.0f;
        gb1 += dz1;
#pragma unroll
        for (int i = 0; i < kPolFeat; ++i) g1[i] = fmaf(s_x[warp][s + u][i], dz1, g1[i]);
      }
      __syncwarp();
    }
  }
  // the upper half of the warps leave their shares, the lower half add theirs
  for (int half = 1; half >= 0; --half) {
    if ((warp >= kGradWarps / 2) == (half == 1)) {
      float* row = s_grad[warp % (kGradWarps / 2)];
      auto put = [&](int c, float v) { row[c] = half ? v : row[c] + v; };
#pragma unroll
      for (int i = 0; i < kPolFeat; ++i) put(kPolOffW1 + i * kPolHidden + lane, g1[i]);
      put(kPolOffB1 + lane, gb1);
#pragma unroll
      for (int i = 0; i < kPolHidden; ++i) put(kPolOffW2 + i * kPolHidden + lane, g2[i]);
      put(kPolOffB2 + lane, gb2);
#pragma unroll
      for (int k = 0; k < kPolArms; ++k) put(kPolOffW3 + lane * kPolArms + k, g3[k]);
      if (lane < kPolArms) put(kPolOffB3 + lane, gb3);
      if (lane == 0) put(kPolWeights, se);
    }
    __syncthreads();
  }
  for (int c = threadIdx.x; c < kGradRow; c += 32 * kGradWarps) {
    float v = 0.0f;
#pragma unroll
    for (int q = 0; q < kGradWarps / 2; ++q) v += s_grad[q][c];
    partial[(size_t)blockIdx.x * kGradRow + c] = v;
  }
}

// Sums `rows` partial gradients: 32 columns a block, eight threads a column, in
// 64 bits (19 additions a thread), so that the sum's own error does not count.
__global__ void __launch_bounds__(256) k_mlp_grad_reduce(const float* __restrict__ partial, int rows,
                                                         float* __restrict__ grad, float* __restrict__ loss) {
  __shared__ double s[8][32];
  const int cx = threadIdx.x & 31, ry = threadIdx.x >> 5, c = blockIdx.x * 32 + cx;
  double v = 0.0;
  if (c < kGradRow) {
#pragma unroll 4
    for (int r = ry; r < rows; r += 8) v += partial[(size_t)r * kGradRow + c];
  }
  s[ry][cx] = v;
  __syncthreads();
  if (ry == 0 && c < kGradRow) {
#pragma unroll
    for (int q = 1; q < 8; ++q) v += s[q][cx];
    if (c < kPolWeights) grad[c] = (float)v;
    else if (loss) *loss = (float)v;
  }
}

__global__ void k_adam(float* __restrict__ w, const float* __restrict__ g, float* __restrict__ m1,
                       float* __restrict__ m2, uint32_t count, float lr, float beta1, float beta2, float eps,
                       float c1, float c2) {
  for (uint64_t i = blockIdx.x * blockDim.x + threadIdx.x; i < count; i += gridDim.x * blockDim.x) {
    const float gi = g[i];
    const float a = beta1 * m1[i] + (1.0f - beta1) * gi;
    const float b = beta2 * m2[i] + (1.0f - beta2) * gi * gi;
    m1[i] = a;
    m2[i] = b;
    w[i] -= lr * (a / c1) / (sqrtf(b / c2) + eps);
  }
}

}  // namespace

// Device pointer of the policy loaded on the current device (nullptr if none).
const float* policy_weights() {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return nullptr;
  std::lock_guard<std::mutex> lock(g_policy_mu);
  return g_policy[dev];
}

}  // namespace sssp

using namespace sssp;

extern "C" sssp_status sssp_policy_load(const float* weights, size_t count) {
  clear_error();
  if (!weights || count != (size_t)kPolWeights)
    return fail(SSSP_ERR_INVALID_ARG, "policy needs %d weights (got %zu)", kPolWeights, count);
  int dev = 0;
  SSSP_CUDA_TRY(cudaGetDevice(&dev));
  if (dev < 0 || dev >= kMaxDevices) return fail(SSSP_ERR_UNSUPPORTED, "device ordinal out of range");
  std::lock_guard<std::mutex> lock(g_policy_mu);
  if (!g_policy[dev]) {
    sssp_status s = dev_alloc(&g_policy[dev], kPolWeights);
    if (s != SSSP_OK) return s;
  }
  SSSP_CUDA_TRY(cudaMemcpy(g_policy[dev], weights, kPolWeights * sizeof(float),
                           is_device_pointer(weights) ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice));
  return SSSP_OK;
}

extern "C" sssp_status sssp_policy_clear(void) {
  int dev = 0;
  SSSP_CUDA_TRY(cudaGetDevice(&dev));
  std::lock_guard<std::mutex> lock(g_policy_mu);
  if (dev >= 0 && dev < kMaxDevices && g_policy[dev]) {
    dev_free(g_policy[dev]);
    g_policy[dev] = nullptr;
  }
  return SSSP_OK;
}

extern "C" sssp_status sssp_policy_features(uint64_t frontier, uint64_t n, uint64_t m, uint64_t phase,
                                            uint64_t edges_prev, uint64_t settled_prev, uint64_t frontier_prev,
                                            float* out8) {
  if (!out8 || n == 0) return fail(SSSP_ERR_INVALID_ARG, "bad feature arguments");
  policy_features(out8, frontier, n, m, phase, edges_prev, settled_prev, frontier_prev);
  return SSSP_OK;
}

extern "C" sssp_status sssp_mlp_forward(const float* w, const float* x, uint32_t batch, float* y, void* stream) {
  clear_error();
  if (!w || !x || !y) return fail(SSSP_ERR_INVALID_ARG, "NULL argument");
  if (batch == 0) return SSSP_OK;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const int blocks = (int)std::min<uint64_t>(((uint64_t)batch + 127) / 128, 1024);
  k_mlp_forward<<<blocks, 128, 0, st>>>(w, x, batch, y);
  SSSP_CUDA_TRY(cudaGetLastError());
  return SSSP_OK;
}

extern "C" sssp_status sssp_mlp_backward(const float* w, const float* x, const float* target, const uint32_t* arm,
                                         uint32_t batch, float* grad, float* loss, void* stream) {
  clear_error();
  if (!w || !x || !target || !arm || !grad || batch == 0) return fail(SSSP_ERR_INVALID_ARG, "NULL or empty argument");
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  // one block per SM, and no more than the samples fill
  const int blocks = (int)std::min<uint32_t>(grad_tiles(batch), (uint32_t)sm_count());
  TmpBuf<float> sbuf(st);
  sssp_status s = sbuf.alloc((size_t)blocks * kGradRow);
  if (s != SSSP_OK) return s;
  k_mlp_grad<<<blocks, 32 * kGradWarps, 0, st>>>(w, x, target, arm, batch, sbuf.p);
  k_mlp_grad_reduce<<<(kGradRow + 31) / 32, 256, 0, st>>>(sbuf.p, blocks, grad, loss);
  SSSP_CUDA_TRY(cudaGetLastError());
  return SSSP_OK;
}

extern "C" sssp_status sssp_mlp_adam(float* w, const float* grad, float* m1, float* m2, uint32_t count, float lr,
                                     float beta1, float beta2, float eps, uint32_t step, void* stream) {
  clear_error();
  if (!w || !grad || !m1 || !m2 || step == 0) return fail(SSSP_ERR_INVALID_ARG, "bad Adam arguments");
  const float c1 = 1.0f - powf(beta1, (float)step), c2 = 1.0f - powf(beta2, (float)step);
  k_adam<<<(int)std::min<uint64_t>(((uint64_t)count + 255) / 256, 1024), 256, 0, static_cast<cudaStream_t>(stream)>>>(
      w, grad, m1, m2, count, lr, beta1, beta2, eps, c1, c2);
  SSSP_CUDA_TRY(cudaGetLastError());
  return SSSP_OK;
}
