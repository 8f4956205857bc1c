// policy.cuh -- the per-phase policy network (device side, shared by the engine
// and the training kernels).
//
// A small MLP picks, at the start of every phase, which fused-threshold arm
// the phase runs with:
//   arm 0: IN-STATIC  | OUT-STATIC, sparse fringe queue
//   arm 1: IN-STATIC  | OUT-STATIC, dense scan of the status array
//   arm 2: IN-SIMPLE  | OUT-STATIC, sparse
//   arm 3: IN-SIMPLE  | OUT-STATIC, dense
// Every arm is a disjunction of sound criteria with a complete disjunct, so the
// choice never changes a distance (Section 3); it changes how many vertices a
// phase settles and what the phase costs.  The network maps 8 features of the
// phase-start state to 4 outputs, the predicted log2 of the phase time per
// settled vertex for each arm; the phase takes the arm with the smallest
// prediction if it beats arm 0 by a margin, else arm 0, the paper's IN+OUT
// (IN-SIMPLE arms only when the in-edge CSR exists; a non-finite prediction
// falls back to arm 0; while the engine keeps the fringe split into near and
// far parts, every phase takes arm 0 without asking the network).
//
// Features (float32, all cheap and identical in every block):
//   f0 = log2(1 + |F|) / 24          f4 = log2(1 + k) / 16     (k = phase index)
//   f1 = |F| / n                      f5 = log2(n) / 32
//   f2 = log2(1 + E_prev) / 24        f6 = (m / n) / 32
//   f3 = log2(1 + S_prev) / 24        f7 = S_prev / (1 + F_prev)
// where E_prev, S_prev, F_prev are the relaxed edges, settled vertices and
// fringe size of phase k-1 (0 for k = 1).
// Weights: one float array, W1[8][32], b1[32], W2[32][32], b2[32], W3[32][4],
// b3[4] (row-major, input index first), ReLU after the two hidden layers.
#pragma once

#include <cstdint>

namespace sssp {

constexpr int kPolFeat = 8;
constexpr int kPolHidden = 32;
constexpr int kPolArms = 4;
constexpr int kPolOffW1 = 0;
constexpr int kPolOffB1 = kPolOffW1 + kPolFeat * kPolHidden;
constexpr int kPolOffW2 = kPolOffB1 + kPolHidden;
constexpr int kPolOffB2 = kPolOffW2 + kPolHidden * kPolHidden;
constexpr int kPolOffW3 = kPolOffB2 + kPolHidden;
constexpr int kPolOffB3 = kPolOffW3 + kPolHidden * kPolArms;
constexpr int kPolWeights = kPolOffB3 + kPolArms;  // 1476

// Feature i from the counts above, as float32: the one formula, for the host
// (policy_features) and for the engine's warps (policy_feature_lane), which have
// one logarithm and one division in a row this way instead of five and eight.
// (A scale by a power of two is exact, before or after.)
__host__ __device__ __forceinline__ float policy_feature(int i, float nF, float n, float m, float k, float e_prev,
                                                         float s_prev, float f_prev) {
  const float x = i == 0 || i == 1 ? nF : i == 2 ? e_prev : i == 4 ? k : i == 5 ? n : i == 6 ? m : s_prev;
  const float num = i < 6 && i != 1 ? log2f(i == 5 ? x : 1.0f + x) : x;
  const float den = i == 1 || i == 6 ? n : i == 7 ? 1.0f + f_prev : i == 4 || i == 5 ? 1.0f : 24.0f;
  const float scale = i == 4 ? 1.0f / 16.0f : i == 5 || i == 6 ? 1.0f / 32.0f : 1.0f;
  return num / den * scale;
}

__host__ __device__ __forceinline__ void policy_features(float* f, uint64_t nF, uint64_t n, uint64_t m, uint64_t k,
                                                         uint64_t e_prev, uint64_t s_prev, uint64_t f_prev) {
  for (int i = 0; i < kPolFeat; ++i)
    f[i] = policy_feature(i, (float)nF, (float)n, (float)m, (float)k, (float)e_prev, (float)s_prev, (float)f_prev);
}

// The same by one full warp, feature i in lane i (i < 8; other lanes: 0).
__device__ __forceinline__ float policy_feature_lane(uint32_t nF, uint32_t n, uint32_t m, uint32_t k,
                                                     uint32_t e_prev, uint32_t s_prev, uint32_t f_prev) {
  const int i = threadIdx.x & 31;
  const float f =
      policy_feature(i, (float)nF, (float)n, (float)m, (float)k, (float)e_prev, (float)s_prev, (float)f_prev);
  return i < kPolFeat ? f : 0.0f;
}

// Place of weight i in a block's shared-memory copy: the matrices of the hidden
// layers four rows at a time, so that a lane reads its column as float4s (a
// forward pass runs with cold instruction caches, and costs what its length does).
__device__ __forceinline__ int policy_place(int i) {
  const int base = i < kPolOffB1 ? kPolOffW1 : kPolOffW2;
  if ((i >= kPolOffB1 && i < kPolOffW2) || i >= kPolOffB2) return i;
  const int r = (i - base) / kPolHidden, c = (i - base) % kPolHidden;
  return base + (r / 4 * kPolHidden + c) * 4 + r % 4;
}

// sum += in[0..4K) * (the lane's column of a matrix placed as above), in order.
template <int K>
__device__ __forceinline__ float policy_column(const float* in, const float* w, float sum) {
  const float4* const x4 = reinterpret_cast<const float4*>(in);
  const float4* const w4 = reinterpret_cast<const float4*>(w) + (threadIdx.x & 31);
#pragma unroll
  for (int q = 0; q < K; ++q) {
    const float4 x = x4[q], c = w4[q * kPolHidden];
    sum = fmaf(x.x, c.x, sum);
    sum = fmaf(x.y, c.y, sum);
    sum = fmaf(x.z, c.z, sum);
    sum = fmaf(x.w, c.w, sum);
  }
  return sum;
}

// Forward pass by one full warp: lane j owns hidden unit j of both layers, and
// lane i < 8 holds feature i in `f`.  Returns the 4 outputs in out[], in every
// lane.  `w`: the weights in shared memory (policy_place); `act`: 64 floats of
// shared memory, 16-byte aligned like w.
__device__ __forceinline__ void policy_forward_warp(const float* w, float f, float* act, float* out) {
  const int lane = threadIdx.x & 31;
  act[lane] = f;
  __syncwarp();
  const float h1 = policy_column<kPolFeat / 4>(act, w + kPolOffW1, w[kPolOffB1 + lane]);
  act[kPolHidden + lane] = fmaxf(h1, 0.0f);
  __syncwarp();
  float h2 = policy_column<kPolHidden / 4>(act + kPolHidden, w + kPolOffW2, w[kPolOffB2 + lane]);
  h2 = fmaxf(h2, 0.0f);
  // the four sums over the lanes, each lane keeping the half it will own:
  // output 2 (lane / 16) + (lane / 8) % 2
  const float4 w3 = reinterpret_cast<const float4*>(w + kPolOffW3)[lane];
  const float y0 = h2 * w3.x, y1 = h2 * w3.y, y2 = h2 * w3.z, y3 = h2 * w3.w;
  const bool hi = (lane & 16) != 0, odd = (lane & 8) != 0;
  const float r0 = (hi ? y2 : y0) + __shfl_xor_sync(0xFFFFFFFFu, hi ? y0 : y2, 16);
  const float r1 = (hi ? y3 : y1) + __shfl_xor_sync(0xFFFFFFFFu, hi ? y1 : y3, 16);
  float r = (odd ? r1 : r0) + __shfl_xor_sync(0xFFFFFFFFu, odd ? r0 : r1, 8);
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) r += __shfl_xor_sync(0xFFFFFFFFu, r, o);
  r += w[kPolOffB3 + (lane >> 3)];
#pragma unroll
  for (int a = 0; a < kPolArms; ++a) out[a] = __shfl_sync(0xFFFFFFFFu, r, a * 8);
}

// Arm with the smallest prediction among the allowed ones (lowest index on
// ties), kept only if it beats arm 0 (the paper's IN+OUT on the sparse queue)
// by kPolicyMargin in log2 time per settled vertex -- the network was fitted on
// smaller graphs, and a switch it is unsure of tends to cost more than it
// saves; arm 0 if any allowed prediction is not finite.
constexpr float kPolicyMargin = 0.35f;

// allow_dense = false (a fringe below n/32) leaves out the dense arms: a scan of
// all n vertices then costs far more per settled vertex than on the small
// training graphs the network has seen.
__device__ __forceinline__ int policy_pick(const float* y, bool allow_simple, bool allow_dense) {
  int best = 0;
  float yb = y[0];
  bool finite = true;
#pragma unroll
  for (int a = 0; a < kPolArms; ++a) {  // (unrolled, so that y stays in registers)
    const bool may = a < 2 || allow_simple;
    finite = finite && (!may || isfinite(y[a]));
    if (may && (allow_dense || !(a & 1)) && y[a] < yb) {
      best = a;
      yb = y[a];
    }
  }
  return finite && yb < y[0] - kPolicyMargin ? best : 0;
}

}  // namespace sssp
