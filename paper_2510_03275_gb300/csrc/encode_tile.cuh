// Upsampling of 8 blocks of weights by one warp through a table with the
// half-shift symmetry (csrc/encode.cu says which and why).
#pragma once

#include "common.cuh"

namespace sdq {

constexpr int kTv = 8;    // virtual rows (row, block) per warp
// Floats between the 8-weight groups of k and k + 4 in the transposed weights
// [k][8]: 4 x 8 plus 8, so that the transposing stores hit 32 banks.
constexpr int kWk4 = 40;

// Floats of the transposed weights of 8 virtual rows of B inputs.
__host__ __device__ constexpr int tile_weight_floats(int B) { return B / 4 * kWk4; }

// x_up of the 8 virtual rows whose weights are in `wt`, pairs (j, j + np) for
// j = lane's first pair + 32 q, q < PT (pairs past `left` of them give
// zeros): acc gets sample j, acc2 sample j + np.  `tp` points at the lane's
// first pair in row 0 of the table's first half (B rows, `ld` apart; shared
// or global memory).  Canonical order: k ascending, every product and every sum rounded, the first product taken as
// is; acc2 subtracts the products of k >= B / 2 that acc adds.
template <int PT>
__device__ __forceinline__ void tile_upsample(const float* tp, int ld, int left, const float* wt, int B,
                                              float (&acc)[kTv][PT], float (&acc2)[kTv][PT]) {
  const int half = B / 2;
  bool in[PT];
#pragma unroll
  for (int q = 0; q < PT; ++q) in[q] = 32 * q < left;
  auto weights = [&](int k, float (&w)[kTv]) {
    const float4* s4 = reinterpret_cast<const float4*>(wt + (k >> 2) * kWk4 + (k & 3) * 8);
    const float4 a = s4[0], b = s4[1];
    w[0] = a.x; w[1] = a.y; w[2] = a.z; w[3] = a.w;
    w[4] = b.x; w[5] = b.y; w[6] = b.z; w[7] = b.w;
  };
  auto table = [&](int k, float (&a)[PT]) {
#pragma unroll
    for (int q = 0; q < PT; ++q) a[q] = in[q] ? tp[(size_t)k * ld + 32 * q] : 0.f;
  };
  {
    float w[kTv], a[PT];
    weights(0, w);
    table(0, a);
#pragma unroll
    for (int v = 0; v < kTv; ++v)
#pragma unroll
      for (int q = 0; q < PT; ++q) acc[v][q] = __fmul_rn(a[q], w[v]);
  }
#pragma unroll 4
  for (int k = 1; k < half; ++k) {
    float w[kTv], a[PT];
    weights(k, w);
    table(k, a);
#pragma unroll
    for (int v = 0; v < kTv; ++v)
#pragma unroll
      for (int q = 0; q < PT; ++q) acc[v][q] = __fadd_rn(acc[v][q], __fmul_rn(a[q], w[v]));
  }
#pragma unroll
  for (int v = 0; v < kTv; ++v)
#pragma unroll
    for (int q = 0; q < PT; ++q) acc2[v][q] = acc[v][q];
#pragma unroll 4
  for (int k = half; k < B; ++k) {
    float w[kTv], a[PT];
    weights(k, w);
    table(k, a);
#pragma unroll
    for (int v = 0; v < kTv; ++v)
#pragma unroll
      for (int q = 0; q < PT; ++q) {
        const float pr = __fmul_rn(a[q], w[v]);
        acc[v][q] = __fadd_rn(acc[v][q], pr);
        acc2[v][q] = __fsub_rn(acc2[v][q], pr);
      }
  }
}

// The first half of the encode table (B x n_b, row k: A_enc[.][k]) to shared
// memory, by the whole CTA.
__device__ __forceinline__ void tile_load_table(float* ts, const float* at, int B, int n_b) {
  const int np = n_b / 2;
  for (int i = threadIdx.x; i < B * np; i += blockDim.x) {
    const int k = i / np;
    ts[i] = __ldg(at + (size_t)k * n_b + (i - k * np));
  }
}

// One step of eq. (8): the code's field (1 or 2 bits) and the new feedback.
template <bool kTernary>
__device__ __forceinline__ uint32_t sd_step(float& integ, float& yp, float x, float alpha, float theta) {
  integ = __fsub_rn(__fadd_rn(integ, x), yp);
  if constexpr (kTernary) {
    const bool pos = integ > theta, neg = integ < -theta;
    yp = pos ? alpha : (neg ? -alpha : 0.f);
    return pos ? 1u : (neg ? 3u : 0u);
  } else {
    const bool pos = integ >= 0.f;
    yp = pos ? alpha : -alpha;
    return pos ? 1u : 0u;
  }
}

}  // namespace sdq
