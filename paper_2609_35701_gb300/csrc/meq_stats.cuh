// Device code of the row / column statistics, shared by the step's kernels and
// the allocation-free statistics call.
#pragma once

#include "meq_elementwise.cuh"

namespace meq {

// sum_{k < count} p[k * stride]: the sums of eight consecutive ranges of
// ceil(count / 8) terms, side by side so that the loads overlap. The order is
// that of fold_block, so an entry's statistics are the same bit for bit
// whether or not the other entries of the state make it fold its partials.
__device__ __forceinline__ float strided_sum8(const float* __restrict__ p, int64_t count, int64_t stride) {
  float a8[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
  const int n = static_cast<int>(count), per = (n + 7) / 8;
  const int64_t range = per * stride;
  int i = 0;
  for (; i < n - 7 * per; ++i, p += stride) {  // all eight ranges have a term i
#pragma unroll
    for (int u = 0; u < 8; ++u) a8[u] += p[u * range];
  }
  for (; i < per; ++i, p += stride) {
#pragma unroll
    for (int u = 0; u < 7; ++u)
      if (u * per + i < n) a8[u] += p[u * range];
  }
  return ((a8[0] + a8[1]) + (a8[2] + a8[3])) + ((a8[4] + a8[5]) + (a8[6] + a8[7]));
}

// Sums of kFoldCols consecutive entries of partial sums [count][len], by a
// block of kThreads: four entries per lane, an eighth of the partials per
// warp, added in a fixed order (strided_sum8's). Thread t < kFoldCols returns the sum of entry
// j0 + t (if it exists).
__device__ __forceinline__ float fold_block(const float* __restrict__ parts, int64_t count, int64_t len, int64_t j0,
                                            float (*sh)[kFoldCols]) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int64_t per = (count + 7) / 8;
  const int64_t k0 = w * per, k1 = min(k0 + per, count);
  float acc[4] = {0.f, 0.f, 0.f, 0.f};
  const float* p = parts + j0 + lane;
  if (j0 + kFoldCols <= len) {
    int64_t k = k0;
    for (; k + 4 <= k1; k += 4) {
      float x[4][4];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int u = 0; u < 4; ++u) x[i][u] = p[(k + i) * len + 32 * u];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int u = 0; u < 4; ++u) acc[u] += x[i][u];
    }
    for (; k < k1; ++k)
#pragma unroll
      for (int u = 0; u < 4; ++u) acc[u] += p[k * len + 32 * u];
  } else {
    for (int64_t k = k0; k < k1; ++k)
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (j0 + lane + 32 * u < len) acc[u] += p[k * len + 32 * u];
  }
#pragma unroll
  for (int u = 0; u < 4; ++u) sh[w][lane + 32 * u] = acc[u];
  __syncthreads();
  const int t = threadIdx.x;
  if (t >= kFoldCols) return 0.f;
  return ((sh[0][t] + sh[1][t]) + (sh[2][t] + sh[3][t])) + ((sh[4][t] + sh[5][t]) + (sh[6][t] + sh[7][t]));
}

// K block sums at once, one barrier for all of them: every warp adds the
// warps' sums up itself (the same tree in each, so all threads get the same
// values). sh holds 32 * K floats that no other call of the block uses.
template <int K>
__device__ __forceinline__ void block_sum_multi(float (&v)[K], float* sh) {
  const unsigned FULL = 0xffffffffu;
#pragma unroll
  for (int k = 0; k < K; ++k)
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v[k] += __shfl_xor_sync(FULL, v[k], o);
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  if (l == 0) {
#pragma unroll
    for (int k = 0; k < K; ++k) sh[32 * k + w] = v[k];
  }
  __syncthreads();
#pragma unroll
  for (int k = 0; k < K; ++k) {
    v[k] = l < static_cast<int>(blockDim.x >> 5) ? sh[32 * k + l] : 0.f;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v[k] += __shfl_xor_sync(FULL, v[k], o);
  }
}

// r (length la) and c (length lb) of one entry, spread over the block. Up to
// kStatRegs values per thread are read once and kept in registers for both
// passes of the CVs and for the scale vector (3 round trips to L2 otherwise).
constexpr int kStatRegs = 32;
struct StatVecs {
  const float *a, *b;
  int64_t la, lb;
  int nk;              // values per thread when they are kept in registers, else 0
  float x[kStatRegs];  // entry threadIdx.x + k * kFinThreads of a followed by b

  __device__ __forceinline__ void load() {
    const int64_t len = la + lb;
    nk = len <= static_cast<int64_t>(kStatRegs) * kFinThreads ? static_cast<int>((len + kFinThreads - 1) / kFinThreads) : 0;
#pragma unroll
    for (int k = 0; k < kStatRegs; ++k) {
      if (k >= nk) break;
      const int i = static_cast<int>(threadIdx.x) + k * kFinThreads;
      x[k] = i < static_cast<int>(la) ? a[i] : (i < static_cast<int>(len) ? b[i - static_cast<int>(la)] : 0.f);
    }
  }
  // f(side, index, value) for every entry of this thread
  template <typename F>
  __device__ __forceinline__ void each(F f) const {
    if (nk) {
      const int na = static_cast<int>(la), n = static_cast<int>(la + lb);
#pragma unroll
      for (int k = 0; k < kStatRegs; ++k) {
        if (k >= nk) break;
        const int i = static_cast<int>(threadIdx.x) + k * kFinThreads;
        if (i < n) f(i < na ? 0 : 1, i < na ? i : i - na, x[k]);
      }
    } else {
#pragma unroll 8
      for (int64_t i = threadIdx.x; i < la; i += kFinThreads) f(0, i, a[i]);
#pragma unroll 8
      for (int64_t i = threadIdx.x; i < lb; i += kFinThreads) f(1, i, b[i]);
    }
  }
};

// Two-pass fp32 CVs of Eq. (8) of r and c over their entries above delta,
// both at once: the mean pass, then the squared deviations.
__device__ __forceinline__ void block_cv2(const StatVecs& v, float delta, float* sh, float* ga, float* gb) {
  float p[4] = {0.f, 0.f, 0.f, 0.f};  // count and sum over r, then over c
  v.each([&](int side, int64_t, float x) {
    const bool in = x > delta, ia = in && side == 0, ib = in && side == 1;
    p[0] += ia ? 1.f : 0.f, p[1] += ia ? x : 0.f;
    p[2] += ib ? 1.f : 0.f, p[3] += ib ? x : 0.f;
  });
  block_sum_multi<4>(p, sh);
  const float mean_a = p[0] > 0.f ? p[1] / p[0] : 0.f;
  const float mean_b = p[2] > 0.f ? p[3] / p[2] : 0.f;
  float q[2] = {0.f, 0.f};
  v.each([&](int side, int64_t, float x) {
    const float d = x - (side == 0 ? mean_a : mean_b);
    q[0] += x > delta && side == 0 ? d * d : 0.f;
    q[1] += x > delta && side == 1 ? d * d : 0.f;
  });
  block_sum_multi<2>(q, sh + 4 * 32);
  *ga = p[0] > 0.f ? sqrtf(q[0] / p[0]) / mean_a : 0.f;
  *gb = p[2] > 0.f ? sqrtf(q[1] / p[2]) / mean_b : 0.f;
}

}  // namespace meq
