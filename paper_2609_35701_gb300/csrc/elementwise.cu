// Bandwidth-bound kernels of the MeqMuon step (everything except the NS GEMMs).
//
//   momentum_norm : B <- mu B + G (Eq. (10)) in place over every matrix, with
//                   deterministic per-chunk partial sums of the squared NS
//                   input; the last chunk of each matrix reduces them into the
//                   X_0 scale alpha0 / ||H||_F of Eq. (5).
//   cast_x0       : X-hat_0 = 16-bit(alpha0 H / ||H||_F) in the oriented NS
//                   layout (transposed through shared memory for tall W).
//   momentum_x0, x0norm : the default: momentum and an unnormalised bf16 X_0 in
//                   one pass, then 1 / ||H||_F.
//   fold, finalize: r, c (Eq. (7)) from the partial sums of squares the last
//                   NS epilogue wrote, gamma_r, gamma_c (Eq. (8)), the
//                   direction (Eq. (11)) and the scale vector of Eq. (9).
//   rowcol, rows, colpart : momentum, row and column statistics of the remaining
//                   2D parameters and vectors (Eqs. (12), (13)).
//   apply         : W <- (1 - lr wd) W - rho lr U~ (Eq. (14)).
#include <algorithm>

#include "meq_elementwise.cuh"
#include "meq_stats.cuh"

namespace meq {
namespace {

__device__ __forceinline__ int64_t mat_begin(const MatInfo& m, int which) {
  return which == 0   ? m.chunk_begin
         : which == 1 ? m.tile_begin
         : which == 2 ? m.hchunk_begin
         : which == 3 ? m.rblk_begin
         : which == 4 ? m.slab_begin
         : which == 5 ? m.xblk_begin
         : which == 6 ? m.fold_begin
                      : m.rc_begin;
}

// Largest i with begin(i) <= key, by a whole warp; begin is nondecreasing in
// i. Entries that own no work of the enumeration share their begin with the
// next entry (or lie past the end), so they are never selected. The lanes
// probe 32 evenly spaced entries at a time: 1024 entries take two dependent
// loads where a binary search took ten, at the head of every block of the
// streaming kernels (Llama-350M, 168 entries: momentum 667 -> 647 us, update
// 484 -> 466 us; two 7B-class layers 881 -> 863 us and 628 -> 617 us).
__device__ __forceinline__ int find_mat(const MatInfo* mats, int nmat, int64_t key, int which) {
  const int lane = threadIdx.x & 31;
  int lo = 0, n = nmat;  // the answer lies in lo .. lo + n - 1
  while (n > 1) {
    const int step = (n + 31) / 32;
    const bool le = lane * step < n && mat_begin(mats[lo + lane * step], which) <= key;
    const int last = 31 - __clz(__ballot_sync(0xffffffffu, le) | 1u);  // lanes 0 .. last hold
    n = min(step, n - last * step);
    lo += last * step;
  }
  return lo;
}

// Row i and column j of flat element e of a matrix with n columns. Every
// model weight has fewer than 2^32 elements, where a 32-bit division is
// several times cheaper than a 64-bit one (measured: about 0.5% of the
// Llama-130M and 350M steps); small32 is uniform over a block, so the
// branch does not diverge.
__device__ __forceinline__ void row_col(int64_t e, int64_t n, bool small32, int64_t& i, int64_t& j) {
  if (small32) {
    const uint32_t eu = static_cast<uint32_t>(e), nu = static_cast<uint32_t>(n);
    const uint32_t iu = eu / nu;
    i = iu;
    j = eu - iu * nu;
  } else {
    i = e / n;
    j = e - i * n;
  }
}

__device__ __forceinline__ float block_sum_f32(float v, float* sh) {
  const unsigned FULL = 0xffffffffu;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(FULL, v, o);
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  __syncthreads();
  if (l == 0) sh[w] = v;
  __syncthreads();
  float r = 0.f;
  if (threadIdx.x == 0) {
    for (int i = 0; i < (int)(blockDim.x >> 5); ++i) r += sh[i];
    sh[0] = r;
  }
  __syncthreads();
  return sh[0];
}

// ------------------------------------------------------------- momentum + norm
__global__ void __launch_bounds__(kThreads) momentum_norm_kernel(const MatInfo* __restrict__ mats, int nmat,
                                                                 const GroupInfo* __restrict__ groups,
                                                                 float* __restrict__ mom,
                                                                 const float* const* __restrict__ grads,
                                                                 const StepScalars* __restrict__ sc,
                                                                 float* __restrict__ partials,
                                                                 unsigned int* __restrict__ counters,
                                                                 float* __restrict__ x0scale,
                                                                 int* __restrict__ nonfinite) {
  pdl_allow_dependents();
  __shared__ float shf[32];
  __shared__ int is_last;
  const int64_t chunk = blockIdx.x;
  const int mi = find_mat(mats, nmat, chunk, 2);
  const MatInfo& M = mats[mi];
  pdl_wait_predecessor();
  const int64_t numel = M.m * M.n;
  const int64_t e0 = (chunk - M.hchunk_begin) * kChunk;
  const int64_t e1 = min(e0 + kChunk, numel);
  const float mu = sc->mu;
  const int nesterov = sc->nesterov;
  float* B = mom + M.mom_off;
  const float* G = grads[mi];
  float ss = 0.f;
  // numel of a matrix need not be a multiple of 4: vector body + scalar tail.
  const int64_t vec_end = e0 + ((e1 - e0) & ~int64_t(3));
  for (int64_t e = e0 + 4 * threadIdx.x; e < vec_end; e += 4 * kThreads) {
    const float4 g = __ldcs(reinterpret_cast<const float4*>(G + e));
    float4 b = *reinterpret_cast<const float4*>(B + e);
    b.x = fmaf(mu, b.x, g.x);
    b.y = fmaf(mu, b.y, g.y);
    b.z = fmaf(mu, b.z, g.z);
    b.w = fmaf(mu, b.w, g.w);
    *reinterpret_cast<float4*>(B + e) = b;
    if (nesterov) {
      const float hx = fmaf(mu, b.x, g.x), hy = fmaf(mu, b.y, g.y), hz = fmaf(mu, b.z, g.z), hw = fmaf(mu, b.w, g.w);
      ss += hx * hx + hy * hy + hz * hz + hw * hw;
    } else {
      ss += b.x * b.x + b.y * b.y + b.z * b.z + b.w * b.w;
    }
  }
  for (int64_t e = vec_end + threadIdx.x; e < e1; e += kThreads) {
    const float g = G[e];
    const float b = fmaf(mu, B[e], g);
    B[e] = b;
    const float h = nesterov ? fmaf(mu, b, g) : b;
    ss += h * h;
  }
  const float part = block_sum_f32(ss, shf);
  if (threadIdx.x == 0) {
    partials[chunk] = part;
    __threadfence();
    const unsigned int nchunks = static_cast<unsigned int>((numel + kChunk - 1) / kChunk);
    const unsigned int prev = atomicAdd(&counters[mi], 1u);
    is_last = (prev + 1 == nchunks);
  }
  __syncthreads();
  if (!is_last) return;
  __threadfence();
  // Last chunk of this matrix: fixed-order fp32 reduction of its partials
  // (fp32 throughout: this GPU's fp64 rate is a small fraction of its fp32 rate).
  const int64_t nchunks = (numel + kChunk - 1) / kChunk;
  float acc = 0.f;
  for (int64_t c = threadIdx.x; c < nchunks; c += kThreads) acc += __ldcg(partials + M.hchunk_begin + c);
  const float total = block_sum_f32(acc, shf);
  if (threadIdx.x == 0) {
    const float nrm = sqrtf(total);
    if (!isfinite(total)) atomicCAS(nonfinite, 0, mi + 1);  // first non-finite entry, 1-based
    // Zero input: U = 0 (Eq. (5) is defined for a nonzero input only).
    x0scale[mi] = nrm > 0.f ? groups[M.group].alpha0 / nrm : 0.f;
    counters[mi] = 0u;
  }
}

__device__ __forceinline__ uint2 pack4_bf16(float a, float b, float c, float d) {
  uint2 w;
  __nv_bfloat162 x = __floats2bfloat162_rn(a, b), y = __floats2bfloat162_rn(c, d);
  w.x = *reinterpret_cast<uint32_t*>(&x);
  w.y = *reinterpret_cast<uint32_t*>(&y);
  return w;
}
__device__ __forceinline__ uint16_t bf16_bits(float v) {
  __nv_bfloat16 h = __float2bfloat16_rn(v);
  return *reinterpret_cast<uint16_t*>(&h);
}

// Hidden weights: B <- mu B + G (Eq. (10)) and X_0 = bf16(H) in the
// oriented NS layout, H being the NS input (B, or G + mu B for Nesterov).
// X_0 is left unnormalised: bf16 has the exponent range of fp32, and the
// first NS products apply 1 / ||H||_F (Eq. (5)) in their epilogues.
// Block t of the enumeration is a flat chunk of kChunk elements of W when
// X_0 has W's layout (B and G are contiguous, so they move as float4s
// whatever the row length), or a 64 x 64 tile of W transposed through shared
// memory when X_0 = W^T (tall W). Each block writes the fixed-order sum of
// squares of its part of H to partials[t]; x0norm_kernel reduces them.
__global__ void __launch_bounds__(kThreads, 8) momentum_x0_kernel(const MatInfo* __restrict__ mats, int nmat,
                                                                 const GroupInfo* __restrict__ groups,
                                                                 float* __restrict__ mom,
                                                                 const float* const* __restrict__ grads,
                                                                 const StepScalars* __restrict__ sc,
                                                                 float* __restrict__ partials) {
  pdl_allow_dependents();
  __shared__ float tile[kCastTile][kCastTile + 1];
  __shared__ float shf[32];
  const int64_t t = blockIdx.x;
  const int mi = find_mat(mats, nmat, t, 5);
  const MatInfo& M = mats[mi];
  pdl_wait_predecessor();
  const GroupInfo& Gi = groups[M.group];
  const int64_t lt = t - M.xblk_begin;
  const float mu = sc->mu;
  const int nesterov = sc->nesterov;
  float* B = mom + M.mom_off;
  const float* G = grads[mi];
  uint16_t* X = static_cast<uint16_t*>(Gi.x0) + M.gidx * Gi.s * Gi.lp;
  float ss = 0.f;
  if (!M.trans) {
    const int64_t e0 = lt * kChunk;
    const int64_t e1 = min(e0 + kChunk, M.m * M.n);
    const bool small32 = M.m * M.n <= static_cast<int64_t>(UINT32_MAX);
    for (int64_t e = e0 + 4 * threadIdx.x; e < e1; e += 4 * kThreads) {
      float h[4];
      if (e + 3 < e1) {
        const float4 g = __ldcs(reinterpret_cast<const float4*>(G + e));
        float4 b = *reinterpret_cast<const float4*>(B + e);
        b.x = fmaf(mu, b.x, g.x), b.y = fmaf(mu, b.y, g.y), b.z = fmaf(mu, b.z, g.z), b.w = fmaf(mu, b.w, g.w);
        *reinterpret_cast<float4*>(B + e) = b;
        if (nesterov) {
          h[0] = fmaf(mu, b.x, g.x), h[1] = fmaf(mu, b.y, g.y), h[2] = fmaf(mu, b.z, g.z), h[3] = fmaf(mu, b.w, g.w);
        } else {
          h[0] = b.x, h[1] = b.y, h[2] = b.z, h[3] = b.w;
        }
      } else {
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          h[u] = 0.f;
          if (e + u < e1) {
            const float g = G[e + u];
            const float b = fmaf(mu, B[e + u], g);
            B[e + u] = b;
            h[u] = nesterov ? fmaf(mu, b, g) : b;
          }
        }
      }
      ss += h[0] * h[0] + h[1] * h[1] + h[2] * h[2] + h[3] * h[3];
      int64_t i, j;
      row_col(e, M.n, small32, i, j);
      if ((M.n & 3) == 0) {
        // four columns of one row (m n is then a multiple of 4, so e + 3 < e1)
        *reinterpret_cast<uint2*>(X + i * Gi.lp + j) = pack4_bf16(h[0], h[1], h[2], h[3]);
      } else {
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          if (e + u < e1) X[i * Gi.lp + j] = bf16_bits(h[u]);
          if (++j == M.n) j = 0, ++i;
        }
      }
    }
  } else {
    const int64_t tiles_n = (M.n + kCastTile - 1) / kCastTile;
    const int64_t r0 = (lt / tiles_n) * kCastTile;
    const int64_t c0 = (lt % tiles_n) * kCastTile;
    const bool vec = (M.n & 3) == 0;
    const int cx = (threadIdx.x & 15) * 4;  // 4 columns
    const int ry = threadIdx.x >> 4;        // rows ry, ry + 16, ry + 32, ry + 48
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int64_t row = r0 + ry + 16 * k, col = c0 + cx;
      float h[4] = {0.f, 0.f, 0.f, 0.f};
      if (row < M.m) {
        if (vec && col + 3 < M.n) {
          const float4 g = __ldcs(reinterpret_cast<const float4*>(G + row * M.n + col));
          float4 b = *reinterpret_cast<const float4*>(B + row * M.n + col);
          b.x = fmaf(mu, b.x, g.x), b.y = fmaf(mu, b.y, g.y), b.z = fmaf(mu, b.z, g.z), b.w = fmaf(mu, b.w, g.w);
          *reinterpret_cast<float4*>(B + row * M.n + col) = b;
          if (nesterov) {
            h[0] = fmaf(mu, b.x, g.x), h[1] = fmaf(mu, b.y, g.y), h[2] = fmaf(mu, b.z, g.z), h[3] = fmaf(mu, b.w, g.w);
          } else {
            h[0] = b.x, h[1] = b.y, h[2] = b.z, h[3] = b.w;
          }
        } else {
#pragma unroll
          for (int u = 0; u < 4; ++u)
            if (col + u < M.n) {
              const float g = G[row * M.n + col + u];
              const float b = fmaf(mu, B[row * M.n + col + u], g);
              B[row * M.n + col + u] = b;
              h[u] = nesterov ? fmaf(mu, b, g) : b;
            }
        }
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        ss += h[u] * h[u];
        tile[ry + 16 * k][cx + u] = h[u];
      }
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int xr = ry + 16 * k;
      const int64_t xrow = c0 + xr, xcol = r0 + cx;
      if (xrow >= M.n) continue;
      if (xcol + 3 < M.m) {
        *reinterpret_cast<uint2*>(X + xrow * Gi.lp + xcol) =
            pack4_bf16(tile[cx][xr], tile[cx + 1][xr], tile[cx + 2][xr], tile[cx + 3][xr]);
      } else {
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (xcol + u < M.m) X[xrow * Gi.lp + xcol + u] = bf16_bits(tile[cx + u][xr]);
      }
    }
  }
  const float part = block_sum_f32(ss, shf);
  if (threadIdx.x == 0) partials[t] = part;
}

// 1 / ||H||_F of every hidden matrix (0 for a zero input, whose U is 0), one
// block per matrix: fixed-order fp32 reduction of the partials its momentum
// blocks wrote (fp32 throughout: this GPU's fp64 rate is a small fraction of
// its fp32 rate).
__global__ void __launch_bounds__(kThreads) x0norm_kernel(const MatInfo* __restrict__ mats,
                                                         const GroupInfo* __restrict__ groups,
                                                         const float* __restrict__ partials,
                                                         float* __restrict__ ginv, int* __restrict__ nonfinite) {
  pdl_allow_dependents();
  __shared__ float shf[32];
  const MatInfo& M = mats[blockIdx.x];
  if (M.kind != KIND_HIDDEN) {
    pdl_wait_predecessor();  // every block of the grid waits: its completion stands for its predecessors'
    return;
  }
  const int64_t nblk = M.trans ? ((M.m + kCastTile - 1) / kCastTile) * ((M.n + kCastTile - 1) / kCastTile)
                               : (M.m * M.n + kChunk - 1) / kChunk;
  const float* part = partials + M.xblk_begin;
  float* out = ginv + groups[M.group].mbase + M.gidx;
  pdl_wait_predecessor();
  float acc = 0.f;
  int64_t c = threadIdx.x;
  for (; c + 3 * kThreads < nblk; c += 4 * kThreads) {
    const float x0 = part[c], x1 = part[c + kThreads], x2 = part[c + 2 * kThreads], x3 = part[c + 3 * kThreads];
    acc += x0, acc += x1, acc += x2, acc += x3;
  }
  for (; c < nblk; c += kThreads) acc += part[c];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if ((threadIdx.x & 31) == 0) shf[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    float total = 0.f;  // the warps one after another: eight adds, fewer cycles than a tree of shuffles
#pragma unroll
    for (int w = 0; w < kThreads / 32; ++w) total += shf[w];
    const float nrm = sqrtf(total);
    if (!isfinite(total)) atomicCAS(nonfinite, 0, static_cast<int>(blockIdx.x) + 1);  // first non-finite entry, 1-based
    *out = nrm > 0.f ? 1.0f / nrm : 0.f;
  }
}

// ------------------------------------------- remaining 2D parameters, vectors
// B <- mu B + G (Eq. (10)) and the row sums of squares of B, one warp per row
// (a vector is a single row; remaining 2D parameters with rows longer than
// kRowColMax). Row sums go to rvec.
__global__ void __launch_bounds__(kThreads) rows_kernel(const MatInfo* __restrict__ mats, int nmat,
                                                       float* __restrict__ mom, const float* const* __restrict__ grads,
                                                       const StepScalars* __restrict__ sc, float* __restrict__ rvec) {
  pdl_allow_dependents();
  const int64_t blk = blockIdx.x;
  const int mi = find_mat(mats, nmat, blk, 3);
  const MatInfo& M = mats[mi];
  pdl_wait_predecessor();
  const int lane = threadIdx.x & 31;
  const int64_t row = (blk - M.rblk_begin) * (kThreads / 32) + (threadIdx.x >> 5);
  if (row >= M.m) return;  // no block-wide synchronisation below
  const float mu = sc->mu;
  float* B = mom + M.mom_off + row * M.n;
  const float* G = grads[mi] + row * M.n;
  float ss = 0.f;
  if ((M.n & 3) == 0) {
    for (int64_t c = 4 * lane; c < M.n; c += 128) {
      const float4 g = __ldcs(reinterpret_cast<const float4*>(G + c));
      float4 b = *reinterpret_cast<const float4*>(B + c);
      b.x = fmaf(mu, b.x, g.x), b.y = fmaf(mu, b.y, g.y), b.z = fmaf(mu, b.z, g.z), b.w = fmaf(mu, b.w, g.w);
      *reinterpret_cast<float4*>(B + c) = b;
      ss += b.x * b.x + b.y * b.y + b.z * b.z + b.w * b.w;
    }
  } else {
    for (int64_t c = lane; c < M.n; c += 32) {
      const float b = fmaf(mu, B[c], G[c]);
      B[c] = b;
      ss += b * b;
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
  if (lane == 0) rvec[M.vec_off + row] = ss;
}

// Both passes over a remaining 2D parameter with rows of up to kRowColMax
// entries in one: a warp keeps a row of B in registers while its sum of
// squares is reduced, then adds the squares of the normalised row (Eq. (12),
// inner operator) to its column sums, so B is read once (12 B / element where
// rows_kernel and colpart_kernel moved 16). One block per slab of M.slab_rows
// rows; slab sizes make whole waves of one block per SM.
template <int kElems, bool kVec>
__device__ __forceinline__ void rowcol_slab(const MatInfo& M, float* B, const float* G, int64_t r0, int64_t r1, float mu,
                                            float eps, float* __restrict__ rss, float* __restrict__ cpart,
                                            float (*sh)[kRowColMax]) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int n = static_cast<int>(M.n);
  // column of value u of this lane
  auto col = [&](int u) { return kVec ? 128 * (u >> 2) + 4 * lane + (u & 3) : 32 * u + lane; };
  float acc[kElems];
#pragma unroll
  for (int u = 0; u < kElems; ++u) acc[u] = 0.f;
  for (int64_t row = r0 + w; row < r1; row += kRowColThreads / 32) {
    float* Br = B + row * n;
    const float* Gr = G + row * n;
    float b[kElems];
    float ss = 0.f;
    if (kVec) {
      float4 g4[kElems / 4], b4[kElems / 4];
#pragma unroll
      for (int k = 0; k < kElems / 4; ++k)
        if (col(4 * k) < n) {
          g4[k] = __ldcs(reinterpret_cast<const float4*>(Gr + col(4 * k)));
          b4[k] = *reinterpret_cast<const float4*>(Br + col(4 * k));
        }
#pragma unroll
      for (int k = 0; k < kElems / 4; ++k) {
        float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
        if (col(4 * k) < n) {
          x = make_float4(fmaf(mu, b4[k].x, g4[k].x), fmaf(mu, b4[k].y, g4[k].y), fmaf(mu, b4[k].z, g4[k].z),
                          fmaf(mu, b4[k].w, g4[k].w));
          *reinterpret_cast<float4*>(Br + col(4 * k)) = x;
        }
        b[4 * k] = x.x, b[4 * k + 1] = x.y, b[4 * k + 2] = x.z, b[4 * k + 3] = x.w;
      }
    } else {
      float g[kElems];
#pragma unroll
      for (int u = 0; u < kElems; ++u) {
        g[u] = b[u] = 0.f;
        if (col(u) < n) g[u] = __ldcs(Gr + col(u)), b[u] = Br[col(u)];
      }
#pragma unroll
      for (int u = 0; u < kElems; ++u) {
        b[u] = fmaf(mu, b[u], g[u]);
        if (col(u) < n) Br[col(u)] = b[u];
      }
    }
#pragma unroll
    for (int u = 0; u < kElems; ++u) ss += b[u] * b[u];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
    if (lane == 0) rss[row] = ss;
    const float rms = sqrtf(ss / static_cast<float>(n));
    const float rinv = rms > eps ? 1.0f / rms : 0.f;
#pragma unroll
    for (int u = 0; u < kElems; ++u) {
      const float x = b[u] * rinv;
      acc[u] = fmaf(x, x, acc[u]);
    }
  }
  // the warps' column sums, in a fixed order: w and w + 8 first, then 0 .. 7
  constexpr int kHalf = kRowColThreads / 64;
  if (w >= kHalf) {
#pragma unroll
    for (int u = 0; u < kElems; ++u)
      if (col(u) < n) sh[w - kHalf][col(u)] = acc[u];
  }
  __syncthreads();
  if (w < kHalf) {
#pragma unroll
    for (int u = 0; u < kElems; ++u)
      if (col(u) < n) sh[w][col(u)] += acc[u];
  }
  __syncthreads();
  for (int c = threadIdx.x; c < n; c += kRowColThreads) {
    float t = 0.f;
#pragma unroll
    for (int i = 0; i < kHalf; ++i) t += sh[i][c];
    cpart[c] = t;
  }
}

__global__ void __launch_bounds__(kRowColThreads, 1) rowcol_kernel(const MatInfo* __restrict__ mats, int nmat,
                                                                  float* __restrict__ mom,
                                                                  const float* const* __restrict__ grads,
                                                                  const StepScalars* __restrict__ sc,
                                                                  float* __restrict__ rvec, float* __restrict__ parts) {
  pdl_allow_dependents();
  __shared__ float sh[kRowColThreads / 64][kRowColMax];
  const int64_t blk = blockIdx.x;
  const int mi = find_mat(mats, nmat, blk, 7);
  const MatInfo& M = mats[mi];
  const int64_t ls = blk - M.rc_begin;
  const int64_t r0 = ls * M.slab_rows;
  const int64_t r1 = min(r0 + M.slab_rows, M.m);
  pdl_wait_predecessor();
  const float mu = sc->mu, eps = sc->eps;
  float* B = mom + M.mom_off;
  const float* G = grads[mi];
  float* rss = rvec + M.vec_off;
  float* cp = parts + M.cpart_off + ls * M.n;
  if ((M.n & 3) == 0) {
    if (M.n <= 256) rowcol_slab<8, true>(M, B, G, r0, r1, mu, eps, rss, cp, sh);
    else if (M.n <= 512) rowcol_slab<16, true>(M, B, G, r0, r1, mu, eps, rss, cp, sh);
    else if (M.n <= 768) rowcol_slab<24, true>(M, B, G, r0, r1, mu, eps, rss, cp, sh);
    else rowcol_slab<32, true>(M, B, G, r0, r1, mu, eps, rss, cp, sh);
  } else {
    if (M.n <= 256) rowcol_slab<8, false>(M, B, G, r0, r1, mu, eps, rss, cp, sh);
    else if (M.n <= 512) rowcol_slab<16, false>(M, B, G, r0, r1, mu, eps, rss, cp, sh);
    else if (M.n <= 768) rowcol_slab<24, false>(M, B, G, r0, r1, mu, eps, rss, cp, sh);
    else rowcol_slab<32, false>(M, B, G, r0, r1, mu, eps, rss, cp, sh);
  }
}

// Column sums of squares of N_r(B) (Eq. (12), inner operator): one block per
// kColSlab rows x 256 columns, deterministic; rows with RMS at or below eps
// contribute nothing.
__global__ void __launch_bounds__(kThreads) colpart_kernel(const MatInfo* __restrict__ mats, int nmat,
                                                          const float* __restrict__ mom, const float* __restrict__ rvec,
                                                          const StepScalars* __restrict__ sc, float* __restrict__ parts) {
  pdl_allow_dependents();
  __shared__ float rinv[kColSlab];
  const int64_t blk = blockIdx.x;
  const int mi = find_mat(mats, nmat, blk, 4);
  const MatInfo& M = mats[mi];
  pdl_wait_predecessor();
  const int64_t ncc = (M.n + kThreads - 1) / kThreads;  // column chunks
  const int64_t lb = blk - M.slab_begin;
  const int64_t ls = lb / ncc;
  const int64_t c = (lb - ls * ncc) * kThreads + threadIdx.x;
  const int64_t r0 = ls * kColSlab;
  const int nr = static_cast<int>(M.m - r0 < kColSlab ? M.m - r0 : kColSlab);
  for (int rr = threadIdx.x; rr < kColSlab; rr += kThreads) {
    float v = 0.f;
    if (rr < nr) {
      const float rms = sqrtf(rvec[M.vec_off + r0 + rr] / static_cast<float>(M.n));
      v = rms > sc->eps ? 1.0f / rms : 0.f;
    }
    rinv[rr] = v;
  }
  __syncthreads();
  if (c >= M.n) return;
  const float* B = mom + M.mom_off + r0 * M.n + c;
  float a4[4] = {0.f, 0.f, 0.f, 0.f};
  int r = 0;
  for (; r + 8 <= nr; r += 8) {
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const float x = B[(r + u) * M.n] * rinv[r + u];
      a4[u & 3] += x * x;
    }
  }
  for (; r < nr; ++r) {
    const float x = B[r * M.n] * rinv[r];
    a4[r & 3] += x * x;
  }
  parts[M.cpart_off + ls * M.n + c] = (a4[0] + a4[1]) + (a4[2] + a4[3]);
}

// ------------------------------------------------------------------ X_0 cast
template <bool kFp16>
__device__ __forceinline__ uint16_t half_bits(float v) {
  if (kFp16) {
    __half h = __float2half_rn(v);
    return *reinterpret_cast<uint16_t*>(&h);
  }
  __nv_bfloat16 h = __float2bfloat16_rn(v);
  return *reinterpret_cast<uint16_t*>(&h);
}

__device__ __forceinline__ uint2 pack4(float a, float b, float c, float d, bool fp16) {
  uint2 w;
  if (fp16) {
    __half2 x = __floats2half2_rn(a, b), y = __floats2half2_rn(c, d);
    w.x = *reinterpret_cast<uint32_t*>(&x);
    w.y = *reinterpret_cast<uint32_t*>(&y);
  } else {
    __nv_bfloat162 x = __floats2bfloat162_rn(a, b), y = __floats2bfloat162_rn(c, d);
    w.x = *reinterpret_cast<uint32_t*>(&x);
    w.y = *reinterpret_cast<uint32_t*>(&y);
  }
  return w;
}

// One 64 x 64 tile of W per block. Threads read 4 consecutive columns
// (128-bit loads when the row length allows) and write 4 consecutive 16-bit
// values; tall matrices go through a shared-memory transpose.
template <bool kFp16>
__global__ void __launch_bounds__(kThreads) cast_x0_kernel(const MatInfo* __restrict__ mats, int nmat,
                                                           const GroupInfo* __restrict__ groups,
                                                           const float* __restrict__ mom,
                                                           const float* const* __restrict__ grads,
                                                           const StepScalars* __restrict__ sc,
                                                           const float* __restrict__ x0scale) {
  pdl_allow_dependents();
  __shared__ float tile[kCastTile][kCastTile + 1];
  const int64_t t = blockIdx.x;
  const int mi = find_mat(mats, nmat, t, 1);
  const MatInfo& M = mats[mi];
  pdl_wait_predecessor();
  const GroupInfo& Gi = groups[M.group];
  const int64_t tiles_n = (M.n + kCastTile - 1) / kCastTile;
  const int64_t lt = t - M.tile_begin;
  const int64_t r0 = (lt / tiles_n) * kCastTile;
  const int64_t c0 = (lt % tiles_n) * kCastTile;
  const float scale = x0scale[mi];
  const float mu = sc->mu;
  const int nesterov = sc->nesterov;
  const float* B = mom + M.mom_off;
  const float* G = grads[mi];
  uint16_t* X = static_cast<uint16_t*>(Gi.x0) + M.gidx * Gi.s * Gi.lp;
  const bool vec = (M.n & 3) == 0;
  const int cx = (threadIdx.x & 15) * 4;  // 4 columns
  const int ry = threadIdx.x >> 4;        // rows ry, ry + 16, ry + 32, ry + 48
  float h[4][4];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const int64_t row = r0 + ry + 16 * k, col = c0 + cx;
#pragma unroll
    for (int u = 0; u < 4; ++u) h[k][u] = 0.f;
    if (row >= M.m) continue;
    if (vec && col + 3 < M.n) {
      float4 b = *reinterpret_cast<const float4*>(B + row * M.n + col);
      if (nesterov) {
        const float4 g = *reinterpret_cast<const float4*>(G + row * M.n + col);
        b.x = fmaf(mu, b.x, g.x), b.y = fmaf(mu, b.y, g.y), b.z = fmaf(mu, b.z, g.z), b.w = fmaf(mu, b.w, g.w);
      }
      h[k][0] = b.x, h[k][1] = b.y, h[k][2] = b.z, h[k][3] = b.w;
    } else {
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (col + u < M.n) {
          float b = B[row * M.n + col + u];
          if (nesterov) b = fmaf(mu, b, G[row * M.n + col + u]);
          h[k][u] = b;
        }
    }
  }
  if (!M.trans) {
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int64_t row = r0 + ry + 16 * k, col = c0 + cx;
      if (row >= M.m) continue;
      if (col + 3 < M.n) {
        *reinterpret_cast<uint2*>(X + row * Gi.lp + col) =
            pack4(h[k][0] * scale, h[k][1] * scale, h[k][2] * scale, h[k][3] * scale, kFp16);
      } else {
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (col + u < M.n) X[row * Gi.lp + col + u] = half_bits<kFp16>(h[k][u] * scale);
      }
    }
  } else {
#pragma unroll
    for (int k = 0; k < 4; ++k)
#pragma unroll
      for (int u = 0; u < 4; ++u) tile[ry + 16 * k][cx + u] = h[k][u] * scale;
    __syncthreads();
    // X row = W column c0 + xr; X columns = W rows r0 + cx .. + 3.
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int xr = ry + 16 * k;
      const int64_t xrow = c0 + xr, xcol = r0 + cx;
      if (xrow >= M.n) continue;
      if (xcol + 3 < M.m) {
        *reinterpret_cast<uint2*>(X + xrow * Gi.lp + xcol) =
            pack4(tile[cx][xr], tile[cx + 1][xr], tile[cx + 2][xr], tile[cx + 3][xr], kFp16);
      } else {
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (xcol + u < M.m) X[xrow * Gi.lp + xcol + u] = half_bits<kFp16>(tile[cx + u][xr]);
      }
    }
  }
}

// ----------------------------------------------------------------- statistics
// The vectors of one entry that come from partial sums: r and c of a hidden
// weight (NS rows and columns, swapped for a transposed one), c of a
// remaining 2D parameter.
struct FoldVec {
  const float* parts;  // [count][len]
  int64_t count, len;
  float* dst;
  float inv;           // 1 / elements summed per entry
};
__device__ __forceinline__ FoldVec fold_vec(const MatInfo& M, int which, const float* parts, float* rvec, float* cvec) {
  FoldVec v;
  if (M.kind == KIND_HIDDEN) {
    const bool cols = (which == 1) != (M.trans != 0);  // which: 0 NS rows, 1 NS columns
    v.parts = parts + (which == 0 ? M.rpart_off : M.cpart_off);
    v.count = ((which == 0 ? M.l() : M.s()) + 31) / 32;
    v.len = which == 0 ? M.s() : M.l();
    v.dst = (cols ? cvec : rvec) + M.vec_off;
    v.inv = 1.0f / static_cast<float>(cols ? M.m : M.n);
  } else {
    v.parts = parts + M.cpart_off;
    v.count = (M.m + M.slab_rows - 1) / M.slab_rows;
    v.len = M.n;
    v.dst = cvec + M.vec_off;
    v.inv = 1.0f / static_cast<float>(M.m);
  }
  return v;
}

// Row i of remaining 2D parameter mi: its RMS in place of the row's sum of
// squares (left there by the row pass), and the row scale of Eq. (12).
__device__ __forceinline__ void two_sided_row(const MatInfo& M, int64_t i, int mi, float delta, float* rvec, float* svec,
                                              int* nonfinite) {
  const float ss = rvec[M.vec_off + i];
  if (!isfinite(ss)) atomicCAS(nonfinite, 0, mi + 1);
  const float rms = sqrtf(ss * (1.0f / static_cast<float>(M.n)));
  rvec[M.vec_off + i] = rms;
  svec[M.vec_off + i] = rms > delta ? 1.0f / rms : 0.f;
}

// r and c (Eq. (7)) from the partial sums of squares, ahead of finalize: a
// block takes kFoldCols consecutive entries of one vector, four per lane, and
// each of its 8 warps an eighth of their partials, added in fixed order. The
// rows of a remaining 2D parameter come first, one per thread.
__global__ void __launch_bounds__(kThreads) fold_kernel(const MatInfo* __restrict__ mats, int nmat,
                                                        const StepScalars* __restrict__ sc,
                                                        const float* __restrict__ parts, float* __restrict__ rvec,
                                                        float* __restrict__ cvec, float* __restrict__ svec,
                                                        float* __restrict__ tvec, int* __restrict__ nonfinite) {
  pdl_allow_dependents();
  __shared__ float sh[kThreads / 32][kFoldCols];
  const int64_t blk = blockIdx.x;
  const int mi = find_mat(mats, nmat, blk, 6);
  const MatInfo& M = mats[mi];
  const int64_t lb = blk - M.fold_begin;
  const int64_t first = M.kind == KIND_HIDDEN ? (M.s() + kFoldCols - 1) / kFoldCols : (M.m + kThreads - 1) / kThreads;
  const int which = lb >= first ? 1 : 0;
  if (M.kind == KIND_TWO_SIDED && which == 0) {
    pdl_wait_predecessor();
    const int64_t i = lb * kThreads + threadIdx.x;
    if (i < M.m) two_sided_row(M, i, mi, sc->eps, rvec, svec, nonfinite);
    return;
  }
  const FoldVec v = fold_vec(M, which, parts, rvec, cvec);
  const int64_t j0 = (lb - (which ? first : 0)) * kFoldCols;
  const int t = threadIdx.x;
  pdl_wait_predecessor();
  const float sum = fold_block(v.parts, v.count, v.len, j0, sh);
  if (t < kFoldCols && j0 + t < v.len) {
    const float rms = sqrtf(sum * v.inv);
    v.dst[j0 + t] = rms;
    if (M.kind == KIND_TWO_SIDED) tvec[M.vec_off + j0 + t] = rms > sc->eps ? 1.0f / rms : 0.f;
  }
}

// Statistics and normalisation scales, one block per parameter.
//   hidden     : r, c of U (Eq. (7)) from the partial sums the last NS
//                epilogue wrote, gamma_r, gamma_c (Eq. (8)), the side of
//                Eq. (11) and its scale vector (Eq. (9)) in svec;
//   remaining 2D: r = row RMS of B, c = column RMS of N_r(B) (Eq. (12)),
//                1/r in svec, 1/c in tvec, their CVs for inspection;
//   vector     : r[0] = RMS of B, 1/r[0] in svec (Eq. (13)).
// folded: r and c of the hidden weights and c of the remaining 2D parameters
// are there already (fold_kernel).
// RMS values at or below eps are treated as zero (scale 0).
__global__ void __launch_bounds__(kFinThreads, 2) finalize_kernel(const MatInfo* __restrict__ mats,
                                                               const StepScalars* __restrict__ sc,
                                                               const float* __restrict__ parts,
                                                               float* __restrict__ rvec, float* __restrict__ cvec,
                                                               float* __restrict__ svec, float* __restrict__ tvec,
                                                               MatStats* __restrict__ stats,
                                                               unsigned long long* __restrict__ dircount,
                                                               int* __restrict__ nonfinite, int folded) {
  pdl_allow_dependents();
  __shared__ float shf[6 * 32];
  const MatInfo& M = mats[blockIdx.x];
  const float delta = sc->eps;  // uploaded before the step's first kernel
  const FoldVec v0 = fold_vec(M, 0, parts, rvec, cvec), v1 = fold_vec(M, 1, parts, rvec, cvec);
  float* r = rvec + M.vec_off;
  float* c = cvec + M.vec_off;
  float* s = svec + M.vec_off;
  const float inv_n = 1.0f / static_cast<float>(M.n);
  pdl_wait_predecessor();
  if (M.kind == KIND_VECTOR) {
    if (threadIdx.x == 0) {
      if (!isfinite(r[0])) atomicCAS(nonfinite, 0, static_cast<int>(blockIdx.x) + 1);
      const float rms = sqrtf(r[0] * inv_n);  // r[0] holds the sum of squares
      r[0] = rms;
      s[0] = rms > delta ? 1.0f / rms : 0.f;
      stats[blockIdx.x].gamma_r = 0.0;
      stats[blockIdx.x].gamma_c = 0.0;
      stats[blockIdx.x].direction = 3;
    }
    return;
  }
  if (!folded) {
    if (M.kind == KIND_TWO_SIDED)
      for (int64_t i = threadIdx.x; i < M.m; i += blockDim.x)
        two_sided_row(M, i, static_cast<int>(blockIdx.x), delta, rvec, svec, nonfinite);
    for (int which = M.kind == KIND_HIDDEN ? 0 : 1; which < 2; ++which) {
      const FoldVec v = which == 0 ? v0 : v1;
      for (int64_t j = threadIdx.x; j < v.len; j += blockDim.x) {
        const float rms = sqrtf(strided_sum8(v.parts + j, v.count, v.len) * v.inv);
        v.dst[j] = rms;
        if (M.kind == KIND_TWO_SIDED) tvec[M.vec_off + j] = rms > delta ? 1.0f / rms : 0.f;
      }
    }
    __syncthreads();
  }
  // Eq. (8) over entries > delta: two passes (mean, then squared deviations),
  // fp32 with fixed-order block reductions.
  StatVecs vecs;
  vecs.a = r, vecs.b = c, vecs.la = M.m, vecs.lb = M.n;
  vecs.load();
  float gam0, gam1;
  block_cv2(vecs, delta, shf, &gam0, &gam1);
  int dir;
  if (M.kind == KIND_TWO_SIDED) {
    dir = 2;  // its scales are written with r and c
  } else if (sc->rule == 1) {
    // Eq. (6): every row scaled by sqrt(max(m, n)), no equilibration
    dir = 4;
    const float f = sqrtf(static_cast<float>(max(M.m, M.n)));
    for (int64_t i = threadIdx.x; i < M.m; i += blockDim.x) s[i] = f;
  } else {
    dir = gam0 >= gam1 - sc->tie_atol ? 0 : 1;
    vecs.each([&](int side, int64_t i, float x) {
      if (side == dir) s[i] = x > delta ? 1.0f / x : 0.0f;  // RMS at or below delta: treated as zero
    });
  }
  if (threadIdx.x == 0) {
    stats[blockIdx.x].gamma_r = static_cast<double>(gam0);
    stats[blockIdx.x].gamma_c = static_cast<double>(gam1);
    stats[blockIdx.x].direction = dir;
    if (dir < 2) dircount[2 * blockIdx.x + dir] += 1ull;  // one block per entry: no other writer
  }
}

// ----------------------------------------------------------------------- apply
// W <- (1 - lr wd) W - rho lr U~ (Eq. (14)), U~ = scaled U (hidden) or scaled
// B (remaining 2D: s_i t_j B_ij; vector: s_0 B_j). Under the Muon rule the
// hidden scale is sqrt(max(m, n)) for every row (Eq. (6)).
__global__ void __launch_bounds__(kThreads, 8) apply_kernel(const MatInfo* __restrict__ mats, int nmat,
                                                         float* const* __restrict__ params,
                                                         const uint16_t* __restrict__ uslab,
                                                         const float* __restrict__ mom,
                                                         const float* __restrict__ svec,
                                                         const float* __restrict__ tvec,
                                                         const MatStats* __restrict__ stats,
                                                         const StepScalars* __restrict__ sc) {
  pdl_allow_dependents();
  const int64_t chunk = blockIdx.x;
  const int mi = find_mat(mats, nmat, chunk, 0);
  const MatInfo& M = mats[mi];
  pdl_wait_predecessor();
  const int64_t numel = M.m * M.n;
  const int64_t e0 = (chunk - M.chunk_begin) * kChunk;
  const int64_t e1 = min(e0 + kChunk, numel);
  const float decay = 1.0f - sc->lr * sc->wd;
  const bool hidden = M.kind == KIND_HIDDEN;
  // hidden: U is fp16(kUScale U) with row stride un; others: the momentum, fp32, contiguous
  const float step = sc->rho * sc->lr * (hidden ? 1.0f / kUScale : 1.0f);
  // mode 0: per-row scale (also the uniform scale of Eq. (6), held per row);
  // 1: per-column scale; 2: row scale x column scale
  const int dir = hidden ? stats[mi].direction : (M.kind == KIND_TWO_SIDED ? 2 : 0);
  const int mode = dir == 4 ? 0 : dir;
  const float* sv = svec + M.vec_off;
  const float* tv = tvec + M.vec_off;
  const uint16_t* U16 = uslab + M.u_off;
  const float* U32 = mom + M.mom_off;
  float* W = params[mi];
  if ((M.n & 3) == 0) {
    // four columns of one row per thread (m n is a multiple of 4, so e + 3 < e1)
    const bool small32 = numel <= static_cast<int64_t>(UINT32_MAX);
    for (int64_t e = e0 + 4 * threadIdx.x; e < e1; e += 4 * kThreads) {
      int64_t i, j;
      row_col(e, M.n, small32, i, j);
      float4 w = *reinterpret_cast<const float4*>(W + e);
      float u[4];
      if (hidden) {
        const uint2 h = __ldcs(reinterpret_cast<const uint2*>(U16 + i * M.un + j));
        const float2 a = __half22float2(*reinterpret_cast<const __half2*>(&h.x));
        const float2 b = __half22float2(*reinterpret_cast<const __half2*>(&h.y));
        u[0] = a.x, u[1] = a.y, u[2] = b.x, u[3] = b.y;
      } else {
        const float4 b = __ldcs(reinterpret_cast<const float4*>(U32 + e));
        u[0] = b.x, u[1] = b.y, u[2] = b.z, u[3] = b.w;
      }
      float s0, s1, s2, s3;
      if (mode == 0) {
        s0 = s1 = s2 = s3 = sv[i];
      } else {
        const float4 s4 = *reinterpret_cast<const float4*>((mode == 1 ? sv : tv) + j);
        s0 = s4.x, s1 = s4.y, s2 = s4.z, s3 = s4.w;
        if (mode == 2) {
          const float si = sv[i];
          s0 *= si, s1 *= si, s2 *= si, s3 *= si;
        }
      }
      w.x = fmaf(decay, w.x, -step * (s0 * u[0]));
      w.y = fmaf(decay, w.y, -step * (s1 * u[1]));
      w.z = fmaf(decay, w.z, -step * (s2 * u[2]));
      w.w = fmaf(decay, w.w, -step * (s3 * u[3]));
      *reinterpret_cast<float4*>(W + e) = w;
    }
  } else {
    // rows of any length: W (and B) are contiguous, so they still move as
    // float4s of flat elements; U's rows start on 16 bytes, so its four values
    // are 2- or 4-byte aligned with the column's parity. Only the group that
    // straddles a row's end (or the matrix's) goes value by value. (One value
    // per thread and pass: 375 us for the update of four 1B-class layers, whose
    // FFN rows are 5461 long; 314 us this way.)
    const bool small32 = numel <= static_cast<int64_t>(UINT32_MAX);
    for (int64_t e = e0 + 4 * threadIdx.x; e < e1; e += 4 * kThreads) {
      int64_t i, j;
      row_col(e, M.n, small32, i, j);
      if (e + 3 < e1 && j + 3 < M.n) {
        float4 w = *reinterpret_cast<const float4*>(W + e);
        float u[4];
        if (hidden) {
          const uint16_t* up = U16 + i * M.un + j;
          if (j & 1) {
            const uint32_t mid = __ldcs(reinterpret_cast<const uint32_t*>(up + 1));
            const float2 m2 = __half22float2(*reinterpret_cast<const __half2*>(&mid));
            u[0] = __half2float(__ushort_as_half(__ldcs(up)));
            u[1] = m2.x, u[2] = m2.y;
            u[3] = __half2float(__ushort_as_half(__ldcs(up + 3)));
          } else {
            const uint32_t lo = __ldcs(reinterpret_cast<const uint32_t*>(up));
            const uint32_t hi = __ldcs(reinterpret_cast<const uint32_t*>(up + 2));
            const float2 a = __half22float2(*reinterpret_cast<const __half2*>(&lo));
            const float2 b = __half22float2(*reinterpret_cast<const __half2*>(&hi));
            u[0] = a.x, u[1] = a.y, u[2] = b.x, u[3] = b.y;
          }
        } else {
          const float4 b = __ldcs(reinterpret_cast<const float4*>(U32 + e));
          u[0] = b.x, u[1] = b.y, u[2] = b.z, u[3] = b.w;
        }
        float f[4];
        const float si = mode == 1 ? 1.f : sv[i];
        const float* cv = mode == 1 ? sv : tv;
#pragma unroll
        for (int k = 0; k < 4; ++k) f[k] = mode == 0 ? si : (mode == 1 ? cv[j + k] : si * cv[j + k]);
        w.x = fmaf(decay, w.x, -step * (f[0] * u[0]));
        w.y = fmaf(decay, w.y, -step * (f[1] * u[1]));
        w.z = fmaf(decay, w.z, -step * (f[2] * u[2]));
        w.w = fmaf(decay, w.w, -step * (f[3] * u[3]));
        *reinterpret_cast<float4*>(W + e) = w;
      } else {
#pragma unroll 1
        for (int64_t ek = e; ek < e1 && ek < e + 4; ++ek) {
          const float u = hidden ? __half2float(__ushort_as_half(U16[i * M.un + j])) : U32[ek];
          const float f = mode == 0 ? sv[i] : (mode == 1 ? sv[j] : sv[i] * tv[j]);
          W[ek] = fmaf(decay, W[ek], -step * (f * u));
          if (++j == M.n) j = 0, ++i;
        }
      }
    }
  }
}

// Elements e0 .. e1 (row-major) of one entry as fp32, for reading back: U
// (raw), or the normalised update that apply_kernel applies, W <- (1 - lr wd) W
// - rho lr U~: U~ = diag(r^-1) U or U diag(c^-1) (Eqs. (9), (11)), sqrt(max(m,
// n)) U under the Eq. (6) rule, N_c(N_r(B)) (Eq. (12)) or B / RMS(B) (Eq.
// (13)), with the same scale factors and operands.
__global__ void __launch_bounds__(kThreads) readback_kernel(MatInfo M, int mi, int raw, int64_t e0, int64_t e1,
                                                            const uint16_t* __restrict__ uslab,
                                                            const float* __restrict__ mom,
                                                            const float* __restrict__ svec,
                                                            const float* __restrict__ tvec,
                                                            const MatStats* __restrict__ stats, float* __restrict__ dst) {
  const bool hidden = M.kind == KIND_HIDDEN;
  const int dir = hidden ? stats[mi].direction : (M.kind == KIND_TWO_SIDED ? 2 : 0);
  const int mode = dir == 4 ? 0 : dir;
  const float* sv = svec + M.vec_off;
  const float* tv = tvec + M.vec_off;
  const uint16_t* U16 = uslab + M.u_off;
  const float* U32 = mom + M.mom_off;
  const float back = hidden ? 1.0f / kUScale : 1.0f;  // a power of two: exact
  const bool small32 = M.m * M.n <= static_cast<int64_t>(UINT32_MAX);
  for (int64_t e = e0 + static_cast<int64_t>(blockIdx.x) * kThreads + threadIdx.x; e < e1;
       e += static_cast<int64_t>(gridDim.x) * kThreads) {
    int64_t i, j;
    row_col(e, M.n, small32, i, j);
    const float u = hidden ? __half2float(__ushort_as_half(U16[i * M.un + j])) : U32[e];
    const float f = raw ? 1.0f : (mode == 0 ? sv[i] : (mode == 1 ? sv[j] : sv[i] * tv[j]));
    dst[e - e0] = (f * u) * back;
  }
}

// Bounded-wait self test: waits on a flag nobody sets and reports a timeout.
__global__ void wait_selftest_kernel(const volatile int* flag, int* err, unsigned long long timeout_ns) {
  unsigned long long t0;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t0));
  for (unsigned int it = 0;; ++it) {
    if (*flag != 0) return;
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    if (t - t0 > timeout_ns || it >= (1u << 28)) {
      atomicCAS(err, 0, DEV_TIMEOUT_TEST);
      return;
    }
  }
}

}  // namespace

cudaError_t launch_momentum_norm(const LaunchCtx& L, cudaStream_t st) {
  return launch_pdl(momentum_norm_kernel, dim3((unsigned)L.total_hchunks), dim3(kThreads), 0, st, 1, L.mats, L.nmat,
                    L.groups, L.mom, L.grads, L.sc, L.partials, L.counters, L.x0scale, L.nonfinite);
}

cudaError_t launch_momentum_x0(const LaunchCtx& L, cudaStream_t st) {
  return launch_pdl(momentum_x0_kernel, dim3((unsigned)L.total_xblks), dim3(kThreads), 0, st, 1, L.mats, L.nmat,
                    L.groups, L.mom, L.grads, L.sc, L.partials);
}

cudaError_t launch_x0norm(const LaunchCtx& L, cudaStream_t st) {
  return launch_pdl(x0norm_kernel, dim3((unsigned)L.nmat), dim3(kThreads), 0, st, 1, L.mats, L.groups,
                    static_cast<const float*>(L.partials), L.ginv, L.nonfinite);
}

cudaError_t launch_rows(const LaunchCtx& L, cudaStream_t st) {
  return launch_pdl(rows_kernel, dim3((unsigned)L.total_rblks), dim3(kThreads), 0, st, 1, L.mats, L.nmat, L.mom,
                    L.grads, L.sc, L.rvec);
}

cudaError_t launch_rowcol(const LaunchCtx& L, cudaStream_t st) {
  return launch_pdl(rowcol_kernel, dim3((unsigned)L.total_rcs), dim3(kRowColThreads), 0, st, 1, L.mats, L.nmat, L.mom,
                    L.grads, L.sc, L.rvec, L.parts);
}

cudaError_t launch_colpart(const LaunchCtx& L, cudaStream_t st) {
  return launch_pdl(colpart_kernel, dim3((unsigned)L.total_slabs), dim3(kThreads), 0, st, 1, L.mats, L.nmat,
                    static_cast<const float*>(L.mom), static_cast<const float*>(L.rvec), L.sc, L.parts);
}

cudaError_t launch_cast_x0(const LaunchCtx& L, bool fp16, cudaStream_t st) {
  if (fp16)
    return launch_pdl(cast_x0_kernel<true>, dim3((unsigned)L.total_tiles), dim3(kThreads), 0, st, 1, L.mats, L.nmat,
                      L.groups, static_cast<const float*>(L.mom), L.grads, L.sc, static_cast<const float*>(L.x0scale));
  return launch_pdl(cast_x0_kernel<false>, dim3((unsigned)L.total_tiles), dim3(kThreads), 0, st, 1, L.mats, L.nmat,
                    L.groups, static_cast<const float*>(L.mom), L.grads, L.sc, static_cast<const float*>(L.x0scale));
}

cudaError_t launch_stats(const LaunchCtx& L, cudaStream_t st) {
  if (L.fold) {
    const cudaError_t e = launch_pdl(fold_kernel, dim3((unsigned)L.total_folds), dim3(kThreads), 0, st, 1, L.mats,
                                     L.nmat, L.sc, static_cast<const float*>(L.parts), L.rvec, L.cvec, L.svec, L.tvec,
                                     L.nonfinite);
    if (e != cudaSuccess) return e;
  }
  return launch_pdl(finalize_kernel, dim3(L.nmat), dim3(kFinThreads), 0, st, 1, L.mats, L.sc,
                    static_cast<const float*>(L.parts), L.rvec, L.cvec, L.svec, L.tvec, L.stats, L.dircount,
                    L.nonfinite, L.fold);
}

cudaError_t launch_apply(const LaunchCtx& L, cudaStream_t st) {
  return launch_pdl(apply_kernel, dim3((unsigned)L.total_chunks), dim3(kThreads), 0, st, 1, L.mats, L.nmat, L.params,
                    static_cast<const uint16_t*>(L.uslab), static_cast<const float*>(L.mom),
                    static_cast<const float*>(L.svec), static_cast<const float*>(L.tvec),
                    static_cast<const MatStats*>(L.stats), L.sc);
}

cudaError_t launch_readback(const LaunchCtx& L, const MatInfo& M, int mi, bool raw, int64_t e0, int64_t e1, float* dst,
                            cudaStream_t st) {
  const int64_t blocks = std::min<int64_t>((e1 - e0 + kThreads - 1) / kThreads, 4096);
  readback_kernel<<<static_cast<unsigned>(blocks), kThreads, 0, st>>>(
      M, mi, raw ? 1 : 0, e0, e1, static_cast<const uint16_t*>(L.uslab), static_cast<const float*>(L.mom),
      static_cast<const float*>(L.svec), static_cast<const float*>(L.tvec), static_cast<const MatStats*>(L.stats), dst);
  return cudaPeekAtLastError();
}

cudaError_t launch_wait_selftest(const int* flag, int* err, unsigned long long timeout_ns, cudaStream_t st) {
  wait_selftest_kernel<<<1, 1, 0, st>>>(flag, err, timeout_ns);
  return cudaGetLastError();
}

}  // namespace meq
