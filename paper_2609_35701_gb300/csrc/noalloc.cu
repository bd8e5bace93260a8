// Row / column statistics of one matrix without any device allocation.
//
// Some callers cannot call cudaMalloc: code that runs inside a framework
// which owns all device memory through its own pool and forbids outside
// allocations, and latency-critical paths that must not allocate after
// start-up (cudaMalloc may synchronise the whole device). For them this file
// provides meq_row_col_stats_noalloc(), the statistics step of the optimizer
// (row / column RMS, their coefficients of variation and the chosen
// normalisation side) for one caller-provided matrix. Its scratch lives in a
// file-scope __device__ array of fixed size that every GPU which loads the
// library holds until the process exits.
//
// It sums squares over blocks of 32 rows x 1024 columns, folds the partials
// with the step's own fold (small matrices: in the last kernel), and forms the
// CVs in two passes, all in fp32 like the full step's statistics, so results
// agree with meq_read_stats up to fp32 summation order. The same kernels, given
// scratch that the caller allocated, give the first point of the CV trajectory
// (meq_ns_cv_trajectory).
//
// Bound by the one read of U. 4096 x 11008 (180 MB, 26.6 us at the measured
// copy rate): 98 us with scalar loads, one thread per column of the fold, a
// CV block that went to L2 six times, and full launch gaps; 41 us now.
#include <mutex>
#include <string>

#include "../../include/meq.h"
#include "meq_stats.cuh"

namespace {

using namespace meq;

constexpr int kNaSlab = 32;        // rows per block
constexpr int kNaChunk = 1024;     // columns per block (four per thread)
constexpr int kMaxDevices = 64;

// 8 MiB of scratch: the row partial sums of squares (ceil(cols / 1024) x
// rows floats) followed by the column partial sums (ceil(rows / 32) x cols).
constexpr long long kScratchFloats = 2ll * 1024 * 1024;
static __device__ __align__(256) float g_stats_scratch[kScratchFloats];

std::mutex g_setup_mu;
float* g_scratch_addr[kMaxDevices] = {nullptr};

// One block per 32-row slab (blockIdx.x) and 1024-column chunk (blockIdx.y):
// the slab's column partial sums of squares over the chunk's columns, and
// the chunk's partial sums of squares of the slab's rows. kVec: rows are a
// multiple of 4 long and U is 16-byte aligned, so a thread takes four
// neighbouring columns, eight 16-byte loads in flight (else four columns 256
// apart, one after the other).
template <bool kVec>
__global__ void __launch_bounds__(kThreads, 3) na_stats_kernel(const float* __restrict__ U, int64_t m, int64_t n,
                                                               float* __restrict__ scratch) {
  pdl_allow_dependents();
  pdl_wait_predecessor();
  __shared__ float shr[kThreads / 32][32];
  const int64_t slab = blockIdx.x, chunk = blockIdx.y;
  const int64_t r0 = slab * kNaSlab;
  const int nr = static_cast<int>(m - r0 < kNaSlab ? m - r0 : kNaSlab);
  const int64_t c1 = (chunk + 1) * kNaChunk < n ? (chunk + 1) * kNaChunk : n;
  const int64_t nchunks = (n + kNaChunk - 1) / kNaChunk;
  const float* Us = U + r0 * n;
  float* rowss = scratch + chunk * m;
  float* cp = scratch + nchunks * m + slab * n;
  float racc[kNaSlab];
#pragma unroll
  for (int r = 0; r < kNaSlab; ++r) racc[r] = 0.f;
  if (kVec) {
    const int64_t c = chunk * kNaChunk + 4 * threadIdx.x;
    if (c < c1) {
      float4 cacc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int rb = 0; rb < kNaSlab; rb += 8) {
        float4 u[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          u[i] = make_float4(0.f, 0.f, 0.f, 0.f);
          if (rb + i < nr) u[i] = __ldcs(reinterpret_cast<const float4*>(Us + (rb + i) * n + c));
        }
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const float x = u[i].x * u[i].x, y = u[i].y * u[i].y, z = u[i].z * u[i].z, w = u[i].w * u[i].w;
          cacc.x += x, cacc.y += y, cacc.z += z, cacc.w += w;
          racc[rb + i] = (x + y) + (z + w);
        }
      }
      // the scratch's column part need not be 16-byte aligned (it follows nchunks * m floats)
      cp[c] = cacc.x, cp[c + 1] = cacc.y, cp[c + 2] = cacc.z, cp[c + 3] = cacc.w;
    }
  } else {
    for (int64_t c = chunk * kNaChunk + threadIdx.x; c < c1; c += kThreads) {
      float cacc = 0.f;
#pragma unroll
      for (int r = 0; r < kNaSlab; ++r) {
        if (r < nr) {
          const float u = Us[r * n + c];
          const float u2 = u * u;
          cacc += u2;
          racc[r] += u2;
        }
      }
      cp[c] = cacc;
    }
  }
  const unsigned FULL = 0xffffffffu;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
  for (int o = 16; o >= 1; o >>= 1) {
#pragma unroll
    for (int i = 0; i < o; ++i) {
      const bool up = (lane & o) != 0;
      const float send = up ? racc[i] : racc[i + o];
      const float keep = up ? racc[i + o] : racc[i];
      racc[i] = keep + __shfl_xor_sync(FULL, send, o);
    }
  }
  shr[w][lane] = racc[0];
  __syncthreads();
  if (threadIdx.x < nr) {
    float s = 0.f;
    for (int i = 0; i < kThreads / 32; ++i) s += shr[i][threadIdx.x];
    rowss[r0 + threadIdx.x] = s;
  }
}

// r (Eq. (7)) from the row partials and c from the column partials, blocks of
// kFoldCols rows first, then of columns; the row sums of squares are kept
// (first row of the scratch) for the CV kernel.
__global__ void __launch_bounds__(kThreads) na_fold_kernel(int64_t m, int64_t n, float* __restrict__ scratch,
                                                           float* __restrict__ r, float* __restrict__ c) {
  pdl_allow_dependents();
  pdl_wait_predecessor();
  __shared__ float sh[kThreads / 32][kFoldCols];
  const int64_t nslabs = (m + kNaSlab - 1) / kNaSlab;
  const int64_t nchunks = (n + kNaChunk - 1) / kNaChunk;
  const int64_t row_blocks = (m + kFoldCols - 1) / kFoldCols;
  const bool rows = blockIdx.x < row_blocks;
  const int64_t len = rows ? m : n;
  const int64_t j0 = (rows ? blockIdx.x : blockIdx.x - row_blocks) * static_cast<int64_t>(kFoldCols);
  const float sum = fold_block(rows ? scratch : scratch + nchunks * m, rows ? nchunks : nslabs, len, j0, sh);
  const int64_t j = j0 + threadIdx.x;
  if (threadIdx.x < kFoldCols && j < len) {
    if (rows) scratch[j] = sum;  // only this block reads or writes these rows' partials
    (rows ? r : c)[j] = sqrtf(sum * (1.0f / static_cast<float>(rows ? n : m)));
  }
}

// gamma_r, gamma_c (Eq. (8), over entries > delta) and the side (Eq. (11)),
// all fp32, in one block. With frob set, r and c are first divided by
// ||U||_F (from the row sums of squares, fixed order), so that they and the
// threshold describe X = U / ||U||_F; a zero U gives zeros. Without a fold
// launch before it, the block folds the partials itself.
__global__ void __launch_bounds__(kFinThreads) na_cv_kernel(int64_t m, int64_t n, float delta, float tie_atol, int frob,
                                                            int folded, float* __restrict__ scratch,
                                                            float* __restrict__ r, float* __restrict__ c,
                                                            double* __restrict__ gammas, int* __restrict__ direction) {
  pdl_allow_dependents();
  pdl_wait_predecessor();
  __shared__ float shf[7 * 32];
  if (!folded) {
    const int64_t nslabs = (m + kNaSlab - 1) / kNaSlab;
    const int64_t nchunks = (n + kNaChunk - 1) / kNaChunk;
    const float* cpart = scratch + nchunks * m;
    for (int64_t i = threadIdx.x; i < m; i += kFinThreads) {
      const float s = strided_sum8(scratch + i, nchunks, m);
      scratch[i] = s;  // only this thread reads or writes row i's partials
      r[i] = sqrtf(s * (1.0f / static_cast<float>(n)));
    }
    for (int64_t j = threadIdx.x; j < n; j += kFinThreads)
      c[j] = sqrtf(strided_sum8(cpart + j, nslabs, n) * (1.0f / static_cast<float>(m)));
    __syncthreads();
  }
  if (frob) {
    float tot[1] = {0.f};
    for (int64_t i = threadIdx.x; i < m; i += kFinThreads) tot[0] += scratch[i];
    block_sum_multi<1>(tot, shf + 6 * 32);
    const float inv = tot[0] > 0.f ? 1.0f / sqrtf(tot[0]) : 0.f;
    for (int64_t i = threadIdx.x; i < m; i += kFinThreads) r[i] *= inv;
    for (int64_t j = threadIdx.x; j < n; j += kFinThreads) c[j] *= inv;
    __syncthreads();
  }
  StatVecs vecs;
  vecs.a = r, vecs.b = c, vecs.la = m, vecs.lb = n;
  vecs.load();
  float g0, g1;
  block_cv2(vecs, delta, shf, &g0, &g1);
  if (threadIdx.x == 0) {
    gammas[0] = static_cast<double>(g0);
    gammas[1] = static_cast<double>(g1);
    *direction = g0 >= g1 - tie_atol ? 0 : 1;
  }
}

// Device address of the scratch array on the current device, looked up once
// per device (the host-side symbol is only a stand-in, not a device address).
cudaError_t scratch_address(float** out) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lock(g_setup_mu);
  if (!g_scratch_addr[dev]) {
    void* p = nullptr;
    e = cudaGetSymbolAddress(&p, g_stats_scratch);
    if (e != cudaSuccess) return e;
    if (p == nullptr) return cudaErrorInvalidSymbol;
    g_scratch_addr[dev] = static_cast<float*>(p);
  }
  *out = g_scratch_addr[dev];
  return cudaSuccess;
}

meq_status na_fail(meq_status s, const std::string& msg) {
  meq::set_global_error(msg);
  return s;
}

}  // namespace

namespace meq {

int64_t row_col_stats_scratch_floats(int64_t rows, int64_t cols) {
  return (cols + kNaChunk - 1) / kNaChunk * rows + (rows + kNaSlab - 1) / kNaSlab * cols;
}

cudaError_t launch_row_col_stats(const float* U, int64_t rows, int64_t cols, float eps, float tie_atol, int frob,
                                 float* scratch, float* r, float* c, double* gammas, int* direction, cudaStream_t st,
                                 const char** failed) {
  const int64_t nslabs = (rows + kNaSlab - 1) / kNaSlab;
  const int64_t nchunks = (cols + kNaChunk - 1) / kNaChunk;
  *failed = "statistics launch";
  const bool vec = (cols & 3) == 0 && (reinterpret_cast<uintptr_t>(U) & 15u) == 0;
  cudaError_t e = launch_pdl(vec ? na_stats_kernel<true> : na_stats_kernel<false>,
                             dim3(static_cast<unsigned>(nslabs), static_cast<unsigned>(nchunks)), dim3(kThreads), 0, st,
                             1, U, rows, cols, scratch);
  if (e != cudaSuccess) return e;
  const int folded = row_col_stats_scratch_floats(rows, cols) > kFoldMinParts ? 1 : 0;
  if (folded) {
    *failed = "fold launch";
    const int64_t blocks = (rows + kFoldCols - 1) / kFoldCols + (cols + kFoldCols - 1) / kFoldCols;
    e = launch_pdl(na_fold_kernel, dim3(static_cast<unsigned>(blocks)), dim3(kThreads), 0, st, 1, rows, cols, scratch, r,
                   c);
    if (e != cudaSuccess) return e;
  }
  *failed = "CV launch";
  return launch_pdl(na_cv_kernel, dim3(1), dim3(kFinThreads), 0, st, 1, rows, cols, eps, tie_atol, frob, folded, scratch,
                    r, c, gammas, direction);
}

}  // namespace meq

extern "C" meq_status meq_row_col_stats_noalloc(const float* U, int64_t rows, int64_t cols, float eps, float tie_atol,
                                                float* r, float* c, double* gammas, int* direction,
                                                void* cuda_stream) {
  if (!U || !r || !c || !gammas || !direction)
    return na_fail(MEQ_ERR_INVALID_ARG, "meq_row_col_stats_noalloc: U, r, c, gammas and direction must not be NULL");
  if (rows <= 0 || cols <= 0 || rows > (int64_t(1) << 20) || cols > (int64_t(1) << 20))
    return na_fail(MEQ_ERR_INVALID_ARG, "meq_row_col_stats_noalloc: rows and cols must be in 1..2^20");
  if (!(eps >= 0.f) || !(tie_atol >= 0.f))
    return na_fail(MEQ_ERR_INVALID_ARG, "meq_row_col_stats_noalloc: eps and tie_atol must be >= 0");
  const int64_t need = meq::row_col_stats_scratch_floats(rows, cols);
  if (need > kScratchFloats)
    return na_fail(MEQ_ERR_INVALID_ARG, "meq_row_col_stats_noalloc: " + std::to_string(rows) + " x " +
                                            std::to_string(cols) + " needs " + std::to_string(need) +
                                            " floats of scratch, above the fixed " + std::to_string(kScratchFloats));
  float* scratch = nullptr;
  cudaError_t e = scratch_address(&scratch);
  if (e != cudaSuccess)
    return na_fail(MEQ_ERR_CUDA, std::string("meq_row_col_stats_noalloc: scratch address lookup: ") + cudaGetErrorString(e));
  const char* what = "";
  e = meq::launch_row_col_stats(U, rows, cols, eps, tie_atol, 0, scratch, r, c, gammas, direction,
                                static_cast<cudaStream_t>(cuda_stream), &what);
  if (e != cudaSuccess)
    return na_fail(MEQ_ERR_CUDA, std::string("meq_row_col_stats_noalloc: ") + what + ": " + cudaGetErrorString(e));
  return MEQ_OK;
}
