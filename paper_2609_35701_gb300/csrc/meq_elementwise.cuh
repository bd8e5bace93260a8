// Launch interface of the bandwidth-bound kernels (internal).
#pragma once

#include "meq_internal.cuh"

namespace meq {

constexpr int kThreads = 256;      // block size of most kernels
constexpr int64_t kChunk = 4096;   // elements per momentum / apply block
constexpr int kCastTile = 64;      // X_0 cast tile (64 x 64 of W)
constexpr int kFinThreads = 512;   // finalize block size (two blocks per SM)
constexpr int kColSlab = 128;      // rows per block of the remaining-2D column pass (at least, in the one-pass form)
constexpr int kRowColMax = 1024;   // longest row of the one-pass form: 32 values per lane, and as many column sums
constexpr int kRowColThreads = 512;
// The partial sums get a launch of their own (fold_kernel) when an entry has
// more of them than this; below, one finalize block reads them in less time
// than a launch takes. Whole steps of one weight, one block per entry -> fold,
// then finalize (partials): 256 x 256 (4.1k) 74.2 -> 75.1 us; 256 x 512 (8.2k)
// 82.1 -> 82.4; 200 x 768 (10.2k) 88.1 -> 87.8; 384 x 768 (18.4k) 97.8 -> 96.5;
// 512 x 1376 (44k) 118.9 -> 115.7; 256 x 4096 (66k) 168.6 -> 161.4; of thirty,
// 256 x 768 (12.3k) 148.5 -> 148.1. Statistics phase: two 7B-class layers 318 ->
// 35 us; two 32000 x 768 embeddings and the Llama-130M weights 79.7 -> 28.3 us.
constexpr int kFoldCols = 128;     // vector entries per block of the fold
constexpr int64_t kFoldMinParts = 8192;

struct MatStats {
  double gamma_r;
  double gamma_c;
  int32_t direction;  // 0 = row (N_r), 1 = column (N_c), 2 = two-sided, 3 = vector, 4 = Eq. (6) shape factor
  int32_t pad;
};

// Device pointers and sizes the elementwise launchers need.
struct LaunchCtx {
  const MatInfo* mats;
  int nmat;
  const GroupInfo* groups;
  float* mom;
  const float* const* grads;
  float* const* params;
  const StepScalars* sc;
  float* partials;
  unsigned int* counters;
  float* x0scale;
  float* ginv;           // 1 / ||H||_F per hidden matrix, ordered group by group
  uint16_t* uslab;       // U of every hidden matrix, fp16, scaled by kUScale
  float* parts;          // NS-row and NS-column partial sums of squares
  float* rvec;
  float* cvec;
  float* svec;           // hidden: scale of the chosen side; others: 1 / row RMS
  float* tvec;           // remaining 2D: 1 / column RMS of the row-normalised momentum
  MatStats* stats;
  unsigned long long* dircount;  // per entry: Eq. (11) row choices, column choices
  int* nonfinite;                // 1 + index of the first entry whose momentum had a non-finite norm, or 0
  int64_t total_chunks, total_hchunks, total_tiles, total_rblks, total_slabs, total_xblks, total_folds, total_rcs;
  int fold;                      // 1: the partial sums are folded by a launch of their own before finalize
  int n_hidden;
};

constexpr int KIND_HIDDEN = 0, KIND_TWO_SIDED = 1, KIND_VECTOR = 2;

cudaError_t launch_momentum_norm(const LaunchCtx& L, cudaStream_t st);
cudaError_t launch_momentum_x0(const LaunchCtx& L, cudaStream_t st);  // fused momentum + bf16 X_0
cudaError_t launch_x0norm(const LaunchCtx& L, cudaStream_t st);       // 1 / ||H||_F from its partials
cudaError_t launch_rowcol(const LaunchCtx& L, cudaStream_t st);    // remaining 2D, rows up to kRowColMax
cudaError_t launch_rows(const LaunchCtx& L, cudaStream_t st);      // remaining 2D with longer rows, vectors
cudaError_t launch_colpart(const LaunchCtx& L, cudaStream_t st);   // remaining 2D with longer rows
cudaError_t launch_cast_x0(const LaunchCtx& L, bool fp16, cudaStream_t st);
cudaError_t launch_stats(const LaunchCtx& L, cudaStream_t st);  // [fold and] finalize of the fused statistics
cudaError_t launch_apply(const LaunchCtx& L, cudaStream_t st);
// Elements e0 .. e1 of entry mi's U (raw) or U~ (the update apply_kernel applies) into dst[0 ..] (device, fp32).
cudaError_t launch_readback(const LaunchCtx& L, const MatInfo& M, int mi, bool raw, int64_t e0, int64_t e1, float* dst,
                            cudaStream_t st);
cudaError_t launch_wait_selftest(const int* flag, int* err, unsigned long long timeout_ns, cudaStream_t st);

}  // namespace meq
