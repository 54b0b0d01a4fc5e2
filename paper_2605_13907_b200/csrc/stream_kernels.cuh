// Host-callable launchers of the streaming (HBM / latency bound) kernels: FP8 block quantisation, merge of
// the per-split log-sum-exp partials, segmented and whole-batch reductions, per-token loss coefficients.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/ais.h"

namespace ais {

constexpr int kDiagBlocks = 592;      // fixed grid of the batch reductions (keeps the summation order fixed)
constexpr int kDiagThreads = 256;
constexpr int kNumMoments = 12;

// One matrix for the row quantiser with fp32 block scales.
struct QuantJob {
    const void* x;
    int64_t rows, ld;
    uint8_t* codes;
    int64_t ldq;
    float* scales;
    int64_t lds;
};
// Group-relative advantages adv[s]; zero_counts [S] and the two counters of the loss kernel (its finished blocks, the row tiles
// to recompute) are cleared for the kernels that count into them; each may be NULL.
struct AdvJob {
    const float* rewards;
    int32_t S, G, std_norm;
    float eps;
    float* adv;
    int32_t* zero_counts;
    uint32_t* tickets;
};
// Opening of a log-prob call: flags[i] = 1 when rows 128 i .. 128 i + 127 contain a row with mask != 0; `clear` (16-byte
// words, may be NULL) is zeroed on the way, and the advantages of the diagnostics that follow are formed (adv.S = 0: none).
struct FlagsJob {
    const uint8_t* mask;
    int64_t T;
    uint8_t* flags;
    void* clear;
    int64_t clear_bytes;
    AdvJob adv;
};
// The end of the batch moments, left to the kernel that follows: partial sums [blocks][kNumMoments], and where the
// diagnostics formed from their totals go.
struct TotalsJob {
    const double* partials;
    int32_t blocks;
    ais_params params;
    ais_diag* diag;
};
// The rectification of a batch (rho, w_tilde) as part of the loss kernel.
struct RectifyJob {
    const float* lp_roll;
    float C;
    TotalsJob totals;
    float *rho, *w_tilde;
    const float* seq_logw;
};

// The scratch rows that the forward pass of the same call has filled with exponentials (exp_form in lmhead.cuh), as part of
// the loss kernel: row factors, target columns, and which row tiles have to be recomputed.
struct KeepJob {
    __nv_bfloat16* U;
    int64_t ldU, rows;         // rows kept (the ones after them are recomputed anyway)
    const int32_t* tokens;
    int32_t V;
    float* scale;              // [T] factor of the row in the dH pass
    uint8_t* redo_flags;       // per row tile
    uint32_t* redo_count;      // zeroed before the launch
};

// Raises the dynamic shared-memory limit of the kernels here that need it (once per device).
cudaError_t stream_prepare();

// Rows quantised with one fp32 scale per `block` elements; one or two matrices (of the same width) and, if not NULL, the
// opening of the log-prob call that follows, in one launch.
cudaError_t launch_quantize(const QuantJob* jobs, int njobs, int64_t cols, int block, const FlagsJob* flags, cudaStream_t stream);

// Blocks running down the columns of x [K, ld] (K a multiple of 128): codes transposed [N, ldq], scales [K / block, lds].
cudaError_t launch_quantize_cols(const void* x, int64_t K, int64_t N, int64_t ld, int block, uint8_t* codes, int64_t ldq,
                                 float* scales, int64_t lds, cudaStream_t stream);

// Microscaling: E8M0 scale per 32 elements, packed in 512-byte chunks of 128 rows x 4 blocks; `scale_bytes` is the
// size of the whole packed array (rows padded to a multiple of 256); the padding rows get the neutral code.
cudaError_t launch_quantize_mx(const void* x, int64_t rows, int64_t cols, int64_t ld, uint8_t* codes, int64_t ldq,
                               uint8_t* scales, size_t scale_bytes, bool fp4 /* E2M1 elements, two per byte */,
                               cudaStream_t stream);

// One scale for the whole matrix (written to *scale on the device), then the codes.
cudaError_t launch_quantize_tensor(const void* x, int64_t rows, int64_t cols, int64_t ld, uint8_t* codes, int64_t ldq,
                                   float* scale, cudaStream_t stream);

// One merge of partial triples laid out [nparts][part_ld]: lp[t] = z_y - lse, lse[t] (may be NULL).
struct CombineJob {
    const float *part_m, *part_s, *part_z;
    int32_t nparts;
    float *lp, *lse;
};
// The batch moments as part of the merge of both passes (batches of at most kMergeMomentRows rows): partial sums
// [merge_moment_blocks(T)][kNumMoments].  adv is there already and n_valid_seq (may be NULL) has been cleared.
constexpr int kMergeRows = 32;                                           // rows of a merging block
constexpr int64_t kMergeMomentRows = int64_t(kDiagBlocks) * kMergeRows;
inline int merge_moment_blocks(int64_t T) { return static_cast<int>((T + kMergeRows - 1) / kMergeRows); }
struct MomentsJob {
    const int32_t* seq_offsets;
    const float* adv;
    int32_t S;
    float C;
    double* partials;
    int32_t* n_valid_seq;
};
// One or two merges (the passes of one call) in one launch, and, if not NULL, the batch moments (two merges, trainer first) or
// the advantages of the diagnostics that follow.
cudaError_t launch_combine(const CombineJob* jobs, int njobs, int64_t part_ld, const uint8_t* mask, int64_t T, uint32_t* status,
                           const AdvJob* adv, const MomentsJob* moments, cudaStream_t stream);
cudaError_t launch_flags(const FlagsJob& job, cudaStream_t stream);

// n_valid_seq[s] = valid rows of sequence s; zeroes `ticket` (the block counter of the reduction that follows).
cudaError_t launch_seq_counts(const uint8_t* mask, const int32_t* seq_offsets, int S, int32_t* n_valid_seq, uint32_t* ticket, cudaStream_t stream);
cudaError_t launch_advantages(const AdvJob& job, cudaStream_t stream);

// n_valid_seq (may be NULL) must have been cleared: the moments kernel adds every sequence's valid rows to it.
cudaError_t launch_diag(const float* lp_train, const float* lp_roll, const uint8_t* mask, const int32_t* seq_offsets,
                        const float* adv, int64_t T, int S, const ais_params& p, double* partials /*[kDiagBlocks][kNumMoments]*/,
                        int32_t* n_valid_seq, float* seq_logw /* [S] scratch: non-NULL selects sequence-level weights */,
                        float* rho, float* w_tilde, ais_diag* diag, bool early /* the log-probs are older than the kernel enqueued last */,
                        int merged_blocks /* > 0: the merge of the log-probs has left this many rows of partial sums */,
                        TotalsJob* later /* not NULL: the loss kernel forms alpha, rho and w_tilde from this */, cudaStream_t stream);

// The two halves of launch_diag: partial moments summed into `moments` [kNumMoments], and everything that follows
// from a (possibly all-reduced) moment vector.
cudaError_t launch_moments(const float* lp_train, const float* lp_roll, const uint8_t* mask, const int32_t* seq_offsets,
                           const float* adv, int64_t T, int S, const ais_params& p, double* partials, int32_t* n_valid_seq,
                           float* seq_logw, double* moments, cudaStream_t stream);
cudaError_t launch_finalize(const double* moments, const float* lp_train, const float* lp_roll, const uint8_t* mask, int64_t T,
                            const ais_params& p, float* rho, float* w_tilde, ais_diag* diag, const int32_t* seq_offsets, int S,
                            const float* seq_logw, cudaStream_t stream);

// coef[t], the row tiles that have a gradient, and the loss; n_valid_seq must already hold the valid counts, ticket zero.
// S_norm is the number of sequences the objective averages over (all data-parallel ranks together).  Rows whose lse is not
// finite (marked by the forward pass) contribute nothing.  Clears `clear` on the way.
cudaError_t launch_loss_coef(const float* lp_train, const float* lp_old, const float* lp_ref, float beta_kl, const uint8_t* mask,
                             const int32_t* seq_offsets, const float* adv, const float* w_tilde, const int32_t* n_valid_seq, int64_t T,
                             int S, int S_norm, float clip_eps, double* partials /*[kDiagBlocks][2]*/, uint32_t* ticket, float* coef,
                             uint8_t* tile_flags, void* clear, size_t clear_bytes, float* loss, ais_diag* diag, const float* lse,
                             const RectifyJob* rectify /* NULL: w_tilde is there already */,
                             const KeepJob* keep /* NULL; only with rectify */, cudaStream_t stream);

}  // namespace ais
