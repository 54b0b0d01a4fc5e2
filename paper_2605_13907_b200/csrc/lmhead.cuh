// Arguments shared by the host launcher and the LM-head tensor-core kernels.
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <stdint.h>

namespace ais {

enum LmheadMode : int {
    kFwdBf16 = 0,   // z = H W^T (bf16), streaming log-sum-exp + target pick -> partial triples
    kFwdFp8  = 1,   // z^ from E4M3 codes with per-block scale promotion, same epilogue
    kBwdP    = 2,   // recompute z (bf16), write u = softmax - onehot as bf16 scratch
    kBwdDh   = 3,   // dH = c (.) (U W), contraction over the vocabulary
    kFwdFp8T = 4,   // E4M3 codes with one scale per tensor: whole contraction in tensor memory, one multiply after
    kBwdDw   = 5,   // dW += U^T H, contraction over the rows (both operands read with the contraction axis as rows)
    kFwdMx   = 6,   // E4M3 codes with one power-of-two (E8M0) scale per 32 elements: hardware block-scaled MMA
    kFwdMx4  = 7,   // packed E2M1 (FP4) codes with one E8M0 scale per 32 elements
    // the same three bf16 passes with W stored [d, V] (one row per hidden unit): the forward passes then read W as an
    // MN-major B operand (four 64-column boxes per stage, like the dH pass of the other layout) and the dH pass reads it
    // K-major (like the forward passes of the other layout)
    kFwdBf16Dv = 8,
    kBwdPDv    = 9,
    kBwdDhDv   = 10,
    // the trainer pass that also stores the exponentials of its logits in the scratch of the dH pass (see exp_form)
    kFwdKeep   = 11,
    kFwdKeepDv = 12
};

// What a mode computes (its epilogue and work-unit shape), whatever the layout of W.
__host__ __device__ constexpr int base_mode(int mode) {
    return mode == kFwdBf16Dv || mode == kFwdKeep || mode == kFwdKeepDv ? kFwdBf16 : mode == kBwdPDv ? kBwdP : mode == kBwdDhDv ? kBwdDh : mode;
}
// B operand stored with the output column as the contiguous axis (MN-major)?
__host__ __device__ constexpr bool b_mn_major(int mode) {
    return mode == kBwdDh || mode == kBwdDw || mode == kFwdBf16Dv || mode == kBwdPDv || mode == kFwdKeepDv;
}

constexpr int kSms = 148;                // SMs of the part; the work splits below are planned for it
constexpr int kMaxRanges = kSms;         // most vocabulary ranges of a row tile
constexpr int kBM = 128;                 // rows per tile (TMEM lanes)
constexpr int kBN = 256;                 // columns per tile (TMEM columns of one accumulator)
constexpr int kStageKBytes = 128;        // bytes of K per shared-memory stage row (one swizzle span)
constexpr int kAStageBytes = kBM * kStageKBytes;
constexpr int kBStageBytes = kBN * kStageKBytes;
constexpr int kStageBytes = kAStageBytes + kBStageBytes;
constexpr int kStages = 4;
// dH pass: a CTA owns two row tiles (256 rows) so that every W tile it loads feeds two accumulators
constexpr int kDhRows = 2 * kBM;
constexpr int kDhStageBytes = 2 * kAStageBytes + kBStageBytes;
constexpr int kDhStages = 3;
// rollout pass with fp32 block scales: a tile is two row tiles (256 rows) x 128 columns, so that a column scale read from
// shared memory serves two rows of a thread
constexpr int kPairRows = 2 * kBM;
constexpr int kPairCols = 128;
static_assert(kDhStages * kDhStageBytes <= kStages * kStageBytes, "the dH stage ring must fit the same shared memory");
constexpr int kNumBarriers = 3 * kStages + 4 + 1;
// microscaling passes: per 128-byte K stage one 512-byte scale chunk for the 128 rows of A and two for the 256 rows of B
// (FP8: 128 elements per stage), twice that with FP4 operands (256 elements per stage)
constexpr int kMxChunkBytes = 512;
constexpr int kMxStageScaleBytes = 6 * kMxChunkBytes;
constexpr int kThreads = 384;            // warp 0 TMA, warp 1 MMA, warps 2..3 idle, warps 4..11 epilogue
constexpr int kEpiWarps = 8;
constexpr int kMxThreads = 512;          // microscaling passes: warps 12..15 move the block scales into tensor memory
constexpr int kSmemBytes = 1024 + kStages * kStageBytes + kStages * kMxStageScaleBytes + kNumBarriers * 8 + 64;

// dH: one partial tile of a split unit, 256 x 256 fp32, ordered for 16-byte accesses with the rows across the lanes:
// [row half][group of 4 columns][128 rows][4 columns]
constexpr int kPartTileFloats = kDhRows * kBN;

// Exponent form of a scratch row.  The gradient of a row is c (softmax - onehot) W = c e^-lse (e^z - e^lse onehot) W, and the
// factor in front does not depend on the column: with U = e^z off the target and (p - 1) e^lse at it, the dH pass only has
// to scale its rows by c e^-lse at the end.  e^z is there before lse, c or alpha are known -- the forward pass forms it for
// its sum -- so a step that runs log-probs and loss in one call stores it there and has no logits to recompute.  bf16 has
// the exponent range of fp32, so the relative rounding is that of softmax itself as long as e^z neither overflows nor loses
// terms that matter: rows with lse in [-20, 59] (terms below e^-67 of the row's sum vanish).  Other rows are in plain form,
// U = c (softmax - onehot) and scale 1; their row tiles are recomputed.  p - 1 at the target comes from the log-prob
// (expm1), so a nearly certain token loses nothing to cancellation.
__host__ __device__ inline bool exp_form(float lse) { return lse >= -20.0f && lse <= 59.0f; }
__device__ __forceinline__ float exp_form_target(float lp, float lse) { return expm1f(lp) * expf(lse); }

// Pacing of the CTAs of a launch (lmhead_common.cuh): stage fills per announcement, counters in the ring.
constexpr int kPaceFills = 16;
constexpr int kPaceSettle = 4;     // stage fills between an announcement and the look at the counter it waits for
constexpr int kPaceRing = 4096;

struct LmheadArgs {
    int64_t rows;          // valid rows handled by this launch
    int64_t row0;          // global index of local row 0 (per-row vectors are indexed globally)
    int32_t n_row_tiles;   // row tiles of 128 rows (dH pass: of 256 rows)
    int32_t ncols;         // output columns: V (forward, recompute) or d (dH)
    int32_t n_col_tiles;
    int32_t ksteps;        // shared-memory stages per accumulator tile
    int32_t nsplit;        // forward / recompute: independent column ranges per row tile
    int32_t block_tiles;   // MN-major B of a [d, V] head: column tiles below this are whole and come by one copy of four blocks
    int32_t sgroups;       // FP8: scale blocks per stage (128 / fp8_block)
    const uint8_t* tile_active;   // one byte per global 128-row tile: 0 = nothing to compute there (may be NULL)
    const int32_t* tokens;
    const uint8_t* mask;
    float* part_m;         // [nsplit*2][part_ld] running maxima (natural log units)
    float* part_s;         // sums of exp(z - m)
    float* part_z;         // target logit or -inf
    int64_t part_ld;
    const float* lse;      // recompute: log-sum-exp of the trainer pass
    __nv_bfloat16* U;      // recompute output / dH input scratch [rows_pad, ldU]
    int64_t ldU;
    const float* scale_a;  // per-tensor FP8: the two scales (one float each, on the device)
    const float* scale_b;
    const float* coef;     // recompute: per-row factor c_t folded into the scratch
    const uint8_t* sf_a;   // microscaling: packed scale chunks of A [row chunks of 128][d/128][512 bytes]
    const uint8_t* sf_b;   // and of B
    int32_t nk4;           // d / 128: scale chunks per 128 rows
    float* dW;             // dW pass: [V, lddw] fp32
    int64_t lddw;
    int32_t dw_accumulate; // dW pass: add to what dW holds instead of overwriting it
    __nv_bfloat16* dH;
    int64_t lddh;
    uint32_t* status;
    int64_t wait_cycles;   // bound of every device-side wait in clock ticks; 0 = the default (about two seconds)
    int32_t split_from;    // dH: units from here on are split along the contraction (the last, partial wave); others whole
    int32_t ksplit;        // dH: ranges of the contraction per split unit (1 = nothing is split)
    float* part_acc;       // dH: fp32 partial tiles of the split units, [slot][kPartTileFloats] (see dh_reduce_kernel)
    int64_t keep_rows;     // kFwdKeep: rows (from the first) whose exponentials go to U
    const float* lp;       // recompute: log-probs of the targets (exponent form)
    const float* row_scale;   // recompute: non-NULL selects the exponent form; dH: factor of every row (0: the row is zero)
    const uint32_t* gate;  // recompute: non-NULL: run only if *gate != 0, and leave the rows of inactive tiles as they are
    uint32_t* pace;        // ring of kPaceRing zeroed counters that keeps the CTAs of the launch in step; NULL = no pacing
    uint32_t* pace_clear;  // ring of the next pass of the same call, cleared by this one; NULL = nothing to clear
    int32_t overlap;       // the pass needs nothing from the kernel before it (the other pass of the same call): it starts
                           // while that one drains and waits for it only at its own end
    int32_t pace_per_unit; // announcements per unit = ceil(largest number of stage fills of a unit / fills per announcement)
};

// Launches one pass.  tmSA / tmSB are only read in kFwdFp8 mode; with an MN-major B tmB maps blocks of 64 columns
// (make_tmap_blocks) and tmSA, for the last column tile of a [d, V] head, plain 64 x 64 boxes.
cudaError_t launch_lmhead(int mode, const CUtensorMap& tmA, const CUtensorMap& tmB, const CUtensorMap& tmSA,
                          const CUtensorMap& tmSB, const LmheadArgs& args, int num_ctas, cudaStream_t stream);
// Sums the partial tiles of a dH launch's split units (args as that launch got them) and writes their part of dH.
cudaError_t launch_dh_reduce(const LmheadArgs& args, cudaStream_t stream);
cudaError_t lmhead_prepare();   // sets the dynamic shared-memory attribute of every instantiation

// The rollout pass with per-block scales (mode kFwdFp8; args.sgroups = 128 / block = 1, 2 or 4).  tmSA / tmSB map the
// block-major scale arrays with boxes of kPairRows (256) and kPairCols (128) rows, each times sgroups blocks.
cudaError_t launch_lmhead_fp8_block(const CUtensorMap& tmA, const CUtensorMap& tmB, const CUtensorMap& tmSA,
                                    const CUtensorMap& tmSB, const LmheadArgs& args, int num_ctas, cudaStream_t stream);
cudaError_t lmhead_fp8_block_prepare();

// The forward and recompute passes (no microscaling) with two row tiles per CTA, and the dW pass: n_row_tiles counts 256-row
// units, tmA has boxes of 256 rows (dW: blocks, make_tmap_blocks).
cudaError_t launch_lmhead_pair(int mode, const CUtensorMap& tmA, const CUtensorMap& tmB, const CUtensorMap& tmB2, const LmheadArgs& args,
                               int num_ctas, cudaStream_t stream);
cudaError_t lmhead_pair_prepare();

}  // namespace ais
