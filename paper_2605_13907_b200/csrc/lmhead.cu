// LM-head tensor-core passes for sm_100a: TMA-fed tcgen05.mma with accumulators in tensor memory and
// fused epilogues (streaming log-sum-exp + target pick, softmax-minus-onehot scratch, dH scaling).
//
// One persistent CTA of three warpgroups per SM.  Warp 0 issues TMA tile loads, warp 1 issues the MMAs
// (warps 2, 3 idle), warps 4..11 are the epilogue: warp w owns TMEM lanes 32*(w%4) .. +31 (one row per
// thread) and column half (w-4)/4 of the 256-column accumulator.  The dH pass gives a CTA two row tiles
// (256 rows, both accumulators) so that every W slice it loads is used twice; its contraction over the
// vocabulary is so long that the one epilogue per unit need not overlap anything.  Two 256-column accumulators
// alternate so that the epilogue of one tile overlaps the MMAs of the next.  The microscaling modes add a fourth
// warpgroup (warps 12..15) that moves each stage's block scales from shared to tensor memory, where the
// block-scaled MMA reads them; their scale columns leave room for one accumulator only.  The rollout pass with
// fp32 per-block scales has a kernel of its own (lmhead_fp8.cu).
//
// The producer and the MMA issuer are one elected thread each (elect.sync; a branch on lane == 0 issues copies and MMAs 10% to 20%
// slower).  Where a stage takes four copies for 512 clocks of MMAs that was the bound: 9,216 rows, d = 4096, 65,536 columns,
// microscaling FP8 2.14 -> 1.91 ms, FP4 1.08 -> 0.91; trainer pass of 613 rows 605 -> 596 us.  What is left there is the MMAs and the
// operand copies together (FP8 1.79 ms; 1.34 without the copies, 1.42 with half the MMAs).
#include <type_traits>

#include "lmhead_common.cuh"
#include "../../include/ais.h"

namespace ais {

namespace {

constexpr int threads_of(int mode) { return (mode == kFwdMx || mode == kFwdMx4) ? kMxThreads : kThreads; }

template <int MODE>
__global__ void __launch_bounds__(threads_of(MODE), 1)
lmhead_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
              const __grid_constant__ CUtensorMap tmB2, const LmheadArgs a) {
    extern __shared__ uint8_t smem_raw[];
    // 1024-byte aligned start, as an offset from the array so that the compiler still knows the address space
    uint8_t* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    uint8_t* stage_base = smem;
    uint8_t* mx_scale_base = smem + kStages * kStageBytes;      // microscaling pass: one scale triple per stage
    uint64_t* bars = reinterpret_cast<uint64_t*>(mx_scale_base + kStages * kMxStageScaleBytes);
    uint64_t* full = bars;                       // [kStages]   TMA -> MMA
    uint64_t* empty = full + kStages;            // [kStages]   MMA -> TMA
    uint64_t* tfull = empty + kStages;           // [2]         MMA -> epilogue
    uint64_t* tempty = tfull + 2;                // [2]         epilogue -> MMA
    uint64_t* done = tempty + 2;                 // [1]         all MMAs of this CTA have completed
    uint64_t* sfull = done + 1;                  // [kStages]   scale warps -> MMA (microscaling passes)
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + kNumBarriers);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
    volatile uint32_t* issued_slot = tmem_slot + 2;     // stage fills the producer has requested (written when it leaves its loop)

    constexpr int BASE = base_mode(MODE);                                       // what is computed, whatever W's layout
    constexpr bool B_MN = b_mn_major(MODE);                                     // B tile arrives as four 64-column boxes
    constexpr bool TWO_ACC = BASE == kBwdDh;                                    // two 128-row tiles per CTA, one B slice
    constexpr int STG = TWO_ACC ? kDhStages : kStages;                          // depth of the stage ring
    constexpr int STG_BYTES = TWO_ACC ? kDhStageBytes : kStageBytes;
    constexpr int A_BYTES = TWO_ACC ? 2 * kAStageBytes : kAStageBytes;
    constexpr bool MX = (MODE == kFwdMx || MODE == kFwdMx4);                    // block scales live in tensor memory
    constexpr bool FP4 = (MODE == kFwdMx4);                                     // 256 packed 4-bit elements per stage
    constexpr int MX_SCALE_BYTES = FP4 ? 6 * kMxChunkBytes : 3 * kMxChunkBytes;
    constexpr int NBUF = (TWO_ACC || MX) ? 1 : 2;                               // accumulator sets that alternate
    constexpr uint32_t kMxScaleCol = 256;                                       // MX: scale columns after the accumulator,
    constexpr uint32_t kMxSetCols = 32;                                         // one set of 32 per stage of the ring
    constexpr int kScaleWarp0 = 12;                                             // MX: first of the four scale warps
    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    const int num_units = count_units<BASE>(a);
    const bool gated = BASE == kBwdP && a.gate != nullptr;
    if (gated) {
        enter_pass(a);
        if (__ldcg(a.gate) == 0u) return;                 // no row tile needs this pass
    }

    if (threadIdx.x == 0) {
        for (int i = 0; i < kStages; ++i) { mbar_init(&full[i], 1); mbar_init(&empty[i], 1); mbar_init(&sfull[i], 4); }
        for (int i = 0; i < 2; ++i) { mbar_init(&tfull[i], 1); mbar_init(&tempty[i], kEpiWarps); }
        mbar_init(done, 1);
        *abort_flag = 0;
        *issued_slot = 0;
        fence_barrier_init();
        tma_prefetch_desc(&tmA);
        tma_prefetch_desc(&tmB);
    }
    if (warp == 1) {
        tmem_alloc(tmem_slot, 512);
        tmem_relinquish();
    }
    if (!gated) enter_pass(a);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;

    // Microscaling pass: its one accumulator is read into registers in one go so that it can go back to the MMA
    // issuer at once; the other warps hand the registers for that to the epilogue (512 x 128 = 256 x 32 + 256 x 224).
    if (warp == 0) {
        // ------------------------------------------------------------------ TMA producer
        if (MX) reg_dealloc<32>();
        if (elect_one()) {
            Pipe st(STG);
            uint32_t issued = 0;
            bool ok = true;
            Pacer pacer(a.pace, a.pace_per_unit);
            int n = 0;                                          // ordinal of this CTA's unit (its wave)
            for (int u = blockIdx.x; u < num_units && ok; u += gridDim.x, ++n) {
                const Unit w = decode_unit<BASE>(a, u);
                if (!unit_active<BASE>(a, w)) {
                    if (pacer.ring) pacer.top_up(n, 0);
                    continue;
                }
                int fills = 0;                                  // stage fills of this unit so far
                for (int t = w.t0; t < w.t1 && ok; ++t) {
                    for (int ks = w.k0; ks < w.k1; ++ks, ++fills) {
                        if (pacer.ring && fills % kPaceFills == 0) pacer.announce(n, fills / kPaceFills);
                        if (pacer.ring && fills % kPaceFills == kPaceSettle) pacer.settle();
                        if (!mbar_wait(&empty[st.idx], st.phase ^ 1u, abort_flag, a.wait_cycles)) { ok = false; break; }
                        uint8_t* sA = stage_base + st.idx * STG_BYTES;
                        uint8_t* sB = sA + A_BYTES;
                        mbar_expect_tx(&full[st.idx], MX ? STG_BYTES + MX_SCALE_BYTES : STG_BYTES);
                        const int kelem = (MODE == kFwdFp8T || MX) ? ks * 128 : ks * 64;
                        if (MX) {
                            // the stage's scales (see the layout at ais_quantize_mxfp8): A's chunk(s) of this row tile, then the
                            // adjacent chunk pair(s) of B's 256 rows; with FP4 a stage spans two chunk columns
                            uint8_t* sS = mx_scale_base + st.idx * kMxStageScaleBytes;
                            constexpr int KC = FP4 ? 2 : 1;                    // chunk columns per stage
                            const int64_t k4 = static_cast<int64_t>(ks) * KC;
#pragma unroll
                            for (int c = 0; c < KC; ++c)
                                bulk_load(sS + c * kMxChunkBytes,
                                          a.sf_a + (static_cast<int64_t>(w.rt >> 1) * a.nk4 + k4 + c) * (2 * kMxChunkBytes) +
                                              (w.rt & 1) * kMxChunkBytes,
                                          kMxChunkBytes, &full[st.idx]);
                            bulk_load(sS + KC * kMxChunkBytes, a.sf_b + (static_cast<int64_t>(t) * a.nk4 + k4) * (2 * kMxChunkBytes),
                                      KC * 2 * kMxChunkBytes, &full[st.idx]);
                        }
                        if (BASE == kBwdDh) {
                            tma_load_2d(sA, &tmA, &full[st.idx], kelem, w.rt * kDhRows);
                            tma_load_2d(sA + kAStageBytes, &tmA, &full[st.idx], kelem, w.rt * kDhRows + kBM);
                        } else {
                            tma_load_2d(sA, &tmA, &full[st.idx], kelem, w.rt * kBM);
                        }
                        if (B_MN) {
                            // B is stored with the output column as the contiguous axis (W[v, n] in the dH pass, W[k, v] in
                            // the forward passes over a [d, V] head): four blocks of 64 columns, one
                            // after the other in shared memory.  One copy for the four: with a copy each the forward pass over a
                            // [d, V] head took 14.2 Mcycles for 9,217 rows, 11.8 now (as much as the other layout).  The last,
                            // partial tile of such a head keeps single boxes, which end at V.
                            if (MODE == kBwdDh || t < a.block_tiles) {
                                tma_load_3d(sB, &tmB, &full[st.idx], 0, kelem, t * (kBN / 64));
                            } else {
#pragma unroll
                                for (int j = 0; j < 4; ++j)
                                    tma_load_2d(sB + j * (kBStageBytes / 4), &tmB2, &full[st.idx], t * kBN + j * 64, kelem);
                            }
                        } else {
                            tma_load_2d(sB, &tmB, &full[st.idx], kelem, t * kBN);
                        }
                        ++issued;
                        st.advance();
                    }
                }
                if (pacer.ring) pacer.top_up(n, (fills + kPaceFills - 1) / kPaceFills);
            }
            if (pacer.ring)                                     // units of the last wave that this CTA does not have
                for (const int waves = (num_units + gridDim.x - 1) / gridDim.x; n < waves; ++n) pacer.top_up(n, 0);
            *issued_slot = issued;
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------------ MMA issuer
        if (MX) reg_dealloc<32>();
        if (elect_one()) {
            constexpr uint32_t idesc =
                (MODE == kFwdFp8T || MX) ? make_idesc(kFmtE4M3, kFmtE4M3, kBM, kBN, 0, 0)
                                  : make_idesc(kFmtBF16, kFmtBF16, kBM, kBN, 0, B_MN ? 1 : 0);
            Pipe st(STG), tb(NBUF);
            bool ok = true;
            for (int u = blockIdx.x; u < num_units && ok; u += gridDim.x) {
                const Unit w = decode_unit<BASE>(a, u);
                if (!unit_active<BASE>(a, w)) continue;
                for (int t = w.t0; t < w.t1 && ok; ++t) {
                    if (!mbar_wait(&tempty[tb.idx], tb.phase ^ 1u, abort_flag, a.wait_cycles)) { ok = false; break; }
                    tc_fence_after();
                    for (int ks = w.k0; ks < w.k1; ++ks) {
                        if (!mbar_wait(&full[st.idx], st.phase, abort_flag, a.wait_cycles)) { ok = false; break; }
                        tc_fence_after();
                        const uint32_t sA = smem_u32(stage_base + st.idx * STG_BYTES);
                        const uint32_t sB = sA + A_BYTES;
                        if (BASE == kBwdDh) {
                            // two row tiles share every B slice: accumulators at TMEM columns 0 and 256
#pragma unroll
                            for (int j = 0; j < 4; ++j) {
                                const uint64_t bdesc = B_MN ? smem_desc_sw128(sB + j * 2048, kBStageBytes / 4, 1024)
                                                            : smem_desc_sw128(sB + j * 32, 16, 1024);
                                const uint32_t accum = (ks > w.k0 || j > 0) ? 1u : 0u;
                                mma_f16(tmem_base, smem_desc_sw128(sA + j * 32, 16, 1024), bdesc, idesc, accum);
                                mma_f16(tmem_base + kBN, smem_desc_sw128(sA + kAStageBytes + j * 32, 16, 1024), bdesc, idesc, accum);
                            }
                        } else if (MX) {
                            // the scale warps have put this stage's scales into its column set: A's chunks first (4 columns
                            // each), then B's (4 columns per 128 rows and chunk).  One block-scaled instruction per 32 bytes
                            // of K, each with its scale id.
                            constexpr int KC = FP4 ? 2 : 1;
                            if (!mbar_wait(&sfull[st.idx], st.phase, abort_flag, a.wait_cycles)) { ok = false; break; }
                            tc_fence_after();
                            const uint32_t tsf = tmem_base + kMxScaleCol + st.idx * kMxSetCols;
#pragma unroll
                            for (int j = 0; j < 4; ++j) {
                                const uint64_t adesc = smem_desc_sw128(sA + j * 32, 16, 1024);
                                const uint64_t bdesc = smem_desc_sw128(sB + j * 32, 16, 1024);
                                const uint32_t accum = (ks > w.k0 || j > 0) ? 1u : 0u;
                                if (FP4) {
                                    // instruction j covers scale blocks 2j, 2j+1: chunk j / 2, bytes 2 (j % 2) and the next
                                    const uint32_t id = 2u * (j & 1), sel = id << 30;
                                    mma_mxf4(tmem_base, adesc, bdesc, make_idesc_mx(kBM, kBN, id, 1u), (tsf + 4 * (j >> 1)) | sel,
                                             (tsf + 4 * KC + 8 * (j >> 1)) | sel, accum);
                                } else {
                                    const uint32_t sel = static_cast<uint32_t>(j) << 30;      // byte of the scale columns
                                    mma_mxf8(tmem_base, adesc, bdesc, make_idesc_mx(kBM, kBN, j), tsf | sel, (tsf + 4) | sel, accum);
                                }
                            }
                        } else {
                            const uint32_t dcol = tmem_base + tb.idx * kBN;
#pragma unroll
                            for (int j = 0; j < 4; ++j) {
                                const uint64_t adesc = smem_desc_sw128(sA + j * 32, 16, 1024);
                                const uint64_t bdesc = B_MN ? smem_desc_sw128(sB + j * 2048, kBStageBytes / 4, 1024)
                                                            : smem_desc_sw128(sB + j * 32, 16, 1024);
                                if (MODE == kFwdFp8T) mma_f8(dcol, adesc, bdesc, idesc, (ks > w.k0 || j > 0) ? 1u : 0u);
                                else mma_f16(dcol, adesc, bdesc, idesc, (ks > w.k0 || j > 0) ? 1u : 0u);
                            }
                        }
                        tc_commit(&empty[st.idx]);
                        st.advance();
                    }
                    if (ok) {
                        tc_commit(&tfull[tb.idx]);
                        tb.advance();
                    }
                }
            }
            // everything issued has to finish before the tensor memory is given back
            tc_commit(done);
        }
    } else if (warp < 4) {
        if (MX) reg_dealloc<32>();          // the idle warps of the first warpgroup give their registers away too
    } else if (MX && warp >= kScaleWarp0) {
        // ------------------------------------------------------------------ scale warps (microscaling passes)
        // A scale chunk in shared memory is 32 rows of 16 bytes: row l holds, for each of four 32-row groups, the
        // four E8M0 bytes of the stage's K blocks.  The MMA reads scales from tensor memory, lane l of every lane
        // quarter, one 32-bit column per group: warp 12 + q copies the stage's chunks to quarter q with plain stores
        // (a tcgen05.cp from the MMA thread would queue in front of the MMAs and costs about a tenth of the pass).
        // A stage's column set is free again once its `empty` barrier has completed, which the producer waited for
        // before the loads that complete `full`.
        reg_dealloc<32>();
        constexpr int KC = FP4 ? 2 : 1;
        const uint32_t lane_addr = static_cast<uint32_t>((warp & 3) * 32) << 16;
        Pipe st(STG);
        bool ok = true;
        for (int u = blockIdx.x; u < num_units && ok; u += gridDim.x) {
            const Unit w = decode_unit<BASE>(a, u);
            if (!unit_active<BASE>(a, w)) continue;
            for (int t = w.t0; t < w.t1 && ok; ++t) {
                for (int ks = w.k0; ks < w.k1; ++ks) {
                    if (!mbar_wait_warp(&full[st.idx], st.phase, abort_flag, a.wait_cycles)) { ok = false; break; }
                    const uint4* src = reinterpret_cast<const uint4*>(mx_scale_base + st.idx * kMxStageScaleBytes) + lane;
                    const uint32_t tsf = tmem_base + lane_addr + kMxScaleCol + st.idx * kMxSetCols;
#pragma unroll
                    for (int c = 0; c < 3 * KC; ++c) tmem_st_32x32b_x4(tsf + 4 * c, src[c * (kMxChunkBytes / 16)]);
                    tmem_st_wait();
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&sfull[st.idx]);
                    st.advance();
                }
            }
        }
    } else {
        // ------------------------------------------------------------------ epilogue warps
        if (MX) reg_alloc<224>();
        const int q = warp & 3;                       // TMEM lane quarter this warp may read
        const int half = (warp - 4) >> 2;             // column half of the accumulator
        const int r_in_tile = q * 32 + lane;
        const uint32_t lane_addr = static_cast<uint32_t>(q * 32) << 16;
        Pipe tb(NBUF);
        bool ok = true;
        uint32_t flags = 0;
        for (int u = blockIdx.x; u < num_units && ok; u += gridDim.x) {
            const Unit w = decode_unit<BASE>(a, u);
            if (!unit_active<BASE>(a, w)) {
                // nothing was loaded or multiplied for this unit: write the neutral output where later passes read it
                if (BASE == kBwdDh && w.slot < 0) {
#pragma unroll
                    for (int sub = 0; sub < 2; ++sub) {
                        const int64_t lr = static_cast<int64_t>(w.rt) * kDhRows + sub * kBM + r_in_tile;
                        if (lr < a.rows) {
                            uint4* dst = reinterpret_cast<uint4*>(a.dH + (a.row0 + lr) * a.lddh + w.t0 * kBN + half * 128);
#pragma unroll
                            for (int j = 0; j < 16; ++j)
                                if (w.t0 * kBN + half * 128 + j * 8 < a.ncols) dst[j] = make_uint4(0, 0, 0, 0);
                        }
                    }
                } else if (BASE == kBwdP && !gated) {
                    const int64_t lr = static_cast<int64_t>(w.rt) * kBM + r_in_tile;
                    if (lr < a.rows) {
                        for (int t = w.t0; t < w.t1; ++t) {
                            uint4* dst = reinterpret_cast<uint4*>(a.U + lr * a.ldU + t * kBN + half * 128);
#pragma unroll
                            for (int j = 0; j < 16; ++j)
                                if (t * kBN + half * 128 + j * 8 < a.ncols) dst[j] = make_uint4(0, 0, 0, 0);
                        }
                    }
                }
                continue;       // forward passes: the rows are masked, the merge kernel never reads their partials
            }
            if (BASE == kBwdDh) {
                // one unit = 256 rows x 256 columns of dH, finished after the whole contraction over the vocabulary
                if (!mbar_wait_warp(&tfull[0], tb.phase, abort_flag, a.wait_cycles)) { ok = false; break; }
                tc_fence_after();
#pragma unroll
                for (int sub = 0; sub < 2; ++sub) {
                    const int64_t lrow2 = static_cast<int64_t>(w.rt) * kDhRows + sub * kBM + r_in_tile;
                    const bool in = lrow2 < a.rows;
                    const int64_t grow2 = a.row0 + lrow2;
                    // (the row's factor, or 1; rows with factor 0 may hold anything, so they are selected away)
                    const float rs = (a.row_scale != nullptr && in) ? a.row_scale[grow2] : 1.f;
                    const uint32_t taddr2 = tmem_base + lane_addr + sub * kBN + half * 128;
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        const int col0 = w.t0 * kBN + half * 128 + c * 32;
                        uint32_t v[32];
                        tmem_ld32(taddr2 + c * 32, v);
                        tmem_ld_wait(v);
                        if (w.slot >= 0) {
                            // one of several ranges of the contraction: the fp32 sums go to the unit's partial tile, 16 bytes
                            // per lane on consecutive addresses
                            float4* dst = reinterpret_cast<float4*>(a.part_acc + static_cast<int64_t>(w.slot) * kPartTileFloats) +
                                          (sub * (kBN / 4) + half * 32 + c * 8) * kBM + r_in_tile;
#pragma unroll
                            for (int j = 0; j < 8; ++j)
                                dst[j * kBM] = make_float4(__uint_as_float(v[4 * j]), __uint_as_float(v[4 * j + 1]),
                                                           __uint_as_float(v[4 * j + 2]), __uint_as_float(v[4 * j + 3]));
                        } else if (in && col0 < a.ncols) {
                            uint32_t pk[16];
#pragma unroll
                            for (int i = 0; i < 32; i += 2) {
                                pk[i >> 1] = rs != 0.f ? pack_bf16(__uint_as_float(v[i]) * rs, __uint_as_float(v[i + 1]) * rs) : 0u;
                            }
                            uint4* dst = reinterpret_cast<uint4*>(a.dH + grow2 * a.lddh + col0);
#pragma unroll
                            for (int j = 0; j < 4; ++j)
                                if (col0 + j * 8 < a.ncols) dst[j] = make_uint4(pk[4 * j], pk[4 * j + 1], pk[4 * j + 2], pk[4 * j + 3]);
                        }
                    }
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&tempty[0]);
                tb.advance();
                continue;
            }
            RowState r = begin_row<MODE>(a, static_cast<int64_t>(w.rt) * kBM + r_in_tile, flags);
            const bool store = r.in && (BASE == kBwdP || r.lrow < a.keep_rows);
            const float tscale = (MODE == kFwdFp8T) ? (*a.scale_a) * (*a.scale_b) : 1.f;
            for (int t = w.t0; t < w.t1 && ok; ++t) {
                const int col_base = t * kBN + half * 128;    // first output column of this thread's half
                {
                    if (!mbar_wait_warp(&tfull[tb.idx], tb.phase, abort_flag, a.wait_cycles)) { ok = false; break; }
                    tc_fence_after();
                }

                const uint32_t taddr = tmem_base + lane_addr + tb.idx * kBN + half * 128;
                uint32_t vv[MX ? 4 : 1][32];
                if (MX) {
                    // the thread's 128 columns at once, then the accumulator is free for the next tile's MMAs
#pragma unroll
                    for (int c = 0; c < 4; ++c) tmem_ld32(taddr + c * 32, vv[MX ? c : 0]);
#pragma unroll
                    for (int c = 0; c < 4; ++c) tmem_ld_wait(vv[MX ? c : 0]);
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&tempty[tb.idx]);
                }
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    const int col0 = col_base + c * 32;
                    float x[32];
                    if (MX) {
#pragma unroll
                        for (int i = 0; i < 32; ++i) x[i] = __uint_as_float(vv[MX ? c : 0][i]);
                    } else {
                        uint32_t v[32];
                        tmem_ld32(taddr + c * 32, v);
                        tmem_ld_wait(v);
#pragma unroll
                        for (int i = 0; i < 32; ++i) x[i] = __uint_as_float(v[i]);
                        if (MODE == kFwdFp8T) {
#pragma unroll
                            for (int i = 0; i < 32; ++i) x[i] *= tscale;
                        }
                    }
                    row_slice<MODE>(a, r, col0, x, store);
                }
                if (!MX) {
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&tempty[tb.idx]);
                }
                tb.advance();
            }
            if (ok && BASE != kBwdP) end_row(a, r, w.part * 2 + half);
        }
        if (flags && a.status) atomicOr(a.status, flags);
    }

    // ---------------------------------------------------------------------- teardown
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        if (lane == 0) mbar_wait_drain(done, 0);   // immediate unless the CTA is giving up early
        __syncwarp();
        tc_fence_after();
        tmem_dealloc(tmem_base, 512);
    }
    if (threadIdx.x == 0 && *abort_flag) {
        // some role gave up on a wait: let the producer's copies still in flight land before the CTA exits
        drain_stage_copies(full, *issued_slot, STG);
        if (a.status) atomicOr(a.status, AIS_FLAG_TIMEOUT);
    }
    leave_pass(a);
}

// dH rows of the units whose contraction was split: the partial tiles are added in the order of their ranges and rounded
// to bf16 once.  A thread owns one row and 16 columns (32 bytes of dH); the partial tiles are read 16 bytes per lane on
// consecutive addresses.  The pass is a plain sweep of ksplit x 256 KB per tile, mostly still in L2 (64 tiles x 9 ranges:
// 151 MB).  Tiles without work have no partial sums and become zeros.
__global__ void __launch_bounds__(256) dh_reduce_kernel(const LmheadArgs a) {
    pdl_enter();
    const int tail = a.n_row_tiles * a.n_col_tiles - a.split_from;
    const int i = blockIdx.x * 256 + threadIdx.x;
    const int row = i & (kBM - 1), cg = (i >> 7) & 15, sub = (i >> 11) & 1, tile = i >> 12;
    Unit w;
    w.rt = (a.split_from + tile) / a.n_col_tiles;
    const int col0 = ((a.split_from + tile) % a.n_col_tiles) * kBN + cg * 16;
    const int64_t lr = static_cast<int64_t>(w.rt) * kDhRows + sub * kBM + row;
    if (lr >= a.rows || col0 >= a.ncols) return;
    float4 acc[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[j] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (unit_active<kBwdDh>(a, w)) {
        const float4* src = reinterpret_cast<const float4*>(a.part_acc + static_cast<int64_t>(tile) * kPartTileFloats) +
                            (sub * (kBN / 4) + cg * 4) * kBM + row;
        const int64_t step = static_cast<int64_t>(tail) * (kPartTileFloats / 4);
#pragma unroll 2
        for (int k = 0; k < a.ksplit; ++k) {
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const float4 v = __ldcs(src + k * step + j * kBM);
                acc[j].x += v.x; acc[j].y += v.y; acc[j].z += v.z; acc[j].w += v.w;
            }
        }
    }
    if (a.row_scale != nullptr) {
        const float rs = a.row_scale[a.row0 + lr];
#pragma unroll
        for (int j = 0; j < 4; ++j)
            acc[j] = rs != 0.f ? make_float4(acc[j].x * rs, acc[j].y * rs, acc[j].z * rs, acc[j].w * rs) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    uint4* dst = reinterpret_cast<uint4*>(a.dH + (a.row0 + lr) * a.lddh + col0);
#pragma unroll
    for (int j = 0; j < 2; ++j)
        dst[j] = make_uint4(pack_bf16(acc[2 * j].x, acc[2 * j].y), pack_bf16(acc[2 * j].z, acc[2 * j].w),
                            pack_bf16(acc[2 * j + 1].x, acc[2 * j + 1].y), pack_bf16(acc[2 * j + 1].z, acc[2 * j + 1].w));
}

}  // namespace

cudaError_t launch_dh_reduce(const LmheadArgs& args, cudaStream_t stream) {
    const int tail = args.n_row_tiles * args.n_col_tiles - args.split_from;
    return launch_pdl(dh_reduce_kernel, tail * 16, 256, 0, stream, args);
}

template <int MODE>
static cudaError_t launch_mode(const CUtensorMap& tmA, const CUtensorMap& tmB, const CUtensorMap& tmB2, const LmheadArgs& args, int num_ctas,
                               cudaStream_t stream) {
    return launch_pdl(lmhead_kernel<MODE>, num_ctas, threads_of(MODE), kSmemBytes, stream, tmA, tmB, tmB2, args);
}

cudaError_t launch_lmhead(int mode, const CUtensorMap& tmA, const CUtensorMap& tmB, const CUtensorMap& tmSA,
                          const CUtensorMap& tmSB, const LmheadArgs& args, int num_ctas, cudaStream_t stream) {
    switch (mode) {
        case kFwdBf16: return launch_mode<kFwdBf16>(tmA, tmB, tmSA, args, num_ctas, stream);
        case kFwdFp8:  return launch_lmhead_fp8_block(tmA, tmB, tmSA, tmSB, args, num_ctas, stream);
        case kBwdP:    return launch_mode<kBwdP>(tmA, tmB, tmSA, args, num_ctas, stream);
        case kBwdDh:   return launch_mode<kBwdDh>(tmA, tmB, tmSA, args, num_ctas, stream);
        case kFwdFp8T: return launch_mode<kFwdFp8T>(tmA, tmB, tmSA, args, num_ctas, stream);
        case kFwdMx:   return launch_mode<kFwdMx>(tmA, tmB, tmSA, args, num_ctas, stream);
        case kFwdMx4:  return launch_mode<kFwdMx4>(tmA, tmB, tmSA, args, num_ctas, stream);
        case kFwdBf16Dv: return launch_mode<kFwdBf16Dv>(tmA, tmB, tmSA, args, num_ctas, stream);
        case kBwdPDv:    return launch_mode<kBwdPDv>(tmA, tmB, tmSA, args, num_ctas, stream);
        case kBwdDhDv:   return launch_mode<kBwdDhDv>(tmA, tmB, tmSA, args, num_ctas, stream);
        case kFwdKeep:   return launch_mode<kFwdKeep>(tmA, tmB, tmSA, args, num_ctas, stream);
        case kFwdKeepDv: return launch_mode<kFwdKeepDv>(tmA, tmB, tmSA, args, num_ctas, stream);
    }
    return cudaErrorInvalidValue;
}

template <int MODE>
static cudaError_t prepare_mode() {
    return cudaFuncSetAttribute(lmhead_kernel<MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes);
}

cudaError_t lmhead_prepare() {
    const cudaError_t all[] = {lmhead_fp8_block_prepare(), lmhead_pair_prepare(), prepare_mode<kFwdBf16>(), prepare_mode<kBwdP>(), prepare_mode<kBwdDh>(),
                               prepare_mode<kFwdFp8T>(), prepare_mode<kFwdMx>(), prepare_mode<kFwdMx4>(),
                               prepare_mode<kFwdBf16Dv>(), prepare_mode<kBwdPDv>(), prepare_mode<kBwdDhDv>(), prepare_mode<kFwdKeep>(),
                               prepare_mode<kFwdKeepDv>()};
    for (const cudaError_t e : all)
        if (e != cudaSuccess) return e;
    return cudaSuccess;
}

}  // namespace ais
