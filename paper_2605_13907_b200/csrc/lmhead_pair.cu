// Forward, recompute and dW passes with two row tiles per CTA: 256 rows x 256 columns, both accumulators of tensor memory, every
// slice of W that a CTA fetches used for two row tiles.  Per 64 K-elements a stage of 64 KB feeds 1,024 clocks of MMAs where
// the one-row-tile kernel (lmhead.cu) needs 48 KB for 512, which is more than L2 delivers to all SMs at that rate: its main
// loop runs at 82% of the tensor rate.  The price is that no third accumulator is left for the next tile while the epilogue
// reads these two.  So the order of the MMAs is skewed at the ends of a tile: the first row tile gets its last two stages
// before the second one, and the next tile's first stages (as many as the ring holds) go to the first row tile alone.  The
// epilogue of an accumulator takes all of it into registers at once (128 per thread) and hands it back before the arithmetic,
// so each of the two is drained while the tensor core works on the other.
// Measured against the one-row-tile kernel (sustained, under the power cap): 9,217 rows at d = 4096, V = 151936 8.57 -> 8.22 ms,
// 20,000 rows at d = 5120, V = 129112 21.6 -> 19.1 ms, 1,024 rows 1.08 -> 1.01 ms.  Without the epilogue's arithmetic it would
// take 2% less, so the skew hides nearly all of it (head 3 / tail 2: 8.01 ms, no tail 8.04, head 1 8.12, head 2 8.13); what is
// left is the power cap.  Batches of few row tiles stay with the other kernel (plan_pass): a CTA per pair halves the units.
//
// The dW pass (256 x 256 of dW per unit, contracted over the rows of the launch) has the same shape with both operands MN-major,
// and an epilogue per 64-row K steps of the batch: at 1,500 rows every 24 stages.  With the epilogue behind the MMAs of both
// accumulators it took 2,540 us for 1,500 rows, 4,275 us for 4,000 and 8.61 ms for 9,217 (d = 4096, V = 151936); drained in turn
// 2,260, 3,950 and 8.32 ms.
//
// Roles as in lmhead.cu: warp 0 copies, warp 1 issues the MMAs, warps 4..11 are the epilogue (lane quarter w % 4, column half
// (w - 4) / 4 of both accumulators: two rows per thread).  The first warpgroup hands registers to the other two
// (384 threads x 168 registers at launch = 128 x 40 + 256 x 232).
#include "lmhead_common.cuh"
#include "../../include/ais.h"

namespace ais {

namespace {

constexpr int kPairStages = kDhStages;
constexpr int kPairStageBytes = kDhStageBytes;
constexpr int kPairBars = 2 * kPairStages + 4 + 1;
constexpr int kPairSmem = 1024 + kPairStages * kPairStageBytes + kPairBars * 8 + 64;
constexpr int kPairTail = 2;                     // stages at the end of a tile that the first row tile gets ahead of the second

// 32 consecutive columns of one row of dW.
__device__ __forceinline__ void store_dw(const LmheadArgs& a, int64_t row, int col0, const uint32_t (&v)[32]) {
    float4* dst = reinterpret_cast<float4*>(a.dW + row * a.lddw + col0);
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        if (col0 + j * 4 >= a.ncols) continue;
        float4 o = make_float4(__uint_as_float(v[4 * j]), __uint_as_float(v[4 * j + 1]), __uint_as_float(v[4 * j + 2]), __uint_as_float(v[4 * j + 3]));
        if (a.dw_accumulate) {
            const float4 old = dst[j];
            o.x += old.x; o.y += old.y; o.z += old.z; o.w += old.w;
        }
        dst[j] = o;
    }
}

template <int MODE>
__global__ void __launch_bounds__(kThreads, 1)
lmhead_pair_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                   const __grid_constant__ CUtensorMap tmB2, const LmheadArgs a) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    uint8_t* stage_base = smem;
    uint64_t* full = reinterpret_cast<uint64_t*>(smem + kPairStages * kPairStageBytes);    // [stages] TMA -> MMA
    uint64_t* empty = full + kPairStages;        // [stages]   MMA -> TMA
    uint64_t* tfull = empty + kPairStages;       // [2]        MMA -> epilogue: accumulator complete
    uint64_t* tempty = tfull + 2;                // [2]        epilogue -> MMA: accumulator in registers
    uint64_t* done = tempty + 2;                 // [1]        all MMAs of this CTA have completed
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(done + 1);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
    volatile uint32_t* issued_slot = tmem_slot + 2;     // stage fills the producer has requested (written when it leaves its loop)

    constexpr int BASE = base_mode(MODE);
    constexpr bool B_MN = b_mn_major(MODE);
    constexpr bool FP8 = MODE == kFwdFp8T;
    constexpr bool DW = MODE == kBwdDw;
    constexpr int UNIT = DW ? kBwdDw : kFwdFp8;  // units of two row tiles, for decode_unit / unit_active
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int num_units = count_units<UNIT>(a);
    const bool gated = BASE == kBwdP && a.gate != nullptr;
    if (gated) {
        enter_pass(a);
        if (__ldcg(a.gate) == 0u) return;                 // no row tile needs this pass
    }

    if (threadIdx.x == 0) {
        for (int i = 0; i < kPairStages; ++i) { mbar_init(&full[i], 1); mbar_init(&empty[i], 1); }
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

    if (warp < 4) {
        reg_dealloc<40>();
        if (warp == 0 && elect_one()) {
            // -------------------------------------------------------------- TMA producer
            Pipe st(kPairStages);
            uint32_t issued = 0;
            bool ok = true;
            Pacer pacer(a.pace, a.pace_per_unit);
            int n = 0;                                          // ordinal of this CTA's unit (its wave)
            for (int u = blockIdx.x; u < num_units && ok; u += gridDim.x, ++n) {
                const Unit w = decode_unit<UNIT>(a, u);
                if (!unit_active<UNIT>(a, w)) {
                    if (pacer.ring) pacer.top_up(n, 0);
                    continue;
                }
                int fills = 0;                                  // stage fills of this unit so far
                for (int t = w.t0; t < w.t1 && ok; ++t) {
                    for (int ks = 0; ks < a.ksteps; ++ks, ++fills) {
                        if (pacer.ring && fills % kPaceFills == 0) pacer.announce(n, fills / kPaceFills);
                        if (pacer.ring && fills % kPaceFills == kPaceSettle) pacer.settle();
                        if (!mbar_wait(&empty[st.idx], st.phase ^ 1u, abort_flag, a.wait_cycles)) { ok = false; break; }
                        uint8_t* sA = stage_base + st.idx * kPairStageBytes;
                        uint8_t* sB = sA + 2 * kAStageBytes;
                        mbar_expect_tx(&full[st.idx], kPairStageBytes);
                        const int kelem = FP8 ? ks * 128 : ks * 64;
                        // dW: the output row is the contiguous axis of A (U[t, v]), four 64-wide blocks of 64 rows t in one copy;
                        // otherwise one box of 256 rows
                        if (DW) tma_load_3d(sA, &tmA, &full[st.idx], 0, kelem, w.rt * (kPairRows / 64));
                        else tma_load_2d(sA, &tmA, &full[st.idx], kelem, w.rt * kPairRows);
                        // MN-major B (H[t, n] of dW, a [d, V] head): four blocks of 64 columns in one copy, except in the last,
                        // partial tile of such a head, whose single boxes end at V.  With a copy for each block the forward pass
                        // over a [d, V] head took 14.2 Mcycles for 9,217 rows instead of 11.8.
                        if (!B_MN) {
                            tma_load_2d(sB, &tmB, &full[st.idx], kelem, t * kBN);
                        } else if (DW || t < a.block_tiles) {
                            tma_load_3d(sB, &tmB, &full[st.idx], 0, kelem, t * (kBN / 64));
                        } else {
#pragma unroll
                            for (int j = 0; j < 4; ++j)
                                tma_load_2d(sB + j * (kBStageBytes / 4), &tmB2, &full[st.idx], t * kBN + j * 64, kelem);
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
        } else if (warp == 1 && elect_one()) {
            // -------------------------------------------------------------- MMA issuer
            constexpr uint32_t idesc = FP8 ? make_idesc(kFmtE4M3, kFmtE4M3, kBM, kBN, 0, 0)
                                           : make_idesc(kFmtBF16, kFmtBF16, kBM, kBN, DW ? 1 : 0, B_MN ? 1 : 0);
            const int K = a.ksteps;
            const int head = K < kPairStages ? K : kPairStages;                 // stages that the first row tile gets alone
            const int tail = K - head < kPairTail ? K - head : kPairTail;
            uint32_t base = 0;                                                  // stages of the tiles before this one
            uint32_t tphase[2] = {0, 0};
            bool ok = true;
            auto wait_stage = [&](int k) {
                const uint32_t n = base + k;
                if (!mbar_wait(&full[n % kPairStages], (n / kPairStages) & 1u, abort_flag, a.wait_cycles)) ok = false;
                tc_fence_after();
                return ok;
            };
            auto wait_acc = [&](int i) {
                if (!mbar_wait(&tempty[i], tphase[i] ^ 1u, abort_flag, a.wait_cycles)) ok = false;
                tc_fence_after();
                tphase[i] ^= 1u;
                return ok;
            };
            auto mma = [&](int k, int i) {                                      // stage k, row tile i
                const uint32_t sA = smem_u32(stage_base + ((base + k) % kPairStages) * kPairStageBytes);
                const uint32_t sB = sA + 2 * kAStageBytes;
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    // MN-major operands: 16 K rows of 128 bytes per instruction, 64-wide blocks of the output axis 8 KB apart
                    const uint64_t adesc = DW ? smem_desc_sw128(sA + i * kAStageBytes + j * 2048, kAStageBytes / 2, 1024)
                                              : smem_desc_sw128(sA + i * kAStageBytes + j * 32, 16, 1024);
                    const uint64_t bdesc = B_MN ? smem_desc_sw128(sB + j * 2048, kBStageBytes / 4, 1024) : smem_desc_sw128(sB + j * 32, 16, 1024);
                    if (FP8) mma_f8(tmem_base + i * kBN, adesc, bdesc, idesc, (k > 0 || j > 0) ? 1u : 0u);
                    else mma_f16(tmem_base + i * kBN, adesc, bdesc, idesc, (k > 0 || j > 0) ? 1u : 0u);
                }
            };
            auto release = [&](int k) { tc_commit(&empty[(base + k) % kPairStages]); };
            for (int u = blockIdx.x; u < num_units && ok; u += gridDim.x) {
                const Unit w = decode_unit<UNIT>(a, u);
                if (!unit_active<UNIT>(a, w)) continue;
                const bool two = second_tile_active(a, w);
                for (int t = w.t0; t < w.t1 && ok; ++t, base += K) {
                    if (!wait_acc(0)) break;
                    for (int k = 0; k < head && ok; ++k)
                        if (wait_stage(k)) {
                            mma(k, 0);
                            if (!two) release(k);
                        }
                    if (!ok) break;
                    if (K == head) tc_commit(&tfull[0]);
                    if (two) {
                        if (!wait_acc(1)) break;
                        for (int k = 0; k < head; ++k) {
                            mma(k, 1);
                            release(k);
                        }
                    }
                    for (int k = head; k < K - tail && ok; ++k)
                        if (wait_stage(k)) {
                            mma(k, 0);
                            if (two) mma(k, 1);
                            release(k);
                        }
                    for (int k = K - tail; k < K && ok; ++k)
                        if (wait_stage(k)) {
                            mma(k, 0);
                            if (!two) release(k);
                        }
                    if (!ok) break;
                    if (K > head) tc_commit(&tfull[0]);
                    if (two) {
                        for (int k = K - tail; k < K; ++k) {
                            mma(k, 1);
                            release(k);
                        }
                        tc_commit(&tfull[1]);
                    }
                }
            }
            // everything issued has to finish before the tensor memory is given back
            tc_commit(done);
        }
    } else {
        // ------------------------------------------------------------------ epilogue warps
        reg_alloc<232>();
        const int q = warp & 3;                       // TMEM lane quarter this warp may read
        const int half = (warp - 4) >> 2;             // column half of the accumulators
        const uint32_t lane_addr = static_cast<uint32_t>(q * 32) << 16;
        const float tscale = FP8 ? (*a.scale_a) * (*a.scale_b) : 1.f;
        uint32_t tphase[2] = {0, 0};
        bool ok = true;
        uint32_t flags = 0;
        for (int u = blockIdx.x; u < num_units && ok; u += gridDim.x) {
            const Unit w = decode_unit<UNIT>(a, u);
            const int64_t lrow0 = static_cast<int64_t>(w.rt) * kPairRows + q * 32 + lane;
            if (!unit_active<UNIT>(a, w)) {
                // nothing was loaded or multiplied for this unit: the recompute pass writes zeros where the dH pass reads;
                // forward passes: the rows are masked, the merge kernel never reads their partials
                if (BASE == kBwdP && !gated)
                    for (int i = 0; i < 2; ++i)
                        if (lrow0 + i * kBM < a.rows)
                            for (int t = w.t0; t < w.t1; ++t) {
                                uint4* dst = reinterpret_cast<uint4*>(a.U + (lrow0 + i * kBM) * a.ldU + t * kBN + half * 128);
#pragma unroll
                                for (int j = 0; j < 16; ++j)
                                    if (t * kBN + half * 128 + j * 8 < a.ncols) dst[j] = make_uint4(0, 0, 0, 0);
                            }
                continue;
            }
            const bool two = second_tile_active(a, w);
            RowState r[2];
            bool store[2];
#pragma unroll
            for (int i = 0; i < 2 && !DW; ++i) {
                r[i] = begin_row<MODE>(a, lrow0 + i * kBM, flags);
                // a gated pass leaves the rows of a tile alone that was not marked, even beside one that was
                const bool mine = !gated || (a.tile_active[a.row0 / kBM + 2 * static_cast<int64_t>(w.rt) + i * (r[i].in ? 1 : 0)] != 0);
                store[i] = r[i].in && (BASE == kBwdP ? mine : r[i].lrow < a.keep_rows);
            }
            for (int t = w.t0; t < w.t1 && ok; ++t) {
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    const int col_base = t * kBN + half * 128;     // first column of this thread's half
                    if (i == 1 && !two) {
                        // the second row tile has no work: rows without gradient become zeros, nothing else is read
                        if (BASE == kBwdP && store[1]) {
#pragma unroll
                            for (int c = 0; c < 4; ++c) {
                                float x[32];
#pragma unroll
                                for (int k = 0; k < 32; ++k) x[k] = 0.f;
                                row_slice<MODE>(a, r[1], col_base + c * 32, x, true);
                            }
                        }
                        continue;
                    }
                    if (!mbar_wait_warp(&tfull[i], tphase[i], abort_flag, a.wait_cycles)) { ok = false; break; }
                    tc_fence_after();
                    tphase[i] ^= 1u;
                    uint32_t v[4][32];
                    const uint32_t taddr = tmem_base + lane_addr + i * kBN + half * 128;
#pragma unroll
                    for (int c = 0; c < 4; ++c) tmem_ld32(taddr + c * 32, v[c]);
#pragma unroll
                    for (int c = 0; c < 4; ++c) tmem_ld_wait(v[c]);
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&tempty[i]);
                    if (DW) {
                        const int64_t row = lrow0 + i * kBM;
                        if (row < a.rows) {
#pragma unroll
                            for (int c = 0; c < 4; ++c)
                                store_dw(a, row, col_base + c * 32, v[c]);
                        }
                        continue;
                    }
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        float x[32];
#pragma unroll
                        for (int k = 0; k < 32; ++k) x[k] = FP8 ? __uint_as_float(v[c][k]) * tscale : __uint_as_float(v[c][k]);
                        row_slice<MODE>(a, r[i], col_base + c * 32, x, store[i]);
                    }
                }
            }
            if (ok && BASE != kBwdP && !DW) {
                end_row(a, r[0], w.part * 2 + half);
                end_row(a, r[1], w.part * 2 + half);
            }
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
        drain_stage_copies(full, *issued_slot, kPairStages);
        if (a.status) atomicOr(a.status, AIS_FLAG_TIMEOUT);
    }
    leave_pass(a);
}

template <int MODE>
cudaError_t launch(const CUtensorMap& tmA, const CUtensorMap& tmB, const CUtensorMap& tmB2, const LmheadArgs& args, int num_ctas, cudaStream_t stream) {
    return launch_pdl(lmhead_pair_kernel<MODE>, num_ctas, kThreads, kPairSmem, stream, tmA, tmB, tmB2, args);
}
template <int MODE>
cudaError_t prepare() {
    return cudaFuncSetAttribute(lmhead_pair_kernel<MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, kPairSmem);
}

}  // namespace

cudaError_t launch_lmhead_pair(int mode, const CUtensorMap& tmA, const CUtensorMap& tmB, const CUtensorMap& tmB2, const LmheadArgs& args,
                               int num_ctas, cudaStream_t stream) {
    switch (mode) {
        case kFwdBf16:   return launch<kFwdBf16>(tmA, tmB, tmB2, args, num_ctas, stream);
        case kFwdBf16Dv: return launch<kFwdBf16Dv>(tmA, tmB, tmB2, args, num_ctas, stream);
        case kFwdKeep:   return launch<kFwdKeep>(tmA, tmB, tmB2, args, num_ctas, stream);
        case kFwdKeepDv: return launch<kFwdKeepDv>(tmA, tmB, tmB2, args, num_ctas, stream);
        case kBwdP:      return launch<kBwdP>(tmA, tmB, tmB2, args, num_ctas, stream);
        case kBwdPDv:    return launch<kBwdPDv>(tmA, tmB, tmB2, args, num_ctas, stream);
        case kFwdFp8T:   return launch<kFwdFp8T>(tmA, tmB, tmB2, args, num_ctas, stream);
        case kBwdDw:     return launch<kBwdDw>(tmA, tmB, tmB2, args, num_ctas, stream);
    }
    return cudaErrorInvalidValue;
}

cudaError_t lmhead_pair_prepare() {
    const cudaError_t all[] = {prepare<kFwdBf16>(), prepare<kFwdBf16Dv>(), prepare<kFwdKeep>(), prepare<kFwdKeepDv>(),
                               prepare<kBwdP>(),    prepare<kBwdPDv>(),    prepare<kFwdFp8T>(),   prepare<kBwdDw>()};
    for (const cudaError_t e : all)
        if (e != cudaSuccess) return e;
    return cudaSuccess;
}

}  // namespace ais
