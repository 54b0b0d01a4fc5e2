// Rollout log-probabilities from E4M3 codes with one fp32 scale per block of 128 / 64 / 32 elements along d.
//
// The scales are arbitrary fp32 numbers, so the hardware's block-scaled MMA kinds (power-of-two scales) do not
// apply: every scale block's partial sum is accumulated alone in tensor memory, read back and promoted on the
// CUDA cores as acc += (partial * sH[row]) * sW[col], two columns per instruction (packed fp32).  One persistent CTA per SM:
//   warp 0      TMA producer: one stage = 128 K-bytes of A (256 rows) and B (128 rows) plus the stage's scale
//               vectors, all completing on the stage's barrier
//   warps 1, 2  MMA issuers: SG blocks per stage, PER = 4 / SG instructions per block and row tile, one commit per block; two
//               256-column tensor-memory buffers alternate between blocks, issuer i owning buffer i
//   warps 4-11  promotion + streaming log-sum-exp.  A tile is two row tiles x 128 columns (partial sums of the second
//               row tile 128 tensor-memory columns further on): warp w reads lane quarter w % 4, column half (w - 4) / 4
//               of both, so a thread owns two rows x 64 columns (128 fp32 sums).  The row scales are two registers; the
//               column scales come as broadcast 16-byte shared-memory loads, each used for both rows.  Pieces of
//               2 x 16 columns are software-pipelined: the load of piece p + 1 is in flight during the arithmetic of
//               piece p, and the buffer goes back to its MMA issuer as soon as the last piece has landed.
// The epilogue never waits for the scales separately: an MMA issuer saw the stage barrier complete before it
// issued the block whose completion the epilogue waits for.  The first warpgroup hands registers to the other
// two (384 threads x 168 registers at launch = 128 x 40 + 256 x 232).
// What bounds it: the promotion warps.  Running free (no barriers, no MMAs; timing-only copy) they take 820 clocks per
// 128 x 256 x 128 of work: arithmetic 570, broadcast loads +110 to +200, tensor-memory loads +110, which add up instead of
// overlapping; with one row tile x 256 columns per tile (each column scale used once) the broadcast loads cost twice that
// and the pass took 1,430 clocks against 1,290 now (9,216 rows, d = 4096, 65,536 columns, same box), with block 32 1,210
// against 1,000 clocks per scale block.  Passing a barrier that completed long ago costs a warp about 250 clocks, which is
// why the next block's barrier is tested before the last arithmetic of this one (block 32: 1,090 -> 1,000).  Sixteen and
// twelve promotion warps (32 columns each) and scale loads hoisted above the waits measured slower or the same.
// With several blocks per stage the two buffers alternate inside a stage, so the loop over its blocks is unrolled by two and
// every tensor-memory address and barrier of a block is a constant offset: block 32 1,005 -> 962 clocks per scale block (8.15 ->
// 7.80 ms, 9,216 rows, d = 4096, 65,536 columns), block 64 4.53 -> 4.35 ms; unrolled by four 1,038 (instruction fetch).
// What the promotion contends for is the path out of shared memory: a broadcast 16-byte load returns 512 bytes, four clocks of
// it, and the MMAs take all of it while they run (8 KB of operands per 64 clocks).  In a copy of the loop with real MMAs and
// without the rest of the kernel a block takes 753 clocks with no MMA, 831 to 840 with the two of block 32 and 1,187 with the eight of
// block 128, against 687, 720 and 791 with the column scales taken as constants; operand copies add nothing to that.  Loads of
// scales by shuffle (1,232), 16x256b tensor-memory loads (eight rows x 16 columns per thread, a third of the scale traffic, but
// half the tensor-memory rate: 1,137) and 128 x 256 tiles of them (1,141) do not get below it.
// How the roles with one thread are entered.  Through elect.sync a stage's copies and a block's MMAs take 10% to 20% less to issue
// than behind `lane == 0` (hand-overs alone, no promotion: 928 -> 847 clocks per block, block 32 414 -> 343).  That shortens what a
// short launch waits for, but in a long one the MMAs then meet the promotion of the block before on the path out of shared memory.
// Block 128, both behind `lane == 0` / issuers elected / both elected (us, in turn on one box; rows x d, columns):
//   pass alone: 600 x 4096, 4,096 30.2 / 29.0 / 29.1;  1,100 x 4096, 16,384 125.4 / 121.4 / 122.8;  3,000 x 2048, 16,384 147.4 / 145.7 /
//   147.7;  6,000 x 1024, 32,000 301 / 304 / 305;  12,000 x 4096, 65,536 4,260 / 4,316 / 4,389;  one row tile, 100 x 4096, 4,096 25.3 /
//   25.9 / 20.6
//   whole step, 9,217 x 4096, 151,936 25,080 / 24,900 / 24,920 (issues that keep pace cost a long pass time and the passes behind it gain
//   more: the step runs at the power cap); log-probs alone 15,840 / 15,830 / 15,980
// Blocks of 64 and 32, behind `lane == 0` and elected: pass alone 12,000 x 4096, 65,536 5,917 and 6,022, 10,407 and 10,506; whole step,
// 9,217 x 4096, 151,936 28,930 and 29,210, 36,890 and 37,360.  Here it is the stages of a tile that decide.
// So the issuers of block 128 are elected, its producer for one row tile only; both roles of smaller blocks are below kElectSteps stages
// per tile (ELECT).
#include <type_traits>

#include "lmhead_common.cuh"
#include "../../include/ais.h"

namespace ais {

namespace {

constexpr int kHalfCols = kPairCols / 2;                              // columns of a promotion warp
constexpr int kPairABytes = kPairRows * kStageKBytes;               // A part of a stage (two row tiles), then B

template <int SG>
struct Fp8Cfg {
    static constexpr int kSlots = (SG == 4) ? 5 : 8;                  // scale slots: more than stages + buffers in flight
    static constexpr int kSlotBytes = SG * (kPairRows + kPairCols) * 4;
    static constexpr int kSlotBOffset = SG * kPairRows * 4;
    static constexpr int kBarriers = 2 * kStages + 4 + kSlots + 1;
    static constexpr int kSmem = 1024 + kStages * kStageBytes + kSlots * kSlotBytes + kBarriers * 8 + 64;
};
static_assert(Fp8Cfg<4>::kSmem <= 232448 && Fp8Cfg<1>::kSmem <= 232448, "shared memory of the FP8 pass");
// With one block per stage a slot's scales are given back without a barrier of the warp between the other lanes' reads and lane 0's
// arrival (a vote orders no memory accesses).  What orders them is the way of the operands: fill m waits for the MMAs of fill
// m - kStages, those waited for the buffer of the block two before theirs, and every warp gave that buffer back behind a
// __syncwarp that follows all its reads of the block before.  So when fill m is requested the scales of fills up to
// m - kStages - 3 have been read, and a slot may be written again that many fills later or more.
static_assert(Fp8Cfg<1>::kSlots >= kStages + 3, "a scale slot is rewritten only after all lanes have read it");

// TILES: row tiles that are promoted, 2, or 1 for a batch of no more than one (kBM rows): half the tensor-memory loads and
// arithmetic, the same scale loads.  100 rows at d = 4096, V = 151936 190 -> 159 us, block 32 (65,536 columns) 264 -> 172.  The last,
// half pair of a longer batch stays with the others: behind whole pairs the launch ends with those, and giving it fewer, longer
// ranges cost more than it saved (613 rows 525 -> 545 us, 1,100 rows 885 -> 926), because pairs that do not walk the vocabulary
// together do not share its codes through L2.
// RUN: blocks that a run of the promotion loop takes, the buffers alternating from buffer 0 on: SG, or with one block per stage and one row
// tile 2 where a tile has an even number of stages (d a multiple of 256: 20 rows x 2048, 32,000 columns 41.9 -> 40.8 us, 100 x 4096,
// 4,096 columns 20.6 -> 20.3), else 1.  With two row tiles runs of two are no faster at d = 4096 (12,000 rows, 65,536 columns 4,316 and
// 4,350 us) and slower where a tile has few stages (d = 256, 20,000 rows, 16,384 columns 196 -> 212, 8,000 and 8,192 56.7 -> 61.0).
template <int SG, int TILES, int RUN, bool ELECT>
__global__ void __launch_bounds__(kThreads, 1)
lmhead_fp8_block_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                        const __grid_constant__ CUtensorMap tmSA, const __grid_constant__ CUtensorMap tmSB,
                        const LmheadArgs a) {
    using C = Fp8Cfg<SG>;
    constexpr int PER = 4 / SG;                     // MMAs (32 K-bytes each) per scale block
    constexpr int MODE = kFwdFp8;
    extern __shared__ uint8_t smem_raw[];
    // 1024-byte aligned start, as an offset from the array so that the compiler still knows the address space
    uint8_t* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    uint8_t* stage_base = smem;
    uint8_t* scale_base = smem + kStages * kStageBytes;
    uint64_t* bars = reinterpret_cast<uint64_t*>(scale_base + C::kSlots * C::kSlotBytes);
    uint64_t* full = bars;                       // [kStages]  TMA -> MMA (operands and scales of the stage)
    uint64_t* empty = full + kStages;            // [kStages]  MMA -> TMA
    uint64_t* tfull = empty + kStages;           // [2]        MMA -> epilogue: a block's partial sums are complete
    uint64_t* tempty = tfull + 2;                // [2]        epilogue -> MMA: the partial sums are in registers
    uint64_t* sempty = tempty + 2;               // [kSlots]   epilogue -> TMA: the stage's scales have been used
    uint64_t* done = sempty + C::kSlots;         // [1]        all MMAs of this CTA have completed
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + C::kBarriers);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
    volatile uint32_t* issued_slot = tmem_slot + 2;     // stage fills the producer has requested (written when it leaves its loop)

    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    const int num_units = a.n_row_tiles * a.nsplit;

    if (threadIdx.x == 0) {
        for (int i = 0; i < kStages; ++i) { mbar_init(&full[i], 1); mbar_init(&empty[i], SG > 1 ? 2 : 1); }   // both issuers use a stage when it holds several blocks
        for (int i = 0; i < 2; ++i) { mbar_init(&tfull[i], 1); mbar_init(&tempty[i], kEpiWarps); }
        for (int i = 0; i < C::kSlots; ++i) mbar_init(&sempty[i], kEpiWarps);
        mbar_init(done, 2);
        *abort_flag = 0;
        *issued_slot = 0;
        fence_barrier_init();
        tma_prefetch_desc(&tmA);
        tma_prefetch_desc(&tmB);
        tma_prefetch_desc(&tmSA);
        tma_prefetch_desc(&tmSB);
    }
    if (warp == 1) {
        tmem_alloc(tmem_slot, 512);
        tmem_relinquish();
    }
    enter_pass(a);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;

    if (warp < 4) {
        reg_dealloc<40>();
        if (warp == 0) {
            // ------------------------------------------------------------------ TMA producer
            if (ELECT && (TILES == 1 || SG > 1) ? elect_one() : lane == 0) {
                Pipe st(kStages), sc(C::kSlots);
                uint32_t issued = 0;
                bool ok = true;
                Pacer pacer(a.pace, a.pace_per_unit);
                int n = 0;                                      // ordinal of this CTA's unit (its wave)
                for (int u = blockIdx.x; u < num_units && ok; u += gridDim.x, ++n) {
                    const Unit w = decode_unit<MODE>(a, u);
                    if (!unit_active<MODE>(a, w)) {
                        if (pacer.ring) pacer.top_up(n, 0);
                        continue;
                    }
                    int fills = 0;                              // stage fills of this unit so far
                    for (int t = w.t0; t < w.t1 && ok; ++t) {
                        for (int ks = 0; ks < a.ksteps; ++ks, ++fills) {
                            if (pacer.ring && fills % kPaceFills == 0) pacer.announce(n, fills / kPaceFills);
                            if (pacer.ring && fills % kPaceFills == kPaceSettle) pacer.settle();
                            if (!mbar_wait(&empty[st.idx], st.phase ^ 1u, abort_flag, a.wait_cycles)) { ok = false; break; }
                            if (!mbar_wait(&sempty[sc.idx], sc.phase ^ 1u, abort_flag, a.wait_cycles)) { ok = false; break; }
                            uint8_t* sA = stage_base + st.idx * kStageBytes;
                            uint8_t* sS = scale_base + sc.idx * C::kSlotBytes;
                            mbar_expect_tx(&full[st.idx], kStageBytes + C::kSlotBytes);
                            tma_load_2d(sS, &tmSA, &full[st.idx], w.rt * kPairRows, ks * SG);
                            tma_load_2d(sS + C::kSlotBOffset, &tmSB, &full[st.idx], t * kPairCols, ks * SG);
                            tma_load_2d(sA, &tmA, &full[st.idx], ks * 128, w.rt * kPairRows);
                            tma_load_2d(sA + kPairABytes, &tmB, &full[st.idx], ks * 128, t * kPairCols);
                            ++issued;
                            st.advance();
                            sc.advance();
                        }
                    }
                    if (pacer.ring) pacer.top_up(n, (fills + kPaceFills - 1) / kPaceFills);
                }
                if (pacer.ring)                                 // units of the last wave that this CTA does not have
                    for (const int waves = (num_units + gridDim.x - 1) / gridDim.x; n < waves; ++n) pacer.top_up(n, 0);
                *issued_slot = issued;
            }
        } else if (warp == 1 || warp == 2) {
            // ------------------------------------------------------------------ MMA issuers
            // Two of them, on two schedulers: issuer `me` owns tensor-memory buffer `me` and takes every other scale
            // block (block n of the CTA goes to buffer n % 2).  One thread cannot keep up: it shares its scheduler with
            // two promotion warps, and wait + four MMAs + two commits took it about 1,300 clocks per block against the
            // 542 the tensor core needs.  The two threads are independent: different buffers, different barriers.
            if (ELECT ? elect_one() : lane == 0) {
                const uint32_t me = warp - 1;
                constexpr uint32_t idesc = make_idesc(kFmtE4M3, kFmtE4M3, kBM, kPairCols, 0, 0);
                const uint64_t desc0 = smem_desc_sw128(0, 16, 1024);           // descriptor of address 0: add (address >> 4)
                const uint32_t dcol = tmem_base + me * (2 * kPairCols);
                Pipe st(kStages);
                uint32_t tphase = 0;                                            // phase of this issuer's buffer barriers
                uint32_t nstage = 0;                                            // stages seen so far (SG == 1: parity picks the owner)
                bool ok = true;
                for (int u = blockIdx.x; u < num_units && ok; u += gridDim.x) {
                    const Unit w = decode_unit<MODE>(a, u);
                    if (!unit_active<MODE>(a, w)) continue;
                    const int nst = (w.t1 - w.t0) * a.ksteps;
                    const bool two = second_tile_active(a, w);
                    for (int i = 0; i < nst && ok; ++i, ++nstage) {
                        if (SG > 1 || (nstage & 1u) == me) {
                            if (!mbar_wait(&full[st.idx], st.phase, abort_flag, a.wait_cycles)) { ok = false; break; }
                            const uint64_t adesc = desc0 + (smem_u32(stage_base + st.idx * kStageBytes) >> 4);
#pragma unroll
                            for (int g = 0; g < SG; ++g) {
                                if (SG > 1 && (g & 1) != static_cast<int>(me)) continue;
                                if (!mbar_wait(&tempty[me], tphase ^ 1u, abort_flag, a.wait_cycles)) { ok = false; break; }
                                tc_fence_after();
#pragma unroll
                                for (int j = 0; j < PER; ++j) {
                                    const uint64_t ad = adesc + 2 * (g * PER + j);       // 32 bytes of K further on
                                    const uint64_t bd = ad + (kPairABytes >> 4);
                                    mma_f8(dcol, ad, bd, idesc, j > 0 ? 1u : 0u);
                                    if (two) mma_f8(dcol + kPairCols, ad + (kAStageBytes >> 4), bd, idesc, j > 0 ? 1u : 0u);
                                }
                                tc_commit(&tfull[me]);
                                tphase ^= 1u;
                            }
                            if (!ok) break;
                            tc_commit(&empty[st.idx]);
                        }
                        st.advance();
                    }
                }
                // everything issued has to finish before the tensor memory is given back
                tc_commit(done);
            }
        }
    } else {
        // ------------------------------------------------------------------ promotion and streaming log-sum-exp
        reg_alloc<232>();
        const int q = warp & 3;                       // TMEM lane quarter this warp may read
        const int half = (warp - 4) >> 2;             // column half of the partial tile
        const uint32_t lane_base = static_cast<uint32_t>(q * 32) << 16;
        Pipe tb(2), sc(C::kSlots);
        bool ok = true;
        uint32_t flags = 0;
        uint32_t va[32], vb[32];
        bool ready = false;                           // the next block was seen complete before its turn
        // piece p: 16 columns of every row tile
        auto ld_piece = [&](uint32_t buf, int p, uint32_t (&v)[32]) {
            const uint32_t at = tmem_base + lane_base + buf * (2 * kPairCols) + half * kHalfCols + p * 16;
            tmem_ld16(at, v, 0);
            if (TILES == 2) tmem_ld16(at + kPairCols, v, 16);
        };
        for (int u = blockIdx.x; u < num_units && ok; u += gridDim.x) {
            const Unit w = decode_unit<MODE>(a, u);
            if (!unit_active<MODE>(a, w)) continue;     // every row masked: the merge kernel never reads these partials
            int64_t grow[2];
            bool rok[2];
            int y[2];
#pragma unroll
            for (int i = 0; i < TILES; ++i) {
                const int64_t lr = static_cast<int64_t>(w.rt) * kPairRows + i * kBM + q * 32 + lane;
                rok[i] = lr < a.rows;
                grow[i] = a.row0 + lr;
                y[i] = -1;
                if (rok[i]) {
                    y[i] = a.tokens[grow[i]];
                    if (a.mask[grow[i]] != 0 && (y[i] < 0 || y[i] >= a.ncols)) { flags |= AIS_FLAG_TOKEN_RANGE; y[i] = -1; }
                }
            }
            float m_run[2] = {kNegBig, kNegBig}, s_run[2] = {0.f, 0.f}, zy[2] = {-INFINITY, -INFINITY};
            for (int t = w.t0; t < w.t1 && ok; ++t) {
                F2 acc[TILES][kHalfCols / 2];                  // columns 2 n, 2 n + 1 of this thread's half, rows of both tiles
#pragma unroll
                for (int n = 0; n < kHalfCols / 2; ++n) acc[0][n] = acc[TILES - 1][n] = F2{0.f, 0.f};
                for (int ks = 0; ks < a.ksteps && ok; ks += RUN / SG) {
                    const float* sS = reinterpret_cast<const float*>(scale_base + sc.idx * C::kSlotBytes);
#pragma unroll(RUN > 1 ? 2 : 1)
                    for (int n = 0; n < RUN; ++n) {
                        const int g = SG > 1 ? n : 0;     // block of its stage
                        if (RUN > 1) tb.idx = n & 1;      // a run starts with buffer 0: known when the loop is unrolled by two
                        if (SG == 1 && n > 0) sS = reinterpret_cast<const float*>(scale_base + sc.idx * C::kSlotBytes);
                        if (!ready && !mbar_wait_warp_spin(&tfull[tb.idx], tb.phase, abort_flag, a.wait_cycles)) { ok = false; break; }
                        tc_fence_after();
                        const uint32_t buf = tb.idx;
                        ld_piece(buf, 0, va);
                        const float sh0 = sS[g * kPairRows + q * 32 + lane], sh1 = sS[g * kPairRows + (TILES - 1) * kBM + q * 32 + lane];
                        const F2 r0 = {sh0, sh0}, r1 = {sh1, sh1};
                        // every lane reads the same column scales: broadcast 16-byte loads, each used for two rows
                        const float4* sw4 = reinterpret_cast<const float4*>(sS + (C::kSlotBOffset / 4) + g * kPairCols + half * kHalfCols);
                        auto promote = [&](auto PP, uint32_t (&v)[32]) {
                            constexpr int pp = decltype(PP)::value;
#pragma unroll
                            for (int j = 0; j < 4; ++j) {
                                const float4 swf = sw4[pp * 4 + j];
                                const F2 c0 = {swf.x, swf.y}, c1 = {swf.z, swf.w};
                                F2* p0 = &acc[0][pp * 8 + 2 * j];
                                F2* p1 = &acc[TILES - 1][pp * 8 + 2 * j];
                                p0[0] = fma2(mul2(F2{__uint_as_float(v[4 * j]), __uint_as_float(v[4 * j + 1])}, r0), c0, p0[0]);
                                p0[1] = fma2(mul2(F2{__uint_as_float(v[4 * j + 2]), __uint_as_float(v[4 * j + 3])}, r0), c1, p0[1]);
                                if (TILES == 1) continue;
                                p1[0] = fma2(mul2(F2{__uint_as_float(v[16 + 4 * j]), __uint_as_float(v[17 + 4 * j])}, r1), c0, p1[0]);
                                p1[1] = fma2(mul2(F2{__uint_as_float(v[18 + 4 * j]), __uint_as_float(v[19 + 4 * j])}, r1), c1, p1[1]);
                            }
                        };
                        using I0 = std::integral_constant<int, 0>;
                        using I1 = std::integral_constant<int, 1>;
                        using I2 = std::integral_constant<int, 2>;
                        using I3 = std::integral_constant<int, 3>;
                        tmem_ld_wait(va);
                        ld_piece(buf, 1, vb);
                        promote(I0{}, va);
                        tmem_ld_wait(vb);
                        ld_piece(buf, 2, va);
                        promote(I1{}, vb);
                        tmem_ld_wait(va);
                        ld_piece(buf, 3, vb);
                        promote(I2{}, va);
                        tmem_ld_wait(vb);
                        // the whole partial tile is in registers: hand the buffer back before the last arithmetic
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(&tempty[buf]);
                        if (RUN > 1) {
                            tb.idx = (n + 1) & 1;
                            tb.phase ^= n & 1;
                        } else {
                            tb.advance();
                        }
                        // ask for the next block's barrier now: the answer comes back behind the last arithmetic
                        const bool seen = mbar_test_wait(&tfull[tb.idx], tb.phase);
                        promote(I3{}, vb);
                        ready = __all_sync(0xffffffffu, seen);
                        if (SG == 1) {                    // the stage's scales have been used (what orders the reads: see kSlots)
                            if (lane == 0) mbar_arrive(&sempty[sc.idx]);
                            sc.advance();
                        }
                    }
                    if (!ok) break;
                    if (SG > 1) {                             // (inside the loop it costs block 32 3%)
                        __syncwarp();
                        if (lane == 0) mbar_arrive(&sempty[sc.idx]);
                        sc.advance();
                    }
                }
                if (!ok) break;
                // streaming log-sum-exp over this thread's columns of its two rows
                const int cbase = t * kPairCols + half * kHalfCols;        // column of acc[.][0].x
#pragma unroll
                for (int i = 0; i < TILES; ++i) {
                    const int yy = y[i] - cbase;
                    if (yy >= 0 && yy < kHalfCols) {
                        // written as a running maximum on purpose: a chain of "if (k == n) z = acc[n]" is folded by
                        // the compiler into acc[k], and a dynamically indexed array leaves the register file
#pragma unroll
                        for (int n = 0; n < kHalfCols / 2; ++n) {
                            zy[i] = fmaxf(zy[i], (yy == 2 * n) ? acc[i][n].x : -INFINITY);
                            zy[i] = fmaxf(zy[i], (yy == 2 * n + 1) ? acc[i][n].y : -INFINITY);
                        }
                    }
                    if (t * kPairCols + kPairCols > a.ncols) {
#pragma unroll
                        for (int n = 0; n < kHalfCols / 2; ++n) {
                            if (cbase + 2 * n >= a.ncols) acc[i][n].x = -INFINITY;
                            if (cbase + 2 * n + 1 >= a.ncols) acc[i][n].y = -INFINITY;
                        }
                    }
                    float cm = acc[i][0].x;
#pragma unroll
                    for (int n = 0; n < kHalfCols / 2; ++n) cm = fmaxf(cm, fmaxf(acc[i][n].x, acc[i][n].y));
                    const float m_new = fmaxf(m_run[i], cm * kLog2e);
                    float add = 0.f;
#pragma unroll
                    for (int n = 0; n < kHalfCols / 2; ++n)
                        add += ex2(fmaf(acc[i][n].x, kLog2e, -m_new)) + ex2(fmaf(acc[i][n].y, kLog2e, -m_new));
                    s_run[i] = fmaf(s_run[i], ex2(m_run[i] - m_new), add);
                    m_run[i] = m_new;
                }
            }
#pragma unroll
            for (int i = 0; i < TILES; ++i)
                if (ok && rok[i]) {
                    const int64_t o = static_cast<int64_t>(w.part * 2 + half) * a.part_ld + grow[i];
                    a.part_m[o] = m_run[i] * kLn2;
                    a.part_s[o] = s_run[i];
                    a.part_z[o] = zy[i];
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
        drain_stage_copies(full, *issued_slot, kStages);
        if (a.status) atomicOr(a.status, AIS_FLAG_TIMEOUT);
    }
    leave_pass(a);
}

}  // namespace

// ELECT with several blocks per stage: below eight stages per tile.  Block 64, behind `lane == 0` and elected, 1,100 and 3,000 rows, 16,384
// columns: d = 256 27.4 and 27.1, 49.0 and 48.5 us; 512 37.3 and 37.2, 70.6 and 70.5; 1024 56.5 and 56.6, 112.6 and 113.0 (600 rows, 4,096
// columns 18.9 and 18.8); 4096 173.3 and 174.6, 387.0 and 390.4.
constexpr int kElectSteps = 8;

template <int SG>
static cudaError_t launch_blocks(const CUtensorMap& tmA, const CUtensorMap& tmB, const CUtensorMap& tmSA, const CUtensorMap& tmSB, const LmheadArgs& args,
                                 int num_ctas, cudaStream_t stream) {
    constexpr int kRun1 = SG == 1 ? 2 : SG;                                // of one row tile
    auto kernel = lmhead_fp8_block_kernel<SG, 2, SG, true>;
    if (SG > 1 && args.ksteps >= kElectSteps) kernel = lmhead_fp8_block_kernel<SG, 2, SG, SG == 1>;
    if (args.rows <= kBM) kernel = SG > 1 || args.ksteps % 2 == 0 ? lmhead_fp8_block_kernel<SG, 1, kRun1, true> : lmhead_fp8_block_kernel<SG, 1, SG, true>;
    return launch_pdl(kernel, num_ctas, kThreads, Fp8Cfg<SG>::kSmem, stream, tmA, tmB, tmSA, tmSB, args);
}

cudaError_t launch_lmhead_fp8_block(const CUtensorMap& tmA, const CUtensorMap& tmB, const CUtensorMap& tmSA,
                                    const CUtensorMap& tmSB, const LmheadArgs& args, int num_ctas, cudaStream_t stream) {
    switch (args.sgroups) {
        case 1: return launch_blocks<1>(tmA, tmB, tmSA, tmSB, args, num_ctas, stream);
        case 2: return launch_blocks<2>(tmA, tmB, tmSA, tmSB, args, num_ctas, stream);
        case 4: return launch_blocks<4>(tmA, tmB, tmSA, tmSB, args, num_ctas, stream);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t lmhead_fp8_block_prepare() {
    cudaError_t e = cudaSuccess;
    auto allow = [&](auto kernel, int bytes) {
        if (e == cudaSuccess) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    };
    allow(lmhead_fp8_block_kernel<1, 1, 1, true>, Fp8Cfg<1>::kSmem);
    allow(lmhead_fp8_block_kernel<1, 1, 2, true>, Fp8Cfg<1>::kSmem);
    allow(lmhead_fp8_block_kernel<1, 2, 1, true>, Fp8Cfg<1>::kSmem);
    allow(lmhead_fp8_block_kernel<2, 1, 2, true>, Fp8Cfg<2>::kSmem);
    allow(lmhead_fp8_block_kernel<2, 2, 2, true>, Fp8Cfg<2>::kSmem);
    allow(lmhead_fp8_block_kernel<2, 2, 2, false>, Fp8Cfg<2>::kSmem);
    allow(lmhead_fp8_block_kernel<4, 1, 4, true>, Fp8Cfg<4>::kSmem);
    allow(lmhead_fp8_block_kernel<4, 2, 4, true>, Fp8Cfg<4>::kSmem);
    allow(lmhead_fp8_block_kernel<4, 2, 4, false>, Fp8Cfg<4>::kSmem);
    return e;
}

}  // namespace ais
