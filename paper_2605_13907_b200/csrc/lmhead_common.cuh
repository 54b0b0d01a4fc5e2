// Device helpers shared by the LM-head tensor-core kernels: stage-ring bookkeeping, warp-wide bounded waits,
// register re-splitting, work-unit decoding and the test for row tiles without work.
#pragma once

#include "../../include/ais.h"
#include "launch.cuh"
#include "lmhead.cuh"
#include "ptx.cuh"

namespace ais {

namespace {

constexpr float kLog2e = 1.4426950408889634f;
constexpr float kLn2 = 0.6931471805599453f;
constexpr float kNegBig = -1.0e30f;

struct Pipe {
    uint32_t idx = 0, phase = 0;
    int n;
    __device__ explicit Pipe(int n_) : n(n_) {}
    __device__ __forceinline__ void advance() {
        if (++idx == static_cast<uint32_t>(n)) { idx = 0; phase ^= 1u; }
    }
};

// Pacing of the persistent CTAs of one launch.  CTAs that share operand tiles through L2 (the column slices of a row
// pair, the row tiles of a vocabulary range) only hit there while they stay within a few dozen stage fills of each
// other, and left alone they drift apart by several per cent of a unit per unit.  Each CTA's producer therefore
// announces every kPaceFills-th stage fill of its n-th unit on a ring of counters in the workspace and lets the slowest
// CTA catch up to within kPaceLag announcements before it goes on.  The wait is advisory and bounded: after
// kPaceWait clock ticks the producer goes on regardless, and after three such give-ups in a row it stops waiting
// for the rest of the launch (it still announces), so CTAs that are not all resident at once cost time, not progress.
// Every announcement index receives exactly gridDim.x arrivals: units without work and the missing units of the
// last wave are announced in one go.
constexpr int kPaceLag = 2;
constexpr long long kPaceWait = 200000;  // clock ticks

struct Pacer {
    uint32_t* ring;      // nullptr: no pacing
    int per_unit;        // announcements per unit (the same for every unit of the launch)
    int strikes = 0;
    const volatile uint32_t* slot = nullptr;   // counter this CTA still has to see reach `want` (nullptr: nothing pending)
    uint32_t want = 0, seen = 0;
    __device__ Pacer(uint32_t* r, int c) : ring(r), per_unit(c) {}
    // Announcement c of unit n.  The counter to wait for is read here and looked at in settle(), a few stage fills
    // later, so that the read's round trip to L2 is not spent waiting.
    __device__ __forceinline__ void announce(int n, int c) {
        const long long k = static_cast<long long>(n) * per_unit + c;
        atomicAdd(&ring[k % kPaceRing], 1u);
        const long long kw = k - kPaceLag;
        if (kw < 0 || strikes >= 3) return;
        want = static_cast<uint32_t>(gridDim.x) * static_cast<uint32_t>(kw / kPaceRing + 1);
        slot = ring + (kw % kPaceRing);
        seen = *slot;
    }
    __device__ __forceinline__ void settle() {
        if (slot == nullptr) return;
        if (seen < want) {
            const long long t0 = clock64();
            while (*slot < want) {
                if (clock64() - t0 > kPaceWait) { ++strikes; slot = nullptr; return; }
            }
        }
        strikes = 0;
        slot = nullptr;
    }
    // announcements c_from .. per_unit - 1 of unit n without waiting (unit ended early, had no work, or does not exist)
    __device__ __forceinline__ void top_up(int n, int c_from) {
        for (int c = c_from; c < per_unit; ++c)
            atomicAdd(&ring[(static_cast<long long>(n) * per_unit + c) % kPaceRing], 1u);
    }
};

// Warp-wide wait: every lane polls (so every lane observes the completed phase itself) and the outcome is
// made uniform, because the tcgen05.ld / __syncwarp that follow need the whole warp.
__device__ __forceinline__ bool mbar_wait_warp(uint64_t* bar, uint32_t parity, volatile int* abort_flag,
                                               long long limit = 0) {
    const bool r = mbar_wait(bar, parity, abort_flag, limit);
    return __all_sync(0xffffffffu, r);
}

__device__ __forceinline__ bool mbar_wait_warp_spin(uint64_t* bar, uint32_t parity, volatile int* abort_flag,
                                                    long long limit = 0) {
    const bool r = mbar_wait_spin(bar, parity, abort_flag, limit);
    return __all_sync(0xffffffffu, r);
}

__device__ __forceinline__ float ex2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

template <int N>
__device__ __forceinline__ void reg_alloc() {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(N));
}
template <int N>
__device__ __forceinline__ void reg_dealloc() {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(N));
}

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
    __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<uint32_t*>(&v);
}

// Which row tile and which column tiles a work unit covers, which K steps, and (split dH units) the partial tile it fills.
struct Unit {
    int rt, t0, t1, part;
    int k0, k1;            // K steps (stage fills per column tile)
    int slot;              // partial tile of a split unit; -1: the unit's result is final
};
template <int MODE>
__device__ __forceinline__ int count_units(const LmheadArgs& a) {
    if (MODE == kBwdDh) return a.split_from + (a.n_row_tiles * a.n_col_tiles - a.split_from) * a.ksplit;
    return MODE == kBwdDw ? a.n_row_tiles * a.n_col_tiles : a.n_row_tiles * a.nsplit;
}
template <int MODE>
__device__ __forceinline__ Unit decode_unit(const LmheadArgs& a, int u) {
    Unit w;
    w.k0 = 0;
    w.k1 = a.ksteps;
    w.slot = -1;
    if (MODE == kBwdDh || MODE == kBwdDw) {
        if (MODE == kBwdDh && u >= a.split_from && a.ksplit > 1) {
            // consecutive units share a range of the contraction, so the CTAs that run together share their operand slices
            const int tail = a.n_row_tiles * a.n_col_tiles - a.split_from;
            w.slot = u - a.split_from;
            const int kr = w.slot / tail;
            w.k0 = static_cast<int>((static_cast<int64_t>(kr) * a.ksteps) / a.ksplit);
            w.k1 = static_cast<int>((static_cast<int64_t>(kr + 1) * a.ksteps) / a.ksplit);
            u = a.split_from + w.slot % tail;
        }
        if (MODE == kBwdDw && a.n_row_tiles < a.n_col_tiles) {
            // dW of a [d, V] head: the few row tiles (their operand stays in L2) vary fastest, so that the scratch is read once;
            // the other order read all of it for every row tile
            w.rt = u % a.n_row_tiles;
            w.t0 = u / a.n_row_tiles;
        } else {
            w.rt = u / a.n_col_tiles;
            w.t0 = u % a.n_col_tiles;
        }
        w.t1 = w.t0 + 1;
        w.part = 0;
    } else {
        w.rt = u / a.nsplit;
        const int c = u % a.nsplit;
        w.t0 = static_cast<int>((static_cast<int64_t>(c) * a.n_col_tiles) / a.nsplit);
        w.t1 = static_cast<int>((static_cast<int64_t>(c + 1) * a.n_col_tiles) / a.nsplit);
        w.part = c;
    }
    return w;
}

// Row tiles in which no row needs computing (all rows masked in the forward passes, all gradient factors zero in
// the backward passes) are skipped by all three roles alike; the epilogue writes the neutral output where one is
// needed.  The dW pass contracts over rows, so it has nothing to skip.
template <int MODE>
__device__ __forceinline__ bool unit_active(const LmheadArgs& a, const Unit& w) {
    if (MODE == kBwdDw || a.tile_active == nullptr) return true;
    const int64_t g = a.row0 / kBM;
    if (MODE == kBwdDh || MODE == kFwdFp8) {                  // units of two row tiles
        const int64_t t0 = g + 2 * static_cast<int64_t>(w.rt);
        const bool second = (2 * static_cast<int64_t>(w.rt) + 1) * kBM < a.rows;
        return a.tile_active[t0] != 0 || (second && a.tile_active[t0 + 1] != 0);
    }
    return a.tile_active[g + w.rt] != 0;
}

// Units of two row tiles: does the second one hold rows to compute?
__device__ __forceinline__ bool second_tile_active(const LmheadArgs& a, const Unit& w) {
    const int64_t second = 2 * static_cast<int64_t>(w.rt) + 1;
    return second * kBM < a.rows && (a.tile_active == nullptr || a.tile_active[a.row0 / kBM + second] != 0);
}

// Opening of a pass, by every thread, after the set-up that touches no global memory.  The trigger comes after the wait,
// so whatever a dependent that does not wait (args.overlap) reads was complete before that dependent could start.
__device__ __forceinline__ void enter_pass(const LmheadArgs& a) {
    if (!a.overlap) pdl_wait();
    pdl_trigger();
    if (a.pace_clear != nullptr)
        for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < kPaceRing / 4; i += gridDim.x * blockDim.x)
            reinterpret_cast<uint4*>(a.pace_clear)[i] = make_uint4(0, 0, 0, 0);
}
// Its end, by every thread: a pass that did not wait at the start completes only after the kernel before it has.
__device__ __forceinline__ void leave_pass(const LmheadArgs& a) {
    if (a.overlap) pdl_wait();
}

// ------------------------------------------------------------------ epilogue of the forward and recompute passes
// One output row of a thread: what its epilogue knows about it and, in the forward passes, its streaming log-sum-exp
// (log2-domain running reference, sum of 2^(z log2e - reference), target logit).
// Recompute: U = mul (e^(z - off) - onehot) in plain form (off = lse, mul = c), mul = 1, off = 0 and `target` at the target
// column in exponent form (exp_form).
constexpr __host__ __device__ bool keep_mode(int mode) { return mode == kFwdKeep || mode == kFwdKeepDv; }
// |reference| (log2 units) up to which the kept exponentials are relative to 0; just above exp_form's largest lse
constexpr float kKeepRange = 86.0f;

struct RowState {
    int64_t lrow, grow;              // row inside the launch, row of the batch
    bool in, valid;
    int y;                           // target column, -1: none
    float m2, s, zy;
    float off2, mul, target;
    bool ef;
};

template <int MODE>
__device__ __forceinline__ RowState begin_row(const LmheadArgs& a, int64_t lrow, uint32_t& flags) {
    constexpr int BASE = base_mode(MODE);
    RowState r;
    r.lrow = lrow;
    r.in = lrow < a.rows;
    r.grow = a.row0 + lrow;
    r.y = -1;
    r.valid = false;
    r.m2 = kNegBig;
    r.s = 0.f;
    r.zy = -INFINITY;
    r.off2 = r.mul = r.target = 0.f;
    r.ef = false;
    if (!r.in) return r;
    r.y = a.tokens[r.grow];
    r.valid = a.mask[r.grow] != 0;
    if (r.valid && (r.y < 0 || r.y >= a.ncols)) { flags |= AIS_FLAG_TOKEN_RANGE; r.y = -1; }
    if (BASE == kBwdP) {
        const float lse = a.lse[r.grow];
        r.mul = a.coef[r.grow];
        if (r.mul == 0.f) r.valid = false;             // rows without gradient are written as exact zeros
        r.ef = a.row_scale != nullptr && exp_form(lse);
        if (r.ef) { r.mul = 1.f; r.target = exp_form_target(a.lp[r.grow], lse); }
        else r.off2 = lse * kLog2e;
    }
    return r;
}

// 32 consecutive logits of the row, from column col0 on.  `store`: the row's scratch is wanted (kFwdKeep, recompute).
template <int MODE>
__device__ __forceinline__ void row_slice(const LmheadArgs& a, RowState& r, int col0, float (&x)[32], bool store) {
    constexpr bool KEEP = keep_mode(MODE);
    uint32_t pk[16];
    if (base_mode(MODE) == kBwdP) {
        if (!store || col0 >= a.ncols) return;
#pragma unroll
        for (int i = 0; i < 32; i += 2) {
            float p0 = r.valid ? ex2(fmaf(x[i], kLog2e, -r.off2)) : 0.f;
            float p1 = r.valid ? ex2(fmaf(x[i + 1], kLog2e, -r.off2)) : 0.f;
            if (col0 + i == r.y) p0 = r.ef ? r.target : p0 - 1.f;
            if (col0 + i + 1 == r.y) p1 = r.ef ? r.target : p1 - 1.f;
            pk[i >> 1] = pack_bf16(r.valid ? r.mul * p0 : 0.f, r.valid ? r.mul * p1 : 0.f);
        }
    } else {
        if (r.y >= col0 && r.y < col0 + 32) {
#pragma unroll
            for (int i = 0; i < 32; ++i)
                if (col0 + i == r.y) r.zy = x[i];
        }
        if (col0 + 32 > a.ncols) {
#pragma unroll
            for (int i = 0; i < 32; ++i)
                if (col0 + i >= a.ncols) x[i] = -INFINITY;
        }
        float cm = x[0];
#pragma unroll
        for (int i = 1; i < 32; ++i) cm = fmaxf(cm, x[i]);
        float m_new = fmaxf(r.m2, cm * kLog2e);
        // reference 0 for every row within range, so that the terms of the sum are what the scratch wants
        if (KEEP && fabsf(m_new) <= kKeepRange) m_new = 0.f;
        float add = 0.f;
        if (KEEP) {
#pragma unroll
            for (int i = 0; i < 32; i += 2) {
                const float e0 = ex2(fmaf(x[i], kLog2e, -m_new)), e1 = ex2(fmaf(x[i + 1], kLog2e, -m_new));
                add += e0;
                add += e1;
                pk[i >> 1] = pack_bf16(e0, e1);
            }
        } else {
#pragma unroll
            for (int i = 0; i < 32; ++i) add += ex2(fmaf(x[i], kLog2e, -m_new));
        }
        r.s = fmaf(r.s, ex2(r.m2 - m_new), add);
        r.m2 = m_new;
        if (!KEEP || !store || col0 >= a.ncols) return;
        if (m_new != 0.f) {                            // rare: this range of the row lies far below the rest, or above
#pragma unroll
            for (int i = 0; i < 32; i += 2)
                pk[i >> 1] = pack_bf16(ex2(fmaf(x[i], kLog2e, -0.f)), ex2(fmaf(x[i + 1], kLog2e, -0.f)));
        }
    }
    uint4* dst = reinterpret_cast<uint4*>(a.U + r.lrow * a.ldU + col0);
#pragma unroll
    for (int j = 0; j < 4; ++j)
        if (col0 + j * 8 < a.ncols) dst[j] = make_uint4(pk[4 * j], pk[4 * j + 1], pk[4 * j + 2], pk[4 * j + 3]);
}

// Forward passes: the row's partial triple for one vocabulary range and column half.
__device__ __forceinline__ void end_row(const LmheadArgs& a, const RowState& r, int part) {
    if (!r.in) return;
    const int64_t o = static_cast<int64_t>(part) * a.part_ld + r.grow;
    a.part_m[o] = r.m2 * kLn2;
    a.part_s[o] = r.s;
    a.part_z[o] = r.zy;
}

// After every role has left its loops: if the CTA gave up on a wait, the tile copies that the producer issued last
// (one per stage of the ring at most) may still be in flight.  Wait for them, so that no copy writes into shared
// memory that the CTA has already given back; `issued` counts the producer's stage fills.
__device__ __forceinline__ void drain_stage_copies(uint64_t* full, uint32_t issued, uint32_t stages) {
    const uint32_t pending = issued < stages ? issued : stages;
    for (uint32_t i = 0; i < pending; ++i) {
        const uint32_t n = issued - 1 - i;                 // n-th fill overall: stage n % stages, phase n / stages
        mbar_wait_drain(&full[n % stages], (n / stages) & 1u);
    }
}

}  // namespace

}  // namespace ais
