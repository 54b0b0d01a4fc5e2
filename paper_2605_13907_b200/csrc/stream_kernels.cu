// Streaming kernels of the AIS path (everything that is not a dense contraction).
#include <type_traits>

#include "stream_kernels.cuh"
#include "launch.cuh"
#include "lmhead.cuh"
#include "ptx.cuh"

#include <cuda_bf16.h>
#include <math.h>

namespace ais {

namespace {

// ------------------------------------------------------------------------------------------------
// Quantisation of the rows of a bf16 matrix: E4M3 with an fp32 scale per 128 / 64 / 32 elements or per tensor, or
// microscaling FP8 / FP4 (E8M0 scale per 32).  Streaming kernels, bound by HBM (3 bytes per element) and close behind it by
// instruction issue: a CTA covers 4 warps x RPW rows x 1024 columns, a lane holds 8 consecutive values per 16-byte load, four
// loads per row segment.  Measured back to back on a 151936 x 4096 head (copy bandwidth 6.5 TB/s): block 128 380 -> 302 us
// (1.89 GB: 6.2 TB/s; 319 us when three heads take turns, so that nothing of one is left in L2) with one residual correction instead of two and the maxima of two loads per shuffle; ten CTAs of four warps per
// SM (48 registers) against five of eight 302 / 305, four 311, six 337, eight 385; microscaling FP8 305, FP4 272 us; a
// persistent form with the next segment prefetched 4.3 to 4.9 TB/s.  Small matrices take RPW = 1: four times the CTAs, no
// serial chain of rows in a warp.
// ------------------------------------------------------------------------------------------------
constexpr int kQCols = 1024;
constexpr int kQThreads = 128;
constexpr int kQIters = kQCols / 256;      // 16-byte loads per lane and row segment
constexpr int kQWarps = kQThreads / 32;

__device__ __forceinline__ uint16_t cvt_e4m3x2(float hi, float lo) {
    uint16_t r;
    asm("cvt.rn.satfinite.e4m3x2.f32 %0, %1, %2;" : "=h"(r) : "f"(hi), "f"(lo));
    return r;
}

// IEEE division kept out of line: it is only reached for scales outside [2^-100, 2^100] and would otherwise
// be inlined eight times into every copy of the hot loop.
__device__ __noinline__ float slow_div(float x, float s) { return __fdiv_rn(x, s); }

// Block maxima of two 16-byte loads at once, on the bf16 bit patterns: |x| is the pattern without its sign bit, and patterns
// of non-negative values order like the values, so packed 16-bit unsigned maxima do the work of eight float compares.
// Low half: the maximum over the lane's block in a, high half: in b.
template <int BLOCK>
__device__ __forceinline__ uint32_t block_amax_pair(const uint4 a, const uint4 b) {
    constexpr int kLanesPerBlock = BLOCK / 8;
    constexpr uint32_t k = 0x7FFF7FFFu;
    const uint32_t ma = __vmaxu2(__vmaxu2(a.x & k, a.y & k), __vmaxu2(a.z & k, a.w & k));
    const uint32_t mb = __vmaxu2(__vmaxu2(b.x & k, b.y & k), __vmaxu2(b.z & k, b.w & k));
    uint32_t m = __vmaxu2(__byte_perm(ma, mb, 0x5410), __byte_perm(ma, mb, 0x7632));
#pragma unroll
    for (int off = 1; off < kLanesPerBlock; off <<= 1) m = __vmaxu2(m, __shfl_xor_sync(0xffffffffu, m, off));
    return m;
}

// Eight bf16 values divided by the block's scale s (y = RN(1 / s)) and rounded to E4M3.
__device__ __forceinline__ uint2 quantize_values(const uint4 raw, float s, float y) {
    const uint32_t w[4] = {raw.x, raw.y, raw.z, raw.w};
    float v[8], qv[8];
    uint2 signs = make_uint2(0, 0);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        v[2 * i] = __uint_as_float(w[i] << 16);
        v[2 * i + 1] = __uint_as_float(w[i] & 0xFFFF0000u);
    }
    if (s > 0x1p-100f && s < 0x1p100f) {
        // x / s from the correctly rounded reciprocal y = RN(1/s), two values per instruction: q0 = RN(x y) is within 2^-23 of
        // x / s, and q1 = RN(q0 + r y) with the residual r = x - s q0 rounds a value within 2^-46 of it.  The code of q1 is that
        // of the correctly rounded quotient: they could only differ where a half-ulp neighbour h of an E4M3 midpoint lies
        // within 2^-46 of x / s.  With S (24 bits) and X (8) the significands of s and x and M 2^20 +- 1, 16 <= M < 32, that of h,
        // |S (M 2^20 +- 1) - X 2^40| <= 8 forces S = a 2^20 + b with |b| <= 8 and b M = -+ a, a <= 16: only S = 2^24 - 1, M = 16,
        // where q1 is right (checked in exact arithmetic).  |x / s| <= 448, so nothing overflows; a quotient that underflows
        // encodes to zero either way.  The sign is put back into the codes because a zero residual sum turns -0 into +0.
        const F2 ys = {y, y}, ns = {-s, -s};
#pragma unroll
        for (int i = 0; i < 8; i += 2) {
            const F2 x = {v[i], v[i + 1]};
            F2 q = mul2(x, ys);
            q = fma2(fma2(ns, q, x), ys, q);
            qv[i] = q.x;
            qv[i + 1] = q.y;
        }
        signs = make_uint2(__byte_perm(w[0], w[1], 0x7531) & 0x80808080u, __byte_perm(w[2], w[3], 0x7531) & 0x80808080u);
    } else {
#pragma unroll
        for (int i = 0; i < 8; ++i) qv[i] = slow_div(v[i], s);      // rare: scale outside the safe exponent range
    }
    uint2 out;
    out.x = static_cast<uint32_t>(cvt_e4m3x2(qv[1], qv[0])) | (static_cast<uint32_t>(cvt_e4m3x2(qv[3], qv[2])) << 16);
    out.y = static_cast<uint32_t>(cvt_e4m3x2(qv[5], qv[4])) | (static_cast<uint32_t>(cvt_e4m3x2(qv[7], qv[6])) << 16);
    out.x |= signs.x;
    out.y |= signs.y;
    return out;
}

// The row segments of a warp: RPW rows one after the other (the loop stays rolled so that the kernel is small in the
// instruction cache; occupancy, not prefetching, hides the load latency), four 16-byte loads per lane each.
// body(row, raw): rows beyond the matrix included, with zeros.
template <int RPW, class Body>
__device__ __forceinline__ void walk_rows(const __nv_bfloat16* __restrict__ x, int64_t rows, int64_t cols, int64_t ld, int64_t row0,
                                          int64_t col0, Body body) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll 1
    for (int rr = 0; rr < RPW; ++rr) {
        const int64_t row = row0 + warp * RPW + rr;
        uint4 raw[kQIters];
#pragma unroll
        for (int it = 0; it < kQIters; ++it) {
            const int64_t col = col0 + it * 256 + lane * 8;
            raw[it] = (row < rows && col < cols) ? __ldg(reinterpret_cast<const uint4*>(x + row * ld + col)) : make_uint4(0, 0, 0, 0);
        }
        body(row, raw);
    }
}

// Row and column of a block's tile: tiles are numbered along the rows first, on grid.x alone (grid.y ends at 65,535 blocks,
// a million rows).
struct QuantTile {
    int64_t row0, col0;
    bool last_rows;          // one of the tiles with the last rows
};
template <int RPW>
__device__ __forceinline__ QuantTile quant_tile(unsigned tiles_x) {
    const unsigned row = blockIdx.x / tiles_x;
    return {static_cast<int64_t>(row) * (kQWarps * RPW), static_cast<int64_t>(blockIdx.x % tiles_x) * kQCols, row == (gridDim.x - 1) / tiles_x};
}

// Group-relative advantage of sequence s (Eq. grpo_adv), and what AdvJob clears for it.
__device__ __forceinline__ void run_advantage(const AdvJob& j, int s) {
    if (s == 0 && j.tickets) j.tickets[0] = j.tickets[1] = 0;
    if (j.zero_counts) j.zero_counts[s] = 0;
    const int g0 = (s / j.G) * j.G;
    double mean = 0.0;
    for (int k = 0; k < j.G; ++k) mean += static_cast<double>(j.rewards[g0 + k]);
    mean /= j.G;
    double a = static_cast<double>(j.rewards[s]) - mean;
    if (j.std_norm) {
        double var = 0.0;
        for (int k = 0; k < j.G; ++k) {
            const double dlt = static_cast<double>(j.rewards[g0 + k]) - mean;
            var += dlt * dlt;
        }
        a /= (sqrt(var / j.G) + static_cast<double>(j.eps));
    }
    j.adv[s] = static_cast<float>(a);
}

// FlagsJob by blocks of kQThreads threads: one warp per 128-row tile, and a thread for each sequence whose advantage is formed on the
// way: with the threads of the tiles alone (a quarter of T) each had several to form, one after the other, ahead of both passes (step
// of 1,024 rows in 4 x 256 sequences 57.8 -> 44.2 us, in 16 x 64 45.3 -> 40.5, of 18,944 rows in 74 x 256 105.6 -> 89.3).
constexpr int kFlagTiles = kQThreads / 32;
inline unsigned flag_blocks(const FlagsJob& f) {
    const int64_t tiles = ((f.T + 127) / 128 + kFlagTiles - 1) / kFlagTiles, seqs = (static_cast<int64_t>(f.adv.S) + kQThreads - 1) / kQThreads;
    return static_cast<unsigned>(tiles > seqs ? tiles : seqs);
}
__device__ __forceinline__ void run_flags(const FlagsJob& f, unsigned block, unsigned nblocks) {
    const int64_t tile = static_cast<int64_t>(block) * kFlagTiles + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (tile * 128 < f.T) {
        bool any = false;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int64_t t = tile * 128 + 32 * j + lane;
            any |= t < f.T && f.mask[t] != 0;
        }
        any = __any_sync(0xffffffffu, any);
        if (lane == 0) f.flags[tile] = any ? 1 : 0;
    }
    if (f.clear)
        for (int64_t k = static_cast<int64_t>(block) * kQThreads + threadIdx.x; k < f.clear_bytes / 16; k += static_cast<int64_t>(nblocks) * kQThreads)
            static_cast<uint4*>(f.clear)[k] = make_uint4(0, 0, 0, 0);
    for (int s = block * kQThreads + threadIdx.x; s < f.adv.S; s += nblocks * kQThreads) run_advantage(f.adv, s);
}
__global__ void __launch_bounds__(kQThreads) flags_kernel(const FlagsJob f) {
    pdl_enter();
    run_flags(f, blockIdx.x, gridDim.x);
}

// Blocks 0 .. n0 - 1 work on job0, the next n1 on job1, the rest on the flags.
template <int BLOCK, int RPW>
__global__ void __launch_bounds__(kQThreads, 10) quantize_kernel(const QuantJob job0, const QuantJob job1, unsigned n0, unsigned n1,
                                                                unsigned tiles_x, int64_t cols, const FlagsJob flags) {
    constexpr int kLanesPerBlock = BLOCK / 8;
    constexpr int kBlocksPerTile = kQCols / BLOCK;
    constexpr int kRows = kQWarps * RPW;
    __shared__ float sc[kBlocksPerTile][kRows + 1];          // scales leave along the rows (block-major)
    pdl_enter();
    if (blockIdx.x >= n0 + n1) {
        run_flags(flags, blockIdx.x - n0 - n1, gridDim.x - n0 - n1);
        return;
    }
    const bool second = blockIdx.x >= n0;
    const QuantJob& job = second ? job1 : job0;
    const unsigned tile = second ? blockIdx.x - n0 : blockIdx.x;
    const __nv_bfloat16* x = static_cast<const __nv_bfloat16*>(job.x);
    const int64_t rows = job.rows, ld = job.ld, ldq = job.ldq, lds = job.lds;
    uint8_t* codes = job.codes;
    float* scales = job.scales;
    const int lane = threadIdx.x & 31;
    const int64_t row0 = static_cast<int64_t>(tile / tiles_x) * kRows, col0 = static_cast<int64_t>(tile % tiles_x) * kQCols;
    walk_rows<RPW>(x, rows, cols, ld, row0, col0, [&](int64_t row, const uint4 (&raw)[kQIters]) {
        // block maxima of the four loads, then lane L of every block's lanes derives scale and reciprocal for load L % 4
        constexpr int kBlkPerIt = 32 / kLanesPerBlock;
        const uint32_t m01 = block_amax_pair<BLOCK>(raw[0], raw[1]), m23 = block_amax_pair<BLOCK>(raw[2], raw[3]);
        static_assert(kQIters == 4 && kLanesPerBlock >= 4, "a lane per load in every block");
        const uint32_t mine = ((lane & 2) ? m23 : m01) >> ((lane & 1) ? 16 : 0) << 16;
        float s_mine = 1.0f, y_mine = 1.0f;
        if (mine != 0u) {
            s_mine = __fdiv_rn(__uint_as_float(mine), 448.0f);
            y_mine = __frcp_rn(s_mine);
        }
        if (lane % kLanesPerBlock < 4) sc[(lane & 3) * kBlkPerIt + lane / kLanesPerBlock][static_cast<int>(row - row0)] = s_mine;
#pragma unroll
        for (int it = 0; it < kQIters; ++it) {
            const int64_t col = col0 + it * 256 + lane * 8;
            const float s = __shfl_sync(0xffffffffu, s_mine, it, kLanesPerBlock);
            const float y = __shfl_sync(0xffffffffu, y_mine, it, kLanesPerBlock);
            if (row < rows && col < cols) *reinterpret_cast<uint2*>(codes + row * ldq + col) = quantize_values(raw[it], s, y);
        }
    });
    __syncthreads();
    const int64_t kb0 = col0 / BLOCK, nkb = cols / BLOCK;
    for (int idx = threadIdx.x; idx < kBlocksPerTile * kRows; idx += kQThreads) {
        const int kb_l = idx / kRows, r_l = idx % kRows;
        if (kb0 + kb_l < nkb && row0 + r_l < rows) scales[(kb0 + kb_l) * lds + row0 + r_l] = sc[kb_l][r_l];
    }
}

// ------------------------------------------------------------------------------------------------
// The same quantisation for a matrix stored with the blocks running DOWN its columns (an LM head kept as [d, V]):
// block kb of column v is x[kb B .. kb B + B - 1, v].  The codes leave transposed, [V, ldq] with the block elements
// contiguous, which is the K-major operand the rollout pass wants; the scales leave block-major [d / B, lds] as always.
// A CTA stages a tile of 128 rows x 128 columns in shared memory (16-byte loads along the rows).  Thread (vp, h) then holds
// rows 32 h .. 32 h + 31 of the column pair vp in registers, one 32-bit word per row, so that maxima and divisions work on
// both columns per instruction; the codes go back through the same shared memory and leave as whole 128-byte rows.
// (One thread per column and 16-bit reads, twice per element, took 574 us for a 4096 x 151936 head.)
// ------------------------------------------------------------------------------------------------
constexpr int kQcTile = 128;
constexpr int kQcPitch = kQcTile / 2 + 4;      // 32-bit words per staged row: 272 bytes
constexpr int kQcOutPitch = kQcTile + 16;      // bytes per column of codes
static_assert(kQcTile * kQcOutPitch <= kQcTile * kQcPitch * 4, "the codes reuse the staged tile's memory");

template <int BLOCK>
__global__ void __launch_bounds__(256) quantize_cols_kernel(const __nv_bfloat16* __restrict__ x, int64_t K, int64_t N, int64_t ld,
                                                            uint8_t* __restrict__ codes, int64_t ldq,
                                                            float* __restrict__ scales, int64_t lds) {
    __shared__ __align__(16) uint32_t tile[kQcTile][kQcPitch];
    __shared__ uint32_t part_max[4][kQcTile / 2];
    pdl_enter();
    const int tid = threadIdx.x;
    const int64_t k0 = static_cast<int64_t>(blockIdx.y) * kQcTile, v0 = static_cast<int64_t>(blockIdx.x) * kQcTile;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const int c = tid + 256 * i, r = c >> 4, c8 = (c & 15) * 8;
        uint4 raw = make_uint4(0, 0, 0, 0);
        if (v0 + c8 < N) raw = __ldg(reinterpret_cast<const uint4*>(x + (k0 + r) * ld + v0 + c8));
        *reinterpret_cast<uint4*>(&tile[r][c8 / 2]) = raw;
    }
    __syncthreads();
    const int vp = tid & 63, h = tid >> 6;
    uint32_t w[32], m = 0;
#pragma unroll
    for (int j = 0; j < 32; ++j) {
        w[j] = tile[32 * h + j][vp];
        m = __vmaxu2(m, w[j] & 0x7FFF7FFFu);
    }
    part_max[h][vp] = m;
    __syncthreads();                                        // the maxima are there, and nobody reads the tile any more
    if (BLOCK == 64) m = __vmaxu2(m, part_max[h ^ 1][vp]);
    if (BLOCK == 128) m = __vmaxu2(__vmaxu2(part_max[0][vp], part_max[1][vp]), __vmaxu2(part_max[2][vp], part_max[3][vp]));
    const uint32_t mlo = m & 0xFFFFu, mhi = m >> 16;
    F2 s = {1.0f, 1.0f};
    if (mlo != 0u) s.x = __fdiv_rn(__uint_as_float(mlo << 16), 448.0f);
    if (mhi != 0u) s.y = __fdiv_rn(__uint_as_float(mhi << 16), 448.0f);
    const F2 y = {__frcp_rn(s.x), __frcp_rn(s.y)}, ns = {-s.x, -s.y};
    const bool fast = s.x > 0x1p-100f && s.x < 0x1p100f && s.y > 0x1p-100f && s.y < 0x1p100f;
    uint8_t* out = reinterpret_cast<uint8_t*>(&tile[0][0]);
#pragma unroll
    for (int g = 0; g < 2; ++g) {                           // sixteen rows of both columns
        uint32_t c0[4], c1[4];
#pragma unroll
        for (int p = 0; p < 8; ++p) {
            F2 q[2];
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                const uint32_t word = w[16 * g + 2 * p + i];
                const F2 v = {__uint_as_float(word << 16), __uint_as_float(word & 0xFFFF0000u)};
                if (fast) {                                  // as in quantize_values, both columns at once
                    const F2 t = mul2(v, y);
                    const F2 u = fma2(fma2(ns, t, v), y, t);
                    q[i] = F2{copysignf(u.x, v.x), copysignf(u.y, v.y)};
                } else {
                    q[i] = F2{slow_div(v.x, s.x), slow_div(v.y, s.y)};
                }
            }
            const uint32_t e0 = cvt_e4m3x2(q[1].x, q[0].x), e1 = cvt_e4m3x2(q[1].y, q[0].y);
            if (p & 1) { c0[p >> 1] |= e0 << 16; c1[p >> 1] |= e1 << 16; }
            else { c0[p >> 1] = e0; c1[p >> 1] = e1; }
        }
        *reinterpret_cast<uint4*>(out + (2 * vp) * kQcOutPitch + 32 * h + 16 * g) = make_uint4(c0[0], c0[1], c0[2], c0[3]);
        *reinterpret_cast<uint4*>(out + (2 * vp + 1) * kQcOutPitch + 32 * h + 16 * g) = make_uint4(c1[0], c1[1], c1[2], c1[3]);
    }
    if (h % (BLOCK / 32) == 0 && v0 + 2 * vp < N) {          // N is a multiple of 8: both columns are in
        float* dst = scales + ((k0 + 32 * h) / BLOCK) * lds + v0 + 2 * vp;
        dst[0] = s.x;
        dst[1] = s.y;
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int c = tid + 256 * i, col = c >> 3, part = (c & 7) * 16;
        if (v0 + col < N)
            *reinterpret_cast<uint4*>(codes + (v0 + col) * ldq + k0 + part) = *reinterpret_cast<const uint4*>(out + col * kQcOutPitch + part);
    }
}

// ------------------------------------------------------------------------------------------------
// Microscaling FP8: 32 consecutive elements share a power-of-two scale 2^X, X = floor(log2 amax) - 8, stored as the
// biased exponent X + 127 (clamped to 0..254; 127 for an all-zero block); the elements are x / 2^X on the E4M3 grid
// (round to nearest even, saturating).  With bf16 inputs everything is exact integer work on exponent fields: the
// block's amax pattern gives the scale code, and the multiplier 2^-X is a float built from its exponent field.
// Four lanes (8 elements each) form a block.  The scale codes leave in the order the block-scaled MMA wants them:
// chunks of 128 rows x 4 blocks, byte (r % 32) * 16 + ((r % 128) / 32) * 4 + kb % 4 of chunk (r / 128, kb / 4); the two
// chunks of a 256-row group are adjacent: chunk start ((r / 256) * (cols / 128) + kb / 4) * 1024 + ((r % 256) / 128) * 512.
// ------------------------------------------------------------------------------------------------
// Microscaling FP4: the same with E2M1 elements (X = floor(log2 amax) - 2), two codes per byte, the element with the lower
// index in the low nibble; a lane turns 8 elements into 4 bytes.  The four scale bytes of a row and 128 columns lie next to
// each other and are written as one word.  Rows that pad the last 256-row group carry the neutral scale 127.
// ------------------------------------------------------------------------------------------------
__device__ __forceinline__ uint32_t cvt_e2m1x2(float hi, float lo) {
    uint32_t r;
    asm("{\n\t.reg .b8 t;\n\tcvt.rn.satfinite.e2m1x2.f32 t, %1, %2;\n\tcvt.u32.u8 %0, t;\n\t}" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}

template <bool FP4, int RPW>
__global__ void __launch_bounds__(kQThreads) quantize_mx_kernel(const __nv_bfloat16* __restrict__ x, int64_t rows,
                                                                             int64_t padded_rows, int64_t cols, int64_t ld,
                                                                             uint8_t* __restrict__ codes, int64_t ldq,
                                                                             uint8_t* __restrict__ scales, unsigned tiles_x) {
    pdl_enter();
    const int lane = threadIdx.x & 31;
    const int64_t nk4 = cols / 128;
    auto scale_word = [&](int64_t row, int64_t k4) {
        return reinterpret_cast<uint32_t*>(scales + ((row >> 8) * nk4 + k4) * 1024 + ((row >> 7) & 1) * 512 + (row & 31) * 16 + ((row & 127) >> 5) * 4);
    };
    const QuantTile tile = quant_tile<RPW>(tiles_x);
    const int64_t col0 = tile.col0;
    if (tile.last_rows)
        for (int64_t i = threadIdx.x; i < (padded_rows - rows) * 8; i += kQThreads)
            if (col0 / 128 + i % 8 < nk4) *scale_word(rows + i / 8, col0 / 128 + i % 8) = 0x7F7F7F7Fu;
    walk_rows<RPW>(x, rows, cols, ld, tile.row0, col0, [&](int64_t row, const uint4 (&raw)[kQIters]) {
            if (row >= rows) return;
            uint32_t pair = 0;
#pragma unroll
            for (int it = 0; it < kQIters; ++it) {
                if (it % 2 == 0) pair = block_amax_pair<32>(raw[it], raw[it + 1]);
                const int64_t col = col0 + it * 256 + lane * 8;
                const uint32_t w[4] = {raw[it].x, raw[it].y, raw[it].z, raw[it].w};
                const uint32_t m = it % 2 == 0 ? pair & 0xFFFFu : pair >> 16;
                const int e = static_cast<int>(m >> 7);         // biased exponent of amax (0 for zero and subnormals)
                const int code = m == 0u ? 127 : max(e - (FP4 ? 2 : 8), 0);
                const float mult = __uint_as_float(static_cast<uint32_t>(254 - code) << 23);      // 2^(127 - code), exact
                // the sixteen lanes of 128 columns hold four blocks: their codes become one word
                uint32_t word = static_cast<uint32_t>(code) << (8 * ((lane >> 2) & 3));
                word |= __shfl_xor_sync(0xffffffffu, word, 4);
                word |= __shfl_xor_sync(0xffffffffu, word, 8);
                if (col >= cols) continue;                      // cols is a multiple of 128: all sixteen lanes agree
                if (FP4) {
                    uint32_t out = 0;
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        out |= cvt_e2m1x2(__uint_as_float(w[i] & 0xFFFF0000u) * mult, __uint_as_float(w[i] << 16) * mult) << (8 * i);
                    *reinterpret_cast<uint32_t*>(codes + row * ldq + col / 2) = out;
                } else {
                    float q[8];
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        q[2 * i] = __uint_as_float(w[i] << 16) * mult;
                        q[2 * i + 1] = __uint_as_float(w[i] & 0xFFFF0000u) * mult;
                    }
                    uint2 out;
                    out.x = static_cast<uint32_t>(cvt_e4m3x2(q[1], q[0])) | (static_cast<uint32_t>(cvt_e4m3x2(q[3], q[2])) << 16);
                    out.y = static_cast<uint32_t>(cvt_e4m3x2(q[5], q[4])) | (static_cast<uint32_t>(cvt_e4m3x2(q[7], q[6])) << 16);
                    *reinterpret_cast<uint2*>(codes + row * ldq + col) = out;
                }
                if ((lane & 15) == 0) *scale_word(row, col / 128) = word;
            }
    });
}

// ------------------------------------------------------------------------------------------------
// Per-tensor dynamic scaling: one scale for the whole matrix.  Pass 1 folds max|x| (as a bf16 bit pattern; the
// patterns of non-negative values order like the values, so an integer atomicMax is exact and order-free)
// into the word that will hold the scale, pass 2 turns it into s = amax / 448, pass 3 quantises.
// ------------------------------------------------------------------------------------------------
template <int RPW>
__global__ void __launch_bounds__(kQThreads) tensor_amax_kernel(const __nv_bfloat16* __restrict__ x, int64_t rows, int64_t cols, int64_t ld,
                                                                uint32_t* __restrict__ amax_bits, unsigned tiles_x) {
    __shared__ uint32_t block_max;
    if (threadIdx.x == 0) block_max = 0;
    pdl_enter();
    __syncthreads();
    uint32_t m = 0;
    const QuantTile tile = quant_tile<RPW>(tiles_x);
    walk_rows<RPW>(x, rows, cols, ld, tile.row0, tile.col0,
                   [&](int64_t, const uint4 (&raw)[kQIters]) {
#pragma unroll
                       for (int it = 0; it < kQIters; ++it)
                           m = __vmaxu2(m, __vmaxu2(__vmaxu2(raw[it].x & 0x7FFF7FFFu, raw[it].y & 0x7FFF7FFFu),
                                                    __vmaxu2(raw[it].z & 0x7FFF7FFFu, raw[it].w & 0x7FFF7FFFu)));
                   });
    m = __reduce_max_sync(0xffffffffu, max(m & 0xFFFFu, m >> 16));
    if ((threadIdx.x & 31) == 0) atomicMax(&block_max, m);
    __syncthreads();
    if (threadIdx.x == 0 && block_max != 0u) atomicMax(amax_bits, block_max);
}

__global__ void tensor_scale_kernel(uint32_t* scale_word) {
    pdl_enter();
    const uint32_t m = *scale_word;                        // bf16 pattern of max|x|
    const float s = (m == 0u) ? 1.0f : __fdiv_rn(__uint_as_float(m << 16), 448.0f);
    *reinterpret_cast<float*>(scale_word) = s;
}

// The rows in the opposite order of the maximum's: what that pass read last is still in L2.
template <int RPW>
__global__ void __launch_bounds__(kQThreads) tensor_quantize_kernel(const __nv_bfloat16* __restrict__ x, int64_t rows, int64_t cols, int64_t ld,
                                                                    uint8_t* __restrict__ codes, int64_t ldq,
                                                                    const float* scale, unsigned tiles_x) {
    pdl_enter();
    const float s = *scale;
    const float y = __frcp_rn(s);
    const QuantTile tile = quant_tile<RPW>(tiles_x);
    const int64_t col0 = tile.col0 + (threadIdx.x & 31) * 8;
    walk_rows<RPW>(x, rows, cols, ld, static_cast<int64_t>((gridDim.x - 1) / tiles_x) * (kQWarps * RPW) - tile.row0, tile.col0, [&](int64_t row, const uint4 (&raw)[kQIters]) {
                       if (row >= rows) return;
#pragma unroll
                       for (int it = 0; it < kQIters; ++it)
                           if (col0 + it * 256 < cols)
                               *reinterpret_cast<uint2*>(codes + row * ldq + col0 + it * 256) = quantize_values(raw[it], s, y);
                   });
}

// ------------------------------------------------------------------------------------------------
// Merge of the per-split (max, sum-exp, target-logit) triples into lp and lse.
// ------------------------------------------------------------------------------------------------
// A block merges 32 rows: lane = row (coalesced), the parts are dealt out to the eight warps and each warp's running
// (max, sum) goes through shared memory to warp 0, in warp order.  With one thread per row the up to 296 parts of a small
// batch were a chain of dependent loads.
constexpr int kCombWarps = 8;
struct MergeState {
    float m[kCombWarps][kMergeRows], s[kCombWarps][kMergeRows], z[kCombWarps][kMergeRows];
};
// One warp's share of the parts of row t (a lane's own).
__device__ __forceinline__ void merge_parts(const CombineJob& job, int64_t part_ld, int64_t t, bool live, int warp, MergeState& st) {
    const float *part_m = job.part_m, *part_s = job.part_s, *part_z = job.part_z;
    const int nparts = job.nparts, lane = threadIdx.x & 31;
    float M = -INFINITY, S = 0.f, Z = -INFINITY;
    if (live) {
#pragma unroll 4
        for (int j = warp; j < nparts; j += kCombWarps) {
            const float m = part_m[j * part_ld + t], s = part_s[j * part_ld + t];
            Z = fmaxf(Z, part_z[j * part_ld + t]);
            const float n = fmaxf(M, m);
            S = S * expf(M - n) + s * expf(m - n);
            M = n;
        }
    }
    st.m[warp][lane] = M;
    st.s[warp][lane] = S;
    st.z[warp][lane] = Z;
}
struct MergedRow { float lp, lse; };
// One warp, behind a barrier: the shares of the eight warps in their order, written to lp and lse (t < T).
__device__ __forceinline__ MergedRow merge_finish(const CombineJob& job, int64_t t, bool live, uint32_t* status, const MergeState& st) {
    const int lane = threadIdx.x & 31;
    float out_lp = 0.f, out_lse = 0.f;
    if (live) {
        float M = st.m[0][lane], Z = st.z[0][lane], S = 0.f;
#pragma unroll
        for (int w = 1; w < kCombWarps; ++w) {
            M = fmaxf(M, st.m[w][lane]);
            Z = fmaxf(Z, st.z[w][lane]);
        }
#pragma unroll
        for (int w = 0; w < kCombWarps; ++w)
            if (w < job.nparts) S += st.s[w][lane] * expf(st.m[w][lane] - M);
        out_lse = M + logf(S);
        out_lp = Z == -INFINITY ? 0.f : Z - out_lse;    // no target logit: token id out of range, flagged by the producer kernel
        if (!isfinite(out_lse) || !isfinite(out_lp)) {
            // a non-finite hidden state or weight reached this row: flag it, give it the neutral log-prob, and mark its
            // log-sum-exp so that the backward pass leaves the row out (gradient factor 0)
            if (status) atomicOr(status, AIS_FLAG_NONFINITE);
            out_lp = 0.f;
            out_lse = __int_as_float(0x7fc00000);
        }
    }
    job.lp[t] = out_lp;
    if (job.lse) job.lse[t] = out_lse;
    return {out_lp, out_lse};
}

__global__ void __launch_bounds__(32 * kCombWarps) combine_kernel(const CombineJob j0, const CombineJob j1, int njobs, int64_t part_ld,
                                                                  const uint8_t* __restrict__ mask, int64_t T, uint32_t* status,
                                                                  const AdvJob adv) {
    pdl_enter();
    if (static_cast<int>(blockIdx.y) == njobs) {                 // the row of blocks behind the merges
        for (int s = blockIdx.x * blockDim.x + threadIdx.x; s < adv.S; s += gridDim.x * blockDim.x) run_advantage(adv, s);
        return;
    }
    __shared__ MergeState st;
    const CombineJob job = blockIdx.y == 0 ? j0 : j1;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t t = static_cast<int64_t>(blockIdx.x) * kMergeRows + lane;
    const bool live = t < T && mask[t] != 0;
    merge_parts(job, part_ld, t, live, warp, st);
    __syncthreads();
    if (warp != 0 || t >= T) return;
    merge_finish(job, t, live, status, st);
}

// ------------------------------------------------------------------------------------------------
// Segmented reductions: valid rows per sequence and group-relative advantages (Eq. grpo_adv).
// ------------------------------------------------------------------------------------------------
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    return v;
}

// Block-wide sum in a fixed order (lanes by butterfly, then warps 0..n-1 serially); result valid in thread 0.
__device__ double block_sum(double v, double* scratch /*[32]*/) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    v = warp_sum(v);
    __syncthreads();
    if (lane == 0) scratch[warp] = v;
    __syncthreads();
    double tot = 0.0;
    if (threadIdx.x == 0) {
        const int nw = (blockDim.x + 31) >> 5;
        for (int i = 0; i < nw; ++i) tot += scratch[i];
    }
    return tot;
}

// Sum of partials[b * stride + offset] over b < nblocks by one warp, in a fixed order: lane l takes blocks l, l + 32, ...
// (loaded sixteen at a time so that the loads overlap), then the shuffle tree of warp_sum.
__device__ __forceinline__ double warp_ordered_sum(const double* partials, int nblocks, int stride, int offset, int lane) {
    double acc = 0.0;
    for (int base = lane; base < nblocks; base += 32 * 16) {
        double v[16];
#pragma unroll
        for (int j = 0; j < 16; ++j) {
            const int b = base + 32 * j;
            v[j] = b < nblocks ? __ldcg(partials + b * stride + offset) : 0.0;      // written by other blocks, possibly of this launch
        }
#pragma unroll
        for (int j = 0; j < 16; ++j) acc += v[j];
    }
    return warp_sum(acc);
}

// The same sums for N values at once (same order each): two barriers for all of them instead of two for each; results in
// out[0 .. N-1], valid for every thread after the call.  Blocks of kDiagThreads.
template <int N>
__device__ __forceinline__ void block_sums(double (&v)[N], double (*scratch)[kDiagThreads / 32] /*[N]*/, double* out) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
    for (int i = 0; i < N; ++i) {
        v[i] = warp_sum(v[i]);
        if (lane == 0) scratch[i][warp] = v[i];
    }
    __syncthreads();
    if (threadIdx.x < N) {
        double tot = 0.0;
#pragma unroll
        for (int i = 0; i < kDiagThreads / 32; ++i) tot += scratch[threadIdx.x][i];
        out[threadIdx.x] = tot;
    }
    __syncthreads();
}

// True in every thread of the block that arrives last at `ticket` (zeroed before the launch): that block sees what all
// blocks wrote before their arrival.
__device__ __forceinline__ bool last_block(uint32_t* ticket) {
    __shared__ bool last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(ticket, 1u) == gridDim.x - 1;
    __syncthreads();
    __threadfence();
    return last;
}

// Valid rows of each sequence: one warp per sequence, 4 mask bytes per lane and load where the row range allows it.
__global__ void __launch_bounds__(256) seq_count_kernel(const uint8_t* __restrict__ mask, const int32_t* __restrict__ seq_offsets,
                                                         int S, int32_t* __restrict__ n_valid_seq, uint32_t* __restrict__ ticket) {
    pdl_enter();
    if (blockIdx.x == 0 && threadIdx.x == 0) *ticket = 0;
    const int s = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (s >= S) return;
    const int lane = threadIdx.x & 31;
    const int64_t b = seq_offsets[s], e = seq_offsets[s + 1];
    const uintptr_t base = reinterpret_cast<uintptr_t>(mask);
    const int64_t b4 = b + static_cast<int64_t>((4 - ((base + b) & 3)) & 3);          // first row on a 4-byte boundary
    int cnt = 0;
    for (int64_t t = b + lane; t < (b4 < e ? b4 : e); t += 32) cnt += mask[t] != 0;
    const int64_t nwords = b4 < e ? (e - b4) / 4 : 0;
    for (int64_t i = lane; i < nwords; i += 32) {
        const uint32_t w = *reinterpret_cast<const uint32_t*>(mask + b4 + 4 * i);
        cnt += ((w & 0xFFu) != 0) + ((w & 0xFF00u) != 0) + ((w & 0xFF0000u) != 0) + ((w & 0xFF000000u) != 0);
    }
    for (int64_t t = b4 + 4 * nwords + lane; t < e; t += 32) cnt += (t >= b4 && mask[t] != 0);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) cnt += __shfl_xor_sync(0xffffffffu, cnt, off);
    if (lane == 0) n_valid_seq[s] = cnt;
}

__global__ void adv_kernel(const AdvJob job) {
    pdl_enter();
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s < job.S) run_advantage(job, s);
}

// Sequence-level importance weight (Eq. is-weight): log w(x) = sum over the valid rows of a sequence of
// lp_train - lp_roll.  One warp per sequence, double accumulation in a fixed order.
__global__ void __launch_bounds__(256) seq_logw_kernel(const float* lp_train, const float* lp_roll,
                                                        const uint8_t* __restrict__ mask, const int32_t* __restrict__ seq_offsets,
                                                        int S, float* __restrict__ seq_logw) {
    pdl_enter();
    const int s = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (s >= S) return;
    const int lane = threadIdx.x & 31;
    double acc = 0.0;
    for (int64_t t = static_cast<int64_t>(seq_offsets[s]) + lane; t < seq_offsets[s + 1]; t += 32)
        if (mask[t]) acc += static_cast<double>(lp_train[t]) - static_cast<double>(lp_roll[t]);
    acc = warp_sum(acc);
    if (lane == 0) seq_logw[s] = static_cast<float>(acc);
}

__device__ __forceinline__ int seq_of_row(const int32_t* __restrict__ seq_offsets, int S, int64_t t) {
    int lo = 0, hi = S;                 // largest s with seq_offsets[s] <= t
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (static_cast<int64_t>(seq_offsets[mid]) <= t) lo = mid; else hi = mid;
    }
    return lo;
}

// The sequences of rows t_first and t_last (t_first <= t_last) found by a whole warp, 32 probes at a time: two rounds of loads
// for up to 1,024 sequences where the binary search of a single thread is a chain of ten.
__device__ __forceinline__ int2 seqs_of_rows_warp(const int32_t* __restrict__ seq_offsets, int S, int64_t t_first, int64_t t_last) {
    const int lane = threadIdx.x & 31;
    int lo[2] = {0, 0}, hi[2] = {S, S};
    const int64_t t[2] = {t_first, t_last};
    while (hi[0] - lo[0] > 1 || hi[1] - lo[1] > 1) {
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const int step = (hi[k] - lo[k] + 31) / 32;
            const int at = lo[k] + (lane + 1) * step;
            const int n = __popc(__ballot_sync(0xffffffffu, at < hi[k] && static_cast<int64_t>(seq_offsets[at < hi[k] ? at : lo[k]]) <= t[k]));
            lo[k] += n * step;
            hi[k] = min(lo[k] + step, hi[k]);
        }
    }
    return make_int2(lo[0], lo[1]);
}
// The largest s in [range.x, range.y] whose first row is not behind t.
__device__ __forceinline__ int seq_in_range(const int32_t* __restrict__ seq_offsets, int2 range, int64_t t) {
    return range.x == range.y ? range.x : range.x + seq_of_row(seq_offsets + range.x, range.y - range.x + 1, t);
}

// Population variance E[x^2] - E[x]^2 in fp64.  The sums reach this point with fp64 accuracy relative to the spread of the data
// (add_run), so what is left is the rounding of the fp64 additions themselves: a result below 2^-44 of the mean square (a few
// hundred ulps of it; a standard deviation below 2.4e-7 of the rms value) is that rounding and is reported as exactly zero.
__device__ __forceinline__ double population_variance(double N, double sum, double sumsq) {
    const double mean = sum / N, ms = sumsq / N;
    const double v = ms - mean * mean;
    return v > ms * 0x1p-44 ? v : 0.0;
}

// The diagnostics and alpha from the ten sums over the batch.
__device__ __noinline__ void derive_diag(const double* m, const ais_params& p, ais_diag* __restrict__ diag) {
    ais_diag d;
    d.status_flags = 0;
    d.reserved = 0;
    d.loss = 0.0;
    d.kl_ref = 0.0;
    const double N = m[0];
    d.n_valid = N;
    if (N <= 0.0) {
        d.mean_w = 1.0; d.cv2 = 0.0; d.ess = 0.0; d.ess_ratio = 1.0; d.alpha_ess = 1.0; d.d_bar = 0.0;
        d.alpha_mis = 0.0; d.std_A = 0.0; d.std_Aw = 0.0; d.delta_sigma = 0.0; d.alpha_var = 0.0;
        d.alpha_adaptive = 0.0; d.kl_k1 = 0.0; d.mean_abs_dp = 0.0;
        d.status_flags |= AIS_FLAG_EMPTY;
    } else {
        auto variance = [&](double sum, double sumsq) { return population_variance(N, sum, sumsq); };
        const double mu = m[1] / N;
        const double var = variance(m[1], m[2]);
        d.mean_w = mu;
        d.cv2 = var / (mu * mu);
        d.ess = m[1] * m[1] / m[2];
        d.ess_ratio = d.ess / N;
        d.alpha_ess = 1.0 / sqrt(1.0 + d.cv2);
        d.d_bar = m[3] / N;
        d.alpha_mis = fmin(1.0, d.d_bar / static_cast<double>(p.delta));
        d.std_A = sqrt(variance(m[4], m[5]));
        d.std_Aw = sqrt(variance(m[6], m[7]));
        d.delta_sigma = d.std_Aw / (d.std_A + static_cast<double>(p.eps));
        d.alpha_var = fmax(0.0, (d.delta_sigma - static_cast<double>(p.gamma)) / static_cast<double>(p.gamma));
        d.alpha_adaptive = fmin(1.0, fmax(0.0, d.alpha_ess - static_cast<double>(p.beta_var) * d.alpha_var)) * d.alpha_mis;
        d.kl_k1 = m[8] / N;
        d.mean_abs_dp = m[9] / N;
    }
    if (isnan(N)) d.status_flags |= AIS_FLAG_TIMEOUT;       // a block of the moments kernel gave up on a bounded wait
    d.alpha = isnan(p.alpha_override) ? d.alpha_adaptive : static_cast<double>(p.alpha_override);
    *diag = d;
}

// alpha alone, the same operations by one warp: lane 0 follows the weights, lanes 1 and 2 the two standard deviations, lane 3
// the log-ratio gap, so that the chain is five divisions and a square root long instead of fifteen.
__device__ __forceinline__ double alpha_by_warp(const double* m, const ais_params& p, int lane) {
    if (!isnan(p.alpha_override)) return static_cast<double>(p.alpha_override);
    const double N = m[0];
    if (N <= 0.0) return 0.0;
    const int at = lane == 0 ? 1 : lane == 1 ? 4 : lane == 2 ? 6 : 3;
    const double first = m[at] / N;                                                      // mu, ..., d_bar
    const double var = lane < 3 ? population_variance(N, m[at], m[at + 1]) : 0.0;
    const double root = sqrt(lane == 0 ? 1.0 + var / (first * first) : var);
    const double std_A = __shfl_sync(0xffffffffu, root, 1), std_Aw = __shfl_sync(0xffffffffu, root, 2);
    const double num = lane == 0 ? 1.0 : lane == 3 ? first : std_Aw;
    const double den = lane == 0 ? root : lane == 3 ? static_cast<double>(p.delta) : std_A + static_cast<double>(p.eps);
    const double q = num / den;                                                          // alpha_ess, delta_sigma, ..., d_bar / delta
    const double alpha_ess = __shfl_sync(0xffffffffu, q, 0), delta_sigma = __shfl_sync(0xffffffffu, q, 1);
    const double alpha_mis = fmin(1.0, __shfl_sync(0xffffffffu, q, 3));
    const double alpha_var = fmax(0.0, (delta_sigma - static_cast<double>(p.gamma)) / static_cast<double>(p.gamma));
    return fmin(1.0, fmax(0.0, alpha_ess - static_cast<double>(p.beta_var) * alpha_var)) * alpha_mis;
}

// Totals over the blocks of a batch reduction, formed by every block of the kernel that follows it (256 threads): thread
// (slice, moment) adds every 25th block's value in block order, ten threads add the slices.  The kernel that produced the
// partial sums is over by then, so nothing has to count arrivals.  Result in t.moments, valid for every thread.
// Each block reads at most 47 KB from L2.  Measured (diagnostics of 1.48 M / 200 k rows, back to back): the last block of the
// moments kernel adding up, deriving alpha and a third kernel reading it 22.1 / 13.5 us, this 18.5 / 12.4 us; the rectifying
// kernel on 444, 296 and 148 blocks instead of 592 18.7, 19.2 and 21.0 us.
constexpr int kSums = 10;                                // slots 10 and 11 are no moments
constexpr int kSlices = kDiagThreads / kSums;
struct Totals {
    double slices[kSlices][kSums];
    double moments[kNumMoments];
    float alpha;
};
__device__ __forceinline__ void form_totals(const TotalsJob& job, Totals& t) {
    const int tid = threadIdx.x;
    if (tid < kSlices * kSums) {
        double acc = 0.0;
        for (int b0 = tid / kSums; b0 < job.blocks; b0 += 12 * kSlices) {
            double v[12];
#pragma unroll
            for (int j = 0; j < 12; ++j) v[j] = b0 + j * kSlices < job.blocks ? job.partials[(b0 + j * kSlices) * kNumMoments + tid % kSums] : 0.0;
#pragma unroll
            for (int j = 0; j < 12; ++j) acc += v[j];
        }
        t.slices[tid / kSums][tid % kSums] = acc;
    }
    __syncthreads();
    if (tid < kNumMoments) {
        double tot = 0.0;
        if (tid < kSums) {
#pragma unroll
            for (int k = 0; k < kSlices; ++k) tot += t.slices[k][tid];
        }
        t.moments[tid] = tot;
    }
    __syncthreads();
}
// alpha of the batch, for every thread; block 0 also writes the diagnostics.
__device__ __forceinline__ float form_alpha(const TotalsJob& job, Totals& t) {
    form_totals(job, t);
    if (threadIdx.x < 32) {
        const double alpha = alpha_by_warp(t.moments, job.params, threadIdx.x);
        if (threadIdx.x == 0) t.alpha = static_cast<float>(alpha);
    } else if (threadIdx.x == 32 && blockIdx.x == 0) {
        derive_diag(t.moments, job.params, job.diag);
    }
    __syncthreads();
    return t.alpha;
}
// The totals on their own: the sums (ais_diag_moments) or, for a batch without rows, the diagnostics.
__global__ void __launch_bounds__(kDiagThreads) totals_kernel(const __grid_constant__ TotalsJob job, double* __restrict__ moments) {
    __shared__ Totals t;
    pdl_enter();
    form_totals(job, t);
    if (moments != nullptr && threadIdx.x < kNumMoments) moments[threadIdx.x] = t.moments[threadIdx.x];
    if (job.diag != nullptr && threadIdx.x == 0) derive_diag(t.moments, job.params, job.diag);
}

// ------------------------------------------------------------------------------------------------
// Whole-batch masked moments in double precision, fixed grid and fixed summation order.
//   0 N   1 sum w   2 sum w^2   3 sum |D|   4 sum A   5 sum A^2   6 sum Aw   7 sum (Aw)^2
//   8 sum (lp_roll - lp_train)   9 sum |exp(lp_train) - exp(lp_roll)|
// ------------------------------------------------------------------------------------------------
// Rows are read VEC at a time (16-byte loads of the two log-prob vectors, one 4-byte load of the mask); the
// sequence of a group's first row comes from a binary search and the following rows only step forward.  The
// exponentials are evaluated in fp32 (the inputs are fp32 and the sums need seven digits at most), the sums
// themselves in fp64.  Two groups are in flight per thread so that the fixed grid keeps HBM busy on long batches.
// rho - 1 = e^x - 1 for a run of n rows.  When every |x| of the run is at most 2^-6 a short series gives it to fp32
// accuracy RELATIVE TO ITSELF (e^x - 1 from a rounded e^x would be good to 1e-7 absolute only, i.e. to a thousandth of a
// weight that differs from 1 by 1e-4); otherwise the fast exponential is used, as everywhere else in these kernels.
template <int N>
__device__ __forceinline__ void rho_minus_one(const float (&x)[N], float (&u)[N]) {
    float amax = 0.f;
#pragma unroll
    for (int j = 0; j < N; ++j) amax = fmaxf(amax, fabsf(x[j]));
    if (amax <= 0x1p-6f) {
#pragma unroll
        for (int j = 0; j < N; ++j)
            u[j] = x[j] * fmaf(x[j], fmaf(x[j], fmaf(x[j], 1.0f / 24.0f, 1.0f / 6.0f), 0.5f), 1.0f);
    } else {
#pragma unroll
        for (int j = 0; j < N; ++j) {
            float e;
            asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e) : "f"(x[j] * 1.4426950408889634f));
            u[j] = e - 1.0f;
        }
    }
}

// Sums of w and w^2 over a short run of rows, in double precision, from fp32 sums of shifted values.  The weights
// enter as u = w - 1 (rho_minus_one above, truncated at C - 1); the run is summed as v = u - p and v^2 about the pivot
// p = u of its first valid row:  with P = 1 + p,  sum w = n P + sum v  and  sum w^2 = n P^2 + 2 P sum v + sum v^2.
// The fp32 roundings then scale with the spread of the run and with |w - 1|, not with the size of w, so that the
// variance formed later as E[w^2] - E[w]^2 in fp64 keeps its digits when the weights differ by 1e-4 of their size,
// and is exactly zero when they are all equal.  All rows of the run share the advantage A.
//   acc: 0 N   1 sum w   2 sum w^2   4 sum A   5 sum A^2   6 sum A w   7 sum (A w)^2
__device__ __forceinline__ void add_run(double* acc, int n, float p, float sv, float sv2, float A) {
    const double nd = static_cast<double>(n), P = 1.0 + static_cast<double>(p), svd = static_cast<double>(sv);
    const double Ad = static_cast<double>(A);
    const double sw = fma(nd, P, svd);
    const double sw2 = static_cast<double>(sv2) + P * fma(nd, P, 2.0 * svd);
    acc[0] += nd;
    acc[1] += sw;
    acc[2] += sw2;
    acc[4] = fma(Ad, nd, acc[4]);
    acc[5] = fma(Ad * Ad, nd, acc[5]);
    acc[6] = fma(Ad, sw, acc[6]);
    acc[7] = fma(Ad * Ad, sw2, acc[7]);
}

// The merge of both passes and the batch moments in one kernel, for batches of up to kMergeMomentRows rows: the sixteen warps
// merge 32 rows as combine_kernel does (eight warps per pass, the same order), then one warp forms the terms of its 32 rows
// and their sums in fp64, one row of partial sums per block.  A small batch is a chain of launches, and the moments kernel (start,
// walk, fp64 sums) is one of them, while every row's log-probs are in a register here.  Steps of d = 256, V = 1024 with the moments
// kernel and without: 512 rows 42.1 -> 39.6 us, 4,096 61.2 -> 58.2, 9,217 68.8 -> 66.2, 12,288 79.7 -> 77.6, 18,944 87.7 -> 86.4; log-probs
// and diagnostics alone 4,096 31.1 -> 28.7, 18,944 51.7 -> 51.1.  The limit is what the buffer of partial sums holds (kDiagBlocks rows of
// them, of which the moments kernel leaves one per 2,048 rows); the gain shrinks towards it because every block behind adds them up.
__global__ void __launch_bounds__(2 * 32 * kCombWarps) merge_moments_kernel(const CombineJob j0, const CombineJob j1, int64_t part_ld,
                                                                            const uint8_t* __restrict__ mask, int64_t T, uint32_t* status,
                                                                            const MomentsJob mj) {
    __shared__ MergeState st[2];
    __shared__ float lp_roll[kMergeRows];
    __shared__ int2 range;
    pdl_enter();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, pass = warp / kCombWarps;
    const int64_t t0 = static_cast<int64_t>(blockIdx.x) * kMergeRows, t = t0 + lane;
    const int64_t last = t0 + kMergeRows <= T ? t0 + kMergeRows - 1 : T - 1;
    const bool live = t < T && mask[t] != 0;
    if (warp == 1) {
        const int2 r = seqs_of_rows_warp(mj.seq_offsets, mj.S, t0, last);
        if (lane == 0) range = r;
    }
    merge_parts(pass == 0 ? j0 : j1, part_ld, t, live, warp % kCombWarps, st[pass]);
    __syncthreads();
    MergedRow row = {0.f, 0.f};
    if (warp % kCombWarps == 0 && t < T) {
        row = merge_finish(pass == 0 ? j0 : j1, t, live, status, st[pass]);
        if (pass == 1) lp_roll[lane] = row.lp;
    }
    __syncthreads();
    if (warp != 0) return;
    const int sq = seq_in_range(mj.seq_offsets, range, t <= last ? t : last);
    double v[kSums] = {};
    if (live) {
        const float lr = lp_roll[lane], x[1] = {row.lp - lr};
        float u[1];
        rho_minus_one(x, u);
        const double w = 1.0 + static_cast<double>(fminf(u[0], mj.C - 1.0f)), A = mj.adv[sq];
        v[0] = 1.0;
        v[1] = w;
        v[2] = w * w;
        v[3] = fabsf(x[0]);
        v[4] = A;
        v[5] = A * A;
        v[6] = A * w;
        v[7] = (A * w) * (A * w);
        v[8] = -x[0];
        v[9] = __expf(lr) * fabsf(u[0]);
    }
    if (mj.n_valid_seq) {
        const int sq0 = __shfl_sync(0xffffffffu, sq, 0);
        if (__all_sync(0xffffffffu, sq == sq0)) {
            const int n = __popc(__ballot_sync(0xffffffffu, live));
            if (lane == 0 && n > 0) atomicAdd(&mj.n_valid_seq[sq0], n);
        } else if (live) {
            atomicAdd(&mj.n_valid_seq[sq], 1);
        }
    }
    double* mine = mj.partials + static_cast<int64_t>(blockIdx.x) * kNumMoments;
#pragma unroll
    for (int i = 0; i < kSums; ++i) {
        v[i] = warp_sum(v[i]);
        if (lane == 0) mine[i] = v[i];
    }
}

template <int VEC>
struct RowGroup {
    float lt[VEC], lr[VEC];
    uint8_t mk[VEC];
    bool any;
};
template <int VEC>
__device__ __forceinline__ RowGroup<VEC> load_group(const float* lp_train, const float* lp_roll,
                                                    const uint8_t* __restrict__ mask, int64_t g) {
    RowGroup<VEC> r;
    if (VEC == 4) {
        const float4 a = reinterpret_cast<const float4*>(lp_train)[g];
        const float4 b = reinterpret_cast<const float4*>(lp_roll)[g];
        const uchar4 m = reinterpret_cast<const uchar4*>(mask)[g];
        r.lt[0] = a.x; r.lt[1 % VEC] = a.y; r.lt[2 % VEC] = a.z; r.lt[3 % VEC] = a.w;
        r.lr[0] = b.x; r.lr[1 % VEC] = b.y; r.lr[2 % VEC] = b.z; r.lr[3 % VEC] = b.w;
        r.mk[0] = m.x; r.mk[1 % VEC] = m.y; r.mk[2 % VEC] = m.z; r.mk[3 % VEC] = m.w;
    } else {
        r.lt[0] = lp_train[g]; r.lr[0] = lp_roll[g]; r.mk[0] = mask[g];
    }
    r.any = false;
#pragma unroll
    for (int j = 0; j < VEC; ++j) r.any |= (r.mk[j] != 0);
    return r;
}

template <int VEC>
__global__ void __launch_bounds__(kDiagThreads) moments_kernel(const float* lp_train, const float* lp_roll,
                                                                const uint8_t* __restrict__ mask,
                                                                const int32_t* __restrict__ seq_offsets,
                                                                const float* adv, int64_t T, int S, float C,
                                                                double* __restrict__ partials, int32_t* __restrict__ n_valid_seq,
                                                                const float* seq_logw) {
    pdl_enter();
    __shared__ double scratch[32];
    double acc[kNumMoments];
#pragma unroll
    for (int i = 0; i < kNumMoments; ++i) acc[i] = 0.0;
    // Every warp owns a contiguous range of row groups and its lanes interleave inside it, so a lane's rows only
    // move forward: one binary search for its first group, then the sequence index steps (the next boundary is kept
    // in a register).  Valid rows are counted per sequence on the way (integer atomics: the result does not depend
    // on their order).  The first-order sums (|D|, D, |dp|) take runs of at most 64 rows in fp32 and those short sums go
    // into the fp64 accumulators; the sums behind the three variances are formed per group of rows by add_run.
    int sq = -1, cur = -1, cnt = 0;
    int64_t next_b = 0;                                   // first row of sequence sq + 1 (or "never" for the last one)
    float f[kNumMoments];
    auto flush = [&]() {
        if (n_valid_seq && cur >= 0 && cnt > 0) atomicAdd(&n_valid_seq[cur], cnt);
        cnt = 0;
    };
    // fp32 runs are kept only for the three first-order sums (3, 8, 9); the sums behind the variances go through add_run
    auto clear = [&]() { f[3] = 0.f; f[8] = 0.f; f[9] = 0.f; };
    auto commit = [&]() {
        acc[3] += static_cast<double>(f[3]);
        acc[8] += static_cast<double>(f[8]);
        acc[9] += static_cast<double>(f[9]);
    };
    auto seek = [&](int64_t t) {
        if (sq < 0) {
            sq = seq_of_row(seq_offsets, S, t);
            next_b = sq + 1 < S ? static_cast<int64_t>(seq_offsets[sq + 1]) : (int64_t(1) << 62);
        }
        while (t >= next_b) {
            ++sq;
            next_b = sq + 1 < S ? static_cast<int64_t>(seq_offsets[sq + 1]) : (int64_t(1) << 62);
        }
    };
    auto add_row = [&](float lt, float lr, float A) {
        const float dl[1] = {lt - lr};
        float u[1];
        rho_minus_one(dl, u);                              // rho - 1; |e^lt - e^lr| = e^lr |rho - 1|
        // sequence-level variant: every row carries its sequence's truncated weight instead of its own
        const float uw = seq_logw ? fminf(__expf(seq_logw[sq]), C) - 1.0f : fminf(u[0], C - 1.0f);
        add_run(acc, 1, uw, 0.f, 0.f, A);
        f[3] += fabsf(dl[0]);
        f[8] -= dl[0];
        f[9] = fmaf(__expf(lr), fabsf(u[0]), f[9]);
        if (sq != cur) { flush(); cur = sq; }
        ++cnt;
    };
    auto add_group = [&](const RowGroup<VEC>& r, int64_t g) {
        if (!r.any) return;
        const int64_t t0 = g * VEC;
        seek(t0);
        if (VEC > 1 && t0 + VEC <= next_b) {
            // the usual case, all rows of the group in one sequence: one advantage and one weight source for the
            // group, masked rows drop out by selection, and the sums that involve A follow from sum w and sum w^2
            const float A = adv[sq];
            const float useq = seq_logw ? fminf(__expf(seq_logw[sq]), C) - 1.0f : 0.f;
            float dl[VEC], u[VEC];
#pragma unroll
            for (int j = 0; j < VEC; ++j) dl[j] = r.mk[j] != 0 ? r.lt[j] - r.lr[j] : 0.f;
            rho_minus_one(dl, u);
            float p = 0.f;
            int n = 0;
#pragma unroll
            for (int j = 0; j < VEC; ++j) {
                const bool on = r.mk[j] != 0;
                f[3] += fabsf(dl[j]);
                f[8] -= dl[j];
                f[9] += on ? __expf(r.lr[j]) * fabsf(u[j]) : 0.f;
                u[j] = seq_logw ? useq : fminf(u[j], C - 1.0f);
                if (on && n == 0) p = u[j];                        // pivot: the first valid row
                n += on ? 1 : 0;
            }
            float sv = 0.f, sv2 = 0.f;
#pragma unroll
            for (int j = 0; j < VEC; ++j) {
                const float v = r.mk[j] != 0 ? u[j] - p : 0.f;
                sv += v;
                sv2 = fmaf(v, v, sv2);
            }
            add_run(acc, n, p, sv, sv2, A);
            if (sq != cur) { flush(); cur = sq; }
            cnt += n;
            return;
        }
#pragma unroll
        for (int j = 0; j < VEC; ++j) {
            if (r.mk[j]) {
                seek(t0 + j);
                add_row(r.lt[j], r.lr[j], adv[sq]);
            }
        }
    };
    const int lane = threadIdx.x & 31;
    const int64_t ngroups = T / VEC;
    const int64_t nwarps = static_cast<int64_t>(gridDim.x) * (blockDim.x >> 5);
    const int64_t gw = static_cast<int64_t>(blockIdx.x) * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const int64_t per = ((ngroups + nwarps - 1) / nwarps + 63) / 64 * 64;             // groups per warp
    const int64_t g_end = (gw + 1) * per < ngroups ? (gw + 1) * per : ngroups;
    int64_t g = gw * per + lane;
    clear();
    for (int pass = 0; g + 32 < g_end; g += 64) {                                      // two groups in flight per lane
        const RowGroup<VEC> r0 = load_group<VEC>(lp_train, lp_roll, mask, g);
        const RowGroup<VEC> r1 = load_group<VEC>(lp_train, lp_roll, mask, g + 32);
        add_group(r0, g);
        add_group(r1, g + 32);
        if ((++pass & 7) == 0) {                                                       // at most 64 rows per fp32 run
            commit();
            clear();
        }
    }
    if (g < g_end) add_group(load_group<VEC>(lp_train, lp_roll, mask, g), g);
    flush();
    // rows after the last whole group: the first threads of the grid, one row each
    {
        const int64_t t = ngroups * VEC + static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
        if (t < T && mask[t]) {
            sq = -1;
            cur = -1;
            seek(t);
            add_row(lp_train[t], lp_roll[t], adv[sq]);
            flush();
        }
    }
    commit();
    for (int i = 0; i < kNumMoments; ++i) {
        const double tot = block_sum(acc[i], scratch);
        if (threadIdx.x == 0) partials[blockIdx.x * kNumMoments + i] = tot;
    }
}

// The same moments for 16-byte aligned inputs, fed by bulk asynchronous copies: a block walks a contiguous range of
// 2048-row tiles; thread 0 keeps three tiles (two log-prob vectors and the mask bytes, 18 KB each) in flight into a
// ring of shared-memory stages, completion arrives on one mbarrier per stage, and every thread takes the eight rows
// 8 tid .. 8 tid + 7 of each tile from shared memory.  Memory latency is carried by the copies in flight (54 KB per
// block, four blocks per SM) instead of by registers, and the work per row is kept to about twenty instructions
// (flush-to-zero exponentials, 32-bit row indices, the group's sequence looked up before the data arrives, the
// per-tile bookkeeping shared by eight rows), because at 9 bytes per row the instruction issue rate is the next limit
// after HBM.  Rows after the last whole tile are read directly.  Summation order is fixed by the grid as above.
constexpr int kMomRows = 2048;
constexpr int kMomStages = 3;
constexpr int kMomStageBytes = kMomRows * 9;
constexpr int kMomSmemBytes = kMomStages * kMomStageBytes + 128;
// 228 KB per SM, 1 KB of it reserved per block: four blocks fit, and all 592 run at once (with three per SM 67 M rows took
// 3.5 TB/s instead of 4.9)
static_assert(4 * (kMomSmemBytes + 1024 + 10 * (kDiagThreads / 32 + 1) * 8 + 64) <= 228 * 1024, "four blocks per SM");


// (add2 / sub2 / mul2 / fma2: the packed two-element fp32 instructions, ptx.cuh.)  The staged kernel is bound by
// instruction issue right after HBM, and half of its per-row work is additions, multiplications and multiply-adds.
__device__ __forceinline__ float ex2_ftz(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// The waiting part of a bounded mbarrier wait, kept out of line so that the loop around it stays small.
__device__ __noinline__ bool mbar_wait_slow(uint64_t* bar, uint32_t parity, int* abort_flag) {
    return mbar_wait(bar, parity, abort_flag);
}

// SEQ: every row carries its sequence's truncated weight instead of its own.  WALKS: the fast walk and, for a block that needs
// it, the exact one (see add_rows) in one kernel, or each in its own -- the fast one leaves in slots 10 and 11 of its partial
// sums which groups it met, and the exact one replaces the sums of the blocks that need it.
enum Walks { kBothWalks, kFastWalk, kExactWalk };
template <bool SEQ, int WALKS>
__global__ void __launch_bounds__(kDiagThreads, 4) moments_staged_kernel(const float* lp_train, const float* lp_roll,
                                                                         const uint8_t* __restrict__ mask,
                                                                         const int32_t* __restrict__ seq_offsets,
                                                                         const float* adv, int T, int S, float C,
                                                                         double* partials, int32_t* __restrict__ n_valid_seq,
                                                                         const float* seq_logw, bool early) {
    static_assert(kDiagThreads * 8 == kMomRows, "one 8-row group per thread and tile");
    extern __shared__ __align__(128) uint8_t stages[];          // kMomStages stages, then the barriers
    uint64_t* full = reinterpret_cast<uint64_t*>(stages + kMomStages * kMomStageBytes);
    __shared__ double scratch[kSums][kDiagThreads / 32];
    __shared__ double totals[kSums];
    __shared__ int abort_flag;
    const int tid = threadIdx.x;
    const int lane = tid & 31;
    const int nfull = T / kMomRows;                    // whole tiles; what is left is one more, read directly
    const int ntiles = (T + kMomRows - 1) / kMomRows;
    const int tile0 = static_cast<int>(static_cast<int64_t>(blockIdx.x) * ntiles / gridDim.x);
    const int tile1 = static_cast<int>(static_cast<int64_t>(blockIdx.x + 1) * ntiles / gridDim.x);
    if (tid == 0) {
        for (int i = 0; i < kMomStages; ++i) mbar_init(&full[i], 1);
        abort_flag = 0;
        fence_barrier_init();
    }
    __syncthreads();
    auto issue = [&](int tile, int st) {               // thread 0: the three copies of one tile onto the stage's barrier
        uint8_t* dst = stages + st * kMomStageBytes;
        const size_t r0 = static_cast<size_t>(tile) * kMomRows;
        mbar_expect_tx(&full[st], kMomStageBytes);
        bulk_load(dst, lp_train + r0, kMomRows * 4, &full[st]);
        bulk_load(dst + kMomRows * 4, lp_roll + r0, kMomRows * 4, &full[st]);
        bulk_load(dst + kMomRows * 8, mask + r0, kMomRows, &full[st]);
    };

    // Everything a thread sums stays in fp32 while it walks its tiles and turns into fp64 once, at the end: the first-order
    // sums (|D|, D, |dp|) as they are, the sums behind the three variances as SHIFTED sums about pivots taken from the
    // thread's own data -- v = (w - 1) - pivot for the weights, dA = A - A_pivot for the advantages, and
    // x = A w - A_pivot (1 + pivot) = A v + dA (1 + pivot) for their product -- so that the fp32 roundings scale with the
    // spread of the data and not with its size, and are exactly zero when all rows are equal.  A thread sees at most
    // 8 ceil(tiles / kDiagBlocks) rows: 16 of 1.48 M, 448 of 67 M.
    float f3, f9, g_v, g_v2, g_dA, g_dA2, g_x, g_x2;
    F2 f8p;                                             // sum of D, two rows at a time
    int nrows;                                          // valid rows of the thread
    int nbig, nsmall;                                   // groups with a gap above 2^-6 / with all gaps below (see add_rows)
    float pivot, A_pivot, dA;
    bool have_pivot;                                    // both pivots come from the thread's first group with a valid row
    constexpr int kNever = 0x7fffffff;
    int sq, cur;
    int next_b;                                         // first row of sequence sq + 1 (or "never" for the last one)
    float A = 0.f, wseq = 0.f;                          // advantage and sequence-level weight of sequence `cur`
    int wsq = -1, wcnt = 0;                             // lane 0: valid rows of the warp's strips counted for sequence wsq
    auto reset = [&]() {
        f3 = f9 = g_v = g_v2 = g_dA = g_dA2 = g_x = g_x2 = 0.f;
        f8p = F2{0.f, 0.f};
        nrows = 0;
        nbig = 0;
        nsmall = 0;
        pivot = A_pivot = dA = 0.f;
        have_pivot = false;
        sq = cur = -1;
        next_b = 0;
    };
    reset();
    auto start_at = [&](int s0) {
        sq = s0;
        next_b = sq + 1 < S ? seq_offsets[sq + 1] : kNever;
    };
    auto seek = [&](int t) {
        while (t >= next_b) start_at(sq + 1);
    };
    auto enter = [&]() {                                // the row's sequence becomes the current one
        if (sq != cur) {
            cur = sq;
            A = adv[sq];
            dA = have_pivot ? A - A_pivot : 0.f;
            if (SEQ) wseq = fminf(__expf(seq_logw[sq]), C);
        }
    };
    // Sums over the rows of a group whose mask byte (rows 0..3 in `m0`, 4..7 in `m1`) is set, all of them in sequence
    // `cur`; returns how many they are.  Rows go two at a time through the packed fp32 instructions.  The weight pivot
    // is w - 1 of the first valid row this thread meets and stays: any value of the data serves.
    // rho - 1 comes from the fast exponential, which is good to 1e-7 ABSOLUTE: enough unless the gaps D themselves are
    // tiny, when it is only a thousandth of a weight that differs from 1 by 1e-4.  The exact walk uses a short series for
    // groups whose |D| are all at most 2^-6 (their sum is), which gives e^D - 1 to fp32 accuracy relative to itself.  Both
    // in one walk cost registers and scheduling freedom (a fifth of the bandwidth), so the fast walk comes first and counts
    // the block's groups above 2^-6; a block that met none walks its tiles a second time, exactly.
    auto add_rows = [&](auto exact, const float (&lt)[8], const float (&lr)[8], uint32_t m0, uint32_t m1) -> int {
        constexpr bool EXACT = decltype(exact)::value;
        const uint32_t v0 = __vcmpne4(m0, 0u), v1 = __vcmpne4(m1, 0u);     // 0xFF in the byte of every valid row
        const int n = (__popc(v0) + __popc(v1)) >> 3;
        bool on[8];
        float dl[8], u[8], e[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) on[j] = ((j < 4 ? v0 : v1) & (0x80u << (8 * (j & 3)))) != 0u;
        float s3 = 0.f;
#pragma unroll
        for (int j = 0; j < 8; j += 2) {
            const F2 d = sub2(F2{lt[j], lt[j + 1]}, F2{lr[j], lr[j + 1]});
            dl[j] = on[j] ? d.x : 0.f;                             // a masked row enters with D = 0
            dl[j + 1] = on[j + 1] ? d.y : 0.f;
            f8p = add2(f8p, F2{dl[j], dl[j + 1]});
            s3 += fabsf(dl[j]);
            s3 += fabsf(dl[j + 1]);
        }
        f3 += s3;
        if (EXACT && s3 <= 0x1p-6f) {
#pragma unroll
            for (int j = 0; j < 8; j += 2) {
                const F2 x = {dl[j], dl[j + 1]};
                F2 q = fma2(x, F2{1.0f / 24.0f, 1.0f / 24.0f}, F2{1.0f / 6.0f, 1.0f / 6.0f});
                q = fma2(x, q, F2{0.5f, 0.5f});
                q = fma2(x, q, F2{1.0f, 1.0f});
                q = mul2(x, q);
                u[j] = q.x;
                u[j + 1] = q.y;
            }
        } else {
            if (!EXACT) {
                nbig += s3 > 0x1p-6f ? 1 : 0;
                nsmall += (s3 <= 0x1p-6f && n > 0) ? 1 : 0;
            }
#pragma unroll
            for (int j = 0; j < 8; j += 2) {
                const F2 x = mul2(F2{dl[j], dl[j + 1]}, F2{1.4426950408889634f, 1.4426950408889634f});
                const F2 r = add2(F2{ex2_ftz(x.x), ex2_ftz(x.y)}, F2{-1.0f, -1.0f});
                u[j] = r.x;
                u[j + 1] = r.y;
            }
        }
#pragma unroll
        for (int j = 0; j < 8; j += 2) {                           // |e^lt - e^lr| = e^lr |rho - 1|
            const F2 y = mul2(F2{on[j] ? lr[j] : 0.f, on[j + 1] ? lr[j + 1] : 0.f}, F2{1.4426950408889634f, 1.4426950408889634f});
            e[j] = ex2_ftz(y.x);
            e[j + 1] = ex2_ftz(y.y);
        }
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            f9 = fmaf(e[j], fabsf(u[j]), f9);
            u[j] = SEQ ? wseq - 1.0f : fminf(u[j], C - 1.0f);      // truncated weight minus one
        }
        if (!have_pivot) {
#pragma unroll
            for (int j = 7; j >= 0; --j) pivot = on[j] ? u[j] : pivot;
            A_pivot = A;
            dA = 0.f;
            have_pivot = n > 0;
        }
        F2 sv = {0.f, 0.f}, sv2 = {0.f, 0.f};
#pragma unroll
        for (int j = 0; j < 8; j += 2) {
            const F2 d = sub2(F2{u[j], u[j + 1]}, F2{pivot, pivot});
            const F2 v = {on[j] ? d.x : 0.f, on[j + 1] ? d.y : 0.f};
            sv = add2(sv, v);
            sv2 = fma2(v, v, sv2);
        }
        const float svs = sv.x + sv.y, sv2s = sv2.x + sv2.y, nf = static_cast<float>(n);
        const float c1 = dA * (1.0f + pivot);                      // x = A v + c1 on every valid row of the group
        g_v += svs;
        g_v2 += sv2s;
        g_dA = fmaf(dA, nf, g_dA);
        g_dA2 = fmaf(dA * dA, nf, g_dA2);
        g_x += fmaf(A, svs, c1 * nf);
        g_x2 += fmaf(A * A, sv2s, fmaf(2.0f * A * c1, svs, c1 * c1 * nf));
        nrows += n;
        return n;
    };

    // One walk over the block's tiles, the `base`-th tile of the stage ring first; the fast one also adds up the valid rows
    // per sequence on the way.
    bool failed = false;
    int issued = tile0;                                 // first tile not yet requested (thread 0)
    const int full1 = tile1 < nfull ? tile1 : nfull;    // tiles of the block that arrive by copy: tile0 .. full1 - 1
    auto fill_ring = [&](int base) {
        issued = tile0;
        if (tid == 0)
            for (; issued < full1 && issued < tile0 + kMomStages; ++issued) issue(issued, (base + issued - tile0) % kMomStages);
    };
    auto walk = [&](auto exact, int base) {
        constexpr bool count = !decltype(exact)::value;
        for (int tile = tile0; tile < tile1; ++tile) {
            const unsigned k = static_cast<unsigned>(base + tile - tile0);
            const unsigned st = k % kMomStages;
            // the group's sequence, advantage and weight source do not depend on the tile's data: fetched before the wait
            const int t0 = tile * kMomRows + 8 * tid;
            seek(t0);
            const bool single = t0 + 8 <= next_b;          // the usual case: the eight rows belong to one sequence
            if (single) enter();
            const uint32_t parity = (k / kMomStages) & 1u;
            bool ok = tile >= nfull || mbar_try_wait(&full[st], parity);
            if (!ok) ok = mbar_wait_slow(&full[st], parity, &abort_flag);
            int n = 0;
            if (ok) {
                float lt[8], lr[8];
                uint2 mk = make_uint2(0, 0);
                if (tile < nfull) {
                    const uint8_t* src = stages + st * kMomStageBytes;
                    const float4* pa = reinterpret_cast<const float4*>(src) + 2 * tid;
                    const float4* pb = reinterpret_cast<const float4*>(src + kMomRows * 4) + 2 * tid;
                    const float4 a0 = pa[0], a1 = pa[1], b0 = pb[0], b1 = pb[1];
                    mk = reinterpret_cast<const uint2*>(src + kMomRows * 8)[tid];
                    lt[0] = a0.x; lt[1] = a0.y; lt[2] = a0.z; lt[3] = a0.w; lt[4] = a1.x; lt[5] = a1.y; lt[6] = a1.z; lt[7] = a1.w;
                    lr[0] = b0.x; lr[1] = b0.y; lr[2] = b0.z; lr[3] = b0.w; lr[4] = b1.x; lr[5] = b1.y; lr[6] = b1.z; lr[7] = b1.w;
                } else {
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        const bool in = t0 + j < T;
                        lt[j] = in ? lp_train[t0 + j] : 0.f;
                        lr[j] = in ? lp_roll[t0 + j] : 0.f;
                        const uint32_t m = in ? mask[t0 + j] : 0u;
                        if (j < 4) mk.x |= m << (8 * j);
                        else mk.y |= m << (8 * (j - 4));
                    }
                }
                if (single) {
                    if ((mk.x | mk.y) != 0u) n = add_rows(exact, lt, lr, mk.x, mk.y);
                } else if ((mk.x | mk.y) != 0u) {
                    const uint64_t m64 = (static_cast<uint64_t>(mk.y) << 32) | mk.x;
                    int j = 0;
                    while (j < 8) {                         // a boundary inside the group: one run of rows per sequence
                        seek(t0 + j);
                        const int left = next_b - (t0 + j);
                        const int j1 = left < 8 - j ? j + left : 8;
                        enter();
                        const uint64_t run = (j1 == 8 ? ~uint64_t(0) : (uint64_t(1) << (8 * j1)) - 1u) & ~((uint64_t(1) << (8 * j)) - 1u);
                        const int nr = add_rows(exact, lt, lr, static_cast<uint32_t>(m64 & run), static_cast<uint32_t>((m64 & run) >> 32));
                        if (count && n_valid_seq && nr > 0) atomicAdd(&n_valid_seq[sq], nr);
                        j = j1;
                    }
                }
            }
            if (count && n_valid_seq) {
                // valid rows per sequence: a warp's 256-row strip usually lies in one sequence, whose count lane 0 keeps in
                // a register until the strip moves on (integer atomics: the result does not depend on their order)
                const int sq0 = __shfl_sync(0xffffffffu, sq, 0);
                if (__all_sync(0xffffffffu, single && sq == sq0)) {
                    const int tot = __reduce_add_sync(0xffffffffu, n);
                    if (lane == 0) {
                        if (sq0 != wsq) {
                            if (wsq >= 0 && wcnt > 0) atomicAdd(&n_valid_seq[wsq], wcnt);
                            wsq = sq0;
                            wcnt = 0;
                        }
                        wcnt += tot;
                    }
                } else if (single && n > 0) {
                    atomicAdd(&n_valid_seq[sq], n);
                }
            }
            // everyone is done with the stage (or someone gave up): the stage can take the tile three ahead
            if (__syncthreads_or(ok ? 0 : 1)) { failed = true; break; }
            if (tid == 0 && issued < full1) { issue(issued, st); ++issued; }
        }
        if (failed && tid == 0) {
            // let the copies still in flight land before the block's shared memory is given up
            for (int i = 0; i < issued - tile0; ++i)
                if (issued - tile0 - i <= kMomStages) {
                    const unsigned q = static_cast<unsigned>(base + i);
                    mbar_wait_drain(&full[q % kMomStages], (q / kMomStages) & 1u);
                }
        }
        if (count && n_valid_seq && lane == 0 && wsq >= 0 && wcnt > 0) atomicAdd(&n_valid_seq[wsq], wcnt);
    };
    // The sequences of the warp's rows of the first tile, before the wait: the offsets are older than the kernel before this
    // one.  So are the rows when that kernel only formed advantages (`early`): their copies start now, too.
    int2 range = make_int2(0, 0);
    if (tile0 < tile1) {
        const int w0 = tile0 * kMomRows + (tid & ~31) * 8;
        range = seqs_of_rows_warp(seq_offsets, S, w0 < T ? w0 : T - 1, w0 + 255 < T ? w0 + 255 : T - 1);
    }
    const int first_sq = seq_in_range(seq_offsets, range, tile0 * kMomRows + 8 * tid < T ? tile0 * kMomRows + 8 * tid : T - 1);
    double* mine = partials + blockIdx.x * kNumMoments;
    if (WALKS == kExactWalk) {
        pdl_enter();
        if (mine[10] != 0.0 || mine[11] == 0.0 || isnan(mine[0])) return;
        fill_ring(0);
        start_at(first_sq);
        walk(std::true_type{}, 0);
    } else {
        if (early) fill_ring(0);
        pdl_enter();
        if (!early) fill_ring(0);
        start_at(first_sq);
        walk(std::false_type{}, 0);
        const bool any_big = __syncthreads_or(nbig) != 0;
        const bool any_small = __syncthreads_or(nsmall) != 0;
        if (WALKS == kBothWalks && !any_big && any_small && !__syncthreads_or(failed ? 1 : 0)) {
            reset();
            start_at(first_sq);
            fill_ring(full1 - tile0);
            walk(std::true_type{}, full1 - tile0);
        }
        if (tid == 0) {
            mine[10] = any_big ? 1.0 : 0.0;
            mine[11] = any_small ? 1.0 : 0.0;
        }
    }
    double acc[kSums];
    {
        // from the shifted sums to the sums of w, w^2, A, A^2, A w, (A w)^2 in fp64, once per thread:
        // w = P + v with P = 1 + pivot;  A = Ap + dA;  A w = K + x with K = Ap P
        const double P = 1.0 + static_cast<double>(pivot), Ap = static_cast<double>(A_pivot), K = Ap * P;
        const double N = static_cast<double>(nrows);
        const double SV = static_cast<double>(g_v), SDA = static_cast<double>(g_dA), SX = static_cast<double>(g_x);
        acc[0] = N;
        acc[1] = fma(P, N, SV);
        acc[2] = static_cast<double>(g_v2) + P * fma(P, N, 2.0 * SV);
        acc[3] = static_cast<double>(f3);
        acc[4] = fma(Ap, N, SDA);
        acc[5] = static_cast<double>(g_dA2) + Ap * fma(Ap, N, 2.0 * SDA);
        acc[6] = fma(K, N, SX);
        acc[7] = static_cast<double>(g_x2) + K * fma(K, N, 2.0 * SX);
        acc[8] = -(static_cast<double>(f8p.x) + static_cast<double>(f8p.y));
        acc[9] = static_cast<double>(f9);
    }
    if (failed) acc[0] = __longlong_as_double(0x7ff8000000000000LL);     // a NaN count marks the batch as not reduced
    block_sums(acc, scratch, totals);
    if (tid < kSums) mine[tid] = totals[tid];
}

// Ratio and rectification weight of a valid row; seq_logw: its sequence's log weight (sequence-level variant) or NULL.
__device__ __forceinline__ void rectify_row(float lt, float lr, float alpha, float C, const float* seq_logw, float& r, float& wt) {
    r = __expf(lt - lr);
    const float w = seq_logw ? __expf(*seq_logw) : r;
    wt = fmaf(alpha, fminf(w, C) - 1.0f, 1.0f);
}

// Forms alpha first, every block for itself (form_alpha).
template <int VEC>
__global__ void __launch_bounds__(kDiagThreads, 4) rectify_kernel(const float* __restrict__ lp_train, const float* __restrict__ lp_roll,
                                                                  const uint8_t* __restrict__ mask, int64_t T, float C,
                                                                  const __grid_constant__ TotalsJob job, float* __restrict__ rho,
                                                                  float* __restrict__ w_tilde, const int32_t* __restrict__ seq_offsets,
                                                                  int S, const float* __restrict__ seq_logw, bool early) {
    // The log-probs and the mask were there before the kernel this one follows (`early`): the first two groups are loaded
    // while that one still runs, the wait is for its sums.
    __shared__ Totals totals;
    const int64_t ngroups = T / VEC;
    const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
    const int64_t g0 = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    RowGroup<VEC> in = {}, next = {};
    auto preload = [&]() {
        if (g0 < ngroups) in = load_group<VEC>(lp_train, lp_roll, mask, g0);
        if (g0 + stride < ngroups) next = load_group<VEC>(lp_train, lp_roll, mask, g0 + stride);
    };
    if (early) preload();
    pdl_enter();
    if (!early) preload();
    const float alpha = form_alpha(job, totals);
    auto one = [&](float lt, float lr, uint8_t mk, float& r, float& wt, int64_t t) {
        r = 1.0f;
        wt = 1.0f;
        if (mk) rectify_row(lt, lr, alpha, C, seq_logw ? seq_logw + seq_of_row(seq_offsets, S, t) : nullptr, r, wt);
    };
    for (int64_t g = g0; g < ngroups; g += stride) {
        float r[VEC], wt[VEC];
#pragma unroll
        for (int j = 0; j < VEC; ++j) one(in.lt[j], in.lr[j], in.mk[j], r[j], wt[j], g * VEC + j);
        if (VEC == 4) {
            if (rho) reinterpret_cast<float4*>(rho)[g] = make_float4(r[0], r[1 % VEC], r[2 % VEC], r[3 % VEC]);
            reinterpret_cast<float4*>(w_tilde)[g] = make_float4(wt[0], wt[1 % VEC], wt[2 % VEC], wt[3 % VEC]);
        } else {
            if (rho) rho[g] = r[0];
            w_tilde[g] = wt[0];
        }
        in = next;
        if (g + 2 * stride < ngroups) next = load_group<VEC>(lp_train, lp_roll, mask, g + 2 * stride);
    }
    for (int64_t t = ngroups * VEC + static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; t < T; t += stride) {
        float r, wt;
        one(lp_train[t], lp_roll[t], mask[t], r, wt, t);
        if (rho) rho[t] = r;
        w_tilde[t] = wt;
    }
}

// ------------------------------------------------------------------------------------------------
// Per-token gradient factor c_t and the surrogate loss (Eq. ais-grpo without the KL term).
// ------------------------------------------------------------------------------------------------
// One thread per group of four rows, one warp per 128-row tile, so that the kernel also says which tiles have a gradient
// (tile_flags) -- and, as its last block, adds up the loss.  VEC: the vectors allow 16-byte accesses.
struct LossArgs {
    const float *lp_train, *lp_old, *lp_ref, *lse, *adv, *w_tilde;
    const uint8_t* mask;
    const int32_t *seq_offsets, *n_valid_seq;
    int64_t T;
    int32_t S, S_norm;
    double beta_kl, clip_eps;
    double* partials;
    float* coef;
    uint8_t* tile_flags;
    uint4* clear;          // pacing rings of the passes that follow
    int32_t nclear;
    uint32_t* ticket;
    float* loss;
    ais_diag* diag;
    RectifyJob rectify;    // rectify.w_tilde != NULL: ratios and weights of the rows are formed here and written on the way
    KeepJob keep;          // keep.scale != NULL: the scratch is in exponent form (with `rectify` only)
};

template <bool VEC, bool RECTIFY>
__global__ void __launch_bounds__(kDiagThreads) loss_coef_kernel(const __grid_constant__ LossArgs a) {
    __shared__ double scratch[2][kDiagThreads / 32];
    __shared__ double totals[2];
    __shared__ std::conditional_t<RECTIFY, Totals, int> batch;
    pdl_enter();
    const int lane = threadIdx.x & 31;
    const int64_t tiles = (a.T + 127) / 128;
    const int64_t nwarps = static_cast<int64_t>(gridDim.x) * (kDiagThreads / 32);
    const int64_t tile0 = static_cast<int64_t>(blockIdx.x) * (kDiagThreads / 32) + (threadIdx.x >> 5);
    // what a thread reads of its four rows
    struct Rows {
        float lt[4], lr[4], lse[4], wt[4];
        uint32_t mk;                                               // mask bytes
        int n;                                                     // rows of the batch among the four
        int2 range;                                                // sequences of the warp's 128 rows
    };
    auto load_rows = [&](int64_t tile, Rows& r) {
        const int64_t t0 = tile * 128 + 4 * lane;
        r.n = t0 + 4 <= a.T ? 4 : t0 < a.T ? static_cast<int>(a.T - t0) : 0;
        r.mk = 0;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            r.lt[j] = j < r.n ? a.lp_train[t0 + j] : 0.f;
            r.lse[j] = j < r.n ? a.lse[t0 + j] : 0.f;
            if (RECTIFY) r.lr[j] = j < r.n ? a.rectify.lp_roll[t0 + j] : 0.f;
        }
        if (VEC && r.n == 4) {
            r.mk = *reinterpret_cast<const uint32_t*>(a.mask + t0);
            if (!RECTIFY) {
                const float4 w4 = *reinterpret_cast<const float4*>(a.w_tilde + t0);
                r.wt[0] = w4.x; r.wt[1] = w4.y; r.wt[2] = w4.z; r.wt[3] = w4.w;
            }
        } else {
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                if (j < r.n) r.mk |= static_cast<uint32_t>(a.mask[t0 + j]) << (8 * j);
                if (!RECTIFY) r.wt[j] = j < r.n ? a.w_tilde[t0 + j] : 0.f;
            }
        }
        r.range = seqs_of_rows_warp(a.seq_offsets, a.S, tile * 128, tile * 128 + 127 < a.T ? tile * 128 + 127 : a.T - 1);
    };
    // The first rows and their sequences are asked for ahead of the sums that alpha waits for: a small batch is one chain of
    // loads (step of 512 rows 42.4 -> 41.4 us, of 3,001 rows, d = 512, V = 4096, 85.8 -> 85.0).
    Rows in;
    if (tile0 < tiles) load_rows(tile0, in);
    float alpha = 0.f;
    if constexpr (RECTIFY) alpha = form_alpha(a.rectify.totals, batch);
    double J = 0.0, KL = 0.0;
    // one valid row of sequence sq: its share of the objective, of the KL estimate, and its gradient factor
    auto one = [&](int64_t t, int sq, float lt, float lse, float wtf) -> float {
        if (!isfinite(lse)) return 0.f;          // the forward pass marked this row (non-finite logits): it takes no part
        const double A = a.adv[sq];
        const int n = a.n_valid_seq[sq] > 0 ? a.n_valid_seq[sq] : 1;
        const double norm = 1.0 / (static_cast<double>(a.S_norm) * static_cast<double>(n));
        const double rho_on = a.lp_old ? exp(static_cast<double>(lt) - static_cast<double>(a.lp_old[t])) : 1.0;
        const double un = rho_on * A;
        const double cl = fmin(fmax(rho_on, 1.0 - a.clip_eps), 1.0 + a.clip_eps) * A;
        const double wt = wtf;
        double c = 0.0;
        J += wt * fmin(un, cl) * norm;
        if (un <= cl) c = wt * A * rho_on * norm;
        if (a.lp_ref) {
            // KL(pi_theta || pi_ref) estimate r - log r - 1, r = pi_ref / pi_theta; its slope in lp_theta is 1 - r
            const double log_r = static_cast<double>(a.lp_ref[t]) - static_cast<double>(lt);
            const double r = exp(log_r);
            KL += (r - log_r - 1.0) * norm;
            c -= a.beta_kl * (1.0 - r) * norm;
        }
        return static_cast<float>(c);
    };
    for (int64_t tile = tile0; tile < tiles; tile += nwarps) {
        if (tile != tile0) load_rows(tile, in);
        const int64_t t0 = tile * 128 + 4 * lane;
        const int rows = in.n;
        const uint32_t mk = in.mk;
        float c[4] = {0.f, 0.f, 0.f, 0.f}, wt[4];
        float rho[4] = {1.f, 1.f, 1.f, 1.f};
#pragma unroll
        for (int j = 0; j < 4; ++j) wt[j] = RECTIFY ? 1.f : in.wt[j];
        if (mk != 0u) {
            int sq = seq_in_range(a.seq_offsets, in.range, t0);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                while (sq + 1 < a.S && static_cast<int64_t>(a.seq_offsets[sq + 1]) <= t0 + j) ++sq;
                if ((mk >> (8 * j)) & 0xFFu) {
                    if (RECTIFY)
                        rectify_row(in.lt[j], in.lr[j], alpha, a.rectify.C, a.rectify.seq_logw ? a.rectify.seq_logw + sq : nullptr, rho[j], wt[j]);
                    c[j] = one(t0 + j, sq, in.lt[j], in.lse[j], wt[j]);
                }
            }
        }
        if (RECTIFY) {
            if (VEC && rows == 4) {
                if (a.rectify.rho) *reinterpret_cast<float4*>(a.rectify.rho + t0) = make_float4(rho[0], rho[1], rho[2], rho[3]);
                *reinterpret_cast<float4*>(a.rectify.w_tilde + t0) = make_float4(wt[0], wt[1], wt[2], wt[3]);
            } else {
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    if (j < rows && a.rectify.rho) a.rectify.rho[t0 + j] = rho[j];
                    if (j < rows) a.rectify.w_tilde[t0 + j] = wt[j];
                }
            }
        }
        if (rows == 4) *reinterpret_cast<float4*>(a.coef + t0) = make_float4(c[0], c[1], c[2], c[3]);     // workspace: aligned
        else
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (j < rows) a.coef[t0 + j] = c[j];
        if (RECTIFY && a.keep.scale != nullptr) {
            bool redo = false;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                if (j >= rows) continue;
                const int64_t t = t0 + j;
                float scale = 0.f;
                if (c[j] != 0.f) {
                    const float lse = in.lse[j];
                    const bool ef = exp_form(lse);
                    scale = ef ? c[j] * expf(-lse) : 1.f;
                    redo |= !ef;
                    const int y = a.keep.tokens[t];
                    if (ef && t < a.keep.rows && y >= 0 && y < a.keep.V)
                        a.keep.U[t * a.keep.ldU + y] = __float2bfloat16(exp_form_target(in.lt[j], lse));
                }
                a.keep.scale[t] = scale;
            }
            redo = __any_sync(0xffffffffu, redo);
            if (lane == 0) {
                a.keep.redo_flags[tile] = redo ? 1 : 0;
                if (redo) atomicAdd(a.keep.redo_count, 1u);
            }
        }
        const bool any = __any_sync(0xffffffffu, c[0] != 0.f || c[1] != 0.f || c[2] != 0.f || c[3] != 0.f);
        if (lane == 0) a.tile_flags[tile] = any ? 1 : 0;
    }
    if (a.clear)
        for (int i = blockIdx.x * kDiagThreads + threadIdx.x; i < a.nclear; i += gridDim.x * kDiagThreads) a.clear[i] = make_uint4(0, 0, 0, 0);
    double sums[2] = {J, KL};
    block_sums(sums, scratch, totals);
    // A single block has its sums at hand and needs no counter of finished blocks (512 rows 41.4 -> 39.2 us).
    double Jall = totals[0], KLall = totals[1];
    if (gridDim.x > 1) {
        if (threadIdx.x < 2) a.partials[2 * blockIdx.x + threadIdx.x] = totals[threadIdx.x];
        if (!last_block(a.ticket) || threadIdx.x >= 32) return;
        Jall = warp_ordered_sum(a.partials, gridDim.x, 2, 0, lane);
        KLall = warp_ordered_sum(a.partials, gridDim.x, 2, 1, lane);
    }
    if (threadIdx.x != 0) return;
    const double total = -Jall + a.beta_kl * KLall;
    if (a.loss) *a.loss = static_cast<float>(total);
    if (a.diag) {
        a.diag->loss = total;
        a.diag->kl_ref = KLall;
    }
}

// 16-byte loads need every per-row vector on a 16-byte boundary (the mask on a 4-byte one).
inline bool vec4_ok(const void* a, const void* b, const void* c, const void* d, const void* m) {
    const uintptr_t f = reinterpret_cast<uintptr_t>(a) | reinterpret_cast<uintptr_t>(b) | reinterpret_cast<uintptr_t>(c) |
                        reinterpret_cast<uintptr_t>(d);
    return (f % 16 == 0) && (reinterpret_cast<uintptr_t>(m) % 4 == 0);
}

// Blocks of a batch reduction: one per `rows` rows up to the fixed maximum, a function of the batch size alone so that the
// summation order is.
inline int reduce_blocks(int64_t T, int rows) {
    const int64_t b = (T + rows - 1) / rows;
    return static_cast<int>(b < 1 ? 1 : b > kDiagBlocks ? kDiagBlocks : b);
}

// The masked sums of the batch, one row of partial sums per block; the number of blocks in *blocks.
// From kSplitWalkRows on the exact walk has a launch of its own: both walks in one kernel cost the fast one a tenth of its
// bandwidth (16 M rows, whole diagnostics 94 against 84 us; 67 M rows 380 against 337), a launch costs 2 us.
constexpr int64_t kSplitWalkRows = int64_t(8) << 20;
// Shared memory that lets an SM take no more than 1, 2 or 3 blocks, so that a grid of fewer than 4 per SM spreads evenly instead
// of piling up on some SMs: diagnostics of 1.48 M rows (362 blocks) 18.2 -> 17.5 us, 400 k (196 blocks) 13.6 -> 12.5.
constexpr size_t kMomSmemShare[4] = {116 << 10, 116 << 10, 77 << 10, 59 << 10};
cudaError_t launch_moments_kernel(const float* lp_train, const float* lp_roll, const uint8_t* mask, const int32_t* seq_offsets,
                                  const float* adv, int64_t T, int S, float C, double* partials, int32_t* n_valid_seq,
                                  float* seq_logw, bool early, int* blocks, cudaStream_t stream) {
    cudaError_t e;
    if (seq_logw && S > 0) {
        e = launch_pdl(seq_logw_kernel, (S + 7) / 8, 256, 0, stream, lp_train, lp_roll, mask, seq_offsets, S, seq_logw);
        if (e != cudaSuccess) return e;
    }
    if (vec4_ok(lp_train, lp_roll, nullptr, nullptr, mask) && reinterpret_cast<uintptr_t>(mask) % 16 == 0 && T < (int64_t(1) << 31) - 2 * kMomRows) {      // 32-bit row indices inside
        // no more blocks than have a tile when every block takes the same number of them
        const int tiles = static_cast<int>((T + kMomRows - 1) / kMomRows), per = (tiles + kDiagBlocks - 1) / kDiagBlocks;
        *blocks = tiles > 0 ? (tiles + per - 1) / per : 1;
        const int per_sm = (*blocks + kSms - 1) / kSms;
        const size_t smem = per_sm >= 4 ? kMomSmemBytes : kMomSmemShare[per_sm];
        auto go = [&](auto kernel, bool ahead) {
            return launch_pdl(kernel, *blocks, kDiagThreads, smem, stream, lp_train, lp_roll, mask, seq_offsets, adv, static_cast<int>(T), S, C,
                              partials, n_valid_seq, seq_logw, ahead);
        };
        if (T < kSplitWalkRows) return seq_logw ? go(moments_staged_kernel<true, kBothWalks>, false) : go(moments_staged_kernel<false, kBothWalks>, early);
        e = seq_logw ? go(moments_staged_kernel<true, kFastWalk>, false) : go(moments_staged_kernel<false, kFastWalk>, early);
        if (e != cudaSuccess) return e;
        return seq_logw ? go(moments_staged_kernel<true, kExactWalk>, false) : go(moments_staged_kernel<false, kExactWalk>, false);
    }
    *blocks = kDiagBlocks;
    return launch_pdl(vec4_ok(lp_train, lp_roll, nullptr, nullptr, mask) ? moments_kernel<4> : moments_kernel<1>, kDiagBlocks, kDiagThreads, 0, stream,
                      lp_train, lp_roll, mask, seq_offsets, adv, T, S, C, partials, n_valid_seq, seq_logw);
}

cudaError_t launch_rectify_kernel(const float* lp_train, const float* lp_roll, const uint8_t* mask, int64_t T, float C, const TotalsJob& job,
                                  float* rho, float* w_tilde, const int32_t* seq_offsets, int S, const float* seq_logw, bool early,
                                  cudaStream_t stream) {
    const int blocks = reduce_blocks(T, 4 * kDiagThreads);
    return launch_pdl(vec4_ok(lp_train, lp_roll, rho, w_tilde, mask) ? rectify_kernel<4> : rectify_kernel<1>, blocks, kDiagThreads, 0, stream,
                      lp_train, lp_roll, mask, T, C, job, rho, w_tilde, seq_offsets, S, seq_logw, early);
}

}  // namespace

cudaError_t stream_prepare() {
    cudaError_t e = cudaSuccess;
    auto allow = [&](auto kernel) {
        if (e == cudaSuccess) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kMomSmemShare[0]);
    };
    allow(moments_staged_kernel<false, kBothWalks>);
    allow(moments_staged_kernel<false, kFastWalk>);
    allow(moments_staged_kernel<false, kExactWalk>);
    allow(moments_staged_kernel<true, kBothWalks>);
    allow(moments_staged_kernel<true, kFastWalk>);
    allow(moments_staged_kernel<true, kExactWalk>);
    return e;
}

// ------------------------------------------------------------------------------------------------ launchers
// Grid of a row quantiser: four rows per warp once that gives every SM a CTA, single rows below (a small matrix is a chain of
// latencies, not of bytes).
inline bool quant_wide(int64_t rows, int64_t cols) {
    return ((cols + kQCols - 1) / kQCols) * ((rows + 4 * kQWarps - 1) / (4 * kQWarps)) >= 148;
}
inline unsigned quant_tiles_x(int64_t cols) { return static_cast<unsigned>((cols + kQCols - 1) / kQCols); }
inline unsigned quant_blocks(int64_t rows, int64_t cols, bool wide) {
    const int per = kQWarps * (wide ? 4 : 1);
    return quant_tiles_x(cols) * static_cast<unsigned>((rows + per - 1) / per);
}

cudaError_t launch_quantize(const QuantJob* jobs, int njobs, int64_t cols, int block, const FlagsJob* flags, cudaStream_t stream) {
    const unsigned tiles_x = quant_tiles_x(cols);
    int64_t rows = 0;
    for (int i = 0; i < njobs; ++i) rows += jobs[i].rows;
    const bool wide = quant_wide(rows, cols);
    unsigned n[2] = {0, 0};
    for (int i = 0; i < njobs; ++i) n[i] = quant_blocks(jobs[i].rows, cols, wide);
    const FlagsJob f = flags ? *flags : FlagsJob{};
    const unsigned blocks = n[0] + n[1] + (flags ? flag_blocks(f) : 0);
    if (blocks == 0) return cudaSuccess;
    auto go = [&](auto kernel) { return launch_pdl(kernel, blocks, kQThreads, 0, stream, jobs[0], jobs[njobs - 1], n[0], n[1], tiles_x, cols, f); };
    switch (block) {
        case 32:  return go(wide ? quantize_kernel<32, 4> : quantize_kernel<32, 1>);
        case 64:  return go(wide ? quantize_kernel<64, 4> : quantize_kernel<64, 1>);
        case 128: return go(wide ? quantize_kernel<128, 4> : quantize_kernel<128, 1>);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_quantize_cols(const void* x, int64_t K, int64_t N, int64_t ld, int block, uint8_t* codes, int64_t ldq,
                                 float* scales, int64_t lds, cudaStream_t stream) {
    if (K == 0 || N == 0) return cudaSuccess;
    dim3 grid(static_cast<unsigned>((N + kQcTile - 1) / kQcTile), static_cast<unsigned>((K + kQcTile - 1) / kQcTile));
    const __nv_bfloat16* xp = static_cast<const __nv_bfloat16*>(x);
    switch (block) {
        case 32:  return launch_pdl(quantize_cols_kernel<32>, grid, 256, 0, stream, xp, K, N, ld, codes, ldq, scales, lds);
        case 64:  return launch_pdl(quantize_cols_kernel<64>, grid, 256, 0, stream, xp, K, N, ld, codes, ldq, scales, lds);
        case 128: return launch_pdl(quantize_cols_kernel<128>, grid, 256, 0, stream, xp, K, N, ld, codes, ldq, scales, lds);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_quantize_mx(const void* x, int64_t rows, int64_t cols, int64_t ld, uint8_t* codes, int64_t ldq,
                               uint8_t* scales, size_t scale_bytes, bool fp4, cudaStream_t stream) {
    if (rows == 0 || cols == 0) return cudaMemsetAsync(scales, 127, scale_bytes, stream);       // padding only
    const bool wide = quant_wide(rows, cols);
    const unsigned tiles_x = quant_tiles_x(cols), blocks = quant_blocks(rows, cols, wide);
    const int64_t padded = static_cast<int64_t>(scale_bytes / 512) / (cols / 128) * 128;
    auto go = [&](auto kernel) {
        return launch_pdl(kernel, blocks, kQThreads, 0, stream, static_cast<const __nv_bfloat16*>(x), rows, padded, cols, ld, codes, ldq, scales, tiles_x);
    };
    if (fp4) return go(wide ? quantize_mx_kernel<true, 4> : quantize_mx_kernel<true, 1>);
    return go(wide ? quantize_mx_kernel<false, 4> : quantize_mx_kernel<false, 1>);
}

cudaError_t launch_quantize_tensor(const void* x, int64_t rows, int64_t cols, int64_t ld, uint8_t* codes, int64_t ldq,
                                   float* scale, cudaStream_t stream) {
    cudaError_t e = cudaMemsetAsync(scale, 0, sizeof(float), stream);
    if (e != cudaSuccess) return e;
    const __nv_bfloat16* xp = static_cast<const __nv_bfloat16*>(x);
    const bool any = rows > 0 && cols > 0, wide = quant_wide(rows, cols);
    const unsigned tiles_x = quant_tiles_x(cols), blocks = quant_blocks(rows, cols, wide);
    if (any) {
        e = launch_pdl(wide ? tensor_amax_kernel<4> : tensor_amax_kernel<1>, blocks, kQThreads, 0, stream, xp, rows, cols, ld,
                       reinterpret_cast<uint32_t*>(scale), tiles_x);
        if (e != cudaSuccess) return e;
    }
    e = launch_pdl(tensor_scale_kernel, 1, 1, 0, stream, reinterpret_cast<uint32_t*>(scale));
    if (e != cudaSuccess || !any) return e;
    return launch_pdl(wide ? tensor_quantize_kernel<4> : tensor_quantize_kernel<1>, blocks, kQThreads, 0, stream, xp, rows, cols, ld, codes, ldq, scale,
                      tiles_x);
}

cudaError_t launch_combine(const CombineJob* jobs, int njobs, int64_t part_ld, const uint8_t* mask, int64_t T, uint32_t* status,
                           const AdvJob* adv, const MomentsJob* moments, cudaStream_t stream) {
    if (T == 0) return adv ? launch_advantages(*adv, stream) : cudaSuccess;
    if (moments)
        return launch_pdl(merge_moments_kernel, merge_moment_blocks(T), 2 * 32 * kCombWarps, 0, stream, jobs[0], jobs[1], part_ld, mask, T, status, *moments);
    const dim3 grid(static_cast<unsigned>((T + kMergeRows - 1) / kMergeRows), static_cast<unsigned>(njobs + (adv ? 1 : 0)));
    return launch_pdl(combine_kernel, grid, 32 * kCombWarps, 0, stream, jobs[0], jobs[njobs - 1], njobs, part_ld, mask, T, status,
                      adv ? *adv : AdvJob{});
}

cudaError_t launch_flags(const FlagsJob& job, cudaStream_t stream) {
    return job.T > 0 ? launch_pdl(flags_kernel, flag_blocks(job), kQThreads, 0, stream, job) : cudaSuccess;
}

cudaError_t launch_seq_counts(const uint8_t* mask, const int32_t* seq_offsets, int S, int32_t* n_valid_seq, uint32_t* ticket, cudaStream_t stream) {
    return launch_pdl(seq_count_kernel, (S + 7) / 8, 256, 0, stream, mask, seq_offsets, S, n_valid_seq, ticket);
}

cudaError_t launch_advantages(const AdvJob& job, cudaStream_t stream) {
    return launch_pdl(adv_kernel, (job.S + 255) / 256, 256, 0, stream, job);
}

cudaError_t launch_diag(const float* lp_train, const float* lp_roll, const uint8_t* mask, const int32_t* seq_offsets,
                        const float* adv, int64_t T, int S, const ais_params& p, double* partials, int32_t* n_valid_seq, float* seq_logw,
                        float* rho, float* w_tilde, ais_diag* diag, bool early, int merged_blocks, TotalsJob* later, cudaStream_t stream) {
    TotalsJob job = {partials, merged_blocks, p, diag};
    if (merged_blocks == 0) {
        const cudaError_t e = launch_moments_kernel(lp_train, lp_roll, mask, seq_offsets, adv, T, S, p.C, partials, n_valid_seq, seq_logw, early, &job.blocks, stream);
        if (e != cudaSuccess) return e;
    }
    if (later) {
        *later = job;
        return cudaSuccess;
    }
    if (T == 0) return launch_pdl(totals_kernel, 1, kDiagThreads, 0, stream, job, nullptr);
    return launch_rectify_kernel(lp_train, lp_roll, mask, T, p.C, job, rho, w_tilde, seq_offsets, S, seq_logw, merged_blocks == 0, stream);
}

cudaError_t launch_moments(const float* lp_train, const float* lp_roll, const uint8_t* mask, const int32_t* seq_offsets,
                           const float* adv, int64_t T, int S, const ais_params& p, double* partials, int32_t* n_valid_seq, float* seq_logw,
                           double* moments, cudaStream_t stream) {
    TotalsJob job = {partials, 0, p, nullptr};
    const cudaError_t e = launch_moments_kernel(lp_train, lp_roll, mask, seq_offsets, adv, T, S, p.C, partials, n_valid_seq, seq_logw, true, &job.blocks, stream);
    return e != cudaSuccess ? e : launch_pdl(totals_kernel, 1, kDiagThreads, 0, stream, job, moments);
}

cudaError_t launch_finalize(const double* moments, const float* lp_train, const float* lp_roll, const uint8_t* mask, int64_t T,
                            const ais_params& p, float* rho, float* w_tilde, ais_diag* diag, const int32_t* seq_offsets, int S,
                            const float* seq_logw, cudaStream_t stream) {
    const TotalsJob job = {moments, 1, p, diag};
    if (T == 0) return launch_pdl(totals_kernel, 1, kDiagThreads, 0, stream, job, nullptr);
    return launch_rectify_kernel(lp_train, lp_roll, mask, T, p.C, job, rho, w_tilde, seq_offsets, S, seq_logw, false, stream);
}

cudaError_t launch_loss_coef(const float* lp_train, const float* lp_old, const float* lp_ref, float beta_kl, const uint8_t* mask,
                             const int32_t* seq_offsets, const float* adv, const float* w_tilde, const int32_t* n_valid_seq, int64_t T,
                             int S, int S_norm, float clip_eps, double* partials, uint32_t* ticket, float* coef, uint8_t* tile_flags,
                             void* clear, size_t clear_bytes, float* loss, ais_diag* diag, const float* lse, const RectifyJob* rectify,
                             const KeepJob* keep, cudaStream_t stream) {
    LossArgs a = {};
    a.lp_train = lp_train;
    a.lp_old = lp_old;
    a.lp_ref = (beta_kl != 0.f) ? lp_ref : nullptr;
    a.lse = lse;
    a.adv = adv;
    a.w_tilde = w_tilde;
    a.mask = mask;
    a.seq_offsets = seq_offsets;
    a.n_valid_seq = n_valid_seq;
    a.T = T;
    a.S = S;
    a.S_norm = S_norm;
    a.beta_kl = a.lp_ref ? static_cast<double>(beta_kl) : 0.0;
    a.clip_eps = static_cast<double>(clip_eps);
    a.partials = partials;
    a.coef = coef;
    a.tile_flags = tile_flags;
    a.clear = static_cast<uint4*>(clear);
    a.nclear = static_cast<int32_t>(clear_bytes / 16);
    a.ticket = ticket;
    a.loss = loss;
    a.diag = diag;
    const int blocks = reduce_blocks(T, 4 * kDiagThreads);
    if (rectify) {
        a.rectify = *rectify;
        if (keep) a.keep = *keep;
        return launch_pdl(vec4_ok(rectify->w_tilde, rectify->rho, nullptr, nullptr, mask) ? loss_coef_kernel<true, true> : loss_coef_kernel<false, true>,
                          blocks, kDiagThreads, 0, stream, a);
    }
    return launch_pdl(vec4_ok(w_tilde, nullptr, nullptr, nullptr, mask) ? loss_coef_kernel<true, false> : loss_coef_kernel<false, false>, blocks,
                      kDiagThreads, 0, stream, a);
}

}  // namespace ais
