// C ABI of the library: argument validation, workspace carving, tensor-map construction and the order
// in which the kernels of each entry point are enqueued.  Declarations and contracts live in include/ais.h.
#include <cuda.h>
#include <cuda_runtime.h>
#include <cudaTypedefs.h>
#include <math.h>
#include <stdint.h>
#include <string.h>

#include <atomic>
#include <mutex>

#include "../../include/ais.h"
#include "host_setup.cuh"
#include "lmhead.cuh"
#include "stream_kernels.cuh"

namespace ais {

namespace {
constexpr int kMaxDevices = 64;
struct DeviceInfo {
    bool ready = false;      // set-up succeeded on this device
    bool wrong_arch = false; // not an sm_100 device: remembered, every later call fails at once
    int num_sms = 0;
};
DeviceInfo g_dev[kMaxDevices];
std::mutex g_mutex;
PFN_cuTensorMapEncodeTiled_v12000 g_encode = nullptr;
std::atomic<long long> g_wait_cycles{0};
}  // namespace

int64_t wait_cycles() { return g_wait_cycles.load(); }

// Per-device set-up, done once per device with that device current: checks the architecture, raises the kernels'
// dynamic shared-memory limit and resolves the driver's tensor-map encoder.  Only the architecture check is
// remembered as a failure; any other failed step (a CUDA call that could not get resources, say) is tried again
// by the next call.
int device_setup(int* num_sms) {
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return AIS_ERR_DEVICE;
    std::lock_guard<std::mutex> lock(g_mutex);
    DeviceInfo& info = g_dev[dev];
    if (info.wrong_arch) return AIS_ERR_DEVICE;
    if (!info.ready) {
        cudaDeviceProp prop;
        if (cudaGetDeviceProperties(&prop, dev) != cudaSuccess) return AIS_ERR_DEVICE;
        if (prop.major != 10) {
            info.wrong_arch = true;
            return AIS_ERR_DEVICE;
        }
        if (!g_encode) {
            void* fn = nullptr;
            cudaDriverEntryPointQueryResult qres;
            if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &qres) != cudaSuccess ||
                qres != cudaDriverEntryPointSuccess || !fn)
                return AIS_ERR_DEVICE;
            g_encode = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(fn);
        }
        if (lmhead_prepare() != cudaSuccess || stream_prepare() != cudaSuccess) return AIS_ERR_DEVICE;
        info.num_sms = prop.multiProcessorCount;
        info.ready = true;
    }
    if (num_sms) *num_sms = info.num_sms;
    return AIS_OK;
}

// 2-D row-major tensor map: dim0 is the contiguous axis.
bool make_tmap(CUtensorMap* map, CUtensorMapDataType dtype, const void* base, uint64_t dim0, uint64_t dim1,
               uint64_t stride1_bytes, uint32_t box0, uint32_t box1, CUtensorMapSwizzle swz) {
    if (!g_encode) return false;
    cuuint64_t dims[2] = {dim0, dim1};
    cuuint64_t strides[1] = {stride1_bytes};
    cuuint32_t box[2] = {box0, box1};
    cuuint32_t estr[2] = {1, 1};
    CUresult r = g_encode(map, dtype, 2, const_cast<void*>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, swz,
                          CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS;
}

bool make_tmap_blocks(CUtensorMap* map, const void* base, uint64_t dim0, uint64_t dim1, uint64_t stride1_bytes) {
    if (!g_encode) return false;
    cuuint64_t dims[3] = {64, dim1, (dim0 + 63) / 64};
    cuuint64_t strides[2] = {stride1_bytes, 128};
    cuuint32_t box[3] = {64, 64, 4};
    cuuint32_t estr[3] = {1, 1, 1};
    return g_encode(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                    CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// The units of a pass are (row tile, vocabulary range) pairs handed round robin to one persistent CTA per SM, so its time
// is waves x tiles of the longest range.  Four ranges for everybody left a response of 613 rows (5 row tiles) on 20 of 148
// SMs (3.2 ms per pass at d = 4096, V = 151936) and ran 79 row tiles as three waves where 2.1 were full.  The number of
// ranges with the least waves x tiles wins, with a handicap for many ranges: the fewer row tiles are in flight, the more
// often W is read, and in the passes that run into the power cap an idle SM costs less than that (2,500 rows: 7 ranges in one
// wave 2.44 ms, 22 in three better filled ones 2.75; 58,142 rows at d = 5120: 7 ranges 58.1 ms, 11 61.5).  The FP8 block
// pass does not reach the cap and takes the balance (11 ranges 48.4 ms, 4 52.3).  From below the number is bounded by L2:
// the hidden rows of the row tiles in flight are read again for every column tile and should take no more than 40 MB of it.
int unit_rows_of(TileKind kind) { return kind == kTileOne ? kBM : kPairRows; }
int tile_cols_of(TileKind kind) { return kind == kTileBlock ? kPairCols : kBN; }
double range_handicap(TileKind kind) { return kind == kTileBlock ? 400.0 : 120.0; }
bool ranges_fit_l2(TileKind kind, int64_t in_flight, int d) {
    return in_flight * (unit_rows_of(kind) / kBM) * d * (kind == kTileBlock ? 128 : 256) <= (int64_t(40) << 20);
}
PassPlan plan_kind(TileKind kind, int64_t rows, int V, int d, int most, int forced, double* cost) {
    const int unit_rows = unit_rows_of(kind), tile_cols = tile_cols_of(kind);
    const int64_t units = rows > 0 ? (rows + unit_rows - 1) / unit_rows : 1;
    const int col_tiles = (V + tile_cols - 1) / tile_cols;
    if (most > col_tiles) most = col_tiles;
    if (most < 1) most = 1;
    int best = 1;
    double best_cost = 0.0;
    for (int s = 1; s <= most; ++s) {
        if (forced > 0 && s != (forced < most ? forced : most)) continue;
        int64_t in_flight = kSms / s > 0 ? kSms / s : 1;
        if (in_flight > units) in_flight = units;
        if (!ranges_fit_l2(kind, in_flight, d) && s < most && forced <= 0) continue;
        const int64_t waves = (units * s + kSms - 1) / kSms;
        const double c = static_cast<double>(waves) * ((col_tiles + s - 1) / s) * (1.0 + s / range_handicap(kind));
        if (best_cost == 0.0 || c < best_cost) { best = s; best_cost = c; }
    }
    // clocks of a tile: 512 per stage and row tile on the tensor cores at best.  One row tile: 620, and no less than its epilogue
    // takes; two: 1,040 plus what the skew at the ends of a tile leaves exposed.
    const double stages = d / 64.0;
    const double tile = kind == kTileTwo ? fmax(1040.0 * stages + 700.0, 7500.0) : fmax(620.0 * stages, 3500.0);
    if (cost) *cost = best_cost * tile;
    return {kind == kTileTwo, best, unit_rows, tile_cols};
}

// Rows x ranges that plan_kind does not exceed for any batch of up to `rows` rows.  Its own choice does not grow with the batch
// (5 row tiles take more ranges than 6), and a workspace sized by it for the largest batch would be too small for a shorter
// one.  The choice s costs no less than units x col_tiles / kSms x (1 + s / h) and no more than that of any t within the L2
// bound, less than (units x t / kSms + 1) x (col_tiles / t + 1) x (1 + t / h); so units x s stays below a line in units for
// every t, and the least of these rises with units.
int64_t most_range_rows(TileKind kind, int64_t rows, int V, int d, int most, int forced) {
    const int64_t units = rows > 0 ? (rows + unit_rows_of(kind) - 1) / unit_rows_of(kind) : 1;
    const int col_tiles = (V + tile_cols_of(kind) - 1) / tile_cols_of(kind);
    if (most > col_tiles) most = col_tiles;
    if (forced > 0) return (forced < most ? forced : most) * units * unit_rows_of(kind);
    const double h = range_handicap(kind), u = static_cast<double>(units);
    double s_u = most * u;
    for (int t = 1; t <= most; ++t)
        if (t == most || ranges_fit_l2(kind, kSms / t, d))
            s_u = fmin(s_u, h * ((u + static_cast<double>(kSms) / t) * (1.0 + static_cast<double>(t) / col_tiles) * (1.0 + t / h) - u));
    return static_cast<int64_t>(ceil(s_u * unit_rows_of(kind)));
}

PassPlan plan_pass(int64_t rows, int V, int d, int most, int forced) {
    double one = 0.0, two = 0.0;
    const PassPlan a = plan_kind(kTileOne, rows, V, d, most, forced, &one), b = plan_kind(kTileTwo, rows, V, d, most, forced, &two);
    return two < one ? b : a;
}

}  // namespace ais

namespace {

using namespace ais;

inline size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }
inline bool aligned(const void* p, size_t a) { return (reinterpret_cast<uintptr_t>(p) % a) == 0; }

int check_shape(const ais_shape* s) {
    if (!s) return AIS_ERR_NULL;
    if (s->T < 0 || s->T > (int64_t(1) << 31) - 1024) return AIS_ERR_SHAPE;
    if (s->d <= 0 || s->V <= 0 || s->P <= 0 || s->G <= 0) return AIS_ERR_SHAPE;
    if (s->d % 128 != 0 || s->V % 8 != 0) return AIS_ERR_SHAPE;
    if (s->fp8_block != 0 && s->fp8_block != 32 && s->fp8_block != 64 && s->fp8_block != 128 && s->fp8_block != AIS_FP8_MX32 &&
        s->fp8_block != AIS_FP4_MX32)
        return AIS_ERR_SHAPE;
    if (s->fp8_block == AIS_FP4_MX32 && (s->d % 256 != 0 || s->ldh % 32 != 0 || s->ldw % 32 != 0)) return AIS_ERR_SHAPE;
    if (s->fp8_block > 0 && s->d % s->fp8_block != 0) return AIS_ERR_SHAPE;
    if (s->w_layout != AIS_W_VD && s->w_layout != AIS_W_DV) return AIS_ERR_SHAPE;
    if (s->w_layout == AIS_W_DV) {
        // [d, V] head: the block-scaled variants and the per-tensor variant take the [V, d] layout only
        if (s->fp8_block != 32 && s->fp8_block != 64 && s->fp8_block != 128) return AIS_ERR_SHAPE;
        if (s->ldh < s->d || s->ldw < s->V) return AIS_ERR_SHAPE;
        if (s->ldh % 16 != 0 || s->ldw % 8 != 0) return AIS_ERR_ALIGN;
    } else {
        if (s->ldh < s->d || s->ldw < s->d) return AIS_ERR_SHAPE;
        if (s->ldh % 16 != 0 || s->ldw % 16 != 0) return AIS_ERR_ALIGN;
    }
    if (static_cast<int64_t>(s->P) * s->G > (1 << 24)) return AIS_ERR_SHAPE;
    if (s->P_total != 0 && (s->P_total < s->P || static_cast<int64_t>(s->P_total) * s->G > (int64_t(1) << 30))) return AIS_ERR_SHAPE;
    return AIS_OK;
}

int check_params(const ais_params* p) {
    if (!p) return AIS_ERR_NULL;
    if (!(p->C >= 1.0f) || !(p->delta > 0.f) || !(p->gamma > 0.f) || !(p->eps >= 0.f) || !(p->clip_eps >= 0.f) ||
        !(p->beta_var >= 0.f))
        return AIS_ERR_PARAM;
    if (!isnan(p->alpha_override) && !(p->alpha_override >= 0.f && p->alpha_override <= 1.f)) return AIS_ERR_PARAM;
    if (p->vocab_chunk < 0 || !(p->beta_kl >= 0.f)) return AIS_ERR_PARAM;
    return AIS_OK;
}

int check_quantize(const void* x, int64_t rows, int64_t cols, int64_t ld, int block, const uint8_t* codes, int64_t ldq,
                   const float* scales, int64_t lds) {
    if (!x || !codes || !scales) return AIS_ERR_NULL;
    if (rows < 0 || cols < 0 || (block != 32 && block != 64 && block != 128)) return AIS_ERR_SHAPE;
    if (cols % block != 0 || ld < cols || ldq < cols || lds < rows) return AIS_ERR_SHAPE;
    if (ld % 8 != 0 || ldq % 8 != 0 || !aligned(x, 16) || !aligned(codes, 8) || !aligned(scales, 4)) return AIS_ERR_ALIGN;
    if (rows > (int64_t(1) << 31) - 1024) return AIS_ERR_SHAPE;
    return AIS_OK;
}

// vocab_chunk asks for its own number of ranges (at most 64); 0: the plan decides.
int forced_ranges(const ais_shape* s, const ais_params* p) {
    if (p->vocab_chunk <= 0) return 0;
    const int n = (s->V + p->vocab_chunk - 1) / p->vocab_chunk;
    return n > 64 ? 64 : n;
}

// dH: the last, partial wave of 256 x 256 output tiles would leave most SMs idle for the length of a whole contraction
// over the vocabulary (16 tiles of 148 SMs for one row pair at d = 4096, 60 of the 800 = 5.4 waves for 10,003 rows at
// d = 5120).  Its tiles are split into ranges of the contraction whose fp32 partial tiles are added afterwards.
// split_cost: microseconds of the tail for ks ranges, from the 0.83 us of a stage fill at 1.5 PFLOP/s and 256 KB written
// and read per partial tile at 6 TB/s plus the extra launch.  A range keeps at least four stage fills (the depth of the
// ring plus one), and the partial tiles number at most kSplitSlots (116 MB).
constexpr int kSplitSlots = 3 * kSms;
constexpr double kFillUs = 0.83, kSplitUs = 6.0, kSlotUs = 0.087;
double split_cost(int tiles, int ks, int ksteps) {
    const double waves = (static_cast<int64_t>(tiles) * ks + kSms - 1) / kSms;
    return waves * ((ksteps + ks - 1) / ks) * kFillUs + (ks > 1 ? kSplitUs + tiles * ks * kSlotUs : 0.0);
}
// Partial tiles that no pass over up to `tiles` output tiles asks pick_ksplit for: a split has to pay for its partial tiles
// within the ksteps x kFillUs of the tail as it is.  Like most_range_rows, for a workspace that serves shorter batches.
int most_split_slots(int64_t tiles, int ksteps) {
    const int64_t tail = tiles < kSms ? tiles : kSms - 1;
    const int64_t ks = ksteps / 4 < 64 ? ksteps / 4 : 64;
    const double paid = (ksteps * kFillUs - kSplitUs) / kSlotUs;
    const double slots = fmin(fmin(static_cast<double>(tail * ks), paid), static_cast<double>(kSplitSlots));
    return ks < 2 || slots < 2.0 ? 0 : static_cast<int>(slots);
}
int pick_ksplit(int tiles, int ksteps, int slots) {
    int best = 1;
    double best_cost = split_cost(tiles, 1, ksteps);
    for (int ks = 2; ks <= 64 && ks * tiles <= slots && ks * 4 <= ksteps; ++ks) {
        const double c = split_cost(tiles, ks, ksteps);
        if (c < 0.97 * best_cost) { best = ks; best_cost = c; }
    }
    return best;
}

constexpr size_t kPaceRingBytes = kPaceRing * sizeof(uint32_t);

struct Layout {
    int64_t t_ld;          // padded length of per-row vectors
    PassPlan train, roll;  // how the two forward passes split
    size_t off_part[2], part_bytes;               // forward partials of the trainer and the rollout pass: max, sum, target planes
    size_t off_diag, off_loss;                    // partial sums of the batch moments and of the loss (doubles)
    size_t off_flags;                             // one byte per 128-row tile: anything to compute there?
    size_t off_pace;                              // two rings of counters that keep the CTAs of a tensor-core launch in step
    size_t off_ticket;                            // counters of the loss kernel
    size_t off_coef, off_nseq;                    // backward: c_t, valid rows per sequence
    size_t off_scale, off_redo;                   // backward, exponent form: row factors, row tiles to recompute
    size_t off_seqw;                              // sequence-level variant: log weight per sequence
    size_t off_split;                             // dH: partial tiles of the split units
    int split_slots, ksplit;                      // how many there is room for; ksplit > 0: ranges fixed by the shape alone
    size_t off_u;                                 // backward scratch
    int64_t ldU;
    size_t fixed_bytes;                           // everything but the scratch rows
    size_t u_row_bytes;
};

Layout compute_layout(const ais_shape* s, const ais_params* p) {
    Layout L;
    L.t_ld = static_cast<int64_t>(align_up(static_cast<size_t>(s->T > 0 ? s->T : 1), 64));
    const int forced = forced_ranges(s, p);
    L.train = plan_pass(s->T, s->V, s->d, kMaxRanges, forced);
    L.roll = s->fp8_block > 0    ? plan_kind(kTileBlock, s->T, s->V, s->d, kMaxRanges, forced, nullptr)
             : s->fp8_block == 0 ? plan_pass(s->T, s->V, s->d / 2, kMaxRanges, forced)
                                 : plan_kind(kTileOne, s->T, s->V, s->d, kMaxRanges, forced, nullptr);
    // every size below is one that a batch of fewer rows does not exceed
    int64_t range_rows = 0;
    auto reserve = [&](TileKind kind, int d) {
        const int64_t r = most_range_rows(kind, s->T, s->V, d, kMaxRanges, forced);
        if (r > range_rows) range_rows = r;
    };
    reserve(kTileOne, s->d);
    reserve(kTileTwo, s->d);
    if (s->fp8_block > 0) {
        reserve(kTileBlock, s->d);
    } else if (s->fp8_block == 0) {
        reserve(kTileOne, s->d / 2);
        reserve(kTileTwo, s->d / 2);
    }
    size_t off = 0;
    L.part_bytes = align_up(2 * static_cast<size_t>(range_rows) * sizeof(float), 256);
    for (int i = 0; i < 2; ++i) { L.off_part[i] = off; off += 3 * L.part_bytes; }
    L.off_flags = off;  off += align_up(static_cast<size_t>(L.t_ld / kBM + 2), 256);
    L.off_pace = off;   off += 2 * kPaceRingBytes;
    L.off_ticket = off; off += 256;
    L.off_diag = off;   off += align_up(static_cast<size_t>(kDiagBlocks) * kNumMoments * sizeof(double), 256);
    L.off_loss = off;   off += align_up(static_cast<size_t>(kDiagBlocks) * 2 * sizeof(double), 256);
    L.off_coef = off;   off += align_up(static_cast<size_t>(L.t_ld) * sizeof(float), 256);
    L.off_nseq = off;   off += align_up(static_cast<size_t>(s->P) * s->G * sizeof(int32_t), 256);
    L.off_scale = off;  off += align_up(static_cast<size_t>(L.t_ld) * sizeof(float), 256);
    L.off_redo = off;   off += align_up(static_cast<size_t>(L.t_ld / kBM + 2), 256);
    L.off_seqw = off;   off += align_up(static_cast<size_t>(s->P) * s->G * sizeof(float), 256);
    {
        // a batch whose dH tiles do not fill one wave gets its ranges from its size alone, so that the split (and with it
        // every bit of dH) is the same whatever the workspace lets a pass hold
        const int64_t tiles = ((s->T + kDhRows - 1) / kDhRows) * ((s->d + kBN - 1) / kBN);
        const int ksteps = (s->V + 63) / 64;
        L.split_slots = most_split_slots(tiles, ksteps);
        L.ksplit = tiles >= kSms ? 0 : tiles > 0 ? pick_ksplit(static_cast<int>(tiles), ksteps, L.split_slots) : 1;
    }
    L.off_split = off;  off += static_cast<size_t>(L.split_slots) * kPartTileFloats * sizeof(float);
    L.off_u = off;
    L.ldU = static_cast<int64_t>(align_up(static_cast<size_t>(s->V), 64));
    L.fixed_bytes = off;
    L.u_row_bytes = static_cast<size_t>(L.ldU) * sizeof(__nv_bfloat16);
    return L;
}

// The layout is a function of the sizes alone, and a program calls with the same ones again and again: each thread keeps its
// last.  The search over ranges takes 2.8 us for a 151,936-row head, a fifth of a diagnostics call of a few thousand rows,
// and a step in one call asks four times.
Layout make_layout(const ais_shape* s, const ais_params* p) {
    struct Key {
        int64_t T;
        int32_t d, V, P, G, fp8_block, vocab_chunk;
    };
    static thread_local Key key = {-1, 0, 0, 0, 0, 0, 0};
    static thread_local Layout layout;
    if (key.T != s->T || key.d != s->d || key.V != s->V || key.P != s->P || key.G != s->G || key.fp8_block != s->fp8_block ||
        key.vocab_chunk != p->vocab_chunk) {
        layout = compute_layout(s, p);
        key = {s->T, s->d, s->V, s->P, s->G, s->fp8_block, p->vocab_chunk};
    }
    return layout;
}

constexpr int64_t kBwdRowsRecommended = 2 * kSms * kBM;

// Points a pass at its pacing ring.  The passes of a call alternate between two rings: the kernel before the first pass
// clears both (ring_bytes of them), every later pass finds its own cleared by the one before it (`clears_next`).
// tiles_per_unit = the largest number of column tiles a unit of the launch walks.  A CTA with only a few announcements to
// make cannot drift far enough to matter and runs without pacing, so small batches have no rings to clear either.
constexpr int64_t kPaceMinFills = 256;
bool arm_pace(LmheadArgs& a, uint8_t* ws, const Layout& L, int tiles_per_unit, int units, int ctas, int pass, bool clears_next) {
    const int64_t fills = static_cast<int64_t>(tiles_per_unit) * a.ksteps;
    const int64_t waves = (units + ctas - 1) / ctas;
    a.pace_clear = clears_next ? reinterpret_cast<uint32_t*>(ws + L.off_pace + ((pass + 1) & 1) * kPaceRingBytes) : nullptr;
    a.pace = ctas < 2 || fills * waves < kPaceMinFills ? nullptr : reinterpret_cast<uint32_t*>(ws + L.off_pace + (pass & 1) * kPaceRingBytes);
    a.pace_per_unit = static_cast<int32_t>((fills + kPaceFills - 1) / kPaceFills);
    return a.pace != nullptr;
}

// Width of a [d, V] head that its map of 64-column blocks covers (below 64 columns no tile uses that map).
uint64_t whole_blocks(uint64_t V) { return V < 64 ? 64 : V / 64 * 64; }

// Rows of backward scratch that the workspace holds: whole row tiles, no more than the batch has.
int64_t scratch_rows(const Layout& L, int64_t T, size_t workspace_bytes) {
    const int64_t rows = static_cast<int64_t>((workspace_bytes - L.fixed_bytes) / L.u_row_bytes) / kBM * kBM;
    const int64_t t_pad = static_cast<int64_t>(align_up(static_cast<size_t>(T), kBM));
    return rows < t_pad ? rows : t_pad;
}

// What ais_step lets neighbouring stages share: a batch of a few hundred rows is a chain of launches, and these are the ones
// whose work fits into a neighbour's.
struct Fuse {
    const QuantJob* quant = nullptr;     // log-probs: quantise these first, in the opening launch
    int* nquant = nullptr;               // how many; zeroed by that launch
    const AdvJob* adv = nullptr;         // log-probs: advantages in the merging launch; diagnostics: they are there already
    const MomentsJob* moments = nullptr; // log-probs: advantages in the opening launch, batch moments in the merging one;
                                         // diagnostics: their partial sums are there already
    TotalsJob* totals = nullptr;         // diagnostics: leave the end (alpha, rho, w_tilde) to the loss, described here
    const RectifyJob* rectify = nullptr; // loss: form them
    int64_t keep_rows = 0;               // log-probs: leave the exponentials of these rows in the scratch; loss: they are there
    const int32_t* counts = nullptr;     // loss: valid rows per sequence are there already, and so is its cleared ticket
};

}  // namespace

extern "C" {

int ais_version(void) { return AIS_VERSION; }

int ais_set_wait_cycles(int64_t cycles) {
    if (cycles < 0) return AIS_ERR_PARAM;
    g_wait_cycles.store(cycles);
    return AIS_OK;
}

const char* ais_strerror(int status) {
    switch (status) {
        case AIS_OK: return "ok";
        case AIS_ERR_NULL: return "a required pointer is NULL";
        case AIS_ERR_SHAPE: return "invalid or inconsistent shape";
        case AIS_ERR_ALIGN: return "pointer or leading dimension not aligned as required";
        case AIS_ERR_WORKSPACE: return "workspace missing, misaligned or too small";
        case AIS_ERR_DEVICE: return "no sm_100 device, or a CUDA call failed";
        case AIS_ERR_PARAM: return "hyper-parameter out of range";
        case AIS_ERR_LIMIT: return "size beyond a fixed limit of this entry point";
        default: return "unknown status";
    }
}

void ais_default_params(ais_params* p) {
    if (!p) return;
    p->C = 5.0f;
    p->delta = 0.02f;
    p->gamma = 1.2f;
    p->eps = 1e-6f;
    p->beta_var = 1.0f;
    p->clip_eps = 0.2f;
    p->alpha_override = NAN;
    p->adv_std_norm = 0;
    p->vocab_chunk = 0;
    p->beta_kl = 0.0f;
    p->seq_level_weights = 0;
}

size_t ais_workspace_min_bytes(const ais_shape* shape, const ais_params* params) {
    if (check_shape(shape) != AIS_OK || check_params(params) != AIS_OK) return 0;
    const Layout L = make_layout(shape, params);
    return L.fixed_bytes + static_cast<size_t>(kBM) * L.u_row_bytes;
}

size_t ais_workspace_bytes(const ais_shape* shape, const ais_params* params) {
    if (check_shape(shape) != AIS_OK || check_params(params) != AIS_OK) return 0;
    const Layout L = make_layout(shape, params);
    int64_t rows = static_cast<int64_t>(align_up(static_cast<size_t>(shape->T > 0 ? shape->T : 1), kBM));
    if (rows > kBwdRowsRecommended) rows = kBwdRowsRecommended;
    return L.fixed_bytes + static_cast<size_t>(rows) * L.u_row_bytes;
}

int ais_quantize_fp8(const void* x, int64_t rows, int64_t cols, int64_t ld, int block, uint8_t* codes, int64_t ldq,
                     float* scales, int64_t lds, void* stream) {
    int st = check_quantize(x, rows, cols, ld, block, codes, ldq, scales, lds);
    if (st != AIS_OK) return st;
    st = device_setup(nullptr);
    if (st != AIS_OK) return st;
    if (rows == 0 || cols == 0) return AIS_OK;
    const QuantJob job = {x, rows, ld, codes, ldq, scales, lds};
    return launch_quantize(&job, 1, cols, block, nullptr, static_cast<cudaStream_t>(stream)) == cudaSuccess ? AIS_OK : AIS_ERR_DEVICE;
}

int ais_quantize_fp8_cols(const void* x, int64_t rows, int64_t cols, int64_t ld, int block, uint8_t* codes, int64_t ldq,
                          float* scales, int64_t lds, void* stream) {
    if (!x || !codes || !scales) return AIS_ERR_NULL;
    if (rows < 0 || cols < 0 || (block != 32 && block != 64 && block != 128)) return AIS_ERR_SHAPE;
    if (rows % 128 != 0 || cols % 8 != 0 || ld < cols || ldq < rows || lds < cols) return AIS_ERR_SHAPE;
    if (ld % 8 != 0 || ldq % 16 != 0 || !aligned(x, 16) || !aligned(codes, 16) || !aligned(scales, 4)) return AIS_ERR_ALIGN;
    if (cols > (int64_t(1) << 31) - 1024 || rows > (int64_t(1) << 24)) return AIS_ERR_SHAPE;
    int st = device_setup(nullptr);
    if (st != AIS_OK) return st;
    return launch_quantize_cols(x, rows, cols, ld, block, codes, ldq, scales, lds, static_cast<cudaStream_t>(stream)) == cudaSuccess
               ? AIS_OK
               : AIS_ERR_DEVICE;
}

int ais_quantize_fp8_tensor(const void* x, int64_t rows, int64_t cols, int64_t ld, uint8_t* codes, int64_t ldq, float* scale,
                            void* stream) {
    if (!x || !codes || !scale) return AIS_ERR_NULL;
    if (rows < 0 || cols < 0 || cols % 8 != 0 || ld < cols || ldq < cols) return AIS_ERR_SHAPE;
    if (ld % 8 != 0 || ldq % 8 != 0 || !aligned(x, 16) || !aligned(codes, 8) || !aligned(scale, 4)) return AIS_ERR_ALIGN;
    if (rows > (int64_t(1) << 31) - 1024) return AIS_ERR_SHAPE;
    int st = device_setup(nullptr);
    if (st != AIS_OK) return st;
    return launch_quantize_tensor(x, rows, cols, ld, codes, ldq, scale, static_cast<cudaStream_t>(stream)) == cudaSuccess
               ? AIS_OK
               : AIS_ERR_DEVICE;
}

size_t ais_mx_scale_bytes(int64_t rows, int64_t cols) {
    if (rows < 0 || cols <= 0 || cols % 128 != 0) return 0;
    const int64_t chunks = (rows + 255) / 256 * 2;          // 128-row chunks, an even number of them
    return static_cast<size_t>(chunks > 0 ? chunks : 2) * static_cast<size_t>(cols / 128) * 512;
}

int ais_quantize_mxfp8(const void* x, int64_t rows, int64_t cols, int64_t ld, uint8_t* codes, int64_t ldq, uint8_t* scales,
                       void* stream) {
    if (!x || !codes || !scales) return AIS_ERR_NULL;
    if (rows < 0 || cols <= 0 || cols % 128 != 0 || ld < cols || ldq < cols) return AIS_ERR_SHAPE;
    if (ld % 8 != 0 || ldq % 8 != 0 || !aligned(x, 16) || !aligned(codes, 8) || !aligned(scales, 16)) return AIS_ERR_ALIGN;
    if (rows > (int64_t(1) << 31) - 1024) return AIS_ERR_SHAPE;
    int st = device_setup(nullptr);
    if (st != AIS_OK) return st;
    return launch_quantize_mx(x, rows, cols, ld, codes, ldq, scales, ais_mx_scale_bytes(rows, cols), false,
                              static_cast<cudaStream_t>(stream)) == cudaSuccess
               ? AIS_OK
               : AIS_ERR_DEVICE;
}

int ais_quantize_mxfp4(const void* x, int64_t rows, int64_t cols, int64_t ld, uint8_t* codes, int64_t ldq, uint8_t* scales,
                       void* stream) {
    if (!x || !codes || !scales) return AIS_ERR_NULL;
    if (rows < 0 || cols <= 0 || cols % 128 != 0 || ld < cols || ldq < cols / 2) return AIS_ERR_SHAPE;
    if (ld % 8 != 0 || ldq % 4 != 0 || !aligned(x, 16) || !aligned(codes, 4) || !aligned(scales, 16)) return AIS_ERR_ALIGN;
    if (rows > (int64_t(1) << 31) - 1024) return AIS_ERR_SHAPE;
    int st = device_setup(nullptr);
    if (st != AIS_OK) return st;
    return launch_quantize_mx(x, rows, cols, ld, codes, ldq, scales, ais_mx_scale_bytes(rows, cols), true,
                              static_cast<cudaStream_t>(stream)) == cudaSuccess
               ? AIS_OK
               : AIS_ERR_DEVICE;
}

static int logprob_fwd(const ais_shape* shape, const ais_params* params, const void* H, const void* W, const uint8_t* qH,
                       const void* sH_, int64_t ldsH, const uint8_t* qW, const void* sW_, int64_t ldsW, const int32_t* tokens,
                       const uint8_t* mask, float* lp_train, float* lse_train, float* lp_roll, float* lse_roll,
                       uint32_t* dev_status, void* workspace, size_t workspace_bytes, void* stream, const Fuse& fuse) {
    int st = check_shape(shape);
    if (st != AIS_OK) return st;
    st = check_params(params);
    if (st != AIS_OK) return st;
    if (!tokens || !mask) return AIS_ERR_NULL;
    const float* sH = static_cast<const float*>(sH_);
    const float* sW = static_cast<const float*>(sW_);
    const bool do_train = lp_train != nullptr, do_roll = lp_roll != nullptr;
    if (do_train && (!H || !W)) return AIS_ERR_NULL;
    if (do_roll && (!qH || !sH || !qW || !sW)) return AIS_ERR_NULL;
    if (do_train && (!aligned(H, 16) || !aligned(W, 16))) return AIS_ERR_ALIGN;
    const bool per_tensor = shape->fp8_block == 0;
    const bool fp4 = shape->fp8_block == AIS_FP4_MX32;
    const bool mx = shape->fp8_block == AIS_FP8_MX32 || fp4;
    if (do_roll) {
        if (!aligned(qH, 16) || !aligned(qW, 16) || !aligned(sH, 4) || !aligned(sW, 4)) return AIS_ERR_ALIGN;
        if (mx && (!aligned(sH, 16) || !aligned(sW, 16))) return AIS_ERR_ALIGN;
        if (!per_tensor && !mx) {
            if (!aligned(sH, 16) || !aligned(sW, 16)) return AIS_ERR_ALIGN;
            if (ldsH < shape->T || ldsW < shape->V) return AIS_ERR_SHAPE;
            if (ldsH % 4 != 0 || ldsW % 4 != 0) return AIS_ERR_ALIGN;
        }
    }
    const Layout L = make_layout(shape, params);
    if (!workspace || !aligned(workspace, 256) || workspace_bytes < L.off_ticket) return AIS_ERR_WORKSPACE;
    int num_sms = 0;
    st = device_setup(&num_sms);
    if (st != AIS_OK) return st;
    if (shape->T == 0 || (!do_train && !do_roll)) return AIS_OK;

    cudaStream_t s = static_cast<cudaStream_t>(stream);
    uint8_t* ws = static_cast<uint8_t*>(workspace);
    LmheadArgs base;
    memset(&base, 0, sizeof(base));
    base.wait_cycles = wait_cycles();
    base.rows = shape->T;
    base.tokens = tokens;
    base.mask = mask;
    base.ncols = shape->V;
    base.part_ld = L.t_ld;
    base.status = dev_status;
    base.tile_active = ws + L.off_flags;         // row tiles without a single valid row are skipped by the tensor-core passes
    const int64_t T = shape->T, V = shape->V, d = shape->d;
    const bool dv = shape->w_layout == AIS_W_DV;

    // One pass: its arguments, its tensor maps, its share of the merge.
    struct Pass {
        LmheadArgs a;
        CUtensorMap tmA, tmB, tmSA, tmSB;
        int mode, units, ctas;
        bool two;
    } pass[2] = {};
    CombineJob jobs[2];
    int n = 0;
    bool paced = false;
    auto add = [&](int mode, const PassPlan& plan, int ksteps, float* lp, float* lse) -> Pass& {
        Pass& p = pass[n];
        p.mode = mode;
        p.two = plan.two;
        p.a = base;
        const int nsplit = plan.ranges;
        p.a.n_row_tiles = static_cast<int32_t>((T + plan.unit_rows - 1) / plan.unit_rows);
        p.a.n_col_tiles = static_cast<int32_t>((V + plan.tile_cols - 1) / plan.tile_cols);
        p.a.nsplit = nsplit;
        p.a.ksteps = ksteps;
        p.a.sgroups = 1;
        float* parts = reinterpret_cast<float*>(ws + L.off_part[n]);
        p.a.part_m = parts;
        p.a.part_s = parts + L.part_bytes / sizeof(float);
        p.a.part_z = parts + 2 * (L.part_bytes / sizeof(float));
        p.units = p.a.n_row_tiles * nsplit;
        p.ctas = p.units < num_sms ? p.units : num_sms;
        paced |= arm_pace(p.a, ws, L, (p.a.n_col_tiles + nsplit - 1) / nsplit, p.units, p.ctas, n, false);
        // the rollout pass needs nothing from the trainer pass: where both fit side by side it does not wait for it.  Larger
        // passes come one after the other: CTAs that start early wait for the rest of their launch in the pacing ring
        // (9,217 rows, both passes: 16.32 ms overlapped, 16.26 not)
        p.a.overlap = n > 0 && pass[0].ctas + p.ctas <= num_sms ? 1 : 0;
        jobs[n] = {p.a.part_m, p.a.part_s, p.a.part_z, plan.parts(), lp, lse};
        ++n;
        return p;
    };
    bool maps = true;
    if (do_train) {
        // W [V, d]: K-major boxes of 64 hidden units x 256 vocabulary rows.  W [d, V]: the vocabulary is the contiguous
        // axis, four blocks of 64 vocabulary columns x 64 hidden units per copy, and single boxes for the last tile
        const bool keep = fuse.keep_rows > 0;
        Pass& p = add(keep ? (dv ? kFwdKeepDv : kFwdKeep) : dv ? kFwdBf16Dv : kFwdBf16, L.train, shape->d / 64, lp_train, lse_train);
        p.a.U = reinterpret_cast<__nv_bfloat16*>(ws + L.off_u);
        p.a.ldU = L.ldU;
        p.a.block_tiles = static_cast<int32_t>(V / kBN);
        p.a.keep_rows = fuse.keep_rows;
        maps &= make_tmap(&p.tmA, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, H, d, T, shape->ldh * 2, 64, L.train.unit_rows, CU_TENSOR_MAP_SWIZZLE_128B) &&
                (dv ? make_tmap_blocks(&p.tmB, W, whole_blocks(V), d, shape->ldw * 2) &&
                          make_tmap(&p.tmSA, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, W, V, d, shape->ldw * 2, 64, 64, CU_TENSOR_MAP_SWIZZLE_128B)
                    : make_tmap(&p.tmB, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, W, d, V, shape->ldw * 2, 64, kBN, CU_TENSOR_MAP_SWIZZLE_128B));
    }
    if (do_roll && (mx || per_tensor)) {
        // Power-of-two scales per 32 elements: the block-scaled MMA applies them.  One scale per tensor: the two meet in the
        // epilogue.  Either way the whole contraction stays in tensor memory.  FP4 codes are two per byte: the maps see
        // d / 2 bytes per row with half the row stride.
        const int64_t kb = fp4 ? d / 2 : d;
        Pass& p = add(per_tensor ? kFwdFp8T : fp4 ? kFwdMx4 : kFwdMx, L.roll, static_cast<int>(kb / 128), lp_roll, lse_roll);
        p.a.sf_a = static_cast<const uint8_t*>(sH_);
        p.a.sf_b = static_cast<const uint8_t*>(sW_);
        p.a.nk4 = shape->d / 128;
        p.a.scale_a = sH;
        p.a.scale_b = sW;
        maps &= make_tmap(&p.tmA, CU_TENSOR_MAP_DATA_TYPE_UINT8, qH, kb, T, fp4 ? shape->ldh / 2 : shape->ldh, 128, L.roll.unit_rows, CU_TENSOR_MAP_SWIZZLE_128B) &&
                make_tmap(&p.tmB, CU_TENSOR_MAP_DATA_TYPE_UINT8, qW, kb, V, fp4 ? shape->ldw / 2 : shape->ldw, 128, kBN, CU_TENSOR_MAP_SWIZZLE_128B);
    } else if (do_roll) {
        // tiles of 256 rows x 128 columns
        const int64_t nkb = d / shape->fp8_block;
        const int sg = 128 / shape->fp8_block;
        Pass& p = add(kFwdFp8, L.roll, shape->d / 128, lp_roll, lse_roll);
        p.a.sgroups = sg;
        maps &= make_tmap(&p.tmA, CU_TENSOR_MAP_DATA_TYPE_UINT8, qH, d, T, shape->ldh, 128, kPairRows, CU_TENSOR_MAP_SWIZZLE_128B) &&
                make_tmap(&p.tmB, CU_TENSOR_MAP_DATA_TYPE_UINT8, qW, d, V, dv ? d : shape->ldw, 128, kPairCols, CU_TENSOR_MAP_SWIZZLE_128B) &&
                make_tmap(&p.tmSA, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, sH, T, nkb, ldsH * 4, kPairRows, sg, CU_TENSOR_MAP_SWIZZLE_NONE) &&
                make_tmap(&p.tmSB, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, sW, V, nkb, ldsW * 4, kPairCols, sg, CU_TENSOR_MAP_SWIZZLE_NONE);
    }
    if (!maps) return AIS_ERR_DEVICE;
    const FlagsJob flags = {mask, T, ws + L.off_flags, paced ? ws + L.off_pace : nullptr, 2 * kPaceRingBytes, fuse.moments ? *fuse.adv : AdvJob{}};
    const int nquant = fuse.nquant ? *fuse.nquant : 0;
    if ((nquant > 0 ? launch_quantize(fuse.quant, nquant, d, shape->fp8_block, &flags, s) : launch_flags(flags, s)) != cudaSuccess)
        return AIS_ERR_DEVICE;
    if (nquant > 0) *fuse.nquant = 0;
    for (int i = 0; i < n; ++i)
        if ((pass[i].two ? launch_lmhead_pair(pass[i].mode, pass[i].tmA, pass[i].tmB, pass[i].tmSA, pass[i].a, pass[i].ctas, s)
                         : launch_lmhead(pass[i].mode, pass[i].tmA, pass[i].tmB, pass[i].tmSA, pass[i].tmSB, pass[i].a, pass[i].ctas, s)) != cudaSuccess)
            return AIS_ERR_DEVICE;
    if (launch_combine(jobs, n, L.t_ld, mask, T, dev_status, fuse.adv, fuse.moments, s) != cudaSuccess) return AIS_ERR_DEVICE;
    return AIS_OK;
}

int ais_logprob_fwd(const ais_shape* shape, const ais_params* params, const void* H, const void* W, const uint8_t* qH,
                    const void* sH, int64_t ldsH, const uint8_t* qW, const void* sW, int64_t ldsW, const int32_t* tokens,
                    const uint8_t* mask, float* lp_train, float* lse_train, float* lp_roll, float* lse_roll,
                    uint32_t* dev_status, void* workspace, size_t workspace_bytes, void* stream) {
    return logprob_fwd(shape, params, H, W, qH, sH, ldsH, qW, sW, ldsW, tokens, mask, lp_train, lse_train, lp_roll, lse_roll,
                       dev_status, workspace, workspace_bytes, stream, Fuse());
}

// What ais_diagnostics refuses.
static int check_diagnostics(const ais_shape* shape, const ais_params* params, const void* lp_train, const void* lp_roll, const void* mask,
                             const void* seq_offsets, const void* rewards, const void* adv, const void* w_tilde, const void* diag,
                             const void* workspace, size_t workspace_bytes) {
    int st = check_shape(shape);
    if (st != AIS_OK) return st;
    st = check_params(params);
    if (st != AIS_OK) return st;
    if (!lp_train || !lp_roll || !mask || !seq_offsets || !rewards || !adv || !w_tilde || !diag) return AIS_ERR_NULL;
    if (!aligned(diag, 8)) return AIS_ERR_ALIGN;
    const Layout L = make_layout(shape, params);
    if (!workspace || !aligned(workspace, 256) || workspace_bytes < (params->seq_level_weights != 0 ? L.off_split : L.off_coef))
        return AIS_ERR_WORKSPACE;
    return AIS_OK;
}

static int diagnostics(const ais_shape* shape, const ais_params* params, const float* lp_train, const float* lp_roll,
                       const uint8_t* mask, const int32_t* seq_offsets, const float* rewards, float* adv, int32_t* n_valid_seq,
                       float* rho, float* w_tilde, ais_diag* diag, void* workspace, size_t workspace_bytes, void* stream, const Fuse& fuse) {
    int st = check_diagnostics(shape, params, lp_train, lp_roll, mask, seq_offsets, rewards, adv, w_tilde, diag, workspace, workspace_bytes);
    if (st != AIS_OK) return st;
    st = device_setup(nullptr);
    if (st != AIS_OK) return st;
    const Layout L = make_layout(shape, params);
    const bool seq_level = params->seq_level_weights != 0;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    uint8_t* ws = static_cast<uint8_t*>(workspace);
    const int S = shape->P * shape->G;
    if (!fuse.adv &&
        launch_advantages({rewards, S, shape->G, params->adv_std_norm, params->eps, adv, n_valid_seq, reinterpret_cast<uint32_t*>(ws + L.off_ticket)}, s) != cudaSuccess)
        return AIS_ERR_DEVICE;
    if (launch_diag(lp_train, lp_roll, mask, seq_offsets, adv, shape->T, S, *params, reinterpret_cast<double*>(ws + L.off_diag),
                    n_valid_seq, seq_level ? reinterpret_cast<float*>(ws + L.off_seqw) : nullptr, rho, w_tilde,
                    diag, !fuse.adv, fuse.moments ? merge_moment_blocks(shape->T) : 0, fuse.totals, s) != cudaSuccess)
        return AIS_ERR_DEVICE;
    return AIS_OK;
}

int ais_diagnostics(const ais_shape* shape, const ais_params* params, const float* lp_train, const float* lp_roll,
                    const uint8_t* mask, const int32_t* seq_offsets, const float* rewards, float* adv, int32_t* n_valid_seq,
                    float* rho, float* w_tilde, ais_diag* diag, void* workspace, size_t workspace_bytes, void* stream) {
    return diagnostics(shape, params, lp_train, lp_roll, mask, seq_offsets, rewards, adv, n_valid_seq, rho, w_tilde, diag, workspace,
                       workspace_bytes, stream, Fuse());
}

int ais_diag_moments(const ais_shape* shape, const ais_params* params, const float* lp_train, const float* lp_roll,
                     const uint8_t* mask, const int32_t* seq_offsets, const float* rewards, float* adv, int32_t* n_valid_seq,
                     double* moments, float* seq_logw, void* workspace, size_t workspace_bytes, void* stream) {
    int st = check_shape(shape);
    if (st != AIS_OK) return st;
    st = check_params(params);
    if (st != AIS_OK) return st;
    if (!lp_train || !lp_roll || !mask || !seq_offsets || !rewards || !adv || !moments) return AIS_ERR_NULL;
    if (params->seq_level_weights != 0 && !seq_logw) return AIS_ERR_NULL;
    if (!aligned(moments, 8)) return AIS_ERR_ALIGN;
    const Layout L = make_layout(shape, params);
    if (!workspace || !aligned(workspace, 256) || workspace_bytes < L.off_coef) return AIS_ERR_WORKSPACE;
    st = device_setup(nullptr);
    if (st != AIS_OK) return st;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    uint8_t* ws = static_cast<uint8_t*>(workspace);
    const int S = shape->P * shape->G;
    if (launch_advantages({rewards, S, shape->G, params->adv_std_norm, params->eps, adv, n_valid_seq, nullptr}, s) != cudaSuccess)
        return AIS_ERR_DEVICE;
    if (launch_moments(lp_train, lp_roll, mask, seq_offsets, adv, shape->T, S, *params, reinterpret_cast<double*>(ws + L.off_diag),
                       n_valid_seq, params->seq_level_weights != 0 ? seq_logw : nullptr, moments, s) != cudaSuccess)
        return AIS_ERR_DEVICE;
    return AIS_OK;
}

int ais_diag_finalize(const ais_shape* shape, const ais_params* params, const double* moments, const float* lp_train,
                      const float* lp_roll, const uint8_t* mask, float* rho, float* w_tilde, ais_diag* diag,
                      const int32_t* seq_offsets, const float* seq_logw, void* stream) {
    int st = check_shape(shape);
    if (st != AIS_OK) return st;
    st = check_params(params);
    if (st != AIS_OK) return st;
    if (!moments || !lp_train || !lp_roll || !mask || !w_tilde || !diag) return AIS_ERR_NULL;
    const bool seq_level = params->seq_level_weights != 0;
    if (seq_level && (!seq_offsets || !seq_logw)) return AIS_ERR_NULL;
    if (!aligned(moments, 8) || !aligned(diag, 8)) return AIS_ERR_ALIGN;
    st = device_setup(nullptr);
    if (st != AIS_OK) return st;
    if (launch_finalize(moments, lp_train, lp_roll, mask, shape->T, *params, rho, w_tilde, diag, seq_offsets,
                        shape->P * shape->G, seq_level ? seq_logw : nullptr, static_cast<cudaStream_t>(stream)) != cudaSuccess)
        return AIS_ERR_DEVICE;
    return AIS_OK;
}

// What ais_loss_bwd refuses.
static int check_loss(const ais_shape* shape, const ais_params* params, const void* H, const void* W, const void* tokens, const void* mask,
                      const void* seq_offsets, const void* lse_train, const void* lp_train, const void* adv, const void* w_tilde, const void* dH,
                      const void* dW, int64_t lddw, const void* workspace, size_t workspace_bytes) {
    int st = check_shape(shape);
    if (st != AIS_OK) return st;
    st = check_params(params);
    if (st != AIS_OK) return st;
    if (!H || !W || !tokens || !mask || !seq_offsets || !lse_train || !lp_train || !adv || !w_tilde || !dH) return AIS_ERR_NULL;
    if (!aligned(H, 16) || !aligned(W, 16) || !aligned(dH, 16)) return AIS_ERR_ALIGN;
    if (dW && (!aligned(dW, 16) || lddw % 4 != 0)) return AIS_ERR_ALIGN;
    if (dW && lddw < (shape->w_layout == AIS_W_DV ? shape->V : shape->d)) return AIS_ERR_SHAPE;
    const Layout L = make_layout(shape, params);
    if (!workspace || !aligned(workspace, 256) || workspace_bytes < L.fixed_bytes + static_cast<size_t>(kBM) * L.u_row_bytes)
        return AIS_ERR_WORKSPACE;
    return AIS_OK;
}

static int loss_bwd(const ais_shape* shape, const ais_params* params, const void* H, const void* W, const int32_t* tokens,
                    const uint8_t* mask, const int32_t* seq_offsets, const float* lse_train, const float* lp_train,
                    const float* lp_old, const float* lp_ref, const float* adv, const float* w_tilde, void* dH, float* loss,
                    ais_diag* diag, float* dW, int64_t lddw, int dw_accumulate,
                    uint32_t* dev_status, void* workspace, size_t workspace_bytes, void* stream, const Fuse& fuse) {
    int st = check_loss(shape, params, H, W, tokens, mask, seq_offsets, lse_train, lp_train, adv, w_tilde, dH, dW, lddw, workspace, workspace_bytes);
    if (st != AIS_OK) return st;
    int num_sms = 0;
    st = device_setup(&num_sms);
    if (st != AIS_OK) return st;
    const Layout L = make_layout(shape, params);

    cudaStream_t s = static_cast<cudaStream_t>(stream);
    uint8_t* ws = static_cast<uint8_t*>(workspace);
    const int S = shape->P * shape->G;
    float* coef = reinterpret_cast<float*>(ws + L.off_coef);
    const int32_t* nseq = fuse.counts;
    uint32_t* ticket = reinterpret_cast<uint32_t*>(ws + L.off_ticket);
    if (!nseq) {
        int32_t* own = reinterpret_cast<int32_t*>(ws + L.off_nseq);
        if (launch_seq_counts(mask, seq_offsets, S, own, ticket, s) != cudaSuccess) return AIS_ERR_DEVICE;
        nseq = own;
    }
    const int P_norm = shape->P_total > 0 ? shape->P_total : shape->P;
    float* scale = reinterpret_cast<float*>(ws + L.off_scale);
    const KeepJob keep = {reinterpret_cast<__nv_bfloat16*>(ws + L.off_u), L.ldU, fuse.keep_rows, tokens, shape->V, scale, ws + L.off_redo, ticket + 1};
    // row tiles whose gradient factors are all zero (masked rows, zero advantage) are skipped by the recompute and dH passes
    if (launch_loss_coef(lp_train, lp_old, lp_ref, params->beta_kl, mask, seq_offsets, adv, w_tilde, nseq, shape->T, S, P_norm * shape->G,
                         params->clip_eps, reinterpret_cast<double*>(ws + L.off_loss), ticket, coef, ws + L.off_flags, ws + L.off_pace,
                         2 * kPaceRingBytes, loss, diag, lse_train, fuse.rectify, fuse.keep_rows > 0 ? &keep : nullptr, s) != cudaSuccess)
        return AIS_ERR_DEVICE;
    if (shape->T == 0) return AIS_OK;

    // the rows go through in passes of what the scratch holds
    const int64_t blk_rows = scratch_rows(L, shape->T, workspace_bytes);
    __nv_bfloat16* U = reinterpret_cast<__nv_bfloat16*>(ws + L.off_u);
    const uint64_t V = static_cast<uint64_t>(shape->V), d = static_cast<uint64_t>(shape->d);

    // tmW_k: W for the recompute pass (contraction over d), tmW_n: W for the dH pass (contraction over V).  With W [V, d]
    // the first is K-major (boxes of 64 hidden units x 256 vocabulary rows) and the second MN-major (blocks of 64 x 64);
    // with W [d, V] it is the other way round (64 x 64 boxes of vocabulary columns x hidden units; boxes of 64 vocabulary
    // columns x 256 hidden units).
    const bool dv = shape->w_layout == AIS_W_DV;
    CUtensorMap tmW_k, tmW_n, tmW_tail, tmU;
    if (!(dv ? make_tmap_blocks(&tmW_k, W, whole_blocks(V), d, shape->ldw * 2) &&
                   make_tmap(&tmW_tail, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, W, V, d, shape->ldw * 2, 64, 64, CU_TENSOR_MAP_SWIZZLE_128B)
             : make_tmap(&tmW_k, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, W, d, V, shape->ldw * 2, 64, kBN, CU_TENSOR_MAP_SWIZZLE_128B)) ||
        !(dv ? make_tmap(&tmW_n, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, W, V, d, shape->ldw * 2, 64, kBN, CU_TENSOR_MAP_SWIZZLE_128B)
             : make_tmap_blocks(&tmW_n, W, d, V, shape->ldw * 2)) ||
        !make_tmap(&tmU, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, U, V, static_cast<uint64_t>(blk_rows), L.ldU * 2, 64, kBM,
                   CU_TENSOR_MAP_SWIZZLE_128B))
        return AIS_ERR_DEVICE;

    int pass = 0;                                           // tensor-core launches so far
    for (int64_t r0 = 0; r0 < shape->T; r0 += blk_rows) {
        const int64_t rows = (shape->T - r0) < blk_rows ? (shape->T - r0) : blk_rows;
        CUtensorMap tmH;
        const __nv_bfloat16* Hc = static_cast<const __nv_bfloat16*>(H) + r0 * shape->ldh;
        const PassPlan plan = rows == shape->T ? L.train : plan_pass(rows, shape->V, shape->d, kMaxRanges, forced_ranges(shape, params));
        if (!make_tmap(&tmH, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, Hc, d, static_cast<uint64_t>(rows), shape->ldh * 2, 64, plan.unit_rows,
                       CU_TENSOR_MAP_SWIZZLE_128B))
            return AIS_ERR_DEVICE;
        LmheadArgs a;
        memset(&a, 0, sizeof(a));
        a.wait_cycles = wait_cycles();
        a.rows = rows;
        a.row0 = r0;
        a.tokens = tokens;
        a.mask = mask;
        a.lse = lse_train;
        a.lp = lp_train;
        a.row_scale = fuse.keep_rows > 0 ? scale : nullptr;
        a.U = U;
        a.ldU = L.ldU;
        a.coef = coef;
        a.dH = static_cast<__nv_bfloat16*>(dH);
        a.lddh = shape->ldh;
        a.status = dev_status;
        a.tile_active = ws + L.off_flags;
        a.sgroups = 1;
        // recompute softmax - onehot into the scratch; rows that the forward pass left there are only redone where they are
        // outside the range of the exponent form (a launch that usually finds its gate closed)
        if (r0 < fuse.keep_rows) {
            a.tile_active = ws + L.off_redo;
            a.gate = ticket + 1;
        }
        a.ncols = shape->V;
        a.n_col_tiles = (shape->V + kBN - 1) / kBN;
        a.n_row_tiles = static_cast<int32_t>((rows + plan.unit_rows - 1) / plan.unit_rows);
        a.nsplit = plan.ranges;
        a.ksteps = shape->d / 64;
        a.block_tiles = shape->V / kBN;
        int units = a.n_row_tiles * a.nsplit;
        int ctas = units < num_sms ? units : num_sms;
        arm_pace(a, ws, L, (a.n_col_tiles + a.nsplit - 1) / a.nsplit, units, ctas, pass, pass > 0);
        ++pass;
        const CUtensorMap& tail_map = dv ? tmW_tail : tmH;
        const int mode = dv ? kBwdPDv : kBwdP;
        if ((plan.two ? launch_lmhead_pair(mode, tmH, tmW_k, tail_map, a, ctas, s) : launch_lmhead(mode, tmH, tmW_k, tail_map, tmW_k, a, ctas, s)) !=
            cudaSuccess)
            return AIS_ERR_DEVICE;
        // dH = c (.) (U W)
        a.tile_active = ws + L.off_flags;
        a.gate = nullptr;
        a.ncols = shape->d;
        a.n_col_tiles = (shape->d + kBN - 1) / kBN;
        a.n_row_tiles = static_cast<int32_t>((rows + kDhRows - 1) / kDhRows);
        a.nsplit = 1;
        a.ksteps = (shape->V + 63) / 64;
        units = a.n_row_tiles * a.n_col_tiles;
        const int tail = units % kSms;
        a.split_from = units;
        a.ksplit = 1;
        if (tail > 0) {
            int ks = L.ksplit > 0 ? L.ksplit : pick_ksplit(tail, a.ksteps, L.split_slots);
            if (ks > 1 && ks * tail > L.split_slots) ks = L.split_slots / tail;
            if (ks > 1) {
                a.split_from = units - tail;
                a.ksplit = ks;
                a.part_acc = reinterpret_cast<float*>(ws + L.off_split);
                units = a.split_from + tail * ks;
            }
        }
        ctas = units < num_sms ? units : num_sms;
        arm_pace(a, ws, L, 1, units, ctas, pass, true);
        ++pass;
        if (launch_lmhead(dv ? kBwdDhDv : kBwdDh, tmU, tmW_n, tmU, tmW_n, a, ctas, s) != cudaSuccess)
            return AIS_ERR_DEVICE;
        if (a.ksplit > 1 && launch_dh_reduce(a, s) != cudaSuccess) return AIS_ERR_DEVICE;
        if (dW) {
            // dW (+)= U^T H over the rows of this pass: both operands are read with the rows as contraction axis;
            // the maps end at `rows`, so rows the scratch still holds from an earlier pass read as zeros
            CUtensorMap tmU_t, tmH_t;
            // (the scratch rows are padded to 64 columns; what the padding holds only reaches outputs that are not stored)
            if (!make_tmap_blocks(&tmU_t, U, V, static_cast<uint64_t>(rows), L.ldU * 2) ||
                !make_tmap_blocks(&tmH_t, Hc, d, static_cast<uint64_t>(rows), shape->ldh * 2))
                return AIS_ERR_DEVICE;
            // output in W's layout: [V, d] = U^T H, or [d, V] = H^T U with the two operands changing places
            const int out_rows = dv ? shape->d : shape->V, out_cols = dv ? shape->V : shape->d;
            LmheadArgs w = a;
            w.rows = out_rows;
            w.row0 = 0;
            w.tile_active = nullptr;         // it contracts over the rows: nothing to skip
            w.n_row_tiles = static_cast<int32_t>((out_rows + kDhRows - 1) / kDhRows);
            w.ncols = out_cols;
            w.n_col_tiles = (out_cols + kBN - 1) / kBN;
            w.ksteps = static_cast<int32_t>((rows + 63) / 64);
            w.dW = dW;
            w.lddw = lddw;
            w.dw_accumulate = (dw_accumulate || r0 > 0) ? 1 : 0;
            units = w.n_row_tiles * w.n_col_tiles;
            const CUtensorMap& tmRow = dv ? tmH_t : tmU_t;
            const CUtensorMap& tmCol = dv ? tmU_t : tmH_t;
            ctas = units < num_sms ? units : num_sms;
            arm_pace(w, ws, L, 1, units, ctas, pass, true);
            ++pass;
            if (launch_lmhead_pair(kBwdDw, tmRow, tmCol, tmCol, w, ctas, s) != cudaSuccess)
                return AIS_ERR_DEVICE;
        }
    }
    return AIS_OK;
}

int ais_loss_bwd(const ais_shape* shape, const ais_params* params, const void* H, const void* W, const int32_t* tokens,
                 const uint8_t* mask, const int32_t* seq_offsets, const float* lse_train, const float* lp_train,
                 const float* lp_old, const float* lp_ref, const float* adv, const float* w_tilde, void* dH, float* loss,
                 ais_diag* diag, float* dW, int64_t lddw, int dw_accumulate,
                 uint32_t* dev_status, void* workspace, size_t workspace_bytes, void* stream) {
    return loss_bwd(shape, params, H, W, tokens, mask, seq_offsets, lse_train, lp_train, lp_old, lp_ref, adv, w_tilde, dH, loss, diag, dW,
                    lddw, dw_accumulate, dev_status, workspace, workspace_bytes, stream, Fuse());
}

int ais_step(const ais_shape* shape, const ais_params* params, const ais_step_args* a, uint32_t stages, void* stream) {
    int st = check_shape(shape);
    if (st != AIS_OK) return st;
    st = check_params(params);
    if (st != AIS_OK) return st;
    if (!a) return AIS_ERR_NULL;
    const int block = shape->fp8_block;
    const bool dv = shape->w_layout == AIS_W_DV, fp4 = block == AIS_FP4_MX32;
    const bool logprob = (stages & AIS_STAGE_LOGPROB) != 0, diag = (stages & AIS_STAGE_DIAGNOSE) != 0, loss = (stages & AIS_STAGE_LOSS) != 0;
    const Layout L = make_layout(shape, params);
    Fuse fuse;
    // codes with fp32 block scales come from the launch that opens the log-probs ([d, V] heads have a quantiser of their own)
    QuantJob quant[2];
    int nquant = 0;
    auto quantize = [&](const void* x, int64_t rows, int64_t ld, uint8_t* codes, int64_t ldq, void* scales, int64_t lds) -> int {
        if (fp4) return ais_quantize_mxfp4(x, rows, shape->d, ld, codes, ldq / 2, static_cast<uint8_t*>(scales), stream);
        if (block == AIS_FP8_MX32) return ais_quantize_mxfp8(x, rows, shape->d, ld, codes, ldq, static_cast<uint8_t*>(scales), stream);
        if (block == 0) return ais_quantize_fp8_tensor(x, rows, shape->d, ld, codes, ldq, static_cast<float*>(scales), stream);
        float* sc = static_cast<float*>(scales);
        if (!logprob || shape->T == 0) return ais_quantize_fp8(x, rows, shape->d, ld, block, codes, ldq, sc, lds, stream);
        const int bad = check_quantize(x, rows, shape->d, ld, block, codes, ldq, sc, lds);
        if (bad == AIS_OK) quant[nquant++] = {x, rows, ld, codes, ldq, sc, lds};
        return bad;
    };
    if ((stages & AIS_STAGE_QUANTIZE_H) && shape->T > 0) st = quantize(a->H, shape->T, shape->ldh, a->qH, shape->ldh, a->sH, a->ldsH);
    if (st == AIS_OK && (stages & AIS_STAGE_QUANTIZE_W))
        st = dv ? ais_quantize_fp8_cols(a->W, shape->d, shape->V, shape->ldw, block, a->qW, shape->d, static_cast<float*>(a->sW), a->ldsW, stream)
                : quantize(a->W, shape->V, shape->ldw, a->qW, shape->ldw, a->sW, a->ldsW);
    // the quantisations that wait for the log-probs' opening launch, when it does not come
    auto flush_quantize = [&]() -> int {
        const int n = nquant;
        nquant = 0;
        if (n == 0) return AIS_OK;
        const int ready = device_setup(nullptr);
        if (ready != AIS_OK) return ready;
        return launch_quantize(quant, n, shape->d, block, nullptr, static_cast<cudaStream_t>(stream)) == cudaSuccess ? AIS_OK : AIS_ERR_DEVICE;
    };
    if (st != AIS_OK) {                                     // W is refused; H may have been accepted
        const int flushed = flush_quantize();
        return flushed != AIS_OK ? flushed : st;
    }
    fuse.quant = quant;
    fuse.nquant = &nquant;
    const int S = shape->P * shape->G;
    const AdvJob adv = {a->rewards, S, shape->G, params->adv_std_norm, params->eps, a->adv, a->n_valid_seq,
                        reinterpret_cast<uint32_t*>(static_cast<uint8_t*>(a->workspace) + L.off_ticket)};
    RectifyJob rectify;
    // The diagnostics' advantages ride on the merge of the log-probs when there is one -- and when the diagnostics are going to
    // run: the merge is checked for what the log-probs need, and the counters that the advantages clear lie behind that.
    if (logprob && diag && shape->T > 0 &&
        check_diagnostics(shape, params, a->lp_train, a->lp_roll, a->mask, a->seq_offsets, a->rewards, a->adv, a->w_tilde, a->diag, a->workspace,
                          a->workspace_bytes) == AIS_OK)
        fuse.adv = &adv;
    // Up to kMergeMomentRows rows the merge forms the batch moments as well (merge_moments_kernel), and the advantages, which
    // they need, ride on the opening launch instead.
    MomentsJob moments = {a->seq_offsets, a->adv, S, params->C, reinterpret_cast<double*>(static_cast<uint8_t*>(a->workspace) + L.off_diag), a->n_valid_seq};
    if (fuse.adv && shape->T <= kMergeMomentRows && params->seq_level_weights == 0) fuse.moments = &moments;
    // What the loss takes over from earlier stages it takes over only when it is going to run.
    const bool loss_runs = loss && shape->T > 0 &&
                           check_loss(shape, params, a->H, a->W, a->tokens, a->mask, a->seq_offsets, a->lse_train, a->lp_train, a->adv, a->w_tilde,
                                      a->dH, a->dW, a->lddw, a->workspace, a->workspace_bytes) == AIS_OK;
    // log-probs and loss in one call: the exponentials of the rows that the scratch holds stay there (dW wants plain form)
    if (fuse.adv && loss_runs && !a->dW && a->n_valid_seq)
        fuse.keep_rows = scratch_rows(L, shape->T, a->workspace_bytes);
    if (logprob)
        st = logprob_fwd(shape, params, a->H, a->W, a->qH, a->sH, a->ldsH, a->qW, a->sW, a->ldsW, a->tokens, a->mask, a->lp_train,
                         a->lse_train, a->lp_roll, a->lse_roll, a->dev_status, a->workspace, a->workspace_bytes, stream, fuse);
    const int flushed = flush_quantize();                   // the log-probs were refused, or none were asked for
    if (flushed != AIS_OK) return flushed;
    if (st != AIS_OK) return st;
    if (diag) {
        // the loss takes the counts from here and forms rho and w_tilde; the diagnostics' advantages have cleared its ticket
        if (loss_runs && a->n_valid_seq) {
            fuse.counts = a->n_valid_seq;
            rectify = {a->lp_roll, params->C, TotalsJob{}, a->rho, a->w_tilde,
                       params->seq_level_weights ? reinterpret_cast<const float*>(static_cast<uint8_t*>(a->workspace) + L.off_seqw) : nullptr};
            fuse.rectify = &rectify;
            fuse.totals = &rectify.totals;
        }
        st = diagnostics(shape, params, a->lp_train, a->lp_roll, a->mask, a->seq_offsets, a->rewards, a->adv, a->n_valid_seq, a->rho,
                         a->w_tilde, a->diag, a->workspace, a->workspace_bytes, stream, fuse);
    }
    if (st == AIS_OK && loss)
        st = loss_bwd(shape, params, a->H, a->W, a->tokens, a->mask, a->seq_offsets, a->lse_train, a->lp_train, a->lp_old, a->lp_ref,
                      a->adv, a->w_tilde, a->dH, a->loss, a->diag, a->dW, a->lddw, static_cast<int>(a->dw_accumulate), a->dev_status,
                      a->workspace, a->workspace_bytes, stream, fuse);
    return st;
}

}  // extern "C"
