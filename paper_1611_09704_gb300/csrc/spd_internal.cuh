// spd_internal.cuh -- device-side structures and launchers shared by the
// translation units of libspd.  Not part of the public ABI (include/spd.h).
#pragma once

#include <cuda_runtime.h>
#include <cuda_fp16.h>
#include <cuda_bf16.h>
#include <stdint.h>

#include "spd.h"

namespace spd {

// ---------------------------------------------------------------- elements

// Value of a stored element as FP32: the raw value, or fmaf(scale, q, offset)
// when a per-row scale is given (FP16 / BF16 storage, Sec. "precision form").
template <int DT> struct Elem;
template <> struct Elem<SPD_F32> {
    using T = float;
    static __device__ __forceinline__ float cvt(T v) { return v; }
};
template <> struct Elem<SPD_F16> {
    using T = __half;
    static __device__ __forceinline__ float cvt(T v) { return __half2float(v); }
};
template <> struct Elem<SPD_BF16> {
    using T = __nv_bfloat16;
    static __device__ __forceinline__ float cvt(T v) { return __bfloat162float(v); }
};

inline size_t elem_bytes(int dt) { return dt == SPD_F32 ? 4 : 2; }

// ------------------------------------------------------------------- MSD

constexpr int kMsdThreads = 256;
constexpr int kMsdUnit = 65536;   // samples of one row per block-partial unit

// (n, T, S) of a piece of the data, Sec. 2.1, written per unit in FP64, plus
// the piece's smallest and largest value: sigma is exactly 0 iff they agree,
// a test that does not depend on how S was rounded.
struct MsdPart {
    double n, T, S, lo, hi;
};

struct MsdArgs {
    const void *data;
    int64_t n_dm, n_samp, stride;
    const float *scale, *offset;
    int64_t units_per_row;
    int vec_ok;          // 16-byte aligned rows: vector loads allowed
    MsdPart *parts;      // [n_dm * units_per_row]
    unsigned *arrived;   // set to 0 (null: nothing), for the merge that follows
    spd_result *result;  // set to 0 (null: nothing)
};

// The arrival counter of a merge: scratch's last place.
inline unsigned *merge_counter(MsdPart *scratch, int n_scratch) {
    return reinterpret_cast<unsigned *>(scratch + n_scratch - 1);
}

// Arguments of the sigma_Nmax pass (Eq. 5): tiles of 8192 starts per row.
struct NmaxArgs {
    const void *data;
    int64_t n_dm, n_samp, stride;
    const float *scale, *offset;
    const spd_msd_stats *msd;   // mean used for centring, per scope entry
    int per_row;
    int vec_ok;                 // rows aligned for 4-element vector loads
    int nmax;
    int nb;                     // staged blocks of 16 samples per tile
    int64_t tiles_per_row;      // partials per row (each covers up to 4 tiles of 8192 starts)
    MsdPart *parts;             // [n_dm * tiles_per_row]
};

// ------------------------------------------------------------------ detect

constexpr int kX = 16;              // consecutive samples owned by one thread

// One group of evaluated widths (host-compiled from the width list).  The
// running boxcar sum B of every start sample i starts as
// B_off(i) = y[i] + ... + y[i+off-1] (read from the tile's compensated prefix
// sums) and then grows one step per member, as in Algorithm 1: from the
// centred samples y (step 1, positions off, off+1, ...) or from the G-sample
// window sums S_G (step G, positions off, off+G, ...).  Member c is the width
// off + (c+1) * step with eval index widx0 + c.  Groups are evaluated in any
// order; in the candidate search a group whose upper bound cannot reach the
// threshold or the current best is skipped.
struct Group {
    int16_t off;
    int16_t count;
    int16_t widx0;
    uint16_t flags;   // bit 0: step G (window sums), else step 1
};
constexpr uint16_t kGroupCoarse = 1;
constexpr uint16_t kGroupRefine = 2;   // widths 1..16 from off 0: per-sample energy test first

constexpr int kMaxCodeGroups = 64;          // groups a packed max can tell apart
constexpr int kMaxEval = SPD_MAX_WIDTHS + 1;
constexpr int kMaxRanges = 8;               // DM ranges searched by one launch

// The width groups of one range.  Member c of group g is the width
// g.off + (c + 1) * step (step G for coarse groups, else 1) with eval index
// g.widx0 + c; eval index 0 is width 1.
struct RangeProg {
    int32_t n_groups;
    int32_t n_eval;     // evaluated widths: width 1 first, then the listed ones
    int32_t wmax;
    int32_t G;          // step of the coarse window sums, 0 if unused
    Group groups[kMaxCodeGroups];
};

// One DM range (a plane with its own widths, MSD and threshold) of a launch.
struct RangeDesc {
    const void *data;
    int64_t n_dm, n_samp, stride;
    const float *scale, *offset;
    const float *inv_tab;       // [entries][n_eval]: 1 / sigma_w, FP32
    const float2 *mu_tab;       // [entries]: mean split into hi + lo FP32
    const int32_t *flags;       // [entries]: nonzero = degenerate sigma
    const float *scr_tab;       // screening: see ConstArgs (null: not screened)
    const float2 *grp_tab;
    int64_t tile0;              // first launch-wide tile index of this range
    int64_t tiles_per_row;
    int32_t vec_ok;             // 16-byte aligned rows: bulk (TMA) copies allowed
    int32_t per_row;            // MSD scope entry = row (else entry 0)
    int32_t R;                  // blocks of 16 positions staged per tile
    int32_t span;               // positions of one tile's window (tile + wmax - 1)
    int32_t dm_offset;          // added to the row index in candidate records
    float threshold;
    int64_t n_emit;             // only starts < n_emit become candidates (n_samp normally)
    int64_t sample_base;        // added to the start sample in candidate records
    int32_t sample_shift;       // records carry start << shift and width << shift
    int32_t reserved0;
    RangeProg prog;
};

// Everything one detect launch needs, passed by value as a __grid_constant__
// kernel parameter (no host-to-device copy of its own, so it can be captured
// in a CUDA graph).
struct Launch {
    int32_t n_ranges;
    int32_t R;                  // shared arrays sized for the widest range
    int32_t raw_bytes;          // bytes of one raw staging buffer (multiple of 16)
    int32_t max_eval;
    int64_t n_tiles;
    spd_candidate *out;
    int64_t capacity;
    spd_result *result;
    float *snr_out;             // plane output (single range) or null
    uint16_t *width_out;
    int64_t out_stride;
    uint64_t wait_ns;           // bound of a wait for a bulk copy
    uint32_t extra_tx;          // test aid: bytes expected beyond each copy (0 in use)
    int32_t kmax;               // search kernel: levels of the block max table
    int32_t units;              // search kernel: units of 16 starts per tile (<= threads)
    int32_t chunk;              // search kernel: tiles per scheduling chunk (set at launch)
    const uint32_t *tile_list;  // search kernel: the tiles to search (null: all n_tiles)
    const uint32_t *tile_count; // and how many they are
    const uint32_t *unit_list;  // then single units (null: none), tile << 8 | unit
    const uint32_t *unit_count;
    int32_t live_blocks, live_halves;   // blocks and half-warps they are searched with
    RangeDesc rng[kMaxRanges];
};

// ------------------------------------------------------------ search kernel

constexpr int kSPad = 20;          // shared words per 16 positions (4 padding words)
constexpr int kSLevels = 5;        // block max table: windows of up to 2^5 blocks

// Bound geometry of one width group (Group) of step d, for the unit of 16
// starts 16t .. 16t+15: its windows end in blocks t + a .. t + b and lie in
// blocks t .. t + e - 1.  The largest block prefix over [t + a, t + b] is
// read as the max of two table windows of 2^lvl blocks at t + a and t + bk
// (lvl = -1: a plain loop over the blocks, for spans longer than the table).
struct GroupGeom {
    int a, bk, lvl, e;
};
__host__ __device__ inline GroupGeom group_geom(int off, int count, int d) {
    GroupGeom q;
    q.a = (off + d) >> 4;
    const int b = (15 + off + count * d) >> 4;
    const int len = b - q.a + 1;
    q.lvl = -1;
    q.bk = b;
    if (len <= (2 << kSLevels)) {
        int k = 0;
        while ((2 << k) <= len) ++k;   // floor(log2(len))
        if (k > kSLevels) k = kSLevels;
        q.lvl = k;
        q.bk = b - (1 << k) + 1;
    }
    q.e = 1 + ((14 + off + count * d) >> 4);
    return q;
}

// Shared memory of one search CTA, in the order the kernel lays it out:
// mbarrier (16 B), one raw staging buffer, then FP32 arrays -- centred samples
// y, in-block prefix sums P and (G > 1) G-sample window sums, each 20 words
// per 16 positions; per block: sums, prefix maxima (level 0 of the table) and
// kmax table levels, prefix minima, energy prefix (RM + 4), four scan
// temporaries; 1/sigma_w per eval index -- then per group two int4 of
// evaluation and bound data, and the width per eval index (uint16).
// RM is a multiple of 4.
struct SearchSmem {
    size_t raw, y, p, g, bs, mx, mn, pq, ex, eq, rh, rl, inv, gr, ew, total;
};
// Plane output (kmax < 0) has no bounds: no array from mx to rl.
__host__ __device__ inline SearchSmem search_smem(int RM, int raw_bytes, int max_eval, int kmax,
                                                  int G) {
    SearchSmem m;
    const size_t blk = (size_t)kSPad * RM * sizeof(float);
    const size_t arr = (size_t)RM * sizeof(float);
    const size_t bnd = kmax < 0 ? 0 : arr;
    m.raw = 16;
    m.y = m.raw + (size_t)raw_bytes;
    m.p = m.y + blk;
    m.g = m.p + blk;
    m.bs = m.g + (G > 1 ? blk : 0);
    m.mx = m.bs + arr;                       // level 0; levels 1..kmax follow
    m.mn = m.mx + (size_t)(1 + kmax) * arr;   // kmax -1: nothing
    m.pq = m.mn + bnd;
    m.ex = m.pq + bnd + 16;
    m.eq = m.ex + bnd;
    m.rh = m.eq + bnd;
    m.rl = m.rh + bnd;
    m.inv = m.rl + bnd;
    m.gr = m.inv + (((size_t)max_eval * sizeof(float) + 15) & ~(size_t)15);
    m.ew = m.gr + (size_t)kMaxCodeGroups * 32;
    m.total = (m.ew + (size_t)max_eval * sizeof(uint16_t) + 15) & ~(size_t)15;
    return m;
}
inline size_t search_smem_bytes(int RM, int raw_bytes, int max_eval, int kmax, int G) {
    return search_smem(RM, raw_bytes, max_eval, kmax, G).total;
}

// ---------------------------------------------------------------- screening

// The candidate search in three launches: a screen of the whole plane that
// reads every sample once and keeps, per unit of 16 starts, only whether any
// candidate can start there; the search kernel over the tiles with many such
// live units; and one half-warp per live unit for the rest.
//
// The screen's bounds are per class of evaluated widths: widths 1..8, 9..16,
// and (2^(c+2), 2^(c+3)] for c = 2 .. 9 (17..32 up to 2049..4096).
constexpr int kScrClasses = 10;
constexpr int kScrTab = 12;         // floats per scope entry: see ConstArgs::scr_tab
constexpr int kScrSlots = 16;       // sets of counters: launches of one call
// Live units of a tile beyond which the tile is searched whole.  A unit stages
// every block that its widths reach, and the half-warps at work on units are as
// many as have room for that in shared memory; a tile is staged once for all its
// units.  So many units took as long as a tile of noise at the search's usual
// thresholds (512 x 262144 samples, ns per unit and per tile of the launch):
// widths to 32 0.84 of 24 (28), to 256 by 8 above 16 1.46 of 27 (19), to 512 by
// 8 3.5 of 40 (11), to 700 6.4 of 43 (7), to 1000 by 16 6.2 of 47 (7), to 2048
// by 64 13.5 of 38 (3), to 4096 by 16 85 of 98 (1).  With 16 for all of them a
// search of widths to 4096 at 5.5 sigma took 21.1 ms, 3.2 with every tile whole.
// The list of units has room for kScrDense of every tile: which way a tile is
// searched depends on its samples alone, not on the order of arrival.
constexpr int kScrDense = 16;
inline int screen_dense(int wmax) {
    const int d = 330 / (((15 + wmax) >> 4) + 1);
    return d < 1 ? 1 : d > kScrDense ? kScrDense : d;
}

__host__ __device__ inline int screen_class(int w) {
    int c = w > 8 ? 1 : 0;
    for (int h = 16; w > h; h *= 2) ++c;
    return c;
}

// Counters of one screened launch, zeroed by the constants kernel.
struct ScreenCtl {
    uint32_t dense;       // tiles in the list of tiles
    uint32_t live;        // units in the list of units
    uint32_t reserved[2];
};

// Where a screened launch keeps its lists (null ctl: not screened).
struct ScreenLists {
    ScreenCtl *ctl;
    uint32_t *tiles;      // launch-wide tile indexes, room for every tile
    uint32_t *units;      // tile << 8 | unit of the tile (under 2^24 tiles)
    int64_t tile_cap;

    // The same lists for launch k of a call: counters of its own.
    ScreenLists slot(int k) const {
        ScreenLists s = *this;
        if (s.ctl) s.ctl += k;
        return s;
    }
};

// Shared words of one half-warp's live unit: y, P and (G > 1) S_G in kSPad
// words per block, then per block its sum, largest prefix and energy prefix.
__host__ __device__ inline int live_words(int blocks, int G) {
    return (blocks * kSPad * (G > 1 ? 3 : 2) + 3 * blocks + 1 + 3) & ~3;   // 16-byte pieces
}

struct ConstArgs {
    const spd_msd_stats *msd;   // [entries]
    int entries;
    int sigma_mode;
    float *inv_tab;
    float2 *mu_tab;
    int32_t *flags;
    // screening (null: not screened).  Per entry: the largest 1/sigma_w of
    // each class, then the largest w / sigma_w^2 of class 0 and of classes 0
    // and 1; per entry and group, the bounds' factors of the search kernel
    float *scr_tab;             // [entries][kScrTab]
    float2 *grp_tab;            // [entries][n_groups]
    ScreenCtl *ctl;             // [kScrSlots], zeroed here
    spd_result *result;   // may be null: status set on a degenerate entry (count untouched)
    int skip_w1;          // eval index 0 (the width-1 start) takes no part: 1/sigma = NaN
};

// Launchers (return cudaGetLastError() of the launch).
cudaError_t launch_msd_partial(const MsdArgs &a, int dtype, cudaStream_t s);
cudaError_t launch_msd_merge(const MsdPart *parts, int64_t n_dm, int64_t units_per_row,
                             int64_t n_samp, int per_row, MsdPart *scratch, int n_scratch,
                             spd_msd_stats *out, const ConstArgs *consts, const RangeProg *prog,
                             cudaStream_t s);
// Global scope: with consts and prog the merge's launch forms the constants
// too.  The partials' launch has set merge_counter(scratch, n_scratch) to 0.
cudaError_t launch_consts(const ConstArgs &a, const RangeProg &prog, cudaStream_t s);
cudaError_t launch_stream_msd(const MsdPart *parts, int64_t n_dm, int64_t upr, int per_row,
                              MsdPart *state, MsdPart *scratch, int n_scratch, spd_msd_stats *out,
                              const ConstArgs *consts, const RangeProg *prog, cudaStream_t s);
// width bytes (a multiple of esz, 2 or 4) of each of n_rows rows.  Addresses
// and row strides are multiples of esz; all device memory.
cudaError_t launch_copy_rows(void *dst, int64_t dst_stride, const void *src, int64_t src_stride,
                             int64_t width, int64_t n_rows, int esz, cudaStream_t s);
cudaError_t launch_zero_parts(MsdPart *p, int64_t n, cudaStream_t s);
int nmax_blocks(int nmax);
// sigma_Nmax partials per row (CTAs of the partial kernel per row).
int64_t nmax_tiles_per_row(int64_t n_samp);
cudaError_t launch_nmax_partial(const NmaxArgs &a, int dtype, cudaStream_t s);
// Fold n_parts partials into *out (the block tree of the final merge).
cudaError_t launch_fold_parts(const MsdPart *parts, int64_t n_parts, MsdPart *scratch,
                              int n_scratch, MsdPart *out, cudaStream_t s);
// Shard partials in shard order -> mean/sd (what 0) or sd_nmax (what 1).
cudaError_t launch_merge_shards(const MsdPart *parts, int n, int what, int nmax,
                                spd_msd_stats *out, cudaStream_t s);
cudaError_t launch_nmax(const NmaxArgs &a, int dtype, MsdPart *scratch, int n_scratch,
                        spd_msd_stats *out, const ConstArgs *consts, const RangeProg *prog,
                        cudaStream_t s);
// The candidate search (search kernel): same launch description with the
// ranges' tiles of 16 * threads starts (threads = 128 or 256), kmax set.
cudaError_t launch_search(const Launch &L, int dtype, int G, bool multi_block, size_t smem,
                          int ctas_per_sm, int threads, cudaStream_t s);
constexpr int kSearchThreads = 256;   // threads of a search CTA by default
constexpr int kPlaneThreads = 256;    // threads of a plane-output CTA
// The screen of a launch's ranges (geometry as for launch_search).
cudaError_t launch_screen(const Launch &L, const ScreenLists &S, int dtype, cudaStream_t s);
// Levels 1 .. `levels` (at most 4) of decimation by 2 of a plane (dequantised)
// into FP32 planes of 16-byte aligned rows: dst[k] (null: not wanted) holds
// n_samp >> (k + 1) sums of 2^(k+1) samples per row.
cudaError_t launch_decimate(const spd_plane &p, float *const *dst, const int64_t *stride,
                            int levels, cudaStream_t s);
cudaError_t launch_threshold_plane(float *snr, uint16_t *width, int64_t n_dm, int64_t n_samp,
                                   int64_t stride, float thr, cudaStream_t s);
cudaError_t launch_threshold(const float *snr, const uint16_t *width, int64_t n_dm,
                             int64_t n_samp, int64_t stride, float thr, spd_candidate *out,
                             int64_t capacity, spd_result *result, cudaStream_t s);
// Per-DM clustering of the candidates of an SNR plane (one warp per row).
cudaError_t launch_cluster(const float *snr, const uint16_t *width, int64_t n_dm,
                           int64_t n_samp, int64_t stride, float thr, int64_t gap,
                           spd_cluster *out, int64_t capacity, spd_result *result,
                           cudaStream_t s);
cudaError_t launch_boxcar_sums(const spd_plane &p, int w, float *out, int64_t out_stride,
                               cudaStream_t s);

}  // namespace spd
