// Internal definitions shared by the host encoder and the CUDA translation unit.
#pragma once
#include <algorithm>
#include <cmath>
#include <cstddef>
#include <cstdint>
#include <cstdlib>
#include <cstring>
#include <memory>
#include <new>
#include <vector>

#include <sys/mman.h>

#include "celty.h"

namespace celty {

constexpr int kGroup = 8;            // entries per 16-byte value vector / 32-bit run word
constexpr int kChunkGroups = 32;     // COLUMN layout: groups per warp-wide chunk (256 entries)
constexpr int kTileSlack = 8;        // LANE_TILE: spare accumulator rows per slab for group-tail slots
// LANE_TILE sub-block header (bytes), ahead of the value vectors and run words:
//   [0,32)   groups of 8 entries that lane L's tile holds (u8)
//   [32,36)  vectors in the sub-block | steps << 16 (u32), steps = the largest group count;  rest zero
constexpr int kSubHeader = 48;
constexpr int kMaxTileRows = 240;    // keeps local rows (and the spare rows after them) in a byte
constexpr int64_t kMaxM = 49152;     // accumulators of one thread block must fit shared memory
constexpr size_t kAlign = 256;
constexpr int kMaxBlocks = 192;      // blocks of the fused kernel the workspace has partial vectors for
// LANE_TILE: a thread block covers at most this many slabs of rows.  The kernels take any value; with one
// slab per block (row parts = slabs, all of a block's warp teams work on different columns of the same rows)
// every configured shape ran as fast or faster on B200 than with 2 or 4, mostly because a block then adds
// fewer rows into y at the end.
constexpr int kSlabsPerBlock = 1;

inline size_t round_up(size_t v, size_t a) { return (v + a - 1) / a * a; }

#ifdef __CUDACC__
#define CELTY_HD __host__ __device__
#else
#define CELTY_HD
#endif

// LANE_TILE row map.  Rows are dealt to the 32 lanes one at a time (row r belongs to lane r mod 32), and
// the groups of 32 consecutive rows are dealt to the S slabs in chunks of C groups, round robin.  Tile
// t = 32*s + L is the ordered set of rows that lane L of slab s receives; local row i of that tile is
//     row = (((i / C) * S + s) * C + i mod C) * 32 + L.
// A lane's local rows grow with the row number, every slab samples the whole height of the matrix (so a
// mask whose density drifts with the row index still gives every lane and every slab the same share),
// and local rows [kC, kC + C) of a slab are the 32*C consecutive rows that start at ((k*S + s)*C)*32:
// the accumulator word (i*32 + L) order of a slab is the order of y, C*32 rows at a time.
CELTY_HD inline int64_t tile_row(int64_t S, int64_t C, int64_t s, int64_t lane, int64_t i)
{
    return (((i / C) * S + s) * C + i % C) * 32 + lane;
}

// Host memory that is not cleared when it is allocated: the encoder's threads write (and so first touch) all of it.  From 2 MB on
// in 2 MB pages where the system grants them on request: 16 threads that first touch 12 MB in 4 KB pages take 0.6 ms, most of it in
// one another's way.
template <typename T>
class Raw {
public:
    Raw() = default;
    Raw(const Raw &o) { allocate(o.n_); if (n_) std::memcpy(p_.get(), o.p_.get(), n_ * sizeof(T)); }
    Raw &operator=(const Raw &) = delete;
    void allocate(size_t n)
    {
        constexpr size_t huge = (size_t)2 << 20;
        const size_t bytes = n * sizeof(T), align = bytes >= huge ? huge : 64;
        p_.reset(static_cast<T *>(std::aligned_alloc(align, round_up(bytes + (bytes == 0), align))));
        if (!p_) throw std::bad_alloc();
        n_ = n;
#ifdef MADV_HUGEPAGE
        if (align == huge) (void)madvise(p_.get(), round_up(bytes, huge), MADV_HUGEPAGE);
#endif
    }
    T *data() { return p_.get(); }
    const T *data() const { return p_.get(); }
    T &operator[](size_t i) { return p_.get()[i]; }
    const T &operator[](size_t i) const { return p_.get()[i]; }
    size_t size() const { return n_; }

private:
    struct Free { void operator()(void *p) const { std::free(p); } };
    std::unique_ptr<T, Free> p_;
    size_t n_ = 0;
};

// Workspace layout (device): all offsets multiples of 256.
struct WorkspaceLayout {
    size_t status_off;   // uint32 status, int32 count, uint32 tickets[2] (and spare words)
    size_t idx_off;      // int32[K]
    size_t val_off;      // uint16[K]
    size_t scratch_off;  // uint32[T + 2] for celty_decode_device
    size_t partial_off;  // float[kMaxBlocks][part_words]: per-block partial sums of the fused kernel (ordered merge), or
                         // uint16[K]: the activations a down projection makes from gate and up (bulk merge)
    size_t total;
};

inline WorkspaceLayout workspace_layout(int64_t K, int64_t T, int64_t part_words)
{
    WorkspaceLayout w{};
    w.status_off = 0;
    w.idx_off = kAlign;
    w.val_off = w.idx_off + round_up((size_t)K * 4, kAlign);
    w.scratch_off = w.val_off + round_up((size_t)K * 2, kAlign);
    w.partial_off = w.scratch_off + round_up((size_t)(T + 2) * 4, kAlign);
    const size_t partials = (size_t)kMaxBlocks * part_words * 4, h = part_words ? (size_t)K * 2 : 0;
    w.total = w.partial_off + round_up(partials > h ? partials : h, kAlign);
    return w;
}

// Shared-memory carve-up of the fused kernel, computed by ONE function for the kernel and for the host
// (which sizes the launch with .total), so that the two can never disagree.
struct FusedSmem {
    size_t acc, ring, bars, flag, items, imeta, zero, keep, wrel, blk, blkw, win, total;   // (32 bits each: 0.5 % slower)
};

// window: bytes of a place of its own for the window of the offset table (launches for several vectors)
CELTY_HD inline FusedSmem fused_smem_layout(int R, int K, int teams, int D, int slot_bytes, int cap, int window = 0)
{
    FusedSmem l;
    uint32_t off = 0;
    l.acc = off;       off += (uint32_t)teams * (R + kTileSlack) * 32 * 4;   // FP32 accumulators, one slab per team
    l.ring = off;      off += (uint32_t)teams * D * slot_bytes;              // bulk-copy ring slots (multiples of 128 bytes)
    l.bars = off;      off += (uint32_t)teams * D * 8 + 8;                   // one "full" mbarrier per slot, one for the offset window
    l.flag = off;      off += (uint32_t)teams * 4 + 8;                       // per team: a wait of one of its warps ran out; the window's; survivors in the last, short word
    off = (off + 15) / 16 * 16;
    l.items = off;     off += (uint32_t)teams * cap * 8;                     // {column, x bits} per looked-up item
    l.imeta = off;     off += (uint32_t)teams * cap * 8;                     // {offset/16, bytes} of its sub-block
    l.zero = off;      off += 16;                                          // the all-zero group that idle lanes fetch
    l.keep = off;      off += ((uint32_t)((K + 31) / 32) * 4 + 15) / 16 * 16;   // one keep bit per activation
    l.wrel = off;      off += ((uint32_t)((K + 31) / 32) * 4 + 15) / 16 * 16;   // survivors before each keep word, in its block of 32
    const uint32_t blocks = ((uint32_t)((K + 1023) / 1024) * 4 + 31) / 32 * 32;   // (eight are read at a time)
    l.blk = off;       off += blocks;                                      // survivors in each block of 32 keep words
    l.blkw = off;      off += 16 * blocks;                                 // per warp: survivors before each block
    l.win = off;
    off += (uint32_t)window;
    l.total = off;
    return l;
}

// The same for k_spmspv_direct.
struct DirectSmem {
    uint32_t ring, bars, flag, items, zero, taken, keep, total;              // (the accumulators lie at 0)
};

inline DirectSmem direct_smem_layout(int R, int K, int G, int D, int slot_bytes, int cap)
{
    DirectSmem l;
    uint32_t off = 0;
    off += (uint32_t)G * (R + kTileSlack) * 32 * 4;                          // FP32 accumulators, one slab per team
    l.ring = off;      off += (uint32_t)G * D * slot_bytes;                  // bulk-copy ring slots (multiples of 128 bytes)
    l.bars = off;      off += (uint32_t)G * D * 8;                           // one "full" mbarrier per slot
    l.flag = off;      off += (uint32_t)G * 4;                               // per team: a warp gave up
    off = (off + 15) / 16 * 16;
    l.zero = off;      off += 16;                                            // the all-zero group that idle lanes fetch
    l.items = off;     off += (uint32_t)G * cap * 8;                         // {offset/16, bytes/16 and x} per column of a team
    l.taken = off;     off += 16;                                            // survivors that the block has taken
    l.keep = off;      off += (uint32_t)((K + 31) / 32) * 4;                 // one keep bit per activation
    l.total = (off + 15) / 16 * 16;
    return l;
}

// k_spmspv_direct: column of x that is the i-th of block b's, where nK blocks share the columns (K or more: block b has no
// i-th column).  Runs of kDirectRun columns go round the blocks, and each round starts kDirectTurn blocks further on.
constexpr int kDirectRun = 2, kDirectTurn = 3;

CELTY_HD inline int direct_column(int i, int b, int nK, float nK_inv)   // nK_inv: 1 / nK to a few units in the last place
{
    const int round = i / kDirectRun, turned = b + round * kDirectTurn;
    const int place = turned - (int)(((float)turned + 0.5f) * nK_inv) * nK;      // modulo nK, exact for turned < 2^14
    return (round * nK + place) * kDirectRun + i % kDirectRun;
}

// Most columns of a block.
inline int direct_columns(int64_t K, int blocks_per_part)
{
    const int64_t round = (int64_t)kDirectRun * blocks_per_part;
    return (int)((K + round - 1) / round) * kDirectRun;
}

// The blocks of a row part form groups, which share the survivors of their columns.  Blocks [0, larger) are in groups of least + 1
// neighbouring ones, those behind them in groups of least.
struct DirectSizes { int32_t least, larger; };

struct DirectGroup { int first, size; float size_inv; };          // blocks [first, first + size)

CELTY_HD inline DirectGroup direct_group(int b, const DirectSizes &z)
{
    DirectGroup g;
    const bool more = b < z.larger;
    g.size = more ? z.least + 1 : z.least;
    g.size_inv = 1.f / (float)g.size;
    const int in = more ? b : b - z.larger;
    g.first = b - in + (int)(((float)in + 0.5f) * g.size_inv) * g.size;
    return g;
}

// Column that a group's ranking lane t (32 * warp + lane) holds (K or more: none): the members' first runs, then their next ones.
CELTY_HD inline int direct_held(int t, const DirectGroup &g, int nK, float nK_inv)
{
    const int run = t / kDirectRun, round = (int)(((float)run + 0.5f) * g.size_inv);
    return direct_column(round * kDirectRun + t % kDirectRun, g.first + run - round * g.size, nK, nK_inv);
}

// Block of the group (counted from its first) that takes the i-th survivor of ranking warp w: the warps start at evenly spaced ones.
CELTY_HD inline int direct_taker(int i, int w, float rankers_inv, const DirectGroup &g)
{
    const int r = i + (int)(((float)(w * g.size) + 0.5f) * rankers_inv);
    return r - (int)(((float)r + 0.5f) * g.size_inv) * g.size;
}

// Groups for a launch of `grid` blocks and P row parts with `warps` warps that can rank: as few as hold all columns, a column per
// lane.  They even out what a group's blocks have, and every ranking warp is another 32 columns.  Device time with up to
// 12 or 16 (pairs) ranking warps / 8 / 5 / 2, in us: 4096 x 4096 5.89 / 5.91 / 6.16 / 6.48;  4096 x 11008 10.8 / 10.9 / 10.9 / 11.3;  8192 x 8192
// 13.5 / 13.6 / 14.2 / 14.2.  Two or four columns per lane are two or four more such look-ups one after the other (small
// layers: 0.2 us each step) and are taken where a group would have less than three members otherwise (wide: more than 128
// columns per block): for two / three / four members 11008 x 4096, N = 4 28.5 / 25.7 / 25.8;  8192 x 28672 at 30 % 24.4 / 23.6 / 23.6;
// 16384 x 12288 at 10 % 10.0 / 10.0 / 10.3;  4096 x 4096, N = 4 13.6 / 13.5 / 14.2;  13824 x 5120 at 50 % 14.0 / 14.0 / 13.7.
struct DirectGroups {
    int rankers;               // warps that rank
    int held;                  // columns per lane of them
    int most;                  // columns that a block may take
    DirectSizes sizes[2];      // in row parts with floor(grid / P) blocks, and in those with one more
};

// Warps that rank, of `most` that can, where blocks have up to `columns`.  Those that neither rank nor stream make the reported list, and a
// block of few columns has done the rest before three of them have.  Device time with 12 / 10 / 8 / 6 / 4, us:
//    512 x 512 (4 columns), 50 % of the activations    -   /  -   / 3.41 / 3.35 / 3.37;  with two 3.32
//   1024 x 1024 (14), 50 %                            3.25 /  -   / 3.24 / 3.24 / 3.24;  with two 3.28
//    600 x 3000 (22), 30 %                            3.66 /  -   / 3.55 / 3.55 / 3.55
//   2048 x 2048 (28), 50 %                            3.57 / 3.54 / 3.52 / 3.54 / 3.56
//   2048 x 3000 (42), 30 %                            3.65 / 3.51 / 3.49 / 3.52 / 3.53
//   1000 x 7000 (48), 10 %, 50 %                      3.79, 4.19 / 3.62, 4.21 / 3.61, 4.22 / 3.62, 4.22 / 3.62, 4.38
//   4096 x 4096 (56), 10 %, 50 %                      3.83, 5.67 / 3.82, 5.66 / 3.83, 5.71 / 3.83, 5.93 / 3.84, 6.01
//   3001 x 5003 (68), 10 %, 50 %                      4.19, 5.76 / 4.21, 5.87 / 4.20, 5.87 / 4.18, 5.97 / 4.26, 6.29
// (In two runs 4096 x 4096 with a magnitude mask took 5.71 and 5.81 with ten and 5.71 with twelve, so that the line lies at 48.  Pairs stream
// with 16 warps whatever ranks: fewer rankers are no more list makers.)
inline int direct_rankers(int columns, int pairs, int most)
{
    return pairs ? most : std::min({most, columns <= 48 ? 10 : most, 1 + columns / 4});
}

inline DirectGroups direct_groups(int64_t K, int grid, int P, int warps, bool wide)
{
    DirectGroups g;
    const int nK = grid / P, columns = direct_columns(K, nK), most = nK + (grid % P ? 1 : 0);
    g.held = 1;
    while (wide && g.held < 4 && 3 * columns > 32 * g.held * warps) g.held *= 2;
    const int members = std::max(1, std::min(most, 32 * g.held * warps / columns)), groups = (most + members - 1) / members;
    const int size = (most + groups - 1) / groups;
    for (int l = 0; l < 2; ++l) {
        const int least = (nK + l) / groups;
        g.sizes[l] = DirectSizes{least, (nK + l - least * groups) * (least + 1)};
    }
    g.rankers = (size * columns + 32 * g.held - 1) / (32 * g.held);
    g.most = std::min(size * columns, g.rankers * (32 * g.held / std::max(1, nK / groups) + 1));
    return g;
}

struct FusedParams {
    const uint32_t *meta;      // [K*S + 1] offset/16 of sub-block (j, s) in the stream
    const uint8_t *stream;
    const uint16_t *x;         // K FP16
    float tau;
    float *y;                  // M
    int32_t *idx;              // global compacted list (API output)
    uint16_t *val;
    int32_t *count;
    uint32_t *status;
    uint32_t *tickets;         // [0] y cleared / partial stored, [1] departed (ordered merge); null (bulk reduce-add merge):
                               // a kernel before this one has cleared y
    float *partials;           // gridDim.x vectors of Sc * R * 32 floats (accumulator layout)
    int M, K, R, S, C;         // rows, columns, local rows per tile, slabs, chunk of the row map (tile_row)
    int G, Sc, P, D;           // teams per slab, slabs per block, row parts, ring depth
    int cl;                    // thread blocks per cluster (1, 2 or 4); blocks of a cluster share a row part
    int pp;                    // 1: two warps per team that take turns at the team's accumulator (see the kernel)
    // mix >= 2 (bulk reduce-add merge without clusters): the gridDim mod P blocks that are left when every row part
    // has floor(gridDim / P) blocks are not given to the first parts (which would then finish early, one slice
    // ahead of the others); each of them serves mix = P / (gridDim mod P) consecutive parts instead, with G / mix
    // teams per slab, so that every part is shared by the same number of teams.  units_inv then holds
    // floor(2^32 / (floor(gridDim / P) * G + G / mix)).
    int mix;
    int slot_bytes;            // ring slot size, multiple of 128
    int cap;                   // columns a team looks up per batch
    int win_cols;              // columns of the offset table a block copies into shared memory at its start
    FusedSmem lay;             // the block's shared memory, worked out once on the host (fused_smem_layout)
    int clear_rows, clear_extra;   // M / gridDim.x and M mod gridDim.x: block b clears clear_rows (+ 1 if b < clear_extra) rows of y
    // teams that share the survivor list of a row part: units = (column slices of the part) * G;
    // units_inv = floor(2^32 / units) for parts with gridDim / cl / P clusters, units_inv_long for those with
    // one cluster more
    uint32_t units_inv, units_inv_long;
    int merge;                 // 0: partial vectors + ordered final sum; 1: bulk reduce-add of row segments into y
    // kBatch: gridDim.y vectors against the same matrix, gridDim.x blocks each (all of them resident at once);
    // vector v = blockIdx.y takes x + v * ldx, y + v * ldy and ticket v
    int64_t ldx, ldy;
    uint32_t spin_limit;       // polls a bounded wait makes before it gives up
    // a1 done by the producer of the activations: when list_count is not null the surviving columns and their
    // values come from this list (any order, every column at most once) and x and tau are not looked at
    const int32_t *list_idx;
    const uint16_t *list_val;
    const int32_t *list_count;
    int32_t *ep_count;         // not null: set to zero for the list that k_epilogue appends to after this kernel
    int image_early;           // 0: the kernel before this one may be writing the image
};

// Parameters of k_spmspv_direct, in the order in which a block looks at them: every 64 bytes of parameters that a kernel
// touches may be a miss of the constant cache on its way.  (As a part of FusedParams, 430 bytes of which a block read here and
// there: 0.1 to 0.15 us per call, 4096 x 4096 6.01 instead of 5.89.)
struct DirectParams {
    const uint32_t *meta;      // as in FusedParams, where nothing else is said
    int32_t K, S, P, G;
    union {
        DirectSizes sizes[2];  // of the groups
        struct { const int32_t *idx; uint32_t units_inv, units_inv_long; } list;        // list builds
    };
    int32_t R, D;
    float *y;
    int32_t clear_rows, clear_extra;

    DirectSmem lay;
    union {
        struct { int32_t rankers; float rankers_inv; };
        const int32_t *list_count;
    };
    int32_t image_early;
    float tau;
    const uint16_t *x;         // list builds: the list's values
    uint32_t *tickets;

    const uint8_t *stream;
    uint32_t G_inv;            // i / G = i * G_inv >> 16 for i < 4096
    int32_t cap, slot_bytes;
    uint32_t spin_limit;
    int32_t M, C;
    int32_t *ep_count;

    int32_t *idx;
    uint16_t *val;
    int32_t *count;
    uint32_t *status;
    int64_t ldx, ldy;
};

// Shape of a fused launch (plan_fused).
struct FusedPlan {
    int G, Sc, P, D, cl, pp, mix, slot_bytes, cap, threads, grid, merge;
    int window;                // bytes of the offset window where it has a place of its own (several vectors), else -1
    int lean;                  // 0: every option compiled in; 1 / 2: the builds for the default launch (without / with warp pairs)
    int direct;                // 1: columns are dealt (k_spmspv_direct)
    int wide;                  // 1: and a ranking lane may hold several
    DirectGroups groups;       // of its blocks (not from a list)
    DirectSmem tables;         // its shared memory
    size_t smem;
};

// A launch worked out once for a handle, a device and a kind of call (prepared_launch): its shape and what of its
// parameters follows from it.
struct PreparedLaunch {
    int device = -1;           // -1: not worked out
    int status = 0;            // what working it out came to
    FusedPlan plan{};
    FusedParams params{};
};

inline size_t fused_smem_bytes(int R, int K, int G, int Sc, int D, int slot_bytes, int cap)
{
    return fused_smem_layout(R, K, G * Sc, D, slot_bytes, cap).total;
}

// Shared memory of the COLUMN kernel.
constexpr int kColumnWindow = 256;     // columns of the offset table a block fetches while the previous kernel ends

struct ColumnSmem { uint32_t acc, dump, spans, items, imeta, window, warps, keep, rank, total; };

CELTY_HD inline ColumnSmem column_smem_layout(int M, int K, int groups, int cap, int own_list)
{
    ColumnSmem l;
    uint32_t off = 0;
    l.acc = off;    off += (uint32_t)groups * ((M + 3) & ~3) * 4u;    // one accumulator per group
    l.dump = off;   off += 32u * 4u;                                 // where the lanes of a column's last chunk put what is no entry
    l.items = off;  off += (uint32_t)cap * 8u;                       // {column, x bits}
    l.imeta = off;  off += (uint32_t)cap * 8u;                       // {offset/16, entries}
    l.window = off; off += own_list ? (uint32_t)kColumnWindow * 8u : 0u;
    l.spans = off;  off += 2u * 32u * 4u;                            // rows spanned by each warp's chunk, two columns deep
    l.warps = off;  off += 33u * 4u;                                 // survivors before each warp's words, and of all
    l.keep = off;   off += own_list ? (uint32_t)((K + 31) / 32) * 4u : 0u;
    l.rank = off;   off += own_list ? (uint32_t)((K + 31) / 32) * 4u : 0u;   // survivors before each keep word
    l.total = (off + 15u) & ~15u;
    return l;
}

// Warps per column and columns in flight of the COLUMN kernel.
struct ColumnShape { int W, groups, cap, own_list; size_t smem; };

inline ColumnShape column_shape(int64_t M, int64_t K, size_t stream_bytes, size_t budget, int grid)
{
    ColumnShape s{};
    const int64_t columns = (K + grid - 1) / grid;                     // a block has, at most
    s.cap = (int)std::min<int64_t>(1024, columns + 1);
    // W warps take ceil(chunks / W) passes over a column, and 32 / W columns are in flight: the split with the fewest
    // passes for a block's share of the columns (taken as half of them; a tenth of a chunk more than the average, so
    // that columns a little longer than that need no pass of their own).  4096 x 4096, 50 %: 11.5 us of
    // device time with the 9 warps for each of 3 columns that this gives, 11.8 with 4 for 8, 12.3 with 6 for 5, 13.2 with 8
    // for 4; 7000 x 2300: 11.4 with the 7 for 4, 11.9 with 16 for 2, 13.3 with 4 for 8; 28672 x 8192, one column at a
    // time: 92.9 with the 29, 94.0 with 32, 110.5 with 16
    const double chunks = (double)stream_bytes / 20.0 / (double)K / kChunkGroups + 0.1;
    const int64_t share = std::max<int64_t>(1, (K / 2 + grid - 1) / grid);
    int64_t best = 0;
    const int64_t room = std::max<int64_t>(1, ((int64_t)budget - 24576) / (4 * ((M + 3) & ~3)));
    for (int w = 1; w <= 32; ++w) {
        const int64_t groups = std::min(std::min(columns, room), (int64_t)(w > 1 ? std::min(15, 32 / w) : 32));   // 15: named barriers
        const int64_t passes = ((share + groups - 1) / groups) * (int64_t)std::ceil(chunks / w);
        if (w == 1 || passes < best) {
            best = passes;
            s.W = w;
            s.groups = (int)groups;
        }
    }
    for (s.own_list = 1; s.own_list >= 0; --s.own_list) {
        // thresholding in the blocks needs 8 bytes per 32 activations; where they leave no room: k_compact
        if (s.own_list && K > 262144) continue;
        for (int g = s.groups; g >= 1; --g) {
            s.smem = column_smem_layout((int)M, (int)K, g, s.cap, s.own_list).total;
            if (s.smem <= budget) { s.groups = g; return s; }
        }
    }
    s.groups = 0;
    return s;
}

// Whether the COLUMN kernel's blocks get their columns dealt (k_spmspv_direct): up to 128 columns per block, at least two warps that
// do not stream, for the list, with a named barrier of their own, and room for the columns.  Where all warps stream, four of those that
// take a column each are given up, or columns in flight that the block's share does not fill, or one of several warps on a column if the
// others need no pass more for it.  A block may have one or two
// columns more than the mean, so where a block's columns take long (more passes over one than there are others in flight) survivors
// are ranked: dealt, 28672 x 8192 at 20 % took 49.8 us instead of 43.4, 20000 x 4000 at 30 % 29.6 instead of 26.6.
inline bool column_dealt(int64_t M, int64_t K, size_t stream_bytes, int grid, size_t budget, ColumnShape *shape, DirectGroups *g)
{
    ColumnShape s = *shape;
    if (!s.own_list || (K + grid - 1) / grid > 128) return false;
    const double chunks = (double)stream_bytes / 20.0 / (double)K / kChunkGroups + 0.1;
    const int most = s.W == 1 ? 28 : 30;                          // warps that stream
    if (s.W == 1) s.groups = std::min(s.groups, most);
    const int64_t share = std::max<int64_t>(1, (K / 2 + grid - 1) / grid);           // as in column_shape
    while (s.W > 1 && s.groups > 1 && (s.W * s.groups > 28 || s.groups > 14) && (share + s.groups - 2) / (s.groups - 1) == (share + s.groups - 1) / s.groups) --s.groups;
    while (s.W > 2 && s.W * s.groups > most && std::ceil(chunks / (s.W - 1)) == std::ceil(chunks / s.W)) --s.W;
    if (std::ceil(chunks / s.W) > s.groups || s.W * s.groups > most || (s.W > 1 && s.groups > 14)) return false;
    const int warps = std::min(16, s.W * s.groups);
    *g = direct_groups(K, grid, 1, warps, false);
    s.smem = column_smem_layout((int)M, (int)K, s.groups, s.cap, s.own_list).total;
    if (direct_columns(K, grid) > 32 * warps || s.smem + (size_t)g->most * 16 > budget) return false;
    *shape = s;
    return true;
}

// A COLUMN launch worked out once for a handle and a device.
struct PreparedColumn {
    int device = -1;           // -1: not worked out
    ColumnShape shape{};
    DirectGroups groups{};
    bool dealt = false;
};

// Launch choices of a handle (celty_set_launch and its neighbours); a default-constructed one is the library's.
struct LaunchKnobs {
    int32_t grid = 0, variant = 0, groups = 0, depth = 0, cluster = 0;
    int32_t pairs = -1;                       // fused kernel, two warps per team that take turns at its accumulator:
                                              // -1 = library's choice, 0 = never, 1 = always
    int32_t reg_rows = 0;                     // register-accumulation study: local rows per lane summed in registers
    uint32_t spin_limit = 0;                  // bounded waits inside the kernels: 0 = the library's limit
    int32_t mix = -1;       // fused kernel, left-over blocks shared between row parts: 0 never, 1 wherever it is even, -1 where it pays
    int32_t lean = -1;      // fused kernel: 0 = always the build with every option compiled in
    int32_t no_overlap = 0; // fused kernel: 1 = plain launch (no programmatic dependent launch)
    int32_t merge = -1;     // fused kernel: -1 = library's choice, 0 = ordered two-stage sum, 1 = bulk reduce-add
};

}  // namespace celty

// The handle.  Host side: logical block pointers and the packed image exactly as it is copied to
// the device.  Device side: caller-owned buffers recorded by celty_bind_device.
struct celty_matrix : celty::LaunchKnobs {
    int64_t M = 0, K = 0;
    int32_t layout = 0;
    int32_t R = 0;          // local rows per tile (LANE_TILE) or M (COLUMN)
    int32_t C = 1;          // LANE_TILE: groups of 32 rows that go to the same slab in a row (see tile_row)
    int64_t T = 1;          // tiles per column (LANE_TILE: 32 * S)
    int64_t S = 1;          // slabs of 32 tiles per column (LANE_TILE), 1 for COLUMN
    int32_t P = 1, Sc = 1;  // LANE_TILE: row parts per column and slabs per part (P * Sc >= S)
    int64_t nnz = 0, n_pad = 0;
    celty::Raw<uint32_t> block_ptr;    // K*T + 1, stored entries before block (j, t)
    celty::Raw<uint8_t> pad_bits;      // one bit per stored entry (logical order): 1 = padding entry
    // image = [meta | stream]
    //   COLUMN:    meta = uint2[K]  {offset/16 of the column block in the stream, entries}
    //   LANE_TILE: meta = uint32[K*S + 1]  offset/16 of sub-block (j, s); sub-blocks are contiguous
    celty::Raw<uint8_t> image;
    size_t meta_bytes = 0;             // stream starts at image[meta_bytes]
    size_t stream_bytes = 0;
    uint32_t max_unit16 = 0;           // largest column block / sub-block in 16-byte units

    // device binding
    uint8_t *d_image = nullptr;
    uint8_t *d_ws = nullptr;
    celty::WorkspaceLayout ws{};
    int32_t last_grid = 0, last_merge = -1;   // what the tickets in the workspace were last used with
    int32_t last_batch_grid[9] = {};          // the same for the tickets of launches that serve 2 .. 8 vectors
    celty::PreparedLaunch prepared[9];        // [0] one vector, [1] one from a list, [v] launches that serve v = 2 .. 8
    celty::PreparedColumn prepared_column;
    void forget_launches()                    // the handle has changed
    {
        for (celty::PreparedLaunch &p : prepared) p.device = -1;
        prepared_column.device = -1;
    }
};
