// ws_kernels.cuh -- launch interface between the C ABI (ws_api.cu) and the
// kernels.  Internal; not installed.
#pragma once
#include "ws_block.cuh"

template <typename T> struct SmallCfg;
template <> struct SmallCfg<float> { static constexpr int M = 16; static constexpr int CAP = 256 * 16; };
template <> struct SmallCfg<double> { static constexpr int M = 16; static constexpr int CAP = 256 * 16; };

// lambda of every segment: an array in device memory, or one value for the
// single segment of a vector call.
struct WsLambda {
    const double* ptr;
    double one;
    __device__ __forceinline__ double at(int seg) const { return ptr ? ptr[seg] : one; }
};

// Opt-in per-launch timing (CUDA events recorded on the launching stream
// around every kernel) and a launch counter.  Host-side only.
enum WsKernelKind {
    WSK_SMALL = 0, WSK_SORT_PLAN, WSK_PARTITION, WSK_BIN_SORT, WSK_OVERSIZE, WSK_TILE_HULL, WSK_ROOT,
    WSK_VALUES, WSK_BIN_OUT, WSK_REGROUP, WSK_OUTPUT, WSK_BWD, WSK_MISC, WSK_TILE_GENERAL, WSK_JUNCTION, WSK_CLIMB, WSK_COUNT
};
struct WsProf {
    bool enabled = false;
    int cap = 0, n = 0;
    cudaEvent_t* ev = nullptr;   // 2 * cap events
    int* kind = nullptr;         // cap
    long long launches = 0;
    void begin(cudaStream_t st, int k) {
        ++launches;
        if (!enabled || n >= cap) return;
        cudaEventRecord(ev[2 * n], st);
        kind[n] = k;
    }
    void end(cudaStream_t st) {
        if (!enabled || n >= cap) return;
        cudaEventRecord(ev[2 * n + 1], st);
        ++n;
    }
};
// Programmatic dependent launch inside one call's chain: a kernel launched by
// ws_launch_chain is placed on the SMs while its predecessor's last CTAs run,
// and waits in ws_chain() for the predecessor's end before it touches memory,
// so the 1.5 to 2 us between two kernels overlap (d = 40960, 15 launches: 127
// -> 104 us).  Every kernel launched this way starts with ws_chain() or
// ws_chain_wait(); a persistent kernel lets its successor in (ws_chain_go) with
// its last tile only.  early = false is a plain launch.
__device__ __forceinline__ void ws_chain_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void ws_chain_go() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void ws_chain() {
    ws_chain_go();
    ws_chain_wait();
}
template <typename... P, typename... A>
inline void ws_launch_if(bool early, void (*kernel)(P...), int grid, int block, size_t smem, cudaStream_t st,
                         A... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3((unsigned)block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = early ? 1 : 0;
    cudaLaunchKernelEx(&cfg, kernel, P(args)...);
}
template <typename... P, typename... A>
inline void ws_launch_chain(void (*kernel)(P...), int grid, int block, size_t smem, cudaStream_t st, A... args) {
    ws_launch_if(true, kernel, grid, block, smem, st, args...);
}
#define WS_LAUNCH(PROF, KIND, ST, ...) \
    do { (PROF)->begin((ST), (KIND)); __VA_ARGS__; (PROF)->end((ST)); } while (0)

// Large-path tile geometry.
constexpr int WS_SORT_NT = 512;              // threads per partition CTA
constexpr int WS_SORT_ITEMS = 12;            // keys per thread
constexpr int WS_SORT_TILE = WS_SORT_NT * WS_SORT_ITEMS;   // 6144 keys per sort tile
// Distribution sort (ws_sort.cu): bins of about WS_BIN_MEAN keys, sorted by
// one CTA up to WS_BIN_CAP keys.  The ratio 1.6 leaves room for the error of
// the sampled map (5 to 14 % standard deviation on N(0, 1), the largest bin 1.2
// to 1.55 times the mean; a mean of 2816 let a few bins of the tails overflow).
constexpr int WS_BWD_BIN_LOG2 = 11, WS_BWD_BIN = 1 << WS_BWD_BIN_LOG2;   // backward: cluster slots per bin (48 KB of sums)
constexpr int WS_BWD_PIECE = 16384; // pairs of a bin that one CTA adds
constexpr int WS_BWD_FAN = 512;    // buckets of one move of the backward
constexpr int WS_BIN_CAP = 4096;
constexpr int WS_BIN_MEAN = 2560;
// Bins that leave a partition's rank word room for the rank.  More of them (a second
// pass of four rounds per tile instead of two, and a word for the top bits) cost 1.4 as
// much to partition, so bins grow to WS_BIN_MEAN_BIG keys first: 1.4e9 weights 74 ms, 81 with more bins.
constexpr int WS_BINS_RANK = 1 << 19;
constexpr int WS_BIN_MEAN_BIG = 3000;
constexpr int WS_FAN = 512;                  // buckets a partition tile counts at a time
constexpr int WS_ONE_LEVEL = 512;            // segments of at most this many bins take one partition pass
constexpr int WS_CELLS = 2048;               // cells of the map (two-level segments; half as many otherwise)
constexpr int WS_HULL_NT = 256;              // threads per hull-tile CTA
constexpr int WS_HULL_M = 16;                // points per thread chunk
constexpr int WS_HULL_TILE = WS_HULL_NT * WS_HULL_M;       // 4096 elements per hull tile

// One tile of a large segment (sort tiles and hull tiles use the same record).
struct TileDesc {
    int64_t kpos;      // first element in the compact key buffer
    int64_t vpos;      // first element in the caller's value array
    int32_t len;       // elements in the tile
    int32_t lseg;      // large-segment index
    int32_t first;     // global index of the segment's first tile (of this kind)
    int32_t tin;       // index of the tile inside its segment
};

// One large segment.
struct LargeSeg {
    int64_t vpos;      // first element in the caller's arrays
    int64_t kpos;      // first element in the compact key buffer
    int64_t len;
    int32_t seg;       // index in the caller's segment list
    int32_t sort_first, sort_count;   // sort tiles
    int32_t hull_first, hull_count;   // hull tiles
    // distribution sort
    int32_t nbins;             // bins of the segment
    int32_t fine_log2;         // first pass: bucket = bin >> fine_log2 (0: one pass only)
    int32_t n_coarse;          // buckets of the first pass
    int32_t ncell;             // cells of the segment's map (a power of two; 0 for one tile, which needs no map)
    int32_t samp_log2;         // sampled elements per sort tile
    int32_t bin_pos, coarse_pos;   // slices of the per-bin / bucket arrays
    int64_t cell_pos;              // and of the cell array
    // backward: bins of cluster slots
    int32_t bb_n, bb_fine;     // bins of the segment; bucket of the first move = bin >> bb_fine (0: one move only)
    int32_t bb_pos, bb_cpos;   // slices of the per-bin / bucket arrays
};

// What a partition pass leaves to undo it.  A tile's keys lie grouped by bucket
// in its staging area; run r of them went to place + delta[r] of the segment.
// 2 bytes per key and a few per run, where a destination per key takes 4, and
// the pass is undone by runs (coalesced) instead of key by key.
struct PassMap {
    uint16_t* loc;      // [n_keys] a key's place in its tile's staging area
    uint32_t* starts;   // [n_sort_tiles][WS_SORT_TILE / 32] a bit at the first place of every run
    uint32_t* delta;    // per run; a tile's runs at tile * WS_FAN (first pass), at its first key (second)
};

// X at the vertices of a hull tile: 64-bit sums of deviations from q0 in units of
// 2^sh (one store of 8 bytes per vertex where 128 bits take a wide product, a
// shift and 16 bytes: tile hulls of 2^26 elements 415 -> 378 us, of 1024 uneven
// segments 820 -> 745), or 128-bit values
// (wide) for the tiles of the general kernel.
struct TileX {
    int64_t q0;
    int32_t sh, wide;
};
__device__ __forceinline__ i128 ws_i128(int64_t hi, uint64_t lo) { return (i128)(((u128)(uint64_t)hi << 64) | lo); }
// a b, and a 2^s for 0 <= s < 64, in two words each (the 128-bit operators take wide
// products and shifts of both words)
__device__ __forceinline__ i128 ws_mul_i64(int64_t a, int64_t b) { return ws_i128(__mul64hi(a, b), (uint64_t)a * (uint64_t)b); }
__device__ __forceinline__ i128 ws_shl_i64(int64_t a, int s) { return ws_i128((a >> 1) >> (63 - s), (uint64_t)a << s); }
struct VertX {
    const i128* x;
    const TileX* h;
    // vertex v of `tile`, at the tile's point p
    // (for searches, which wait for one load after the other: all that a vertex needs is loaded side by
    // side and picked without a branch, so that the loads of two vertices overlap as well)
    __device__ __forceinline__ i128 at(int64_t tile, int v, int p) const {
        const i128* b = x + tile * (WS_HULL_TILE + 1);
        const ulonglong2 w = __ldg(reinterpret_cast<const ulonglong2*>(b + v));
        const int64_t s = __ldg(reinterpret_cast<const int64_t*>(b) + v);
        const TileX t = h[tile];
        const i128 q = ws_mul_i64(p, t.q0) + ws_shl_i64(s, t.sh);
        const uint64_t m = t.wide ? ~0ull : 0ull;
        return ws_i128((int64_t)((w.y & m) | ((uint64_t)(q >> 64) & ~m)), (w.x & m) | ((uint64_t)q & ~m));
    }
    __device__ __forceinline__ i128 at(const TileX& t, int64_t tile, int v, int p) const {
        const i128* b = x + tile * (WS_HULL_TILE + 1);
        if (t.wide) return b[v];
        return (i128)p * (i128)t.q0 + ((i128)reinterpret_cast<const int64_t*>(b)[v] << t.sh);
    }
    // at(tile, v + 1, p + n) - at(tile, v, p), with the tile's TileX at hand
    __device__ __forceinline__ i128 step(const TileX& t, int64_t tile, int v, int n) const {
        const i128* b = x + tile * (WS_HULL_TILE + 1);
        if (t.wide) return b[v + 1] - b[v];
        const int64_t* q = reinterpret_cast<const int64_t*>(b) + v;
        return (i128)t.q0 * (int64_t)n + ((i128)(q[1] - q[0]) << t.sh);
    }
};

// Work words of the backward (device memory).
struct BwdWork {
    int n_bins, two_level;
    size_t zero_bytes;             // emax .. n_items: one block, cleared by every backward
    int32_t* emax;                 // [n_lseg] largest grad_out exponent
    uint32_t* cnt;                 // [n_bins] pairs
    uint32_t* extra;               // [n_bins] tiles of one cluster (they move no pairs)
    uint32_t* xlo;                 // [n_bins] the slots these add to: WS_BWD_BIN - the first one (0: none)
    uint32_t* xhi;                 // [n_bins] and the last one + 1
    uint32_t* arrive;              // [n_bins] finished pieces
    int32_t* n_items;              // pieces of the split bins
    const int2* map;               // [n_bins] (segment, bucket of the first move that starts here or -1)
    unsigned long long* start;     // [n_bins + 1]
    unsigned long long *cur1, *cur2;   // cursors of the moves
    uint2* items;                  // (bin, piece)
};

// Sort control words, cleared before every sort.
struct SortCtl {
    uint32_t bar;          // grid barrier of the plan kernel
    uint32_t abort;        // a barrier gave up: the keys are not moved
    uint32_t over_count;   // bins above WS_BIN_CAP
    uint32_t over_bar;     // grid barrier of the oversize kernel
    unsigned long long over_diff;   // key bits that vary inside any class above WS_BIN_CAP
    uint32_t over_items;   // classes to sort, up to WS_BIN_CAP keys
    uint32_t over_big;     // and above
    int32_t gen_count;     // hull tiles for the general kernel
    int32_t pad;
};

// Map header of a segment: cell = (key - kmin) >> shift.
struct SortHdr {
    uint64_t kmin;
    uint64_t mag;     // FP64: magnitudes below this count as it (see squeeze)
    uint64_t dlo, dhi;   // smallest and largest sample above kmin
    int32_t shift;
};

// A bin above WS_BIN_CAP.
struct OverBin {
    int64_t start;          // first key
    int32_t n;
    int32_t first_tile;     // of the oversize kernel's tiles
    int32_t lseg;
    int32_t nspl;           // splitters of its classes
};

// Its classes: 2 i + 1 the keys equal to splitter i, 2 i those between splitters
// i - 1 and i (see ws_sort.cu).
constexpr int OVER_SPL = 255;
template <typename K>
struct OverTab {
    K spl[OVER_SPL];                  // ascending, different
    uint32_t cnt[2 * OVER_SPL + 1];   // keys per class
    uint32_t cur[OVER_SPL + 1];       // write cursors of the classes between splitters
};
// Classes of N keys; spl: OVER_SPL + 1 entries, ~0 beyond the splitters.  The searches
// take one step after the other side by side (their loads overlap).
template <typename K, int N>
__device__ __forceinline__ void ws_over_classes(const K* spl, int n, const K (&key)[N], int (&cls)[N]) {
#pragma unroll
    for (int k = 0; k < N; ++k) cls[k] = 0;   // splitters below the key, so far
    for (int step = 1 << (31 - __clz(n | 1)); step > 0; step >>= 1) {
#pragma unroll
        for (int k = 0; k < N; ++k) cls[k] += spl[cls[k] + step - 1] < key[k] ? step : 0;
    }
#pragma unroll
    for (int k = 0; k < N; ++k) cls[k] = 2 * cls[k] + (cls[k] < n && spl[cls[k]] == key[k] ? 1 : 0);
}

// A class between splitters that is to be sorted.
struct OverClass {
    int64_t start;
    int32_t n;
    int32_t first_tile;        // above WS_BIN_CAP keys: of the radix passes' tiles
    unsigned long long diff;   // and the key bits that vary inside it
};

// A piece of a node hull: vertices [lo, hi) of hull tile `tile`; cum = rank of
// its first vertex within the node hull; off = fixed-point prefix X at the
// tile's first point, relative to the node's first point.
struct __align__(16) Piece {
    int32_t tile;
    uint16_t lo, hi;
    int32_t cum;
    int32_t pad;
    i128 off;
};

// Value and cluster id of one element, on its way back to the caller's order.
template <typename T> struct OutPair;
template <> struct __align__(8) OutPair<float> { float val; int32_t id; };
template <> struct __align__(16) OutPair<double> { double val; int32_t id, pad; };

// Constants of the exact hull test at one fixed-point unit scale of a
// segment: the units of a one-binade hull tile (ulps of its binade) or the
// segment's own scale.  Computed once per segment (k_scales) so that tiles do
// no FP64 or wide-integer set-up work.
struct TileScale {
    SegConst sc;      // hull-test constants at this scale
    float muq;        // lambda 2^L / (d - 1) in units, for the FP32 filter
    int fast;         // muq usable by the filter
    uint64_t modd;    // odd part of lambda 2^L (0 when lambda = 0) and its exponent
    int sodd;
    int pad;
    int64_t t11;      // lower bound of 2 lambda 2^L / (d - 1): two adjacent elements
                      // collide at once (IC round 1) if their gap <= t11 units
};
constexpr int WS_NSCALE = 64;   // per segment: binade shifts 0 .. FIX_OFS, then the segment scale last

// The constants at a segment's own scale (with lambda / (d - 1) in FP64: one
// division per segment, not one per thread of every later kernel).
__device__ __forceinline__ SegConst ws_seg_scale(const TileScale* scales, int lseg) {
    return scales[(size_t)lseg * WS_NSCALE + WS_NSCALE - 1].sc;
}

// Per-segment run-time values computed on the device.
struct SegRuntime {
    int64_t n_clusters;
    int64_t table_pos;  // first cluster value of the segment
    int32_t emax;
    int32_t pad;
};

template <typename T>
cudaError_t ws_launch_small(const T* values, const int64_t* offsets, const int32_t* seg_list, int n_list,
                            WsLambda lambdas, T* out, int32_t* ids, int64_t* n_clusters, int fp64,
                            const WsEpi& ep, uint32_t* status, cudaStream_t st, WsProf* prof, int32_t* gen_list,
                            int32_t* gen_count, int ic_cap, const int32_t* ids_prev);
template <typename T>
cudaError_t ws_launch_small_backward(const T* g, const int32_t* ids, const int64_t* offsets, const int32_t* seg_list,
                                     int n_list, T* gin, uint32_t* status, cudaStream_t st, WsProf* prof);

// Launch shapes of a plan's sort (host).
struct WsSortShape {
    bool wide = false;                                 // 32-bit bin numbers
    int hist_cap = 0;                                  // shared words of the plan kernel (bins counted, samples kept)
    int max_bins = 0;                                  // of the longest segment
    int samp_max = 0;                                  // log2 of the most samples per tile
    int plan_grid = 1, part_grid = 1, over_grid = 1;   // CTAs resident at once
    int out_extra = 1;                                 // CTAs of the way back for the oversize bins
};
template <typename T> cudaError_t ws_sort_prepare(int max_bins, int n_tiles, int samp_max, WsSortShape* sh);

// Large path workspace pointers (all device).
template <typename T>
struct LargeWork {
    typedef typename KeyOf<T>::K K;
    int n_lseg, n_sort_tiles, n_hull_tiles;
    int64_t n_keys;
    const LargeSeg* lsegs;
    const TileDesc* sort_tiles;
    const TileDesc* hull_tiles;
    K* keys_a;
    K* keys_b;
    // sort: the first sort_zero_bytes from ctl on are cleared before every sort
    SortCtl* ctl;
    size_t sort_zero_bytes;
    unsigned long long* seg_hi;   // [n_lseg] largest sampled key
    unsigned long long* seg_lo;   // [2][n_lseg] complements of the smallest sampled key and nonzero magnitude
    uint32_t* seg_en;        // [n_lseg] INT_MAX - smallest effective exponent of a nonzero value
    uint32_t* cells;         // [3 cells] sampled keys per cell, then per part of a cell
    uint32_t* bin_cnt;       // [n_bins]
    // (not cleared)
    int n_bins, two_level;
    WsSortShape sort_shape;
    void* bins;              // [2][n_keys] bin of every key (16 bits, or 32 in plans with longer segments)
    uint32_t* bin_start;     // [n_bins] first key of every bin, relative to its segment
    uint32_t* cur1;          // [coarse buckets] write cursors of the first pass
    uint32_t* cur2;          // [n_bins] write cursors of the second pass
    const int32_t* bin_seg;  // [n_bins] segment of every bin
    OverBin* over;           // [n_bins] oversize bins
    void* over_tabs;         // [n_keys / WS_BIN_CAP + 1] OverTab: their classes
    OverClass* over_items;   // [n_keys / WS_BIN_CAP + 1][OVER_SPL + 1] classes to sort
    OverClass* over_big;     // [n_keys / WS_BIN_CAP + 1] those above WS_BIN_CAP keys
    uint32_t* over_cnt;      // [n_keys / (WS_SORT_TILE / 2) + 1][256] digit counts of their tiles
    int32_t* seg_emin;       // [n_lseg] smallest effective exponent of a nonzero value
    // hull
    uint16_t* vp;            // [n_hull_tiles][WS_HULL_TILE + 1] vertex points (tile-local)
    i128* vx;                // [n_hull_tiles][WS_HULL_TILE + 1] X at vertices (tile-local; see TileX)
    TileX* hx;               // [n_hull_tiles]
    int32_t* nvert;          // [n_hull_tiles]
    i128* tile_total;        // [n_hull_tiles] node total X, stored at the node's first tile
    int32_t* arrive;         // [levels][n_hull_tiles] merge-tree arrival counters (cleared with the sort's words)
    Piece* pieces;           // [n_hull_tiles]
    int32_t* npieces;        // [n_hull_tiles] pieces of the node whose first tile is this index
    int32_t* tile_piece;     // [n_hull_tiles] piece index in the root list or -1
    int32_t* gen_list;       // [n_hull_tiles] tiles whose hull the general kernel builds
    int32_t* keepR;          // [n_hull_tiles] junction results (ws_tile.cu)
    int32_t* keepL;          // [n_hull_tiles]
    int32_t* jflag0;         // [n_hull_tiles]
    int32_t* seg_mode;       // [n_lseg] 0: junctions resolved, 3: one cluster unless seg_below (then the tree of merges)
    i128* tile_base;         // [n_hull_tiles] X at every hull tile's first point (segment frame)
    TileScale* scales;       // [n_lseg][WS_NSCALE]
    int32_t* tile_rounds;    // [n_hull_tiles] in-tile IC rounds to converge, -1 chain + trees, -2 general kernel
    int ic_cap;              // in-tile IC round cap (0: chain + trees only)
    i128* seg_total;         // [n_lseg] X of the whole segment
    int32_t* seg_below;      // [n_lseg] a tile-hull vertex lies below the segment's chord
    SegRuntime* rt;          // [n_lseg]
    T* cval;                 // [n_keys + n_lseg] cluster values
    uint2* rank_words;       // [n_hull_tiles][WS_HULL_TILE / 32] cluster starts among 32 sorted positions, starts before
    // way back to the caller's order
    PassMap map1, map2;      // how to undo the first pass and the second (two-level plans)
    uint16_t* bin_idx;       // [n_keys] for every sorted position, its key's place in the unsorted bin
    OutPair<T>* pairs_a;     // [n_keys] in the first pass's order (two-level segments)
    OutPair<T>* pairs_b;     // [n_keys] in bin order; before that, scratch of the oversize bins' sort
    // backward
    T* bsum;                 // [n_keys + n_lseg] cluster means
    int32_t* bcnt;           // [n_keys + n_lseg] cluster sizes
    unsigned long long* bacc;   // [n_keys + n_lseg][2] exact cluster sums (128-bit, low word first)
    BwdWork bwd;
    WsProf* prof;            // host-side launch accounting
};

// way_back: also record where every key goes (map1, map2, bin_idx).
template <typename T>
cudaError_t ws_large_sort(const LargeWork<T>& W, const T* values, bool way_back, uint32_t* status,
                          uint64_t spin_limit, cudaStream_t st, typename KeyOf<T>::K** sorted);
// Lean tile hulls and the junction resolution (ws_tile.cu).
template <typename T>
cudaError_t ws_large_hull_fast(const LargeWork<T>& W, typename KeyOf<T>::K* sorted, WsLambda lambdas,
                               uint32_t* status, cudaStream_t st);
template <typename T>
cudaError_t ws_large_junctions(const LargeWork<T>& W, cudaStream_t st);
template <typename T>
cudaError_t ws_large_prox(const LargeWork<T>& W, const T* values, WsLambda lambdas, T* out, int32_t* ids,
                          int64_t* n_clusters, int fp64, const WsEpi& ep, uint32_t* status, uint64_t spin_limit,
                          cudaStream_t st);
template <typename T>
cudaError_t ws_large_backward(const LargeWork<T>& W, const T* g, const int32_t* ids, T* gin, uint32_t* status,
                              cudaStream_t st);
template <typename T>
cudaError_t ws_large_copy_sorted(const LargeWork<T>& W, const typename KeyOf<T>::K* sorted, T* dst, cudaStream_t st);
// R(w) and the weight-sharing measure per large segment (ws_stats.cu);
// `partial` holds ws_R_partial_bytes(n_sort_tiles) bytes of device scratch.
template <typename T>
cudaError_t ws_large_R(const LargeWork<T>& W, const T* values, double* R_out, double* metric_out, uint32_t* status,
                       uint64_t spin_limit, void* partial, cudaStream_t st);
size_t ws_R_partial_bytes(int n_sort_tiles);
template <typename T>
cudaError_t ws_tiny_R(const T* values, int64_t d, double* R_out, double* metric_out, WsProf* prof, cudaStream_t st);
// d <grad_out, out> / d lambda per segment, partition held fixed (ws_stats.cu);
// `partial` as for ws_large_R.
template <typename T>
cudaError_t ws_dlambda(const T* g, const int32_t* ids, const int64_t* d_offsets, const int32_t* d_small, int n_small,
                       int64_t n_seg, const LargeWork<T>& W, double* out, uint32_t* status, void* partial,
                       cudaStream_t st);
