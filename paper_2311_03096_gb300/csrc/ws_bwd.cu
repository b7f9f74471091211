// ws_bwd.cu -- the backward of the prox with the partition held fixed: every
// element's gradient is the mean of grad_out over its cluster (the Jacobian
// of the cluster means; a cluster moves as one particle, Sec. 3).
//
// The cluster sums are exact and deterministic: every grad_out value is
// converted to a 128-bit integer at a per-segment scale (exact for values
// within SH binades of the segment's largest |g|: 71 for float, 42 for
// double; smaller ones keep their top bits), and the integers are added with
// 64-bit atomics that carry into the high word explicitly.  Integer addition
// is associative, so the sum -- hence the mean -- does not depend on the
// order of the additions, and its error does not grow with the cluster size
// (one rounding when the mean is formed).
//
// Device-wide segments: the (grad_out, id) pairs are moved into bins of
// WS_BWD_BIN consecutive cluster slots, whose sums fit the shared memory of one
// CTA.  k_bwd_prep finds the segment's scale and counts the bins, k_bwd_scan
// turns the counts into bin starts, k_bwd_part moves the pairs (in one pass up
// to WS_BWD_FAN bins, in two above, as the forward's sort), k_bwd_bins adds a
// bin's pairs into limbs in shared memory and writes the means, k_bwd_apply
// gathers them.  A bin with more than PIECE pairs is added by several CTAs
// (128-bit global atomics per slot, the last one writes the means).  A tile whose
// elements all share one cluster adds its sum once and moves no pairs, so a
// single huge cluster costs one atomic per tile.  The pairs borrow buffers of the
// forward, which the backward does not otherwise use.
//
// FP32 2^24, clusters of a few elements, us: prep 52 (issue, the bins' adds),
// scan 10, moves 71 + 67 (shared-memory wavefronts, 0.67 of the pipe), bins 123
// (issue, 0.71: half the adds, half the conversions of 15 million means), apply
// 76 (one line per lane and clock of the L1: 0.75 of that).  Three 64-bit global
// atomics per pair instead of the bins took 876 in all; in every case measured
// (from 5000 elements to 2^25, from one cluster to all distinct) the bins are
// faster: 7 clusters of 2^24 elements 2825 -> 426, one cluster beside short ones
// 1508 -> 420, 100000 elements 90 -> 30, 2^25 FP64 2201 -> 1492.
// One-CTA segments: the same arithmetic in shared memory (k_small_backward).
#include "ws_kernels.cuh"

namespace {

constexpr int BTILE = WS_SORT_TILE;   // elements per tile (the sort tiles of the plan)
constexpr int PNT = WS_SORT_NT, ITEMS = WS_SORT_ITEMS;
constexpr int ANT = 256;              // k_bwd_bins
constexpr int PIECE = WS_BWD_PIECE;
constexpr int CHUNK = 8 * ANT;        // pairs of one step of k_bwd_bins
constexpr int EXTRA = 4 * 152;        // CTAs of k_bwd_bins for the split bins
constexpr int MAIN = 8192;            // and for the others at most (empty bins cost a CTA's launch: 24576 of them 50 us)
constexpr int HIST_MAX = 16384;       // bins that k_bwd_prep counts in shared memory

template <typename T> struct BwdFix;
template <> struct BwdFix<float> { static constexpr int SH = 71, BIAS = 127, MANT = 23; };
template <> struct BwdFix<double> { static constexpr int SH = 42, BIAS = 1023, MANT = 52; };

// g * 2^(SH - emax + BIAS + MANT) as an integer (exact unless g is more than
// SH binades below 2^emax; then truncated toward zero).
template <typename T>
__device__ __forceinline__ i128 ws_bwd_fix(T g, int emax) {
    typedef KeyOf<T> KO;
    const uint64_t b = (uint64_t)KO::bits(g);
    int e = (int)((b >> KO::MANT) & KO::EXPMASK);
    uint64_t m = b & ((1ull << KO::MANT) - 1ull);
    if (e == 0) e = 1; else m |= (1ull << KO::MANT);
    const int sh = e - emax + BwdFix<T>::SH;
    u128 mag;
    if (sh >= 0) mag = (u128)m << sh;
    else mag = (sh > -64) ? (u128)(m >> (-sh)) : (u128)0;
    const bool neg = (b >> (KO::BITS - 1)) & 1ull;
    return neg ? -(i128)mag : (i128)mag;
}

// mean = S / cnt * 2^-(SH - emax + BIAS + MANT)
template <typename T>
__device__ __forceinline__ T ws_bwd_mean(i128 S, int cnt, int emax) {
    const int Lg = BwdFix<T>::SH - emax + BwdFix<T>::BIAS + BwdFix<T>::MANT;
    if (sizeof(T) == 4) {
        // as ws_i128_to_float_scaled(S, 0) / cnt * 2^-Lg with one scaling: powers of two commute with
        // the division (no step leaves the normal range), and one multiplication rounds like ldexpf
        const u128 mag = S < 0 ? (u128)(-S) : (u128)S;
        const int sh = max(ws_bitlen128(mag) - 62, 0);
        const float f = ws_u64_to_float((uint64_t)(mag >> sh)) / (float)cnt;
        const int e = sh - Lg;
        const float r = e >= -126 && e <= 127 ? f * __int_as_float((e + 127) << 23) : ldexpf(f, e);
        return (T)(S < 0 ? -r : r);
    }
    return (T)ldexp(ws_div_i128_n(S, cnt), -Lg);
}

__device__ __forceinline__ void ws_atomic_add_i128(unsigned long long* lo_hi, i128 v) {
    const unsigned long long lo = (unsigned long long)(uint64_t)v;
    const unsigned long long hi = (unsigned long long)(uint64_t)((u128)v >> 64);
    const unsigned long long old = atomicAdd(lo_hi, lo);
    atomicAdd(lo_hi + 1, hi + (old + lo < old ? 1ull : 0ull));
}

template <typename T> __device__ __forceinline__ int ws_g_exp(T g) { return g != (T)0 ? ws_eff_exp(g) : 0; }

template <typename T> __device__ __forceinline__ T ws_g_of_bits(typename KeyOf<T>::K b) {
    if (sizeof(T) == 4) return (T)__uint_as_float((uint32_t)b);
    return (T)__longlong_as_double((long long)b);
}

// Sum of v over the lanes in `peers` (every one of them calls with the same
// mask; the groups of a __match_any_sync may call side by side).  |v| < 2^95
// (a ws_bwd_fix value), so v + 2^95 lies in [0, 2^96): its four 24-bit limbs
// are summed separately -- at most 32 * (2^24 - 1) < 2^29 each, no carry is
// lost -- and recombined.  Exact.
__device__ __forceinline__ i128 ws_group_sum_i96(unsigned peers, i128 v) {
    const u128 o = (u128)(v + ((i128)1 << 95));
    const uint32_t lo = (uint32_t)(uint64_t)o, mid = (uint32_t)(uint64_t)(o >> 32),
                   hi = (uint32_t)(uint64_t)(o >> 64);
    const uint32_t s0 = __reduce_add_sync(peers, lo & 0xffffffu);
    const uint32_t s1 = __reduce_add_sync(peers, (lo >> 24) | ((mid & 0xffffu) << 8));
    const uint32_t s2 = __reduce_add_sync(peers, (mid >> 16) | ((hi & 0xffu) << 16));
    const uint32_t s3 = __reduce_add_sync(peers, hi >> 8);
    const u128 S = (u128)s0 + ((u128)s1 << 24) + ((u128)s2 << 48) + ((u128)s3 << 72);
    return (i128)S - (i128)__popc(peers) * ((i128)1 << 95);
}

// Sums in shared memory, as five signed 19-bit limbs per cluster.  A grad_out
// value of MANT + 1 bits falls into at most three of them (four for double),
// each one 32-bit shared-memory add without a returned value (native; a 64-bit
// shared atomic is a compare-and-swap loop), and 4096 adds of 19 bits cannot
// overflow 32.  The limbs recombine to the integer that 128-bit additions give.
constexpr int LIMBS = 5, LIMB_BITS = 19;   // 95 bits: every ws_bwd_fix value
constexpr uint32_t LIMB_MASK = (1u << LIMB_BITS) - 1u;

// p[l * STRIDE] += limb l of ws_bwd_fix(g, emax)
template <typename T, int STRIDE>
__device__ __forceinline__ void ws_limb_add(int* p, T g, int emax) {
    typedef KeyOf<T> KO;
    static_assert(LIMBS * LIMB_BITS >= BwdFix<T>::SH + BwdFix<T>::MANT + 1, "every value fits");
    // grad_out = +-m 2^sh in units of the fixed point, as in ws_bwd_fix
    if (sizeof(T) == 4) {   // (32-bit arithmetic: the integer pipe bounds the kernels)
        const uint32_t b = (uint32_t)KO::bits(g);
        const int ex = (int)((b >> 23) & 255u);
        uint32_t m = (b & 0x7fffffu) | (ex ? 0x800000u : 0u);
        int sh = max(ex, 1) - emax + BwdFix<T>::SH;
        if (sh < 0) { m = sh > -32 ? m >> (-sh) : 0u; sh = 0; }
        const int l0 = (sh * 27) >> 9;   // sh / 19 for 0 <= sh <= 94
        const int r = sh - LIMB_BITS * l0;
        const uint32_t lo = m << r, hi = __funnelshift_l(m, 0u, r);   // m << r: 42 bits
        const int sg = (int)b >> 31;     // 0 or -1: x ^ sg - sg is +-x
        p += l0 * STRIDE;
        const uint32_t v0 = lo & LIMB_MASK, v1 = __funnelshift_r(lo, hi, LIMB_BITS) & LIMB_MASK,
                       v2 = hi >> (2 * LIMB_BITS - 32);
        if (v0) atomicAdd(p, ((int)v0 ^ sg) - sg);
        if (v1) atomicAdd(p + STRIDE, ((int)v1 ^ sg) - sg);
        if (v2) atomicAdd(p + 2 * STRIDE, ((int)v2 ^ sg) - sg);
        return;
    }
    const uint64_t b = (uint64_t)KO::bits(g);
    int ex = (int)((b >> KO::MANT) & KO::EXPMASK);
    uint64_t m = b & ((1ull << KO::MANT) - 1ull);
    if (ex == 0) ex = 1; else m |= 1ull << KO::MANT;
    int sh = ex - emax + BwdFix<T>::SH;
    if (sh < 0) { m = sh > -64 ? m >> (-sh) : 0ull; sh = 0; }
    const bool neg = (b >> (KO::BITS - 1)) & 1ull;
    const int l0 = (sh * 27) >> 9;   // sh / 19 for 0 <= sh <= 94
    const int r = sh - LIMB_BITS * l0;
    p += l0 * STRIDE;
    auto add = [&](int l, uint32_t v) {
        if (v) atomicAdd(p + l * STRIDE, neg ? -(int)v : (int)v);
    };
    const uint64_t w = m << r;   // (the low 64 of 71 bits)
    add(0, (uint32_t)w & LIMB_MASK);
    add(1, (uint32_t)(w >> LIMB_BITS) & LIMB_MASK);
    add(2, (uint32_t)(w >> (2 * LIMB_BITS)) & LIMB_MASK);
    add(3, (uint32_t)((m >> (3 * LIMB_BITS - 18)) >> (18 - r)) & LIMB_MASK);   // (m << r) >> 57, r <= 18
}
template <int STRIDE>
__device__ __forceinline__ i128 ws_limb_sum(const int* p) {
    const int64_t A = (int64_t)p[0] + ((int64_t)p[STRIDE] << LIMB_BITS);
    const int64_t B = (int64_t)p[2 * STRIDE] + ((int64_t)p[3 * STRIDE] << LIMB_BITS);
    return (i128)A + ((i128)B << (2 * LIMB_BITS)) + ((i128)p[4 * STRIDE] << (4 * LIMB_BITS));
}

// 1. per segment the largest exponent of grad_out; per bin the elements of the
// tiles that are not one cluster (cnt) and the tiles that are (extra).  Up to
// HIST_MAX bins are counted in shared memory by a persistent grid.
template <typename T>
__global__ void __launch_bounds__(PNT, 3) k_bwd_prep(const T* __restrict__ g, const int32_t* __restrict__ ids,
                                                     const TileDesc* __restrict__ tiles, int n_tiles,
                                                     const LargeSeg* __restrict__ lsegs, int n_hist, int32_t* seg_emax,
                                                     uint32_t* cnt, uint32_t* extra, uint32_t* xlo, uint32_t* xhi,
                                                     uint32_t* status) {
    extern __shared__ uint32_t hist[];   // [n_hist]
    const int t = threadIdx.x, lane = t & 31;
    for (int b = t; b < n_hist; b += PNT) hist[b] = 0;
    bool bad = false;
    for (int tile = blockIdx.x; tile < n_tiles; tile += gridDim.x) {
        const TileDesc td = tiles[tile];
        const LargeSeg& ls = lsegs[td.lseg];
        const int64_t slen = ls.len;
        const int bpos = ls.bb_pos;
        int idv[ITEMS];
        T gv[ITEMS];
#pragma unroll
        for (int k = 0; k < ITEMS; ++k) {   // (indices clamped into the tile: every load in bounds)
            const int i = min(t + k * PNT, td.len - 1);
            idv[k] = __ldg(ids + td.vpos + i);
            gv[k] = __ldg(g + td.vpos + i);
        }
        const int id0 = __ldg(ids + td.vpos);
        int e = 0;
        bool same = true;
#pragma unroll
        for (int k = 0; k < ITEMS; ++k) {
            e = max(e, ws_g_exp(gv[k]));
            same &= idv[k] == id0;
        }
        e = __reduce_max_sync(0xffffffffu, e);
        if (lane == 0 && e > *(volatile int32_t*)(seg_emax + td.lseg)) atomicMax(seg_emax + td.lseg, e);
        if (__syncthreads_and(same)) {   // (also the barrier after the clearing of hist)
            if (id0 < 0 || (int64_t)id0 >= slen) bad = true;
            else if (t == 0 && td.len < slen) {   // (the only tile of its segment writes the mean itself)
                const int b = bpos + (id0 >> WS_BWD_BIN_LOG2), r = id0 & (WS_BWD_BIN - 1);
                atomicAdd(extra + b, 1u);
                atomicMax(xlo + b, (uint32_t)(WS_BWD_BIN - r));
                atomicMax(xhi + b, (uint32_t)(r + 1));
            }
            continue;
        }
#pragma unroll
        for (int k = 0; k < ITEMS; ++k) {
            const bool here = t + k * PNT < td.len;
            const bool ok = here && idv[k] >= 0 && (int64_t)idv[k] < slen;
            bad |= here && !ok;
            const int b = bpos + (idv[k] >> WS_BWD_BIN_LOG2);
            const unsigned crowd = ws_crowd(b, ok);
            uint32_t add = ok ? 1u : 0u;
            if ((crowd >> lane) & 1u) add = lane == __ffs((int)crowd) - 1 ? (uint32_t)__popc(crowd) : 0u;
            if (add) {
                if (n_hist) atomicAdd(&hist[b], add);
                else atomicAdd(cnt + b, add);
            }
        }
    }
    if (bad) ws_flag(status, WS_STATUS_INTERNAL);
    __syncthreads();
    for (int b = t; b < n_hist; b += PNT)
        if (hist[b]) atomicAdd(cnt + b, hist[b]);
}

// 2. the starts of the bins in the pair buffers and the cursors of the moves
// (one CTA); the pieces of the bins with more than PIECE pairs.  A thread takes two
// neighbouring bins of each of four rows, so that its loads and stores are next to
// its neighbours' (eight in a row each: 33 us for 24576 bins, now 19).
constexpr int SCAN_NT = 1024, SCAN_ROWS = 4;
__global__ void __launch_bounds__(SCAN_NT) k_bwd_scan(const uint32_t* __restrict__ cnt, int n_bins,
                                                      const int2* __restrict__ map, unsigned long long* start,
                                                      unsigned long long* cur1, unsigned long long* cur2,
                                                      uint2* items, int32_t* n_items) {
    ws_chain();
    __shared__ long long wsum[SCAN_ROWS * SCAN_NT / 32 + 1];   // totals of a row's warps, then what is before them
    __shared__ uint2 split[SCAN_NT];   // (bin, first item) of the split bins of one step
    __shared__ int n_split, s_items;
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    if (t == 0) s_items = 0;
    long long run = 0;
    const int n_pad = (n_bins + 7) & ~7;   // (as the arrays; no pairs and no buckets beyond n_bins)
    for (int b0 = 0; b0 < n_bins; b0 += SCAN_ROWS * 2 * SCAN_NT) {
        uint2 c[SCAN_ROWS];
        int2 first[SCAN_ROWS];
        long long inc[SCAN_ROWS];
        bool big = false;
#pragma unroll
        for (int r = 0; r < SCAN_ROWS; ++r) {
            const int b = b0 + 2 * (r * SCAN_NT + t);
            c[r] = make_uint2(0, 0);
            first[r] = make_int2(-1, -1);
            if (b < n_pad) {
                c[r] = __ldg(reinterpret_cast<const uint2*>(cnt + b));
                const int4 m = __ldg(reinterpret_cast<const int4*>(map + b));
                first[r] = make_int2(m.y, m.w);
            }
            big |= c[r].x > (uint32_t)PIECE || c[r].y > (uint32_t)PIECE;
        }
#pragma unroll
        for (int r = 0; r < SCAN_ROWS; ++r) {
            inc[r] = ws_warp_incl_scan<long long>((long long)c[r].x + (long long)c[r].y);
            if (lane == 31) wsum[r * (SCAN_NT / 32) + w] = inc[r];
        }
        __syncthreads();
        if (w == 0) {   // (four totals a lane)
            static_assert(SCAN_ROWS * SCAN_NT / 32 == 128, "four totals a lane of one warp");
            long long v[4], sum = 0;
#pragma unroll
            for (int k = 0; k < 4; ++k) { v[k] = wsum[4 * lane + k]; sum += v[k]; }
            long long before = ws_warp_incl_scan<long long>(sum) - sum;
#pragma unroll
            for (int k = 0; k < 4; ++k) { wsum[4 * lane + k] = before; before += v[k]; }
            if (lane == 31) wsum[128] = before;
        }
        __syncthreads();
#pragma unroll
        for (int r = 0; r < SCAN_ROWS; ++r) {
            const int b = b0 + 2 * (r * SCAN_NT + t);
            if (b < n_pad) {
                const long long own = (long long)c[r].x + (long long)c[r].y;
                ulonglong2 q;
                q.x = (unsigned long long)(run + wsum[r * (SCAN_NT / 32) + w] + inc[r] - own);
                q.y = q.x + c[r].x;
                if (first[r].x >= 0) cur1[first[r].x] = q.x;   // (the first bin of a bucket of the first move)
                if (first[r].y >= 0) cur1[first[r].y] = q.y;
                *reinterpret_cast<ulonglong2*>(start + b) = q;
                *reinterpret_cast<ulonglong2*>(cur2 + b) = q;
            }
        }
        run += wsum[128];
        if (!__syncthreads_or(big)) continue;   // (also the end of this step's use of wsum)
#pragma unroll 1
        for (int k = 0; k < 2 * SCAN_ROWS; ++k) {
            const int b = b0 + 2 * ((k >> 1) * SCAN_NT + t) + (k & 1);
            const uint32_t ck = b < n_bins ? __ldg(cnt + b) : 0u;
            if (t == 0) n_split = 0;
            __syncthreads();
            if (ck > (uint32_t)PIECE)
                split[atomicAdd(&n_split, 1)] =
                    make_uint2((uint32_t)b, (uint32_t)atomicAdd(&s_items, (int)((ck + PIECE - 1) / PIECE)));
            __syncthreads();
            for (int i = t >> 5; i < n_split; i += SCAN_NT / 32) {
                const uint2 sp = split[i];
                const uint32_t np = (__ldg(cnt + sp.x) + PIECE - 1) / PIECE;
                for (uint32_t q = t & 31; q < np; q += 32) items[sp.y + q] = make_uint2(sp.x, q);
            }
            __syncthreads();
        }
    }
    __syncthreads();
    if (t == 0) { start[n_bins] = (unsigned long long)run; *n_items = s_items; }
}

// The slots whose sums are formed in global memory start from zero: those of split
// bins, and from the first to the last one that whole tiles add to (a warp per bin).
// (With whole bins there, segments of one cluster cleared and read 40 KB each: 2000 of
// 10000 elements 248 us, now 211.)
__global__ void __launch_bounds__(256) k_bwd_clear(const uint32_t* __restrict__ cnt,
                                                   const uint32_t* __restrict__ extra,
                                                   const uint32_t* __restrict__ xlo, const uint32_t* __restrict__ xhi,
                                                   int n_bins, const int2* __restrict__ map,
                                                   const LargeSeg* __restrict__ lsegs, unsigned long long* acc,
                                                   int32_t* gcnt) {
    ws_chain();
    const int lane = threadIdx.x & 31;
    // (eight lanes look at a bin each, the warp clears those that need it)
    const int nw = (int)gridDim.x * 8 * 8;
    for (int b0 = ((int)blockIdx.x * 8 + (int)(threadIdx.x >> 5)) * 8; b0 < n_bins; b0 += nw) {
        const int mine = b0 + lane;
        const bool need = lane < 8 && mine < n_bins && (cnt[mine] > PIECE || extra[mine] != 0);
        for (unsigned todo = __ballot_sync(0xffffffffu, need); todo; todo &= todo - 1) {
            const int b = b0 + __ffs((int)todo) - 1;
            const int lseg = map[b].x;
            const LargeSeg& ls = lsegs[lseg];
            const int64_t r0 = (int64_t)(b - ls.bb_pos) << WS_BWD_BIN_LOG2;
            const int64_t r1 = min(r0 + WS_BWD_BIN, ls.len), slot0 = ls.kpos + lseg;
            const bool split = cnt[b] > PIECE;
            const int64_t a = split ? r0 : r0 + WS_BWD_BIN - xlo[b], z = split ? r1 : r0 + xhi[b];
            for (int64_t r = a + lane; r < z; r += 32) {
                acc[2 * (slot0 + r)] = 0ull;
                acc[2 * (slot0 + r) + 1] = 0ull;
                gcnt[slot0 + r] = 0;
            }
        }
    }
}

// 3. moves the pairs into their buckets (FIRST) or, inside the buckets of a
// long segment, into their bins.  The pairs of one tile are grouped in shared
// memory (one atomic per pair ranks it), each run reserved with one global
// atomic and copied out by consecutive threads.
template <typename T>
struct BwdPartSmem {
    typename KeyOf<T>::K g[BTILE];
    int32_t id[BTILE];
    uint32_t cnt[WS_BWD_FAN];
    uint32_t first[WS_BWD_FAN];              // the run's start inside the tile
    unsigned long long base[WS_BWD_FAN];     // and its destination
    int wsum[PNT / 32];
    long long wlo[PNT / 32], whi[PNT / 32];
};

template <typename T, bool FIRST>
__global__ void __launch_bounds__(PNT, 2) k_bwd_part(const typename KeyOf<T>::K* __restrict__ g_in,
                                                     const int32_t* __restrict__ id_in,
                                                     typename KeyOf<T>::K* __restrict__ g_a, int32_t* __restrict__ id_a,
                                                     typename KeyOf<T>::K* __restrict__ g_b, int32_t* __restrict__ id_b,
                                                     const TileDesc* __restrict__ tiles, int n_tiles,
                                                     const LargeSeg* __restrict__ lsegs,
                                                     const unsigned long long* __restrict__ start,
                                                     unsigned long long* cursor, const int32_t* __restrict__ seg_emax,
                                                     unsigned long long* acc, int32_t* gcnt, T* mean,
                                                     int64_t n_pairs) {
    typedef KeyOf<T> KO;
    typedef typename KO::K K;
    static_assert(WS_BWD_FAN == PNT, "one bucket per thread");
    extern __shared__ __align__(16) unsigned char part_raw[];
    BwdPartSmem<T>& s = *reinterpret_cast<BwdPartSmem<T>*>(part_raw);
    ws_chain_wait();
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    struct Src { int64_t pos; int len; };
    auto source = [&](int tile) {
        Src r;
        const TileDesc& td = tiles[tile];
        if (FIRST) { r.pos = td.vpos; r.len = td.len; return r; }
        const LargeSeg& sg = lsegs[td.lseg];
        r.pos = 0;
        r.len = 0;
        if (sg.bb_fine == 0) return r;
        const int64_t p0 = (int64_t)start[sg.bb_pos] + (int64_t)td.tin * BTILE;
        const int64_t p1 = (int64_t)start[sg.bb_pos + sg.bb_n];
        r.pos = p0;
        r.len = (int)max((int64_t)0, min((int64_t)BTILE, p1 - p0));
        return r;
    };
    K gv[ITEMS];
    int32_t idv[ITEMS];
    auto load = [&](const Src& r) {
#pragma unroll
        for (int k = 0; k < ITEMS; ++k) {
            const int p = t + k * PNT;
            idv[k] = -1;
            if (p < r.len) {
                gv[k] = __ldg(g_in + r.pos + p);
                idv[k] = __ldg(id_in + r.pos + p);
            }
        }
    };
    int tile = blockIdx.x;
    if (tile >= n_tiles) return;
    Src cur = source(tile);
    load(cur);
    while (tile < n_tiles) {
        const int nxt = tile + (int)gridDim.x;
        const Src ns = nxt < n_tiles ? source(nxt) : Src{0, 0};
        const int lseg = tiles[tile].lseg;
        const LargeSeg& sg = lsegs[lseg];
        const int fl = sg.bb_fine, len = cur.len;
        bool skip = len == 0;
        if (FIRST) {
            const int id0 = __ldg(id_in + cur.pos);
            const int slen = (int)min(sg.len, (int64_t)INT32_MAX);
            bool same = true;
#pragma unroll
            for (int k = 0; k < ITEMS; ++k) {
                if (t + k * PNT < len) same &= idv[k] == id0;
                if (idv[k] >= slen) idv[k] = -1;
            }
            if (__syncthreads_and(same)) {
                // one cluster: the exact sum, once
                skip = true;
                if (id0 >= 0 && id0 < slen) {   // (uniform)
                    const int emax = seg_emax[lseg];
                    i128 sum = 0;
#pragma unroll
                    for (int k = 0; k < ITEMS; ++k)
                        if (t + k * PNT < len) sum += ws_bwd_fix<T>(ws_g_of_bits<T>(gv[k]), emax);
                    sum = ws_warp_reduce_i128(sum);
                    if (lane == 0) { s.wlo[w] = (long long)(uint64_t)sum; s.whi[w] = (long long)(uint64_t)((u128)sum >> 64); }
                    __syncthreads();
                    if (t == 0) {
                        i128 tot = 0;
                        for (int k = 0; k < PNT / 32; ++k)
                            tot += (i128)(((u128)(uint64_t)s.whi[k] << 64) | (u128)(uint64_t)s.wlo[k]);
                        const int64_t slot = sg.kpos + lseg + id0;
                        if (len == slen) mean[slot] = ws_bwd_mean<T>(tot, len, emax);
                        else {
                            ws_atomic_add_i128(acc + 2 * slot, tot);
                            atomicAdd(gcnt + slot, len);
                        }
                    }
                }
            }
        }
        if (skip) {   // (uniform)
            if (nxt < n_tiles) load(ns);
            __syncthreads();
            tile = nxt;
            cur = ns;
            continue;
        }
        // the tile's buckets: all of the segment's, or the bins of its first to last bucket
        const int sh = WS_BWD_BIN_LOG2 + (FIRST ? fl : 0);
        int base = 0, nbk = ((sg.bb_n - 1) >> fl) + 1;
        if (!FIRST) {
            base = ((__ldg(id_in + cur.pos) >> WS_BWD_BIN_LOG2) >> fl) << fl;
            const int hi = (((__ldg(id_in + cur.pos + len - 1) >> WS_BWD_BIN_LOG2) >> fl) + 1) << fl;
            nbk = max(min(sg.bb_n, hi) - base, 1);
        }
        K* go = FIRST && fl != 0 ? g_a : g_b;
        int32_t* io = FIRST && fl != 0 ? id_a : id_b;
        for (int r0 = 0; r0 < nbk; r0 += WS_BWD_FAN) {
            const uint32_t off = (uint32_t)(base + r0);
            __syncthreads();   // (the previous use of the shared memory is over)
            s.cnt[t] = 0;
            __syncthreads();
            uint32_t rk[ITEMS];
#pragma unroll
            for (int k = 0; k < ITEMS; ++k) {
                const uint32_t b = (uint32_t)(idv[k] >> sh) - off;   // (id -1: above every bucket, or refused below)
                rk[k] = 0;
                if (idv[k] >= 0 && b < WS_BWD_FAN) rk[k] = atomicAdd(&s.cnt[b], 1u);
            }
            __syncthreads();
            const uint32_t c = s.cnt[t];
            s.base[t] = c ? atomicAdd(cursor + (FIRST ? sg.bb_cpos : sg.bb_pos) + off + t, (unsigned long long)c) : 0ull;
            int total;
            s.first[t] = (uint32_t)ws_block_excl_scan<PNT, int>((int)c, s.wsum, &total);
            __syncthreads();
#pragma unroll
            for (int k = 0; k < ITEMS; ++k) {
                const uint32_t b = (uint32_t)(idv[k] >> sh) - off;
                if (idv[k] >= 0 && b < WS_BWD_FAN) {
                    const uint32_t j = s.first[b] + rk[k];
                    s.g[j] = gv[k];
                    s.id[j] = idv[k];
                }
            }
            __syncthreads();
            // (the registers are free: the next tile's loads overlap the copy)
            if (r0 + WS_BWD_FAN >= nbk) {
                if (nxt < n_tiles) load(ns);
                else ws_chain_go();
            }
#pragma unroll 4
            for (int j = t; j < total; j += PNT) {
                const int32_t id = s.id[j];
                const uint32_t b = (uint32_t)(id >> sh) - off;
                const int64_t pos = (int64_t)s.base[b] + (int64_t)((uint32_t)j - s.first[b]);
                if (pos < n_pairs) {   // (always)
                    go[pos] = s.g[j];
                    io[pos] = id;
                }
            }
        }
        tile = nxt;
        cur = ns;
    }
}

// 4. the sums of a bin's slots in shared memory, and its means.  CTA b takes
// bin b (and b + MAIN ..); the last EXTRA CTAs the pieces of the split ones.  Pairs are added in
// steps of CHUNK; with more than 4096 of them the limbs are normalised after
// every step (the top limb's carries go to the upper half of the counter, whose
// lower half holds at most PIECE).
struct BwdBinSmem {
    int limb[LIMBS][WS_BWD_BIN];
    int cnt[WS_BWD_BIN];
};

template <typename T>
__global__ void __launch_bounds__(ANT, 4) k_bwd_bins(const typename KeyOf<T>::K* __restrict__ g_b,
                                                     const int32_t* __restrict__ id_b,
                                                     const uint32_t* __restrict__ cnt,
                                                     const uint32_t* __restrict__ extra,
                                                     const uint32_t* __restrict__ xlo,
                                                     const uint32_t* __restrict__ xhi, int n_bins,
                                                     const int2* __restrict__ map, const LargeSeg* __restrict__ lsegs,
                                                     const unsigned long long* __restrict__ start,
                                                     const uint2* __restrict__ items,
                                                     const int32_t* __restrict__ n_items, uint32_t* arrive,
                                                     const int32_t* __restrict__ seg_emax, unsigned long long* acc,
                                                     int32_t* gcnt, T* mean) {
    typedef KeyOf<T> KO;
    typedef typename KO::K K;
    static_assert(PIECE < 32768, "the counter's lower half");
    extern __shared__ __align__(16) unsigned char bin_raw[];
    BwdBinSmem& s = *reinterpret_cast<BwdBinSmem*>(bin_raw);
    __shared__ int s_last;
    ws_chain();
    const int t = threadIdx.x, lane = t & 31;
    auto run = [&](int bin, int piece) {   // (piece -1: the whole bin)
        const int nbin = (int)cnt[bin];
        const bool more = extra[bin] != 0;
        if (nbin == 0 && !more) return;
        const int lseg = map[bin].x;
        const LargeSeg& ls = lsegs[lseg];
        const int r0 = (bin - ls.bb_pos) << WS_BWD_BIN_LOG2;
        const int nr = (int)min((int64_t)WS_BWD_BIN, ls.len - r0);
        const int64_t slot0 = ls.kpos + lseg + r0;
        const int emax = seg_emax[lseg];
        // (what whole tiles added, and to which slots)
        const int xa = more ? WS_BWD_BIN - (int)xlo[bin] : 0, xz = more ? (int)xhi[bin] : 0;
        auto tiles_cnt = [&](int r) { return gcnt[slot0 + r]; };
        auto tiles_sum = [&](int r) { return (i128)(((u128)acc[2 * (slot0 + r) + 1] << 64) | (u128)acc[2 * (slot0 + r)]); };
        if (nbin == 0) {   // (no pairs: only these)
            for (int r = xa + t; r < xz; r += ANT) {
                const int c = tiles_cnt(r);
                if (c) mean[slot0 + r] = ws_bwd_mean<T>(tiles_sum(r), c, emax);
            }
            return;
        }
        const int64_t p0 = (int64_t)start[bin] + (piece > 0 ? (int64_t)piece * PIECE : 0);
        const int n = piece < 0 ? nbin : min(PIECE, nbin - piece * PIECE);
        __syncthreads();   // (the previous use of the shared memory is over)
        for (int i = t; i < (int)(sizeof(BwdBinSmem) / sizeof(int4)); i += ANT)
            reinterpret_cast<int4*>(&s)[i] = make_int4(0, 0, 0, 0);
        __syncthreads();
        for (int c0 = 0; c0 < n; c0 += CHUNK) {
            K gv[8];
            int idv[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                if (c0 + k * ANT >= n) break;   // (uniform)
                const int64_t j = p0 + min(c0 + k * ANT + t, n - 1);
                gv[k] = __ldg(g_b + j);
                idv[k] = __ldg(id_b + j);
            }
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                if (c0 + k * ANT >= n) break;
                const bool in = c0 + k * ANT + t < n;
                const int r = idv[k] & (WS_BWD_BIN - 1);
                const T gk = ws_g_of_bits<T>(gv[k]);
                const unsigned crowd = ws_crowd(r, in);
                if ((crowd >> lane) & 1u) {
                    const i128 sum = ws_group_sum_i96(crowd, ws_bwd_fix<T>(gk, emax));
                    if (lane == __ffs((int)crowd) - 1) {
#pragma unroll
                        for (int l = 0; l < LIMBS - 1; ++l)
                            atomicAdd(&s.limb[l][r], (int)((uint32_t)(uint64_t)((u128)sum >> (l * LIMB_BITS)) & LIMB_MASK));
                        atomicAdd(&s.limb[LIMBS - 1][r], (int)(sum >> ((LIMBS - 1) * LIMB_BITS)));
                        atomicAdd(&s.cnt[r], __popc(crowd));
                    }
                } else if (in) {
                    ws_limb_add<T, WS_BWD_BIN>(&s.limb[0][r], gk, emax);
                    atomicAdd(&s.cnt[r], 1);
                }
            }
            __syncthreads();
            if (n > 4096) {
                for (int r = t; r < nr; r += ANT) {
                    int carry = 0;
#pragma unroll
                    for (int l = 0; l < LIMBS; ++l) {
                        const int v = s.limb[l][r];
                        // (v + carry stays below 2^31: 2049 values of 19 bits and a carry of 12)
                        const int x = v + carry;
                        carry = x >> LIMB_BITS;
                        s.limb[l][r] = x & (int)LIMB_MASK;
                    }
                    s.cnt[r] += carry * 65536;
                }
                __syncthreads();
            }
        }
        // the count and the sum of slot r
        auto slot_cnt = [&](int r) { return s.cnt[r] & 0xffff; };
        auto slot_sum = [&](int r) {
            return ws_limb_sum<WS_BWD_BIN>(&s.limb[0][r]) + ((i128)(s.cnt[r] >> 16) << (LIMBS * LIMB_BITS));
        };
        if (piece < 0) {
            for (int r = t; r < nr; r += ANT) {
                int c = slot_cnt(r);
                i128 S = slot_sum(r);
                if (r >= xa && r < xz) {
                    c += tiles_cnt(r);
                    S += tiles_sum(r);
                }
                if (c) mean[slot0 + r] = ws_bwd_mean<T>(S, c, emax);
            }
            return;
        }
        for (int r = t; r < nr; r += ANT) {
            const int c = slot_cnt(r);
            if (c) {
                ws_atomic_add_i128(acc + 2 * (slot0 + r), slot_sum(r));
                atomicAdd(gcnt + slot0 + r, c);
            }
        }
        // the piece that comes last forms the means
        __threadfence();
        __syncthreads();
        if (t == 0) s_last = atomicAdd(arrive + bin, 1u) == (uint32_t)((nbin + PIECE - 1) / PIECE) - 1u;
        __syncthreads();
        if (!s_last) return;
        __threadfence();
        for (int r = t; r < nr; r += ANT) {
            const int c = __ldcg(gcnt + slot0 + r);
            if (c == 0) continue;
            const i128 S = (i128)(((u128)__ldcg(acc + 2 * (slot0 + r) + 1) << 64) | (u128)__ldcg(acc + 2 * (slot0 + r)));
            mean[slot0 + r] = ws_bwd_mean<T>(S, c, emax);
        }
    };
    const int n_main = (int)gridDim.x - EXTRA;
    if ((int)blockIdx.x < n_main) {
        for (int b = blockIdx.x; b < n_bins; b += n_main)
            if (cnt[b] <= PIECE) run(b, -1);
        return;
    }
    const int ni = *n_items;
    for (int i = (int)blockIdx.x - n_main; i < ni; i += EXTRA) {
        const uint2 it = items[i];
        run((int)it.x, (int)it.y);
    }
}

// 5. every element takes its cluster's mean
template <typename T>
__global__ void __launch_bounds__(PNT) k_bwd_apply(const int32_t* __restrict__ ids, const TileDesc* __restrict__ tiles,
                                                   const LargeSeg* __restrict__ lsegs, const T* __restrict__ mean,
                                                   T* gin) {
    ws_chain();
    const TileDesc td = tiles[blockIdx.x];
    const LargeSeg& ls = lsegs[td.lseg];
    const int64_t slot0 = ls.kpos + td.lseg, slen = ls.len;
    int idv[ITEMS];
    T v[ITEMS];
#pragma unroll
    for (int k = 0; k < ITEMS; ++k) {
        const int i = threadIdx.x + k * PNT;
        idv[k] = i < td.len ? __ldg(ids + td.vpos + i) : -1;
        if ((int64_t)idv[k] >= slen) idv[k] = -1;
    }
#pragma unroll
    for (int k = 0; k < ITEMS; ++k)
        if (idv[k] >= 0) v[k] = __ldg(mean + slot0 + idv[k]);
#pragma unroll
    for (int k = 0; k < ITEMS; ++k)
        if (idv[k] >= 0) gin[td.vpos + threadIdx.x + k * PNT] = v[k];
}

// One-CTA segments: the same limbs, one CTA per segment.  Bound by the adds and
// the conversions; 12.6M elements in rows of 3072: 482 us with 64-bit atomics
// behind a warp match, 90 with the limbs.
template <typename T, int NT, int CAP>
__global__ void __launch_bounds__(NT, 2) k_small_backward(const T* __restrict__ g, const int32_t* __restrict__ ids,
                                                          const int64_t* __restrict__ offsets,
                                                          const int32_t* __restrict__ seg_list, T* gin,
                                                          uint32_t* status) {
    typedef KeyOf<T> KO;
    constexpr int PER = CAP / NT;
    static_assert(CAP % NT == 0, "whole elements per thread");
    static_assert((long long)CAP * ((1 << LIMB_BITS) - 1) < (1ll << 31), "no limb overflows");
    extern __shared__ __align__(16) unsigned char smem_raw[];
    int* limb = reinterpret_cast<int*>(smem_raw);   // [LIMBS][CAP]
    int* cnt = limb + LIMBS * CAP;                  // [CAP]
    __shared__ int s_emax;
    const int seg = seg_list[blockIdx.x];
    const int64_t a0 = offsets[seg];
    const int n = (int)(offsets[seg + 1] - a0);
    if (n <= 0) return;
    if (n > CAP) { if (threadIdx.x == 0) ws_flag(status, WS_STATUS_INTERNAL); return; }
    const int t = threadIdx.x, lane = t & 31;
    if (t == 0) s_emax = 0;
    T gv[PER];
    int idv[PER];
#pragma unroll
    for (int k = 0; k < PER; ++k) {
        const int i = t + k * NT;
        gv[k] = i < n ? __ldg(g + a0 + i) : (T)0;
        idv[k] = i < n ? __ldg(ids + a0 + i) : -1;
    }
    for (int i = t; i < (n + 3) / 4; i += NT) {
#pragma unroll
        for (int l = 0; l <= LIMBS; ++l) reinterpret_cast<int4*>(limb + l * CAP)[i] = make_int4(0, 0, 0, 0);
    }
    int e = 0;
    bool bad = false;
#pragma unroll
    for (int k = 0; k < PER; ++k) {
        e = max(e, ws_g_exp(gv[k]));
        if (idv[k] < 0 || idv[k] >= n) { bad |= t + k * NT < n; idv[k] = -1; }
    }
    if (bad) ws_flag(status, WS_STATUS_INTERNAL);
    e = __reduce_max_sync(0xffffffffu, e);
    __syncthreads();
    if (lane == 0) atomicMax(&s_emax, e);
    __syncthreads();
    const int emax = s_emax;
#pragma unroll
    for (int k = 0; k < PER; ++k) {
        const int id = idv[k];
        if (id < 0) continue;
        ws_limb_add<T, CAP>(limb + id, gv[k], emax);
        atomicAdd(cnt + id, 1);
    }
    __syncthreads();
    // the mean of slot r replaces its low limbs (only this thread touches slot r)
    for (int r = t; r < n; r += NT) {
        const int c = cnt[r];
        if (c == 0) continue;
        const i128 S = ws_limb_sum<CAP>(limb + r);
        const T mean = ws_bwd_mean<T>(S, c, emax);
        if (sizeof(T) == 4) limb[r] = __float_as_int((float)mean);
        else {
            const long long q = __double_as_longlong((double)mean);
            limb[r] = (int)(uint32_t)(uint64_t)q;
            limb[CAP + r] = (int)(uint32_t)((uint64_t)q >> 32);
        }
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < PER; ++k) {
        const int id = idv[k];
        if (id < 0) continue;
        T v;
        if (sizeof(T) == 4) v = (T)__int_as_float(limb[id]);
        else v = (T)__longlong_as_double((long long)(((uint64_t)(uint32_t)limb[CAP + id] << 32) | (uint32_t)limb[id]));
        gin[a0 + t + k * NT] = v;
    }
}

}  // namespace

template <typename T>
cudaError_t ws_large_backward(const LargeWork<T>& W, const T* g, const int32_t* ids, T* gin, uint32_t* status,
                              cudaStream_t st) {
    if (W.n_lseg == 0) return cudaSuccess;
    typedef typename KeyOf<T>::K K;
    cudaError_t e = cudaMemsetAsync(W.bwd.emax, 0, W.bwd.zero_bytes, st);
    if (e) return e;
    const BwdWork& B = W.bwd;
    const int nt = W.n_sort_tiles;
    // the pairs borrow buffers of the forward (n_keys entries each)
    K *g_a = W.keys_a, *g_b = W.keys_b;
    int32_t *id_a = reinterpret_cast<int32_t*>(W.cval), *id_b = reinterpret_cast<int32_t*>(W.bins);
    const int n_hist = B.n_bins <= HIST_MAX ? B.n_bins : 0;
    const size_t hsm = sizeof(uint32_t) * n_hist, psm = sizeof(BwdPartSmem<T>), bsm = sizeof(BwdBinSmem);
    if ((e = cudaFuncSetAttribute(k_bwd_prep<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, 4 * HIST_MAX)) ||
        (e = cudaFuncSetAttribute(k_bwd_part<T, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)psm)) ||
        (e = cudaFuncSetAttribute(k_bwd_part<T, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)psm)) ||
        (e = cudaFuncSetAttribute(k_bwd_bins<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bsm)))
        return e;
    const int grid = std::min(nt, 2 * 152);
    WS_LAUNCH(W.prof, WSK_BWD, st,
              (k_bwd_prep<T><<<std::min(nt, 3 * 152), PNT, hsm, st>>>(g, ids, W.sort_tiles, nt, W.lsegs, n_hist, B.emax, B.cnt, B.extra,
                                                     B.xlo, B.xhi, status)));
    WS_LAUNCH(W.prof, WSK_BWD, st,
              ws_launch_chain(k_bwd_scan, 1, SCAN_NT, 0, st, B.cnt, B.n_bins, B.map, B.start, B.cur1, B.cur2, B.items,
                              B.n_items));
    WS_LAUNCH(W.prof, WSK_BWD, st,
              ws_launch_chain(k_bwd_clear, std::min((B.n_bins + 63) / 64, 8 * 152), 256, 0, st, B.cnt, B.extra, B.xlo, B.xhi,
                              B.n_bins, B.map, W.lsegs, W.bacc, W.bcnt));
    WS_LAUNCH(W.prof, WSK_BWD, st,
              ws_launch_chain(k_bwd_part<T, true>, grid, PNT, psm, st, reinterpret_cast<const K*>(g), ids, g_a, id_a,
                              g_b, id_b, W.sort_tiles, nt, W.lsegs, B.start, B.cur1, B.emax, W.bacc, W.bcnt,
                              W.bsum, W.n_keys));
    if (B.two_level)
        WS_LAUNCH(W.prof, WSK_BWD, st,
                  ws_launch_chain(k_bwd_part<T, false>, grid, PNT, psm, st, g_a, id_a, g_a, id_a, g_b, id_b,
                                  W.sort_tiles, nt, W.lsegs, B.start, B.cur2, B.emax, W.bacc, W.bcnt, W.bsum,
                                  W.n_keys));
    WS_LAUNCH(W.prof, WSK_BWD, st,
              ws_launch_chain(k_bwd_bins<T>, std::min(B.n_bins, MAIN) + EXTRA, ANT, bsm, st, g_b, id_b, B.cnt, B.extra, B.xlo, B.xhi,
                              B.n_bins, B.map, W.lsegs, B.start, B.items, B.n_items, B.arrive, B.emax, W.bacc, W.bcnt, W.bsum));
    // (a gather that lives off the caches: a plain launch)
    WS_LAUNCH(W.prof, WSK_BWD, st,
              ws_launch_if(nt <= 2 * 152, k_bwd_apply<T>, nt, PNT, 0, st, ids, W.sort_tiles, W.lsegs, W.bsum, gin));
    return cudaGetLastError();
}

template <typename T>
cudaError_t ws_launch_small_backward(const T* g, const int32_t* ids, const int64_t* offsets, const int32_t* seg_list,
                                     int n_list, T* gin, uint32_t* status, cudaStream_t st, WsProf* prof) {
    constexpr int NT = 512;
    constexpr int CAP = SmallCfg<T>::CAP;
    if (n_list <= 0) return cudaSuccess;
    const size_t smem = (size_t)CAP * (LIMBS + 1) * sizeof(int);
    auto k = k_small_backward<T, NT, CAP>;
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e) return e;
    WS_LAUNCH(prof, WSK_BWD, st, (k<<<n_list, NT, smem, st>>>(g, ids, offsets, seg_list, gin, status)));
    return cudaGetLastError();
}

template cudaError_t ws_large_backward<float>(const LargeWork<float>&, const float*, const int32_t*, float*,
                                              uint32_t*, cudaStream_t);
template cudaError_t ws_large_backward<double>(const LargeWork<double>&, const double*, const int32_t*, double*,
                                               uint32_t*, cudaStream_t);
template cudaError_t ws_launch_small_backward<float>(const float*, const int32_t*, const int64_t*, const int32_t*,
                                                     int, float*, uint32_t*, cudaStream_t, WsProf*);
template cudaError_t ws_launch_small_backward<double>(const double*, const int32_t*, const int64_t*,
                                                      const int32_t*, int, double*, uint32_t*, cudaStream_t,
                                                      WsProf*);
