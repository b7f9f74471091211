// ws_sort.cu -- sort of the keys of the large segments (the pre-processing
// every prox algorithm of Sec. 4 assumes), as a distribution sort.
//
// Only keys move: because equal weights always share a cluster, the result of
// the prox never depends on the order of ties, so no index payload is sorted,
// no pass has to be stable, and a pass needs no look-back over earlier tiles:
//   k_sort_plan   samples every segment, fits a monotone map key -> bin (a
//                 piecewise linear image of the sampled distribution, so that
//                 bins come out about equal whatever the distribution), counts
//                 every key's bin, and turns the counts into bin starts;
//   k_part        moves the keys into their bins: one pass for segments of at
//                 most WS_ONE_LEVEL bins, otherwise a pass into buckets of
//                 2^fine_log2 bins and a second one inside the buckets.  A
//                 tile ranks its keys with one shared-memory atomic each and
//                 reserves its runs with one global atomic per bucket;
//   k_bin_sort    sorts every bin in one CTA;
//   k_oversize    sorts the bins that do not fit one CTA (heavy ties, or a
//                 distribution that the map does not resolve), returns at once
//                 when there are none.
// The map only decides how even the bins are: it is monotone in the key by
// construction, so the result is the sorted sequence for any input.
//
// Measured against 8-bit LSD passes with decoupled look-back (a histogram and
// four passes of 0.322 ms at 2^26 FP32 keys, eight passes for FP64; 0.245 of
// HBM, bound by the stable in-warp ranking), us:
//   FP32 2^26    1394 -> 882 (plan 150, partition 2 x 217, bins 293, oversize 6)
//   FP32 2^24     398 -> 271 (68, 2 x 58, 82, 6)
//   FP64 2^22     319 -> 147 (53, 2 x 23, 41, 6)
//   1024 FP32 segments of 16 .. 2^20 elements (9.7e7 keys)   2085 -> 1310
// without the records of the way back; with them 2^26 980 (2 x 249, bins 334).
// The partition is bound by shared-memory wavefronts (17 per 32 keys: the
// counters, the staging and the copy out; 0.7 of the pipe), the bin sort by
// issue (0.65) and the same pipe, the plan by the read of the values (0.104 of
// its 0.150 ms) and four barriers.
#include <algorithm>
#include <type_traits>

#include "ws_kernels.cuh"

namespace {

constexpr int PLAN_NT = 1024;
constexpr int PLAN_SMP = 8;   // samples per lane of a segment of one tile
// Up to this many segments of one tile are counted by the whole CTA one after the
// other, more by a warp each (15 us for 6144 elements).
constexpr int PLAN_ONE = 8;
static_assert(WS_SORT_TILE <= 3 * WS_BIN_MEAN, "such a segment has at most three bins");
constexpr int OVER_NT = WS_SORT_NT;

__device__ __forceinline__ uint32_t ld_acquire_u32(const uint32_t* p) {
    uint32_t v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// Barrier over a cooperative grid: arrivals are counted in *ctr (cleared
// before the launch).  A wait that gives up sets the timeout status and the
// abort word, and sync() is false then, for the whole CTA: what the other CTAs
// were to write before the barrier may be missing.  The plan kernel goes on
// without waiting (it indexes with nothing from another CTA but what it clamps);
// the oversize kernel leaves (it indexes with other CTAs' tile numbers, which
// may be an earlier call's).
struct GridBarrier {
    uint32_t* ctr;
    uint32_t* abort;
    uint32_t* status;
    uint64_t limit;
    uint32_t target;
    bool dead;   // (thread 0)
    __device__ __forceinline__ bool sync() {
        __syncthreads();
        if (threadIdx.x == 0) {
            target += gridDim.x;
            __threadfence();
            atomicAdd(ctr, 1u);
            uint64_t it = 0;
            while (!dead && (int32_t)(ld_acquire_u32(ctr) - target) < 0) {
                if (++it > limit) {
                    dead = true;
                    atomicExch(abort, 1u);
                    ws_flag(status, WS_STATUS_TIMEOUT);
                    break;
                }
                ws_backoff((int)min(it, (uint64_t)1 << 20));
            }
            __threadfence();
        }
        return !__syncthreads_or(dead);   // (dead: thread 0's, false elsewhere)
    }
};

// ---------------------------------------------------------------------------
// The map of a segment.  The sampled key range is cut into ncell cells of
// equal width, a cell with many samples into 2^bits equal parts (so that a
// part holds about the same number of samples wherever there are enough of
// them, and the density changes little inside one).  Knot i is the expected
// number of bins filled by the keys below part i; inside a part the map is
// linear in the key, with a slope rounded down by 2^-20.  Every step rounds
// monotonically, so the image of a part never passes the next knot and the map
// is monotone over the whole key range.  Keys above the sampled range go to
// the last bin, keys below it to the first.
// ---------------------------------------------------------------------------
struct MapTab {
    uint32_t split[WS_CELLS + 1];       // first part | width of a part << 16 (log2; the last entry: above the range)
    float2 knots[2 * WS_CELLS + 1];     // map value at the start of the part, its slope
};

// FP64 keys as the map sees them: magnitudes below m (the binade of the
// smallest sampled one) count as m, and the gap between -m and m closes.  The
// key range of values of both signs spans 2 x 1023 binades, nearly all of them
// between -m and m and empty; cells cut from all of it were two or four binades
// wide, their parts too coarse at the ends of a distribution, and bins overflowed
// (1 to 4 of them cost the oversize kernel's 115 us and 60 us on the way back:
// 700001 N(0, 1) weights 392 us with them, 222 without).  Monotone in the key.
template <typename T>
__device__ __forceinline__ typename KeyOf<T>::K squeeze(typename KeyOf<T>::K k, uint64_t m) {
    typedef typename KeyOf<T>::K K;
    if (sizeof(K) == 4) return k;   // (512 binades of keys: cells of half a binade)
    const K z = (K)1 << (KeyOf<T>::BITS - 1);   // the key of +0
    return k >= z ? z + (max(k - z, (K)m) - (K)m) : z - 1 - (max(z - 1 - k, (K)m) - (K)m);
}

template <typename T>
struct KeyMap {
    typedef typename KeyOf<T>::K K;
    K kmin;
    uint64_t mag;
    int shift;
    uint32_t ncell, last;
    __device__ __forceinline__ void init(const SortHdr& h, int ncell_, int nbins) {
        kmin = (K)h.kmin;
        mag = h.mag;
        shift = h.shift;
        ncell = (uint32_t)ncell_;
        last = (uint32_t)(nbins - 1);
    }
    // position inside a part of width 2^s2, at most 24 bits of it
    __device__ __forceinline__ static uint32_t low(K d, int s2) {
        const K x = d & (((K)1 << s2) - 1);
        return (uint32_t)(sizeof(K) == 4 ? x : x >> max(s2 - 24, 0));
    }
    // slope of a part of width 2^s2 that covers db bins
    __device__ __forceinline__ static float slope(float db, int s2) {
        return ldexpf(db * (1.0f - 1.0f / 1048576.0f), -(sizeof(K) == 4 ? s2 : min(s2, 24)));
    }
    __device__ __forceinline__ uint32_t bin(K key, const MapTab& m) const {
        const K k = squeeze<T>(key, mag);
        const K d = max(k, kmin) - kmin;
        const uint32_t e = m.split[(uint32_t)min(d >> shift, (K)ncell)];
        const int s2 = (int)(e >> 16);
        const K in = d & (((K)1 << shift) - 1);
        const uint32_t i = min((e & 0xffffu) + (uint32_t)(in >> s2), 2u * WS_CELLS);
        const float2 kn = m.knots[i];
        return min(__float2uint_rz(fmaf((float)low(d, s2), kn.y, kn.x)), last);   // (below 0: bin 0)
    }
};

// Sampled element j of m = 2^mlog of a tile: a pair of neighbours (one sector)
// at a pseudo-random place of every (m / 2)-th of the tile; all elements of a
// tile of at most m.
__device__ __forceinline__ int sample_pos(int tile, int j, int len, int mlog) {
    if (len <= (1 << mlog)) return j;
    const uint32_t q = (uint32_t)j >> 1;
    uint32_t h = (uint32_t)tile * 0x9E3779B9u + q * 0x85EBCA6Bu;
    h ^= h >> 15; h *= 0x2C1B3C6Du; h ^= h >> 13;
    return min((int)((q * (uint32_t)len + __umulhi(h, (uint32_t)len)) >> (mlog - 1)) + (j & 1), len - 1);
}

// ---------------------------------------------------------------------------
// Plan: sample, map, bin counts, bin starts.  A cooperative grid with one
// barrier between the phases.  Bound by the read of the values (the count)
// and, for short segments, by the barriers (about 2 us each).
// ---------------------------------------------------------------------------
struct PlanSmem {
    unsigned long long hi, lo, mag;
    int emin;
    int map;   // the CTA has tiles of segments with a map
    int n_one;   // segments of one tile that the CTA counts together
    struct { unsigned long long s1, s2; int tile, c1, c2, emin; } one[PLAN_ONE];
    int wsum[PLAN_NT / 32];
};

// Segments of one tile (S.n_one of the CTA's tiles): their bins start at quantiles
// of a sample, which a warp finds, and the elements are counted against these.  No
// other CTA needs any of it in the plan, so that it stands where the CTA maps the
// elements of its longer segments.  Out of line: inlined it cost the plans of longer
// segments 2 us (instruction fetches).  true: a weight that is not finite.
template <typename T, typename B>
__device__ __noinline__ bool plan_one(PlanSmem& S, const T* __restrict__ values, const TileDesc* __restrict__ tiles, int t0,
                                      int t1, const LargeSeg* __restrict__ lsegs, B* bins, uint32_t* bin_cnt,
                                      uint32_t* bin_start, uint32_t* cur1, int32_t* seg_emin) {
    typedef KeyOf<T> KO;
    typedef typename KO::K K;
    const int t = threadIdx.x, lane = t & 31, w = t >> 5, n_one = S.n_one;
    const bool cta = n_one <= PLAN_ONE;   // (else a warp for each)
    bool bad = false;
    auto split = [&](const TileDesc& td, const LargeSeg& sg, int tile, K& s1, K& s2) {
        const int nb = sg.nbins;
        s1 = s2 = ~(K)0;   // the bins after the first start at these keys
        if (nb == 1) return;
        const int m = 1 << sg.samp_log2;
        K smp[PLAN_SMP];
#pragma unroll
        for (int q = 0; q < PLAN_SMP; ++q) {
            const int j = lane + 32 * q;
            smp[q] = j < m ? KO::to_key(__ldg(values + td.vpos + sample_pos(tile, j, td.len, sg.samp_log2))) : ~(K)0;
        }
        // the samples of rank m / nb and 2 m / nb, bit by bit
        const int r1 = m / nb, r2 = nb > 2 ? 2 * m / nb : m;
        s1 = s2 = 0;
#pragma unroll 1
        for (K bit = (K)1 << (KO::BITS - 1); bit != 0; bit >>= 1) {
            uint32_t c = 0;   // samples below s1 | bit, and below s2 | bit
#pragma unroll
            for (int q = 0; q < PLAN_SMP; ++q) c += (smp[q] < (s1 | bit) ? 1u : 0u) + (smp[q] < (s2 | bit) ? 0x10000u : 0u);
            c = __reduce_add_sync(WS_FULL_MASK, c);
            if ((int)(c & 0xffffu) <= r1) s1 |= bit;
            if ((int)(c >> 16) <= r2) s2 |= bit;
        }
    };
    auto done = [&](const TileDesc& td, const LargeSeg& sg, int c1, int c2, int emin) {   // (one thread)
        seg_emin[td.lseg] = emin;
        const int at[4] = {0, td.len - c1, td.len - c2, td.len}, nb = sg.nbins;
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            if (q >= nb) break;
            const int end = q + 1 == nb ? td.len : at[q + 1];
            bin_cnt[sg.bin_pos + q] = (uint32_t)(end - at[q]);
            bin_start[sg.bin_pos + q] = (uint32_t)at[q];
            cur1[sg.coarse_pos + q] = (uint32_t)at[q];
        }
    };
    if (cta) {
        if (w < n_one) {
            const int tile = S.one[w].tile;
            const TileDesc td = tiles[tile];
            K s1, s2;
            split(td, lsegs[td.lseg], tile, s1, s2);
            if (lane == 0) {
                S.one[w].s1 = s1;
                S.one[w].s2 = s2;
                S.one[w].c1 = S.one[w].c2 = 0;
                S.one[w].emin = 0x7fffffff;
            }
        }
        __syncthreads();
    }
    const int i0 = cta ? t : lane, step = cta ? PLAN_NT : 32;
    for (int q = cta ? 0 : w; q < (cta ? n_one : t1 - t0); q += cta ? 1 : PLAN_NT / 32) {
        const int tile = cta ? S.one[q].tile : t0 + q;
        const TileDesc td = tiles[tile];
        const LargeSeg& sg = lsegs[td.lseg];
        if (sg.sort_count != 1) continue;
        const int nb = sg.nbins, len = td.len;
        K s1, s2;
        if (cta) { s1 = (K)S.one[q].s1; s2 = (K)S.one[q].s2; }
        else split(td, sg, tile, s1, s2);
        const T* src = values + td.vpos;
        B* bo = bins + td.kpos;
        K amax = 0, amin = ~(K)0;   // (as in phase 4)
        int c1 = 0, c2 = 0;         // keys from s1 on, and from s2 on
        for (int i = i0; i - lane < len; i += step * 8) {
            T v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) v[u] = __ldg(src + min(i + step * u, len - 1));
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const bool in = i + step * u < len;
                const K mag = (K)KO::bits(v[u]) & (~(K)0 >> 1), k = KO::to_key(v[u]);
                amax = max(amax, mag);
                amin = min(amin, mag - 1);
                const int b1 = nb > 1 && k >= s1, b2 = nb > 2 && k >= s2;
                c1 += in && b1;
                c2 += in && b2;
                if (in) bo[i + step * u] = (B)(b1 + b2);
            }
        }
        bad |= (amax >> KO::MANT) >= (K)KO::EXPMASK;
        int emin = amin != ~(K)0 ? max((int)((amin + 1) >> KO::MANT), 1) : 0x7fffffff;
        emin = __reduce_min_sync(WS_FULL_MASK, emin);
        c1 = __reduce_add_sync(WS_FULL_MASK, c1);
        c2 = __reduce_add_sync(WS_FULL_MASK, c2);
        if (lane == 0) {
            if (cta) { atomicAdd(&S.one[q].c1, c1); atomicAdd(&S.one[q].c2, c2); atomicMin(&S.one[q].emin, emin); }
            else done(td, sg, c1, c2, emin);
        }
    }
    if (cta) {
        __syncthreads();
        if (t < n_one) {
            const TileDesc td = tiles[S.one[t].tile];
            done(td, lsegs[td.lseg], S.one[t].c1, S.one[t].c2, S.one[t].emin);
        }
    }
    return bad;
}

template <typename T, typename B>
__global__ void __launch_bounds__(PLAN_NT, 1) k_sort_plan(const T* __restrict__ values,
                                                          const TileDesc* __restrict__ tiles, int n_tiles,
                                                          const LargeSeg* __restrict__ lsegs, int n_lseg,
                                                          SortCtl* ctl, unsigned long long* seg_hi,
                                                          unsigned long long* seg_lo, uint32_t* seg_en,
                                                          uint32_t* cells, uint32_t* bin_cnt, B* bins,
                                                          uint32_t* bin_start, uint32_t* cur1, uint32_t* cur2,
                                                          int32_t* seg_emin, int max_bins, int hist_cap, int samp_max,
                                                          uint64_t spin_limit, uint32_t* status) {
    typedef KeyOf<T> KO;
    typedef typename KO::K K;
    __shared__ PlanSmem S;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    MapTab& tab = *reinterpret_cast<MapTab*>(smem_raw);
    uint32_t* hist = reinterpret_cast<uint32_t*>(smem_raw + sizeof(MapTab));      // [hist_cap]
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    GridBarrier bar{&ctl->bar, &ctl->abort, status, spin_limit, 0u, false};
    // this CTA's tiles, contiguous
    const int t0 = (int)((int64_t)n_tiles * blockIdx.x / gridDim.x);
    const int t1 = (int)((int64_t)n_tiles * (blockIdx.x + 1) / gridDim.x);
    const int seg0 = t0 < t1 ? tiles[t0].lseg : -1;
    // the CTA's sampled keys stay in the (later) histogram's shared memory if they fit
    K* cache = reinterpret_cast<K*>(hist);
    const bool cached = ((size_t)(t1 - t0) << samp_max) * sizeof(K) <= (size_t)hist_cap * sizeof(uint32_t);

    // 1. range of the sampled keys (one warp per tile; the CTA's first segment
    // is combined in shared memory)
    if (t == 0) { S.hi = 0; S.lo = 0; S.mag = 0; S.map = 0; S.n_one = 0; }
    __syncthreads();
    bool bad = false;
    for (int tile = t0 + w; tile < t1; tile += PLAN_NT / 32) {
        const TileDesc td = tiles[tile];
        const LargeSeg& sg = lsegs[td.lseg];
        if (sg.sort_count == 1) {   // no map: plan_one below
            if (lane == 0) {
                const int q = atomicAdd(&S.n_one, 1);
                if (q < PLAN_ONE) S.one[q].tile = tile;
            }
            continue;
        }
        if (lane == 0) S.map = 1;
        const int ml = sg.samp_log2;
        const int m = min(td.len, 1 << ml);
        K hi = 0, lo = 0, mg = 0;   // (lo, mg: complements, so that 0 is neutral)
        K* keep = cache + ((size_t)(tile - t0) << samp_max);
#pragma unroll 4
        for (int j = lane; j < m; j += 32) {
            const K k = KO::to_key(__ldg(values + td.vpos + sample_pos(tile, j, td.len, ml)));
            if (cached) keep[j] = k;
            hi = max(hi, k);
            lo = max(lo, (K)~k);
            if (sizeof(K) == 8) {
                const K z = (K)1 << (KO::BITS - 1), a = k >= z ? k - z : z - 1 - k;
                if (a != 0) mg = max(mg, (K)~a);
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            hi = max(hi, ws_shfl_xor_k(hi, o));
            lo = max(lo, ws_shfl_xor_k(lo, o));
            if (sizeof(K) == 8) mg = max(mg, ws_shfl_xor_k(mg, o));
        }
        if (lane == 0) {
            if (td.lseg == seg0) {
                atomicMax(&S.hi, (unsigned long long)hi);
                atomicMax(&S.lo, (unsigned long long)lo);
                if (sizeof(K) == 8) atomicMax(&S.mag, (unsigned long long)mg);
            } else {
                atomicMax(seg_hi + td.lseg, (unsigned long long)hi);
                atomicMax(seg_lo + td.lseg, (unsigned long long)lo);
                if (sizeof(K) == 8) atomicMax(seg_lo + n_lseg + td.lseg, (unsigned long long)mg);
            }
        }
    }
    __syncthreads();
    if (t == 0 && S.map) {   // (S.hi, S.lo: 0 if the first segment has one bin)
        atomicMax(seg_hi + seg0, S.hi);
        atomicMax(seg_lo + seg0, S.lo);
        if (sizeof(K) == 8) atomicMax(seg_lo + n_lseg + seg0, S.mag);
    }
    const int tm = S.map ? t1 : t0;   // (uniform; the tile loops below are for segments with a map)
    bar.sync();

    // header of a segment from its sampled range
    auto header = [&](int lseg, const LargeSeg& sg) {
        SortHdr h;
        h.mag = 0;
        if (sizeof(K) == 8) {   // (a whole binade: cells stay aligned with the binades)
            const unsigned long long c = __ldcg(seg_lo + n_lseg + lseg);
            h.mag = c ? (~c >> KO::MANT) << KO::MANT : 0ull;
        }
        const K hi = squeeze<T>((K)__ldcg(seg_hi + lseg), h.mag),
                lo = squeeze<T>((K)~(K)__ldcg(seg_lo + lseg), h.mag);
        // cells aligned in the key space, so that no cell (or part of one)
        // straddles a binade, where the density per key jumps by two
        const K range = hi > lo ? hi - lo : (K)0;
        const int cl = 31 - __clz(sg.ncell);
        const int bl = range ? 64 - __clzll((long long)(uint64_t)range) : 0;
        h.shift = max(bl - cl, 0);
        if (hi > lo && (hi >> h.shift) - (lo >> h.shift) >= (K)sg.ncell) ++h.shift;
        h.kmin = (uint64_t)((lo >> h.shift) << h.shift);
        h.dlo = (uint64_t)lo - h.kmin;
        h.dhi = (uint64_t)max(hi, lo) - h.kmin;
        return h;
    };
    // f(offset above kmin) for every sample of tiles [ta, tb) of one segment
    auto samples = [&](const LargeSeg& sg, const SortHdr& h, int ta, int tb, auto f) {
        const int m = 1 << sg.samp_log2;
#pragma unroll 4
        for (int i = t; i < (tb - ta) << sg.samp_log2; i += PLAN_NT) {
            const int tile = ta + (i >> sg.samp_log2), j = i & (m - 1);
            const int64_t o = (int64_t)(tile - sg.sort_first) * WS_SORT_TILE;
            const int len = (int)min((int64_t)WS_SORT_TILE, sg.len - o);
            if (j < len) {
                const K k = squeeze<T>(
                    cached ? cache[((size_t)(tile - t0) << samp_max) + j]
                           : KO::to_key(__ldg(values + sg.vpos + o + sample_pos(tile, j, len, sg.samp_log2))),
                    h.mag);
                f(k > (K)h.kmin ? k - (K)h.kmin : (K)0);
            }
        }
    };

    // 2. sampled keys per cell (counted in shared memory, added to the
    // segment's cells once per CTA)
    for (int ta = t0; ta < tm;) {
        const int lseg = tiles[ta].lseg;
        const LargeSeg sg = lsegs[lseg];
        const int tb = min(t1, sg.sort_first + sg.sort_count);
        if (sg.sort_count == 1) { ta = tb; continue; }   // (uniform)
        const SortHdr h = header(lseg, sg);
        uint32_t* sc = tab.split;   // [ncell]
        for (int i = t; i < sg.ncell; i += PLAN_NT) sc[i] = 0;
        __syncthreads();
        samples(sg, h, ta, tb, [&](K d) { atomicAdd(&sc[(uint32_t)min(d >> h.shift, (K)(sg.ncell - 1))], 1u); });
        __syncthreads();
        for (int i = t; i < sg.ncell; i += PLAN_NT)
            if (sc[i]) atomicAdd(cells + sg.cell_pos + i, sc[i]);
        __syncthreads();
        ta = tb;
    }
    bar.sync();

    // Parts of every cell, from the cell counts (every CTA for the segments
    // it needs; into tab.split): a cell of c samples gets 2^floor(log2(c / thr))
    // parts, thr = the larger of 96 samples (10 % noise) and 1 / ncell of all
    // (so at most ncell parts beside one per cell).  Cells with less than 8 thr
    // are cut down to 48 samples a part if that fits: in the tails the density
    // varies more inside a cell than the noise costs.  Returns the number.
    auto parts_of = [&](const LargeSeg& sg, const SortHdr& h) -> int {
        constexpr int PER = WS_CELLS / PLAN_NT;
        int v[PER], bits[PER], sum;
#pragma unroll
        for (int i = 0; i < PER; ++i) {
            const int c = t * PER + i;
            v[i] = c < sg.ncell ? (int)__ldcg(cells + sg.cell_pos + c) : 0;
        }
        const int m = 1 << sg.samp_log2, tail = (int)(sg.len - (int64_t)(sg.sort_count - 1) * WS_SORT_TILE);
        int tot = (sg.sort_count - 1) * m + min(tail, m);   // the segment's samples
        const int thr = max(96, tot / sg.ncell + 1);
        const int bmax = min(h.shift, 12);
        auto log2_of = [](int q) { return q > 0 ? 31 - __clz(q) : 0; };
        int ex = 0;
        for (int fine = 1; fine >= 0; --fine) {
            sum = 0;
#pragma unroll
            for (int i = 0; i < PER; ++i) {
                bits[i] = log2_of(v[i] / thr);
                if (fine && bits[i] < 3) bits[i] = min(log2_of(v[i] / 48), 3);
                bits[i] = min(bits[i], bmax);
                if (t * PER + i < sg.ncell) sum += 1 << bits[i];
            }
            ex = ws_block_excl_scan<PLAN_NT, int>(sum, S.wsum, &tot);
            if (tot <= 2 * sg.ncell) break;   // (uniform; always without the fine cut)
        }
#pragma unroll
        for (int i = 0; i < PER; ++i) {
            const int c = t * PER + i;
            if (c < sg.ncell) {
                tab.split[c] = (uint32_t)min(ex, 2 * sg.ncell) | ((uint32_t)(h.shift - bits[i]) << 16);
                ex += 1 << bits[i];
            }
        }
        if (t == 0) tab.split[sg.ncell] = (uint32_t)min(tot, 2 * sg.ncell) | ((uint32_t)h.shift << 16);
        __syncthreads();
        return min(tot, 2 * sg.ncell);
    };

    // 3. sampled keys per part
    for (int ta = t0; ta < tm;) {
        const int lseg = tiles[ta].lseg;
        const LargeSeg sg = lsegs[lseg];
        const int tb = min(t1, sg.sort_first + sg.sort_count);
        if (sg.sort_count == 1) { ta = tb; continue; }   // (uniform)
        const SortHdr h = header(lseg, sg);
        const int parts = parts_of(sg, h);
        uint32_t* sc = reinterpret_cast<uint32_t*>(tab.knots);   // [parts]
        for (int i = t; i < parts; i += PLAN_NT) sc[i] = 0;
        __syncthreads();
        const K mask = (K)(((K)1 << h.shift) - 1);
        samples(sg, h, ta, tb, [&](K d) {
            const uint32_t c = (uint32_t)min(d >> h.shift, (K)(sg.ncell - 1));
            const uint32_t e = tab.split[c];
            const uint32_t i = (e & 0xffffu) + (uint32_t)((d & mask) >> (int)(e >> 16));
            if (i < (uint32_t)parts) atomicAdd(&sc[i], 1u);
        });
        __syncthreads();
        uint32_t* gp = cells + sg.cell_pos + sg.ncell;
        for (int i = t; i < parts; i += PLAN_NT)
            if (sc[i]) atomicAdd(gp + i, sc[i]);
        __syncthreads();
        ta = tb;
    }
    bar.sync();

    if (S.n_one > 0) bad = plan_one<T, B>(S, values, tiles, t0, t1, lsegs, bins, bin_cnt, bin_start, cur1, seg_emin);

    // 4. knots of every segment (every CTA for the segments it needs), the bin
    // of every key, finiteness, smallest exponent
    for (int ta = t0; ta < tm;) {
        const int lseg = tiles[ta].lseg;
        const LargeSeg sg = lsegs[lseg];
        const int tb = min(t1, sg.sort_first + sg.sort_count);
        if (sg.sort_count == 1) { ta = tb; continue; }   // (uniform)
        const bool local = sg.nbins <= hist_cap;
        const SortHdr h = header(lseg, sg);
        const int parts = parts_of(sg, h);
        {
            constexpr int PER = 2 * WS_CELLS / PLAN_NT;
            int v[PER], sum = 0;
#pragma unroll
            for (int i = 0; i < PER; ++i) {
                const int c = t * PER + i;
                v[i] = c < parts ? (int)__ldcg(cells + sg.cell_pos + sg.ncell + c) : 0;
                sum += v[i];
            }
            int tot;
            int ex = ws_block_excl_scan<PLAN_NT, int>(sum, S.wsum, &tot);
            const float scale = (float)sg.nbins / (float)max(tot, 1);
#pragma unroll
            for (int i = 0; i < PER; ++i) {
                const int c = t * PER + i;
                if (c < parts) tab.knots[c].x = fminf((float)ex * scale, (float)sg.nbins);
                ex += v[i];
            }
            if (t == 0) tab.knots[parts] = make_float2((float)sg.nbins, 0.0f);
            __syncthreads();
            for (int c = t; c < sg.ncell; c += PLAN_NT) {
                const uint32_t e = tab.split[c];
                const int s2 = (int)(e >> 16);
                const int q1 = min((int)(e & 0xffffu) + (1 << (h.shift - s2)), parts);
                for (int q = (int)(e & 0xffffu); q < q1; ++q)
                    tab.knots[q].y = KeyMap<T>::slope(tab.knots[q + 1].x - tab.knots[q].x, s2);
            }
            __syncthreads();
            if (t == 0) {
                // The parts of the smallest and the largest sample are filled from and up to these
                // only (a distribution with a hard edge: the bins there held two times the mean and
                // more).  Below the first: bin 0; above the last: the last bin.
                auto part_at = [&](K d, int& s2) {
                    const uint32_t e = tab.split[(uint32_t)min(d >> h.shift, (K)(sg.ncell - 1))];
                    s2 = (int)(e >> 16);
                    return (int)min((e & 0xffffu) + (uint32_t)((d & (((K)1 << h.shift) - 1)) >> s2), (uint32_t)(parts - 1));
                };
                int s0, s1;
                const int q0 = part_at((K)h.dlo, s0), q1 = part_at((K)h.dhi, s1);
                const float w0 = ldexpf(1.0f, sizeof(K) == 4 ? s0 : min(s0, 24)), l0 = (float)KeyMap<T>::low((K)h.dlo, s0);
                const float l1 = (float)KeyMap<T>::low((K)h.dhi, s1) + 1.0f;
                if (q0 < q1) {
                    // (the start moves by at most 64 times the part's bins: its rounding, 2^-18 of them, stays
                    // inside the slope's 2^-16)
                    if ((w0 - l0) * 64.0f >= w0) {
                        const float y = (tab.knots[q0 + 1].x - tab.knots[q0].x) * (1.0f - 1.0f / 65536.0f) / (w0 - l0);
                        tab.knots[q0] = make_float2(tab.knots[q0].x - l0 * y, y);
                    }
                    tab.knots[q1].y = (tab.knots[q1 + 1].x - tab.knots[q1].x) / l1;
                }
            }
        }
        KeyMap<T> map;
        map.init(h, sg.ncell, sg.nbins);
        if (local)
            for (int i = t; i < sg.nbins; i += PLAN_NT) hist[i] = 0;
        if (t == 0) S.emin = 0x7fffffff;
        __syncthreads();
        const int64_t o0 = (int64_t)(ta - sg.sort_first) * WS_SORT_TILE;
        const int64_t n = min((int64_t)(tb - sg.sort_first) * WS_SORT_TILE, sg.len) - o0;
        const T* src = values + sg.vpos + o0;
        B* bo = bins + sg.kpos + o0;   // (16-byte aligned keys: 8-byte aligned at least for two-byte bins)
        uint32_t* gcnt = bin_cnt + sg.bin_pos;
        K amax = 0, amin = ~(K)0;   // largest magnitude bits; smallest ones minus 1 (zero wraps to the largest)
        auto bin_of = [&](T v) -> uint32_t {
            const K mag = (K)KO::bits(v) & (~(K)0 >> 1);
            amax = max(amax, mag);
            amin = min(amin, mag - 1);
            const uint32_t b = map.bin(KO::to_key(v), tab);
            if (local) atomicAdd(&hist[b], 1u);
            else atomicAdd(gcnt + b, 1u);
            return b;
        };
        if (((uintptr_t)src & 15) == 0) {
            // 16-byte loads, four in flight per thread
            constexpr int VEC = 16 / (int)sizeof(T), U = 4;
            const int64_t nv = n / VEC;
            const uint4* vs = reinterpret_cast<const uint4*>(src);
            auto one = [&](const uint4& q, int64_t i) {
                const T* e = reinterpret_cast<const T*>(&q);
                __align__(16) B r[VEC];
#pragma unroll
                for (int k = 0; k < VEC; ++k) r[k] = (B)bin_of(e[k]);
                if (sizeof(r) == 16) *reinterpret_cast<uint4*>(bo + i * VEC) = *reinterpret_cast<const uint4*>(r);
                else if (sizeof(r) == 8) *reinterpret_cast<uint2*>(bo + i * VEC) = *reinterpret_cast<const uint2*>(r);
                else *reinterpret_cast<uint32_t*>(bo + i * VEC) = *reinterpret_cast<const uint32_t*>(r);
            };
            int64_t i = t;
            for (; i + (U - 1) * PLAN_NT < nv; i += U * PLAN_NT) {
                uint4 buf[U];
#pragma unroll
                for (int u = 0; u < U; ++u) buf[u] = __ldg(vs + i + u * PLAN_NT);
#pragma unroll
                for (int u = 0; u < U; ++u) one(buf[u], i + u * PLAN_NT);
            }
            for (; i < nv; i += PLAN_NT) one(__ldg(vs + i), i);
            for (int64_t k = nv * VEC + t; k < n; k += PLAN_NT) bo[k] = (B)bin_of(src[k]);
        } else {
            constexpr int U = 8;
            int64_t i = t;
            for (; i + (U - 1) * PLAN_NT < n; i += U * PLAN_NT) {
                T v[U];
#pragma unroll
                for (int u = 0; u < U; ++u) v[u] = __ldg(src + i + u * PLAN_NT);
#pragma unroll
                for (int u = 0; u < U; ++u) bo[i + u * PLAN_NT] = (B)bin_of(v[u]);
            }
            for (; i < n; i += PLAN_NT) bo[i] = (B)bin_of(src[i]);
        }
        bad |= (amax >> KO::MANT) >= (K)KO::EXPMASK;
        int emin = amin != ~(K)0 ? max((int)((amin + 1) >> KO::MANT), 1) : 0x7fffffff;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) emin = min(emin, __shfl_xor_sync(WS_FULL_MASK, emin, o));
        if (lane == 0 && emin != 0x7fffffff) atomicMin(&S.emin, emin);
        __syncthreads();
        if (t == 0 && S.emin != 0x7fffffff) atomicMax(seg_en + lseg, (uint32_t)(0x7fffffff - S.emin));
        if (local)
            for (int q = t; q < sg.nbins; q += PLAN_NT)
                if (hist[q]) atomicAdd(gcnt + q, hist[q]);
        __syncthreads();
        ta = tb;
    }
    if (bad) ws_flag(status, WS_STATUS_NONFINITE);
    bar.sync();

    // 5. bin starts and the passes' cursors: a CTA per segment and run of
    // PLAN_NT bins, which adds up the counts before its run itself
    for (int c0 = 0; c0 < max_bins; c0 += PLAN_NT) {
        const int first = (int)(((int64_t)blockIdx.x + (int64_t)gridDim.x * (c0 / PLAN_NT) - c0 / PLAN_NT) % gridDim.x);
        for (int lseg = first; lseg < n_lseg; lseg += gridDim.x) {
            const LargeSeg sg = lsegs[lseg];
            if (c0 >= sg.nbins || sg.sort_count == 1) continue;   // (uniform)
            const uint32_t* c = bin_cnt + sg.bin_pos;
            int before = 0;
#pragma unroll 8
            for (int b = t; b < c0; b += PLAN_NT) before += (int)__ldcg(c + b);
            int base;
            ws_block_excl_scan<PLAN_NT, int>(before, S.wsum, &base);
            const int b = c0 + t;
            const int own = b < sg.nbins ? (int)__ldcg(c + b) : 0;
            const uint32_t start = (uint32_t)(base + ws_block_excl_scan<PLAN_NT, int>(own, S.wsum, nullptr));
            if (b < sg.nbins) {
                bin_start[sg.bin_pos + b] = start;
                if (sg.fine_log2 == 0) cur1[sg.coarse_pos + b] = start;
                else {
                    cur2[sg.bin_pos + b] = start;
                    if ((b & ((1 << sg.fine_log2) - 1)) == 0) cur1[sg.coarse_pos + (b >> sg.fine_log2)] = start;
                }
            }
            if (c0 == 0 && t == 0) seg_emin[lseg] = (int32_t)(0x7fffffffu - __ldcg(seg_en + lseg));
        }
    }
}

// ---------------------------------------------------------------------------
// Partition passes.  FIRST: the values into buckets of 2^fine_log2 bins (to
// keys_a) or straight into bins (one-level segments, to keys_b).  Otherwise:
// the buckets of two-level segments into bins (keys_a to keys_b); a tile lies
// in one bucket or two as a rule, and takes further rounds of WS_FAN bins
// where its buckets are sparse.
// ---------------------------------------------------------------------------
template <typename T, typename B>
struct PartSmem {
    typename KeyOf<T>::K key[WS_SORT_TILE];
    B bin[WS_SORT_TILE];
    uint32_t cnt[WS_FAN];
    uint2 run[WS_FAN];        // start of the bucket's run inside the tile, and its destination
    uint32_t starts[WS_SORT_TILE / 32];   // a bit at the first place of every run
    int wsum[WS_SORT_NT / 32];
    int tie;                              // bucket of a heavy tie in the tile before, or -1
};

// Ranks of a warp's keys (w: bin << 13 per key, the rank goes below) where many are in
// bucket `tie`: these are counted by votes, and added once.
__device__ __noinline__ void part_rank_tied(uint32_t* w, uint32_t* cnt, uint32_t tie, int bsh, uint32_t off, int len) {
    const int t = threadIdx.x, lane = t & 31;
    uint32_t met = 0;
#pragma unroll 1
    for (int p = t; p < WS_SORT_TILE; p += WS_SORT_NT) {
        const uint32_t x = w[p], b = (x >> bsh) - off;
        const bool in = p < len && b < WS_FAN;
        const unsigned m = __ballot_sync(WS_FULL_MASK, in && b == tie);
        if (in)
            w[p] = (x & ~0x1fffu) |
                   (b == tie ? met + (uint32_t)__popc(m & ((1u << lane) - 1u)) : atomicAdd(&cnt[b], 1u));
        met += (uint32_t)__popc(m);
    }
    uint32_t at = lane == 0 ? atomicAdd(&cnt[tie], met) : 0u;
    at = __shfl_sync(WS_FULL_MASK, at, 0);
#pragma unroll 1
    for (int p = t; p < len; p += WS_SORT_NT)
        if ((w[p] >> bsh) - off == tie) w[p] += at;
}

template <typename T, typename B, bool FIRST, bool TOP>
__global__ void __launch_bounds__(WS_SORT_NT, sizeof(T) == 4 ? 3 : 2) k_part(
    const T* __restrict__ values, const typename KeyOf<T>::K* __restrict__ keys_in, const B* __restrict__ bins_in,
    typename KeyOf<T>::K* __restrict__ out_a, typename KeyOf<T>::K* __restrict__ out_b, B* __restrict__ bins_out,
    PassMap map,   // (map.loc nullable: how to undo the pass)
    const TileDesc* __restrict__ tiles, int n_tiles, const LargeSeg* __restrict__ lsegs, uint32_t* cursor,
    const SortCtl* ctl) {
    typedef KeyOf<T> KO;
    typedef typename KO::K K;
    constexpr int NT = WS_SORT_NT, ITEMS = WS_SORT_ITEMS;
    static_assert(WS_FAN == NT, "one bucket per thread");
    extern __shared__ __align__(16) unsigned char smem_raw[];
    PartSmem<T, B>& s = *reinterpret_cast<PartSmem<T, B>*>(smem_raw);
    ws_chain_wait();
    if (ctl->abort) return;
    const int t = threadIdx.x;
    // the next tile of this CTA from `tile` on that this pass moves
    auto next_tile = [&](int tile) {
        if (!FIRST)
            while (tile < n_tiles && lsegs[tiles[tile].lseg].fine_log2 == 0) tile += gridDim.x;
        return tile;
    };
    K key[ITEMS];         // (loaded raw; made keys when the tile's turn comes, so that the loads stay in flight)
    // bin << 13 | rank.  TOP (more than 2^19 bins): the bin's top bit is in `top`, a bit per key
    uint32_t br[ITEMS], top = 0;
    auto load = [&](const TileDesc& td) {
        const K* src = FIRST ? reinterpret_cast<const K*>(values) + td.vpos : keys_in + td.kpos;
        const B* bsrc = bins_in + td.kpos;
#pragma unroll
        for (int k = 0; k < ITEMS; ++k) {
            const int p = t + k * NT;
            if (p < td.len) {
                key[k] = __ldg(src + p);
                br[k] = __ldg(bsrc + p);
            }
        }
    };
    int tile = next_tile(blockIdx.x);
    if (tile >= n_tiles) return;
    load(tiles[tile]);
    if (t == 0) s.tie = -1;
    while (tile < n_tiles) {
        const int nxt = next_tile(tile + gridDim.x);
        const int len = tiles[tile].len;
        const LargeSeg& sg = lsegs[tiles[tile].lseg];
        const int fl = sg.fine_log2;
        // the tile's buckets: all of the segment's (first pass), the bins of
        // its first to last bucket (second)
        int base = 0, nbk = sg.n_coarse;
        if (!FIRST) {
            const int64_t k0 = tiles[tile].kpos;
            base = ((int)__ldg(bins_in + k0) >> fl) << fl;
            nbk = max(min(sg.nbins, (((int)__ldg(bins_in + k0 + len - 1) >> fl) + 1) << fl) - base, 1);
        }
        const int bsh = FIRST ? 13 + fl : 13;
        uint32_t jb = 0, rb = 0;   // places and runs of the rounds before
#pragma unroll
        for (int k = 0; k < ITEMS; ++k) {
            if (FIRST) key[k] = KO::key_of_bits(key[k]);
            if (TOP) top = (k ? top : 0u) | ((br[k] >> 19) & 1u) << k;
            br[k] <<= 13;
        }
        auto bin_of = [&](int k) -> uint32_t { return TOP ? (br[k] >> 13) | ((top >> k) & 1u) << 19 : br[k] >> 13; };
        auto bucket_of = [&](int k, uint32_t off) -> uint32_t {   // (WS_FAN and above: not of this round)
            return (TOP ? bin_of(k) >> (bsh - 13) : br[k] >> bsh) - off;
        };
        for (int r0 = 0; r0 < nbk; r0 += WS_FAN) {
            const uint32_t off = (uint32_t)(base + r0);
            __syncthreads();   // (the previous use of the shared memory is over)
            s.cnt[t] = 0;
            if (r0 == 0 && t < WS_SORT_TILE / 32) s.starts[t] = 0;
            // A heavy tie's adds to its bucket would go one by one: where a bucket took a third of the tile
            // before, a warp counts its keys for that bucket by votes and adds them once.  2^26 weights: 99 %
            // zeros 835 -> 600 us for both passes, one value 779 -> 546.  With few buckets the adds are as
            // fast: 8192 segments of 4097 183 us, by votes 207.
            const int tie = nbk >= 8 ? s.tie : -1;
            __syncthreads();
            if (t == 0) s.tie = -1;
            if (tie < 0) {
#pragma unroll
                for (int k = 0; k < ITEMS; ++k) {
                    const uint32_t b = bucket_of(k, off);
                    if (t + k * NT < len && b < WS_FAN) br[k] = (br[k] & ~0x1fffu) | atomicAdd(&s.cnt[b], 1u);
                }
            } else {   // (through the staging area: out of line, and the loop above keeps its registers)
                uint32_t* w = reinterpret_cast<uint32_t*>(s.key);
#pragma unroll
                for (int k = 0; k < ITEMS; ++k) w[t + k * NT] = TOP ? min(bucket_of(k, off), (uint32_t)WS_FAN) << 13 : br[k];
                part_rank_tied(w, s.cnt, (uint32_t)tie, TOP ? 13 : bsh, TOP ? 0u : off, len);
#pragma unroll
                for (int k = 0; k < ITEMS; ++k) br[k] = TOP ? (br[k] & ~0x1fffu) | (w[t + k * NT] & 0x1fffu) : w[t + k * NT];
            }
            __syncthreads();
            // start inside the tile, and the run's destination
            const uint32_t c = s.cnt[t];
            if (c > WS_SORT_TILE / 3) atomicMax(&s.tie, t);
            const uint32_t g =
                c ? atomicAdd(cursor + (FIRST ? sg.coarse_pos : sg.bin_pos + base) + r0 + t, c) : 0u;
            // (places in the low half, runs in the high one)
            int tot2;
            const uint32_t ex2 =
                (uint32_t)ws_block_excl_scan<NT, int>((int)(c | (c ? 0x10000u : 0u)), s.wsum, &tot2);
            const uint32_t ex = ex2 & 0xffffu;
            const int total = tot2 & 0xffff;
            s.run[t] = make_uint2(ex, g);
            if (map.loc && c) {
                const uint32_t j = jb + ex;
                map.delta[(FIRST ? (int64_t)tile * WS_FAN : tiles[tile].kpos) + rb + (ex2 >> 16)] = g - j;
                atomicOr(&s.starts[j >> 5], 1u << (j & 31));
            }
            __syncthreads();
            const int64_t kp = tiles[tile].kpos;
#pragma unroll
            for (int k = 0; k < ITEMS; ++k) {
                const uint32_t b = bucket_of(k, off);
                if (t + k * NT < len && b < WS_FAN) {
                    const uint2 run = s.run[b];
                    const uint32_t rk = br[k] & 0x1fffu, j = run.x + rk;
                    s.key[j] = key[k];
                    s.bin[j] = (B)bin_of(k);
                    if (map.loc) map.loc[kp + t + k * NT] = (uint16_t)(jb + j);
                }
            }
            __syncthreads();
            // (the key registers are free: the next tile's loads overlap the copy)
            if (r0 + WS_FAN >= nbk) {
                if (nxt < n_tiles) load(tiles[nxt]);
                else ws_chain_go();
            }
            // bucket runs, copied out by consecutive threads
            K* dst = (FIRST && fl != 0 ? out_a : out_b) + sg.kpos;
            B* bdst = bins_out + sg.kpos;
            const uint32_t slen = (uint32_t)sg.len;
#pragma unroll 4
            for (int j = t; j < total; j += NT) {
                const B bn = s.bin[j];
                const uint2 run = s.run[((uint32_t)bn >> (bsh - 13)) - off];
                const uint32_t p = run.y + (uint32_t)j - run.x;
                if (p < slen) {   // (always)
                    dst[p] = s.key[j];
                    if (FIRST && fl != 0) bdst[p] = bn;
                }
            }
            jb += (uint32_t)total;
            rb += (uint32_t)tot2 >> 16;
        }
        if (map.loc && t < WS_SORT_TILE / 32) map.starts[(int64_t)tile * (WS_SORT_TILE / 32) + t] = s.starts[t];
        tile = nxt;
    }
}

// ---------------------------------------------------------------------------
// Sort of one bin per CTA: the keys into 1024 groups by a monotone linear map
// of the bin's range (2.5 keys each on average), every group of at most 8 keys
// in one thread's registers by a sorting network, larger ones (one in 500; more
// in the tails, where the density varies inside a bin) by a warp that counts
// ranks.  A bin with a group of more than BIN_WARP_MAX keys (unless they are
// equal) takes LSD radix passes over the bits that vary in it.
//
// PLACE: the place of every key in the unsorted bin is wanted too.  What is
// sorted then are words of the key above the bin's smallest (its top 20 bits;
// 52 for FP64) and the place in the low 12 bits, so that the sort moves one
// word per key either way.  Where the bin spans more than that (short
// segments, bins near zero), keys with the same top bits are put in order
// after it.
// ---------------------------------------------------------------------------
constexpr int BIN_NT = 256;
constexpr int BIN_ITEMS = WS_BIN_CAP / BIN_NT;
constexpr int BIN_REG = 12;                      // keys per thread kept in registers
constexpr int BIN_GPT = 4;                       // groups per thread
constexpr int BIN_GROUPS = BIN_GPT * BIN_NT;
constexpr int BIN_NET = 8;
constexpr int BIN_WARP_MAX = 256;
constexpr int BIN_RUN_MAX = 32;                  // keys with the same top bits that one thread orders

template <typename T>
struct BinSmem {
    typedef typename KeyOf<T>::K K;
    K key[WS_BIN_CAP];               // keys, or words
    union {
        uint32_t cnt[BIN_GROUPS];
        struct {
            uint32_t whist[(BIN_NT / 32) * 256];
            uint32_t dcount[256], dstart[256];
        } radix;
    } u;
    K lo, hi;
    uint32_t late[WS_BIN_CAP - BIN_REG * BIN_NT];    // group << 16 | rank of the keys not in registers
    int wsum[BIN_NT / 32];
    int n_list, radix_needed, skew;
    uint32_t list[WS_BIN_CAP / (BIN_NET + 1) + 1];   // start << 16 | keys of the groups for the warps
};

// Batcher's odd-even merge sorting network.
template <int N, typename K>
__device__ __forceinline__ void sort_network(K (&v)[N]) {
#pragma unroll
    for (int p = 1; p < N; p *= 2)
#pragma unroll
        for (int k = p; k >= 1; k /= 2)
#pragma unroll
            for (int j = k % p; j + k < N; j += 2 * k)
#pragma unroll
                for (int i = 0; i < k; ++i)
                    if (j + i + k < N && (j + i) / (2 * p) == (j + i + k) / (2 * p)) {
                        const K a = v[j + i], c = v[j + i + k];
                        v[j + i] = min(a, c);
                        v[j + i + k] = max(a, c);
                    }
}

template <int N, typename K>
__device__ __forceinline__ void sort_group(K* key, int n) {
    K v[N];
#pragma unroll
    for (int i = 0; i < N; ++i) v[i] = i < n ? key[i] : ~(K)0;
    sort_network<N, K>(v);
#pragma unroll
    for (int i = 0; i < N; ++i)
        if (i < n) key[i] = v[i];
}

__device__ __forceinline__ uint32_t warp_min_k(uint32_t v) { return __reduce_min_sync(WS_FULL_MASK, v); }
__device__ __forceinline__ uint32_t warp_max_k(uint32_t v) { return __reduce_max_sync(WS_FULL_MASK, v); }
__device__ __forceinline__ uint64_t warp_min_k(uint64_t v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = min(v, ws_shfl_xor_k(v, o));
    return v;
}
__device__ __forceinline__ uint64_t warp_max_k(uint64_t v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = max(v, ws_shfl_xor_k(v, o));
    return v;
}

// Sort of n keys or words by one warp: ranks by counting (ties by place).
// Words that are equal above the place are left alone (any order will do).
// Keys of which few differ (weights that are already shared) are written as
// runs.  false: more than BIN_WARP_MAX and neither.
template <bool PLACE, typename K>
__device__ __noinline__ bool sort_warp(K* key, int n) {
    const int lane = threadIdx.x & 31;
    constexpr int PER = BIN_WARP_MAX / 32;
    if (PLACE && n > 16) {
        const K k0 = key[0] >> 12;
        bool same = true;
        for (int j = lane; same && j - lane < n; j += 32) same = __all_sync(WS_FULL_MASK, j >= n || (key[j] >> 12) == k0);
        if (same) return true;
        if (n > BIN_WARP_MAX) return false;
    }
    bool runs = false;
    if (!PLACE && n > 16) {   // (at most 8 different ones among the first 32)
        const unsigned peers = __match_any_sync(WS_FULL_MASK, (unsigned long long)key[min(lane, n - 1)]);
        runs = n > BIN_WARP_MAX || __popc(__ballot_sync(WS_FULL_MASK, lane == __ffs((int)peers) - 1)) <= 8;
    }
    if (runs) {
        // lane d gets the d-th smallest value and where its run ends
        K mine = 0, prev = 0;
        int end = n, done = 0;
        for (int d = 0; d < 32 && done < n; ++d) {
            K lo = ~(K)0;
            for (int j = lane; j < n; j += 32) {
                const K x = key[j];
                if (d == 0 || x > prev) lo = min(lo, x);
            }
            lo = warp_min_k(lo);
            int c = 0;
            for (int j = lane; j < n; j += 32) c += key[j] == lo;
            done += __reduce_add_sync(WS_FULL_MASK, c);
            if (lane == d) { mine = lo; end = done; }
            prev = lo;
        }
        __syncwarp();
        if (done == n) {
            for (int d = 0, j0 = 0; d < 32 && j0 < n; ++d) {
                const K x = ws_shfl_k(mine, d);
                const int j1 = __shfl_sync(WS_FULL_MASK, end, d);
                for (int j = j0 + lane; j < j1; j += 32) key[j] = x;
                j0 = j1;
            }
            return true;
        }
        if (n > BIN_WARP_MAX) return false;
    }
    K v[PER];
    int r[PER];
#pragma unroll
    for (int k = 0; k < PER; ++k) {
        v[k] = lane + 32 * k < n ? key[lane + 32 * k] : ~(K)0;
        r[k] = 0;
    }
#pragma unroll 4
    for (int j = 0; j < n; ++j) {
        const K x = key[j];
#pragma unroll
        for (int k = 0; k < PER; ++k) {
            if (32 * k >= n) break;   // (uniform)
            r[k] += (x < v[k] || (!PLACE && x == v[k] && j < lane + 32 * k)) ? 1 : 0;   // (places: all words differ)
        }
    }
    __syncwarp();
#pragma unroll
    for (int k = 0; k < PER; ++k)
        if (lane + 32 * k < n) key[r[k]] = v[k];
    return true;
}

// LSD radix passes, 8-bit digits that vary (diff), over a bin's n keys in
// s.key; with PLACE over the words that are there already (words: they hold every
// bit that varies), or else over the keys src[place], s.key holding the places.
// The rare path: out of line.
template <typename T, bool PLACE>
__device__ __noinline__ void bin_radix(BinSmem<T>& s, const typename KeyOf<T>::K* src, int n,
                                       typename KeyOf<T>::K diff, bool words) {
    typedef typename KeyOf<T>::K K;
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    if (!words) {
        for (int i = t; i < n; i += BIN_NT) s.key[i] = PLACE ? (K)i : src[i];
        __syncthreads();
    }
    for (int pass = 0; pass < KeyOf<T>::BITS / 8; ++pass) {
        if (((diff >> (8 * pass)) & 0xff) == 0) continue;
        K key[BIN_ITEMS];
        uint32_t dg[BIN_ITEMS];
        bool valid[BIN_ITEMS];
        int pos[BIN_ITEMS];
#pragma unroll
        for (int k = 0; k < BIN_ITEMS; ++k) {
            const int p = w * 32 * BIN_ITEMS + k * 32 + lane;
            valid[k] = p < n;
            key[k] = valid[k] ? s.key[p] : (K)0;
            const K kk = PLACE && !words ? (valid[k] ? __ldg(src + (uint32_t)key[k]) : (K)0) : key[k];
            dg[k] = (uint32_t)((kk >> (8 * pass)) & 0xff);
        }
        __syncthreads();
        ws_rank_digits<BIN_NT, BIN_ITEMS, 1>(dg, valid, pos, s.u.radix.whist, s.u.radix.dcount, s.u.radix.dstart);
#pragma unroll
        for (int k = 0; k < BIN_ITEMS; ++k)
            if (valid[k]) s.key[pos[k]] = key[k];
        __syncthreads();
    }
}

// Monotone image of a double in FP32 by truncation (no FP64 conversion).
__device__ __forceinline__ float ws_trunc_f32(float v) { return v; }
__device__ __forceinline__ float ws_trunc_f32(double v) {
    const uint64_t b = (uint64_t)__double_as_longlong(v);
    const int e = (int)((b >> 52) & 0x7ff) - 896;
    const uint32_t sign = (uint32_t)(b >> 32) & 0x80000000u;
    uint32_t m = (uint32_t)(b >> 29) & 0x7fffffu;
    if (e <= 0) return __uint_as_float(sign);
    if (e >= 255) return __uint_as_float(sign | 0x7f7fffffu);
    return __uint_as_float(sign | ((uint32_t)e << 23) | m);
}

constexpr int OVER_SAMPLE = 1024;   // keys at most
// Splitters of a bin, by one warp: quantiles of a sorted sample, each value once.
// (A value of more than two gaps between them is among them, so a class between
// splitters holds less than 3 / (quantiles + 1) of the bin, but for the sample's error.)
// Enters the bin in the list; the counts of its classes are cleared.
template <typename K>
__device__ __noinline__ void over_sample(K* s, const K* __restrict__ src, int n, int64_t start, int lseg, SortCtl* ctl,
                                         OverBin* over, OverTab<K>* tabs) {
    const int lane = threadIdx.x & 31;
    const uint32_t entry = lane == 0 ? atomicAdd(&ctl->over_count, 1u) : 0u;   // (back with the sample)
    int ns = 0;
    OverTab<K>* tab = nullptr;
    // a small sample for a bin that a few classes cut; a large one for a large bin of many different values
    for (int m = n < 16384 ? 64 : 256;; m = OVER_SAMPLE) {
#pragma unroll 4
        for (int j = lane; j < m; j += 32) s[j] = __ldg(src + ((uint64_t)(2 * j + 1) * (uint64_t)n) / (uint32_t)(2 * m));
        __syncwarp();
        for (int k = 2; k <= m; k <<= 1)
            for (int d = k >> 1; d > 0; d >>= 1) {
#pragma unroll 4
                for (int q = lane; q < m / 2; q += 32) {
                    const int i = 2 * q - (q & (d - 1)), j = i + d;
                    const K a = s[i], b = s[j];
                    if ((a > b) == ((i & k) == 0)) { s[i] = b; s[j] = a; }
                }
                __syncwarp();
            }
        tab = tabs + __shfl_sync(WS_FULL_MASK, entry, 0);
        // a splitter for every 256 keys (classes that one CTA sorts in a microsecond or two)
        const int q = min(min(OVER_SPL, m - 1), n / 256);
        ns = 0;
        for (int c0 = 1; c0 <= q; c0 += 32) {
            const int c = c0 + lane;
            const bool in = c <= q;
            const K v = s[in ? c * m / (q + 1) : 0];
            const bool take = in && (c == 1 || v != s[(c - 1) * m / (q + 1)]);
            const unsigned vote = __ballot_sync(WS_FULL_MASK, take);
            if (take) tab->spl[ns + __popc(vote & ((1u << lane) - 1u))] = v;
            ns += __popc(vote);
        }
        if (m == OVER_SAMPLE || n < (1 << 17) || ns < 64) break;   // (uniform)
        __syncwarp();
    }
    for (int j = lane; j < 2 * ns + 1; j += 32) tab->cnt[j] = 0;
    for (int j = lane; j < ns + 1; j += 32) tab->cur[j] = 0;
    if (lane == 0) {
        OverBin ob;
        ob.start = start;
        ob.n = n;
        ob.first_tile = 0;
        ob.lseg = lseg;
        ob.nspl = ns;
        over[entry] = ob;
    }
}

template <typename T, bool PLACE>
__global__ void __launch_bounds__(BIN_NT, 4) k_bin_sort(const typename KeyOf<T>::K* __restrict__ keys,
                                                        typename KeyOf<T>::K* __restrict__ sorted,
                                                        const int32_t* __restrict__ bin_seg,
                                                        const LargeSeg* __restrict__ lsegs,
                                                        const uint32_t* __restrict__ bin_start,
                                                        const uint32_t* __restrict__ bin_cnt,
                                                        uint16_t* __restrict__ bin_idx,   // (PLACE)
                                                        SortCtl* ctl, OverBin* over,
                                                        OverTab<typename KeyOf<T>::K>* tabs, int64_t n_keys) {
    typedef KeyOf<T> KO;
    typedef typename KO::K K;
    extern __shared__ __align__(16) unsigned char bin_smem_raw[];
    BinSmem<T>& s = *reinterpret_cast<BinSmem<T>*>(bin_smem_raw);
    ws_chain();
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    if (ctl->abort) {   // the keys were not moved: a sequence that is sorted, so that later steps see a valid one
        for (int64_t i = (int64_t)blockIdx.x * BIN_NT + t; i < n_keys; i += (int64_t)gridDim.x * BIN_NT)
            sorted[i] = KO::to_key((T)0);
        return;
    }
    const int bin = blockIdx.x;
    const int64_t start = lsegs[bin_seg[bin]].kpos + (int64_t)bin_start[bin];
    const int n = (int)bin_cnt[bin];
    if (n <= 0) return;
    if (n > WS_BIN_CAP) {
        // to the oversize kernel, with the splitters that it needs (here they cost no time of their own)
        if (t < 32) over_sample<K>(s.key, keys + start, n, start, bin_seg[bin], ctl, over, tabs);
        return;
    }
    const K* src = keys + start;
    reinterpret_cast<uint4*>(s.u.cnt)[t] = make_uint4(0, 0, 0, 0);
    if (t == 0) { s.lo = ~(K)0; s.hi = 0; s.n_list = 0; s.radix_needed = 0; s.skew = 0; }
    // the first BIN_REG keys of a thread stay in registers; the few beyond (a
    // bin 1.2 times the mean or more) are read again, and their group kept in
    // shared memory
    K key[BIN_REG];
#pragma unroll
    for (int k = 0; k < BIN_REG; ++k) {
        const int p = t + k * BIN_NT;
        key[k] = p < n ? __ldg(src + p) : (K)0;
    }
    K lo = ~(K)0, hi = 0;
#pragma unroll
    for (int k = 0; k < BIN_REG; ++k) {
        if (k * BIN_NT >= n) break;   // (uniform)
        if (t + k * BIN_NT < n) { lo = min(lo, key[k]); hi = max(hi, key[k]); }
    }
    for (int p = t + BIN_REG * BIN_NT; p < n; p += BIN_NT) { const K k = __ldg(src + p); lo = min(lo, k); hi = max(hi, k); }
    lo = warp_min_k(lo);
    hi = warp_max_k(hi);
    __syncthreads();
    if (lane == 0) { ws_atomic_min_k(&s.lo, lo); ws_atomic_max_k(&s.hi, hi); }
    __syncthreads();
    lo = s.lo;
    hi = s.hi;
    // group: linear in the key where sign and exponent are shared (the value is
    // linear in the key there), else linear in the value; but linear in the key
    // again where the bin spans several binades and most of it lies in a sixteenth of
    // the span next to zero (heavy tails: a few groups held such a bin, which took
    // radix passes: R of 4097 Cauchy weights 96 -> 69 us, of 20000 104 -> 61)
    bool by_key = ((lo ^ hi) >> KO::MANT) == 0;
    const int range_bits = 64 - __clzll((long long)((uint64_t)(hi - lo) | 1ull));
    const int dsh = max(0, range_bits - 24);
    const int cut = PLACE ? max(0, range_bits - (KO::BITS - 12)) : 0;   // key bits that the words leave out
    const float x0 = ws_trunc_f32(KO::from_key(lo)), x1 = ws_trunc_f32(KO::from_key(hi));
    if ((hi >> KO::MANT) - (lo >> KO::MANT) >= 3) {   // (uniform)
        const bool both = ((lo ^ hi) >> (KO::BITS - 1)) != 0;   // (signs)
        const float near0 = (both ? 0.0f : fminf(fabsf(x0), fabsf(x1))) + (x1 - x0) * 0.0625f;
        int c = 0;
#pragma unroll
        for (int k = 0; k < BIN_REG; ++k)
            c += t + k * BIN_NT < n && fabsf(ws_trunc_f32(KO::from_key(key[k]))) < near0 ? 1 : 0;
        c = __reduce_add_sync(WS_FULL_MASK, c);
        if (lane == 0) atomicAdd(&s.skew, c);
        __syncthreads();
        by_key = 2 * s.skew > min(n, BIN_REG * BIN_NT);
    }
    const float span = by_key ? (float)(uint32_t)((hi - lo) >> dsh) + 1.0f : x1 - x0;
    const float scale = (span > 0.0f && span <= 3.0e38f) ? (float)BIN_GROUPS / span : 0.0f;
    auto group_of = [&](K k) -> uint32_t {   // group << 16 | rank
        const float f = by_key ? (float)(uint32_t)((k - lo) >> dsh) : ws_trunc_f32(KO::from_key(k)) - x0;
        const uint32_t b = min((uint32_t)(int)(f * scale), (uint32_t)BIN_GROUPS - 1u);
        return (b << 16) | atomicAdd(&s.u.cnt[b], 1u);
    };
    auto word_of = [&](K k, int p) -> K { return PLACE ? (K)((((k - lo) >> cut) << 12) | (K)p) : k; };
    uint32_t br[BIN_REG];
#pragma unroll
    for (int k = 0; k < BIN_REG; ++k) {
        if (k * BIN_NT >= n) break;   // (uniform)
        const int p = t + k * BIN_NT;
        if (p < n) {
            br[k] = group_of(key[k]);
            key[k] = word_of(key[k], p);
        }
    }
    for (int p = t + BIN_REG * BIN_NT; p < n; p += BIN_NT) s.late[p - BIN_REG * BIN_NT] = group_of(__ldg(src + p));
    __syncthreads();
    // this thread's four groups
    static_assert(BIN_GPT == 4 && BIN_NT == 256, "a thread's group counts are one 16-byte word; eight warps");
    const uint4 c4 = reinterpret_cast<const uint4*>(s.u.cnt)[t];
    const int sum = (int)(c4.x + c4.y + c4.z + c4.w);
    const int inc = ws_warp_incl_scan<int>(sum);
    if (lane == 31) s.wsum[w] = inc;
    __syncthreads();
    const int wt = s.wsum[lane & 7];
    const int g0 = inc - sum + __reduce_add_sync(WS_FULL_MASK, lane < w ? wt : 0);
    reinterpret_cast<uint4*>(s.u.cnt)[t] =
        make_uint4((uint32_t)g0, g0 + c4.x, g0 + c4.x + c4.y, g0 + c4.x + c4.y + c4.z);
    __syncthreads();
#pragma unroll
    for (int k = 0; k < BIN_REG; ++k) {
        if (k * BIN_NT >= n) break;   // (uniform)
        if (t + k * BIN_NT < n) s.key[s.u.cnt[br[k] >> 16] + (br[k] & 0xffffu)] = key[k];
    }
    for (int p = t + BIN_REG * BIN_NT; p < n; p += BIN_NT) {
        const uint32_t b = s.late[p - BIN_REG * BIN_NT];
        s.key[s.u.cnt[b >> 16] + (b & 0xffffu)] = word_of(__ldg(src + p), p);
    }
    __syncthreads();
    {
        const int c[BIN_GPT] = {(int)c4.x, (int)c4.y, (int)c4.z, (int)c4.w};
        int g = g0;
#pragma unroll
        for (int i = 0; i < BIN_GPT; ++i) {
            if (c[i] <= BIN_NET) sort_group<BIN_NET, K>(s.key + g, c[i]);
            else s.list[atomicAdd(&s.n_list, 1)] = ((uint32_t)g << 16) | (uint32_t)c[i];
            g += c[i];
        }
    }
    __syncthreads();
    const int nl = s.n_list;
    if (nl > 0) {   // (uniform)
        for (int i = w; i < nl; i += BIN_NT / 32)
            if (!sort_warp<PLACE, K>(s.key + (s.list[i] >> 16), (int)(s.list[i] & 0xffffu)) && lane == 0)
                s.radix_needed = 1;
        __syncthreads();
    }
    bool radix = s.radix_needed != 0;   // (uniform: the last write is before the barrier above)
    if (PLACE && cut > 0 && !radix) {
        // runs with the same top bits: the thread of a run's first word orders it by the whole keys
        // (a run too long for that is a word of the barrier, not of shared memory: a warp that
        // has found one must not change the condition above for a warp that comes to it later)
        bool long_run = false;
        for (int i = t; i < n; i += BIN_NT) {
            const K top = s.key[i] >> 12;
            if (i > 0 && (s.key[i - 1] >> 12) == top) continue;
            int e = i + 1;
            while (e < n && e - i <= BIN_RUN_MAX && (s.key[e] >> 12) == top) ++e;
            if (e - i > BIN_RUN_MAX) { long_run = true; continue; }
            for (int a = i + 1; a < e; ++a) {
                const K wa = s.key[a], ka = __ldg(src + ((uint32_t)wa & 0xfffu));
                int j = a - 1;
                while (j >= i && __ldg(src + ((uint32_t)s.key[j] & 0xfffu)) > ka) { s.key[j + 1] = s.key[j]; --j; }
                s.key[j + 1] = wa;
            }
        }
        radix = __syncthreads_or(long_run) != 0;
        if (radix) {
            // (a long run of ties is in order as it is: one pass looks for a key below its neighbour)
            bool inverted = false;
            for (int i = t + 1; i < n; i += BIN_NT) {
                const K a = s.key[i - 1], b = s.key[i];
                if ((a >> 12) == (b >> 12))
                    inverted |= __ldg(src + ((uint32_t)a & 0xfffu)) > __ldg(src + ((uint32_t)b & 0xfffu));
            }
            radix = __syncthreads_or(inverted) != 0;
        }
    }
    if (radix) {   // (uniform; every word of the steps above has been read)
        const K vary = (K)(~(uint64_t)0 >> (64 - range_bits));
        if (PLACE && cut == 0) bin_radix<T, PLACE>(s, src, n, (K)(vary << 12), true);
        else bin_radix<T, PLACE>(s, src, n, vary | (lo ^ hi), false);
    }
    K* dst = sorted + start;
#pragma unroll 4
    for (int p = t; p < n; p += BIN_NT) {
        const K c = s.key[p];
        if (PLACE) {
            const uint32_t q = (uint32_t)c & 0xfffu;
            dst[p] = cut > 0 || radix ? __ldg(src + q) : lo + (c >> 12);
            bin_idx[start + p] = (uint16_t)q;
        } else {
            dst[p] = c;
        }
    }
}

// ---------------------------------------------------------------------------
// Oversize bins, as a cooperative grid with a barrier between the steps.  Such a
// bin is a heavy tie as a rule (zeros, weights that are already shared) with a few
// neighbours, sometimes a spike that the map does not resolve.  The splitters that
// k_bin_sort took from a sample of it cut its keys into the classes "equal to
// splitter i" and "between splitters".  The ties are written as runs (they need
// neither moving nor sorting); what lies between goes to a class's region of a
// scratch buffer, which one CTA sorts.  A class between splitters that is still
// above WS_BIN_CAP takes LSD radix passes over the digits that vary.  The bin's
// keys stay in keys_b and its classes in `tabs` (the way back finds a key's place
// by its class).  Bound by latency (two barriers and two reads of the keys: 20 us)
// up to about 2^22 keys, by the reads above.  Against LSD passes over whole bins
// and a bisection of every element in its bin by 64 CTAs, FP32 ws_prox, lambda
// 1e-2, us (the radix sort with a lookup by value before both):
//   2^26   50 % zeros 10240 (18890; 10900), 99 % 3670 (21620; 4010), 7 values 3280
//          (4700; 3720), 1000 values 3680 (6170; 3930), one value 1350 (2200; 2160)
//   2^24   50 % zeros 5500 (7410; 5590), 99 % 1170 (5170; 1260), 7 values 900 (1230; 1030)
//   2^20   1 % zeros 334 (394; 374), 50 % 300 (508; 369), 99 % 246 (596; 297)
// (the rest of such a call is the tree of merges around the huge cluster).  Spikes
// of a million different FP64 values that lie within 2^-30 of each other stay slower
// than under the radix sort (2^24: 5600; 1620): their classes take its passes, and
// a bisection for every element of the way back.
// ---------------------------------------------------------------------------
template <typename T>
struct OverSmem {
    typedef typename KeyOf<T>::K K;
    union {
        struct {                               // counting and placing: the table of the current bin
            K spl[OVER_SPL + 1];
            uint32_t start[2 * OVER_SPL + 2];  // start of every class in the bin
            uint32_t cnt[2 * OVER_SPL + 1];
            uint32_t place[OVER_SPL + 1];
        } split;
        struct {
            K key[WS_BIN_CAP];
            uint32_t whist[(OVER_NT / 32) * 256];
            uint32_t dcount[256], dstart[256], base[256];
        } sort;
    } u;
    int first[OVER_NT];   // first tile of every bin of a short list
    int wsum[OVER_NT / 32];
    int carry;
    int ent;
    unsigned long long diff;
};

// Sort of a class between splitters by the CTA, n <= WS_BIN_CAP keys: a bitonic
// network in shared memory (1280 keys 3 us; LSD passes over their four digits took 15).
template <typename T>
__device__ __noinline__ void over_sort_class(OverSmem<T>& s, const typename KeyOf<T>::K* src,
                                             typename KeyOf<T>::K* dst, int n) {
    typedef typename KeyOf<T>::K K;
    constexpr int NT = OVER_NT;
    const int t = threadIdx.x;
    K* key = s.u.sort.key;
    int m = 64;
    while (m < n) m <<= 1;
    __syncthreads();   // (the previous use of the shared memory is over)
    for (int i = t; i < m; i += NT) key[i] = i < n ? __ldcg(src + i) : ~(K)0;
    for (int k = 2; k <= m; k <<= 1)
        for (int d = k >> 1; d > 0; d >>= 1) {
            // (a warp's 32 pairs lie in one run of 64 keys while d < 64: only the steps across such runs, and the
            // first one after them, need the CTA)
            if (d >= 32 || k == 2) __syncthreads(); else __syncwarp();
            for (int q = t; q < m / 2; q += NT) {
                const int i = 2 * q - (q & (d - 1)), j = i + d;
                const K a = key[i], b = key[j];
                if ((a > b) == ((i & k) == 0)) { key[i] = b; key[j] = a; }
            }
        }
    __syncthreads();
    for (int i = t; i < n; i += NT) dst[i] = key[i];
}

template <typename T>
__global__ void __launch_bounds__(OVER_NT, 2) k_oversize(typename KeyOf<T>::K* ka,
                                                         const typename KeyOf<T>::K* __restrict__ kb,
                                                         typename KeyOf<T>::K* kt, int64_t n_keys, SortCtl* ctl,
                                                         OverBin* over, OverTab<typename KeyOf<T>::K>* tabs,
                                                         OverClass* items, OverClass* big, uint32_t* over_cnt,
                                                         uint64_t spin_limit, uint32_t* status) {
    typedef KeyOf<T> KO;
    typedef typename KO::K K;
    constexpr int NT = OVER_NT, ITEMS = WS_SORT_ITEMS, TILE = WS_SORT_TILE, P = KO::BITS / 8;
    extern __shared__ __align__(16) unsigned char over_smem_raw[];
    OverSmem<T>& s = *reinterpret_cast<OverSmem<T>*>(over_smem_raw);
    const int cnt = (int)ctl->over_count;
    if (cnt == 0 || ctl->abort) return;
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    GridBarrier bar{&ctl->over_bar, &ctl->abort, status, spin_limit, 0u, false};
    // tiles of the bins, in list order: a short list is numbered by every CTA for itself
    // (the first one writes the numbers down), a long one by one CTA
    auto number_tiles = [&](auto* list, int m) {
        if (t == 0) s.carry = 0;
        __syncthreads();
        for (int e0 = 0; e0 < m; e0 += NT) {
            const int e = e0 + t;
            const int nt = e < m ? (__ldcg(&list[e].n) + TILE - 1) / TILE : 0;
            int tot;
            const int ex = ws_block_excl_scan<NT, int>(nt, s.wsum, &tot);
            if (m <= NT) s.first[t] = ex;
            if (e < m && blockIdx.x == 0) __stcg(&list[e].first_tile, s.carry + ex);
            __syncthreads();
            if (t == 0) s.carry += tot;
            __syncthreads();
        }
        return s.carry;
    };
    int n_tiles = 0;
    const bool listed = cnt <= NT;
    if (listed) n_tiles = number_tiles(over, cnt);
    else {
        if (blockIdx.x == 0) number_tiles(over, cnt);
        if (!bar.sync()) return;
        n_tiles = __ldcg(&over[cnt - 1].first_tile) + (__ldcg(&over[cnt - 1].n) + TILE - 1) / TILE;
    }
    auto first_of = [&](int e) -> int { return listed ? s.first[e] : __ldcg(&over[e].first_tile); };
    // this CTA's tiles, contiguous: a table serves all tiles of its bin
    const int t0 = (int)((int64_t)n_tiles * blockIdx.x / gridDim.x);
    const int t1 = (int)((int64_t)n_tiles * (blockIdx.x + 1) / gridDim.x);
    auto first_entry = [&]() -> int {   // bin of tile t0
        int lo = 0, hi = cnt - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (first_of(mid) <= t0) lo = mid; else hi = mid - 1;
        }
        return lo;
    };
    const int e_first = t0 < t1 ? first_entry() : cnt;
    // 1. keys per class.  The counts of a bin's tiles are added up in shared memory.
    {
        int tile = t0;
        for (int e = e_first; tile < t1; ++e) {
            const int64_t st = over[e].start;
            const int ne = over[e].n, f = first_of(e), S = over[e].nspl;
            const K spl = t < OVER_SPL ? __ldcg(&tabs[e].spl[t]) : (K)0;   // (beyond S: not used)
            const int te = min(t1, f + (ne + TILE - 1) / TILE);
            __syncthreads();
            for (int j = t; j < 2 * OVER_SPL + 1; j += NT) s.u.split.cnt[j] = 0;
            if (t <= OVER_SPL) s.u.split.spl[t] = t < S ? spl : ~(K)0;
            __syncthreads();
            for (; tile < te; ++tile) {
                const int o0 = (tile - f) * TILE, n = min(TILE, ne - o0);
                K key[ITEMS];
#pragma unroll
                for (int k = 0; k < ITEMS; ++k) key[k] = t + k * NT < n ? __ldg(kb + st + o0 + t + k * NT) : (K)0;
                int cls[ITEMS];
                ws_over_classes<K, ITEMS>(s.u.split.spl, S, key, cls);
#pragma unroll
                for (int k = 0; k < ITEMS; ++k) {
                    if (k * NT >= n) break;   // (uniform)
                    const bool in = t + k * NT < n;
                    const unsigned crowd = ws_crowd(cls[k], in);
                    if ((crowd >> lane) & 1u) {
                        if (lane == __ffs((int)crowd) - 1) atomicAdd(&s.u.split.cnt[cls[k]], (uint32_t)__popc(crowd));
                    } else if (in) {
                        atomicAdd(&s.u.split.cnt[cls[k]], 1u);
                    }
                }
            }
            __syncthreads();
            for (int j = t; j < 2 * S + 1; j += NT)
                if (s.u.split.cnt[j]) atomicAdd(&tabs[e].cnt[j], s.u.split.cnt[j]);
        }
    }
    if (!bar.sync()) return;
    // 2. the runs of ties, and the keys between splitters into the regions of their classes
    {
        int tile = t0;
        for (int e = e_first; tile < t1; ++e) {
            const int64_t st = over[e].start;
            const int ne = over[e].n, f = first_of(e), S = over[e].nspl;
            const K spl = t < OVER_SPL ? __ldcg(&tabs[e].spl[t]) : (K)0;   // (beyond S: not used)
            const int te = min(t1, f + (ne + TILE - 1) / TILE);
            __syncthreads();
            if (t <= OVER_SPL) s.u.split.spl[t] = t < S ? spl : ~(K)0;
            {
                static_assert(2 * OVER_SPL + 2 <= OVER_NT && OVER_SPL < WS_BIN_CAP / 4, "a thread per class; the sample fits");
                const int all = t < 2 * OVER_SPL + 1 ? (int)__ldcg(&tabs[e].cnt[t]) : 0, c = t < 2 * S + 1 ? all : 0;
                const int ex = ws_block_excl_scan<NT, int>(c, s.wsum, nullptr);
                if (t < 2 * S + 2) s.u.split.start[t] = (uint32_t)ex;
                // (the bin's first tile lists the classes to sort)
                if (tile == f && (t & 1) == 0 && c > 1) {
                    OverClass oc = {};
                    oc.start = st + ex;
                    oc.n = c;
                    if (c <= WS_BIN_CAP) items[atomicAdd(&ctl->over_items, 1u)] = oc;
                    else big[atomicAdd(&ctl->over_big, 1u)] = oc;
                }
            }
            __syncthreads();
            for (; tile < te; ++tile) {
                const int o0 = (tile - f) * TILE, n = min(TILE, ne - o0);
                K key[ITEMS];
                int cls[ITEMS];
                uint32_t cr[ITEMS];   // class between splitters << 16 | rank among the tile's
#pragma unroll
                for (int k = 0; k < ITEMS; ++k) key[k] = t + k * NT < n ? __ldg(kb + st + o0 + t + k * NT) : (K)0;
                if (t <= OVER_SPL) s.u.split.cnt[t] = 0;
                __syncthreads();
                ws_over_classes<K, ITEMS>(s.u.split.spl, S, key, cls);
                bool any = false;
#pragma unroll
                for (int k = 0; k < ITEMS; ++k) {
                    cr[k] = 0xffffffffu;
                    if (t + k * NT < n && (cls[k] & 1) == 0) {
                        cr[k] = ((uint32_t)cls[k] << 15) | atomicAdd(&s.u.split.cnt[cls[k] >> 1], 1u);
                        any = true;
                    }
                }
                if (__syncthreads_or(any)) {
                    if (t <= S) {
                        const uint32_t c = s.u.split.cnt[t];
                        if (c) s.u.split.place[t] = s.u.split.start[2 * t] + atomicAdd(&tabs[e].cur[t], c);
                    }
                    __syncthreads();
#pragma unroll
                    for (int k = 0; k < ITEMS; ++k)
                        if (cr[k] != 0xffffffffu) {
                            const uint32_t c = cr[k] >> 16, p = s.u.split.place[c] + (cr[k] & 0xffffu);
                            // (a class of one key needs no sorting)
                            K* to = s.u.split.start[2 * c + 1] - s.u.split.start[2 * c] == 1u ? ka : kt;
                            if (p < (uint32_t)ne) to[st + p] = key[k];
                        }
                }
                for (int j = 0; j < S; ++j) {
                    const int a = max((int)s.u.split.start[2 * j + 1], o0), b = min((int)s.u.split.start[2 * j + 2], o0 + n);
                    const K v = s.u.split.spl[j];
                    for (int i = a + t; i < b; i += NT) ka[st + i] = v;
                }
                __syncthreads();
            }
        }
    }
    if (!bar.sync()) return;
    // 3. the classes between splitters
    const int n_items = (int)__ldcg(&ctl->over_items);
    for (int i = blockIdx.x; i < n_items; i += gridDim.x)
        over_sort_class<T>(s, kt + __ldcg(&items[i].start), ka + __ldcg(&items[i].start), __ldcg(&items[i].n));
    const int n_big = (int)__ldcg(&ctl->over_big);
    if (n_big == 0) return;   // (uniform over the grid)
    // 4. those above WS_BIN_CAP: LSD radix passes, which alternate between keys_a and a second
    // scratch buffer so that the last one writes keys_a
    K* kt2 = kt + n_keys;
    if (blockIdx.x == 0) number_tiles(big, n_big);
    if (!bar.sync()) return;
    const int b_tiles = __ldcg(&big[n_big - 1].first_tile) + (__ldcg(&big[n_big - 1].n) + TILE - 1) / TILE;
    // entry of a tile (all threads; ends synchronised)
    auto entry = [&](int tile) -> int {
        __syncthreads();
        if (t == 0) {
            int lo = 0, hi = n_big - 1;
            while (lo < hi) {
                const int mid = (lo + hi + 1) >> 1;
                if (__ldcg(&big[mid].first_tile) <= tile) lo = mid; else hi = mid - 1;
            }
            s.ent = lo;
            s.diff = 0;
        }
        __syncthreads();
        return s.ent;
    };
    auto passes_before = [&](unsigned long long diff, int p) {   // passes that the digits below p need
        int c = 0;
        for (int q = 0; q < p; ++q) c += ((diff >> (8 * q)) & 0xffull) != 0;
        return c;
    };
    // where pass i of m writes, and where it reads
    auto out_of = [&](int i, int m) -> K* { return ((m - 1 - i) & 1) ? kt2 : ka; };
    auto in_of = [&](int i, int m) -> const K* { return i == 0 ? kt : out_of(i - 1, m); };
    // bits that vary
    for (int tile = blockIdx.x; tile < b_tiles; tile += gridDim.x) {
        const int e = entry(tile);
        const int64_t st = __ldcg(&big[e].start);
        const int o0 = (tile - __ldcg(&big[e].first_tile)) * TILE, n = min(TILE, __ldcg(&big[e].n) - o0);
        const K k0 = __ldcg(kt + st);
        K d = 0;
        for (int i = t; i < n; i += NT) d |= __ldcg(kt + st + o0 + i) ^ k0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) d |= ws_shfl_xor_k(d, o);
        if (lane == 0 && d) atomicOr(&s.diff, (unsigned long long)d);
        __syncthreads();
        if (t == 0 && s.diff) {
            atomicOr(&big[e].diff, s.diff);
            atomicOr(&ctl->over_diff, s.diff);
        }
    }
    if (!bar.sync()) return;
    const unsigned long long all = __ldcg(&ctl->over_diff);
    for (int p = 0; p < P; ++p) {
        if (((all >> (8 * p)) & 0xffull) == 0) continue;   // (uniform over the grid)
        // digit counts of every tile
        for (int tile = blockIdx.x; tile < b_tiles; tile += gridDim.x) {
            const int e = entry(tile);
            const unsigned long long diff = __ldcg(&big[e].diff);
            if (((diff >> (8 * p)) & 0xffull) == 0) continue;
            const K* src = in_of(passes_before(diff, p), passes_before(diff, P)) + __ldcg(&big[e].start);
            const int o0 = (tile - __ldcg(&big[e].first_tile)) * TILE, n = min(TILE, __ldcg(&big[e].n) - o0);
            uint32_t* dcount = s.u.sort.dcount;
            if (t < 256) dcount[t] = 0;
            __syncthreads();
            for (int i = t; i < n; i += NT) atomicAdd(&dcount[(int)((__ldcg(src + o0 + i) >> (8 * p)) & 0xff)], 1u);
            __syncthreads();
            if (t < 256) __stcg(over_cnt + (size_t)tile * 256 + t, dcount[t]);
        }
        if (!bar.sync()) return;
        // counts -> first position of every (tile, digit), one CTA per class
        for (int e = blockIdx.x; e < n_big; e += gridDim.x) {
            const unsigned long long diff = __ldcg(&big[e].diff);
            if (((diff >> (8 * p)) & 0xffull) == 0) continue;
            uint32_t* c = over_cnt + (size_t)__ldcg(&big[e].first_tile) * 256;
            const int nt = (__ldcg(&big[e].n) + TILE - 1) / TILE;
            __syncthreads();
            uint32_t run = 0;
            if (t < 256) {
                int i = 0;
                for (; i + 8 <= nt; i += 8) {
                    uint32_t v[8];
#pragma unroll
                    for (int u = 0; u < 8; ++u) v[u] = __ldcg(c + (size_t)(i + u) * 256 + t);
#pragma unroll
                    for (int u = 0; u < 8; ++u) { __stcg(c + (size_t)(i + u) * 256 + t, run); run += v[u]; }
                }
                for (; i < nt; ++i) {
                    const uint32_t v = __ldcg(c + (size_t)i * 256 + t);
                    __stcg(c + (size_t)i * 256 + t, run);
                    run += v;
                }
            }
            const int ex = ws_block_excl_scan<NT, int>((int)run, s.wsum, nullptr);
            if (t < 256)
                for (int i = 0; i < nt; ++i) __stcg(c + (size_t)i * 256 + t, __ldcg(c + (size_t)i * 256 + t) + (uint32_t)ex);
        }
        if (!bar.sync()) return;
        // stable scatter
        for (int tile = blockIdx.x; tile < b_tiles; tile += gridDim.x) {
            const int e = entry(tile);
            const unsigned long long diff = __ldcg(&big[e].diff);
            if (((diff >> (8 * p)) & 0xffull) == 0) continue;
            const int i = passes_before(diff, p), m = passes_before(diff, P);
            const int64_t st = __ldcg(&big[e].start);
            const K* src = in_of(i, m) + st;
            K* dst = out_of(i, m) + st;
            const int ne = __ldcg(&big[e].n);
            const int o0 = (tile - __ldcg(&big[e].first_tile)) * TILE, n = min(TILE, ne - o0);
            K key[ITEMS];
            uint32_t dg[ITEMS];
            bool valid[ITEMS];
            int pos[ITEMS];
#pragma unroll
            for (int k = 0; k < ITEMS; ++k) {
                const int q = w * 32 * ITEMS + k * 32 + lane;
                valid[k] = q < n;
                key[k] = valid[k] ? __ldcg(src + o0 + q) : (K)0;
                dg[k] = (uint32_t)((key[k] >> (8 * p)) & 0xff);
            }
            uint32_t* base = s.u.sort.base;
            if (t < 256) base[t] = __ldcg(over_cnt + (size_t)tile * 256 + t);
            ws_rank_digits<NT, ITEMS, 1>(dg, valid, pos, s.u.sort.whist, s.u.sort.dcount, s.u.sort.dstart);
#pragma unroll
            for (int k = 0; k < ITEMS; ++k)
                if (valid[k]) {
                    const uint32_t q = base[dg[k]] + (uint32_t)pos[k] - s.u.sort.dstart[dg[k]];
                    if (q < (uint32_t)ne) dst[q] = key[k];
                }
        }
        if (!bar.sync()) return;
    }
    // classes of equal keys
    for (int tile = blockIdx.x; tile < b_tiles; tile += gridDim.x) {
        const int e = entry(tile);
        if (__ldcg(&big[e].diff) != 0) continue;
        const int64_t st = __ldcg(&big[e].start);
        const int o0 = (tile - __ldcg(&big[e].first_tile)) * TILE, n = min(TILE, __ldcg(&big[e].n) - o0);
        for (int i = t; i < n; i += NT) ka[st + o0 + i] = __ldcg(kt + st + o0 + i);
    }
}

// Shared memory of the plan kernel for hist_cap bins counted locally.
size_t plan_smem(int hist_cap) { return sizeof(MapTab) + 4 * (size_t)hist_cap; }

}  // namespace

// Launch shapes of a plan's sort (and the kernels' shared-memory limits on
// the plan's device).  max_bins: of its longest segment; samp_max: log2 of the
// largest number of samples per tile.
template <typename T, typename B, bool TOP>
static cudaError_t sort_prepare(int max_bins, int n_tiles, WsSortShape* sh) {
    constexpr int HIST_MAX = 45056;
    auto* kp = k_sort_plan<T, B>;
    auto* k1 = k_part<T, B, true, TOP>;
    auto* k2 = k_part<T, B, false, TOP>;
    auto* ko = k_oversize<T>;
    const size_t ksm = sizeof(PartSmem<T, B>);
    cudaError_t e = cudaFuncSetAttribute(kp, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)plan_smem(HIST_MAX));
    if (!e) e = cudaFuncSetAttribute(k1, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ksm);
    if (!e) e = cudaFuncSetAttribute(k2, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ksm);
    auto *kb0 = k_bin_sort<T, false>, *kb1 = k_bin_sort<T, true>;
    if (!e) e = cudaFuncSetAttribute(kb0, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(BinSmem<T>));
    if (!e) e = cudaFuncSetAttribute(kb1, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(BinSmem<T>));
    if (!e) e = cudaFuncSetAttribute(ko, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(OverSmem<T>));
    if (e) return e;
    int dev = 0, sms = 0, np = 0, n1 = 0, no = 0;
    if ((e = cudaGetDevice(&dev))) return e;
    if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev))) return e;
    // shared words of the plan kernel (one CTA per SM): the bins of the longest
    // segment and the CTA's samples, as far as they fit
    sh->plan_grid = std::min(sms, n_tiles);
    const int64_t keep = ((int64_t)((n_tiles + sh->plan_grid - 1) / sh->plan_grid) << sh->samp_max) *
                         (int64_t)(sizeof(typename KeyOf<T>::K) / 4);
    sh->hist_cap = (int)std::min<int64_t>(std::max<int64_t>(std::max<int64_t>(max_bins, 1024), keep), HIST_MAX);
    if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&np, kp, PLAN_NT, plan_smem(sh->hist_cap)))) return e;
    if (np < 1) return cudaErrorInvalidConfiguration;
    if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n1, k1, WS_SORT_NT, ksm))) return e;
    if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&no, ko, OVER_NT, sizeof(OverSmem<T>)))) return e;
    sh->part_grid = std::max(1, sms * n1);
    sh->over_grid = std::max(1, sms * no);
    sh->out_extra = std::min((sizeof(T) == 4 ? 6 : 3) * sms, n_tiles);   // (as many as are resident at once)
    return cudaSuccess;
}

template <typename T>
cudaError_t ws_sort_prepare(int max_bins, int n_tiles, int samp_max, WsSortShape* sh) {
    sh->wide = max_bins > 65536;
    sh->samp_max = samp_max;
    sh->max_bins = max_bins;
    if (max_bins > WS_BINS_RANK) return sort_prepare<T, uint32_t, true>(max_bins, n_tiles, sh);
    return sh->wide ? sort_prepare<T, uint32_t, false>(max_bins, n_tiles, sh)
                    : sort_prepare<T, uint16_t, false>(max_bins, n_tiles, sh);
}

template <typename T, typename B, bool TOP>
static cudaError_t sort_run(const LargeWork<T>& W, const T* values, bool way_back, uint32_t* status,
                            uint64_t spin_limit, cudaStream_t st) {
    typedef typename KeyOf<T>::K K;
    cudaError_t e = cudaMemsetAsync(W.ctl, 0, W.sort_zero_bytes, st);
    if (e) return e;
    const WsSortShape& sh = W.sort_shape;
    // bins of the keys: in the caller's order, then in the first pass's
    B* bins = (B*)W.bins;
    B* bins2 = bins + W.n_keys;
    {
        int n_tiles = W.n_sort_tiles, n_lseg = W.n_lseg, hc = sh.hist_cap, sm = sh.samp_max, mb = sh.max_bins;
        const TileDesc* tiles = W.sort_tiles;
        const LargeSeg* lsegs = W.lsegs;
        void* args[] = {(void*)&values, &tiles, &n_tiles, &lsegs, &n_lseg, (void*)&W.ctl, (void*)&W.seg_hi,
                        (void*)&W.seg_lo, (void*)&W.seg_en, (void*)&W.cells, (void*)&W.bin_cnt, &bins,
                        (void*)&W.bin_start, (void*)&W.cur1, (void*)&W.cur2, (void*)&W.seg_emin, &mb, &hc, &sm, &spin_limit,
                        &status};
        WS_LAUNCH(W.prof, WSK_SORT_PLAN, st,
                  e = cudaLaunchCooperativeKernel((const void*)k_sort_plan<T, B>,
                                                  dim3(sh.plan_grid), dim3(PLAN_NT), args,
                                                  plan_smem(sh.hist_cap), st));
        if (e) return e;
    }
    const size_t ksm = sizeof(PartSmem<T, B>);
    const int grid = std::min(sh.part_grid, W.n_sort_tiles);
    const T* no_values = nullptr;
    K* no_keys = nullptr;
    B* no_bins = nullptr;
    WS_LAUNCH(W.prof, WSK_PARTITION, st,
              ws_launch_chain(k_part<T, B, true, TOP>, grid, WS_SORT_NT, ksm, st, values, no_keys, bins, W.keys_a,
                              W.keys_b, bins2, way_back ? W.map1 : PassMap{}, W.sort_tiles, W.n_sort_tiles, W.lsegs,
                              W.cur1, W.ctl));
    if (W.two_level)
        WS_LAUNCH(W.prof, WSK_PARTITION, st,
                  ws_launch_chain(k_part<T, B, false, TOP>, grid, WS_SORT_NT, ksm, st, no_values, W.keys_a, bins2, no_keys,
                                  W.keys_b, no_bins, way_back ? W.map2 : PassMap{}, W.sort_tiles, W.n_sort_tiles,
                                  W.lsegs, W.cur2, W.ctl));
    WS_LAUNCH(W.prof, WSK_BIN_SORT, st,
              ws_launch_chain(way_back ? k_bin_sort<T, true> : k_bin_sort<T, false>, W.n_bins, BIN_NT,
                              sizeof(BinSmem<T>), st, W.keys_b, W.keys_a, W.bin_seg, W.lsegs, W.bin_start, W.bin_cnt,
                              W.bin_idx, W.ctl, W.over, reinterpret_cast<OverTab<K>*>(W.over_tabs), W.n_keys));
    {
        K* ka = W.keys_a;
        K* kb = W.keys_b;
        K* kt = reinterpret_cast<K*>(W.pairs_b);   // (two buffers of n_keys: a pair takes at least two keys)
        static_assert(sizeof(OutPair<T>) >= 2 * sizeof(K), "the scratch fits");
        OverTab<K>* tabs = reinterpret_cast<OverTab<K>*>(W.over_tabs);
        void* args[] = {&ka, &kb, &kt, (void*)&W.n_keys, (void*)&W.ctl, (void*)&W.over, &tabs, (void*)&W.over_items,
                        (void*)&W.over_big, (void*)&W.over_cnt, &spin_limit, &status};
        WS_LAUNCH(W.prof, WSK_OVERSIZE, st,
                  e = cudaLaunchCooperativeKernel((const void*)k_oversize<T>,
                                                  dim3(std::min(sh.over_grid, W.n_sort_tiles)), dim3(OVER_NT), args,
                                                  sizeof(OverSmem<T>),
                                                  st));
        if (e) return e;
    }
    return cudaGetLastError();
}

template <typename T>
cudaError_t ws_large_sort(const LargeWork<T>& W, const T* values, bool way_back, uint32_t* status,
                          uint64_t spin_limit, cudaStream_t st, typename KeyOf<T>::K** sorted) {
    *sorted = nullptr;
    if (W.n_sort_tiles == 0) return cudaSuccess;
    *sorted = W.keys_a;
    if (W.sort_shape.max_bins > WS_BINS_RANK)
        return sort_run<T, uint32_t, true>(W, values, way_back, status, spin_limit, st);
    return W.sort_shape.wide ? sort_run<T, uint32_t, false>(W, values, way_back, status, spin_limit, st)
                             : sort_run<T, uint16_t, false>(W, values, way_back, status, spin_limit, st);
}

template cudaError_t ws_sort_prepare<float>(int, int, int, WsSortShape*);
template cudaError_t ws_sort_prepare<double>(int, int, int, WsSortShape*);
template cudaError_t ws_large_sort<float>(const LargeWork<float>&, const float*, bool, uint32_t*, uint64_t,
                                          cudaStream_t, uint32_t**);
template cudaError_t ws_large_sort<double>(const LargeWork<double>&, const double*, bool, uint32_t*, uint64_t,
                                           cudaStream_t, uint64_t**);
