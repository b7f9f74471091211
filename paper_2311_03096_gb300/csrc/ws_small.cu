// ws_small.cu -- fused single-CTA prox for short segments (n <= 4096, float
// and double): one CTA loads a segment once, sorts (key, index)
// pairs in shared memory, builds the exact hull, and writes values and cluster
// ids straight to their original positions.  HBM traffic is the I/O floor:
// read w, write out and id (12 B/element for float).  The lean kernel
// (k_small) builds the hull by Imminent Collisions rounds with a fallback to
// chains and bridge trees; the general kernel (k_small_general) takes the rare
// segments whose fixed-point sums need 128 bits.
#include "ws_hull.cuh"
#include "ws_kernels.cuh"

namespace {

// Shared memory of one segment, laid out so that three CTAs fit on an SM:
// buffers whose lifetimes do not overlap share storage.
//   r1: digit counters of the sort  |  hull vertex list + cluster-start bits
//   r2: sort keys (dead after the prefix sums)  |  chunk hulls  |  values
template <typename T, int NT, int M>
struct SmallSmem {
    typedef typename KeyOf<T>::K K;
    static constexpr int CAP = NT * M;
    static_assert(32 % M == 0 || M % 32 == 0, "a thread's marks must lie in one 32-bit word");
    uint16_t idx[CAP];
    TilePrefix<NT, M> pre;  // fixed-point prefix sums of the sorted segment
    union {
        struct {
            uint32_t whist[(NT / 32) * 256];
            uint32_t dcount[256], dstart[256];
        } sort;
        uint32_t cnt[CAP];              // bucket counts, then starts: two per word
        struct {
            uint16_t V[CAP + 2];        // hull vertices (points)
            uint32_t mark[CAP / 32];    // bit p: a cluster starts at sorted position p
            uint16_t multi[CAP / 2];    // clusters of two or more elements
        } ids;
    } r1;
    union {
        K keys[CAP];
        HullSmem<NT, M> hull;
        T val[CAP];
    } r2;
    int wsum_i[NT / 32];
    wsh::Ends ends;
    K kmin, kmax;
    int flags;
    int emin;
    int n_multi;
    SegConst sc, sct;
    float muq, muqt;
    int fast, fastt;
};

// One bucket of the interpolation bucket sort, entries [b0, b1) of (keys, idx)
// through the slot maps kp and ip, by key (ties may end in any order): up to
// four entries by a sorting network in registers, more by insertion.
template <typename K, typename KP, typename IP>
__device__ __forceinline__ void small_sort_bucket(int b0, int b1, K* keys, uint16_t* idx, KP kp, IP ip) {
    if (b1 - b0 <= 4) {
        K k[4];
        uint16_t x[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const bool in = b0 + j < b1;
            k[j] = in ? keys[kp(b0 + j)] : ~(K)0;
            x[j] = in ? idx[ip(b0 + j)] : (uint16_t)0;
        }
        auto cs = [&](int a, int b) {
            const bool sw = k[a] > k[b];
            const K ka = sw ? k[b] : k[a], kb = sw ? k[a] : k[b];
            const uint16_t xa = sw ? x[b] : x[a], xb = sw ? x[a] : x[b];
            k[a] = ka; k[b] = kb; x[a] = xa; x[b] = xb;
        };
        cs(0, 1); cs(2, 3); cs(0, 2); cs(1, 3); cs(1, 2);
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (b0 + j < b1) { keys[kp(b0 + j)] = k[j]; idx[ip(b0 + j)] = x[j]; }
        return;
    }
    for (int a = b0 + 1; a < b1; ++a) {
        const K kk = keys[kp(a)];
        const uint16_t ii = idx[ip(a)];
        int j = a - 1;
        while (j >= b0 && keys[kp(j)] > kk) {
            keys[kp(j + 1)] = keys[kp(j)];
            idx[ip(j + 1)] = idx[ip(j)];
            --j;
        }
        keys[kp(j + 1)] = kk;
        idx[ip(j + 1)] = ii;
    }
}

// The general one-CTA prox of one segment (every input, including values
// whose fixed-point sums need 128 bits): used for the segments the lean
// kernel below sends here.
template <typename T, int NT, int M>
__device__ __forceinline__ void small_general_segment(SmallSmem<T, NT, M>& s, int seg, const T* __restrict__ values,
                                                      const int64_t* __restrict__ offsets,
                                                      const WsLambda& lambdas, T* out, int32_t* ids,
                                                      int64_t* n_clusters, int fp64, const WsEpi& ep,
                                                      int ic_cap, uint32_t* status) {
    typedef KeyOf<T> KO;
    typedef typename KO::K K;
    typedef SmallSmem<T, NT, M> S;
    constexpr int CAP = S::CAP;
    constexpr int ITEMS = M;   // items per thread in the sort
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;

    const int64_t a0 = offsets[seg];
    const int n = (int)(offsets[seg + 1] - a0);
    const double lam = lambdas.at(seg);
    if (!(lam >= 0.0) || !(lam <= 1.7976931348623157e308)) {
        if (t == 0) ws_flag(status, WS_STATUS_BAD_LAMBDA);
        return;
    }
    if (n <= 0 || n > CAP) {
        if (n > CAP && t == 0) ws_flag(status, WS_STATUS_INTERNAL);
        if (n == 0 && t == 0 && n_clusters) n_clusters[seg] = 0;
        return;
    }

    // ---- load (striped per warp, coalesced), map to keys, check finiteness
    if (t == 0) { s.flags = 0; s.emin = 0x7fffffff; s.n_multi = 0; }
    __syncthreads();
    bool bad = false;
#pragma unroll
    for (int k = 0; k < ITEMS; ++k) {
        int p = w * 32 * ITEMS + k * 32 + lane;
        if (p < n) {
            T v = values[a0 + p];
            bad |= !ws_isfinite(v);
            s.r2.keys[p] = KO::to_key(v);
            s.idx[p] = (uint16_t)p;
        }
    }
    if (bad) atomicOr(&s.flags, 1);
    __syncthreads();
    if (s.flags) {
        if (t == 0) ws_flag(status, WS_STATUS_NONFINITE);
        return;
    }
    if (n == 1) {
        if (t == 0) {
            const T x = values[a0];   // d = 1: no shift (the 1/(d-1) factor is vacuous)
            out[a0] = fp64 ? (T)ws_epilogue<double>((double)x, 0.0, ep.beta, ep.gamma, ep.on != 0)
                           : (T)ws_epilogue<float>((float)x, 0.0f, ep.beta_f, ep.gamma_f, ep.on != 0);
            if (ids) ids[a0] = 0;
            if (n_clusters) n_clusters[seg] = 1;
        }
        return;
    }

    // ---- sort (key, idx) in shared memory: the interpolation bucket sort of
    // k_small (two buckets per element; eight radix passes took 42 us of a
    // single FP64 segment of 4096), LSD radix passes where a bucket is large
    bool radix;
    {
        K kk[ITEMS], lo = ~(K)0, hi = 0;
        if (t == 0) { s.kmin = ~(K)0; s.kmax = 0; }
        for (int i = t; i < n; i += NT) s.r1.cnt[i] = 0;
#pragma unroll
        for (int k = 0; k < ITEMS; ++k) {
            const int p = t + k * NT;
            kk[k] = p < n ? s.r2.keys[p] : (K)0;
            if (p < n) { lo = min(lo, kk[k]); hi = max(hi, kk[k]); }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            lo = min(lo, ws_shfl_xor_k(lo, o));
            hi = max(hi, ws_shfl_xor_k(hi, o));
        }
        __syncthreads();
        if (lane == 0) { ws_atomic_min_k(&s.kmin, lo); ws_atomic_max_k(&s.kmax, hi); }
        __syncthreads();
        const float f0 = (float)KO::from_key(s.kmin), span = (float)KO::from_key(s.kmax) - f0;
        const float scale = (span > 0.0f && span <= 3.0e38f) ? (float)(2 * n) / span : 0.0f;
        uint32_t br[ITEMS];   // bucket << 16 | rank
#pragma unroll
        for (int k = 0; k < ITEMS; ++k) {
            if (t + k * NT < n) {
                const float f = ((float)KO::from_key(kk[k]) - f0) * scale;
                const uint32_t b = (uint32_t)min(2 * n - 1, max(0, (int)f)), up = (b & 1u) << 4;
                const uint32_t old = atomicAdd(&s.r1.cnt[b >> 1], 1u << up);
                br[k] = (b << 16) | ((old >> up) & 0xffffu);
            }
        }
        __syncthreads();
        int sum = 0, big = 0;
        uint32_t c[M], multi = 0;   // (multi: bit j, bucket 2 t M + j holds two or more)
#pragma unroll
        for (int i = 0; i < M; ++i) {   // (this thread's 32 consecutive buckets)
            c[i] = t * M + i < n ? s.r1.cnt[t * M + i] : 0u;
            const int c0 = (int)(c[i] & 0xffffu), c1 = (int)(c[i] >> 16);
            sum += c0 + c1;
            big = max(big, max(c0, c1));
            multi |= (c0 >= 2 ? 1u : 0u) << (2 * i) | (c1 >= 2 ? 2u : 0u) << (2 * i);
        }
        int run = ws_block_excl_scan<NT, int>(sum, s.wsum_i, nullptr);
#pragma unroll
        for (int i = 0; i < M; ++i) {
            if (t * M + i < n) s.r1.cnt[t * M + i] = (uint32_t)run | ((uint32_t)(run + (int)(c[i] & 0xffffu)) << 16);
            run += (int)(c[i] & 0xffffu) + (int)(c[i] >> 16);
        }
        radix = __syncthreads_or(big > 32);
        if (!radix) {
            auto start = [&](int b) { return (int)((s.r1.cnt[b >> 1] >> ((b & 1) << 4)) & 0xffffu); };
#pragma unroll
            for (int k = 0; k < ITEMS; ++k)
                if (t + k * NT < n) {
                    const int q = start((int)(br[k] >> 16)) + (int)(br[k] & 0xffffu);
                    s.r2.keys[q] = kk[k];
                    s.idx[q] = (uint16_t)(t + k * NT);
                }
            __syncthreads();
            // (spread over the CTA: the fullest buckets are neighbours)
            uint16_t* list = reinterpret_cast<uint16_t*>(&s.pre);   // (not in use yet; at most n / 2 entries)
            static_assert(sizeof(s.pre) >= sizeof(uint16_t) * CAP / 2, "the list fits");
            if (multi) {
                int at = atomicAdd(&s.n_multi, __popc(multi));
                for (; multi; multi &= multi - 1) list[at++] = (uint16_t)(2 * t * M + __ffs((int)multi) - 1);
            }
            __syncthreads();
            for (int i = t; i < s.n_multi; i += NT) {
                const int b = list[i];
                small_sort_bucket<K>(start(b), b + 1 < 2 * n ? start(b + 1) : n, s.r2.keys, s.idx,
                                     [](int p) { return p; }, [](int p) { return p; });
            }
            __syncthreads();
        }
    }
    for (int pass = 0; radix && pass < KO::BITS / 8; ++pass) {
        K kk[ITEMS];
        uint16_t ii[ITEMS];
        uint32_t dg[ITEMS];
        bool valid[ITEMS];
        int pos[ITEMS];
#pragma unroll
        for (int k = 0; k < ITEMS; ++k) {
            int p = w * 32 * ITEMS + k * 32 + lane;
            valid[k] = p < n;
            kk[k] = valid[k] ? s.r2.keys[p] : (K)0;
            ii[k] = valid[k] ? s.idx[p] : (uint16_t)0;
            dg[k] = (uint32_t)((kk[k] >> (8 * pass)) & 0xff);
        }
        __syncthreads();
        ws_rank_digits<NT, ITEMS, 1>(dg, valid, pos, s.r1.sort.whist, s.r1.sort.dcount, s.r1.sort.dstart);
#pragma unroll
        for (int k = 0; k < ITEMS; ++k)
            if (valid[k]) { s.r2.keys[pos[k]] = kk[k]; s.idx[pos[k]] = ii[k]; }
        __syncthreads();
    }

    // ---- fixed point and prefix sums (blocked: thread t owns sorted [t*M, t*M+M))
    int64_t q0;
    i128 total;
    int bsh;
    K kr[M];
    int emin = 0x7fffffff;   // smallest effective exponent of a nonzero value
#pragma unroll
    for (int i = 0; i < M; ++i) {
        kr[i] = (t * M + i < n) ? s.r2.keys[t * M + i] : (K)0;
        const T x = KO::from_key(kr[i]);
        if (t * M + i < n && x != (T)0) emin = min(emin, ws_eff_exp(x));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) emin = min(emin, __shfl_xor_sync(WS_FULL_MASK, emin, o));
    if (lane == 0) atomicMin(&s.emin, emin);
    __syncthreads();
    const K kfirst = s.r2.keys[0], klast = s.r2.keys[n - 1];
    const T xlo = KO::from_key(kfirst), xhi = KO::from_key(klast);
    const int emax = ws_fix_scale<T>(max(ws_eff_exp(xlo), ws_eff_exp(xhi)), s.emin);
    // (two warps: FP64 divisions take a few microseconds each)
    if (t == 0) {
        s.sc = ws_seg_const<T>(n, lam, emax);
        bool f;
        s.muq = ws_muq_f(s.sc, f);
        s.fast = f ? 1 : 0;
    }
    if (t == 32) {
        const int sh0 = ws_eff_exp(xlo) - emax + KO::FIX_OFS;
        s.sct = ws_seg_const_L(n, lam, KO::L_BASE - emax - (sh0 > 0 ? sh0 : 0));
        bool f;
        s.muqt = ws_muq_f(s.sct, f);
        s.fastt = f ? 1 : 0;
    }
    // (the prefix sums end with a barrier; the keys' storage is reused from here on)
    // this thread's entry of the chain thresholds at the scale the segment's mode
    // uses; the prefix stores it after its first barrier (the keys are dead then)
    static_assert(M * M <= NT, "one threshold entry per thread");
    int thr_v = 0;
    if (t < M * M) {
        int shb;
        const bool tbin = ws_tile_binade<T>(kfirst, klast, n, emax, shb);
        uint64_t mlam;
        int sx;
        ws_thr_consts(lam, KO::L_BASE - emax - (tbin && shb > 0 ? shb : 0), mlam, sx);
        thr_v = ws_thr_entry<M>(t, mlam, sx, n > 1 ? (uint64_t)(n - 1) : 1ull);
    }
    const int mode = ws_tile_prefix<T, NT, M>(s.pre, kr, kfirst, klast, n, emax, q0, total, bsh,
                                              t < M * M ? s.r2.hull.thr + t : nullptr, thr_v);
    const SegConst& sc = s.sc;

    // ---- exact hull (in-CTA merge)
    int nv;
    if (mode == WS_TILE_BINADE) {
        TilePtsDev<M> P = ws_dev_pts<M>(s.pre.s64, s.muqt, s.fastt != 0, (uint64_t)(klast - kfirst), n, s.sct);
        P.thr = s.r2.hull.thr;
        ws_cta_hull<NT, M, TilePtsDev<M>, true>(s.r2.hull, n, P, s.sct, &nv);
    } else if (mode == WS_TILE_NARROW) {
        const uint64_t range = (uint64_t)(ws_fixed<T>(xhi, emax) - q0);
        TilePtsDev<M> P = ws_dev_pts<M>(s.pre.s64, s.muq, s.fast != 0, range, n, sc);
        P.thr = s.r2.hull.thr;
        ws_cta_hull<NT, M, TilePtsDev<M>, true>(s.r2.hull, n, P, sc, &nv);
    } else {
        static_assert(NT == wsh::NT && M == wsh::M, "the rounds' tile");
        const TilePtsWide<M> P{s.pre.s64, s.pre.base, s.muq, s.fast != 0};
        if (ic_cap <= 0 || !wsh::wide_rounds(s.r2.hull, s.ends, n, P, sc, ic_cap, &nv))
            ws_cta_hull<NT, M>(s.r2.hull, n, P, sc, &nv);
    }
    auto X = [&](int p) -> i128 { return ws_tile_X<M>(s.pre.s64, s.pre.base, mode, q0, bsh, p); };
    {
        int l = s.r2.hull.lo[t], h = s.r2.hull.hi[t], o = s.r2.hull.cum[t];
        for (int i = l; i < h; ++i) s.r1.ids.V[o + (i - l)] = s.r2.hull.H[i * NT + t];
    }
    for (int i = t; i < CAP / 32; i += NT) s.r1.ids.mark[i] = 0u;
    __syncthreads();   // the chunk hulls are dead from here on (their storage holds the values)
    const int c = nv - 1;
    if (s.r1.ids.V[0] != 0 || s.r1.ids.V[c] != n) { if (t == 0) ws_flag(status, WS_STATUS_INTERNAL); }

    // ---- cluster values (a one-element cluster reads its weight back from the input).
    // FP32 arithmetic on deviation tiles: mean = x_first + (sum of deviations / n)
    // 2^-L, all terms exact but the last conversions (error a few FP32 ulps of
    // max |w|); otherwise from the exact 128-bit cluster sum.
    const bool dev32 = !fp64 && mode != WS_TILE_WIDE;
    const int Ldev = mode == WS_TILE_BINADE ? s.sct.L : sc.L;
    const float x0f = (float)xlo;
    // Single weights first, four of a thread's on their way together; the
    // other clusters from a list, so that no lane waits for a neighbour's
    // division.
    if (t == 0) s.n_multi = 0;
    __syncthreads();
    constexpr int VU = 4;
    for (int r0 = t; r0 < c; r0 += NT * VU) {
        T xv[VU];
#pragma unroll
        for (int u = 0; u < VU; ++u) {
            const int r = min(r0 + u * NT, c - 1), a = s.r1.ids.V[r];
            xv[u] = s.r1.ids.V[r + 1] - a == 1 ? __ldg(values + a0 + s.idx[a]) : (T)0;
        }
#pragma unroll
        for (int u = 0; u < VU; ++u) {
            const int r = r0 + u * NT;
            if (r >= c) break;
            const int a = s.r1.ids.V[r], b = s.r1.ids.V[r + 1];
            atomicOr(&s.r1.ids.mark[a >> 5], 1u << (a & 31));
            if (b - a > 1) { s.r1.ids.multi[atomicAdd(&s.n_multi, 1)] = (uint16_t)r; continue; }
            s.r2.val[r] = dev32 ? (T)ws_epilogue<float>((float)xv[u], sc.mu_f * (float)(n - a - b), ep.beta_f,
                                                        ep.gamma_f, ep.on != 0)
                                : ValueOut<T>::value((i128)0, a, b, xv[u], sc, fp64 != 0, ep);
        }
    }
    __syncthreads();
    for (int q = t; q < s.n_multi; q += NT) {
        const int r = s.r1.ids.multi[q], a = s.r1.ids.V[r], b = s.r1.ids.V[r + 1];
        if (dev32) {
            const float mean = x0f + ldexpf(ws_u64_to_float((uint64_t)(s.pre.s64[ws_sidx<M>(b)] -
                                                                       s.pre.s64[ws_sidx<M>(a)])) /
                                                (float)(b - a),
                                            -Ldev);
            s.r2.val[r] = (T)ws_epilogue<float>(mean, sc.mu_f * (float)(n - a - b), ep.beta_f, ep.gamma_f,
                                                ep.on != 0);
        } else {
            s.r2.val[r] = ValueOut<T>::value(X(b) - X(a), a, b, (T)0, sc, fp64 != 0, ep);
        }
    }
    __syncthreads();

    // ---- cluster id of every sorted position, then scatter to the original order
    const uint32_t mymarks = (s.r1.ids.mark[(t * M) >> 5] >> ((t * M) & 31)) & (uint32_t)((1ull << M) - 1ull);
    int tot;
    int run = ws_block_excl_scan<NT, int>(__popc(mymarks), s.wsum_i, &tot);
    for (int i = 0; i < M; ++i) {
        int p = t * M + i;
        if (p < n) {
            run += (mymarks >> i) & 1u;
            int r = run - 1;
            int64_t o = a0 + s.idx[p];
            out[o] = s.r2.val[r];
            if (ids) ids[o] = r;
        }
    }
    if (t == 0 && n_clusters) n_clusters[seg] = c;
}

template <typename T, int NT, int M>
__global__ void __launch_bounds__(NT, 3) k_small_general(const T* __restrict__ values,
                                                      const int64_t* __restrict__ offsets,
                                                      const int32_t* __restrict__ gen_list,
                                                      const int32_t* __restrict__ gen_count,
                                                      const WsLambda lambdas, T* out, int32_t* ids,
                                                      int64_t* n_clusters, int fp64, const WsEpi ep,
                                                      int ic_cap, uint32_t* status) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    SmallSmem<T, NT, M>& s = *reinterpret_cast<SmallSmem<T, NT, M>*>(smem_raw);
    ws_chain();
    const int cnt = *gen_count;
    for (int i = blockIdx.x; i < cnt; i += gridDim.x) {
        small_general_segment<T, NT, M>(s, gen_list[i], values, offsets, lambdas, out, ids, n_clusters, fp64, ep,
                                        ic_cap, status);
        __syncthreads();
    }
}

// ---------------------------------------------------------------------------
// The lean one-CTA prox: keys and their original positions sorted in shared
// memory, then the hull of the sorted segment by the Imminent Collisions
// rounds with the chain-and-tree fallback (ws_hull.cuh), cluster ids from the
// cluster-start bitmap, values scattered back through the positions.
// Segments whose prefix sums need 128 bits (or whose bridge walks are too
// long) are appended to gen_list for the general kernel above.
// Bound by issue (0.64; 470 thread instructions per weight), instruction fetches
// and the barriers between its phases.  Rows of the MLP (8202 of 3072 or 4096, lambda 1e-3 .. 1):
// 809 us with three CTAs per SM (74 KB of shared memory, 80 registers), one
// decision per boundary and round and a value loop that searched the bitmap;
// 676 with the rounds of ws_hull.cuh, 601 with four CTAs (57 KB, 64 registers), 579
// with the loops over shared memory rolled (fetching instructions is the first stall).
// ---------------------------------------------------------------------------
template <typename T>
struct LeanSmem {
    typedef typename KeyOf<T>::K K;
    static constexpr int CAP = wsh::TILE;               // 4096 elements, float and double
    // Arrays read in blocks of 16 consecutive entries per thread are padded
    // (keys: one slot per 16, 16-bit arrays: two) so those reads do not
    // collide in the shared-memory banks; see kpad / ipad.
    uint16_t idx[CAP + CAP / 8];                        // original position of every sorted element
    // One after the other: the sort; the prefix sums and the rounds.  At the
    // end the prefix-sum slot of a cluster's first point takes the cluster's
    // value (FP32: and id), and the lane stacks' storage the first point of
    // every original position's cluster.  Four CTAs then fit on an SM (FP32).
    union {
        struct {
            K keys[CAP + CAP / 16];
            union {
                uint32_t cnt[CAP + CAP / 16];   // bucket counts, then starts: two per word (words padded like the keys: kpad)
                struct {
                    uint32_t whist[(wsh::NT / 32) * 256];
                    uint32_t dcount[256], dstart[256];
                } radix;
            };
        } sort;
        wsh::Smem h;
    } u;
    uint16_t cid[sizeof(T) == 8 ? CAP : 1];   // FP64: cluster id by first point
    K kmin, kmax;
    int bmax;
    int wsumi[wsh::NT / 32];
    uint32_t starts[wsh::TILE / 32 + 1];   // bit p: a cluster starts at sorted position p
    TileScale ts;
    SegConst sc;    // the segment's global fixed-point scale (cluster values)
    int64_t t11;    // round-1 gap threshold (tile units)
    int flags, emin;
    int inexact;    // the fixed point truncates some values
};

// Exclusive scan of one int per thread over the CTA with a single barrier:
// every thread reads the warp totals itself.  wsum (one word per warp) must
// not be written again before the next barrier of the caller.
__device__ __forceinline__ int lean_excl_scan(int v, int* wsum, int* total) {
    constexpr int NW = wsh::NT / 32;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int inc = ws_warp_incl_scan<int>(v);
    if (lane == 31) wsum[w] = inc;
    __syncthreads();
    int base = 0, tot = 0;
#pragma unroll
    for (int k = 0; k < NW; ++k) {
        const int x = wsum[k];
        base += k < w ? x : 0;
        tot += x;
    }
    *total = tot;
    return base + inc - v;
}

__device__ __forceinline__ int lean_kpad(int p) { return p + (p >> 4); }          // keys, counts
__device__ __forceinline__ int lean_ipad(int p) { return p + ((p >> 4) << 1); }   // 16-bit arrays

// The rare paths of k_small live out of line so that the common path's code
// stays compact in the instruction cache.  All threads of the CTA call each.

// LSD radix sort, 8-bit digits, of the n (key, original position) pairs in
// s.u.sort.keys / s.idx (any order on entry; sorted on return).  Every pass takes
// position w*32*M + k*32 + l of the previous one, which the stable ranking
// keeps in order.
template <typename T>
__device__ __noinline__ void small_radix(LeanSmem<T>& s, int n) {
    typedef KeyOf<T> KO;
    typedef typename KO::K K;
    constexpr int NT = wsh::NT, M = wsh::M;
    const int t = threadIdx.x, l = t & 31, w = t >> 5;
    for (int pass = 0; pass < KO::BITS / 8; ++pass) {
        K key[M];
        uint16_t ii[M];
        uint32_t dg[M];
        bool valid[M];
        int pos[M];
#pragma unroll
        for (int k = 0; k < M; ++k) {
            const int p = w * 32 * M + k * 32 + l;
            valid[k] = p < n;
            key[k] = valid[k] ? s.u.sort.keys[lean_kpad(p)] : (K)0;
            ii[k] = valid[k] ? s.idx[lean_ipad(p)] : (uint16_t)0;
            dg[k] = (uint32_t)((key[k] >> (8 * pass)) & 0xff);
        }
        __syncthreads();
        ws_rank_digits<NT, M, 1>(dg, valid, pos, s.u.sort.radix.whist, s.u.sort.radix.dcount, s.u.sort.radix.dstart);
#pragma unroll
        for (int k = 0; k < M; ++k)
            if (valid[k]) { s.u.sort.keys[lean_kpad(pos[k])] = key[k]; s.idx[lean_ipad(pos[k])] = ii[k]; }
        __syncthreads();
    }
}

// The hull by chains and trees when the rounds hit their cap (no CTA cap:
// never fails).  Ends synchronised.
__device__ __noinline__ void small_chain_tree(wsh::Smem& h, const wsh::Test& tst, int first, int last, int n,
                                              int64_t Xf) {
    wsh::chain_tree_hull(h, tst, threadIdx.x, first, last, n, Xf, 1 << 30);
}

// Warm start: the runs of equal earlier cluster ids (low 16 bits; any values
// are valid) along the sorted order, then candidate_boundaries on the
// round-1 survivors G.  The earlier
// ids are staged by original position in `cprev` (the lane stacks' storage,
// which only a segment whose rounds hit their cap uses, later).  Prefix sums of every point must be written
// (the barriers here publish them).
template <typename T>
__device__ __noinline__ uint32_t small_warm(LeanSmem<T>& s, const wsh::Test& tst, const int32_t* ids_prev,
                                            int64_t a0, int first, int n, uint32_t G) {
    constexpr int M = wsh::M;
    const int t = threadIdx.x;
    uint16_t* cprev = s.u.h.st;   // (st, lo and hi are one run of 16-bit words)
    static_assert(sizeof(s.u.h.st) + sizeof(s.u.h.lo) + sizeof(s.u.h.hi) >= sizeof(s.idx), "the earlier ids fit");
    if (first < n) {
        const int32_t* src = ids_prev + a0 + first;
        if (first + M <= n && (((uintptr_t)src) & 15) == 0) {
#pragma unroll
            for (int i = 0; i < M; i += 4) {
                const int4 q = __ldcs(reinterpret_cast<const int4*>(src + i));
                cprev[lean_ipad(first + i)] = (uint16_t)q.x;
                cprev[lean_ipad(first + i + 1)] = (uint16_t)q.y;
                cprev[lean_ipad(first + i + 2)] = (uint16_t)q.z;
                cprev[lean_ipad(first + i + 3)] = (uint16_t)q.w;
            }
        } else {
            for (int i = 0; i < M && first + i < n; ++i) cprev[lean_ipad(first + i)] = (uint16_t)src[i];
        }
    }
    __syncthreads();
    // bit i: a run starts at point first + i
    uint32_t R = 0;
    if (first < n) {
        uint16_t cp = first >= 1 ? cprev[lean_ipad(s.idx[lean_ipad(first - 1)])] : (uint16_t)0;
#pragma unroll
        for (int i = 0; i < M; ++i) {
            const int p = first + i;
            if (p < n) {
                const uint16_t c = cprev[lean_ipad(s.idx[lean_ipad(p)])];
                if (p >= 1 && c != cp) R |= 1u << i;
                cp = c;
            }
        }
    }
    return wsh::candidate_boundaries(s.u.h, tst, t, first, n, R, G);
}

// A cluster's value from its exact 128-bit sum (FP64 arithmetic or storage).
template <typename T>
__device__ __noinline__ T small_value(int64_t xd, int a, int b, int64_t q0, int up, T xs, const SegConst* sc,
                                      bool fp64, const WsEpi* ep) {
    const i128 SX = (i128)(b - a) * (i128)q0 + ((i128)xd << up);
    return ValueOut<T>::value(SX, a, b, xs, *sc, fp64, *ep);
}

template <typename T>
__global__ void __launch_bounds__(wsh::NT, sizeof(T) == 4 ? 4 : 2) k_small(const T* __restrict__ values,
                                                   const int64_t* __restrict__ offsets,
                                                   const int32_t* __restrict__ seg_list,
                                                   const WsLambda lambdas, T* out, int32_t* ids,
                                                   int64_t* n_clusters, int fp64, const WsEpi ep, uint32_t* status,
                                                   int32_t* gen_list, int32_t* gen_count, int ic_cap,
                                                   const int32_t* ids_prev) {   // (may alias ids)
    typedef KeyOf<T> KO;
    typedef typename KO::K K;
    typedef LeanSmem<T> S;
    constexpr int NT = wsh::NT, M = wsh::M, CAP = S::CAP;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    S& s = *reinterpret_cast<S*>(smem_raw);
    wsh::Smem& h = s.u.h;
    auto kpad = [](int p) { return p + (p >> 4); };          // keys
    auto ipad = [](int p) { return p + ((p >> 4) << 1); };   // 16-bit arrays
    const int t = threadIdx.x, l = t & 31, w = t >> 5;
    const int seg = seg_list[blockIdx.x];
    const int64_t a0 = offsets[seg];
    const int n = (int)(offsets[seg + 1] - a0);
    const double lam = lambdas.at(seg);
    if (!(lam >= 0.0) || !(lam <= 1.7976931348623157e308)) {
        if (t == 0) ws_flag(status, WS_STATUS_BAD_LAMBDA);
        return;
    }
    if (n <= 0 || n > CAP) {
        if (n > CAP && t == 0) ws_flag(status, WS_STATUS_INTERNAL);
        if (n == 0 && t == 0 && n_clusters) n_clusters[seg] = 0;
        return;
    }
    // ---- load this thread's 16 consecutive elements (16-byte loads when whole and aligned)
    const int first = t * M;
    K key[M];
    bool bad = false;
    int emin = 0x7fffffff;
    {
        T v[M];
        const T* src = values + a0 + first;
        if (first + M <= n && (((uintptr_t)src) & 15) == 0) {
            constexpr int NV = M * (int)sizeof(T) / 16;
            uint4 buf[NV];
#pragma unroll
            for (int i = 0; i < NV; ++i) buf[i] = __ldcs(reinterpret_cast<const uint4*>(src) + i);
            const T* bv = reinterpret_cast<const T*>(buf);
#pragma unroll
            for (int i = 0; i < M; ++i) v[i] = bv[i];
        } else {
#pragma unroll
            for (int i = 0; i < M; ++i) v[i] = (first + i < n) ? src[i] : (T)0;
        }
#pragma unroll
        for (int i = 0; i < M; ++i) {
            if (first + i < n) {
                bad |= !ws_isfinite(v[i]);
                if (v[i] != (T)0) emin = min(emin, ws_eff_exp(v[i]));
            }
            key[i] = KO::to_key(v[i]);
        }
    }
    if (t == 0) {
        s.emin = 0x7fffffff;
        s.kmin = ~(K)0;
        s.kmax = 0;
        s.bmax = 0;
    }
    if (__syncthreads_or(bad)) {
        if (t == 0) ws_flag(status, WS_STATUS_NONFINITE);
        return;
    }
    if (n == 1) {
        if (t == 0) {
            const T x = KO::from_key(key[0]);   // d = 1: no shift (the 1/(d-1) factor is vacuous)
            out[a0] = fp64 ? (T)ws_epilogue<double>((double)x, 0.0, ep.beta, ep.gamma, ep.on != 0)
                           : (T)ws_epilogue<float>((float)x, 0.0f, ep.beta_f, ep.gamma_f, ep.on != 0);
            if (ids) ids[a0] = 0;
            if (n_clusters) n_clusters[seg] = 1;
        }
        return;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) emin = min(emin, __shfl_xor_sync(WS_FULL_MASK, emin, o));
    if (l == 0) atomicMin(&s.emin, emin);

    // ---- sort (key, original position).  First an interpolation bucket sort:
    // bucket(x) = floor((x - x_min) 2n / (x_max - x_min)) in FP32 is monotone
    // in x (every step rounds monotonically), so equal keys share a bucket and
    // sorting each bucket by key sorts the segment; for the smooth
    // distributions of weights a bucket holds half an element on average (n
    // buckets: more and larger buckets to sort, rows of the MLP 610 us).  If a bucket is
    // larger than BUCKET_MAX the segment takes the LSD radix passes instead.
    constexpr int BUCKET_MAX = 32;
    {
        K lo = ~(K)0, hi = 0;
#pragma unroll
        for (int i = 0; i < M; ++i)
            if (first + i < n) { lo = min(lo, key[i]); hi = max(hi, key[i]); }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            lo = min(lo, ws_shfl_xor_k(lo, o));
            hi = max(hi, ws_shfl_xor_k(hi, o));
        }
        uint32_t* cnt = s.u.sort.cnt;
        for (int i = t; i < n; i += NT) cnt[kpad(i)] = 0;
        if (l == 0) { ws_atomic_min_k(&s.kmin, lo); ws_atomic_max_k(&s.kmax, hi); }
    }
    __syncthreads();
    // ---- the fixed point of the segment, from its extreme keys (the first and
    // last sorted ones): a segment whose prefix sums need more than 64 bits
    // goes to the general kernel before any sorting
    const K kfirst = s.kmin, klast = s.kmax;
    const T xlo = KO::from_key(kfirst), xhi = KO::from_key(klast);
    const int emax = ws_fix_scale<T>(max(ws_eff_exp(xlo), ws_eff_exp(xhi)), s.emin);
    if (t == 0) {
        const int top = max(ws_eff_exp(xlo), ws_eff_exp(xhi));
        ws_note_scale<T>(top, s.emin, status);
        s.inexact = s.emin <= top && top - s.emin > KO::FIX_OFS;
    }
    int sh;
    const bool bin = ws_tile_binade<T>(kfirst, klast, n, emax, sh);
    const int64_t q0 = ws_fixed<T>(xlo, emax);
    const uint64_t range = bin ? (uint64_t)(klast - kfirst) : (uint64_t)(ws_fixed<T>(xhi, emax) - q0);
    const bool lean = ws_lean_x(range, n);   // prefix sums in 64 bits
    const bool d64 = ws_lean_tile(range, n);  // every Delta too
    if (!lean) {   // (uniform)
        if (t == 0) gen_list[atomicAdd(gen_count, 1)] = seg;
        return;
    }
    bool radix = false;
    {
        uint32_t* cnt = s.u.sort.cnt;
        const float f0 = (float)KO::from_key(s.kmin), f1 = (float)KO::from_key(s.kmax);
        const float span = f1 - f0;
        const float scale = (span > 0.0f && span <= 3.0e38f) ? (float)(2 * n) / span : 0.0f;
        uint32_t br[M];   // bucket << 16 | rank
#pragma unroll
        for (int i = 0; i < M; ++i) {
            if (first + i < n) {
                const float f = ((float)KO::from_key(key[i]) - f0) * scale;
                const uint32_t b = (uint32_t)min(2 * n - 1, max(0, (int)f));
                const uint32_t up = (b & 1u) << 4;
                const uint32_t old = atomicAdd(&cnt[kpad((int)(b >> 1))], 1u << up);
                br[i] = (b << 16) | ((old >> up) & 0xffffu);
            }
        }
        __syncthreads();
        // bucket starts: this thread's 32 consecutive buckets, then the CTA scan
        uint32_t c[M], multi = 0;   // (multi: bit j, bucket 2 first + j holds two or more)
        int sum = 0, big = 0;
#pragma unroll
        for (int i = 0; i < M; ++i) {
            c[i] = (first + i < n) ? cnt[kpad(first + i)] : 0u;
            const int c0 = (int)(c[i] & 0xffffu), c1 = (int)(c[i] >> 16);
            sum += c0 + c1;
            big = max(big, max(c0, c1));
            multi |= (c0 >= 2 ? 1u : 0u) << (2 * i) | (c1 >= 2 ? 2u : 0u) << (2 * i);
        }
        int tot;
        int run = lean_excl_scan(sum, s.wsumi, &tot);
#pragma unroll
        for (int i = 0; i < M; ++i)
            if (first + i < n) {
                const uint32_t mid = (uint32_t)run + (c[i] & 0xffffu);
                cnt[kpad(first + i)] = (uint32_t)run | (mid << 16);
                run = (int)(mid + (c[i] >> 16));
            }
        radix = __syncthreads_or(big > BUCKET_MAX);
        if (!radix) {
            auto start_of_bucket = [&](int b) { return (int)((cnt[kpad(b >> 1)] >> ((b & 1) << 4)) & 0xffffu); };
#pragma unroll
            for (int i = 0; i < M; ++i)
                if (first + i < n) {
                    const int pp = start_of_bucket((int)(br[i] >> 16)) + (int)(br[i] & 0xffffu);
                    s.u.sort.keys[kpad(pp)] = key[i];
                    s.idx[ipad(pp)] = (uint16_t)(first + i);
                }
            __syncthreads();
            while (multi) {
                const int i = 2 * first + __ffs((int)multi) - 1;
                multi &= multi - 1;
                const int b0 = start_of_bucket(i);
                const int b1 = i + 1 < 2 * n ? start_of_bucket(i + 1) : n;
                small_sort_bucket<K>(b0, b1, s.u.sort.keys, s.idx, kpad, ipad);
            }
            __syncthreads();
        }
    }
    // ---- otherwise: LSD radix sort, 8-bit digits (out of line)
    if (radix) {
#pragma unroll
        for (int k = 0; k < M; ++k)
            if (first + k < n) { s.u.sort.keys[kpad(first + k)] = key[k]; s.idx[ipad(first + k)] = (uint16_t)(first + k); }
        __syncthreads();
        small_radix<T>(s, n);
    }

    // ---- the sorted segment as one hull tile: this thread's 16 sorted keys
    K kr[M];
#pragma unroll
    for (int i = 0; i < M; ++i) kr[i] = (first + i < n) ? s.u.sort.keys[kpad(first + i)] : s.u.sort.keys[0];
    const K kprev = (t > 0 && first < n) ? s.u.sort.keys[kpad(first - 1)] : kfirst;
    __syncthreads();   // (the keys are read; the prefix sums take their place)
    if (t == 0) {   // (no FP64 on this critical path)
        s.sc = ws_seg_const_f(n, lam, KO::L_BASE - emax, fp64 != 0);
        TileScale& ts = s.ts;
        ts.sc = bin ? ws_seg_const_f(n, lam, s.sc.L - sh, false) : s.sc;
        bool f;
        ts.muq = ws_muq_f(ts.sc, f);
        ts.fast = f ? 1 : 0;
        if (ts.sc.mlam == 0) { ts.modd = 0; ts.sodd = 0; }
        else { const int tz = __ffsll((long long)ts.sc.mlam) - 1; ts.modd = ts.sc.mlam >> tz; ts.sodd = ts.sc.s + tz; }
        // lower bound of floor(2 mu) (muq is within 1e-6 relative of mu)
        const float m2 = 2.0f * ts.muq * (1.0f - 1.0e-6f);
        s.t11 = !f ? (int64_t)-1 : (m2 < 3.9e18f ? (int64_t)floorf(m2) - 1 : (int64_t)3.9e18);
        h.general = 0;
    }
    auto devk = [&](K k) -> int64_t {
        return bin ? (int64_t)(k - kfirst) : ws_fixed<T>(KO::from_key(k), emax) - q0;
    };
    auto dev = [&](int i) -> int64_t { return devk(kr[i]); };
    // the deviations, once: their running sums (this lane's prefix sums
    // relative to its first point) go straight into the prefix-sum slots (the
    // sort's scratch is dead); the lane's offset is added below
    int64_t csum = 0;
#pragma unroll
    for (int i = 0; i < M; ++i)
        if (first + i < n) {
            csum += dev(i);
            wsh::xref(h, first + i + 1) = csum;
        }
    const int64_t winc = ws_warp_incl_scan<long long>((long long)csum);
    if (l == 31) h.wtot[w] = winc;
    if (t == 0) wsh::xref(h, 0) = 0;
    __syncthreads();
    int64_t wbase = 0;
    for (int k = 0; k < w; ++k) wbase += h.wtot[k];
    const int64_t Xf = wbase + winc - csum;
    const int last = min(first + M, n);
    wsh::Test tst;
    tst.sc = s.ts.sc;
    tst.P.s64 = nullptr;
    tst.P.muq = s.ts.muq;
    tst.P.fast = s.ts.fast != 0;
    tst.P.d64 = d64;
    tst.P.thr = nullptr;
    tst.P.modd = s.ts.modd;
    tst.P.sodd = s.ts.sodd;
    // round 1 of the Imminent Collisions rounds: point p stays a boundary iff
    // y_{p-1} < y_p, i.e. the gap x_p - x_{p-1} exceeds 2 lambda/(d-1) = 2 mu.
    // t11 is a lower bound of floor(2 mu) in tile units, so a few points at
    // the threshold may stay too: a superset of the hull vertices is all the
    // rounds need (their first round tests every boundary exactly).  Warm:
    // of these, the candidate's run boundaries and the points below their
    // run's chord.
    // (with the lane's offset added to its prefix sums)
    uint32_t B = 0;
    if (first < n) {
        const int64_t t11 = s.t11;
        int64_t dprev = devk(kprev), prevX = 0;
#pragma unroll 4
        for (int i = 0; i < M; ++i) {
            const int p = first + i;
            if (p < n) {
                int64_t& slot = wsh::xref(h, p + 1);
                const int64_t Xl = slot;
                const int64_t di = Xl - prevX;   // the deviation of element p
                prevX = Xl;
                slot = Xl + Xf;
                if (p >= 1 && di - dprev > t11) B |= 1u << i;
                dprev = di;
            }
        }
    }
    if (ids_prev) B = small_warm<T>(s, tst, ids_prev, a0, first, n, B);
    int rounds = 0, prev = 0, next = n;
    bool converged = false;
    if (ic_cap > 0) converged = wsh::ic_rounds(h.e, [&](int p) { return wsh::xat(h, p); }, tst, t, first, n, B,
                                                    ic_cap, rounds, prev, next);
    uint16_t* st16 = reinterpret_cast<uint16_t*>(s.starts);
    if (converged) {
        st16[t] = (uint16_t)(B | (t == 0 ? 1u : 0u));
    } else {
        small_chain_tree(h, tst, first, last, n, Xf);
        st16[t] = 0;
        __syncthreads();
        for (int k = h.lo[t]; k < (int)h.hi[t]; ++k) {
            const int p = h.st[k * NT + t];
            if (p < n) atomicOr(&s.starts[p >> 5], 1u << (p & 31));
        }
    }
    __syncthreads();
    // ---- cluster ids: rank of every start; values of the clusters this thread starts
    const uint32_t mine = (uint32_t)st16[t] & (first < n ? (n - first >= M ? 0xffffu : ((1u << (n - first)) - 1u)) : 0u);
    int C;
    const int base = lean_excl_scan(__popc(mine), h.wsum, &C);
    // neighbouring starts outside this thread's chunk
    if (!converged) {
        next = n;
        for (int wd = (first + M) >> 5; (wd << 5) < n; ++wd) {
            uint32_t bits = s.starts[wd];
            if ((wd << 5) < first + M) bits &= 0xffffffffu << ((first + M) & 31);
            if (bits) { next = min((wd << 5) + __ffs((int)bits) - 1, n); break; }
        }
        prev = 0;   // (position 0 is a start)
        for (int wd = min(first, n) >> 5; wd >= 0; --wd) {
            uint32_t bits = s.starts[wd];
            if ((wd << 5) + 31 >= first) bits &= (1u << (first & 31)) - 1u;
            if (bits) { prev = (wd << 5) + 31 - __clz((int)bits); break; }
        }
    }
    // ---- the value of every cluster, into the slot of its first point.  That
    // slot is read as the end of the cluster before it, by this thread except
    // for its first start, which waits for the barrier.
    auto put = [&](int a, T val, int r) {
        if (sizeof(T) == 4) *reinterpret_cast<uint2*>(&wsh::xref(h, a)) = make_uint2(__float_as_uint((float)val), (uint32_t)r);
        else { *reinterpret_cast<double*>(&wsh::xref(h, a)) = (double)val; s.cid[a] = (uint16_t)r; }
    };
    T v0 = (T)0;
    if (mine) {
        const int Lt = s.ts.sc.L;
        // 2^-L as a factor where it is a normal number (then x 2^-L rounds as ldexpf does)
        const bool fac = Lt >= -126 && Lt <= 126;
        const float down = fac ? __uint_as_float((uint32_t)(127 - Lt) << 23) : 0.0f;
        const bool inexact = s.inexact != 0;
        const float mu_f = s.sc.mu_f, x0f = (float)xlo;
        uint32_t rest = mine;
        int a = first + __ffs((int)rest) - 1, r = base;
        int64_t Xa = wsh::xat(h, a);
        rest &= rest - 1;
        while (true) {
            const int b = rest ? first + __ffs((int)rest) - 1 : next;
            const int64_t Xb = wsh::xat(h, b), xd = Xb - Xa;
            T val;
            if (KO::BITS == 32 && !fp64) {
                // FP32: mean = x_0 + (deviation sum / count) in tile units; every
                // term exact but the conversions (a few FP32 ulps of max |w|).
                // A single weight comes back exactly from its deviation.
                float mean;
                if (b - a == 1) {
                    if (bin) mean = (float)KO::from_key((K)(kfirst + (K)xd));
                    else if (!inexact && fac && q0 + xd != 0) {   // (zeros keep their sign)
                        const int64_t q = q0 + xd;
                        const float f = ws_u64_to_float((uint64_t)(q < 0 ? -q : q));
                        mean = (q < 0 ? -f : f) * down;
                    } else mean = (float)values[a0 + s.idx[ipad(a)]];
                } else {
                    const float f = ws_u64_to_float((uint64_t)xd) / (float)(b - a);
                    mean = x0f + (fac ? f * down : ldexpf(f, -Lt));
                }
                val = (T)ws_epilogue<float>(mean, mu_f * (float)(n - a - b), ep.beta_f, ep.gamma_f, ep.on != 0);
            } else {
                const T xs = b - a == 1 ? values[a0 + s.idx[ipad(a)]] : (T)0;
                val = small_value<T>(xd, a, b, q0, bin ? sh : 0, xs, &s.sc, fp64 != 0, &ep);
            }
            if (r == base) v0 = val;
            else put(a, val, r);
            if (!rest) break;
            rest &= rest - 1;
            ++r;
            a = b;
            Xa = Xb;
        }
    }
    __syncthreads();   // (every prefix sum is read)
    if (mine) put(first + __ffs((int)mine) - 1, v0, base);
    // ---- the cluster (its first point) of every original position, then this
    // thread's 16 consecutive outputs (coalesced stores)
    uint16_t* start_of = h.st;   // (st, lo and hi are one run of 16-bit words)
    {
        int a = prev;
#pragma unroll 4
        for (int i = 0; i < M; ++i) {
            const int p = first + i;
            if ((mine >> i) & 1u) a = p;
            if (p < n) start_of[ipad(s.idx[ipad(p)])] = (uint16_t)a;
        }
    }
    __syncthreads();
    if (first < n) {
        T* od = out + a0 + first;
        int32_t* id = ids ? ids + a0 + first : nullptr;
        const bool whole = first + M <= n && (((uintptr_t)od) & 15) == 0 && (!id || (((uintptr_t)id) & 15) == 0);
        // (four at a time: the loop is rolled for the instruction cache)
#pragma unroll 1
        for (int j = 0; j < M; j += 4) {
            __align__(16) T ov[4];
            __align__(16) int32_t oi[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int a = (first + j + i < n) ? (int)start_of[ipad(first + j + i)] : 0;
                if (sizeof(T) == 4) {
                    const uint2 q = *reinterpret_cast<const uint2*>(&wsh::xref(h, a));
                    ov[i] = (T)__uint_as_float(q.x);
                    oi[i] = (int32_t)q.y;
                } else {
                    ov[i] = (T)*reinterpret_cast<const double*>(&wsh::xref(h, a));
                    oi[i] = (int32_t)s.cid[a];
                }
            }
            if (whole) {
#pragma unroll
                for (int i = 0; i < (int)sizeof(T) / 4; ++i)
                    __stcs(reinterpret_cast<uint4*>(od + j) + i, reinterpret_cast<const uint4*>(ov)[i]);
                if (id) __stcs(reinterpret_cast<uint4*>(id + j), *reinterpret_cast<const uint4*>(oi));
            } else {
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    if (first + j + i < n) {
                        od[j + i] = ov[i];
                        if (id) id[j + i] = oi[i];
                    }
            }
        }
    }
    if (t == 0 && n_clusters) n_clusters[seg] = C;
}

}  // namespace

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------
template <typename T>
cudaError_t ws_launch_small(const T* values, const int64_t* offsets, const int32_t* seg_list, int n_list,
                            WsLambda lambdas, T* out, int32_t* ids, int64_t* n_clusters, int fp64,
                            const WsEpi& ep, uint32_t* status, cudaStream_t st, WsProf* prof, int32_t* gen_list,
                            int32_t* gen_count, int ic_cap, const int32_t* ids_prev) {
    constexpr int NT = 256;
    constexpr int M = SmallCfg<T>::M;
    if (n_list <= 0) return cudaSuccess;
    cudaError_t e = cudaMemsetAsync(gen_count, 0, sizeof(int32_t), st);
    if (e != cudaSuccess) return e;
    const size_t smem = sizeof(LeanSmem<T>);
    e = cudaFuncSetAttribute(k_small<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    WS_LAUNCH(prof, WSK_SMALL, st,
              (k_small<T><<<n_list, NT, smem, st>>>(values, offsets, seg_list, lambdas, out, ids, n_clusters, fp64, ep,
                                                    status, gen_list, gen_count, ic_cap, ids_prev)));
    // the segments the lean kernel passed on (none on ordinary inputs): a
    // small grid that walks the list
    const size_t gsmem = sizeof(SmallSmem<T, NT, M>);
    auto gk = k_small_general<T, NT, M>;
    e = cudaFuncSetAttribute(gk, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)gsmem);
    if (e != cudaSuccess) return e;
    WS_LAUNCH(prof, WSK_SMALL, st,
              ws_launch_chain(gk, n_list < 456 ? n_list : 456, NT, gsmem, st, values, offsets, gen_list, gen_count,
                              lambdas, out, ids, n_clusters, fp64, ep, ic_cap, status));
    return cudaGetLastError();
}

template cudaError_t ws_launch_small<float>(const float*, const int64_t*, const int32_t*, int, WsLambda, float*,
                                            int32_t*, int64_t*, int, const WsEpi&, uint32_t*, cudaStream_t, WsProf*,
                                            int32_t*, int32_t*, int, const int32_t*);
template cudaError_t ws_launch_small<double>(const double*, const int64_t*, const int32_t*, int, WsLambda,
                                             double*, int32_t*, int64_t*, int, const WsEpi&, uint32_t*, cudaStream_t,
                                             WsProf*, int32_t*, int32_t*, int, const int32_t*);
