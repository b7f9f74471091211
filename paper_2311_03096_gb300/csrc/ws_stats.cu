// ws_stats.cu -- R(w) and the weight-sharing measure of a vector, on the
// sorted keys of the device-wide path.
//
// R(w) = 1/(d-1) sum_{i>j} |w_i - w_j| (Eq. (1)) is evaluated the way the
// appendix "Computing R" does it: sort, then R = 1/(d-1) sum_k (2k - d - 1) x_k
// (k = 1..d, x sorted ascending), an O(d) reduction after the sort.  The sum
// is accumulated exactly in 128-bit fixed point (q = x 2^L as in the hull:
// |q| <= 2^58, |2k - d - 1| < 2^31, so every term and the total fit) and
// rounded once at the end.  The weight-sharing measure of the CIFAR10
// experiment is #distinct nonzero weights / #nonzero weights (0 when every
// weight is zero); on sorted keys a distinct value is a key that differs
// from its predecessor.
#include <algorithm>

#include "ws_kernels.cuh"

namespace {

struct RPartial {
    i128 s;             // sum of (2k - d - 1) q_k over the tile
    long long distinct; // nonzero keys that differ from their predecessor
    long long nonzero;
};

template <typename T>
__global__ void __launch_bounds__(256) k_R_tiles(const typename KeyOf<T>::K* __restrict__ sorted,
                                                 const TileDesc* __restrict__ tiles,
                                                 const LargeSeg* __restrict__ lsegs,
                                                 const int32_t* __restrict__ seg_emin, RPartial* part) {
    typedef KeyOf<T> KO;
    typedef typename KO::K K;
    __shared__ i128 ws128[8];
    ws_chain();
    const TileDesc td = tiles[blockIdx.x];
    const LargeSeg ls = lsegs[td.lseg];
    const K* seg = sorted + ls.kpos;
    const T xlo = KO::from_key(seg[0]), xhi = KO::from_key(seg[ls.len - 1]);
    const int E = ws_fix_scale<T>(max(ws_eff_exp(xlo), ws_eff_exp(xhi)), seg_emin[td.lseg]);
    const K kz = KO::to_key((T)0), knz = KO::to_key(-(T)0);
    const int64_t j0 = (int64_t)td.tin * WS_SORT_TILE;
    // sum of coef_j q_j over this thread's elements, coef_j = 2j - len + 1
    // (2k - d - 1 with k = j + 1).  Its elements lie 256 apart, so with c its
    // last coefficient the sum is c Q - 512 W, Q the sum of its q and W that of
    // its earlier elements' running sums: 64-bit additions and, every four
    // elements (the sums stay below 2^61), two 128-bit products.
    constexpr int U = 4;
    i128 acc = 0;
    int dis = 0, nz = 0;
    for (int i0 = threadIdx.x; i0 < td.len; i0 += 256 * U) {
        K k[U], before[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int64_t j = j0 + min(i0 + u * 256, td.len - 1);
            k[u] = __ldg(seg + j);
            before[u] = j > 0 ? __ldg(seg + j - 1) : ~k[u];
        }
        int64_t Q = 0, Wq = 0;
        int c = 0;
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (i0 + u * 256 < td.len) {
                const bool nonzero = k[u] != kz && k[u] != knz;
                nz += nonzero;
                dis += nonzero && before[u] != k[u];
                Wq += Q;
                Q += ws_fixed<T>(KO::from_key(k[u]), E);   // (|Q| <= 2^60, |Wq| <= 6 x 2^58)
                c = u;
            }
        }
        const int64_t coef = 2 * (j0 + i0 + c * 256) - ls.len + 1;
        acc += (i128)coef * Q - (i128)512 * Wq;
    }
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    acc = ws_warp_reduce_i128(acc);
    dis = __reduce_add_sync(0xffffffffu, dis);
    nz = __reduce_add_sync(0xffffffffu, nz);
    __shared__ int wsd[8], wsn[8];
    if (lane == 0) { ws128[w] = acc; wsd[w] = dis; wsn[w] = nz; }
    __syncthreads();
    if (threadIdx.x == 0) {
        RPartial p;
        p.s = 0; p.distinct = 0; p.nonzero = 0;
        for (int k = 0; k < 8; ++k) { p.s += ws128[k]; p.distinct += wsd[k]; p.nonzero += wsn[k]; }
        part[blockIdx.x] = p;
    }
}

// One CTA per segment adds its tiles' partial sums.
template <typename T>
__global__ void __launch_bounds__(256) k_R_final(const LargeSeg* __restrict__ lsegs, const TileDesc* __restrict__ tiles,
                                                const typename KeyOf<T>::K* __restrict__ sorted,
                                                const int32_t* __restrict__ seg_emin, const RPartial* part,
                                                double* R_out, double* metric_out, uint32_t* status) {
    typedef KeyOf<T> KO;
    __shared__ RPartial wp[8];
    ws_chain();
    const LargeSeg ls = lsegs[blockIdx.x];
    i128 s = 0;
    long long dis = 0, nz = 0;
#pragma unroll 4
    for (int t = threadIdx.x; t < ls.sort_count; t += 256) {
        const RPartial p = part[ls.sort_first + t];
        s += p.s; dis += p.distinct; nz += p.nonzero;
    }
    s = ws_warp_reduce_i128(s);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        dis += __shfl_xor_sync(0xffffffffu, dis, o);
        nz += __shfl_xor_sync(0xffffffffu, nz, o);
    }
    if ((threadIdx.x & 31) == 0) { wp[threadIdx.x >> 5].s = s; wp[threadIdx.x >> 5].distinct = dis; wp[threadIdx.x >> 5].nonzero = nz; }
    __syncthreads();
    if (threadIdx.x != 0) return;
    for (int k = 1; k < 8; ++k) { s += wp[k].s; dis += wp[k].distinct; nz += wp[k].nonzero; }
    const T xlo = KO::from_key(sorted[ls.kpos]), xhi = KO::from_key(sorted[ls.kpos + ls.len - 1]);
    const int E = ws_fix_scale<T>(max(ws_eff_exp(xlo), ws_eff_exp(xhi)), seg_emin[blockIdx.x]);
    ws_note_scale<T>(max(ws_eff_exp(xlo), ws_eff_exp(xhi)), seg_emin[blockIdx.x], status);
    const int L = KO::L_BASE - E;
    if (R_out) R_out[ls.seg] = ls.len > 1 ? ldexp(ws_i128_to_double(s), -L) / (double)(ls.len - 1) : 0.0;
    if (metric_out) metric_out[ls.seg] = nz > 0 ? (double)dis / (double)nz : 0.0;
}

}  // namespace

template <typename T>
cudaError_t ws_large_R(const LargeWork<T>& W, const T* values, double* R_out, double* metric_out, uint32_t* status,
                       uint64_t spin_limit, void* partial, cudaStream_t st) {
    typedef typename KeyOf<T>::K K;
    if (W.n_lseg == 0) return cudaSuccess;
    K* sorted = nullptr;
    cudaError_t e = ws_large_sort<T>(W, values, false, status, spin_limit, st, &sorted);
    if (e) return e;
    RPartial* part = reinterpret_cast<RPartial*>(partial);
    WS_LAUNCH(W.prof, WSK_MISC, st,
              ws_launch_chain(k_R_tiles<T>, W.n_sort_tiles, 256, 0, st, sorted, W.sort_tiles, W.lsegs, W.seg_emin, part));
    WS_LAUNCH(W.prof, WSK_MISC, st,
              ws_launch_chain(k_R_final<T>, W.n_lseg, 256, 0, st, W.lsegs, W.sort_tiles, sorted, W.seg_emin, part, R_out,
                              metric_out, status));
    return cudaGetLastError();
}

namespace {
template <typename T>
__global__ void k_R_tiny(const T* values, int64_t d, double* R_out, double* metric_out) {
    if (R_out) *R_out = 0.0;   // d <= 1: no pairs
    if (metric_out) *metric_out = (d == 1 && values[0] != (T)0) ? 1.0 : 0.0;
}
}  // namespace

template <typename T>
cudaError_t ws_tiny_R(const T* values, int64_t d, double* R_out, double* metric_out, WsProf* prof, cudaStream_t st) {
    WS_LAUNCH(prof, WSK_MISC, st, (k_R_tiny<T><<<1, 1, 0, st>>>(values, d, R_out, metric_out)));
    return cudaGetLastError();
}
template cudaError_t ws_tiny_R<float>(const float*, int64_t, double*, double*, WsProf*, cudaStream_t);
template cudaError_t ws_tiny_R<double>(const double*, int64_t, double*, double*, WsProf*, cudaStream_t);

size_t ws_R_partial_bytes(int n_sort_tiles) { return sizeof(RPartial) * (size_t)(n_sort_tiles > 0 ? n_sort_tiles : 1); }

template cudaError_t ws_large_R<float>(const LargeWork<float>&, const float*, double*, double*, uint32_t*, uint64_t,
                                       void*, cudaStream_t);
template cudaError_t ws_large_R<double>(const LargeWork<double>&, const double*, double*, double*, uint32_t*,
                                        uint64_t, void*, cudaStream_t);

// ---------------------------------------------------------------------------
// d out / d lambda with the partition held fixed (Sec. 3: a cluster moves
// with the mean velocity of its particles).  A cluster on sorted positions
// a..b (1-based) has d out / d lambda = (d + 1 - a - b)/(d - 1); with 0-based
// start s and size m that is (d - 2s - m)/(d - 1).  Starts follow from the
// cluster sizes because cluster ids are ranked by value.  The result per
// segment is sum_i grad_out[i] * d out_i / d lambda (the sums of tiles are
// added with FP64 atomics: their order is not fixed).
// ---------------------------------------------------------------------------
namespace {

template <typename T, int NT, int CAP>
__global__ void __launch_bounds__(NT) k_dlam_small(const T* __restrict__ g, const int32_t* __restrict__ ids,
                                                   const int64_t* __restrict__ offsets,
                                                   const int32_t* __restrict__ seg_list, double* out,
                                                   uint32_t* status) {
    __shared__ int cnt[CAP];
    __shared__ int start[CAP];
    __shared__ int wsum[NT / 32];
    __shared__ double wacc[NT / 32];
    constexpr int PER = CAP / NT;
    const int seg = seg_list[blockIdx.x];
    const int64_t a0 = offsets[seg];
    const int n = (int)(offsets[seg + 1] - a0);
    if (n <= 1) return;   // d <= 1: no shift
    if (n > CAP) { if (threadIdx.x == 0) ws_flag(status, WS_STATUS_INTERNAL); return; }
    const int t = threadIdx.x;
    for (int i = t; i < CAP; i += NT) cnt[i] = 0;
    __syncthreads();
    for (int i = t; i < n; i += NT) {
        const int id = ids[a0 + i];
        if (id < 0 || id >= n) { ws_flag(status, WS_STATUS_INTERNAL); continue; }
        atomicAdd(&cnt[id], 1);
    }
    __syncthreads();
    int run = 0;
#pragma unroll
    for (int k = 0; k < PER; ++k) run += cnt[t * PER + k];
    int tot;
    int ex = ws_block_excl_scan<NT, int>(run, wsum, &tot);
#pragma unroll
    for (int k = 0; k < PER; ++k) { start[t * PER + k] = ex; ex += cnt[t * PER + k]; }
    __syncthreads();
    double acc = 0.0;
    for (int i = t; i < n; i += NT) {
        const int id = ids[a0 + i];
        if (id < 0 || id >= n) continue;
        acc += (double)g[a0 + i] * (double)(n - 2 * start[id] - cnt[id]) / (double)(n - 1);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if ((t & 31) == 0) wacc[t >> 5] = acc;
    __syncthreads();
    if (t == 0) {
        double s = 0.0;
        for (int w = 0; w < NT / 32; ++w) s += wacc[w];
        atomicAdd(&out[seg], s);
    }
}

// Cluster sizes.  Distinct ids: one global atomic each, bound by the L1 (a line
// per lane and clock; 91 us at 2^24).  Adds to one address go one by one (0.6 ns),
// so a tile in which at least HOT of 256 sampled ids meet another one of their warp
// is left to k_dlam_crowded, which adds into a hash table in shared memory first,
// one global add per id and tile (what finds no place in four probes is added
// directly).  2^24 elements, dlambda in all, us: one cluster 10740 -> 190, 7
// clusters 2660 -> 183, one of half the elements 5520 -> 251.  (A kernel of its
// own: with the table's shared memory the direct adds take 120 us.)
constexpr int HOT = 3;
__global__ void __launch_bounds__(256) k_dlam_count(const int32_t* __restrict__ ids, const TileDesc* __restrict__ tiles,
                                                    const LargeSeg* __restrict__ lsegs, int32_t* cnt,
                                                    uint8_t* crowded, uint32_t* status) {
    const TileDesc td = tiles[blockIdx.x];
    const LargeSeg ls = lsegs[td.lseg];
    const int64_t slot0 = ls.kpos + td.lseg;
    constexpr int U = 8;   // (loads issued together)
    bool hot = false;
    for (int i0 = threadIdx.x, first = 1; i0 - (int)threadIdx.x < td.len; i0 += 256 * U, first = 0) {
        int id[U];
#pragma unroll
        for (int u = 0; u < U; ++u) id[u] = i0 + u * 256 < td.len ? __ldg(ids + td.vpos + i0 + u * 256) : 0;
        if (first) {   // (uniform)
            const unsigned peers = __match_any_sync(0xffffffffu, id[0]);
            hot = __syncthreads_count(i0 < td.len && __popc(peers) > 1) >= HOT;
            if (threadIdx.x == 0) crowded[blockIdx.x] = hot ? 1 : 0;
        }
        if (hot) return;
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (i0 + u * 256 >= td.len) break;
            if (id[u] < 0 || id[u] >= ls.len) { ws_flag(status, WS_STATUS_INTERNAL); continue; }
            atomicAdd(&cnt[slot0 + id[u]], 1);
        }
    }
}

constexpr int DC_NT = 512, TAB_LOG2 = 12;
__device__ __forceinline__ void dlam_crowded_tile(const TileDesc& td, const int32_t* __restrict__ ids,
                                                  const LargeSeg* __restrict__ lsegs, int32_t* cnt, int* tk, int* tc,
                                                  uint32_t* status) {
    constexpr int PER = WS_SORT_TILE / DC_NT, TAB = 1 << TAB_LOG2;
    const int64_t slot0 = lsegs[td.lseg].kpos + td.lseg, slen = lsegs[td.lseg].len;
    const int t = threadIdx.x, lane = t & 31;
    int id[PER];
    bool bad = false;
#pragma unroll
    for (int k = 0; k < PER; ++k) {
        const int i = t + k * DC_NT;
        id[k] = i < td.len ? __ldg(ids + td.vpos + i) : -1;
        if (i < td.len && (id[k] < 0 || (int64_t)id[k] >= slen)) { bad = true; id[k] = -1; }
    }
    if (bad) ws_flag(status, WS_STATUS_INTERNAL);
    __syncthreads();   // (the previous use of the table is over)
    for (int i = t; i < TAB; i += DC_NT) { tk[i] = -1; tc[i] = 0; }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < PER; ++k) {
        const unsigned crowd = ws_crowd(id[k], id[k] >= 0);
        int add = id[k] >= 0 ? 1 : 0;
        if ((crowd >> lane) & 1u) add = lane == __ffs((int)crowd) - 1 ? __popc(crowd) : 0;
        if (add == 0) continue;
        uint32_t h = ((uint32_t)id[k] * 0x9E3779B1u) >> (32 - TAB_LOG2);
        int probe = 0;
        for (; probe < 4; ++probe, h = (h + 1) & (TAB - 1)) {
            int q = *(volatile int*)&tk[h];
            if (q == -1) {
                q = atomicCAS(&tk[h], -1, id[k]);
                if (q == -1) q = id[k];
            }
            if (q == id[k]) { atomicAdd(&tc[h], add); break; }
        }
        if (probe == 4) atomicAdd(&cnt[slot0 + id[k]], add);
    }
    __syncthreads();
    for (int i = t; i < TAB; i += DC_NT)
        if (tc[i]) atomicAdd(&cnt[slot0 + tk[i]], tc[i]);
}
__global__ void __launch_bounds__(DC_NT) k_dlam_crowded(const int32_t* __restrict__ ids,
                                                        const TileDesc* __restrict__ tiles, int n_tiles,
                                                        const LargeSeg* __restrict__ lsegs, int32_t* cnt,
                                                        const uint8_t* __restrict__ crowded, uint32_t* status) {
    __shared__ int tk[1 << TAB_LOG2], tc[1 << TAB_LOG2];
    ws_chain();
    for (int tile = blockIdx.x; tile < n_tiles; tile += gridDim.x)
        if (crowded[tile]) dlam_crowded_tile(tiles[tile], ids, lsegs, cnt, tk, tc, status);   // (uniform)
}

// Cluster starts in two passes over the counts, in chunks of 4096 slots (one
// CTA; 16-byte loads, warp w the slots [512 w, 512 w + 512) of its chunk):
// WRITE false: csum[b] = total of chunk b; then, with csum scanned, WRITE true:
// key[s] = 2 start(s) + cnt[s], start counted over all slots.  32-bit wrapping
// arithmetic: len - 2 start - size of a cluster in its segment, which fits, is
// len + 2 start(first slot of the segment) - key[s].
constexpr int DL_CHUNK = 4096;
template <bool WRITE>
__global__ void __launch_bounds__(256) k_dlam_starts(const int32_t* __restrict__ cnt, int64_t S, uint32_t* key,
                                                     int32_t* csum) {
    ws_chain();
    __shared__ int wsum[8];
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    const int64_t b0 = (int64_t)blockIdx.x * DL_CHUNK + 512 * w + 4 * lane;
    int4 v[4];
    int inc[4], tot = 0;   // inclusive within the warp's rows of 128
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int64_t s = b0 + 128 * k;
        if (s + 4 <= S) v[k] = __ldg(reinterpret_cast<const int4*>(cnt + s));
        else {
            v[k].x = s < S ? cnt[s] : 0;
            v[k].y = s + 1 < S ? cnt[s + 1] : 0;
            v[k].z = s + 2 < S ? cnt[s + 2] : 0;
            v[k].w = 0;
        }
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int sum = v[k].x + v[k].y + v[k].z + v[k].w;
        if (WRITE) {
            const int i = ws_warp_incl_scan<int>(sum);
            inc[k] = tot + i - sum;
            tot += __shfl_sync(0xffffffffu, i, 31);
        } else {
            tot += sum;
        }
    }
    if (!WRITE) tot = __reduce_add_sync(0xffffffffu, tot);
    if (lane == 0) wsum[w] = tot;
    __syncthreads();
    if (!WRITE) {
        if (t == 0) {
            int all = 0;
            for (int k = 0; k < 8; ++k) all += wsum[k];
            csum[blockIdx.x] = all;
        }
        return;
    }
    int base = csum[blockIdx.x];
    for (int k = 0; k < w; ++k) base += wsum[k];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int64_t s = b0 + 128 * k;
        const uint32_t e0 = (uint32_t)(base + inc[k]), e1 = e0 + v[k].x, e2 = e1 + v[k].y, e3 = e2 + v[k].z;
        const uint4 q = make_uint4(2 * e0 + v[k].x, 2 * e1 + v[k].y, 2 * e2 + v[k].z, 2 * e3 + v[k].w);
        if (s + 4 <= S) *reinterpret_cast<uint4*>(key + s) = q;
        else {
            if (s < S) key[s] = q.x;
            if (s + 1 < S) key[s + 1] = q.y;
            if (s + 2 < S) key[s + 2] = q.z;
        }
    }
}

// exclusive scan of the chunk totals, in place (one CTA, carried across rounds)
__global__ void __launch_bounds__(1024) k_dlam_scan_totals(int32_t* csum, int nb) {
    ws_chain();
    __shared__ int wsum[32];
    __shared__ int carry;
    if (threadIdx.x == 0) carry = 0;
    __syncthreads();
    for (int b0 = 0; b0 < nb; b0 += 1024) {
        const int b = b0 + (int)threadIdx.x;
        const int v = b < nb ? csum[b] : 0;
        int tot;
        const int ex = ws_block_excl_scan<1024, int>(v, wsum, &tot);
        if (b < nb) csum[b] = carry + ex;
        __syncthreads();
        if (threadIdx.x == 0) carry += tot;
        __syncthreads();
    }
}

// Sum of grad_out x (len - 2 start - size) over one sort tile: every product as
// an integer of up to 84 bits, in units of 2^-113 of its warp's largest (a
// product more than 28 binades below it, 58 for FP32, loses the bits below
// that), the sums in 128 bits, one rounding and one division at the end.  The
// scale comes from the products: the largest gradient may have weight 0 or 1,
// and an integer of the gradient alone at its scale lost what others, with
// weights up to the length, add (FP64 products did not).  FP64 multiplies and
// adds per element took 266 us at 2^24 (GB300 runs them at a small fraction of
// the FP32 rate; two gathers per element beside them) and round more.
constexpr int DL_NT = 512;
template <typename T>
__global__ void __launch_bounds__(DL_NT, sizeof(T) == 4 ? 1 : 2) k_dlam_apply(const T* __restrict__ g, const int32_t* __restrict__ ids,
                                                      const TileDesc* __restrict__ tiles,
                                                      const LargeSeg* __restrict__ lsegs,
                                                      const int32_t* __restrict__ cnt,
                                                      const uint32_t* __restrict__ key, double* out) {
    ws_chain();
    typedef KeyOf<T> KO;
    constexpr int PER = WS_SORT_TILE / DL_NT;
    __shared__ long long wlo[DL_NT / 32], whi[DL_NT / 32];
    __shared__ int we[DL_NT / 32];
    const TileDesc td = tiles[blockIdx.x];
    const LargeSeg& ls = lsegs[td.lseg];
    const int64_t slot0 = ls.kpos + td.lseg;
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    T gv[PER];
    int id[PER];
#pragma unroll
    for (int k = 0; k < PER; ++k) {
        const int i = t + k * DL_NT;
        gv[k] = i < td.len ? __ldg(g + td.vpos + i) : (T)0;
        id[k] = i < td.len ? __ldg(ids + td.vpos + i) : -1;
    }
    // len + 2 start of the segment's first slot, modulo 2^32
    const uint32_t top = (uint32_t)ls.len + key[slot0] - (uint32_t)cnt[slot0];
    uint32_t kv[PER];
    int e = 0;
    bool odd = false;
#pragma unroll
    for (int k = 0; k < PER; ++k) {
        if (id[k] < 0 || (int64_t)id[k] >= ls.len) { id[k] = -1; gv[k] = (T)0; }
        kv[k] = id[k] >= 0 ? __ldg(key + slot0 + id[k]) : 0u;
        odd |= !ws_isfinite(gv[k]);
    }
#pragma unroll
    for (int k = 0; k < PER; ++k) {   // (the weight; one bit above the product's binade)
        const int32_t wt = id[k] >= 0 ? (int32_t)(top - kv[k]) : 0;
        kv[k] = (uint32_t)wt;
        if (gv[k] != (T)0 && wt != 0) e = max(e, ws_eff_exp(gv[k]) + 32 - __clz(abs(wt)));
    }
    // every warp at its own scale (no barrier while the weights arrive)
    int emax = __reduce_max_sync(0xffffffffu, e);
    if (__any_sync(0xffffffffu, odd)) {   // infinities and NaN: as FP64 arithmetic has it
        double acc = 0.0;
#pragma unroll
        for (int k = 0; k < PER; ++k)
            if (id[k] >= 0) acc += (double)gv[k] * ((double)(int32_t)kv[k] / (double)(ls.len - 1));
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        if (lane == 0) atomicAdd(&out[ls.seg], acc);
#pragma unroll
        for (int k = 0; k < PER; ++k) kv[k] = 0;   // (nothing left to add)
        emax = 0;
    }
    i128 acc = 0;
#pragma unroll
    for (int k = 0; k < PER; ++k) {
        const uint64_t b = (uint64_t)KO::bits(gv[k]);
        int ex = (int)((b >> KO::MANT) & KO::EXPMASK);
        uint64_t m = b & ((1ull << KO::MANT) - 1ull);
        if (ex == 0) ex = 1; else m |= 1ull << KO::MANT;
        const int32_t wt = (int32_t)kv[k];
        const uint64_t aw = (uint32_t)abs(wt);
        const u128 p = sizeof(T) == 4 ? (u128)(m * aw) : (u128)m * aw;   // < 2^(MANT + 1 + bits of the weight)
        const int up = ex - emax + 112 - KO::MANT;   // (then < 2^113: 6144 of them fit)
        if (wt == 0) continue;
        u128 q;
        if (up < 0) q = up > -128 ? p >> -up : (u128)0;   // (rare)
        else if (sizeof(T) == 4) q = p << up;
        else {   // (up <= 59)
            const uint64_t lo = (uint64_t)p, hi = (uint64_t)(p >> 64);
            q = ((u128)((hi << up) | ((lo >> 1) >> (63 - up))) << 64) | (lo << up);
        }
        acc += ((b >> (KO::BITS - 1)) & 1ull) != (uint64_t)(wt < 0) ? -(i128)q : (i128)q;
    }
    acc = ws_warp_reduce_i128(acc);
    if (lane == 0) { wlo[w] = (long long)(uint64_t)acc; whi[w] = (long long)(uint64_t)((u128)acc >> 64); we[w] = emax; }
    __syncthreads();
    if (t == 0) {
        emax = 0;
        for (int k = 0; k < DL_NT / 32; ++k) emax = max(emax, we[k]);
        i128 S = 0;
        for (int k = 0; k < DL_NT / 32; ++k)
            S += (i128)(((u128)(uint64_t)whi[k] << 64) | (u128)(uint64_t)wlo[k]) >> min(emax - we[k], 127);
        // product = q 2^(emax - bias - 112)
        const int bias = KO::EXPMASK >> 1;
        const double v = ws_i128_to_double(S) / (double)(ls.len - 1);
        if (S != 0) atomicAdd(&out[ls.seg], ldexp(v, emax - bias - 112));
    }
}

}  // namespace

template <typename T>
cudaError_t ws_dlambda(const T* g, const int32_t* ids, const int64_t* d_offsets, const int32_t* d_small, int n_small,
                       int64_t n_seg, const LargeWork<T>& W, double* out, uint32_t* status, void* partial,
                       cudaStream_t st) {
    cudaError_t e = cudaMemsetAsync(out, 0, sizeof(double) * (size_t)n_seg, st);
    if (e) return e;
    if (n_small > 0) {
        WS_LAUNCH(W.prof, WSK_BWD, st,
                  (k_dlam_small<T, 256, SmallCfg<T>::CAP><<<n_small, 256, 0, st>>>(g, ids, d_offsets, d_small, out,
                                                                                   status)));
    }
    if (W.n_lseg > 0) {
        const int64_t S = W.n_keys + W.n_lseg;
        int32_t* cnt = W.bcnt;
        uint32_t* key = reinterpret_cast<uint32_t*>(W.bsum);
        int32_t* csum = reinterpret_cast<int32_t*>(partial);
        uint8_t* crowded = reinterpret_cast<uint8_t*>(W.keys_a);   // (the sort's buffer, free here)
        const int nb = (int)((S + DL_CHUNK - 1) / DL_CHUNK);
        e = cudaMemsetAsync(cnt, 0, sizeof(int32_t) * (size_t)S, st);
        if (e) return e;
        WS_LAUNCH(W.prof, WSK_BWD, st,
                  (k_dlam_count<<<W.n_sort_tiles, 256, 0, st>>>(ids, W.sort_tiles, W.lsegs, cnt, crowded, status)));
        WS_LAUNCH(W.prof, WSK_BWD, st,
                  ws_launch_chain(k_dlam_crowded, std::min(W.n_sort_tiles, 3 * 152), DC_NT, 0, st, ids, W.sort_tiles,
                                  W.n_sort_tiles, W.lsegs, cnt, crowded, status));
        WS_LAUNCH(W.prof, WSK_BWD, st, ws_launch_chain(k_dlam_starts<false>, nb, 256, 0, st, cnt, S, key, csum));
        WS_LAUNCH(W.prof, WSK_BWD, st, ws_launch_chain(k_dlam_scan_totals, 1, 1024, 0, st, csum, nb));
        WS_LAUNCH(W.prof, WSK_BWD, st, ws_launch_chain(k_dlam_starts<true>, nb, 256, 0, st, cnt, S, key, csum));
        WS_LAUNCH(W.prof, WSK_BWD, st,
                  ws_launch_if(W.n_sort_tiles <= 2 * 152, k_dlam_apply<T>, W.n_sort_tiles, DL_NT, 0, st, g, ids,
                               W.sort_tiles, W.lsegs, cnt, key, out));
    }
    return cudaGetLastError();
}

template cudaError_t ws_dlambda<float>(const float*, const int32_t*, const int64_t*, const int32_t*, int, int64_t,
                                       const LargeWork<float>&, double*, uint32_t*, void*, cudaStream_t);
template cudaError_t ws_dlambda<double>(const double*, const int32_t*, const int64_t*, const int32_t*, int, int64_t,
                                        const LargeWork<double>&, double*, uint32_t*, void*, cudaStream_t);
