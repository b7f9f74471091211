// ws_large.cu -- the device-wide path for segments longer than one CTA:
//   sorted keys -> per-tile exact hulls -> tree of bridge merges across tiles
//   -> cluster values and starts -> the sort's passes undone, to the caller's order.
//
// The hull of the points P_p = (p, S_p) (see ws_common.cuh) is built tile by
// tile (4096 elements per CTA); adjacent tile hulls are then merged up a
// binary tree.  A merge keeps a prefix of the left hull and a suffix of the
// right one (the bridge is the common lower tangent, Search Collisions'
// Merge step of Sec. 4.3 re-derived on convex chains), so a node's hull is a
// list of "pieces" -- contiguous vertex ranges of tile hulls -- and a merge
// only edits the two lists where they meet.  The root list is the cluster
// partition: its consecutive vertices bound the clusters.
#include <algorithm>

#include "ws_hull.cuh"
#include "ws_kernels.cuh"

namespace {

constexpr int HT = WS_HULL_TILE;
constexpr int HNT = WS_HULL_NT;
constexpr int HM = WS_HULL_M;

// ---------------------------------------------------------------------------
// 2. merging two adjacent node hulls (run by the CTA that arrives last)
//
// Piece lists are rewritten in place as the tree climbs, by whichever CTA
// merges a node, so they are read through L2 (ld.global.cg): an SM's L1 may
// still hold a line of a list another SM has since rewritten.
// ---------------------------------------------------------------------------
__device__ __forceinline__ Piece ws_ld_piece(const Piece* p) {
    const uint4* q = reinterpret_cast<const uint4*>(p);
    uint4 a = __ldcg(q), b = __ldcg(q + 1);
    Piece r;
    *reinterpret_cast<uint4*>(&r) = a;
    *(reinterpret_cast<uint4*>(&r) + 1) = b;
    return r;
}
__device__ __forceinline__ void ws_st_piece(Piece* p, const Piece& v) {
    uint4* q = reinterpret_cast<uint4*>(p);
    __stcg(q, *reinterpret_cast<const uint4*>(&v));
    __stcg(q + 1, *(reinterpret_cast<const uint4*>(&v) + 1));
}
__device__ __forceinline__ i128 ws_ld_i128(const i128* p) {
    const uint4 v = __ldcg(reinterpret_cast<const uint4*>(p));
    return *reinterpret_cast<const i128*>(&v);
}

struct NodeView {
    const Piece* pc;   // piece list
    int np;            // pieces
    const uint16_t* vp;
    VertX vx;
    int hull_first;    // global index of the segment's first hull tile
    i128 base;         // X offset of this node's first point in the merge frame
    __device__ __forceinline__ int find(int r) const {   // piece holding rank r
        int lo = 0, hi = np - 1;
        while (lo < hi) {
            int mid = (lo + hi + 1) >> 1;
            if (ws_ld_piece(pc + mid).cum <= r) lo = mid; else hi = mid - 1;
        }
        return lo;
    }
    __device__ __forceinline__ void get(int r, int64_t& pt, i128& X) const {
        const Piece p = ws_ld_piece(pc + find(r));
        const int v = p.lo + (r - p.cum), at = vp[(size_t)p.tile * (HT + 1) + v];
        pt = (int64_t)(p.tile - hull_first) * HT + at;
        X = base + p.off + vx.at(p.tile, v, at);
    }
    __device__ __forceinline__ int count() const {
        if (np == 0) return 0;
        const Piece p = ws_ld_piece(pc + np - 1);
        return p.cum + (p.hi - p.lo);
    }
};

__device__ __forceinline__ void ws_piece_vertex(const Piece& q, int v, const uint16_t* vp, const VertX& vx,
                                                int hull_first, i128 base, int64_t& pt, i128& X) {
    const int at = vp[(size_t)q.tile * (HT + 1) + v];
    pt = (int64_t)(q.tile - hull_first) * HT + at;
    X = base + q.off + vx.at(q.tile, v, at);
}

// Bridge between two node hulls by walking outward from their junction
// (the linear merge of two convex chains), stepping through the piece lists
// directly.  Returns false (no result) after too many steps; the caller then
// runs the galloping search.  Same outputs as ws_bridge.
__device__ bool ws_bridge_walk(const Piece* PL, int npL, const Piece* PR, int npR, const uint16_t* vp,
                               const VertX& vx, int hull_first, i128 baseR, const SegConst& sc, int& flag, int& istar,
                               int& jstar) {
    int lp = npL - 1, rp = 0;
    Piece qL = ws_ld_piece(PL + lp), qR = ws_ld_piece(PR + rp);
    int lv = qL.hi - 1, rv = qR.lo;   // L_p and R_0: the junction
    auto prevL = [&](int& p, Piece& q, int& v) -> bool {
        if (v > q.lo) { --v; return true; }
        if (p == 0) return false;
        --p; q = ws_ld_piece(PL + p); v = q.hi - 1; return true;
    };
    auto nextR = [&](int& p, Piece& q, int& v) -> bool {
        if (v + 1 < q.hi) { ++v; return true; }
        if (p + 1 >= npR) return false;
        ++p; q = ws_ld_piece(PR + p); v = q.lo; return true;
    };
    int64_t pj; i128 Xj;
    ws_piece_vertex(qR, rv, vp, vx, hull_first, baseR, pj, Xj);
    if (!prevL(lp, qL, lv) || !nextR(rp, qR, rv)) { flag = 0; return true; }
    int64_t pl, pr; i128 Xl, Xr;
    ws_piece_vertex(qL, lv, vp, vx, hull_first, 0, pl, Xl);
    ws_piece_vertex(qR, rv, vp, vx, hull_first, baseR, pr, Xr);
    if (ws_convex(Xl, Xj, Xr, pl, pj, pr, sc)) { flag = 0; return true; }
    flag = 1;
    int steps = 0;
    constexpr int WALK_MAX = 32;
    while (true) {
        bool moved = false;
        while (true) {
            int p2 = lp, v2 = lv;
            Piece q2 = qL;
            if (!prevL(p2, q2, v2)) break;
            int64_t pm; i128 Xm;
            ws_piece_vertex(q2, v2, vp, vx, hull_first, 0, pm, Xm);
            if (ws_convex(Xm, Xl, Xr, pm, pl, pr, sc)) break;
            lp = p2; qL = q2; lv = v2; pl = pm; Xl = Xm; moved = true;
            if (++steps > WALK_MAX) return false;
        }
        while (true) {
            int p2 = rp, v2 = rv;
            Piece q2 = qR;
            if (!nextR(p2, q2, v2)) break;
            int64_t pn; i128 Xn;
            ws_piece_vertex(q2, v2, vp, vx, hull_first, baseR, pn, Xn);
            if (ws_convex(Xl, Xr, Xn, pl, pr, pn, sc)) break;
            rp = p2; qR = q2; rv = v2; pr = pn; Xr = Xn; moved = true;
            if (++steps > WALK_MAX) return false;
        }
        if (!moved) break;
    }
    istar = qL.cum + (lv - qL.lo);
    jstar = qR.cum + (rv - qR.lo);
    return true;
}

constexpr int MW = 16;   // vertices of each child prefetched around the junction

struct MergeSmem {
    int is, js, pl, pr, npL, npR;
    i128 totL, totR;
    int wsi[8];
    // window: the last MW vertices of L (index 0 = L_p, the junction, going
    // left) and the first MW of R (index 0 = R_0 = junction, going right)
    Piece wpL[MW], wpR[MW];        // the pieces at the ends of the two lists
    int nwpL, nwpR;
    int wLn, wRn;                  // vertices in each window
    int wLpc[MW], wLv[MW], wRpc[MW], wRv[MW];   // (piece slot in the list, vertex index)
    int64_t wLpt[MW], wRpt[MW];
    i128 wLX[MW], wRX[MW];
    int ok;
    int cand_i[HNT / 32], cand_s[HNT / 32], cand_j[HNT / 32];   // parallel search: one candidate per warp
};

// Vertex of rank r of a node hull whose piece list is cached in shared memory.
__device__ __forceinline__ void ws_cached_vertex(const Piece* c, int np, int r, const uint16_t* vp, const VertX& vx,
                                                 int hull_first, i128 base, int64_t& pt, i128& X) {
    int lo = 0, hi = np - 1;   // the last piece whose first rank is <= r
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (c[mid].cum <= r) lo = mid; else hi = mid - 1;
    }
    ws_piece_vertex(c[lo], c[lo].lo + (r - c[lo].cum), vp, vx, hull_first, base, pt, X);
}
__device__ __forceinline__ int ws_cached_find(const Piece* c, int np, int r) {
    int lo = 0, hi = np - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (c[mid].cum <= r) lo = mid; else hi = mid - 1;
    }
    return lo;
}

// The bridge of two node hulls searched by the whole CTA, for merges whose
// bridge lies beyond the prefetched window (typically near the root, where
// one side loses thousands of vertices).  Same definitions as ws_bridge:
// right(i, j) = R_{j+1} on or below the line (L_i, R_j); tangent(i) = the
// first j with !right(i, j) (right(i, .) is true then false along the convex
// chain R); survives(i) = i == 0 or L_{i-1}, L_i, R_tangent(i) convex
// (survivors are a prefix of L); istar = the last survivor below the
// junction, jstar = tangent(istar).  Each round of the outer search gives
// one candidate i to each warp; a warp finds tangent(i) by a 32-way search
// (every lane tests one j), so a merge costs about log_9(p) * log_33(q)
// rounds instead of a serial gallop through global memory.  Requires the
// junction not to be a vertex and both hulls to have >= 2 vertices.  The
// piece lists are copied into `cache` (capacity >= npL + npR).  All threads
// call it; it ends synchronised with m.is/js/pl/pr set and m.ok = 1.
__device__ void ws_parallel_bridge(Piece* cache, MergeSmem& m, const Piece* PL, const Piece* PR, const uint16_t* vp,
                                   const VertX& vx, int hull_first, const SegConst& sc) {
    constexpr int NW = HNT / 32;
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    const int npL = m.npL, npR = m.npR;
    Piece* cL = cache;
    Piece* cR = cache + npL;
    for (int k = t; k < npL + npR; k += HNT) cache[k] = ws_ld_piece(k < npL ? PL + k : PR + (k - npL));
    __syncthreads();
    const int p = cL[npL - 1].cum + (cL[npL - 1].hi - cL[npL - 1].lo) - 1;   // L_p = R_0: the junction
    const int q = cR[npR - 1].cum + (cR[npR - 1].hi - cR[npR - 1].lo) - 1;
    const i128 baseR = m.totL;
    if (p < 1 || q < 1) return;   // (not reached from the window walk) left to the serial search
    if (t == 0) {   // the junction stays a vertex: keep all of L, drop R_0 (as ws_bridge's flag 0)
        int64_t pa, pb, pc;
        i128 Xa, Xb, Xc;
        ws_cached_vertex(cL, npL, p - 1, vp, vx, hull_first, 0, pa, Xa);
        ws_cached_vertex(cL, npL, p, vp, vx, hull_first, 0, pb, Xb);
        ws_cached_vertex(cR, npR, 1, vp, vx, hull_first, baseR, pc, Xc);
        m.cand_s[0] = ws_convex(Xa, Xb, Xc, pa, pb, pc, sc) ? 1 : 0;
        if (m.cand_s[0]) {
            m.is = p; m.js = 1;
            m.pl = ws_cached_find(cL, npL, p);
            m.pr = ws_cached_find(cR, npR, 1);
            m.ok = 1;
        }
    }
    __syncthreads();
    const bool junction_vertex = m.cand_s[0] != 0;
    __syncthreads();   // every thread has read the flag before the search reuses cand_s
    if (junction_vertex) return;   // (m.ok set)
    // first j in [0, q] with !right(i, j), by the whole warp
    auto tangent = [&](int64_t pi, const i128& Xi) -> int {
        int jl = -1, jh = q;   // right(i, jl) (or jl = -1), !right(i, jh) (jh = q: no R_{q+1})
        while (jh - jl > 1) {
            const int span = jh - jl - 1;   // candidates jl + 1 .. jh - 1
            const int j = (span <= 32) ? jl + 1 + lane : jl + 1 + (int)(((long long)span * lane) >> 5);
            const bool valid = j < jh;
            bool rt = false;
            if (valid) {
                int64_t pj, pk;
                i128 Xj, Xk;
                ws_cached_vertex(cR, npR, j, vp, vx, hull_first, baseR, pj, Xj);
                ws_cached_vertex(cR, npR, j + 1, vp, vx, hull_first, baseR, pk, Xk);
                rt = !ws_convex(Xi, Xj, Xk, pi, pj, pk, sc);
            }
            const unsigned bt = __ballot_sync(WS_FULL_MASK, valid && rt);
            const unsigned bf = __ballot_sync(WS_FULL_MASK, valid && !rt);
            if (bt) jl = __shfl_sync(WS_FULL_MASK, j, 31 - __clz((int)bt));
            if (bf) jh = __shfl_sync(WS_FULL_MASK, j, __ffs((int)bf) - 1);
        }
        return jh;
    };
    int good = 0, bad = p, jgood = -1;   // survives(good), !survives(bad) (bad = p: the junction)
    while (bad - good > 1) {
        const int span = bad - good - 1;
        const int c = (span <= NW) ? good + 1 + w : good + 1 + (int)(((long long)span * w) / NW);
        if (c < bad) {
            int64_t pc;
            i128 Xc;
            ws_cached_vertex(cL, npL, c, vp, vx, hull_first, 0, pc, Xc);
            const int jt = tangent(pc, Xc);
            if (lane == 0) {
                int64_t pm, pt;
                i128 Xm, Xt;
                ws_cached_vertex(cL, npL, c - 1, vp, vx, hull_first, 0, pm, Xm);
                ws_cached_vertex(cR, npR, jt, vp, vx, hull_first, baseR, pt, Xt);
                m.cand_i[w] = c;
                m.cand_j[w] = jt;
                m.cand_s[w] = ws_convex(Xm, Xc, Xt, pm, pc, pt, sc) ? 1 : 0;
            }
        } else if (lane == 0) {
            m.cand_i[w] = -1;
        }
        __syncthreads();
        int ng = good, nb = bad, nj = jgood;
        for (int k = 0; k < NW; ++k) {
            const int ci = m.cand_i[k];
            if (ci < 0) continue;
            if (m.cand_s[k]) { if (ci > ng) { ng = ci; nj = m.cand_j[k]; } }
            else if (ci < nb) nb = ci;
        }
        good = ng; bad = nb; jgood = nj;
        __syncthreads();
    }
    if (jgood < 0 && w == 0) {   // istar = 0 was never a candidate: its tangent
        int64_t p0;
        i128 X0;
        ws_cached_vertex(cL, npL, 0, vp, vx, hull_first, 0, p0, X0);
        const int jt = tangent(p0, X0);
        if (lane == 0) m.cand_j[0] = jt;
    }
    __syncthreads();
    if (t == 0) {
        const int js = jgood >= 0 ? jgood : m.cand_j[0];
        m.is = good;
        m.js = js;
        m.pl = ws_cached_find(cL, npL, good);
        m.pr = js <= q ? ws_cached_find(cR, npR, js) : npR;
        m.ok = 1;
    }
    __syncthreads();
}

// Merge the node hulls whose piece lists start at Lg and Rg (global hull-tile
// indices, Rg > Lg adjacent); the result replaces the list at Lg.  All
// threads of the CTA call this.  Warp 0 first gathers, in parallel, the
// vertices next to the junction (usually all the bridge needs); thread 0
// walks them in shared memory and falls back to the global search only if
// the bridge leaves that window.
__device__ __noinline__ void ws_merge_children(MergeSmem& m, Piece* pieces, int32_t* npieces, i128* ntotal, int Lg, int Rg,
                                  const uint16_t* vp, const VertX& vx, int hull_first, const SegConst& sc,
                                  Piece* cache, int cache_cap) {
    const int t = threadIdx.x;
    Piece* PL = pieces + Lg;
    Piece* PR = pieces + Rg;
    if (t < 32) {
        const int npL = __ldcg(npieces + Lg), npR = __ldcg(npieces + Rg);
        // the last MW pieces of L (slot 0 = last) and the first MW of R
        if (t < MW) { if (t < npL) m.wpL[t] = ws_ld_piece(PL + npL - 1 - t); }
        else { const int k = t - MW; if (k < npR) m.wpR[k] = ws_ld_piece(PR + k); }
        if (t == 0) {
            m.npL = npL; m.npR = npR;
            m.totL = ws_ld_i128(ntotal + Lg);
            m.totR = ws_ld_i128(ntotal + Rg);
            m.nwpL = min(npL, MW); m.nwpR = min(npR, MW);
        }
        __syncwarp();
        if (t == 0) {   // enumerate the window's vertices
            int n = 0;
            for (int k = 0; k < m.nwpL && n < MW; ++k) {
                const Piece q = m.wpL[k];
                for (int v = q.hi - 1; v >= (int)q.lo && n < MW; --v) { m.wLpc[n] = npL - 1 - k; m.wLv[n] = v; ++n; }
            }
            m.wLn = n;
            n = 0;
            for (int k = 0; k < m.nwpR && n < MW; ++k) {
                const Piece q = m.wpR[k];
                for (int v = q.lo; v < (int)q.hi && n < MW; ++v) { m.wRpc[n] = k; m.wRv[n] = v; ++n; }
            }
            m.wRn = n;
        }
        __syncwarp();
        if (t < MW) {
            if (t < m.wLn) {
                const Piece q = m.wpL[npL - 1 - m.wLpc[t]];
                ws_piece_vertex(q, m.wLv[t], vp, vx, hull_first, 0, m.wLpt[t], m.wLX[t]);
            }
        } else {
            const int k = t - MW;
            if (k < m.wRn) {
                const Piece q = m.wpR[m.wRpc[k]];
                ws_piece_vertex(q, m.wRv[k], vp, vx, hull_first, m.totL, m.wRpt[k], m.wRX[k]);
            }
        }
        __syncwarp();
        if (t == 0) {
            // walk in the window: li indexes wL (0 = junction), rj indexes wR (0 = junction)
            const int nL = m.wLn, nR = m.wRn;
            int flag = 0, li = 0, rj = 0;
            bool ok = true;
            const bool Lmore = nL == MW, Rmore = nR == MW;   // a list may continue past the window
            if (nL >= 2 && nR >= 2) {
                if (!ws_convex(m.wLX[1], m.wLX[0], m.wRX[1], m.wLpt[1], m.wLpt[0], m.wRpt[1], sc)) {
                    flag = 1; li = 1; rj = 1;
                    while (ok) {
                        bool moved = false;
                        while (true) {
                            if (li + 1 >= nL) { if (Lmore) ok = false; break; }
                            if (ws_convex(m.wLX[li + 1], m.wLX[li], m.wRX[rj], m.wLpt[li + 1], m.wLpt[li], m.wRpt[rj], sc))
                                break;
                            ++li; moved = true;
                        }
                        if (!ok) break;
                        while (true) {
                            if (rj + 1 >= nR) { if (Rmore) ok = false; break; }
                            if (ws_convex(m.wLX[li], m.wRX[rj], m.wRX[rj + 1], m.wLpt[li], m.wRpt[rj], m.wRpt[rj + 1], sc))
                                break;
                            ++rj; moved = true;
                        }
                        if (!moved) break;
                    }
                }
            } else if (!(nL == 1 || nR == 1)) {
                ok = false;
            }
            if (ok) {
                // (the pieces named here are in the window: its copies, not global memory)
                if (flag == 0) {   // junction stays: keep all of L, drop R_0
                    m.pl = npL - 1;
                    const Piece qL = m.wpL[0];
                    m.is = qL.cum + (qL.hi - qL.lo) - 1;
                    m.js = 1;
                    if (nR >= 2) { m.pr = m.wRpc[1]; } else { m.pr = npR; }
                } else {
                    m.pl = m.wLpc[li];
                    m.pr = m.wRpc[rj];
                    const Piece qL = m.wpL[npL - 1 - m.pl];
                    const Piece qR = m.wpR[m.pr];
                    m.is = qL.cum + (m.wLv[li] - qL.lo);
                    m.js = qR.cum + (m.wRv[rj] - qR.lo);
                }
                if (nL == 1 || nR == 1) { m.pl = npL - 1; m.is = -1; m.pr = (nR >= 2) ? m.wRpc[1] : npR; m.js = 1; }
            }
            m.ok = ok ? 1 : 0;
        }
        __syncwarp();
    }
    __syncthreads();
    // the bridge reaches beyond the window: the CTA searches it in parallel
    // (the serial walk and gallop below remain for lists too long to cache)
    if (!m.ok && m.npL + m.npR <= cache_cap) ws_parallel_bridge(cache, m, PL, PR, vp, vx, hull_first, sc);
    if (t == 0) {
        const int npL = m.npL, npR = m.npR;
        const i128 totL = m.totL;
        if (!m.ok) {   // the bridge reaches beyond the window: global walk, then the gallop
            NodeView L{PL, npL, vp, vx, hull_first, 0};
            NodeView R{PR, npR, vp, vx, hull_first, totL};
            const int nL = L.count(), nR = R.count();
            int flag = 0, is = nL - 1, js = 0;
            if (nL > 0 && nR > 0) {
                if (!ws_bridge_walk(PL, npL, PR, npR, vp, vx, hull_first, totL, sc, flag, is, js)) {
                    auto gl = [&](int r, int64_t& pt, i128& X) { L.get(r, pt, X); };
                    auto gr = [&](int r, int64_t& pt, i128& X) { R.get(r, pt, X); };
                    ws_bridge(gl, nL - 1, gr, nR - 1, sc, flag, is, js);
                }
                if (flag == 0) { is = nL - 1; js = 1; }
            }
            m.pl = (nL > 0) ? L.find(is) : -1;
            m.pr = (nR > 0 && js < nR) ? R.find(js) : npR;
            m.is = is; m.js = js;
        }
        if (m.pl >= 0 && m.is >= 0) {   // truncate the left list after istar
            const int slot = npL - 1 - m.pl;
            Piece q = slot < m.nwpL ? m.wpL[slot] : ws_ld_piece(PL + m.pl);
            q.hi = (uint16_t)(q.lo + (m.is - q.cum) + 1);
            ws_st_piece(PL + m.pl, q);
        }
        if (m.pr < npR) {  // the right list starts at jstar
            const bool in_window = m.pr < m.nwpR;
            Piece q = in_window ? m.wpR[m.pr] : ws_ld_piece(PR + m.pr);
            q.lo = (uint16_t)(q.lo + (m.js - q.cum));
            ws_st_piece(PR + m.pr, q);
            if (in_window) m.wpR[m.pr] = q;   // the copy below reads the window
        }
    }
    __syncthreads();
    const int keepL = m.pl + 1, firstR = m.pr, keepR = m.npR - m.pr;
    const i128 totL = m.totL;
    // Move the right suffix down behind the left prefix (dst <= src: chunked),
    // rebasing offsets onto the left node's first point.  Ranks of the kept
    // left pieces are unchanged; the right ones shift uniformly: the first
    // kept right piece starts at rank istar + 1.
    const int shift = m.is + 1 - m.js;
    for (int b = 0; b < keepR; b += 256) {
        Piece v;
        const bool has = b + t < keepR;
        if (has) {
            const int k = firstR + b + t;
            v = k < m.nwpR ? m.wpR[k] : ws_ld_piece(PR + k);
            v.off += totL;
            v.cum = (b + t == 0) ? m.is + 1 : v.cum + shift;
        }
        __syncthreads();
        if (has) ws_st_piece(PL + keepL + b + t, v);
        __syncthreads();
    }
    const int np = keepL + keepR;
    if (t == 0) {
        __stcg(npieces + Lg, np);
        const i128 tot = m.totL + m.totR;
        __stcg(reinterpret_cast<uint4*>(ntotal + Lg), *reinterpret_cast<const uint4*>(&tot));
    }
}

// ---------------------------------------------------------------------------
// 1. per-tile hull
// ---------------------------------------------------------------------------
struct TileHullSmem {
    TilePrefix<HNT, HM> pre;
    HullSmem<HNT, HM> hull;
    wsh::Ends ends;
    SegConst sc;     // global fixed-point scale of the segment
    SegConst sct;    // scale of this tile when it lies in one binade
    float muq, muqt;
    int fast, fastt;
};

// The general tile kernel: the exact hull of a tile whose prefix sums need
// 128 bits (or whose bridge walks were too long for the lean kernel of
// ws_tile.cu, which lists such tiles in gen_list).  A small grid walks the
// list.  Four CTAs per SM (64 registers, 412/788 bytes of spills in FP64): many
// tiles are what it takes long for.  8192 FP64 segments of 4097: 833 us; with
// three CTAs and 76/76 bytes 990, with two and no spills 909.  A lone vector with
// two such tiles would gain: 4194001 FP64 weights 460, 446 with two CTAs.
template <typename T>
__global__ void __launch_bounds__(HNT, 4) k_tile_hull(const typename KeyOf<T>::K* __restrict__ sorted,
                                                   const TileDesc* __restrict__ htiles,
                                                   const LargeSeg* __restrict__ lsegs,
                                                   WsLambda lambdas, SegRuntime* rt,
                                                   uint16_t* vp, i128* vx, TileX* hx, int32_t* nvert, i128* tile_total,
                                                   const int32_t* __restrict__ gen_list,
                                                   const int32_t* __restrict__ gen_count,
                                                   const int32_t* __restrict__ seg_emin, int ic_cap, uint32_t* status) {
    typedef KeyOf<T> KO;
    typedef typename KO::K K;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    TileHullSmem& s = *reinterpret_cast<TileHullSmem*>(smem_raw);
    const int t = threadIdx.x;
    ws_chain();
    const int n_list = *gen_count;
    for (int li = blockIdx.x; li < n_list; li += gridDim.x) {
    __syncthreads();   // (the previous tile's shared memory is dead)
    const int tile = gen_list[li];
    const TileDesc td = htiles[tile];
    const LargeSeg ls = lsegs[td.lseg];
    const double lam = lambdas.at(ls.seg);
    const bool lam_ok = lam >= 0.0 && lam <= 1.7976931348623157e308;
    const double lamv = lam_ok ? lam : 0.0;
    const int n = td.len;
    const K* kp = sorted + td.kpos;
    const K kfirst = kp[0], klast = kp[n - 1];
    const T xlo = KO::from_key(sorted[ls.kpos]), xhi = KO::from_key(sorted[ls.kpos + ls.len - 1]);
    const int emax = ws_fix_scale<T>(max(ws_eff_exp(xlo), ws_eff_exp(xhi)), seg_emin[td.lseg]);
    if (t == 0) {
        if (!lam_ok) ws_flag(status, WS_STATUS_BAD_LAMBDA);
        if (td.tin == 0) rt[td.lseg].emax = emax;
        s.sc = ws_seg_const<T>(ls.len, lamv, emax);
        bool f;
        s.muq = ws_muq_f(s.sc, f);
        s.fast = f ? 1 : 0;
    }
    if (t == 32) {   // (two warps: FP64 divisions take a few microseconds each)
        const int sh = ws_eff_exp(KO::from_key(kfirst)) - emax + KO::FIX_OFS;
        s.sct = ws_seg_const_L(ls.len, lamv, KO::L_BASE - emax - (sh > 0 ? sh : 0));
        bool f;
        s.muqt = ws_muq_f(s.sct, f);
        s.fastt = f ? 1 : 0;
    }
    // this thread's 16 consecutive sorted keys (vector loads when whole and aligned)
    K kr[HM];
    {
        const int first = t * HM;
        const K* src = kp + first;
        if (first + HM <= n && (((uintptr_t)src) & 15) == 0) {
            constexpr int NV = HM * (int)sizeof(K) / 16;
            const uint4* v4 = reinterpret_cast<const uint4*>(src);
            uint4 buf[NV];
#pragma unroll
            for (int i = 0; i < NV; ++i) buf[i] = v4[i];
            const K* bk = reinterpret_cast<const K*>(buf);
#pragma unroll
            for (int i = 0; i < HM; ++i) kr[i] = bk[i];
        } else {
#pragma unroll
            for (int i = 0; i < HM; ++i) kr[i] = (first + i < n) ? src[i] : (K)0;
        }
    }
    // this thread's entry of the chain thresholds, at the scale the tile's mode uses
    // (computed while the keys are in flight; stored by the prefix after its first barrier)
    static_assert(HM * HM <= HNT, "one threshold entry per thread");
    int thr_v = 0;
    if (t < HM * HM) {
        int shb;
        const bool tbin = ws_tile_binade<T>(kfirst, klast, n, emax, shb);
        uint64_t mlam;
        int sx;
        ws_thr_consts(lamv, KO::L_BASE - emax - (tbin && shb > 0 ? shb : 0), mlam, sx);
        thr_v = ws_thr_entry<HM>(t, mlam, sx, ls.len > 1 ? (uint64_t)(ls.len - 1) : 1ull);
    }
    int64_t q0;
    i128 total;
    int bsh;
    const int mode = ws_tile_prefix<T, HNT, HM>(s.pre, kr, kfirst, klast, n, emax, q0, total, bsh,
                                                t < HM * HM ? s.hull.thr + t : nullptr, thr_v);
    int nv;
    if (mode == WS_TILE_BINADE) {
        TilePtsDev<HM> P = ws_dev_pts<HM>(s.pre.s64, s.muqt, s.fastt != 0, (uint64_t)(klast - kfirst), n, s.sct);
        P.thr = s.hull.thr;
        ws_cta_hull<HNT, HM>(s.hull, n, P, s.sct, &nv);
    } else if (mode == WS_TILE_NARROW) {
        const uint64_t range = (uint64_t)(ws_fixed<T>(KO::from_key(klast), emax) - q0);
        TilePtsDev<HM> P = ws_dev_pts<HM>(s.pre.s64, s.muq, s.fast != 0, range, n, s.sc);
        P.thr = s.hull.thr;
        ws_cta_hull<HNT, HM>(s.hull, n, P, s.sc, &nv);
    } else {
        const TilePtsWide<HM> P{s.pre.s64, s.pre.base, s.muq, s.fast != 0};
        if (ic_cap <= 0 || !wsh::wide_rounds(s.hull, s.ends, n, P, s.sc, ic_cap, &nv))
            ws_cta_hull<HNT, HM>(s.hull, n, P, s.sc, &nv);
    }
    {
        const int l = s.hull.lo[t], h = s.hull.hi[t], o = s.hull.cum[t];
        const size_t b = (size_t)tile * (HT + 1);
        for (int i = l; i < h; ++i) {
            const int pnt = s.hull.H[i * HNT + t];
            vp[b + o + (i - l)] = (uint16_t)pnt;
            vx[b + o + (i - l)] = ws_tile_X<HM>(s.pre.s64, s.pre.base, mode, q0, bsh, pnt);
        }
    }
    if (t == 0) {
        nvert[tile] = nv;
        hx[tile] = TileX{0, 0, 1};
        __stcg(reinterpret_cast<uint4*>(tile_total + tile), *reinterpret_cast<const uint4*>(&total));
    }
    }
}

// ---------------------------------------------------------------------------
// 3. the tree of bridge merges across tiles, for segments whose junctions do
// not resolve locally and are not one cluster (seg_mode 3 with seg_below).  All tile hulls are written.  A CTA takes
// one hull tile after another (a small grid); for each it starts the tile's
// node list, then climbs: at each level the CTA that arrives second merges
// the two children of the parent, the first one goes on to its next tile.
// Nobody waits.
// ---------------------------------------------------------------------------
constexpr int CLIMB_CACHE = 1024;   // piece lists up to this long are searched from shared memory

struct ClimbSmem {
    MergeSmem ms;
    Piece cache[CLIMB_CACHE];
    int go;
    SegConst sc;
};

__global__ void __launch_bounds__(HNT) k_climb(const TileDesc* __restrict__ htiles, const LargeSeg* __restrict__ lsegs,
                                               const TileScale* __restrict__ scales, const uint16_t* vp, const VertX vx,
                                               const int32_t* __restrict__ nvert, i128* tile_total, Piece* pieces,
                                               int32_t* npieces, int32_t* arrive, int n_hull,
                                               const int32_t* __restrict__ seg_mode,
                                               const int32_t* __restrict__ seg_below) {
    __shared__ ClimbSmem s;
    const int t = threadIdx.x;
    ws_chain();
    auto to_climb = [&](int lseg) { return seg_mode[lseg] == 3 && seg_below[lseg] != 0; };
    // Most calls have no segment left for the tree: all threads check this
    // CTA's tiles at once, instead of one tile per round trip in the loop below.
    bool any = false;
    for (int tile = blockIdx.x + t * gridDim.x; tile < n_hull; tile += HNT * gridDim.x)
        any |= to_climb(htiles[tile].lseg);
    if (!__syncthreads_or(any)) return;
    for (int tile = blockIdx.x; tile < n_hull; tile += gridDim.x) {
    const TileDesc td = htiles[tile];
    if (!to_climb(td.lseg)) continue;   // (uniform)
    __syncthreads();   // (the previous tile's shared memory is dead)
    const LargeSeg ls = lsegs[td.lseg];
    if (t == 0) {
        s.sc = ws_seg_scale(scales, td.lseg);
        Piece pc;
        pc.tile = tile; pc.lo = 0; pc.hi = (uint16_t)nvert[tile]; pc.cum = 0; pc.pad = 0; pc.off = 0;
        ws_st_piece(pieces + tile, pc);
        __stcg(npieces + tile, 1);
    }
    __syncthreads();
    const int nt = ls.hull_count, tin = td.tin;
    for (int level = 0; (1 << level) < nt; ++level) {
        const int span = 1 << level;
        const int parent_base = (tin >> (level + 1)) << (level + 1);
        const int right_base = parent_base + span;
        if (right_base >= nt) continue;   // no right sibling: the parent is this node
        __threadfence();                  // this CTA's writes of the child are visible GPU-wide ...
        __syncthreads();
        if (t == 0) {                     // ... before its arrival is counted
            const int old = atomicAdd(&arrive[(size_t)(level + 1) * n_hull + ls.hull_first + parent_base], 1);
            __threadfence();
            s.go = (old == 1);
        }
        __syncthreads();
        if (!s.go) break;
        ws_merge_children(s.ms, pieces, npieces, tile_total, ls.hull_first + parent_base, ls.hull_first + right_base,
                          vp, vx, ls.hull_first, s.sc, s.cache, CLIMB_CACHE);
    }
    }
}

// ---------------------------------------------------------------------------
// 4. root of each segment: cluster count, piece index per tile
// ---------------------------------------------------------------------------
// `parts` CTAs per segment share the numbering; the first also writes the list
// of a segment that the chord check left as one cluster (its first and its last
// point).
__global__ void __launch_bounds__(256) k_root(const LargeSeg* __restrict__ lsegs, const int32_t* __restrict__ nvert,
                                              const i128* __restrict__ tile_base, const int32_t* __restrict__ seg_mode,
                                              const int32_t* __restrict__ seg_below, Piece* pieces, int32_t* npieces,
                                              int32_t* tile_piece, SegRuntime* rt, int64_t* n_clusters_out,
                                              int parts) {
    ws_chain();
    const int lseg = blockIdx.x / parts, part = blockIdx.x % parts;
    const LargeSeg& ls = lsegs[lseg];
    const int h0 = ls.hull_first;
    if (seg_mode[lseg] == 3 && !seg_below[lseg]) {   // (uniform)
        if (part != 0 || threadIdx.x != 0) return;
        const int kl = ls.hull_count - 1, nvl = nvert[h0 + kl];
        Piece a;
        a.tile = h0; a.lo = 0; a.hi = 1; a.cum = 0; a.pad = 0; a.off = 0;
        int np = 1;
        if (kl == 0) {   // one tile: the chord is its hull
            a.hi = (uint16_t)nvl;
        } else {
            Piece z;
            z.tile = h0 + kl; z.lo = (uint16_t)(nvl - 1); z.hi = (uint16_t)nvl; z.cum = 1; z.pad = 0;
            z.off = tile_base[h0 + kl];
            pieces[h0 + 1] = z;
            tile_piece[h0 + kl] = 1;
            np = 2;
        }
        pieces[h0] = a;
        npieces[h0] = np;
        tile_piece[h0] = 0;
        const int64_t c = kl == 0 ? nvl - 1 : 1;
        rt[lseg].n_clusters = c;
        rt[lseg].table_pos = ls.kpos + lseg;
        if (n_clusters_out) n_clusters_out[ls.seg] = c;
        return;
    }
    const Piece* P = pieces + h0;
    const int np = npieces[h0];
    for (int i = part * 256 + threadIdx.x; i < np; i += 256 * parts) tile_piece[P[i].tile] = i;
    if (part == 0 && threadIdx.x == 0) {
        const Piece last = P[np - 1];
        const int64_t c = (int64_t)last.cum + (last.hi - last.lo) - 1;
        rt[lseg].n_clusters = c;
        rt[lseg].table_pos = ls.kpos + lseg;
        if (n_clusters_out) n_clusters_out[ls.seg] = c;
    }
}

// ---------------------------------------------------------------------------
// 5. cluster values, and for every 32 sorted positions the bitmap of cluster
// starts among them with the number of starts before them (one CTA per hull
// tile).  The cluster of a sorted position is then one word away; no search by
// value is needed.  A cluster of at most SUM_MAX elements takes its exact sum
// from the tile's keys (4 bytes per element, in shared memory) instead of the
// prefix sums at its two vertices (16 bytes each): the same integer.  Bound by
// issue (0.66; the values' 64-bit sums and one division per cluster); from the
// prefix sums alone it took 460 us at 2^26, lambda 1e-2, instead of 311.  SUM_MAX
// 2, 4, 8, 16: 457, 357, 295, 295 us there, 95, 90, 84, 79 at 2^24, lambda 1, 60, 63,
// 64, 65 for FP64 2^22, lambda 1 (eight sums of 2^58 are the most that 64 bits hold).
// ---------------------------------------------------------------------------
constexpr int HTW = HT / 32;   // rank words per hull tile
constexpr int SUM_MAX = 8;

template <typename T>
__global__ void __launch_bounds__(256, 6) k_values(const TileDesc* __restrict__ htiles, const LargeSeg* __restrict__ lsegs,
                                                const TileScale* __restrict__ scales, const SegRuntime* __restrict__ rt,
                                                const typename KeyOf<T>::K* __restrict__ sorted,
                                                const uint16_t* __restrict__ vp, const VertX vx,
                                                const Piece* __restrict__ pieces,
                                                const int32_t* __restrict__ npieces,
                                                const int32_t* __restrict__ tile_piece, T* cval, uint2* rank_words,
                                                int fp64, const WsEpi ep, uint32_t* status) {
    typedef KeyOf<T> KO;
    typedef typename KO::K K;
    __shared__ __align__(16) K key[HT];
    __shared__ uint32_t words[HTW];
    __shared__ int wsum[8];
    __shared__ int s_base;
    ws_chain();
    const int tile = blockIdx.x, t = threadIdx.x;
    const int tp = tile_piece[tile];
    const TileDesc td = htiles[tile];
    const TileX tx = vx.h[tile];
    const LargeSeg& ls = lsegs[td.lseg];
    const int h0 = ls.hull_first;
    const int64_t kpos = ls.kpos, n_clusters = rt[td.lseg].n_clusters, table_pos = rt[td.lseg].table_pos;
    if (n_clusters == 1 && tp < 0) return;   // (one cluster: every position has it)
    const Piece* P = pieces + h0;
    const int np = npieces[h0];
    if (t < HTW) words[t] = 0;
    if (tp >= 0 && n_clusters != 1) {
        // (a segment's keys start on 16 bytes, and so does each of its tiles)
        constexpr int VEC = 16 / (int)sizeof(K);
        const uint4* src = reinterpret_cast<const uint4*>(sorted + td.kpos);
        const int nv = td.len / VEC;
        for (int i = t; i < nv; i += 256) reinterpret_cast<uint4*>(key)[i] = __ldg(src + i);
        for (int i = nv * VEC + t; i < td.len; i += 256) key[i] = sorted[td.kpos + i];
    }
    if (t == 0) {
        // starts before this tile; a junction point that the tile on the left
        // keeps as its last vertex is this tile's position 0
        int prev, base;
        if (tp >= 0) { prev = tp - 1; base = P[tp].cum; }
        else {
            int lo = 0, hi = np - 1;   // last piece of an earlier tile (piece 0 is tile 0's)
            while (lo < hi) {
                const int mid = (lo + hi + 1) >> 1;
                if (P[mid].tile < tile) lo = mid; else hi = mid - 1;
            }
            prev = lo;
            base = P[lo].cum + (P[lo].hi - P[lo].lo);
        }
        int bit0 = 0;
        if (prev >= 0) {
            const Piece q = P[prev];
            bit0 = q.tile == tile - 1 && vp[(size_t)q.tile * (HT + 1) + q.hi - 1] == HT;
        }
        s_base = base - bit0;
        words[0] = (uint32_t)bit0;
    }
    __syncthreads();
    if (tp >= 0) {
        const int emax = rt[td.lseg].emax;
        const SegConst sc = ws_seg_scale(scales, td.lseg);
        const Piece pc = P[tp];
        const uint16_t* vpt = vp + (size_t)tile * (HT + 1);
        const int64_t p0 = (int64_t)td.tin * HT;
        int sh = 0;
        const bool bin = n_clusters != 1 && ws_tile_binade<T>(key[0], key[td.len - 1], td.len, emax, sh);
        const int64_t q0 = bin ? ws_fixed<T>(KO::from_key(key[0]), emax) : 0;
        int i = pc.lo + t;
        int al = i < pc.hi ? vpt[i] : 0, bl = i + 1 < pc.hi ? vpt[i + 1] : -1;
        while (i < pc.hi) {
            const int in = i + 256;   // (the next vertices are on their way while this one's value is formed)
            const int an = in < pc.hi ? vpt[in] : 0, bn = in + 1 < pc.hi ? vpt[in + 1] : -1;
            const int64_t r = (int64_t)pc.cum + (i - pc.lo);
            if (r < n_clusters) {   // (the final vertex, point d, opens no cluster)
                const int64_t a = p0 + al;
                int64_t b = p0 + bl;
                i128 SX = 0;
                T xs = (T)0;
                bool done = false;
                if (bl >= 0 && bl - al <= SUM_MAX && n_clusters != 1) {
                    xs = KO::from_key(key[al]);
                    int64_t q = 0;   // (|q| <= 8 x 2^58)
                    const int n = bl - al;
                    if (n > 1) {
                        if (bin) {   // (deviations from the tile's first key, in ulps of its binade)
                            uint64_t dev = 0;
                            for (int j = al; j < bl; ++j) dev += (uint64_t)(key[j] - key[0]);
                            q = (int64_t)n * q0 + (int64_t)(dev << sh);
                        } else {
                            for (int j = al; j < bl; ++j) q += ws_fixed<T>(KO::from_key(key[j]), emax);
                        }
                    }
                    if (sizeof(T) == 4 && !fp64) {
                        cval[table_pos + r] = (T)ValueOut<float>::value64(q, n, (int)(sc.d - a - b), (float)xs, sc, ep);
                        done = true;
                    }
                    SX = (i128)q;
                } else {
                    bool ok = true;
                    if (bl >= 0) {
                        SX = vx.step(tx, tile, i, bl - al);
                    } else if (tp + 1 < np) {
                        const Piece q = P[tp + 1];
                        const int at = vp[(size_t)q.tile * (HT + 1) + q.lo];
                        b = (int64_t)(q.tile - h0) * HT + at;
                        SX = q.off + vx.at(q.tile, q.lo, at) - (pc.off + vx.at(tile, i, al));
                    } else {
                        ok = false;
                        ws_flag(status, WS_STATUS_INTERNAL);
                    }
                    if (ok) {
                        if (b - a == 1) xs = KO::from_key(sorted[kpos + a]);
                    } else b = a + 1;
                }
                if (!done) cval[table_pos + r] = ValueOut<T>::value(SX, a, b, xs, sc, fp64 != 0, ep);
                if (al < HT) atomicOr(&words[al >> 5], 1u << (al & 31));
            }
            i = in;
            al = an;
            bl = bn;
        }
    }
    if (n_clusters == 1) return;
    __syncthreads();
    const uint32_t wd = t < HTW ? words[t] : 0u;
    const int ex = ws_block_excl_scan<256, int>(__popc(wd), wsum, nullptr);
    if (t < HTW) rank_words[(size_t)tile * HTW + t] = make_uint2(wd, (uint32_t)(s_base + ex));
}

// Cluster of a sorted position from its rank word.
__device__ __forceinline__ int ws_cluster_at(uint2 rw, uint32_t pos) {
    return (int)rw.y + __popc(rw.x & (0xffffffffu >> (31u - (pos & 31u)))) - 1;
}

// ---------------------------------------------------------------------------
// 6. the way back to the caller's order: the passes of the sort undone one by
// one.  Every step reads and writes runs (a bin, a tile's bucket runs), never
// single elements all over memory, which is what a lookup of every weight by
// value costs (one or two random sectors each).  Against a table of clusters
// with a directory of 2^22 value buckets and such a lookup, us: 2^26 FP32
// lambda 1e-2: table 449 + lookup 1533 -> values 289, bins 199, regroup 228,
// output 233; 2^24 lambda 1: 120 + 42 + 212 -> 82, 53, 65, 61; 1024 uneven
// segments: 878 + 101 + 1241 -> 498, 309, 340 (no second pass).  The sort pays
// for it by writing where the keys go: 6 bytes per key and a few per run.
// ---------------------------------------------------------------------------
// Bins: value and cluster of every sorted position, put into the order the
// partition left the bin in (in shared memory).  One CTA per bin; the CTAs after
// those share the tiles of the oversize bins.

// Oversize bins, elements [o0, o0 + n) of a bin at a time: an element takes its
// place from the classes that the sort cut the bin into.  One cluster holds a tie,
// so the ties' values are looked up once per bin, and only the elements between
// splitters look for their key (by bisection, in their class).
template <typename T>
struct OverOutSmem {
    typename KeyOf<T>::K spl[OVER_SPL + 1];
    uint32_t start[2 * OVER_SPL + 2];
    OutPair<T> tie[OVER_SPL];
    int wsum[8];
};
template <typename T>
__device__ __noinline__ void bin_out_oversize(OverOutSmem<T>& s, int cta, int n_ctas, int cnt,
                                              const LargeSeg* __restrict__ lsegs, const SegRuntime* __restrict__ rt,
                                              const uint2* __restrict__ rank_words, const T* __restrict__ cval,
                                              const typename KeyOf<T>::K* __restrict__ sorted,
                                              const typename KeyOf<T>::K* __restrict__ keys,
                                              const OverBin* __restrict__ over,
                                              const OverTab<typename KeyOf<T>::K>* __restrict__ tabs, OutPair<T>* pairs) {
    typedef typename KeyOf<T>::K K;
    constexpr int TILE = WS_SORT_TILE, U = 4;
    const int t = threadIdx.x;
    // this CTA's tiles, contiguous: a table serves all tiles of its bin
    const int n_tiles = over[cnt - 1].first_tile + (over[cnt - 1].n + TILE - 1) / TILE;
    int tile = (int)((int64_t)n_tiles * cta / n_ctas);
    const int t1 = (int)((int64_t)n_tiles * (cta + 1) / n_ctas);
    int e = 0;
    for (int hi = cnt - 1; e < hi;) {
        const int mid = (e + hi + 1) >> 1;
        if (over[mid].first_tile <= tile) e = mid; else hi = mid - 1;
    }
    for (; tile < t1; ++e) {
        const OverBin ob = over[e];
        const int te = min(t1, ob.first_tile + (ob.n + TILE - 1) / TILE);
        const LargeSeg& sg = lsegs[ob.lseg];
        const int64_t c = rt[ob.lseg].n_clusters;
        if (c == 1) { tile = te; continue; }   // (one cluster: every element has it)
        const uint2* sw = rank_words + (size_t)sg.hull_first * HTW;
        const T* cv = cval + rt[ob.lseg].table_pos;
        const uint32_t pos0 = (uint32_t)(ob.start - sg.kpos);   // the bin's first sorted position
        auto pair_at = [&](uint32_t r) {
            const uint32_t p = pos0 + min(r, (uint32_t)ob.n - 1u);
            OutPair<T> o = {};
            o.id = ws_cluster_at(__ldg(sw + (p >> 5)), p);
            o.val = __ldg(cv + min(max((int64_t)o.id, (int64_t)0), c - 1));
            return o;
        };
        const int S = ob.nspl;
        __syncthreads();   // (the previous bin's table is dead)
        // (two classes a thread: between splitters, and equal to the next one)
        static_assert(OVER_SPL < 256, "a thread per splitter");
        const int between = t <= S ? (int)tabs[e].cnt[2 * t] : 0, tie = t < S ? (int)tabs[e].cnt[2 * t + 1] : 0;
        const int ex = ws_block_excl_scan<256, int>(between + tie, s.wsum, nullptr);
        if (t <= S) {
            s.start[2 * t] = (uint32_t)ex;
            s.start[2 * t + 1] = (uint32_t)(ex + between);
            if (tie > 0) s.tie[t] = pair_at((uint32_t)(ex + between));
        }
        if (t <= OVER_SPL) s.spl[t] = t < S ? tabs[e].spl[t] : ~(K)0;
        __syncthreads();
        const K* sk = sorted + ob.start;
        const int o0 = (tile - ob.first_tile) * TILE, o1 = min((te - ob.first_tile) * TILE, ob.n);
        for (int i0 = o0 + t; i0 < o1; i0 += 256 * U) {
            K k[U];
#pragma unroll
            for (int u = 0; u < U; ++u) k[u] = __ldg(keys + ob.start + min(i0 + u * 256, o1 - 1));
            int cl[U];
            ws_over_classes<K, U>(s.spl, S, k, cl);
            // (first position whose key is not below the element's; the searches go side by side)
            uint32_t r[U], m[U], more = 0;
#pragma unroll
            for (int u = 0; u < U; ++u) {
                r[u] = s.start[cl[u]];
                m[u] = cl[u] & 1 ? 0u : s.start[cl[u] + 1] - r[u];
                more |= m[u];
            }
            for (; more != 0; more >>= 1) {
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const uint32_t half = m[u] >> 1;
                    const bool below = m[u] != 0 && sk[min(r[u] + half, (uint32_t)ob.n - 1u)] < k[u];
                    if (below) r[u] += half + 1;
                    m[u] = below ? m[u] - half - 1 : half;
                }
            }
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (i0 + u * 256 < o1) pairs[ob.start + i0 + u * 256] = cl[u] & 1 ? s.tie[cl[u] >> 1] : pair_at(r[u]);
        }
        tile = te;
    }
}

// (FP64: the staged pairs allow three CTAs; at six, 24/32 bytes of spills cost 5 of 64 us for 7.4M weights)
template <typename T>
__global__ void __launch_bounds__(256, sizeof(T) == 4 ? 6 : 3) k_bin_out(const LargeSeg* __restrict__ lsegs, const SegRuntime* __restrict__ rt,
                                                 const int32_t* __restrict__ bin_seg,
                                                 const uint32_t* __restrict__ bin_start,
                                                 const uint32_t* __restrict__ bin_cnt, int n_bins,
                                                 const uint16_t* __restrict__ bin_idx,
                                                 const uint2* __restrict__ rank_words, const T* __restrict__ cval,
                                                 const typename KeyOf<T>::K* __restrict__ sorted,
                                                 const typename KeyOf<T>::K* __restrict__ keys,
                                                 const SortCtl* __restrict__ ctl, const OverBin* __restrict__ over,
                                                 const OverTab<typename KeyOf<T>::K>* __restrict__ tabs, OutPair<T>* pairs) {
    typedef typename KeyOf<T>::K K;
    __shared__ uint2 rw[HTW + 2];
    extern __shared__ __align__(16) unsigned char pair_smem_raw[];
    OutPair<T>* stage = reinterpret_cast<OutPair<T>*>(pair_smem_raw);   // [WS_BIN_CAP]
    const int t = threadIdx.x;
    ws_chain();
    if ((int)blockIdx.x < n_bins) {
        const int bin = blockIdx.x;
        const int lseg = bin_seg[bin];
        const LargeSeg& sg = lsegs[lseg];
        const int64_t c = rt[lseg].n_clusters;
        const int n = (int)bin_cnt[bin];
        const uint32_t s0 = bin_start[bin];
        if (c == 1 || n <= 0 || n > WS_BIN_CAP || (int64_t)s0 + n > sg.len) return;
        const int64_t g = sg.kpos + s0;
        constexpr int U = 6;   // (a bin of the usual size in two steps)
        const uint32_t w0 = s0 >> 5, nw = ((s0 + n - 1) >> 5) - w0 + 1;
        const T* cv = cval + rt[lseg].table_pos;
        if (t < nw) rw[t] = rank_words[(size_t)sg.hull_first * HTW + w0 + t];   // (nw <= HTW + 1)
        for (int b0 = 0; b0 < n; b0 += 256 * U) {
            const int i0 = b0 + t;
            uint16_t q[U];
            T v[U];
#pragma unroll
            for (int u = 0; u < U; ++u) q[u] = i0 + u * 256 < n ? __ldg(bin_idx + g + i0 + u * 256) : (uint16_t)0;
            if (b0 == 0) __syncthreads();   // (the rank words; the places are on their way)
            auto id_at = [&](int u) {
                const uint32_t p = s0 + min(i0 + u * 256, n - 1);
                return ws_cluster_at(rw[(p >> 5) - w0], p);
            };
#pragma unroll
            for (int u = 0; u < U; ++u) v[u] = __ldg(cv + min(max(id_at(u), 0), (int)c - 1));
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (i0 + u * 256 < n) {
                    OutPair<T> o = {};
                    o.val = v[u];
                    o.id = id_at(u);
                    stage[min((uint32_t)q[u], (uint32_t)n - 1u)] = o;
                }
        }
        __syncthreads();
        for (int i = t; i < n; i += 256) pairs[g + i] = stage[i];
        return;
    }
    const int cnt = (int)ctl->over_count;
    if (cnt == 0 || ctl->abort) return;
    bin_out_oversize<T>(*reinterpret_cast<OverOutSmem<T>*>(pair_smem_raw), (int)blockIdx.x - n_bins,
                        (int)gridDim.x - n_bins, cnt, lsegs, rt, rank_words, cval, sorted, keys, over, tabs, pairs);
}

// A pass undone tile by tile: the tile's pairs are read run by run into shared
// memory, where every element then finds its own.  Bound by DRAM latency and
// bytes (2^26: 18 bytes per element, 0.78 of the copy rate).  A gather of every
// pair through a 4-byte destination took one line per lane and clock of the L1
// and 20 bytes: regroup 245 -> 228 us, output 286 -> 233 at 2^26, 406 -> 340 for
// 1024 uneven segments.
constexpr int GNT = WS_SORT_NT;

// The places of this thread's elements t + k GNT, two to a word (loaded first: they
// arrive while the tile is staged).
__device__ __forceinline__ void ws_load_places(uint32_t (&pl)[WS_SORT_TILE / GNT / 2], const uint16_t* loc, int len) {
#pragma unroll
    for (int k = 0; k < WS_SORT_TILE / GNT; k += 2) {
        const int a = min((int)threadIdx.x + k * GNT, len - 1), b = min((int)threadIdx.x + (k + 1) * GNT, len - 1);
        pl[k / 2] = (uint32_t)__ldg(loc + a) | ((uint32_t)__ldg(loc + b) << 16);
    }
}

// The tile's pairs, run by run (neighbouring lanes read neighbouring pairs), into
// the tile's staging order.  Bounds hold whatever the maps contain.
template <typename T>
__device__ __forceinline__ void ws_stage_tile(OutPair<T>* stage, uint32_t* words, uint32_t* pre, int* wsum,
                                              const PassMap& m, int tile, int64_t dpos, int max_run, int len,
                                              const OutPair<T>* __restrict__ src, uint32_t last) {
    constexpr int W = WS_SORT_TILE / 32, U = 6;
    static_assert(W <= GNT && WS_SORT_TILE % (GNT * U) == 0, "a thread per word; whole steps");
    const int t = threadIdx.x;
    const uint32_t wd = t < W ? __ldg(m.starts + (int64_t)tile * W + t) : 0u;
    const int ex = ws_block_excl_scan<GNT, int>(__popc(wd), wsum, nullptr);
    if (t < W) { words[t] = wd; pre[t] = (uint32_t)ex; }
    __syncthreads();
    for (int j0 = t; j0 < len; j0 += GNT * U) {
        uint32_t p[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int j = min(j0 + u * GNT, len - 1);
            const int r = (int)pre[j >> 5] + __popc(words[j >> 5] & (0xffffffffu >> (31 - (j & 31)))) - 1;
            p[u] = min((uint32_t)j + __ldg(m.delta + dpos + max(min(r, max_run - 1), 0)), last);
        }
        OutPair<T> o[U];
#pragma unroll
        for (int u = 0; u < U; ++u) o[u] = src[p[u]];
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (j0 + u * GNT < len) stage[j0 + u * GNT] = o[u];
    }
    __syncthreads();
}

template <typename T>
__global__ void __launch_bounds__(GNT, sizeof(T) == 4 ? 3 : 2) k_regroup(
    const TileDesc* __restrict__ tiles, const LargeSeg* __restrict__ lsegs, const SegRuntime* __restrict__ rt,
    const PassMap map, const OutPair<T>* __restrict__ from, OutPair<T>* __restrict__ to) {
    extern __shared__ __align__(16) unsigned char pair_smem_raw[];
    __shared__ uint32_t words[WS_SORT_TILE / 32], pre[WS_SORT_TILE / 32];
    __shared__ int wsum[GNT / 32];
    OutPair<T>* stage = reinterpret_cast<OutPair<T>*>(pair_smem_raw);   // [WS_SORT_TILE]
    ws_chain();
    const TileDesc td = tiles[blockIdx.x];
    const LargeSeg& sg = lsegs[td.lseg];
    if (sg.fine_log2 == 0 || rt[td.lseg].n_clusters == 1) return;
    uint32_t pl[WS_SORT_TILE / GNT / 2];
    ws_load_places(pl, map.loc + td.kpos, td.len);
    ws_stage_tile<T>(stage, words, pre, wsum, map, blockIdx.x, td.kpos, td.len, td.len, from + sg.kpos,
                     (uint32_t)sg.len - 1u);
#pragma unroll
    for (int k = 0; k < WS_SORT_TILE / GNT; ++k) {
        const int i = threadIdx.x + k * GNT;
        if (i < td.len) to[td.kpos + i] = stage[min((int)(pl[k / 2] >> (16 * (k & 1)) & 0xffffu), td.len - 1)];
    }
}

// First pass undone: value and id of every element, in the caller's order.
template <typename T>
__global__ void __launch_bounds__(GNT, sizeof(T) == 4 ? 3 : 2) k_output(
    const TileDesc* __restrict__ tiles, const LargeSeg* __restrict__ lsegs, const SegRuntime* __restrict__ rt,
    const T* __restrict__ cval, const PassMap map, const OutPair<T>* __restrict__ pairs_a,
    const OutPair<T>* __restrict__ pairs_b, T* out, int32_t* ids) {
    extern __shared__ __align__(16) unsigned char pair_smem_raw[];
    __shared__ uint32_t words[WS_SORT_TILE / 32], pre[WS_SORT_TILE / 32];
    __shared__ int wsum[GNT / 32];
    OutPair<T>* stage = reinterpret_cast<OutPair<T>*>(pair_smem_raw);   // [WS_SORT_TILE]
    ws_chain();
    const TileDesc td = tiles[blockIdx.x];
    const LargeSeg& sg = lsegs[td.lseg];
    if (rt[td.lseg].n_clusters == 1) {   // one cluster (large lambda): every weight gets its value
        const T v = cval[rt[td.lseg].table_pos];
        for (int i = threadIdx.x; i < td.len; i += GNT) {
            __stcs(out + td.vpos + i, v);
            if (ids) __stcs(ids + td.vpos + i, 0);
        }
        return;
    }
    uint32_t pl[WS_SORT_TILE / GNT / 2];
    ws_load_places(pl, map.loc + td.kpos, td.len);
    ws_stage_tile<T>(stage, words, pre, wsum, map, blockIdx.x, (int64_t)blockIdx.x * WS_FAN, WS_FAN, td.len,
                     (sg.fine_log2 ? pairs_a : pairs_b) + sg.kpos, (uint32_t)sg.len - 1u);
#pragma unroll
    for (int k = 0; k < WS_SORT_TILE / GNT; ++k) {
        const int i = threadIdx.x + k * GNT;
        if (i >= td.len) break;
        const OutPair<T> o = stage[min((int)(pl[k / 2] >> (16 * (k & 1)) & 0xffffu), td.len - 1)];
        __stcs(out + td.vpos + i, o.val);
        if (ids) __stcs(ids + td.vpos + i, o.id);
    }
}

template <typename T>
__global__ void k_copy_sorted(const typename KeyOf<T>::K* __restrict__ sorted, const TileDesc* __restrict__ tiles,
                              T* dst) {
    const TileDesc td = tiles[blockIdx.x];
    for (int i = threadIdx.x; i < td.len; i += 256) dst[td.vpos + i] = KeyOf<T>::from_key(sorted[td.kpos + i]);
}

}  // namespace

// ---------------------------------------------------------------------------
// host-side sequencing of the large path
// ---------------------------------------------------------------------------
template <typename T>
cudaError_t ws_large_prox(const LargeWork<T>& W, const T* values, WsLambda lambdas, T* out, int32_t* ids,
                          int64_t* n_clusters, int fp64, const WsEpi& ep, uint32_t* status, uint64_t spin_limit,
                          cudaStream_t st) {
    typedef typename KeyOf<T>::K K;
    if (W.n_lseg == 0) return cudaSuccess;
    K* sorted = nullptr;
    cudaError_t e = ws_large_sort<T>(W, values, true, status, spin_limit, st, &sorted);
    if (e) return e;
    // tile hulls: the lean kernel, then the general one for the tiles it flagged
    e = ws_large_hull_fast<T>(W, sorted, lambdas, status, st);
    if (e) return e;
    size_t smem = sizeof(TileHullSmem);
    e = cudaFuncSetAttribute(k_tile_hull<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e) return e;
    const int small_grid = W.n_hull_tiles < 4 * 152 ? W.n_hull_tiles : 4 * 152;
    WS_LAUNCH(W.prof, WSK_TILE_GENERAL, st,
              ws_launch_chain(k_tile_hull<T>, small_grid, HNT, smem, st, sorted, W.hull_tiles, W.lsegs, lambdas, W.rt,
                              W.vp, W.vx, W.hx, W.nvert, W.tile_total, W.gen_list, &W.ctl->gen_count, W.seg_emin, W.ic_cap,
                              status));
    // across tiles: junction bridges and the per-segment resolution, then the
    // tree of merges for the segments that need it
    e = ws_large_junctions<T>(W, st);
    if (e) return e;
    WS_LAUNCH(W.prof, WSK_CLIMB, st,
              ws_launch_chain(k_climb, small_grid, HNT, 0, st, W.hull_tiles, W.lsegs, W.scales, W.vp, VertX{W.vx, W.hx}, W.nvert,
                              W.tile_total, W.pieces, W.npieces, W.arrive, W.n_hull_tiles, W.seg_mode, W.seg_below));
    // CTAs per segment of the numbering: one per 1024 tiles of an average segment
    const int parts = std::max(1, std::min(16, W.n_hull_tiles / W.n_lseg / 1024));
    WS_LAUNCH(W.prof, WSK_ROOT, st,
              ws_launch_chain(k_root, W.n_lseg * parts, 256, 0, st, W.lsegs, W.nvert, W.tile_base, W.seg_mode,
                              W.seg_below, W.pieces, W.npieces, W.tile_piece, W.rt, n_clusters, parts));
    WS_LAUNCH(W.prof, WSK_VALUES, st,
              ws_launch_chain(k_values<T>, W.n_hull_tiles, 256, 0, st, W.hull_tiles, W.lsegs, W.scales, W.rt, sorted,
                              W.vp, VertX{W.vx, W.hx}, W.pieces, W.npieces, W.tile_piece, W.cval, W.rank_words, fp64, ep, status));
    // back to the caller's order
    const size_t osm = sizeof(OutPair<T>) * WS_BIN_CAP;
    static_assert(sizeof(OverOutSmem<T>) <= sizeof(OutPair<T>) * WS_BIN_CAP, "in the same shared memory");
    e = cudaFuncSetAttribute(k_bin_out<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)osm);
    if (e) return e;
    WS_LAUNCH(W.prof, WSK_BIN_OUT, st,
              ws_launch_chain(k_bin_out<T>, W.n_bins + W.sort_shape.out_extra, 256, osm, st, W.lsegs, W.rt, W.bin_seg, W.bin_start,
                              W.bin_cnt, W.n_bins, W.bin_idx, W.rank_words, W.cval, sorted, W.keys_b, W.ctl, W.over,
                              reinterpret_cast<const OverTab<K>*>(W.over_tabs), W.pairs_b));
    const size_t gsm = sizeof(OutPair<T>) * WS_SORT_TILE;
    if ((e = cudaFuncSetAttribute(k_regroup<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)gsm)) ||
        (e = cudaFuncSetAttribute(k_output<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)gsm)))
        return e;
    // (beside the end of their predecessors the two ways back through large grids lose more than the
    // launch gains: 2^26 2540 us per call against 2435, 1024 uneven segments 3490 against 3420; up to two
    // tiles per SM it gains 4 us of 104)
    const bool early = W.n_sort_tiles <= 2 * 152;
    if (W.two_level)
        WS_LAUNCH(W.prof, WSK_REGROUP, st,
                  ws_launch_if(early, k_regroup<T>, W.n_sort_tiles, GNT, gsm, st, W.sort_tiles, W.lsegs, W.rt, W.map2,
                                  W.pairs_b, W.pairs_a));
    WS_LAUNCH(W.prof, WSK_OUTPUT, st,
              ws_launch_if(early, k_output<T>, W.n_sort_tiles, GNT, gsm, st, W.sort_tiles, W.lsegs, W.rt, W.cval, W.map1,
                              W.pairs_a, W.pairs_b, out, ids));
    return cudaGetLastError();
}

template <typename T>
cudaError_t ws_large_copy_sorted(const LargeWork<T>& W, const typename KeyOf<T>::K* sorted, T* dst,
                                 cudaStream_t st) {
    if (W.n_sort_tiles == 0) return cudaSuccess;
    WS_LAUNCH(W.prof, WSK_MISC, st, (k_copy_sorted<T><<<W.n_sort_tiles, 256, 0, st>>>(sorted, W.sort_tiles, dst)));
    return cudaGetLastError();
}

#define WS_INST(T)                                                                                                  \
    template cudaError_t ws_large_prox<T>(const LargeWork<T>&, const T*, WsLambda, T*, int32_t*, int64_t*, int, \
                                          const WsEpi&, uint32_t*, uint64_t, cudaStream_t);                         \
    template cudaError_t ws_large_copy_sorted<T>(const LargeWork<T>&, const typename KeyOf<T>::K*, T*, cudaStream_t);
WS_INST(float)
WS_INST(double)
