// Candidate scan of PLD+ -- Eq. 1 (Sec. 4.2) with the longest-suffix n-gram rule --
// as device building blocks shared by pldp_find_candidates and the drafting calls.
//
// A CTA owns a contiguous chunk of one context and each of its warps a contiguous
// segment of the chunk, 128 positions an iteration (a 16-byte vector per lane).  The
// tokens before a vector's are in the lanes below it, so the suffix-match lengths of
// all 128 positions come from shuffles and compares, without another load and
// without a loop over the matches.  A warp keeps only the positions with the longest
// match it has met so far, in ascending order, in a short list in shared memory: a
// shorter match can no longer be a candidate.  One pass over the ids is thus enough,
// however often x_t occurs (text repeats its frequent tokens thousands of times in a
// long context); a list that overflows is written by a second pass over its segment.
//
// What bounds it: the ids' DRAM round trips (8 vectors in flight per lane) and, for a
// frequent x_t, about 60 instructions per iteration that meets one.  Before, every
// occurrence walked its suffix with one dependent load per token and the positions
// were written by a second pass with two CTA barriers per 1024 positions: on 32k-token
// Zipf contexts (batch 128) the drafting launch took 1240-1490 us and now 125-190 us,
// what is left being the scores of its hundreds of candidates; pldp_find_candidates on
// 16k-token contexts (batch 64, L2 flushed) went from 12.2 to 8.2 us.
#pragma once

#include "pldp_internal.cuh"

namespace pldp {

constexpr int kScanThreads = 256;
constexpr int kScanWarps = kScanThreads / 32;
constexpr int kScanTile = 128;          // positions per warp iteration: a 16-byte vector per lane
constexpr int kScanMaxCluster = 8;      // portable cluster size
constexpr int64_t kScanChunkUnit = int64_t(kScanTile) * kScanWarps;   // a chunk is a multiple of this

// How ids are read: through the read-only cache (a context that no kernel of
// the call writes), or through L2 (a context that the same kernel has just
// appended to, which the read-only path is not guaranteed to see).
struct ReadOnlyIds {
    static __device__ __forceinline__ int32_t one(const int32_t* p) { return __ldg(p); }
    static __device__ __forceinline__ int4 four(const int4* p) { return __ldg(p); }
};
struct CoherentIds {
    static __device__ __forceinline__ int32_t one(const int32_t* p) { return __ldcg(p); }
    static __device__ __forceinline__ int4 four(const int4* p) { return __ldcg(p); }
};

// Positions 4q .. 4q + 3 of a context; positions outside [0, lim) read as 0 (with VEC,
// lim is a multiple of 4 and rows are 16-byte aligned).
template <bool VEC, typename RD>
__device__ __forceinline__ int4 scan_load(const int32_t* __restrict__ row, int64_t q, int64_t lim) {
    int4 v = make_int4(0, 0, 0, 0);
    const int64_t p = 4 * q;
    if constexpr (VEC) {
        if (q >= 0 && p < lim) v = RD::four(reinterpret_cast<const int4*>(row) + q);
    } else {
        if (p >= 0 && p < lim) v.x = RD::one(row + p);
        if (p + 1 >= 0 && p + 1 < lim) v.y = RD::one(row + p + 1);
        if (p + 2 >= 0 && p + 2 < lim) v.z = RD::one(row + p + 2);
        if (p + 3 >= 0 && p + 3 < lim) v.w = RD::one(row + p + 3);
    }
    return v;
}

// The vector `back` (1 or 2) places before each lane's: from the lanes below, and for
// the first lanes from the last lanes of the warp's previous vectors (vp).
__device__ __forceinline__ int4 scan_before(const int4& v, const int4& vp, int back, int lane) {
    const bool hi = lane >= 32 - back;
    const int src = (lane + 32 - back) & 31;
    int4 r;
    r.x = __shfl_sync(0xFFFFFFFFu, hi ? vp.x : v.x, src);
    r.y = __shfl_sync(0xFFFFFFFFu, hi ? vp.y : v.y, src);
    r.z = __shfl_sync(0xFFFFFFFFu, hi ? vp.z : v.z, src);
    r.w = __shfl_sync(0xFFFFFFFFu, hi ? vp.w : v.w, src);
    return r;
}

// Suffix-match lengths of the lane's four positions p .. p + 3 (those below `lim`;
// 0 where the token is not x_t), capped at n_max and at the tokens there are.
// suf = x_t, x_{t-1}, ...
__device__ __forceinline__ void scan_match(const int4& v, const int4& vp, int64_t p, int64_t lim,
                                           const int32_t* suf, int n_max, int lane, int (&m)[4]) {
    const int32_t xt = suf[0];
    bool ok[4] = {v.x == xt && p < lim, v.y == xt && p + 1 < lim, v.z == xt && p + 2 < lim, v.w == xt && p + 3 < lim};
#pragma unroll
    for (int c = 0; c < 4; ++c) m[c] = ok[c] ? 1 : 0;
    if (n_max > 1) {                                          // the tokens at p - 8 .. p + 3
        const int4 b1 = scan_before(v, vp, 1, lane);
        int32_t w[12] = {0, 0, 0, 0, b1.x, b1.y, b1.z, b1.w, v.x, v.y, v.z, v.w};
        if (n_max > 5) {
            const int4 b2 = scan_before(v, vp, 2, lane);
            w[0] = b2.x;
            w[1] = b2.y;
            w[2] = b2.z;
            w[3] = b2.w;
        }
#pragma unroll
        for (int k = 1; k < PLDP_MAX_NGRAM; ++k) {
            if (k >= n_max) break;
            const int32_t s = suf[k];
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                ok[c] = ok[c] && p + c >= k && w[8 + c - k] == s;
                m[c] += ok[c] ? 1 : 0;
            }
        }
    }
}

// Calls put(index, position) for the lane's positions with m == level, index counting
// the warp's from `base` in ascending position order; returns how many the warp has.
template <typename Put>
__device__ __forceinline__ int scan_put(const int (&m)[4], int level, int64_t p, int base, int lane, Put put) {
    const unsigned lt = (1u << lane) - 1u;
    int off = base, n = 0;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        const unsigned bal = __ballot_sync(0xFFFFFFFFu, m[c] == level);
        off += __popc(bal & lt);
        n += __popc(bal);
    }
#pragma unroll
    for (int c = 0; c < 4; ++c)
        if (m[c] == level) put(off++, p + c);
    return n;
}

// One warp's scan of positions [s0, s0 + nit * kScanTile), those below `lim`, U vectors
// in flight per lane.  begin() issues the first loads (ids up to `cap` may be read), so
// that they can be under way before the suffix and the context length are known.
template <bool VEC, typename RD, int U>
struct WarpScan {
    const int32_t* row;
    int64_t q0, cap;                     // the lane's first vector; readable positions
    int nit, lane;
    int4 v[U], vp;

    __device__ __forceinline__ void load(int it0) {
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (it0 + u < nit) v[u] = scan_load<VEC, RD>(row, q0 + static_cast<int64_t>(it0 + u) * 32, cap);
    }
    __device__ __forceinline__ void begin(const int32_t* r, int64_t s0, int iters, int64_t cap_, int lane_) {
        row = r;
        lane = lane_;
        cap = cap_;
        nit = iters;
        q0 = (s0 >> 2) + lane;
        vp = make_int4(0, 0, 0, 0);      // lanes 30, 31: the vectors before the segment
        if (lane >= 30 && nit > 0) vp = scan_load<VEC, RD>(row, q0 - 32, cap);
        load(0);
    }
    // each(m, p): the match lengths of a tile with at least one occurrence of x_t.  One
    // copy of the tile's code walks the vectors by shifting them down (after an L2 flush
    // the kernel's code comes from DRAM: unrolled over the vectors, it cost a
    // drafting call 2-6 us of instruction fetch); tiles without x_t skip it.
    template <typename Each>
    __device__ __forceinline__ void run(int64_t lim, const int32_t* suf, int n_max, Each each) {
        const int32_t xt = suf[0];
#pragma unroll 1
        for (int it0 = 0; it0 < nit && 4 * (q0 - lane) + static_cast<int64_t>(it0) * kScanTile < lim; it0 += U) {
            if (it0 > 0) load(it0);
            unsigned tiles = 0;                               // bit u: this lane has x_t in vector u
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (it0 + u < nit && (v[u].x == xt || v[u].y == xt || v[u].z == xt || v[u].w == xt)) tiles |= 1u << u;
            tiles = __reduce_or_sync(0xFFFFFFFFu, tiles);     // bit u: the warp has
            const int4 last = v[U - 1];
            int64_t p = 4 * (q0 + static_cast<int64_t>(it0) * 32);
#pragma unroll 1
            for (; tiles != 0; tiles >>= 1, p += kScanTile) {
                if (tiles & 1u) {
                    int m[4];
                    scan_match(v[0], vp, p, lim, suf, n_max, lane, m);
                    each(m, p);
                }
                vp = v[0];
#pragma unroll
                for (int k = 0; k + 1 < U; ++k) v[k] = v[k + 1];
            }
            vp = last;
        }
    }
};

// What a CTA found: per warp the longest match length and how many positions have it,
// the first LW of them listed in ascending order.
template <int LW>
struct ScanLists {
    int32_t suf[PLDP_MAX_NGRAM];         // x_t, x_{t-1}, ... (n_max of them)
    int32_t pos[kScanWarps][LW];
    int wm[kScanWarps], wc[kScanWarps];
};

// A warp's pass: leaves its longest match length, their count and its list in `sl`.
template <typename Scan, int LW>
__device__ __forceinline__ void scan_lists(Scan& sc, int64_t lim, int n_max, int warp, ScanLists<LW>& sl) {
    int wm = 0, wc = 0;
    sc.run(lim, sl.suf, n_max, [&](const int (&m)[4], int64_t p) {
        const int mx = __reduce_max_sync(0xFFFFFFFFu, max(max(m[0], m[1]), max(m[2], m[3])));
        if (mx < wm) return;                                  // warp-uniform
        if (mx > wm) {
            wm = mx;
            wc = 0;
        }
        wc += scan_put(m, wm, p, wc, sc.lane, [&](int i, int64_t j) {
            if (i < LW) sl.pos[warp][i] = static_cast<int32_t>(j);
        });
    });
    if (sc.lane == 0) {
        sl.wm[warp] = wm;
        sl.wc[warp] = wc;
    }
}

// The CTA's longest match length, the positions that have it, how many of them lie in
// warps below this one, and whether some warp's list does not hold all of its own.
// Called by every thread after a barrier.
struct CtaMatches {
    int m, cnt, base;
    bool over;
};
template <int LW>
__device__ __forceinline__ CtaMatches cta_matches(const ScanLists<LW>& sl, int warp) {
    CtaMatches r = {0, 0, 0, false};
#pragma unroll
    for (int w = 0; w < kScanWarps; ++w) r.m = max(r.m, sl.wm[w]);
#pragma unroll
    for (int w = 0; w < kScanWarps; ++w) {
        const int c = (r.m > 0 && sl.wm[w] == r.m) ? sl.wc[w] : 0;
        r.base += w < warp ? c : 0;
        r.cnt += c;
        r.over |= c > LW;
    }
    return r;
}

// The warp's positions of match length `level`, by a second pass over its segment (the
// list does not hold them all): put(at + i, j) for the i-th of them, those below C_cap.
// Out of line: few launches run it.
template <bool VEC, typename RD, typename Put>
__device__ __noinline__ void scan_again(const int32_t* __restrict__ row, int64_t s0, int nit, int64_t lim, int64_t cap,
                                        const int32_t* suf, int n_max, int level, int64_t at, int C_cap, int lane,
                                        Put put) {
    WarpScan<VEC, RD, 8> sc;
    sc.begin(row, s0, nit, cap, lane);
    sc.run(lim, suf, n_max, [&](const int (&m)[4], int64_t p) {
        const int64_t base = at;
        at += scan_put(m, level, p, 0, lane, [&](int i, int64_t j) {
            if (base + i < C_cap) put(base + i, static_cast<int32_t>(j));
        });
    });
}

// Writes the warp's positions of match length `level` as candidates at, at + 1, ... in
// ascending order (those below C_cap): put(i, j) for every one of them.
template <bool VEC, typename RD, int LW, typename Put>
__device__ __forceinline__ void scan_emit(const int32_t* __restrict__ row, int64_t s0, int nit, int64_t lim,
                                          int64_t cap, int n_max, int level, int64_t at, int C_cap, int warp, int lane,
                                          const ScanLists<LW>& sl, Put put) {
    if (level < 1 || sl.wm[warp] != level || at >= C_cap) return;
    const int n = sl.wc[warp];
    if (n > LW) {
        scan_again<VEC, RD>(row, s0, nit, lim, cap, sl.suf, n_max, level, at, C_cap, lane, put);
        return;
    }
    for (int i = lane; i < n; i += 32)
        if (at + i < C_cap) put(at + i, sl.pos[warp][i]);
}

// A CTA's outcome as its cluster's peers see it.
struct ScanPeer {
    int m, cnt, over;
};

// n* = the longest match length of the cluster's CTAs (0 below n_min), the candidates
// in all and those in CTAs before `rank`.
struct ScanTotal {
    int nstar, total, before;
    bool over;
};
__device__ __forceinline__ ScanTotal scan_total(const ScanPeer* tab, int CL, int rank, int n_min) {
    ScanTotal r = {0, 0, 0, false};
    for (int k = 0; k < CL; ++k) r.nstar = max(r.nstar, tab[k].m);
    if (r.nstar < n_min) r.nstar = 0;
    if (r.nstar > 0)
        for (int k = 0; k < CL; ++k)
            if (tab[k].m == r.nstar) {
                r.total += tab[k].cnt;
                r.before += k < rank ? tab[k].cnt : 0;
                r.over |= tab[k].over != 0;
            }
    return r;
}

// Cluster barriers, split so that work runs between the two halves.  (A cluster of one
// CTA passes them at once.)
__device__ __forceinline__ void cluster_arrive_relaxed() {
    asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_arrive() {
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() {
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// Cluster size and chunk (a multiple of kScanChunkUnit) for scanning T_cap positions of
// B sequences: one CTA per `per_cta` positions, at most a portable cluster, and no more
// CTAs in all than `resident` (so the grid is a single wave).
inline void scan_shape(int64_t T_cap, int B, int resident, int64_t per_cta, int* CL_out,
                       int64_t* chunk_out) {
    int64_t CL = (T_cap + per_cta - 1) / per_cta;
    const int per_seq = resident / (B > 0 ? B : 1);
    if (CL > per_seq) CL = per_seq;
    CL = CL < 1 ? 1 : (CL > kScanMaxCluster ? kScanMaxCluster : CL);
    int64_t chunk = (T_cap + CL - 1) / CL;
    chunk = (chunk + kScanChunkUnit - 1) / kScanChunkUnit * kScanChunkUnit;
    if (chunk < kScanChunkUnit) chunk = kScanChunkUnit;
    CL = (T_cap + chunk - 1) / chunk;
    *CL_out = static_cast<int>(CL < 1 ? 1 : CL);
    *chunk_out = chunk;
}

}  // namespace pldp
