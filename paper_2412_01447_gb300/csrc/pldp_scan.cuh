// Candidate scan of PLD+ -- Eq. 1 (Sec. 4.2) with the longest-suffix n-gram rule --
// as device building blocks shared by pldp_find_candidates and the drafting calls.
//
// A CTA owns a contiguous chunk of one context and each of its warps a contiguous
// segment of the chunk, 1024 positions a round: eight 16-byte vectors per lane, a bit
// per position in a lane's mask.  The positions equal to x_{t-k} are a mask of 32
// compares; moved up by k positions (shifts inside a lane, one or two shuffles for what
// crosses lanes) it says where the k-th token of the suffix matches, so the longest
// match of the round is a chain of ANDs, whatever the number of matches.  A warp keeps
// only the positions with the longest match it has met so far, in ascending order, in a
// short list in shared memory: a shorter match can no longer be a candidate.  One pass
// over the ids is thus enough, however often x_t occurs (text repeats its frequent
// tokens thousands of times in a long context); a list that overflows is written by a
// second pass over its segment.
//
// What bounds it: the ids' DRAM round trips (8 vectors in flight per lane).  Match
// lengths worked out per position cost 150 instructions per 128 positions wherever x_t
// is frequent (drafting batch 128 x 32k Zipf tokens through the index: 34 us, 21 us with
// masks; its scanning kernel 22 -> 17 us).  Before that, every occurrence walked its
// suffix with one dependent load per token and the positions were written by a second
// pass with two CTA barriers per 1024 positions, which took most of 1240-1490 us of a
// drafting launch over 32k-token Zipf contexts (batch 128).  pldp_find_candidates, batch
// 64 x 16k, L2 flushed: 12.2 -> 8-9.6 us.
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

// Where a lane's vectors hold token s: bit 4 u + c for component c of vector u.
template <int U>
__device__ __forceinline__ uint32_t scan_equal(const int4 (&v)[U], int32_t s) {
    static_assert(U <= 8, "a bit per position");
    uint32_t m = 0;
#pragma unroll
    for (int u = 0; u < U; ++u) {
        m |= v[u].x == s ? 1u << (4 * u) : 0u;
        m |= v[u].y == s ? 2u << (4 * u) : 0u;
        m |= v[u].z == s ? 4u << (4 * u) : 0u;
        m |= v[u].w == s ? 8u << (4 * u) : 0u;
    }
    return m;
}

// The mask f moved up by k positions (1 <= k < 8): a bit stays in its lane or comes from
// one of the two lanes below; the first lanes take theirs from the vector before, in the
// last lanes (before a round's first vectors: fp, the mask of lanes 30 and 31 there).
__device__ __forceinline__ uint32_t scan_move(uint32_t f, uint32_t fp, int k, int lane) {
    const int a = k >> 2, r = k & 3;
    auto below = [&](int d) -> uint32_t {
        return __shfl_sync(0xFFFFFFFFu, lane >= 32 - d ? (f << 4) | fp : f, (lane + 32 - d) & 31);
    };
    const uint32_t near = a ? below(1) : f;
    if (r == 0) return near;
    const uint32_t far = below(a + 1);
    const uint32_t keep = 0x11111111u * ((0xFu << r) & 0xFu);    // components that stay in their lane
    return ((near << r) & keep) | ((far >> (4 - r)) & ~keep);
}

// One warp's scan of positions [s0, s0 + nit * kScanTile), those below a limit, U
// vectors in flight per lane (AHEAD: the next U too, while these are worked on).
// begin() issues the first loads (ids up to `cap` may be read), so that they can be
// under way before the suffix and the context length are known.
template <bool VEC, typename RD, int U, bool AHEAD = false>
struct WarpScan {
    const int32_t* row;
    int64_t q0, cap;                     // the lane's first vector; readable positions
    int nit, lane;
    int4 v[U], vp;

    __device__ __forceinline__ void load(int4 (&x)[U], int it0) const {
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (it0 + u < nit) x[u] = scan_load<VEC, RD>(row, q0 + static_cast<int64_t>(it0 + u) * 32, cap);
    }
    __device__ __forceinline__ void begin(const int32_t* r, int64_t s0, int iters, int64_t cap_, int lane_) {
        row = r;
        lane = lane_;
        cap = cap_;
        nit = iters;
        q0 = (s0 >> 2) + lane;
        vp = make_int4(0, 0, 0, 0);      // lanes 30, 31: the vectors before the segment
        if (lane >= 30 && nit > 0) vp = scan_load<VEC, RD>(row, q0 - 32, cap);
#pragma unroll
        for (int u = 0; u < U; ++u) v[u] = make_int4(0, 0, 0, 0);
        load(v, 0);
    }
    // each(m, mask, p) for every round with an occurrence of x_t = suf[0]: its longest
    // suffix match m (at most n_max) and the positions that have it, bit 4 u + c of a
    // lane's mask standing for p + u * kScanTile + c.
    template <typename Each>
    __device__ __forceinline__ void run(int64_t lim, const int32_t* suf, int n_max, Each each) {
        const int32_t xt = suf[0];
#pragma unroll 1
        for (int it0 = 0; it0 < nit; it0 += U) {
            const int64_t p = 4 * (q0 + static_cast<int64_t>(it0) * 32);      // the lane's first position
            if (p - 4 * lane >= lim) break;                                   // warp-uniform
            int4 nx[AHEAD ? U : 1];
            if constexpr (AHEAD) {
#pragma unroll
                for (int u = 0; u < U; ++u) nx[u] = make_int4(0, 0, 0, 0);
                load(nx, it0 + U);
            } else if (it0 > 0) {
                load(v, it0);
            }
            uint32_t mask = scan_equal<U>(v, xt);
            if (it0 + U > nit) mask &= (1u << (4 * (nit - it0))) - 1u;
            if (p - 4 * lane + static_cast<int64_t>(U) * kScanTile > lim) {   // the context ends in this round
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const int64_t left = lim - (p + u * kScanTile);
                    if (left < 4) mask &= ~((0xFu << (left > 0 ? static_cast<int>(left) : 0) & 0xFu) << (4 * u));
                }
            }
            if (__any_sync(0xFFFFFFFFu, mask != 0)) {
                int m = 1;
#pragma unroll 1
                for (; m < n_max; ++m) {                                      // mask: matches of m tokens
                    const int32_t sk = suf[m];
                    const int4 before[1] = {vp};
                    uint32_t f = scan_move(scan_equal<U>(v, sk), scan_equal<1>(before, sk), m, lane);
                    if (p < m) f &= ~0u << (m - p < 4 ? static_cast<int>(m - p) : 4);   // no token there
                    f &= mask;
                    if (!__any_sync(0xFFFFFFFFu, f != 0)) break;
                    mask = f;
                }
                each(m, mask, p);
            }
            vp = v[U - 1];
            if constexpr (AHEAD) {
#pragma unroll
                for (int u = 0; u < U; ++u) v[u] = nx[u];
            }
        }
    }
};

// put(i, j) for the i-th of the warp's positions in a round's mask (see WarpScan::run),
// counting from `base` in ascending order; returns how many there are.
template <typename Put>
__device__ __forceinline__ int scan_put(uint32_t mask, int64_t p, int base, int lane, Put put) {
    const unsigned lt = (1u << lane) - 1u;
    uint32_t tiles = (mask | mask >> 1 | mask >> 2 | mask >> 3) & 0x11111111u;
    tiles = __reduce_or_sync(0xFFFFFFFFu, tiles);
    int n = 0;
#pragma unroll 1
    for (; tiles != 0; tiles &= tiles - 1u) {
        const int at = __ffs(tiles) - 1;                          // 4 u
        const uint32_t nib = mask >> at;
        int off = base + n;
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const unsigned bal = __ballot_sync(0xFFFFFFFFu, (nib >> c) & 1u);
            off += __popc(bal & lt);
            n += __popc(bal);
        }
#pragma unroll
        for (int c = 0; c < 4; ++c)
            if ((nib >> c) & 1u) put(off++, p + (at >> 2) * kScanTile + c);
    }
    return n;
}

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
    sc.run(lim, sl.suf, n_max, [&](int m, uint32_t mask, int64_t p) {
        if (m < wm) return;                                       // warp-uniform
        if (m > wm) {
            wm = m;
            wc = 0;
        }
        wc += scan_put(mask, p, wc, sc.lane, [&](int i, int64_t j) {
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
    sc.run(lim, suf, n_max, [&](int m, uint32_t mask, int64_t p) {
        if (m != level) return;
        const int64_t base = at;
        at += scan_put(mask, p, 0, lane, [&](int i, int64_t j) {
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
