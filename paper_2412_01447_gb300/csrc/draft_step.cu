// pldp_draft_step: the drafting half of a PLD+ step -- candidate search (Eq. 1
// with the longest-suffix n-gram rule), ranking by hidden states (Eq. 3) and/or
// by attentions (Eq. 2), and draft extraction (Sec. 4.3) -- in one call; and
// pldp_verify_greedy_draft / pldp_verify_sample_draft: greedy or sampling
// verification (Sec. 4.4) followed by the next step's drafting.  The kernels:
//  * draft_step_kernel scans the contexts (below);
//  * draft_index_kernel looks the occurrences up in the incremental token index
//    (further down), one CTA per sequence;
//  * verify_draft_kernel runs the finish of verification (on the greedy pass's
//    row keys, or on the draws of sampling) and then the indexed drafting in the
//    same CTA;
//  * score_deferred_kernel, behind each of these, scores the sequences with many
//    candidates;
//  * index_build_kernel, with index_clear_kernel before it for large batches, builds
//    the index.
//
// The scanning kernel: one thread-block cluster per sequence, a chunk of the context
// per CTA.  Each CTA
//  1. scans its chunk once and keeps the positions with the longest suffix match it
//     met (pldp_scan.cuh), starts their hidden rows towards L2, and tells the
//     cluster's other CTAs its longest match and how many positions have it;
//  2. after the cluster barrier knows n*, the candidate list and its order; the
//     candidates are dealt out evenly to the cluster's CTAs, which read each other's
//     lists over distributed shared memory and score them -- cos(H_{j-1}, H_{t-1})
//     and the max (or sum) of the selected attention rows at key j, both in one round
//     trip to memory;
//  3. sends its best keys to CTA 0, which writes the choices and the draft.
// Only candidates are scored, whatever the number of occurrences of x_t.  A sequence
// with many of them (a frequent x_t in new text, Eq. 1's unigram match) is left to a
// second launch behind it, score_deferred_kernel, which deals all such candidates of
// the batch out to the whole GPU; so do the indexed kernels.
//
// Every score is the sum of the same partial sums in the same order (a fixed share per
// thread of a CTA, combined in warp order), whether a CTA scores one candidate with
// all its warps (cta_score) or each warp takes its own (warp_score), so results are
// deterministic and do not depend on the path.  Results are those of
// pldp_find_candidates, pldp_rank_hidden, pldp_rank_attention and pldp_extract_draft
// called in turn (fp32 score sums are split differently, so scores can differ in
// their last bits).
#include <climits>
#include <type_traits>

#include "pldp_rank.cuh"
#include "pldp_scan.cuh"
#include "pldp_verify.cuh"

namespace pldp {
namespace {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
// Workspace per sequence.  The scanning call needs a DeferSlot each and one more; the size
// stays what callers know it to be.
constexpr size_t kSeqWs = 16 + 256 * 16;
constexpr int64_t kPositionsPerCta = 1024;                     // scanned by a CTA at least; the batch sets the rest
constexpr int kScanLoads = 8;                                  // vectors of ids in flight per lane (scan kernel)
constexpr int kListPerWarp = 128;                              // positions listed per warp (scan kernel)
constexpr int kList = kListPerWarp * kWarps;                   // ... and per CTA
constexpr int kRescanPerWarp = 128;                            // the same for the rescan of the indexed kernels
constexpr int kRescanRounds = 5;                               // rounds of 1024 positions a warp keeps masks of there
constexpr int kScoreUnroll = 2;                                // 16-byte row loads in flight
constexpr int kScoreBatch = 2;                                 // candidates scored by the whole CTA at once (scan kernel)
constexpr int kMaxScoreBatch = 4;                              // ... and at most (the indexed kernel)
// Scoring passes of a CTA; a sequence with more candidates is deferred.  Two passes cost
// what the deferred launch does, which runs either way: on Zipf contexts 2 against 4
// measured 31.2 / 32.0 us (drafting, batch 128 x 32k) and 1385 / 1400 us (index build and
// 8 fused steps); one pass defers what uniform text often has (5-8 occurrences).
constexpr int kCtaPasses = 2;
constexpr int kMaxUnit = 64;                                   // candidates per unit of the deferred scoring, at most
constexpr int kSpeculate = kMaxScoreBatch;                     // occurrences scored before their suffix match
constexpr int kPrefetchOcc = 32;                                // occurrences whose rows are prefetched otherwise
constexpr size_t kMaxQueryBytes = 196608;
constexpr int kMaxSelRows = 8192;
constexpr int64_t kMaxPositions = int64_t(1) << 27;            // (j << 4) | m fits 31 bits

struct NoHidden {};

struct DraftParams {
    const int32_t* ids;
    int64_t ids_stride;
    const int32_t* seq_len;
    int64_t T_cap;
    int ngram_min, ngram_max;
    int32_t* cand_pos;
    int C_cap;
    int32_t* cand_count;
    int32_t* match_len;
    const void* H;
    bool h_bf16;
    int64_t d;
    int64_t h_seq_stride;
    float threshold;
    float* h_scores;
    int32_t* best_h;
    float* best_h_score;
    const void* A;
    bool a_bf16;
    int R;
    int64_t a_row_stride;
    int64_t a_key_stride;
    int64_t a_seq_stride;
    const int32_t* row_idx;
    int n_sel;
    int agg;
    float* a_scores;
    int32_t* best_a;
    float* best_a_score;
    int draft_from;       // 0: hidden choice, 1: attention choice
    int K;
    int32_t* draft;
    int32_t* draft_len;
    uint32_t* status;
    int B;
    struct DeferSlot* defer;   // [B + 1], all zero between calls; null: nothing is deferred
    bool count;                // the sequences decided on are counted (see score_deferred_kernel)
};

// What the drafting kernels leave to score_deferred_kernel: `pending` candidates of a
// sequence (its list is written); the best keys and the units done, while it runs.
// Slot B counts its CTAs out.
struct alignas(16) DeferSlot {
    unsigned long long h, a;
    unsigned pending, done;
    unsigned decided;          // slot B, indexed drafting: sequences decided on, and kDeferred times those left
    unsigned pad;
};
constexpr unsigned kDeferred = 1u << 16;                       // (at most 65535 sequences)
static_assert(sizeof(DeferSlot) == 32 && 2 * sizeof(DeferSlot) <= kSeqWs, "B + 1 slots fit the workspace");

// One thread, once per sequence and launch of an indexed drafting kernel: whether the
// sequence's `pending` candidates (0: none) are left to score_deferred_kernel.
__device__ __forceinline__ void decide(const DraftParams& p, int b, unsigned pending) {
    if (p.defer == nullptr) return;
    if (pending != 0) p.defer[b].pending = pending;
    if (p.count) atomicAdd(&p.defer[p.B].decided, pending != 0 ? 1u + kDeferred : 1u);
}

template <int NB>
__device__ __forceinline__ float (&part_buf(float (&part)[kMaxScoreBatch][kWarps][4]))[NB][kWarps][4] {
    return *reinterpret_cast<float(*)[NB][kWarps][4]>(&part[0]);
}

struct StepShared {
    alignas(16) float part[2][kMaxScoreBatch][kWarps][4];   // per-warp partials: dot, |a|^2, |q|^2, attention
    unsigned long long wkey[2][kWarps];      // per-warp best keys (hidden, attention)
};

// Eq. 3 and Eq. 2 for candidates j[0 .. nb) of sequence b (nb <= NB), by all
// threads of the CTA: thread i takes 16-byte chunks i, i + 256, ... of H_{j-1}
// and H_{t-1} and selected rows i, i + 256, ...; partial sums meet in `part`
// and are combined in warp order.  The candidates of one pass share the loads of
// H_{t-1} and are otherwise independent: a score does not depend on which pass
// or slot computes it.  The attention values of each thread's first selected row
// are loaded before the hidden rows are used, so both arrive in one round trip.
// Scores are returned in thread 0: the cosine (-inf when j = 0 has no H_{j-1})
// and the attention max / sum.  CTA-uniform call with one barrier; callers
// alternate `part` buffers.
template <typename TH, int NB>
__device__ __forceinline__ void cta_score(const DraftParams& p, int b, const int64_t (&j)[NB], int nb, int64_t t,
                                          float (&part)[NB][kWarps][4], float (&s_h)[NB], float (&s_a)[NB]) {
    constexpr bool HAS_H = !std::is_same<TH, NoHidden>::value;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const bool is_max = p.agg == PLDP_AGG_MAX;
    bool h_ok[NB], a_ok[NB];
    bool any_h = false;
#pragma unroll
    for (int h = 0; h < NB; ++h) {
        h_ok[h] = HAS_H && h < nb && j[h] >= 1 && j[h] < t;
        a_ok[h] = p.A != nullptr && h < nb && j[h] >= 0 && j[h] < t;
        any_h |= h_ok[h];
    }
    float dot[NB], na[NB], nq = 0.f, acc[NB];
#pragma unroll
    for (int h = 0; h < NB; ++h) {
        dot[h] = 0.f;
        na[h] = 0.f;
        acc[h] = is_max ? -INFINITY : 0.0f;
    }
    const size_t a_es = p.a_bf16 ? 2 : 4;
    const void* ab = p.A ? static_cast<const char*>(p.A) + static_cast<int64_t>(b) * p.a_seq_stride * a_es : nullptr;
    float av[NB];                                                 // selected row `tid`, in flight with H
    {
        const int r = (p.A != nullptr && tid < p.n_sel) ? (p.row_idx ? __ldg(p.row_idx + tid) : tid) : -1;
        const bool rv = r >= 0 && r < p.R;
#pragma unroll
        for (int h = 0; h < NB; ++h)
            av[h] = (rv && a_ok[h]) ? load_attn(ab, static_cast<int64_t>(r) * p.a_row_stride + j[h] * p.a_key_stride, p.a_bf16) : NAN;
    }
    if constexpr (HAS_H) {
        if (any_h) {
            constexpr int E = 16 / sizeof(TH);
            const TH* hb = static_cast<const TH*>(p.H) + static_cast<int64_t>(b) * p.h_seq_stride;
            const TH* qrow = hb + (t - 1) * p.d;                  // H_{t-1}
            const TH* arow[NB];
#pragma unroll
            for (int h = 0; h < NB; ++h) arow[h] = h_ok[h] ? hb + (j[h] - 1) * p.d : qrow;   // H_{j-1}
            const int64_t nch = p.d / E;
            for (int64_t c0 = tid; c0 < nch; c0 += static_cast<int64_t>(kThreads) * kScoreUnroll) {
                uint4 q[kScoreUnroll], a[NB][kScoreUnroll];
#pragma unroll
                for (int u = 0; u < kScoreUnroll; ++u) {
                    const int64_t c = c0 + static_cast<int64_t>(kThreads) * u;
                    if (c < nch) {
                        q[u] = ld_stream16(qrow + c * E);
#pragma unroll
                        for (int h = 0; h < NB; ++h)
                            if (h_ok[h]) a[h][u] = ld_stream16(arow[h] + c * E);
                    }
                }
#pragma unroll
                for (int u = 0; u < kScoreUnroll; ++u) {
                    if (c0 + static_cast<int64_t>(kThreads) * u >= nch) continue;
                    float dead0 = 0.f, dead1 = 0.f;                 // |H_{t-1}|^2 once for the pass
                    accum16<TH>(q[u], q[u], dead0, dead1, nq);
#pragma unroll
                    for (int h = 0; h < NB; ++h) {
                        float dead2 = 0.f;
                        if (h_ok[h]) accum16<TH>(a[h][u], q[u], dot[h], na[h], dead2);
                    }
                }
            }
        }
    }
    if (p.A != nullptr) {
#pragma unroll
        for (int h = 0; h < NB; ++h)
            if (av[h] == av[h]) acc[h] = is_max ? fmaxf(acc[h], av[h]) : acc[h] + av[h];
        for (int k = tid + kThreads; k < p.n_sel; k += kThreads) {
            const int r = p.row_idx ? __ldg(p.row_idx + k) : k;
            const bool rv = r >= 0 && r < p.R;
            float v[NB];
#pragma unroll
            for (int h = 0; h < NB; ++h)
                v[h] = (rv && a_ok[h]) ? load_attn(ab, static_cast<int64_t>(r) * p.a_row_stride + j[h] * p.a_key_stride, p.a_bf16) : NAN;
#pragma unroll
            for (int h = 0; h < NB; ++h)
                if (v[h] == v[h]) acc[h] = is_max ? fmaxf(acc[h], v[h]) : acc[h] + v[h];
        }
    }
    // warp totals by reduce-scatter: lane l ends with one of them
    if constexpr (HAS_H) {
        float w[2 * NB];                                          // dot products, then |H_{j-1}|^2
#pragma unroll
        for (int h = 0; h < NB; ++h) {
            w[h] = dot[h];
            w[NB + h] = na[h];
        }
        const float tw = warp_reduce_scatter<2 * NB>(w, false);
        constexpr int SW = 32 / (2 * NB);                         // lanes holding each total
        const int iw = lane / SW;
        if (lane % SW == 0) part[iw % NB][warp][iw < NB ? 0 : 1] = tw;
        nq = warp_sum(nq);
        if (lane < NB) part[lane][warp][2] = nq;
    } else {
        if (lane < NB) part[lane][warp][0] = part[lane][warp][1] = part[lane][warp][2] = 0.f;
    }
    {
        const float ta = warp_reduce_scatter<NB>(acc, is_max);
        constexpr int SA = 32 / NB;
        if (lane % SA == 0) part[lane / SA][warp][3] = ta;
    }
    __syncthreads();
    if (warp == 0) {
        // lane (h, w) = (lane / kWarps, lane % kWarps) takes warp w's partials of
        // candidate h; the kWarps lanes of a candidate combine them in a fixed tree
        static_assert(NB * kWarps <= 32, "a lane per (candidate, warp)");
        const int h = lane / kWarps, w = lane % kWarps;
        float4 v = make_float4(0.f, 0.f, 0.f, is_max ? -INFINITY : 0.f);
        if (h < NB) v = *reinterpret_cast<const float4*>(&part[h][w][0]);
#pragma unroll
        for (int o = kWarps / 2; o > 0; o >>= 1) {
            v.x += __shfl_xor_sync(0xFFFFFFFFu, v.x, o);
            v.y += __shfl_xor_sync(0xFFFFFFFFu, v.y, o);
            v.z += __shfl_xor_sync(0xFFFFFFFFu, v.z, o);
            const float x = __shfl_xor_sync(0xFFFFFFFFu, v.w, o);
            v.w = is_max ? fmaxf(v.w, x) : v.w + x;
        }
        bool hv = false, avl = false;
#pragma unroll
        for (int k = 0; k < NB; ++k)
            if (k == h) {
                hv = h_ok[k];
                avl = a_ok[k];
            }
        const float sh_ = hv ? finish_cosine(v.x, v.y, v.z) : -INFINITY;
        const float sa_ = avl ? v.w : -INFINITY;
#pragma unroll
        for (int k = 0; k < NB; ++k) {
            s_h[k] = __shfl_sync(0xFFFFFFFFu, sh_, k * kWarps);
            s_a[k] = __shfl_sync(0xFFFFFFFFu, sa_, k * kWarps);
        }
    }
}

// This warp's share of |H_{t-1}|^2, in cta_score's order; sum_shares combines the eight.
template <typename TH>
__device__ __forceinline__ float query_norm_share(const DraftParams& p, int b, int64_t t) {
    if constexpr (std::is_same<TH, NoHidden>::value) {
        return 0.f;
    } else {
        constexpr int E = 16 / sizeof(TH);
        const TH* qrow = static_cast<const TH*>(p.H) + static_cast<int64_t>(b) * p.h_seq_stride + (t - 1) * p.d;
        const int64_t nch = p.d / E;
        float nq = 0.f;
        if (t >= 2)
            for (int64_t c = threadIdx.x; c < nch; c += kThreads) {
                const uint4 q = __ldg(reinterpret_cast<const uint4*>(qrow) + c);
                float dead0 = 0.f, dead1 = 0.f;
                accum16<TH>(q, q, dead0, dead1, nq);
            }
        return warp_sum(nq);
    }
}
__device__ __forceinline__ float sum_shares(const float (&x)[kWarps]) {
    static_assert(kWarps == 8, "cta_score's tree over eight warps");
    return ((x[0] + x[4]) + (x[2] + x[6])) + ((x[1] + x[5]) + (x[3] + x[7]));
}

// Eq. 3 (dot product and |H_{j-1}|^2) and Eq. 2 for one candidate j by one warp, the
// results (in every lane) those of cta_score bit for bit: lane l forms the partial sums
// of the CTA's threads l, 32 + l, ..., 224 + l in eight accumulators, each in that
// thread's order, and they are reduced over the lanes and then over the eight in the
// CTA's order.  Eight 16-byte loads of the row are in flight per lane (sixteen measured
// 0.5-1.5 us more per launch); the query row is read through L1, which the CTA's warps
// share.
template <typename TH>
__device__ __forceinline__ void warp_score(const DraftParams& p, int b, int64_t j, int64_t t, float& dot, float& na,
                                           float& s_a) {
    constexpr bool HAS_H = !std::is_same<TH, NoHidden>::value;
    const int lane = threadIdx.x & 31;
    const bool is_max = p.agg == PLDP_AGG_MAX;
    const bool h_ok = HAS_H && j >= 1 && j < t, a_ok = p.A != nullptr && j >= 0 && j < t;
    dot = 0.f;
    na = 0.f;
    s_a = -INFINITY;
    // the attention values of the first 128 selected rows are requested before the
    // hidden row is used, so both arrive in one round trip
    const int64_t a_es = p.a_bf16 ? 2 : 4;
    const char* ab =
        p.A ? static_cast<const char*>(p.A) + (static_cast<int64_t>(b) * p.a_seq_stride + j * p.a_key_stride) * a_es : nullptr;
    auto attn = [&](int k) -> float {                             // NaN: no such row
        if (!a_ok || k >= p.n_sel) return NAN;
        const int r = p.row_idx ? __ldg(p.row_idx + k) : k;
        return (r >= 0 && r < p.R) ? load_attn(ab, static_cast<int64_t>(r) * p.a_row_stride, p.a_bf16) : NAN;
    };
    constexpr int kEarly = 4;
    float av[kEarly];
#pragma unroll
    for (int w = 0; w < kEarly; ++w) av[w] = attn(32 * w + lane);
    if constexpr (HAS_H) {
        if (h_ok) {                                               // warp-uniform
            constexpr int E = 16 / sizeof(TH), U = kWarps;
            const TH* hb = static_cast<const TH*>(p.H) + static_cast<int64_t>(b) * p.h_seq_stride;
            const uint4* qrow = reinterpret_cast<const uint4*>(hb + (t - 1) * p.d);
            const TH* arow = hb + (j - 1) * p.d;
            const int nch = static_cast<int>(p.d / E);
            float v[2 * kWarps];                                  // dot of share w, then |H_{j-1}|^2 of share w
#pragma unroll
            for (int i = 0; i < 2 * kWarps; ++i) v[i] = 0.f;
#pragma unroll 1
            for (int c0 = lane; c0 < nch; c0 += 32 * U) {
                uint4 a[U];
#pragma unroll
                for (int u = 0; u < U; ++u)
                    if (c0 + 32 * u < nch) a[u] = ld_stream16(arow + static_cast<int64_t>(c0 + 32 * u) * E);
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    if (c0 + 32 * u >= nch) continue;
                    const uint4 q = __ldg(qrow + c0 + 32 * u);
                    float dead = 0.f;
                    accum16<TH>(a[u], q, v[u % kWarps], v[kWarps + u % kWarps], dead);
                }
            }
            float r = warp_reduce_scatter<2 * kWarps>(v, false);  // lane l: value l / 2
            r += __shfl_xor_sync(0xFFFFFFFFu, r, 8);
            r += __shfl_xor_sync(0xFFFFFFFFu, r, 4);
            r += __shfl_xor_sync(0xFFFFFFFFu, r, 2);
            dot = __shfl_sync(0xFFFFFFFFu, r, 0);
            na = __shfl_sync(0xFFFFFFFFu, r, 16);
        }
    }
    if (a_ok) {                                                   // warp-uniform
        float acc[kWarps];
#pragma unroll
        for (int w = 0; w < kWarps; ++w) {
            acc[w] = is_max ? -INFINITY : 0.0f;
            const float x = w < kEarly ? av[w] : attn(32 * w + lane);
            if (x == x) acc[w] = is_max ? fmaxf(acc[w], x) : acc[w] + x;
        }
#pragma unroll 1
        for (int k0 = kThreads; k0 < p.n_sel; k0 += kThreads) {
            float x[kWarps];
#pragma unroll
            for (int w = 0; w < kWarps; ++w) x[w] = attn(k0 + 32 * w + lane);
#pragma unroll
            for (int w = 0; w < kWarps; ++w)
                if (x[w] == x[w]) acc[w] = is_max ? fmaxf(acc[w], x[w]) : acc[w] + x[w];
        }
        float r = warp_reduce_scatter<kWarps>(acc, is_max);       // lane l: value l / 4
#pragma unroll
        for (int o = 16; o >= 4; o >>= 1) {
            const float x = __shfl_xor_sync(0xFFFFFFFFu, r, o);
            r = is_max ? fmaxf(r, x) : r + x;
        }
        s_a = r;
    }
}

// The best keys a thread has scored.
struct BestKeys {
    unsigned long long h, a;
};

// Takes in the scores of the candidate with list index i at position j.
template <typename TH>
__device__ __forceinline__ void take_score(const DraftParams& p, int i, int64_t j, float s_h, float s_a, float* hsc,
                                           float* asc, BestKeys& best) {
    if (!std::is_same<TH, NoHidden>::value) {
        if (hsc) hsc[i] = s_h;
        if (j >= 1 && s_h > p.threshold) {
            const unsigned long long key = pack_key(s_h, static_cast<uint32_t>(j));
            best.h = key > best.h ? key : best.h;
        }
    }
    if (p.A != nullptr) {
        if (asc) asc[i] = s_a;
        const unsigned long long key = pack_key(s_a, static_cast<uint32_t>(j));
        best.a = key > best.a ? key : best.a;
    }
}

// One warp: the choices of both rankings (best keys hk, ak) and the draft (Sec. 4.3),
// with draft_tok(i, j*) giving token j* + 1 + i.
template <bool HAS_H, typename Tok>
__device__ __forceinline__ void write_choice(const DraftParams& p, int b, int64_t t, unsigned long long hk,
                                             unsigned long long ak, int lane, Tok draft_tok) {
    const int32_t bh = hk == 0 ? -1 : static_cast<int32_t>(key_index(hk));
    const int32_t ba = ak == 0 ? -1 : static_cast<int32_t>(key_index(ak));
    const int64_t js = p.draft_from == 0 ? bh : ba;
    int64_t dl = 0;
    if (js >= 0 && js < t) dl = (t - js < p.K) ? (t - js) : p.K;
    for (int i = lane; i < p.K; i += 32)
        p.draft[static_cast<int64_t>(b) * p.K + i] = (i < dl) ? draft_tok(i, js) : -1;
    if (lane != 0) return;
    if (HAS_H) {
        p.best_h[b] = bh;
        if (p.best_h_score) p.best_h_score[b] = bh >= 0 ? key_value(hk) : -INFINITY;
    }
    if (p.A != nullptr) {
        p.best_a[b] = ba;
        if (p.best_a_score) p.best_a_score[b] = ba >= 0 ? key_value(ak) : -INFINITY;
    }
    p.draft_len[b] = static_cast<int32_t>(dl);
}

// One thread: the candidate list's size and length, and the status bits of drafting.
__device__ __forceinline__ void write_counts(const DraftParams& p, int b, int nstar, int total, bool bad_rows) {
    p.cand_count[b] = total;
    p.match_len[b] = nstar;
    if (p.status && total > p.C_cap) atomicOr(p.status + b, PLDP_ST_CAND_OVERFLOW);
    if (p.status && bad_rows) atomicOr(p.status + b, PLDP_ST_ROW_INDEX);
}

// The scores of the sequences that the drafting kernel before it left (`defer`), spread
// over the whole GPU: the deferred candidates of the batch are cut into units of a few
// per warp, about one unit per CTA, whatever sequences they belong to.  A unit's CTA
// scores a candidate per warp at a time and adds its best keys to the sequence's slot;
// the CTA that completes a sequence writes its choices and draft.  Nothing waits.
//
// What bounds it: latency, about 9 us from the drafting kernel's end to its own with one
// candidate per warp (the slots, the candidates, their rows, the keys and the count, the
// draft: a round trip to memory each), then the translation of the rows' addresses: they
// are random 8 KB rows of a tensor of tens of GB, and the first half of one arrives 4-8 us
// after its load, about 500 rows/us in all (23 us for the 7154 candidates of a fused step
// of batch 128 x 32k).  Sending the rows to L2 while the drafting kernel ends, loading the
// next candidate's row while one is summed, and scoring with whole CTAs gave nothing.
//
// The same work by the sequences' own CTAs (up to 8, one in the indexed kernels) took
// 100-400 us of a drafting launch on Zipf contexts while the other SMs were idle: drafting
// batch 128 x 32k 125-190 -> 30 us (28 now); index build + 8 fused steps of it 6083 -> 1400
// us (1100 now).
//
// A batch without deferred sequences (uniform contexts, where x_t occurs a few times) pays
// for the launch all the same, most of it the boundary between two kernels: fused step of
// batch 128 x 32k uniform tokens 74.7 us without it, 76.5 with a grid of one CTA, 76.8 with
// every CTA waiting for the drafting kernel and then finding nothing.  COUNTED (behind
// indexed drafting of more sequences than half the SMs, which counts those it has decided
// on): when all are and none is left, every CTA but the first leaves before the wait, 76.4;
// the first stays until the drafting kernel is complete, since the stream's next work relies
// on this launch for that.  Where the drafting CTAs leave room for these, they are all there
// by then, and the counts cost 0.15 us a call and give nothing; behind the scanning kernel
// they cost as much as they gave (draft_step, 2 x 128k Zipf tokens, 12.2 -> 12.4 us).
template <typename TH, bool COUNTED>
__global__ void __launch_bounds__(kThreads, 2) score_deferred_kernel(const DraftParams p, int B) {
    constexpr bool HAS_H = !std::is_same<TH, NoHidden>::value;
    __shared__ int n_of[kThreads];                                // deferred candidates of this tile's sequences
    __shared__ int start[kThreads];                               // their first units, counted from the tile's
    __shared__ int wsum[kWarps];
    __shared__ unsigned long long wkey[2][kWarps];
    __shared__ float wnq[kWarps];
    __shared__ int last;
    if constexpr (COUNTED) {
        const bool none = threadIdx.x == 0 && ld_relaxed(&p.defer[B].decided) == static_cast<unsigned>(B);
        if (__syncthreads_or(none) && blockIdx.x != 0) return;
    }
    pdl_enter();
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    DeferSlot* slots = p.defer;
    const int G = static_cast<int>(gridDim.x);
    // (no more than a list holds, whatever was in scratch that was not cleared)
    auto pending = [&](int b) -> unsigned {
        const unsigned n = __ldcg(&slots[b].pending), cap = static_cast<unsigned>(p.C_cap);
        return n < cap ? n : cap;
    };
    const int n0 = tid < B ? static_cast<int>(pending(tid)) : 0;   // the first tile's
    unsigned sum = n0, seqs = n0 > 0;
    for (int b = tid + kThreads; b < B; b += kThreads) {
        const unsigned n = pending(b);
        sum += n;
        seqs += n > 0;
    }
    sum = __reduce_add_sync(0xFFFFFFFFu, sum);
    seqs = __reduce_add_sync(0xFFFFFFFFu, seqs);
    if (lane == 0) {
        wsum[warp] = static_cast<int>(sum);
        n_of[warp] = static_cast<int>(seqs);
    }
    __syncthreads();
    int64_t all = 0, heavy = 0;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) {
        all += wsum[w];
        heavy += n_of[w];
    }
    if (all == 0) {
        if (COUNTED && blockIdx.x == 0 && tid == 0) slots[B].decided = 0;
        return;
    }
    // The last CTA to have read every `pending` clears them on its way out: known at once
    // when they are one tile, else after the last tile.
    bool clears = false;
    auto count_in = [&]() { clears = tid == 0 && atomicAdd(&slots[B].done, 1u) == static_cast<unsigned>(G - 1); };
    if (B <= kThreads) count_in();
    // units of U candidates, a multiple of one per warp, at most one unit per CTA where
    // that fits (the last unit of every sequence may be short)
    const int64_t ctas = (2 * heavy < G ? G - heavy : (G + 1) / 2) * kWarps;
    const int64_t per = (all + ctas - 1) / ctas * kWarps;
    const int U = per < kMaxUnit ? static_cast<int>(per) : kMaxUnit;
    int64_t unit0 = 0;                                            // units of the tiles before
    for (int b0 = 0; b0 < B; b0 += kThreads) {
        // the tile's units: an exclusive scan over its sequences
        const int n = b0 == 0 ? n0 : b0 + tid < B ? static_cast<int>(pending(b0 + tid)) : 0;
        const int units = (n + U - 1) / U;
        int incl = units;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xFFFFFFFFu, incl, o);
            if (lane >= o) incl += v;
        }
        __syncthreads();                                          // wsum, n_of and start have been read
        if (lane == 31) wsum[warp] = incl;
        __syncthreads();
        int before = 0, total = 0;
#pragma unroll
        for (int w = 0; w < kWarps; ++w) {
            before += w < warp ? wsum[w] : 0;
            total += wsum[w];
        }
        n_of[tid] = n;
        start[tid] = before + incl - units;
        __syncthreads();
        const int64_t skip = (unit0 + G - 1 - blockIdx.x) / G;    // this CTA's units below unit0
        for (int64_t u = skip * G + blockIdx.x - unit0; u < total; u += G) {
            int lo = 0, hi = kThreads - 1;                        // the last sequence that starts at or below u
            while (lo < hi) {
                const int mid = (lo + hi + 1) >> 1;
                if (start[mid] <= u) lo = mid;
                else hi = mid - 1;
            }
            const int b = b0 + lo, nb = n_of[lo];
            const int k0 = static_cast<int>(u - start[lo]) * U, k1 = k0 + U < nb ? k0 + U : nb;
            const int64_t t = static_cast<int64_t>(p.seq_len[b]) - 1;
            const int64_t row0 = static_cast<int64_t>(b) * p.C_cap;
            // this warp's candidates k0 + warp, k0 + warp + kWarps, ...: lane i the i-th
            const int kl = k0 + warp + lane * kWarps;
            const int32_t jl = kl < k1 ? p.cand_pos[row0 + kl] : -1;
            const int cnt = k1 > k0 + warp ? (k1 - k0 - warp + kWarps - 1) / kWarps : 0;
            const float nqs = query_norm_share<TH>(p, b, t);
            if (lane == 0) wnq[warp] = nqs;
            float dl = 0.f, nl = 0.f, al = 0.f;
            for (int i = 0; i < cnt; ++i) {
                const int64_t j = __shfl_sync(0xFFFFFFFFu, jl, i);
                if (HAS_H && i + 1 < cnt) {                       // the next row heads for L2
                    const int64_t jn = __shfl_sync(0xFFFFFFFFu, jl, i + 1);
                    const int64_t h_es = p.h_bf16 ? 2 : 4;
                    if (lane == 0 && jn >= 1 && jn < t)
                        prefetch_l2_bulk(static_cast<const char*>(p.H) +
                                             (static_cast<int64_t>(b) * p.h_seq_stride + (jn - 1) * p.d) * h_es,
                                         static_cast<uint32_t>(p.d * h_es));
                }
                float dot, na, s_a;
                warp_score<TH>(p, b, j, t, dot, na, s_a);
                if (lane == i) {
                    dl = dot;
                    nl = na;
                    al = s_a;
                }
            }
            __syncthreads();                                      // every share of the query norm is in
            BestKeys best = {0, 0};
            if (lane < cnt) {
                const float s_h = (HAS_H && jl >= 1 && jl < t) ? finish_cosine(dl, nl, sum_shares(wnq)) : -INFINITY;
                take_score<TH>(p, kl, jl, s_h, al, p.h_scores ? p.h_scores + row0 : nullptr,
                               p.a_scores ? p.a_scores + row0 : nullptr, best);
            }
            const unsigned long long hw = warp_max_u64(best.h), aw = warp_max_u64(best.a);
            if (lane == 0) {
                wkey[0][warp] = hw;
                wkey[1][warp] = aw;
            }
            __syncthreads();
            if (tid == 0) {
                unsigned long long hk = 0, ak = 0;
#pragma unroll
                for (int w = 0; w < kWarps; ++w) {
                    hk = wkey[0][w] > hk ? wkey[0][w] : hk;
                    ak = wkey[1][w] > ak ? wkey[1][w] : ak;
                }
                if (hk) atomicMax(&slots[b].h, hk);
                if (ak) atomicMax(&slots[b].a, ak);
                __threadfence();                                  // the keys before the count
                last = atomicAdd(&slots[b].done, 1u) == static_cast<unsigned>((nb + U - 1) / U - 1);
                __threadfence();
            }
            __syncthreads();
            if (last && warp == 0) {                              // the sequence is complete
                const unsigned long long hk = __ldcg(&slots[b].h), ak = __ldcg(&slots[b].a);
                const int32_t* row = p.ids + static_cast<int64_t>(b) * p.ids_stride;
                write_choice<HAS_H>(p, b, t, hk, ak, lane, [&](int i, int64_t js) -> int32_t { return row[js + 1 + i]; });
                __syncwarp();
                if (lane == 0) {
                    slots[b].h = 0;
                    slots[b].a = 0;
                    slots[b].done = 0;
                }
            }
            // (wkey and wnq are rewritten only after the next unit's first barrier or by
            // their own warps; `last` after its second)
        }
        unit0 += total;
    }
    if (B > kThreads) {
        __syncthreads();                                          // this CTA's reads are done
        count_in();
    }
    if (!__syncthreads_or(clears)) return;
    for (int b = tid; b < B; b += kThreads) slots[b].pending = 0;
    if (tid == 0) {
        slots[B].done = 0;
        if (COUNTED) slots[B].decided = 0;
    }
}

// What the rescan keeps per warp: every round's longest match and its mask (see
// WarpScan::run) for the first kRescanRounds rounds of 1024 positions, i.e. contexts of
// up to 40k tokens; of a longer context a list of positions.
union RescanShared {
    struct {
        uint32_t mask[kScanWarps][kRescanRounds][32];
        int32_t suf[PLDP_MAX_NGRAM];
        int wm[kScanWarps], wc[kScanWarps];
        uint8_t level[kScanWarps][kRescanRounds];
    };
    ScanLists<kRescanPerWarp> sl;
};

// The candidates of a sequence whose occurrences were not gathered (a token the index
// cannot answer for): one CTA scans the context and writes the candidate list, its first
// `keep` entries to `first` (shared) too.  With the rounds' masks kept, the list is
// written without reading the ids again, however long it is (a token that makes up 8 % of
// 32k tokens overflowed a warp's list of 128, and its second pass took 18 us: index build
// and 8 fused steps of batch 128 x 32k 1252 -> 1142 us).  Kept out of line: its registers
// do not weigh on the common path.  CTA-uniform call, a barrier at the end.
template <bool IVEC, typename RD>
__device__ __noinline__ void rescan(const DraftParams& p, int64_t t, const int32_t* row, int32_t* cand_row,
                                    RescanShared& rs, int32_t* first, int keep, int& nstar, int& total) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t seg = (t + kScanChunkUnit - 1) / kScanChunkUnit * kScanTile;      // positions per warp
    const int64_t s0 = warp * seg;
    const int nit = static_cast<int>(seg / kScanTile);
    if (IVEC && lane == 0 && s0 < t)                              // the warp's ids head for L2 all at once
        prefetch_l2_bulk(row + s0, static_cast<uint32_t>((s0 + seg < t ? seg : (t - s0 + 3) & ~int64_t(3)) * 4));
    WarpScan<IVEC, RD, kScanLoads, true> sc;
    sc.begin(row, s0, nit, p.T_cap, lane);
    auto put = [&](int64_t i, int32_t j) {
        cand_row[i] = j;
        if (i < keep) first[i] = j;
    };
    if (nit <= kRescanRounds * kScanLoads) {
        if (tid < PLDP_MAX_NGRAM) rs.suf[tid] = (tid < p.ngram_max && t - tid >= 0) ? RD::one(row + t - tid) : 0;
        if (lane < kRescanRounds) rs.level[warp][lane] = 0;
        __syncthreads();                                          // the suffix is in
        int wm = 0, wc = 0;                                       // wc: this lane's
        sc.run(t, rs.suf, p.ngram_max, [&](int m, uint32_t mask, int64_t q) {
            if (m < wm) return;                                   // warp-uniform
            if (m > wm) wc = 0;
            wm = m;
            wc += __popc(mask);
            const int r = static_cast<int>((q - 4 * lane - s0) / (kScanTile * kScanLoads));
            rs.mask[warp][r][lane] = mask;
            if (lane == 0) rs.level[warp][r] = static_cast<uint8_t>(m);
        });
        wc = static_cast<int>(__reduce_add_sync(0xFFFFFFFFu, static_cast<unsigned>(wc)));
        if (lane == 0) {
            rs.wm[warp] = wm;
            rs.wc[warp] = wc;
        }
        __syncthreads();
        int best = 0, cnt = 0, at = 0;
#pragma unroll
        for (int w = 0; w < kScanWarps; ++w) best = max(best, rs.wm[w]);
#pragma unroll
        for (int w = 0; w < kScanWarps; ++w) {
            const int c = rs.wm[w] == best ? rs.wc[w] : 0;
            at += w < warp ? c : 0;
            cnt += c;
        }
        nstar = best >= p.ngram_min ? best : 0;
        total = nstar > 0 ? cnt : 0;
        if (nstar > 0 && wm == nstar)
            for (int r = 0; r * kScanLoads < nit && at < p.C_cap; ++r) {
                if (rs.level[warp][r] != nstar) continue;
                const int base = at;
                at += scan_put(rs.mask[warp][r][lane], s0 + r * (kScanTile * kScanLoads) + 4 * lane, 0, lane,
                               [&](int i, int64_t j) {
                                   if (base + i < p.C_cap) put(base + i, static_cast<int32_t>(j));
                               });
            }
    } else {
        ScanLists<kRescanPerWarp>& sl = rs.sl;
        if (tid < PLDP_MAX_NGRAM) sl.suf[tid] = (tid < p.ngram_max && t - tid >= 0) ? RD::one(row + t - tid) : 0;
        __syncthreads();                                          // the suffix is in
        scan_lists(sc, t, p.ngram_max, warp, sl);
        __syncthreads();
        const CtaMatches cm = cta_matches(sl, warp);
        nstar = cm.m >= p.ngram_min ? cm.m : 0;
        total = nstar > 0 ? cm.cnt : 0;
        scan_emit<IVEC, RD>(row, s0, nit, t, p.T_cap, p.ngram_max, nstar, cm.base, p.C_cap, warp, lane, sl, put);
    }
    __syncthreads();
}

// Per-sequence outputs of a context length outside [0, T_cap].
template <bool HAS_H>
__device__ __forceinline__ void no_draft(const DraftParams& p, int b) {
    for (int i = threadIdx.x; i < p.K; i += kThreads) p.draft[static_cast<int64_t>(b) * p.K + i] = -1;
    if (threadIdx.x != 0) return;
    p.cand_count[b] = 0;
    p.match_len[b] = 0;
    if (HAS_H) {
        p.best_h[b] = -1;
        if (p.best_h_score) p.best_h_score[b] = -INFINITY;
    }
    if (p.A != nullptr) {
        p.best_a[b] = -1;
        if (p.best_a_score) p.best_a_score[b] = -INFINITY;
    }
    p.draft_len[b] = 0;
    if (p.status) atomicOr(p.status + b, PLDP_ST_SEQ_LEN);
}

// The scanning kernel's shared memory.
struct ScanStepShared {
    StepShared st;
    ScanLists<kListPerWarp> sl;
    int32_t list[kList];                                          // this CTA's longest matches, ascending
    int32_t mine[kList];                                          // the candidates this CTA scores
    ScanPeer tab[kScanMaxCluster];                                // every CTA's outcome
    unsigned long long key[kScanMaxCluster][2];                   // CTA 0: every CTA's best keys
};

template <typename TH, bool IVEC>
__global__ void __launch_bounds__(kThreads, 3) draft_step_kernel(const DraftParams p, int CL, int64_t chunk) {
    constexpr bool HAS_H = !std::is_same<TH, NoHidden>::value;
    __shared__ ScanStepShared sh;
    pdl_enter();
    const int b = blockIdx.x / CL;
    const int rank = blockIdx.x - b * CL;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int32_t* row = p.ids + static_cast<int64_t>(b) * p.ids_stride;
    const bool has_a = p.A != nullptr;
    const int64_t h_es = p.h_bf16 ? 2 : 4;
    // The chunk's first ids do not depend on seq_len: their loads go out first, bounded
    // by the row's capacity, and land while seq_len and the suffix arrive.
    const int64_t seg = chunk / kScanWarps;
    const int64_t s0 = static_cast<int64_t>(rank) * chunk + warp * seg;
    const int nit = static_cast<int>(seg / kScanTile);
    WarpScan<IVEC, ReadOnlyIds, kScanLoads> sc;
    sc.begin(row, s0, nit, p.T_cap, lane);
    const int64_t L = p.seq_len[b];
    const int64_t t = L - 1;
    if (L < 0 || L > p.T_cap) {                                   // the same for every CTA of the cluster
        if (rank == 0) no_draft<HAS_H>(p, b);
        return;
    }
    cg::cluster_group cluster = cg::this_cluster();
    if (CL > 1) cluster_arrive_relaxed();                         // this CTA runs: its shared memory may be written
    if (tid < PLDP_MAX_NGRAM)                                     // x_t and the n_max - 1 tokens before it
        sh.sl.suf[tid] = (tid < p.ngram_max && t - tid >= 0) ? __ldg(row + t - tid) : 0;
    const char* hrows = static_cast<const char*>(p.H) + static_cast<int64_t>(b) * p.h_seq_stride * h_es;
    if (HAS_H && tid == 32 && rank == 0 && t >= 2)                // H_{t-1}: every score reads it
        prefetch_l2_bulk(hrows + (t - 1) * p.d * h_es, static_cast<uint32_t>(p.d * h_es));
    bool bad = false;                                             // a selected row outside [0, R)
    if (rank == 0 && has_a && p.row_idx)
        for (int k = tid; k < p.n_sel; k += kThreads) {
            const int r = __ldg(p.row_idx + k);
            bad |= r < 0 || r >= p.R;
        }
    bad = __syncthreads_or(bad) != 0;

    // ---- 1. this chunk's longest matches -----------------------------------------------------
    scan_lists(sc, t, p.ngram_max, warp, sh.sl);
    __syncthreads();
    const CtaMatches cm = cta_matches(sh.sl, warp);
    if (!cm.over && cm.m > 0 && sh.sl.wm[warp] == cm.m)           // their list, in order
        for (int i = lane; i < sh.sl.wc[warp]; i += 32) {
            const int32_t j = sh.sl.pos[warp][i];
            sh.list[cm.base + i] = j;
            if (HAS_H && j >= 1 && cm.m >= p.ngram_min && cm.base + i < kWarps)   // likely candidates
                prefetch_l2_bulk(hrows + (j - 1) * p.d * h_es, static_cast<uint32_t>(p.d * h_es));
        }
    if (CL > 1) {
        cluster_wait();
        if (tid < CL) *cluster.map_shared_rank(&sh.tab[rank], tid) = ScanPeer{cm.m, cm.cnt, cm.over ? 1 : 0};
        cluster_arrive();
        cluster_wait();                                           // every CTA's outcome and list are in
    } else {
        if (tid == 0) sh.tab[0] = ScanPeer{cm.m, cm.cnt, cm.over ? 1 : 0};
        __syncthreads();
    }

    // ---- 2. the candidate list; every CTA scores its share -----------------------------------
    const ScanTotal tt = scan_total(sh.tab, CL, rank, p.ngram_min);
    const int n = tt.total < p.C_cap ? tt.total : p.C_cap;
    const int n_local = n > rank ? (n - rank + CL - 1) / CL : 0;
    int32_t* cand_row = p.cand_pos + static_cast<int64_t>(b) * p.C_cap;
    float* hsc = (HAS_H && p.h_scores) ? p.h_scores + static_cast<int64_t>(b) * p.C_cap : nullptr;
    float* asc = (has_a && p.a_scores) ? p.a_scores + static_cast<int64_t>(b) * p.C_cap : nullptr;
    BestKeys best = {0, 0};
    if (!tt.over) {
        for (int k = tid; k < n_local; k += kThreads) {           // candidate rank + CL k: whose list, and where
            int i = rank + CL * k, r = 0;
            while (sh.tab[r].m != tt.nstar || i >= sh.tab[r].cnt) {
                if (sh.tab[r].m == tt.nstar) i -= sh.tab[r].cnt;
                ++r;
            }
            const int32_t j = CL > 1 ? *cluster.map_shared_rank(&sh.list[i], r) : sh.list[i];
            sh.mine[k] = j;
            cand_row[rank + CL * k] = j;
        }
        __syncthreads();
    } else {
        // more matches in a warp's segment than its list holds: the list goes through
        // the caller's candidate row
        scan_emit<IVEC, ReadOnlyIds>(row, s0, nit, t, p.T_cap, p.ngram_max, tt.nstar,
                                     static_cast<int64_t>(tt.before) + cm.base, p.C_cap, warp, lane, sh.sl,
                                     [&](int64_t i, int32_t j) { cand_row[i] = j; });
        if (CL > 1) {
            cluster_arrive();
            cluster_wait();
        } else {
            __syncthreads();
        }
    }
    const bool deferred = p.defer != nullptr && n > kCtaPasses * kScoreBatch * CL;
    if (!deferred) {
        for (int k0 = 0; k0 < n_local; k0 += kScoreBatch) {
            int64_t j[kScoreBatch];
#pragma unroll
            for (int h = 0; h < kScoreBatch; ++h)
                j[h] = k0 + h >= n_local ? -1 : tt.over ? __ldcg(cand_row + rank + CL * (k0 + h)) : sh.mine[k0 + h];
            const int nb = n_local - k0 < kScoreBatch ? n_local - k0 : kScoreBatch;
            float s_h[kScoreBatch], s_a[kScoreBatch];
            cta_score<TH, kScoreBatch>(p, b, j, nb, t, part_buf<kScoreBatch>(sh.st.part[(k0 / kScoreBatch) & 1]), s_h, s_a);
            if (tid == 0)
#pragma unroll
                for (int h = 0; h < kScoreBatch; ++h)
                    if (h < nb) take_score<TH>(p, rank + CL * (k0 + h), j[h], s_h[h], s_a[h], hsc, asc, best);
        }
    }

    // ---- 3. best of each ranking, then the draft (Sec. 4.3) ----------------------------------
    unsigned long long hk = warp_max_u64(best.h), ak = warp_max_u64(best.a);
    if (lane == 0) {
        sh.st.wkey[0][warp] = hk;
        sh.st.wkey[1][warp] = ak;
    }
    __syncthreads();
    if (tid < 2) {
        unsigned long long k = 0;
#pragma unroll
        for (int w = 0; w < kWarps; ++w) k = sh.st.wkey[tid][w] > k ? sh.st.wkey[tid][w] : k;
        *(CL > 1 ? cluster.map_shared_rank(&sh.key[rank][tid], 0) : &sh.key[0][tid]) = k;
    }
    if (CL > 1) {
        cluster_arrive();
        cluster_wait();                                           // no CTA leaves while its list may be read
    }
    if (rank != 0 || warp != 0) return;
    __syncwarp();
    hk = 0;
    ak = 0;
    for (int r = 0; r < CL; ++r) {
        hk = sh.key[r][0] > hk ? sh.key[r][0] : hk;
        ak = sh.key[r][1] > ak ? sh.key[r][1] : ak;
    }
    if (lane == 0) {
        write_counts(p, b, tt.nstar, tt.total, bad);
        if (deferred) p.defer[b].pending = static_cast<unsigned>(n);
    }
    if (!deferred)
        write_choice<HAS_H>(p, b, t, hk, ak, lane, [&](int i, int64_t js) -> int32_t { return __ldg(row + js + 1 + i); });
}

// ---------------------------------------------------------------------------
// The incremental token index: drafting without rescanning the context.
//
// Per sequence b and token v the index holds one 64-byte entry (half a line): how
// often v occurs among the indexed positions, then up to kIndexSlots of those
// positions (in no particular order); ilen[b] is the number of positions indexed
// (0 .. ilen-1), -1 when the index of b is unusable.  A step with t = seq_len - 1:
//  * reads x_t's entry in one request (a word per lane); when the count is at
//    most kIndexSlots the slots are every occurrence before ilen, and the
//    positions appended since (ilen .. t-1, read anyway) supply the rest;
//  * otherwise (a frequent token, a stale or unusable index) falls back to the
//    rescan of the context, so results are those of the scan either way;
//  * appends positions ilen .. t-1 to the index and sets ilen = t.  Each
//    appended position takes its slot with an atomic on its token's count; the
//    answer is used (the slot written) only at the end of the CTA, and tokens
//    equal to x_t take theirs only after x_t's entry has been read.
// With at most kSpeculate occurrences (most steps) every occurrence is scored
// while its suffix-match length is found, in one round trip to memory: its
// preceding tokens, the K tokens after it, H_{j-1} and the attention values at
// j are loaded together, and n* then picks the candidates among the scored
// occurrences.  With more, scoring all of them would cost more than it saves
// (each needs a d-element row and R scattered attention values): the suffix
// matches come first, then only the candidates are scored, with the tokens
// after them read in the same round trip.  One CTA per sequence.
// ---------------------------------------------------------------------------
constexpr int kIndexSlots = 15;
constexpr int kEntryWords = 1 + kIndexSlots;       // count, then the slots: 64 bytes, half a line
constexpr int kNewCap = kThreads;                  // appended positions taken in one step
constexpr int kOccCap = kIndexSlots + kNewCap;
constexpr int kDraftWin = 32;                      // draft tokens staged per occurrence (a lane each)

static_assert(kEntryWords * 4 == 64 && kEntryWords <= 32, "an entry is 64 bytes, a word per lane");

struct IndexView {
    DeferSlot* defer;   // [B + 1], after the entries; null where the memory ends with these
    int32_t* ilen;      // [B]
    int32_t* flags;     // [B], build scratch
    int32_t* entries;   // [B][V][kEntryWords]
    int V;
};

// Kept below 10 KB a CTA: the streaming pass that runs before the fused kernel leaves
// the SMs configured for little shared memory, and CTAs that need more wait for an SM
// to drain (16 KB measured 2.2 us more per step at the sustained-loop shape).
struct IndexShared {
    union {
        struct {
            int32_t occ[kOccCap];          // occurrences of x_t, ascending
            int32_t occ_m[kOccCap];        // their suffix-match lengths
            int32_t occ_new[kNewCap];      // the appended occurrences, ascending
        };
        RescanShared rs;                   // the rescan, which has no occurrences at hand
    };
    int32_t cand[kOccCap];             // the candidates (match length >= n*), ascending
    int32_t newtok[kNewCap];           // ids of positions il .. t-1
    int32_t suf[PLDP_MAX_NGRAM];       // x_t, x_{t-1}, ...
    int nocc, ncand, nstar, bad_token, indexed, wmax[kWarps];
};

__device__ __forceinline__ int32_t* index_entry(const IndexView& ix, int b, int32_t tok) {
    return ix.entries + (static_cast<int64_t>(b) * ix.V + tok) * kEntryWords;
}

// Counts one more occurrence of token tok in sequence b's index: returns the slot
// it takes (the old count; >= kIndexSlots: none), or -1 for a token outside [0, V).
__device__ __forceinline__ int index_take(const IndexView& ix, int b, int32_t tok) {
    if (tok < 0 || tok >= ix.V) return -1;
    return atomicAdd(index_entry(ix, b, tok), 1);
}

// Writes position q into the slot taken by index_take.
__device__ __forceinline__ void index_put(const IndexView& ix, int b, int32_t tok, int slot, int64_t q) {
    if (slot >= 0 && slot < kIndexSlots) index_entry(ix, b, tok)[1 + slot] = static_cast<int32_t>(q);
}

__device__ __forceinline__ bool index_insert(const IndexView& ix, int b, int64_t q, int32_t tok) {
    const int slot = index_take(ix, b, tok);
    index_put(ix, b, tok, slot, q);
    return slot >= 0;
}

// The indexed drafting of sequence b by the whole CTA, for context length L.
// RD: how ids are read -- CoherentIds when this kernel has just appended to the
// context (verification fused in front), else through the read-only cache.
// PRE: the indexed length is il_in and the ids it starts from -- is.newtok (the
// positions appended since, when they fit) and is.suf (x_t, x_{t-1}, ...) -- are
// already in shared memory, written before the CTA's last barrier.
template <typename TH, bool IVEC, typename RD, bool PRE = false>
__device__ __forceinline__ void index_draft(const DraftParams& p, const IndexView& ix, int b, int64_t L,
                                            StepShared& sh, IndexShared& is, int64_t il_in = 0) {
    constexpr bool HAS_H = !std::is_same<TH, NoHidden>::value;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t il = PRE ? il_in : static_cast<int64_t>(ix.ilen[b]);
    const bool valid = L >= 0 && L <= p.T_cap;
    const int64_t t = L - 1;
    const int32_t* row = p.ids + static_cast<int64_t>(b) * p.ids_stride;
    const bool has_a = p.A != nullptr;
    const size_t h_es = p.h_bf16 ? 2 : 4;
    bool bad = false;                                             // a selected row outside [0, R)
    if (has_a && valid && p.row_idx)
        for (int k = tid; k < p.n_sel; k += kThreads) {
            const int r = __ldg(p.row_idx + k);
            bad |= r < 0 || r >= p.R;
        }
    if (tid == 0) is.bad_token = 0;
    bad = __syncthreads_or(bad) != 0;
    if (!valid) {
        no_draft<HAS_H>(p, b);
        if (tid == 0) decide(p, b, 0);
        return;
    }
    // usable: the index covers a prefix of the context; small: what was appended fits the CTA
    const bool usable = il >= 0 && il <= t;
    const int64_t nnew = usable ? t - il : 0;
    const bool small = usable && nnew <= kNewCap;
    if (tid == 0 && HAS_H && t >= 2)                              // H_{t-1}: every candidate's score reads it
        prefetch_l2_bulk(static_cast<const char*>(p.H) + (static_cast<int64_t>(b) * p.h_seq_stride + (t - 1) * p.d) * h_es,
                         static_cast<uint32_t>(p.d * h_es));
    if (!PRE) {
        if (small && tid < nnew) is.newtok[tid] = RD::one(row + il + tid);
        if (tid < PLDP_MAX_NGRAM) is.suf[tid] = (tid < p.ngram_max && t - tid >= 0) ? RD::one(row + t - tid) : 0;
    }
    __syncthreads();
    const int32_t xt = is.suf[0];
    const bool lookup = small && t >= 1 && xt >= 0 && xt < ix.V;
    int32_t ev = 0;                                               // x_t's entry, word `lane` (warp 0)
    if (lookup && tid < kEntryWords) ev = __ldcg(index_entry(ix, b, xt) + tid);
    // this thread's appended position (small): its token and the slot it takes
    const bool mine = small && tid < nnew;
    const int32_t mytok = mine ? is.newtok[tid] : 0;
    int myslot = -1;
    if (mine && mytok != xt) myslot = index_take(ix, b, mytok);  // other entries: no wait for x_t's
    if (mine && (mytok < 0 || mytok >= ix.V)) atomicOr(&is.bad_token, 1);
    if (warp == 0 && lookup) {
        // the appended occurrences (ascending) while the entry is on its way
        int nn = 0;
        for (int c0 = 0; c0 < nnew; c0 += 32) {
            const bool hit = c0 + lane < nnew && is.newtok[c0 + lane] == xt;
            const unsigned bal = __ballot_sync(0xFFFFFFFFu, hit);
            if (hit) is.occ_new[nn + __popc(bal & ((1u << lane) - 1u))] = static_cast<int32_t>(il + c0 + lane);
            nn += __popc(bal);
        }
        const int nold = __shfl_sync(0xFFFFFFFFu, ev, 0);
        const bool ok = nold >= 0 && nold <= kIndexSlots;         // else the slots do not hold them all
        if (ok) {
            if (lane >= 1 && lane <= nold) {                      // the indexed ones (all before il), ranked
                int rank = 0;
                for (int k = 1; k <= nold; ++k) rank += __shfl_sync((1u << (nold + 1)) - 2u, ev, k) < ev ? 1 : 0;
                is.occ[rank] = ev;
            }
            __syncwarp();
            for (int k = lane; k < nn; k += 32) is.occ[nold + k] = is.occ_new[k];
        }
        if (lane == 0) {
            is.indexed = ok;
            is.nocc = ok ? nold + nn : 0;
        }
    }
    __syncthreads();                                              // x_t's entry has been read
    const bool indexed = lookup && is.indexed;
    if (mine && mytok == xt) myslot = index_take(ix, b, mytok);
    if (usable && !small) {                                       // a long append: inserted in turn
        bool badtok = false;
        for (int64_t q = il + tid; q < t; q += kThreads) badtok |= !index_insert(ix, b, q, RD::one(row + q));
        if (badtok) atomicOr(&is.bad_token, 1);
    }

    int32_t* cand_row = p.cand_pos + static_cast<int64_t>(b) * p.C_cap;
    float* hsc = (HAS_H && p.h_scores) ? p.h_scores + static_cast<int64_t>(b) * p.C_cap : nullptr;
    float* asc = (has_a && p.a_scores) ? p.a_scores + static_cast<int64_t>(b) * p.C_cap : nullptr;
    const int nocc = indexed ? is.nocc : 0;
    // More occurrences than are scored at once: the suffix matches come first, and
    // meanwhile the rows of (up to kPrefetchOcc of) the occurrences head for L2 --
    // H_{j-1} with one bulk prefetch, the attention values at key j when the
    // selected rows of a key are side by side -- so that the candidates' scoring,
    // a round trip later, finds them there.
    if (indexed && nocc > kSpeculate && tid < nocc && tid < kPrefetchOcc) {
        const int64_t j = is.occ[tid];
        if (HAS_H && j >= 1 && j < t)
            prefetch_l2_bulk(static_cast<const char*>(p.H) + (static_cast<int64_t>(b) * p.h_seq_stride + (j - 1) * p.d) * h_es,
                             static_cast<uint32_t>(p.d * h_es));
        if (has_a && p.a_row_stride == 1 && !p.row_idx && j >= 0 && j < t) {
            const size_t a_es = p.a_bf16 ? 2 : 4;
            const char* run = static_cast<const char*>(p.A) + (static_cast<int64_t>(b) * p.a_seq_stride + j * p.a_key_stride) * a_es;
            const char* end = run + static_cast<int64_t>(p.R) * a_es;          // every address inside the run
            for (const char* a = run; a < end; a += 128) asm volatile("prefetch.global.L2 [%0];" ::"l"(a));
            asm volatile("prefetch.global.L2 [%0];" ::"l"(end - 1));
        }
    }

    // One thread: the counts, and the index's new state.
    auto counts = [&](int nstar, int total) {
        write_counts(p, b, nstar, total, bad);
        // the index now covers 0 .. t-1 (or is unusable: a token it cannot hold, or stale)
        if (usable) ix.ilen[b] = is.bad_token ? -1 : static_cast<int32_t>(t);
        else if (il > t && il > 0) ix.ilen[b] = -1;             // shrunk (an empty context keeps il = 0)
    };

    // ---- the list scored: every occurrence, or the candidates --------------------------
    // spec: at most kSpeculate occurrences, all scored at once; their suffix matches
    // are read in the same round trip and n* then picks the candidates among them.
    // Otherwise the candidates (the first C_cap) are known first, from the occurrences'
    // suffix matches or from a rescan of the context: a few go through the same code,
    // kSpeculate a pass (one loop with one call of the scorer: a second copy, run only by
    // the sequences with more, cost them its instruction fetch); many are left to
    // score_deferred_kernel.
    constexpr int NB = kSpeculate;
    BestKeys best = {0, 0};
    int nstar = 0, total = 0;
    const bool spec = indexed && nocc <= kSpeculate;
    if (indexed && !spec) {
        int mloc = 0;
        for (int i = tid; i < nocc; i += kThreads) {
            const int64_t j = is.occ[i];
            int32_t pv[PLDP_MAX_NGRAM - 1];                       // x_{j-1}, x_{j-2}, ... all requested at once
#pragma unroll
            for (int m = 1; m < PLDP_MAX_NGRAM; ++m) {
                const int64_t q = j - m;
                pv[m - 1] = (m < p.ngram_max && q >= 0) ? (q >= il ? is.newtok[q - il] : RD::one(row + q)) : 0;
            }
            int m = 1;
#pragma unroll
            for (int k = 1; k < PLDP_MAX_NGRAM; ++k)
                if (m == k && k < p.ngram_max && j - k >= 0 && pv[k - 1] == is.suf[k]) m = k + 1;
            is.occ_m[i] = m;
            mloc = m > mloc ? m : mloc;
        }
        mloc = __reduce_max_sync(0xFFFFFFFFu, mloc);
        if (lane == 0) is.wmax[warp] = mloc;
        __syncthreads();
        if (warp == 0) {
            int mx = 0;
#pragma unroll
            for (int w = 0; w < kWarps; ++w) mx = is.wmax[w] > mx ? is.wmax[w] : mx;
            const int ns = mx >= p.ngram_min ? mx : 0;           // m <= ngram_max already
            int base = 0;
            if (ns > 0)
                for (int c0 = 0; c0 < nocc; c0 += 32) {
                    const bool c = c0 + lane < nocc && is.occ_m[c0 + lane] >= ns;
                    const unsigned bal = __ballot_sync(0xFFFFFFFFu, c);
                    if (c) {
                        const int r = base + __popc(bal & ((1u << lane) - 1u));
                        is.cand[r] = is.occ[c0 + lane];
                        if (r < p.C_cap) cand_row[r] = is.occ[c0 + lane];
                    }
                    base += __popc(bal);
                }
            if (lane == 0) {
                is.nstar = ns;
                is.ncand = base;
            }
        }
        __syncthreads();
        nstar = is.nstar;
        total = is.ncand;
    } else if (!indexed) {
        rescan<IVEC, RD>(p, t, row, cand_row, is.rs, is.cand, kOccCap, nstar, total);
    }

    const int n = spec ? nocc : (total < p.C_cap ? total : p.C_cap);
    const bool deferred = p.defer != nullptr && n > kCtaPasses * NB;
    if (tid == 0) decide(p, b, deferred ? static_cast<unsigned>(n) : 0u);
    if (deferred) {
        if (mine) index_put(ix, b, mytok, myslot, il + tid);      // the slot taken above
        if (tid == 0) counts(nstar, total);
        return;
    }
    {
        const int32_t* list = spec ? is.occ : is.cand;
        int32_t pre[PLDP_MAX_NGRAM - 1];                          // spec, thread h < n: x_{j-1}, x_{j-2}, ...
        const int64_t jm = (spec && tid < n) ? list[tid] : -1;
#pragma unroll
        for (int m = 1; m < PLDP_MAX_NGRAM; ++m) {
            const int64_t q = jm - m;
            pre[m - 1] = (jm >= 0 && m < p.ngram_max && q >= 0) ? (q >= il ? is.newtok[q - il] : RD::one(row + q)) : 0;
        }
        const bool staged = p.K <= kDraftWin;                     // warp 0, lane i: token i after list[h], h < NB
        int32_t dv[NB];
        int64_t j0[NB];
#pragma unroll
        for (int h = 0; h < NB; ++h) {
            j0[h] = h < n ? list[h] : -1;
            const int64_t q = j0[h] + 1 + lane;
            dv[h] = (staged && warp == 0 && h < n && lane < p.K && q <= t) ? RD::one(row + q) : -1;
        }
        float s_h[NB], s_a[NB];
        for (int i0 = 0; i0 < n; i0 += NB) {                      // one pass but for many candidates
            const int nb = n - i0 < NB ? n - i0 : NB;
            int64_t j[NB];
#pragma unroll
            for (int h = 0; h < NB; ++h) j[h] = h < nb ? list[i0 + h] : -1;
            cta_score<TH, NB>(p, b, j, nb, t, part_buf<NB>(sh.part[(i0 / NB) & 1]), s_h, s_a);
            if (!spec && warp == 0)                               // candidates: keys now, in every lane
#pragma unroll
                for (int h = 0; h < NB; ++h)
                    if (h < nb)
                        take_score<TH>(p, i0 + h, j[h], s_h[h], s_a[h], lane == 0 ? hsc : nullptr,
                                       lane == 0 ? asc : nullptr, best);
        }
        if (mine) index_put(ix, b, mytok, myslot, il + tid);      // the slot taken above
        if (warp != 0) return;
        if (spec) {
            // n* among the scored occurrences (n <= NB: one pass), then their keys
            int m = 0;
            if (lane < n) {
                m = 1;
#pragma unroll
                for (int k = 1; k < PLDP_MAX_NGRAM; ++k)
                    if (m == k && k < p.ngram_max && jm - k >= 0 && pre[k - 1] == is.suf[k]) m = k + 1;
            }
            int mh[NB], mx = 0;
#pragma unroll
            for (int h = 0; h < NB; ++h) {
                mh[h] = __shfl_sync(0xFFFFFFFFu, m, h);
                mx = mh[h] > mx ? mh[h] : mx;
            }
            nstar = mx >= p.ngram_min ? mx : 0;                   // m <= ngram_max already
            int r = 0;                                            // candidates: ascending, as the occurrences
            if (nstar > 0)
#pragma unroll
                for (int h = 0; h < NB; ++h) {
                    if (h >= n || mh[h] < nstar) continue;
                    if (r < p.C_cap) {
                        if (lane == 0) cand_row[r] = static_cast<int32_t>(j0[h]);
                        take_score<TH>(p, r, j0[h], s_h[h], s_a[h], lane == 0 ? hsc : nullptr,
                                       lane == 0 ? asc : nullptr, best);
                    }
                    ++r;
                }
            total = r;
        }
        if (lane == 0) counts(nstar, total);
        write_choice<HAS_H>(p, b, t, best.h, best.a, lane, [&](int i, int64_t js) -> int32_t {
            if (staged && i == lane) {
                int32_t v = -1;
                bool found = false;
#pragma unroll
                for (int h = 0; h < NB; ++h)
                    if (h < n && j0[h] == js) {
                        v = dv[h];
                        found = true;
                    }
                if (found) return v;
            }
            return RD::one(row + js + 1 + i);
        });
    }
}

template <typename TH, bool IVEC>
__global__ void __launch_bounds__(kThreads, 1) draft_index_kernel(const DraftParams p, const IndexView ix) {
    __shared__ StepShared sh;
    __shared__ IndexShared is;
    pdl_enter();
    index_draft<TH, IVEC, ReadOnlyIds>(p, ix, blockIdx.x, p.seq_len[blockIdx.x], sh, is);
}

// Verification of the current step -- the finish of greedy verification: the
// accepted length, the bonus token and the append (Sec. 4.4) -- and then, in the
// same CTA, the next step's drafting with the token index.  One CTA per
// sequence, launched behind the verification's argmax pass (greedy: the targets
// are the row keys) or behind the draws of sampling verification (va.row_draws).  The draft step
// starts from the context the finish has just written: its length is known
// without a read, and the appended ids are read through L2.
constexpr int kOldWin = 32;                        // old-context tokens read before the wait (a lane each)

template <typename TH, bool IVEC>
__global__ void __launch_bounds__(kThreads, 1) verify_draft_kernel(const VerifyArgs va, const DraftParams p,
                                                                    const IndexView ix) {
    __shared__ StepShared sh;
    __shared__ IndexShared is;
    __shared__ long long L_after;
    __shared__ int32_t oldwin[kOldWin];                          // x_{Lw}, ..., x_{Lw + kOldWin - 1}
    const int b = blockIdx.x;
    // Read before the wait, since the argmax pass does not write them (its
    // predecessors, which did, completed before it started): the indexed length,
    // the last kOldWin tokens of the context as it was before this step's append --
    // the drafting's appended ids and suffix reach back into them -- and the
    // finish's draft, draft length and context length.
    const int64_t il = ix.ilen[b];
    const int64_t L_old = va.seq_len ? static_cast<int64_t>(va.seq_len[b]) : -1;
    const int64_t Lw = L_old - kOldWin;
    const int32_t* row_b = p.ids + static_cast<int64_t>(b) * p.ids_stride;
    FinishIn fin = {};
    if (threadIdx.x < kOldWin) {
        const int64_t q = Lw + threadIdx.x;
        oldwin[threadIdx.x] = (L_old >= 1 && L_old <= p.T_cap && q >= 0) ? __ldcg(row_b + q) : 0;
        fin = finish_inputs(va, b, static_cast<int>(threadIdx.x));    // the draft: not written by the pass
    }
    pdl_enter();                                                  // the pass's row keys are final
    if (threadIdx.x < 32) {
        const int lane = static_cast<int>(threadIdx.x);
        __syncwarp();                                             // oldwin written by this warp
        FinishOut fo;
        const int64_t r0 = static_cast<int64_t>(b) * (va.K + 1);
        const RowTokens src{va.row_draws ? nullptr : va.row_keys + r0, va.row_draws ? va.row_draws + r0 : nullptr};
        const int64_t L1 = finish_sequence(va, b, lane, src, &fo, &fin);
        if (lane == 0) L_after = L1;
        // The drafting's first reads come from what the finish holds: the ids appended
        // since the index was brought up to date (il .. t-1) and the suffix x_t, x_{t-1},
        // ...; positions the finish wrote come from its draft and bonus, older ones from L2.
        if (L1 >= 0 && L1 <= p.T_cap) {
            const int64_t t = L1 - 1;
            const int64_t L0 = fo.appended ? L1 - fo.n - 1 : L1;  // the first appended position
            const int32_t* row = p.ids + static_cast<int64_t>(b) * p.ids_stride;
            const int32_t* dr = va.draft + static_cast<int64_t>(b) * va.K;
            auto tok = [&](int64_t q) -> int32_t {
                if (q >= L0) return q - L0 < fo.n ? dr[q - L0] : fo.bonus;
                if (L0 == L_old && q >= Lw) return oldwin[q - Lw];     // read before the wait
                return __ldcg(row + q);
            };
            const bool usable = il >= 0 && il <= t;
            const int64_t nnew = usable ? t - il : 0;
            if (usable && nnew <= kNewCap)
                for (int64_t k = lane; k < nnew; k += 32) is.newtok[k] = tok(il + k);
            if (lane < PLDP_MAX_NGRAM) is.suf[lane] = (lane < p.ngram_max && t - lane >= 0) ? tok(t - lane) : 0;
        } else if (lane < PLDP_MAX_NGRAM) {
            is.suf[lane] = 0;                                     // no last token (as the drafting reads it)
        }
    }
    __syncthreads();                                              // the append is visible to the whole CTA
    const int64_t L = L_after >= 0 ? static_cast<int64_t>(L_after) : static_cast<int64_t>(__ldcg(p.seq_len + b));
    index_draft<TH, IVEC, CoherentIds, true>(p, ix, b, L, sh, is, il);
}

// Index build: positions 0 .. seq_len-2 of every sequence, by a cluster per sequence that
// clears the sequence's entries and then inserts its positions.  Only the first half of
// an entry is cleared (a 32-byte sector: the count and seven slots; a slot is read only
// below the count), which is all that most entries of a vocabulary ever see.
//
// What bounds it: the clearing, V * 32 bytes a sequence (525 MB at batch 128, V = 128256:
// 85 us alone), and the atomics: those of a text's frequent tokens take turns on a few
// entries, and entries that have left L2 come back from memory.  Batch 16 x 8k,
// V = 128256: 64 -> 28 us against a memset of everything, a kernel that inserted and one
// that wrote the lengths; batch 64 x 16k, V = 32000: 69 -> 38 us; batch 1 x 4k: 19.5 -> 13 us.
//
// More sequences than clusters of 8 at once and entries beyond what L2 holds of those under
// way: one launch clears them all at the memory's rate, and smaller clusters insert all the
// sequences in one wave.  By clusters of 8 that clear and insert in turn, a few sequences at
// a time, each wave waited for its frequent tokens.  Batch 128 x 32k, V = 128256, against
// those and (in brackets) the three kernels: Zipf tokens whose ids are in the order of their
// frequency, as a tokenizer's roughly are, 272 -> 203 (243) us, named at random 233 -> 186
// (230), uniform tokens 207 -> 236 (306); 200 x 4k, V = 152000, 226 -> 184 (290); 300 x 16k,
// V = 128256, in order 463 -> 344 (435).
constexpr int kBuildThreads = 1024;
constexpr int kBuildLoads = 4;                     // positions in flight per thread
constexpr int kClearThreads = 512;
// Tokens counted (and cleared) at a time, when there are more sequences than clusters at
// once: entries then wait less long for their positions.  Inserting alone, uniform tokens at
// the first size above: 248 us against 266 by 65536 (Zipf in order 217 / 205).  With the
// clearing, batch 128 x 32k, V = 50257, Zipf: 147 / 131 us against 164 / 152 in one pass.
constexpr int64_t kBuildTokens = 32768;
// The largest vocabulary whose entries the clusters clear themselves: batch 128 x 32k,
// V = 50257, Zipf 137 / 127 us (cleared first 133 / 127), uniform 127 (188); the same of
// V = 66000, Zipf 184 / 166 us (148 / 143), uniform 150 (205); 64 x 16k, V = 100000, Zipf
// 90 / 80 us (80 / 84), uniform 80 (84).
constexpr int kBuildClearTokens = 65536;

__global__ void __launch_bounds__(kClearThreads) index_clear_kernel(uint4* __restrict__ entries, int64_t sectors) {
    pdl_enter();
    const int64_t step = static_cast<int64_t>(gridDim.x) * kClearThreads;
#pragma unroll 4
    for (int64_t u = static_cast<int64_t>(blockIdx.x) * kClearThreads + threadIdx.x; u < 2 * sectors; u += step)
        entries[(u >> 1) * (kEntryWords / 4) + (u & 1)] = make_uint4(0u, 0u, 0u, 0u);
}

__global__ void __launch_bounds__(kBuildThreads, 2)
index_build_kernel(const int32_t* __restrict__ ids, int64_t ids_stride, const int32_t* __restrict__ seq_len, int B,
                   int64_t T_cap, IndexView ix, uint32_t* __restrict__ status, int S,
                   int64_t tokens, bool clear) {
    pdl_enter();
    const int b = blockIdx.x / S;
    const int rank = blockIdx.x - b * S;
    const int tid = threadIdx.x;
    const int64_t L = seq_len[b];
    const bool valid = L >= 0 && L <= T_cap;
    const int64_t t = valid ? L - 1 : 0;
    if (rank == 0 && tid == 0) {
        ix.flags[b] = 0;
        if (ix.defer != nullptr) {
            ix.defer[b] = DeferSlot{};
            if (b == 0) ix.defer[B] = DeferSlot{};
        }
    }
    const int step = S * kBuildThreads, first = rank * kBuildThreads + tid;
    uint4* entries = reinterpret_cast<uint4*>(index_entry(ix, b, 0));   // four vectors each
    const int32_t* row = ids + static_cast<int64_t>(b) * ids_stride;
    bool bad = false;                              // a token the index cannot hold
    for (int64_t v0 = 0; v0 < ix.V; v0 += tokens) {                    // cluster-uniform
        const int64_t v1 = v0 + tokens < ix.V ? v0 + tokens : ix.V;
        if (clear)
#pragma unroll 4
            for (int64_t u = 2 * v0 + first; u < 2 * v1; u += step)
                entries[(u >> 1) * (kEntryWords / 4) + (u & 1)] = make_uint4(0u, 0u, 0u, 0u);   // a sector per two lanes
        if (S > 1) {
            cluster_arrive();
            cluster_wait();
        } else {
            __syncthreads();
        }
        for (int64_t q0 = first; q0 < t; q0 += static_cast<int64_t>(step) * kBuildLoads) {
            int32_t tok[kBuildLoads];
            int slot[kBuildLoads];
#pragma unroll
            for (int u = 0; u < kBuildLoads; ++u) {
                const int64_t q = q0 + static_cast<int64_t>(u) * step;
                tok[u] = q < t ? __ldg(row + q) : static_cast<int32_t>(v0);
                bad |= tok[u] < 0 || tok[u] >= ix.V;
            }
#pragma unroll
            for (int u = 0; u < kBuildLoads; ++u) {
                const bool in = q0 + static_cast<int64_t>(u) * step < t && tok[u] >= v0 && tok[u] < v1;
                slot[u] = in ? index_take(ix, b, tok[u]) : kIndexSlots;
            }
#pragma unroll
            for (int u = 0; u < kBuildLoads; ++u) index_put(ix, b, tok[u], slot[u], q0 + static_cast<int64_t>(u) * step);
        }
    }
    if (bad) atomicOr(ix.flags + b, 1);
    if (S > 1) {
        cluster_arrive();
        cluster_wait();
    } else {
        __syncthreads();
    }
    if (rank != 0 || tid != 0) return;
    const bool bad_token = __ldcg(ix.flags + b) != 0;
    ix.ilen[b] = (!valid || bad_token) ? -1 : static_cast<int32_t>(L >= 1 ? L - 1 : 0);
    if (status && !valid) atomicOr(status + b, PLDP_ST_SEQ_LEN);
    if (status && bad_token) atomicOr(status + b, PLDP_ST_TOKEN_RANGE);
}

// Byte offsets of the index parts (ilen, flags, entries, the drafting calls' scratch),
// 256-byte aligned.  Memory without the last part (an index was its first `defer` bytes
// before deferred scoring was there) does too: its sequences score their own candidates.
struct IndexLayout {
    size_t ilen, flags, entries, defer, total;
};
inline IndexLayout index_layout(int B, int V) {
    auto up = [](size_t x) { return (x + 255) / 256 * 256; };
    IndexLayout l;
    l.ilen = 0;
    l.flags = up(static_cast<size_t>(B) * 4);
    l.entries = l.flags + up(static_cast<size_t>(B) * 4);
    l.defer = l.entries + up(static_cast<size_t>(B) * V * kEntryWords * 4);
    l.total = l.defer + up((static_cast<size_t>(B) + 1) * sizeof(DeferSlot));
    return l;
}
inline IndexView index_view(void* base, size_t bytes, int B, int V) {
    const IndexLayout l = index_layout(B, V);
    char* c = static_cast<char*>(base);
    return IndexView{bytes < l.total ? nullptr : reinterpret_cast<DeferSlot*>(c + l.defer), reinterpret_cast<int32_t*>(c + l.ilen),
                     reinterpret_cast<int32_t*>(c + l.flags), reinterpret_cast<int32_t*>(c + l.entries), V};
}

// Whether a drafting kernel that scores up to `here` candidates of a sequence by itself
// may have to leave some: then its launch is followed by score_deferred_kernel's.
inline bool may_defer(const DraftParams& p, int64_t here) { return p.C_cap > here && p.T_cap > here; }

template <typename TH>
pldp_status launch_deferred(const DraftParams& p, int B, cudaStream_t s, const char* what) {
    const auto kernel = p.count ? score_deferred_kernel<TH, true> : score_deferred_kernel<TH, false>;
    int64_t blocks = resident_blocks(reinterpret_cast<const void*>(kernel), kThreads, 0);
    const int64_t most = p.C_cap < p.T_cap ? p.C_cap : p.T_cap;               // candidates of a sequence
    const int64_t need = (most + kWarps - 1) / kWarps * B;                    // units of one per warp
    if (blocks > need) blocks = need;
    const cudaError_t e =
        launch_pdl(kernel, dim3(static_cast<unsigned>(blocks)), dim3(kThreads), 0, s, 0, p, B);
    if (e != cudaSuccess) return fail(PLDP_ERR_CUDA, "%s: launch failed: %s", what, cudaGetErrorString(e));
    return PLDP_OK;
}

template <typename TH, bool IVEC>
pldp_status launch_t(const DraftParams& p0, int B, cudaStream_t s) {
    int CL;
    int64_t chunk;
    scan_shape(p0.T_cap, B, resident_blocks(reinterpret_cast<const void*>(&draft_step_kernel<TH, IVEC>), kThreads, 0),
               kPositionsPerCta, &CL, &chunk);
    DraftParams p = p0;
    if (!may_defer(p, static_cast<int64_t>(kCtaPasses) * kScoreBatch * CL)) p.defer = nullptr;
    const cudaError_t e = launch_pdl(draft_step_kernel<TH, IVEC>, dim3(static_cast<unsigned>(B) * CL), dim3(kThreads), 0,
                                     s, CL > 1 ? CL : 0, p, CL, chunk);
    if (e != cudaSuccess) return fail(PLDP_ERR_CUDA, "draft_step: launch failed: %s", cudaGetErrorString(e));
    return p.defer ? launch_deferred<TH>(p, B, s, "draft_step") : PLDP_OK;
}

template <typename TH, bool IVEC>
pldp_status launch_index_t(const DraftParams& p0, const IndexView& ix, int B, cudaStream_t s) {
    DraftParams p = p0;
    p.defer = may_defer(p, kCtaPasses * kMaxScoreBatch) ? ix.defer : nullptr;
    p.count = p.defer != nullptr && 2 * B > sm_count();
    cudaError_t e = launch_pdl(draft_index_kernel<TH, IVEC>, dim3(static_cast<unsigned>(B)), dim3(kThreads), 0, s, 0,
                               p, ix);
    if (e != cudaSuccess) return fail(PLDP_ERR_CUDA, "draft_step (indexed): launch failed: %s", cudaGetErrorString(e));
    return p.defer ? launch_deferred<TH>(p, B, s, "draft_step (indexed)") : PLDP_OK;
}

template <typename TH>
pldp_status launch_draft_step(const DraftParams& p, int B, cudaStream_t s, bool ivec, const IndexView* ix) {
    if (ix) return ivec ? launch_index_t<TH, true>(p, *ix, B, s) : launch_index_t<TH, false>(p, *ix, B, s);
    return ivec ? launch_t<TH, true>(p, B, s) : launch_t<TH, false>(p, B, s);
}

// The checks and argument block of pldp_draft_step (`what` names the call in
// messages).  empty: B == 0, nothing to launch.
pldp_status prepare_draft(const pldp_draft_step_args* a, const char* what, DraftParams& p, IndexView& ixv,
                          bool& has_ix, bool& ivec, bool& empty) {
    const int B = a->B;
    if (B < 0) return fail(PLDP_ERR_INVALID_ARG, "%s: B < 0", what);
    if (B > 65535) return fail(PLDP_ERR_UNSUPPORTED, "%s: B > 65535", what);
    if (a->T_cap < 0 || a->T_cap > kMaxPositions)
        return fail(PLDP_ERR_INVALID_ARG, "%s: T_cap outside [0, 2^27]", what);
    if (a->ids_stride < a->T_cap) return fail(PLDP_ERR_INVALID_ARG, "%s: ids_stride < T_cap", what);
    if (a->ngram_min < 1 || a->ngram_max < a->ngram_min || a->ngram_max > PLDP_MAX_NGRAM)
        return fail(PLDP_ERR_INVALID_ARG, "%s: need 1 <= ngram_min <= ngram_max <= %d", what,
                    PLDP_MAX_NGRAM);
    if (a->C_cap < 0) return fail(PLDP_ERR_INVALID_ARG, "%s: C_cap < 0", what);
    if (a->K < 1) return fail(PLDP_ERR_INVALID_ARG, "%s: K < 1", what);
    if (!a->H && !a->A) return fail(PLDP_ERR_INVALID_ARG, "%s: neither H nor A given", what);
    if (a->draft_from != 0 && a->draft_from != 1)
        return fail(PLDP_ERR_INVALID_ARG, "%s: draft_from must be 0 (hidden) or 1 (attention)", what);
    if ((a->draft_from == 0 && !a->H) || (a->draft_from == 1 && !a->A))
        return fail(PLDP_ERR_INVALID_ARG, "%s: draft_from names a ranking that is not given", what);
    size_t qbytes = 0, h_es = 0;
    if (a->H) {
        if (a->h_dtype != PLDP_F32 && a->h_dtype != PLDP_BF16)
            return fail(PLDP_ERR_UNSUPPORTED, "%s: unsupported hidden dtype %d", what, (int)a->h_dtype);
        h_es = a->h_dtype == PLDP_F32 ? 4 : 2;
        if (a->d < 1) return fail(PLDP_ERR_INVALID_ARG, "%s: d < 1", what);
        qbytes = static_cast<size_t>(a->d) * h_es;
        if (qbytes > kMaxQueryBytes)
            return fail(PLDP_ERR_UNSUPPORTED, "%s: d * sizeof(dtype) > %zu", what, kMaxQueryBytes);
        if (a->h_seq_stride < a->T_cap * a->d)
            return fail(PLDP_ERR_INVALID_ARG, "%s: h_seq_stride < T_cap*d", what);
        if (a->threshold != a->threshold) return fail(PLDP_ERR_INVALID_ARG, "%s: threshold is NaN", what);
    }
    int sel = 0;
    if (a->A) {
        if (a->a_dtype != PLDP_F32 && a->a_dtype != PLDP_BF16)
            return fail(PLDP_ERR_UNSUPPORTED, "%s: unsupported attention dtype %d", what, (int)a->a_dtype);
        if (a->agg != PLDP_AGG_MAX && a->agg != PLDP_AGG_SUM)
            return fail(PLDP_ERR_INVALID_ARG, "%s: unknown aggregation %d", what, (int)a->agg);
        if (a->R < 1) return fail(PLDP_ERR_INVALID_ARG, "%s: R < 1", what);
        if (const char* why = attention_layout_error(a->R, a->T_cap, a->a_row_stride,
                                                     a->a_key_stride == 0 ? 1 : a->a_key_stride, a->a_seq_stride))
            return fail(PLDP_ERR_INVALID_ARG, "%s: attention layout: %s", what, why);
        sel = a->row_idx ? a->n_sel : a->R;
        if (sel < 1 || sel > kMaxSelRows)
            return fail(PLDP_ERR_INVALID_ARG, "%s: need 1 <= n_sel <= %d", what, kMaxSelRows);
    }
    empty = B == 0;
    if (empty) return PLDP_OK;
    if (!a->ids || !a->seq_len || !a->cand_count || !a->match_len || !a->draft || !a->draft_len ||
        (a->C_cap > 0 && !a->cand_pos) || (a->H && !a->best_h) || (a->A && !a->best_a))
        return fail(PLDP_ERR_INVALID_ARG, "%s: null pointer", what);
    has_ix = a->index != nullptr;
    if (a->index) {
        if (a->V < 1) return fail(PLDP_ERR_INVALID_ARG, "%s: V < 1 with an index", what);
        const size_t need = index_layout(B, a->V).defer;
        if (a->index_bytes < need || !aligned16(a->index))
            return fail(PLDP_ERR_INVALID_ARG, "%s: index needs %zu bytes, 16-byte aligned", what, need);
        ixv = index_view(a->index, a->index_bytes, B, a->V);
    } else if (!a->workspace || a->workspace_bytes < static_cast<size_t>(B) * kSeqWs || !aligned16(a->workspace)) {
        return fail(PLDP_ERR_INVALID_ARG, "%s: workspace needs %zu bytes, 16-byte aligned", what,
                    static_cast<size_t>(B) * kSeqWs);
    }
    if (a->H && !(aligned16(a->H) && qbytes % 16 == 0 && (a->h_seq_stride * h_es) % 16 == 0))
        return fail(PLDP_ERR_UNSUPPORTED,
                    "draft_step: hidden rows must be 16-byte aligned (the separate calls accept any layout)");

    p = DraftParams{};
    p.ids = a->ids;
    p.ids_stride = a->ids_stride;
    p.seq_len = a->seq_len;
    p.T_cap = a->T_cap;
    p.ngram_min = a->ngram_min;
    p.ngram_max = a->ngram_max;
    p.cand_pos = a->cand_pos;
    p.C_cap = a->C_cap;
    p.cand_count = a->cand_count;
    p.match_len = a->match_len;
    p.H = a->H;
    p.h_bf16 = a->h_dtype == PLDP_BF16;
    p.d = a->d;
    p.h_seq_stride = a->h_seq_stride;
    p.threshold = a->threshold;
    p.h_scores = a->h_scores;
    p.best_h = a->best_h;
    p.best_h_score = a->best_h_score;
    p.A = a->A;
    p.a_bf16 = a->a_dtype == PLDP_BF16;
    p.R = a->R;
    p.a_row_stride = a->a_row_stride;
    p.a_key_stride = a->a_key_stride == 0 ? 1 : a->a_key_stride;
    p.a_seq_stride = a->a_seq_stride;
    p.row_idx = a->row_idx;
    p.n_sel = sel;
    p.agg = static_cast<int>(a->agg);
    p.a_scores = a->a_scores;
    p.best_a = a->best_a;
    p.best_a_score = a->best_a_score;
    p.draft_from = a->draft_from;
    p.K = a->K;
    p.draft = a->draft;
    p.draft_len = a->draft_len;
    p.status = a->status;
    p.B = B;
    p.defer = has_ix ? nullptr : reinterpret_cast<DeferSlot*>(a->workspace);
    ivec = aligned16(a->ids) && a->ids_stride % 4 == 0 && a->T_cap % 4 == 0;
    return PLDP_OK;
}

template <typename TH, bool IVEC>
pldp_status launch_verify_draft_t(const VerifyArgs& va, const DraftParams& p0, const IndexView& ix, int B,
                                  cudaStream_t s) {
    DraftParams p = p0;
    p.defer = may_defer(p, kCtaPasses * kMaxScoreBatch) ? ix.defer : nullptr;
    p.count = p.defer != nullptr && 2 * B > sm_count();
    const cudaError_t e = launch_pdl(verify_draft_kernel<TH, IVEC>, dim3(static_cast<unsigned>(B)), dim3(kThreads), 0,
                                     s, 0, va, p, ix);
    if (e != cudaSuccess) return fail(PLDP_ERR_CUDA, "verify_draft: launch failed: %s", cudaGetErrorString(e));
    return p.defer ? launch_deferred<TH>(p, B, s, "verify_draft") : PLDP_OK;
}

template <typename TH>
pldp_status launch_verify_draft(const VerifyArgs& va, const DraftParams& p, const IndexView& ix, int B, bool ivec,
                                cudaStream_t s) {
    return ivec ? launch_verify_draft_t<TH, true>(va, p, ix, B, s) : launch_verify_draft_t<TH, false>(va, p, ix, B, s);
}

}  // namespace
}  // namespace pldp

using namespace pldp;

extern "C" PLDP_API size_t pldp_draft_workspace_size(int B) {
    return B < 0 ? 0 : static_cast<size_t>(B) * kSeqWs;
}

extern "C" PLDP_API pldp_status pldp_draft_step(const pldp_draft_step_args* a, void* stream) {
    if (!a) return fail(PLDP_ERR_INVALID_ARG, "draft_step: null argument block");
    DraftParams p;
    IndexView ixv = {};
    bool has_ix = false, ivec = false, empty = false;
    const pldp_status st = prepare_draft(a, "draft_step", p, ixv, has_ix, ivec, empty);
    if (st != PLDP_OK || empty) return st;
    const int B = a->B;
    const IndexView* ix = has_ix ? &ixv : nullptr;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (!a->H) return launch_draft_step<NoHidden>(p, B, s, ivec, ix);
    if (a->h_dtype == PLDP_BF16) return launch_draft_step<__nv_bfloat16>(p, B, s, ivec, ix);
    return launch_draft_step<float>(p, B, s, ivec, ix);
}

extern "C" PLDP_API pldp_status pldp_verify_greedy_draft(const pldp_verify_draft_args* a, void* stream) {
    if (!a) return fail(PLDP_ERR_INVALID_ARG, "verify_greedy_draft: null argument block");
    const pldp_draft_step_args& n = a->next;
    if (!n.index) return fail(PLDP_ERR_INVALID_ARG, "verify_greedy_draft: the next draft needs a token index");
    if (a->V < 1) return fail(PLDP_ERR_INVALID_ARG, "verify_greedy_draft: V < 1");
    if (n.V != a->V) return fail(PLDP_ERR_INVALID_ARG, "verify_greedy_draft: the index's V differs from the logits'");
    if (a->dtype != PLDP_F32 && a->dtype != PLDP_BF16)
        return fail(PLDP_ERR_UNSUPPORTED, "verify_greedy_draft: unsupported dtype %d", (int)a->dtype);
    if (n.T_cap > INT32_MAX) return fail(PLDP_ERR_INVALID_ARG, "verify_greedy_draft: bad T_cap");
    DraftParams p;
    IndexView ixv = {};
    bool has_ix = false, ivec = false, empty = false;
    const pldp_status st = prepare_draft(&n, "verify_greedy_draft", p, ixv, has_ix, ivec, empty);
    if (st != PLDP_OK || empty) return st;
    const int B = n.B, K = n.K;
    if (!a->logits || !a->draft || !a->draft_len || !a->accept_len || !a->next_token)
        return fail(PLDP_ERR_INVALID_ARG, "verify_greedy_draft: null pointer");
    const size_t need = pldp_verify_workspace_size(B, K, a->V);
    if (!a->workspace || a->workspace_bytes < need || !aligned16(a->workspace))
        return fail(PLDP_ERR_INVALID_ARG, "verify_greedy_draft: workspace needs %zu bytes, 16-byte aligned", need);
    // verification appends to the context the next draft reads: next.ids and next.seq_len
    VerifyArgs va = verify_args(B, K, a->V, a->draft, a->draft_len, a->argmax, a->accept_len, a->next_token,
                                const_cast<int32_t*>(n.ids), n.ids_stride, const_cast<int32_t*>(n.seq_len), n.T_cap,
                                a->kv_keep_len, n.status);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const pldp_status sp = launch_verify_pass(a->logits, a->dtype, va, a->workspace, s, "verify_greedy_draft");
    if (sp != PLDP_OK) return sp;
    if (!n.H) return launch_verify_draft<NoHidden>(va, p, ixv, B, ivec, s);
    if (n.h_dtype == PLDP_BF16) return launch_verify_draft<__nv_bfloat16>(va, p, ixv, B, ivec, s);
    return launch_verify_draft<float>(va, p, ixv, B, ivec, s);
}

extern "C" PLDP_API size_t pldp_verify_sample_draft_workspace_size(int B, int K, int V, pldp_dtype dtype) {
    return sample_draft_workspace_size(B, K, V, dtype);
}

extern "C" PLDP_API pldp_status pldp_verify_sample_draft(const pldp_verify_sample_draft_args* a, void* stream) {
    if (!a) return fail(PLDP_ERR_INVALID_ARG, "verify_sample_draft: null argument block");
    const pldp_draft_step_args& n = a->next;
    if (!n.index) return fail(PLDP_ERR_INVALID_ARG, "verify_sample_draft: the next draft needs a token index");
    if (a->V < 1) return fail(PLDP_ERR_INVALID_ARG, "verify_sample_draft: V < 1");
    if (n.V != a->V) return fail(PLDP_ERR_INVALID_ARG, "verify_sample_draft: the index's V differs from the logits'");
    if (a->dtype != PLDP_F32 && a->dtype != PLDP_BF16)
        return fail(PLDP_ERR_UNSUPPORTED, "verify_sample_draft: unsupported dtype %d", (int)a->dtype);
    if (!(a->temperature > 0.f) || isinf(a->temperature))
        return fail(PLDP_ERR_INVALID_ARG, "verify_sample_draft: temperature must be positive and finite");
    if (n.T_cap > INT32_MAX) return fail(PLDP_ERR_INVALID_ARG, "verify_sample_draft: bad T_cap");
    if (n.K >= 1 && static_cast<int64_t>(n.K) + 1 > 12288)
        return fail(PLDP_ERR_UNSUPPORTED, "verify_sample_draft: K > 12287");
    DraftParams p;
    IndexView ixv = {};
    bool has_ix = false, ivec = false, empty = false;
    const pldp_status st = prepare_draft(&n, "verify_sample_draft", p, ixv, has_ix, ivec, empty);
    if (st != PLDP_OK || empty) return st;
    const int B = n.B, K = n.K;
    if (!a->logits || !a->uniforms || !a->draft || !a->draft_len || !a->accept_len || !a->next_token)
        return fail(PLDP_ERR_INVALID_ARG, "verify_sample_draft: null pointer");
    const size_t need = sample_draft_workspace_size(B, K, a->V, a->dtype);
    if (!a->workspace || a->workspace_bytes < need || !aligned16(a->workspace))
        return fail(PLDP_ERR_INVALID_ARG, "verify_sample_draft: workspace needs %zu bytes, 16-byte aligned", need);
    // verification appends to the context the next draft reads: next.ids and next.seq_len
    VerifyArgs va = verify_args(B, K, a->V, a->draft, a->draft_len, a->sampled, a->accept_len, a->next_token,
                                const_cast<int32_t*>(n.ids), n.ids_stride, const_cast<int32_t*>(n.seq_len), n.T_cap,
                                a->kv_keep_len, n.status);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const pldp_status sp = launch_sample_draws(a->logits, a->dtype, va, a->temperature, a->uniforms, a->workspace, s,
                                               "verify_sample_draft");
    if (sp != PLDP_OK) return sp;
    if (!n.H) return launch_verify_draft<NoHidden>(va, p, ixv, B, ivec, s);
    if (n.h_dtype == PLDP_BF16) return launch_verify_draft<__nv_bfloat16>(va, p, ixv, B, ivec, s);
    return launch_verify_draft<float>(va, p, ixv, B, ivec, s);
}

extern "C" PLDP_API size_t pldp_index_size(int B, int V) {
    if (B < 0 || V < 1) return 0;
    return index_layout(B, V).total;
}

extern "C" PLDP_API pldp_status pldp_index_build(const int32_t* ids, int64_t ids_stride, const int32_t* seq_len,
                                                 int B, int64_t T_cap, int V, void* index, size_t index_bytes,
                                                 uint32_t* status, void* stream) {
    if (B < 0) return fail(PLDP_ERR_INVALID_ARG, "index_build: B < 0");
    if (B > 65535) return fail(PLDP_ERR_UNSUPPORTED, "index_build: B > 65535");
    if (V < 1) return fail(PLDP_ERR_INVALID_ARG, "index_build: V < 1");
    if (T_cap < 0 || T_cap > kMaxPositions) return fail(PLDP_ERR_INVALID_ARG, "index_build: T_cap outside [0, 2^27]");
    if (ids_stride < T_cap) return fail(PLDP_ERR_INVALID_ARG, "index_build: ids_stride < T_cap");
    if (B == 0) return PLDP_OK;
    if (!ids || !seq_len || !index) return fail(PLDP_ERR_INVALID_ARG, "index_build: null pointer");
    const size_t need = index_layout(B, V).defer;
    if (index_bytes < need || !aligned16(index))
        return fail(PLDP_ERR_INVALID_ARG, "index_build: index needs %zu bytes, 16-byte aligned", need);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const IndexView ix = index_view(index, index_bytes, B, V);
    // a cluster of 8 where its CTAs have a few entries or positions a thread
    const int64_t work = T_cap > V ? T_cap : V;
    int64_t S = work / (4 * kBuildThreads);
    S = S < 1 ? 1 : (S > kScanMaxCluster ? kScanMaxCluster : S);
    const int64_t ctas = resident_blocks(reinterpret_cast<const void*>(&index_build_kernel), kBuildThreads, 0);
    const int64_t tokens = B > ctas / S ? kBuildTokens : V;
    const bool clear_first = B > ctas / S && V > kBuildClearTokens;
    if (clear_first) {
        while (S > 1 && B * S > ctas) S /= 2;                    // all sequences at once
        const cudaError_t e = launch_pdl(index_clear_kernel, dim3(8 * sm_count()), dim3(kClearThreads), 0, s, 0,
                                         reinterpret_cast<uint4*>(ix.entries), static_cast<int64_t>(B) * V);
        if (e != cudaSuccess) return fail(PLDP_ERR_CUDA, "index_build: launch failed: %s", cudaGetErrorString(e));
    }
    const cudaError_t e = launch_pdl(index_build_kernel, dim3(static_cast<unsigned>(B * S)), dim3(kBuildThreads), 0, s,
                                     S > 1 ? static_cast<int>(S) : 0, ids, ids_stride, seq_len, B, T_cap, ix, status,
                                     static_cast<int>(S), tokens, !clear_first);
    if (e != cudaSuccess) return fail(PLDP_ERR_CUDA, "index_build: launch failed: %s", cudaGetErrorString(e));
    return PLDP_OK;
}
