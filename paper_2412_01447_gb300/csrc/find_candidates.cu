// pldp_find_candidates: the candidate search of PLD+ (Eq. 1, Sec. 4.2, with the
// longest-suffix n-gram rule) as its own kernel -- one thread-block cluster per
// sequence running the scan of pldp_scan.cuh.  Each CTA scans its chunk once, the
// cluster's CTAs tell each other their longest match and its count over distributed
// shared memory, and the CTAs that hold the longest write their positions.
#include "pldp_scan.cuh"

namespace pldp {
namespace {

constexpr int64_t kPositionsPerCta = 1024;   // at least; the batch sets the rest (one wave)
constexpr int kFindList = 128;               // positions listed per warp

template <bool VEC>
__global__ void __launch_bounds__(kScanThreads, 3)
find_candidates_kernel(const int32_t* __restrict__ ids, int64_t ids_stride,
                       const int32_t* __restrict__ seq_len, int64_t T_cap, int ngram_min,
                       int ngram_max, int32_t* __restrict__ cand_pos, int C_cap,
                       int32_t* __restrict__ cand_count, int32_t* __restrict__ match_len,
                       uint32_t* __restrict__ status, int CL, int64_t chunk) {
    __shared__ ScanLists<kFindList> sl;
    __shared__ ScanPeer tab[kScanMaxCluster];
    pdl_enter();
    const int b = blockIdx.x / CL;
    const int rank = blockIdx.x - b * CL;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int32_t* row = ids + static_cast<int64_t>(b) * ids_stride;
    // the chunk's first ids are requested before the context length is known
    const int64_t seg = chunk / kScanWarps;
    const int64_t s0 = static_cast<int64_t>(rank) * chunk + warp * seg;
    const int nit = static_cast<int>(seg / kScanTile);
    WarpScan<VEC, ReadOnlyIds, 8> sc;
    sc.begin(row, s0, nit, T_cap, lane);

    // Every CTA of the cluster sees the same seq_len, so these exits are
    // cluster-uniform and no CTA is left waiting at a cluster barrier.
    const int64_t L = seq_len[b];
    const int64_t t = L - 1;
    if (L < 0 || L > T_cap || t < 1) {
        if (rank == 0 && tid == 0) {
            cand_count[b] = 0;
            match_len[b] = 0;
            if ((L < 0 || L > T_cap) && status) status[b] |= PLDP_ST_SEQ_LEN;
        }
        return;
    }
    if (CL > 1) cluster_arrive_relaxed();                 // this CTA runs: its shared memory may be written
    if (tid < PLDP_MAX_NGRAM) sl.suf[tid] = (tid < ngram_max && t - tid >= 0) ? __ldg(row + t - tid) : 0;
    __syncthreads();
    scan_lists(sc, t, ngram_max, warp, sl);
    __syncthreads();
    const CtaMatches cm = cta_matches(sl, warp);
    if (CL > 1) {
        cluster_wait();
        if (tid < CL)
            *cg::this_cluster().map_shared_rank(&tab[rank], tid) = ScanPeer{cm.m, cm.cnt, cm.over ? 1 : 0};
        cluster_arrive();
        cluster_wait();                                   // every CTA's outcome is in
    } else {
        if (tid == 0) tab[0] = ScanPeer{cm.m, cm.cnt, cm.over ? 1 : 0};
        __syncthreads();
    }
    const ScanTotal st = scan_total(tab, CL, rank, ngram_min);
    if (rank == 0 && tid == 0) {
        cand_count[b] = st.total;
        match_len[b] = st.nstar;
        if (status && st.total > C_cap) status[b] |= PLDP_ST_CAND_OVERFLOW;
    }
    int32_t* dst = cand_pos + static_cast<int64_t>(b) * C_cap;
    scan_emit<VEC, ReadOnlyIds>(row, s0, nit, t, T_cap, ngram_max, st.nstar, static_cast<int64_t>(st.before) + cm.base,
                                C_cap, warp, lane, sl, [&](int64_t i, int32_t j) { dst[i] = j; });
}

}  // namespace
}  // namespace pldp

using namespace pldp;

extern "C" PLDP_API pldp_status pldp_find_candidates(const int32_t* ids, int64_t ids_stride,
                                                     const int32_t* seq_len, int B, int64_t T_cap,
                                                     int ngram_min, int ngram_max,
                                                     int32_t* cand_pos, int C_cap,
                                                     int32_t* cand_count, int32_t* match_len,
                                                     uint32_t* status, void* stream) {
    if (B < 0) return fail(PLDP_ERR_INVALID_ARG, "find_candidates: B < 0");
    if (T_cap < 0 || T_cap > INT32_MAX)
        return fail(PLDP_ERR_INVALID_ARG, "find_candidates: T_cap outside [0, 2^31)");
    if (ids_stride < T_cap) return fail(PLDP_ERR_INVALID_ARG, "find_candidates: ids_stride < T_cap");
    if (ngram_min < 1 || ngram_max < ngram_min || ngram_max > PLDP_MAX_NGRAM)
        return fail(PLDP_ERR_INVALID_ARG, "find_candidates: need 1 <= ngram_min <= ngram_max <= %d",
                    PLDP_MAX_NGRAM);
    if (C_cap < 0) return fail(PLDP_ERR_INVALID_ARG, "find_candidates: C_cap < 0");
    if (B == 0) return PLDP_OK;
    if (!ids || !seq_len || !cand_count || !match_len || (C_cap > 0 && !cand_pos))
        return fail(PLDP_ERR_INVALID_ARG, "find_candidates: null pointer");

    const bool vec = aligned16(ids) && ids_stride % 4 == 0 && T_cap % 4 == 0;
    const void* fn = vec ? reinterpret_cast<const void*>(&find_candidates_kernel<true>)
                         : reinterpret_cast<const void*>(&find_candidates_kernel<false>);
    int CL;
    int64_t chunk;
    scan_shape(T_cap, B, resident_blocks(fn, kScanThreads, 0), kPositionsPerCta, &CL, &chunk);
    if (static_cast<int64_t>(B) * CL > INT32_MAX)
        return fail(PLDP_ERR_INVALID_ARG, "find_candidates: B too large");

    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(static_cast<unsigned>(B * CL));
    cfg.blockDim = dim3(kScanThreads);
    cfg.dynamicSmemBytes = 0;
    cfg.stream = static_cast<cudaStream_t>(stream);
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = CL;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    cudaError_t e;
    if (vec)
        e = cudaLaunchKernelEx(&cfg, find_candidates_kernel<true>, ids, ids_stride, seq_len, T_cap,
                               ngram_min, ngram_max, cand_pos, C_cap, cand_count, match_len, status,
                               CL, chunk);
    else
        e = cudaLaunchKernelEx(&cfg, find_candidates_kernel<false>, ids, ids_stride, seq_len, T_cap,
                               ngram_min, ngram_max, cand_pos, C_cap, cand_count, match_len, status,
                               CL, chunk);
    if (e != cudaSuccess)
        return fail(PLDP_ERR_CUDA, "find_candidates: launch failed: %s", cudaGetErrorString(e));
    return PLDP_OK;
}
