"""The one-pass candidate scan at the sizes where it can go wrong, against the oracle:
contexts around the tile (128 positions), the chunk unit (1024) and a cluster's chunks,
one CTA or a full cluster, rows that take 16-byte or 4-byte loads, suffixes that reach
over lanes, tiles, warps and CTAs (n up to 8), and x_t so frequent that a warp's list
(128 positions) overflows; then the drafting calls on such lists, whose many candidates
are scored by a warp each."""
import numpy as np
import pytest
import torch

import oracle
import paper_2412_01447_gb300 as pk
from tests._parity import Buffers, gpu_step, host, snapshot
from tests.test_gpu_fused import _compare, i32

pytestmark = pytest.mark.gpu
DEV = "cuda"


def _contexts(T, V, B, seed):
    rng = np.random.default_rng(seed)
    ids = rng.integers(0, V, size=(B, T)).astype(np.int32)
    lens = np.full(B, T, np.int32)
    for b in range(B):
        if b:
            lens[b] = rng.integers(0, T + 1)
        t = int(lens[b]) - 1
        for at in (9, 131, 1027, T // 2):              # copies of the last 9 tokens, over the boundaries
            if t > 9 and at < t - 9:
                ids[b, at - 9:at + 1] = ids[b, t - 9:t + 1]
    return ids, lens


@pytest.mark.parametrize("T", [1, 2, 9, 127, 128, 129, 132, 1023, 1024, 1028, 8192, 9001, 70000])
@pytest.mark.parametrize("V,B", [(1, 2), (3, 1), (40, 5), (5000, 200)])
def test_find_candidates_edges(lib, T, V, B):
    if T * B > 2_000_000:
        B = 9
    ids, lens = _contexts(T, V, B, T + V)
    for ngram, C in (((1, 1), 1500), ((1, 3), 64), ((3, 5), 1024), ((2, 8), 200000)):
        buf = Buffers(B, 8, 8, C, DEV)
        buf.cand.fill_(-7)
        lib.pldp_find_candidates(i32(ids), i32(lens), ngram[0], ngram[1], buf.cand, buf.cnt, buf.ml, buf.status)
        g = snapshot(buf)
        o_cand, o_cnt, o_ml, o_st = oracle.find_candidates(ids, lens, ngram[0], ngram[1], C)
        assert np.array_equal(g["cnt"], o_cnt) and np.array_equal(g["ml"], o_ml)
        assert np.array_equal(g["status"].view(np.uint32), o_st)
        for b in range(B):
            n = min(o_cnt[b], C)
            assert np.array_equal(g["cand"][b, :n], o_cand[b, :n]), b
            assert (g["cand"][b, n:] == -7).all()      # slots past the list are left alone


# lists that overflow (V = 1, 2) or not; one to eight CTAs a sequence; hidden rows of one
# and of several passes of a warp, attention sums over more rows than a CTA has threads
@pytest.mark.parametrize("T,V,B,d,R,agg,dtype", [
    (9000, 1, 3, 64, 20, 0, torch.bfloat16), (9000, 2, 150, 64, 8, 1, torch.bfloat16),
    (6000, 12, 4, 4096, 300, 1, torch.float32), (6001, 12, 4, 4104, 300, 1, torch.bfloat16),
    (700, 6, 5, 1000, 600, 0, torch.float32),
    # the rescan's masks at their last context length, and the lists beyond it
    (40960, 3, 3, 64, 8, 0, torch.bfloat16), (42001, 3, 3, 64, 8, 0, torch.bfloat16),
    (50000, 400, 3, 64, 8, 1, torch.bfloat16),
    # around what a CTA scores by itself (8 or 4 a CTA), and more sequences than a tile of the deferred launch
    (90, 10, 40, 64, 8, 0, torch.bfloat16), (200, 7, 700, 64, 8, 1, torch.bfloat16)])
@pytest.mark.parametrize("ngram", [(1, 1), (1, 3)])
def test_many_candidates(lib, T, V, B, d, R, agg, dtype, ngram):
    K, C = 6, 1100
    ids, lens = _contexts(T, V, B, T + V + B)
    gen = torch.Generator(device=DEV).manual_seed(T)
    H = torch.randn((B, T, d), generator=gen, device=DEV).to(dtype)
    A = torch.rand((B, R, T), generator=gen, device=DEV).to(dtype)
    L = i32(lens)
    index = torch.empty(pk.pldp_index_size(B, V), dtype=torch.uint8, device=DEV)
    pk.pldp_index_build(i32(ids), L, V, index)
    out = []
    for ix in (None, index):                           # scanned, then through the index's rescan
        buf = Buffers(B, K, 8, C, DEV)
        pk.pldp_draft_step(i32(ids), L, ngram[0], ngram[1], buf.cand, buf.cnt, buf.ml, K, buf.draft, buf.dlen,
                           None if ix is not None else buf.dws, H=H, best_h=buf.best_h, h_scores=buf.scores_h,
                           best_h_score=buf.bscore_h, A=A, best_a=buf.best_a, agg=agg, a_scores=buf.scores_a,
                           best_a_score=buf.bscore_a, status=buf.status, index=ix, V=V)
        out.append(snapshot(buf))
        assert not buf.dws.any()                       # the scratch is left zeroed
        _compare(out[-1], ids, lens, H, A, None, agg, ngram, C, K, "hidden")
    for k in ("cand", "scores_h", "scores_a", "best_h", "best_a", "draft"):
        assert np.array_equal(out[0][k], out[1][k], equal_nan=True), k


# calls that leave some, all or none of their sequences to the deferred launch, in turn on the
# same scratch, invalid lengths among them: every call's results are its own and the scratch
# is left zeroed (one sequence, one tile of the deferred launch and several, grids of one wave
# of drafting CTAs and more)
@pytest.mark.parametrize("B,T", [(1, 3000), (37, 2000), (256, 600), (700, 600)])
def test_deferred_in_turn(lib, B, T):
    K, C, V, d = 5, 256, 600, 64
    rng = np.random.default_rng(B)
    gen = torch.Generator(device=DEV).manual_seed(B)
    H = torch.randn((B, T, d), generator=gen, device=DEV).to(torch.bfloat16)
    buf = Buffers(B, K, 8, C, DEV)
    index = torch.empty(pk.pldp_index_size(B, V), dtype=torch.uint8, device=DEV)
    slots = index.numel() - (32 * (B + 1) + 255) // 256 * 256
    for heavy in (0.0, 1.0, 0.0, 0.3, 0.0, 0.02):
        ids = rng.integers(0, V, size=(B, T)).astype(np.int32)
        lens = np.full(B, T, np.int32)
        for b in np.nonzero(rng.random(B) < heavy)[0]:
            ids[b, rng.integers(0, T, size=T // 4)] = ids[b, T - 1]
        if B > 1:
            lens[rng.integers(0, B)] = T + 1
            lens[rng.integers(0, B)] = rng.integers(0, 3)
        L = i32(lens)
        pk.pldp_index_build(i32(ids), L, V, index)
        for ix in (None, index):
            out = buf if ix is None else Buffers(B, K, 8, C, DEV)
            out.status.zero_()
            pk.pldp_draft_step(i32(ids), L, 1, 3, out.cand, out.cnt, out.ml, K, out.draft, out.dlen,
                               None if ix is not None else buf.dws, H=H, best_h=out.best_h, h_scores=out.scores_h,
                               best_h_score=out.bscore_h, status=out.status, index=ix, V=V)
            _compare(snapshot(out), ids, lens, H, None, None, 0, (1, 3), C, K, "hidden")
            assert not buf.dws.any() and not index[slots:slots + 32 * (B + 1)].any()
