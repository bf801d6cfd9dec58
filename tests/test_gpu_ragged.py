"""Verification where rows of logits are not a whole number of 16 bytes (a vocabulary with
an added token): the streaming passes cut rows inside vectors.  Greedy argmaxes against the
oracle bit for bit, sampling draws as in test_gpu_sample.py, at row lengths around the
limits of the paths, with maxima and ties at the rows' ends."""
import numpy as np
import pytest
import torch

import oracle
import paper_2412_01447_gb300 as pk
from tests._parity import host
from tests.test_gpu_sample import _f64, _run, _valid_draw

pytestmark = pytest.mark.gpu
DEV = "cuda"


# 2 KB is the shortest row of the streaming pass (1024 bf16, 512 fp32); every remainder of a vector
@pytest.mark.parametrize("V,dtype", [(1023, torch.bfloat16), (1025, torch.bfloat16), (1031, torch.bfloat16),
                                     (2049, torch.bfloat16), (32001, torch.bfloat16), (511, torch.float32),
                                     (513, torch.float32), (1026, torch.float32), (32003, torch.float32)]
                         + [(V + r, torch.bfloat16) for V in (1024, 2048) for r in range(2, 7)]
                         + [(12001, torch.float32), (12002, torch.float32)])
@pytest.mark.parametrize("B,K", [(1, 1), (5, 7), (64, 10)])
def test_greedy(lib, V, dtype, B, K):
    rng = np.random.default_rng(V + B)
    x = rng.integers(-3, 4, size=(B * (K + 1), V)).astype(np.float32)     # every row's maximum occurs many times
    for r in range(x.shape[0]):
        kind = r % 5
        if kind < 4:
            x[r] -= 10.0                                                   # one or two clear maxima
            x[r, {0: 0, 1: V - 1, 2: rng.integers(0, V), 3: V - 2}[kind]] = 2.0
            if kind == 2:
                x[r, rng.integers(0, V)] = 2.0
    logits = torch.from_numpy(x).reshape(B, K + 1, V).to(dtype).to(DEV)
    draft = torch.randint(0, V, (B, K), dtype=torch.int32, device=DEV)
    dlen = torch.full((B,), K, dtype=torch.int32, device=DEV)
    o = oracle.verify_greedy(host(logits), host(draft), host(dlen))
    shifted = torch.empty(logits.numel() + 1, dtype=dtype, device=DEV)[1:].reshape(logits.shape)   # unaligned logits
    shifted.copy_(logits)
    for lg in (logits, shifted):
        ws = torch.zeros(pk.pldp_verify_workspace_size(B, K, V), dtype=torch.uint8, device=DEV)
        am = torch.full((B, K + 1), -1, dtype=torch.int32, device=DEV)
        acc, nxt = torch.zeros_like(dlen), torch.zeros_like(dlen)
        pk.pldp_verify_greedy(lg, draft, dlen, acc, nxt, ws, argmax=am)
        assert np.array_equal(host(am), o["argmax"])
        assert np.array_equal(host(acc), o["accept_len"]) and np.array_equal(host(nxt), o["next_token"])
        assert not ws.any()


@pytest.mark.parametrize("B,K,dtype", [(2, 12, torch.bfloat16), (3, 12, torch.float32), (3, 13, torch.float32)])
def test_greedy_wide(lib, B, K, dtype):
    test_greedy(lib, 128255, dtype, B, K)


# NaN is no maximum: whole rows, whole lanes (32 bf16 or 16 fp32 a segment) and all but a
# few elements of a row; the streaming path against the element loads, which take one
# element at a time
@pytest.mark.parametrize("V,dtype,B", [(1025, torch.bfloat16, 6), (5003, torch.bfloat16, 6), (5003, torch.float32, 220)])
def test_greedy_nan(lib, V, dtype, B):
    K = 7
    gen = torch.Generator(device=DEV).manual_seed(V)
    logits = torch.randn((B, K + 1, V), generator=gen, device=DEV).to(dtype)
    logits[0] = float("nan")
    logits[1, :, 3:] = float("nan")
    logits[2] = torch.where(torch.rand((K + 1, V), generator=gen, device=DEV) < 0.999, float("nan"), -3.0).to(dtype)
    logits[3] = torch.where(torch.rand((K + 1, V), generator=gen, device=DEV) < 0.5, float("nan"), float("-inf")).to(dtype)
    logits[4, :, : V // 2] = float("nan")
    draft = torch.zeros((B, K), dtype=torch.int32, device=DEV)
    dlen = torch.zeros(B, dtype=torch.int32, device=DEV)
    shifted = torch.empty(logits.numel() + 1, dtype=dtype, device=DEV)[1:].reshape(logits.shape)   # unaligned logits
    shifted.copy_(logits)
    got = []
    for lg in (logits, shifted):
        ws = torch.zeros(pk.pldp_verify_workspace_size(B, K, V), dtype=torch.uint8, device=DEV)
        am = torch.full((B, K + 1), -7, dtype=torch.int32, device=DEV)
        acc, nxt = torch.zeros_like(dlen), torch.zeros_like(dlen)
        pk.pldp_verify_greedy(lg, draft, dlen, acc, nxt, ws, argmax=am)
        got.append(host(am))
    assert np.array_equal(got[0], got[1])
    assert (got[0] >= 0).all() and (got[0][0] == 0).all()


# a last piece with and without room for the elements that a cut row start moves there
# (1017 and 1021 of 1024, 509 and 510 of 512), rows shorter than a vector, several pieces
@pytest.mark.parametrize("V,dtype", [(3, torch.bfloat16), (1017, torch.bfloat16), (1021, torch.bfloat16),
                                     (2041, torch.bfloat16), (32001, torch.bfloat16), (509, torch.float32),
                                     (510, torch.float32), (32003, torch.float32), (128255, torch.bfloat16)]
                         + [(1024 + r, torch.bfloat16) for r in range(1, 8)])
@pytest.mark.parametrize("T", [0.6, 1.0])
def test_sampling(lib, V, dtype, T):
    B, K = 5, 12
    gen = torch.Generator(device=DEV).manual_seed(V)
    logits = (torch.randn((B, K + 1, V), generator=gen, device=DEV) * 2).to(dtype)
    logits[:, ::3, 0] += 9.0                             # weight at the rows' ends
    logits[:, 1::3, V - 1] += 9.0
    u = torch.rand((B, K + 1), generator=gen, device=DEV)
    u[0, :3] = torch.tensor([0.0, 1.0, 0.999999], device=DEV)
    draft, dlen = torch.zeros((B, K), dtype=torch.int32, device=DEV), torch.zeros(B, dtype=torch.int32, device=DEV)
    _, ys, _ = _run(logits, u, draft, dlen, T)
    o = oracle.verify_sample(host(logits), host(u), host(draft), host(dlen), T)["sampled"]
    l64 = _f64(logits)
    diff = np.argwhere(ys != o)
    assert len(diff) <= 2, diff
    for b, i in diff:
        assert _valid_draw(l64[b, i], T, float(u[b, i]), int(ys[b, i])), (b, i, ys[b, i], o[b, i])


# masks that hold the type's lowest value or a large one: whole rows, whole 2 KB pieces and lanes of them;
# whole vectors, cut rows and unaligned (element) loads
@pytest.mark.parametrize("V,dtype,off", [(4096, torch.bfloat16, 0), (4097, torch.bfloat16, 0), (4096, torch.float32, 0),
                                         (4097, torch.float32, 0), (4097, torch.bfloat16, 1)])
@pytest.mark.parametrize("T", [0.3, 1.0, 2.0])
@pytest.mark.parametrize("lowest", [None, -1e9, -1e4])
def test_sampling_masked(lib, V, dtype, off, T, lowest):
    B, K = 3, 7
    gen = torch.Generator(device=DEV).manual_seed(V)
    logits = torch.empty(B * (K + 1) * V + off, dtype=dtype, device=DEV)[off:].view(B, K + 1, V)
    logits.copy_(torch.randn((B, K + 1, V), generator=gen, device=DEV) * 2)
    low = lowest if lowest is not None else torch.finfo(dtype).min
    logits[:, 0] = low
    logits[:, 1, :3000] = low                            # pieces without weight before the row's
    logits[:, 2, 100:] = low
    logits[:, 3, 1:] = low                               # one token left
    logits[:, 4][torch.rand((B, V), generator=gen, device=DEV) < 0.9] = low
    u = torch.rand((B, K + 1), generator=gen, device=DEV)
    draft, dlen = torch.zeros((B, K), dtype=torch.int32, device=DEV), torch.zeros(B, dtype=torch.int32, device=DEV)
    _, ys, _ = _run(logits, u, draft, dlen, T)
    o = oracle.verify_sample(host(logits), host(u), host(draft), host(dlen), T)["sampled"]
    l64 = _f64(logits)
    for b, i in np.argwhere(ys != o):
        assert _valid_draw(l64[b, i], T, float(u[b, i]), int(ys[b, i])), (b, i, ys[b, i], o[b, i])
