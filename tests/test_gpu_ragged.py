"""Verification where rows of logits are not a whole number of 16 bytes (a vocabulary with
an added token): the streaming pass cuts rows inside vectors.  Argmaxes against the oracle
bit for bit, at row lengths around the limits of the paths, with maxima and ties at the
rows' ends."""
import numpy as np
import pytest
import torch

import oracle
import paper_2412_01447_gb300 as pk
from tests._parity import host

pytestmark = pytest.mark.gpu
DEV = "cuda"


# 2 KB is the shortest row of the streaming pass (1024 bf16, 512 fp32)
@pytest.mark.parametrize("V,dtype", [(1023, torch.bfloat16), (1025, torch.bfloat16), (1031, torch.bfloat16),
                                     (2049, torch.bfloat16), (32001, torch.bfloat16), (511, torch.float32),
                                     (513, torch.float32), (1026, torch.float32), (32003, torch.float32)])
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
