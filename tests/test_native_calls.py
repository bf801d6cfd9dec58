"""The binding's native checks (csrc/host_calls.cpp) against the Python ones: the same
calls are made, with the same results, and what a check refuses is refused the same way."""
import os
import subprocess
import sys

import pytest
import torch

import paper_2412_01447_gb300 as pk
import workloads as wl
from paper_2412_01447_gb300 import _build
from tests._parity import Buffers, snapshot

DEV = "cuda"


def test_nothing_is_taken_off_the_device():
    """Host tensors, wrong counts of arguments and other kinds are left to Python."""
    pk.build()
    pk._load()
    c = pk._calls
    x, y = torch.zeros((2, 8), dtype=torch.int32), torch.zeros(2, dtype=torch.int32)
    assert c.find_candidates(x, y, 1, 3, x, y, y, None, None, None) is None
    assert c.find_candidates(x) is None and c.top_heads(None, 1, y, None) is None
    assert c.draft_step(x, y, 1, 3, x, y, y, 4, x, y, None, None, {"H": None}) is None
    assert c.verify_greedy(None, x, y, y, y, y, None, None, None, None, None, None, None) is None
    with pytest.raises(ValueError):
        c.bind((1, 2))


@pytest.fixture(scope="session")
def any_device():
    """The native checks built without the device check, so that host tensors reach the
    rest of them (bound to recorders here, never to the library)."""
    pk.build()
    pk._load()
    return _build.build_calls(out=os.path.join(_build.BUILD_DIR, "any_device", "_pldp_calls.so"),
                              extra_flags=["-DPLDP_TEST_ANY_DEVICE"])


def test_a_build_belongs_to_its_torch_and_python(monkeypatch):
    """The extension of another torch or Python is not taken for this one's."""
    mine = _build.calls_path()
    monkeypatch.setattr(torch, "__version__", "0.0.0+other")
    assert _build.calls_path() != mine
    monkeypatch.undo()
    monkeypatch.setattr(_build.sysconfig, "get_config_var", lambda name: ".cpython-00-other.so")
    assert _build.calls_path() != mine


def test_the_library_does_not_need_the_extension(monkeypatch, tmp_path):
    """Without a C++ compiler the library is built and linked all the same and an extension
    of older sources goes; one that does not load is left out."""
    pk.build()
    path = tmp_path / "_pldp_calls.so"
    monkeypatch.setattr(_build, "calls_path", lambda: str(path))
    path.write_bytes(b"not a library")
    lib = pk._load()
    with pytest.warns(RuntimeWarning, match="ctypes"):
        assert pk._load_calls(lib) is None
    monkeypatch.setenv("CXX", str(tmp_path / "no-such-compiler"))
    os.utime(path, (1, 1))
    with pytest.warns(RuntimeWarning, match="ctypes"):
        _build.build()
    assert not path.exists() and pk._load_calls(lib) is None
    monkeypatch.setattr(_build, "LIB", str(tmp_path / "libpldp.so"))
    monkeypatch.setattr(_build, "BUILD_DIR", str(tmp_path / "_build"))
    monkeypatch.setattr(_build, "sources", lambda: [os.path.join(_build.CSRC, "abi.cu")])
    with pytest.warns(RuntimeWarning, match="ctypes"):
        assert os.path.exists(_build.build())


VMAP = """
import ctypes, importlib.util, sys
import torch
spec = importlib.util.spec_from_file_location("_pldp_calls", sys.argv[1])
c = importlib.util.module_from_spec(spec)
spec.loader.exec_module(c)
made = []
@ctypes.CFUNCTYPE(ctypes.c_int)
def call():
    made.append(1)
    return 0
c.bind((ctypes.cast(call, ctypes.c_void_p).value,) * 12)
i = lambda *s: torch.zeros(s, dtype=torch.int32)
B, C, T = 2, 3, 16
calls = [lambda x: c.rank_hidden(x, i(B), i(B, C), i(B), i(B), None, None, 0.0, None, 0),
         lambda x: c.rank_attention(x, i(B), i(B, C), i(B), i(B), None, 0, None, None, None, 0),
         lambda x: c.identify_heads(i(B, T), i(B), x, i(T), 8, None, None, 0),
         lambda x: c.verify_greedy(x, i(B, T - 1), i(B), i(B), i(B), i(64), None, None, None, None, None, None, 0)]
for f in calls:
    assert f(torch.zeros(B, T, T)) == 0                  # a plain tensor: the call is made
    n, got = len(made), []
    torch.vmap(lambda x: (got.append(f(x)), x)[1])(torch.zeros(2, B, T, T))
    assert got == [None] and len(made) == n, got         # one without storage: left to Python
print("left to python")
"""


def test_a_tensor_without_storage_is_left_to_python(any_device):
    """torch.vmap hands a function tensors that pass every check of type, shape and
    strides and whose data pointer raises: in a child process, since that once raised
    without the interpreter's lock."""
    r = subprocess.run([sys.executable, "-c", VMAP, any_device], capture_output=True, text=True, timeout=600)
    assert r.returncode == 0 and "left to python" in r.stdout, (r.returncode, r.stdout, r.stderr[-2000:])


def _steps(buf, inp, w, index, calls):
    """Every call of a decode step once, through the native checks or without them."""
    B, K, V = w.B, w.K, w.V
    ids, L, H, A = inp["ids"].clone(), inp["seq_len"].clone(), inp["H"], inp["A"]
    rows = torch.arange(0, w.R, 2, dtype=torch.int32, device=DEV)
    u = torch.linspace(0.05, 0.95, B * (K + 1), device=DEV).reshape(B, K + 1)
    ws = torch.zeros(pk.pldp_verify_sample_draft_workspace_size(B, K, V), dtype=torch.uint8, device=DEV)
    counts = torch.zeros(w.R, dtype=torch.int32, device=DEV)
    top = torch.zeros(3, dtype=torch.int32, device=DEV)
    kw = dict(H=H, best_h=buf.best_h, h_scores=buf.scores_h, A=A, best_a=buf.best_a, row_idx=rows, agg=1,
              a_scores=buf.scores_a, draft_from="attention", status=buf.status, threshold=-0.5)
    out = []
    pk.pldp_find_candidates(ids, L, 1, 3, buf.cand, buf.cnt, buf.ml, buf.status, T_cap=w.T)
    pk.pldp_rank_hidden(H, L, buf.cand, buf.cnt, buf.best_h, scores=buf.scores_h, best_score=buf.bscore_h)
    pk.pldp_rank_attention(A, L, buf.cand, buf.cnt, buf.best_a, row_idx=rows, agg=1, scores=buf.scores_a)
    pk.pldp_extract_draft(ids, L, buf.best_h, buf.draft, buf.dlen)
    pk.pldp_verify_greedy(inp["logits"], buf.draft, buf.dlen, buf.acc, buf.nxt, buf.ws, argmax=buf.argmax)
    pk.pldp_verify_sample(inp["logits"], u, buf.draft, buf.dlen, buf.acc, buf.nxt, ws, temperature=0.7)
    out.append(snapshot(buf))
    pk.pldp_index_build(ids, L, V, index, status=buf.status)
    pk.pldp_draft_step(ids, L, 1, 3, buf.cand, buf.cnt, buf.ml, K, buf.draft, buf.dlen, buf.dws, **kw)
    pk.pldp_verify_greedy_draft(inp["logits"], buf.draft, buf.dlen, buf.acc, buf.nxt, buf.ws, ids, L, 1, 3, buf.cand,
                                buf.cnt, buf.ml, buf.draft, buf.dlen, index, argmax=buf.argmax, **kw)
    pk.pldp_verify_sample_draft(inp["logits"], u, buf.draft, buf.dlen, buf.acc, buf.nxt, ws, ids, L, 1, 3, buf.cand,
                                buf.cnt, buf.ml, buf.draft, buf.dlen, index, kv_keep_len=buf.kv, **kw)
    pk.pldp_identify_heads(inp["ids"], inp["seq_len"] - 1, A.contiguous(), counts, max_suffix=16)
    pk.pldp_top_heads(counts, 3, top)
    out.append(snapshot(buf))
    return out + [dict(ids=ids.cpu().numpy(), L=L.cpu().numpy(), counts=counts.cpu().numpy(), top=top.cpu().numpy())]


@pytest.mark.gpu
def test_native_and_python_calls_agree(lib, monkeypatch):
    w = wl.CONFIGS["attention_b32_ctx8k"].replace(B=3, prompt_len=600, out_len=200, V=4000, d=256, h_dtype="bf16",
                                                  layers=2, heads=4, planted_heads=2, C_cap=64)
    inp = wl.single_step(w, device=DEV)
    index = torch.empty(pk.pldp_index_size(w.B, w.V), dtype=torch.uint8, device=DEV)
    taken = []

    class Counted:
        def __getattr__(self, name):
            def call(*args):
                rc = getattr(native, name)(*args)
                taken.append((name, rc))
                return rc
            return call

    native = pk._calls
    assert native is not None
    got = []
    for calls in (Counted(), None):
        monkeypatch.setattr(pk, "_calls", calls)
        got.append(_steps(Buffers(w.B, w.K, w.V, w.C_cap, DEV), inp, w, index, calls))
    assert len(taken) == 12 and all(rc == 0 for _, rc in taken), taken
    for a, b in zip(*got):
        for k in a:
            assert (a[k] == b[k]).all() or ((a[k] != a[k]) == (b[k] != b[k])).all(), k


@pytest.mark.gpu
def test_errors_of_the_library_are_raised(lib):
    """A call whose buffers pass and that the library refuses raises its message."""
    ids = torch.zeros((2, 64), dtype=torch.int32, device=DEV)
    L = torch.full((2,), 10, dtype=torch.int32, device=DEV)
    buf = Buffers(2, 4, 8, 8, DEV)
    with pytest.raises(pk.PldpError, match="ngram"):
        pk.pldp_find_candidates(ids, L, 3, 1, buf.cand, buf.cnt, buf.ml)
    with pytest.raises(TypeError):
        pk.pldp_draft_step(ids, L, 1, 3, buf.cand, buf.cnt, buf.ml, 4, buf.draft, buf.dlen, buf.dws, no_such=1)
    with pytest.raises(ValueError):
        pk.pldp_extract_draft(ids, L, buf.best_h, buf.draft.t(), buf.dlen)
