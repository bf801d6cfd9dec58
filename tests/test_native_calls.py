"""The binding's native checks (csrc/host_calls.cpp) against the Python ones: the same
calls are made, with the same results, and what a check refuses is refused the same way."""
import ctypes
import importlib.util
import inspect
import os
import subprocess
import sys
import types

import numpy as np
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


class Recorder:
    """The library's entry points, each writing down the arguments it is called with."""

    def __init__(self, lib):
        self.made, self.rc, self.fns = [], 0, {}
        for f in pk._CALLS:
            self.fns[f] = ctypes.CFUNCTYPE(ctypes.c_int, *getattr(lib, f).argtypes)(self._entry(f))
        self.addresses = tuple(ctypes.cast(self.fns[f], ctypes.c_void_p).value for f in pk._CALLS)

    def _entry(self, name):
        def entry(*args):
            self.made.append((name, *(bytes(a.contents) if hasattr(a, "contents") else repr(a) for a in args)))
            return self.rc
        return entry

    def pldp_last_error(self):
        return b"refused"

    def __getattr__(self, name):
        return self.fns[name]


B, C, K, V, T, D, R = 3, 5, 4, 16, 40, 8, 6


def _i(*shape):
    return torch.zeros(shape, dtype=torch.int32)


def _f(*shape, dtype=torch.float32):
    return torch.zeros(shape, dtype=dtype)


def _call_arguments():
    """A call of every function with all of its arguments, and the same without the optional ones."""
    H, A = _f(B, T, D, dtype=torch.bfloat16), _f(B, R, T)
    lists = dict(cand_pos=_i(B, C), cand_count=_i(B))
    ctx = dict(ids=_i(B, T + 4)[:, :T], seq_len=_i(B))
    opt = dict(status=_i(B), stream=7)
    find = dict(ngram_min=1, ngram_max=3, match_len=_i(B), **lists)
    both = dict(H=H, best_h=_i(B), h_scores=_f(B, C), best_h_score=_f(B), threshold=0.25, A=A, best_a=_i(B),
                row_idx=_i(2), agg=1, a_scores=_f(B, C), best_a_score=_f(B), draft_from="attention", status=_i(B), T_cap=T - 8)
    ver = dict(logits=_f(B, K + 1, V, dtype=torch.bfloat16), draft=_i(B, K), draft_len=_i(B), accept_len=_i(B),
               next_token=_i(B), workspace=_f(64))
    app = dict(ids=ctx["ids"], seq_len=ctx["seq_len"], kv_keep_len=_i(B), T_cap=T - 8, **opt)
    nxt = dict(next_draft=_i(B, K), next_draft_len=_i(B), index=_f(64), kv_keep_len=_i(B), stream=7, **ctx, **find, **both)
    u = dict(uniforms=_f(B, K + 1), temperature=0.7, sampled=_i(B, K + 1))
    full = {
        "pldp_find_candidates": dict(**ctx, **find, **opt, T_cap=T - 8),
        "pldp_rank_hidden": dict(H=H, seq_len=_i(B), **lists, best_pos=_i(B), scores=_f(B, C), best_score=_f(B),
                                 threshold=0.25, **opt),
        "pldp_rank_attention": dict(A=A.transpose(1, 2).contiguous().transpose(1, 2), seq_len=_i(B), **lists, best_pos=_i(B),
                                    row_idx=_i(2), agg=1, scores=_f(B, C), best_score=_f(B), **opt),
        "pldp_extract_draft": dict(**ctx, best_pos=_i(B), draft=_i(B, K), draft_len=_i(B), T_cap=T - 8, stream=7),
        "pldp_draft_step": dict(**ctx, **find, K=K, draft=_i(B, K), draft_len=_i(B), workspace=_f(64), stream=7, index=_f(64),
                                V=V, **both),
        "pldp_index_build": dict(**ctx, V=V, index=_f(64), T_cap=T - 8, **opt),
        "pldp_verify_greedy": dict(**ver, argmax=_i(B, K + 1), **app),
        "pldp_verify_greedy_draft": dict(**ver, argmax=_i(B, K + 1), **nxt),
        "pldp_verify_sample": dict(**ver, **u, **app),
        "pldp_verify_sample_draft": dict(**ver, **u, **nxt),
        "pldp_identify_heads": dict(ids=ctx["ids"], pos=_i(B), A=A, counts=_i(R), max_suffix=9, r_star=_i(B), **opt),
        "pldp_top_heads": dict(counts=_i(R), k=2, row_idx=_i(2), stream=7),
    }
    assert set(full) == set(pk._CALLS)
    needed = {f: [p.name for p in inspect.signature(getattr(pk, f)).parameters.values()
                  if p.default is p.empty and p.kind != p.VAR_KEYWORD] for f in full}
    plain = {f: {**{k: a[k] for k in needed[f]}, "stream": 0, **({"H": H, "best_h": a["best_h"]} if "best_h" in a else {})}
             for f, a in full.items()}
    return full, plain


def _variants(x):
    """Other things in the place of an argument: kinds, sizes, strides and ranges that a check is for."""
    if isinstance(x, torch.Tensor):
        yield from (None, 3, [1], x.numpy() if x.dtype != torch.bfloat16 else 1.5, x.long(), x.to(torch.float16), x.float(),
                    x.to(torch.bfloat16), x.to(torch.uint32) if x.dtype == torch.int32 else x.double(), x[:-1], x[..., :-1],
                    x[..., :-1].contiguous(), x.flatten(), x.unsqueeze(0), torch.stack([x, x], -1)[..., 0],
                    torch.cat([x, x]), torch.cat([x, x], -1), torch.empty(0, dtype=x.dtype), x.new_zeros(()))
        if x.dim() > 1:
            yield from (x.transpose(-1, -2), x.transpose(0, 1), x[:, :-1], x[:, :-1].contiguous(), x[:, 1:], torch.cat([x, x], 1),
                        x[:1].expand(x.shape))
        if x.is_floating_point():
            yield torch.nn.Parameter(x)
    elif isinstance(x, str):
        yield from ("hidden", "x", 0, 1, 2, True, None, np.int64(1), [])
    else:
        yield from (None, 0, 1, -1, 5, T, T + 1, 2**31 - 1, 2**31, -2**31, -2**31 - 1, 2**40, 2**63, -2**70, 0.0, 1.0, 1.5,
                    float("nan"), float("-inf"), 1e300, True, "1", np.int32(2), np.float32(0.5))


def test_native_and_python_checks_agree(any_device, monkeypatch):
    """Every argument of every call in turn replaced by other things: the native form makes
    the call that the Python form makes, argument for argument, or leaves it to Python.
    Without a GPU: host tensors in both forms, the entry points replaced."""
    spec = importlib.util.spec_from_file_location("_pldp_calls", any_device)
    native = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(native)
    rec = Recorder(pk._load())
    native.bind(rec.addresses)
    monkeypatch.setattr(pk, "_load", lambda: rec)
    monkeypatch.setattr(torch.Tensor, "is_cuda", True, raising=False)

    def outcome(f, args, calls):
        monkeypatch.setattr(pk, "_calls", calls)
        rec.made.clear()
        try:
            getattr(pk, f)(**args)
            return list(rec.made)
        except Exception as e:
            return [*rec.made, type(e), str(e)]

    def agree(f, args, what):
        a, b = outcome(f, args, native), outcome(f, args, None)
        assert a == b, (f, what, a, b)
        return a

    for arguments in _call_arguments():
        for f, args in arguments.items():
            taken = getattr(native, f[5:])
            made = agree(f, args, "as it is")
            assert len(made) == 1 and made[0][0] == f, made
            spy = types.SimpleNamespace(**{f[5:]: lambda *a: seen.append(taken(*a)) or seen[-1]})
            seen = []
            outcome(f, args, spy)
            assert seen == [0], (f, "not taken natively")
            rec.rc = 3
            assert agree(f, args, "refused by the library")[1] is pk.PldpError
            rec.rc = 0
            for name, x in args.items():
                for i, y in enumerate(_variants(x)):
                    agree(f, {**args, name: y}, (name, i, y))
            agree(f, {k: v for k, v in args.items() if k not in ("best_h", "best_a", "V")}, "outputs missing")
            agree(f, {**args, "no_such": 1}, "a keyword it does not have")


def _steps(buf, inp, w, index):
    """Every call of a decode step once; what each of the two halves leaves."""
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
        buf = Buffers(w.B, w.K, w.V, w.C_cap, DEV)
        for t in vars(buf).values():                     # outputs that a call does not write compare too
            if t.dtype != torch.uint8 and t is not buf.status:
                t.fill_(-77)
        index.zero_()                                    # a build leaves half of most entries as they are
        got.append(_steps(buf, inp, w, index))
    assert len(taken) == 12 and all(rc == 0 for _, rc in taken), taken
    for a, b in zip(*got):
        assert a.keys() == b.keys()
        for k in a:
            assert np.array_equal(a[k], b[k], equal_nan=a[k].dtype.kind == "f"), k


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
