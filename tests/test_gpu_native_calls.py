"""The native call path of api.py (csrc/bysdf_torch.cpp) against the general one
through ctypes: plain calls take it and give the same bits, and whatever is not
plain gives the same result or the same exception as without it."""
import numpy as np
import pytest
import torch

from paper_2401_12724_gb300 import _native as N
from paper_2401_12724_gb300 import api
from paper_2401_12724_gb300 import inputs as I

pytestmark = pytest.mark.gpu


class Spy:
    """N.calls, counting the calls it took and the ones it left."""

    def __init__(self, calls):
        self.calls, self.took, self.left = calls, 0, 0

    def __getattr__(self, name):
        def call(*args):
            r = getattr(self.calls, name)(*args)
            if r is NotImplemented:
                self.left += 1
            else:
                self.took += 1
            return r
        return call


@pytest.fixture
def spy(monkeypatch):
    N.load()
    assert N.calls is not None
    s = Spy(N.calls)
    monkeypatch.setattr(N, "calls", s)
    return s


def flat(r):
    if isinstance(r, dict):
        return [(k, v) for k, v in r.items()]
    return list(enumerate(r)) if isinstance(r, tuple) else [(0, r)]


def outcome(fn):
    try:
        r = flat(fn())
        torch.cuda.synchronize()
        return "ok", [(k, None if v is None else v.cpu()) for k, v in r]
    except Exception as e:
        return type(e).__name__, str(e)


def same(monkeypatch, fn):
    a = outcome(fn)
    with monkeypatch.context() as m:
        m.setattr(N, "calls", None)
        b = outcome(fn)
    assert a[0] == b[0], (a, b)
    if a[0] != "ok":
        assert a == b
        return a[0]
    assert [k for k, _ in a[1]] == [k for k, _ in b[1]]
    for (k, x), (_, y) in zip(a[1], b[1]):
        assert (x is None and y is None) or \
            (x.dtype == y.dtype and x.shape == y.shape and torch.equal(x, y)), k
    return "ok"


def batch(n, sort=True, seed=5):
    rec = I.random_records(n, n_mat=8, seed=seed, wi_mode="cosine", sample=True, sorted_ids=sort)
    seg = I.seg_offsets_from_ids(rec["mat_id"], 8) if sort else None
    return api.records_to_device(rec, seg_offsets=seg)


def ops(M, d, n, stream=None, det=True):
    """The calls of the native path; the gradients in the deterministic form, whose sums
    have one order."""
    x = torch.linspace(-1, 1, 3 * n, device="cuda").reshape(3, n)
    w = torch.linspace(0.5, 2, n, device="cuda")
    kw = dict(stream=stream)
    return {
        "eval": lambda: api.eval(M, d, **kw),
        "eval_no_pdf": lambda: api.eval(M, d, with_pdf=False, **kw),
        "sample": lambda: api.sample(M, d, **kw),
        "sample_u": lambda: api.sample(M, d, d.get("u1"), d.get("u0"), **kw),
        "pdf": lambda: api.pdf(M, d, **kw),
        "fused": lambda: api.eval_sample_pdf(M, d, **kw),
        "backward": lambda: api.eval_backward(M, d, x, deterministic=det, **kw),
        "ext": lambda: api.eval_backward_ext(M, d, x, deterministic=det, **kw),
        "ext_dirs": lambda: api.eval_backward_ext(M, d, x, deterministic=det, dirs=True, **kw),
        "l2": lambda: api.eval_l2_backward(M, d, x, deterministic=det, **kw),
        "l2_weighted": lambda: api.eval_l2_backward(M, d, x, w, deterministic=det, with_f=False,
                                                    **kw),
    }


@pytest.mark.parametrize("n,sort", [(0, False), (1, False), (777, True), (50_001, True)])
def test_plain_calls_take_the_native_path(spy, monkeypatch, n, sort):
    M, d = api.Materials(I.materials(2)), batch(n, sort)
    # (the deterministic gradients are refused in any order, both ways)
    streams = [None, torch.cuda.Stream(), torch.cuda.Stream().cuda_stream]
    for st in streams:
        torch.cuda.synchronize()
        for name, fn in ops(M, d, n, st).items():
            before = spy.took
            same(monkeypatch, fn)
            assert spy.took == before + 1 and spy.left == 0, name
    if n > 1:
        with torch.cuda.stream(torch.cuda.Stream()):
            for fn in ops(M, d, n).values():
                assert same(monkeypatch, fn) == "ok"
        # any order: one record per material, whose sums have one term
        r = {k: v[..., :8].contiguous() for k, v in d.items() if k != "seg_offsets"}
        r["mat_id"] = torch.arange(8, dtype=torch.int32, device="cuda")
        for fn in ops(M, r, 8, det=False).values():
            assert same(monkeypatch, fn) == "ok"
        assert spy.left == 0


def test_the_workspace_grows_with_the_batch(spy, monkeypatch):
    M = api.Materials(I.materials(2))
    for n in (100, 200_000, 50):
        d = batch(n)
        for fn in ops(M, d, n).values():
            assert same(monkeypatch, fn) == "ok"
        assert M._ws.numel() >= M.lib.bysdf_workspace_size(M.handle, n)
    assert spy.left == 0


class Sub(torch.Tensor):
    pass


class Records(dict):
    pass


CHANGES = {
    "strided": lambda d: {**d, "wi": torch.stack([d["wi"]] * 2, -1)[..., 0]},
    "transposed": lambda d: {**d, "wi": d["wi"].t().contiguous().t()},
    "missing plane": lambda d: {k: v for k, v in d.items() if k != "u"},
    "no plane": lambda d: {**d, "v": None},
    "host plane": lambda d: {**d, "v": d["v"].cpu()},
    "array": lambda d: {**d, "v": d["v"].cpu().numpy()},
    "number": lambda d: {**d, "v": 1.0},
    "unaligned": lambda d: {**d, "v": torch.cat([d["v"][:1], d["v"]])[1:]},
    "no wo": lambda d: {k: v for k, v in d.items() if k != "wo"},
    "no ids": lambda d: {k: v for k, v in d.items() if k not in ("mat_id", "seg_offsets")},
    "ids None": lambda d: {**d, "mat_id": None, "ratio": None},
    "no random numbers": lambda d: {k: v for k, v in d.items() if k != "u1"},
    "subclass": lambda d: {**d, "h": d["h"].as_subclass(Sub)},
    "parameter": lambda d: {**d, "h": torch.nn.Parameter(d["h"])},
    "dict subclass": lambda d: Records(d),
    "scalar h": lambda d: {**d, "h": d["h"][0]},
}


@pytest.mark.parametrize("change", list(CHANGES))
def test_other_records_give_what_the_general_path_gives(spy, monkeypatch, change):
    n = 333
    M, d = api.Materials(I.materials(2)), CHANGES[change](batch(n))
    seen = [same(monkeypatch, fn) for fn in ops(M, d, n).values()]
    if change in ("parameter", "dict subclass", "subclass", "ids None"):
        assert set(seen) == {"ok"}
    elif change in ("strided", "transposed", "missing plane", "no plane", "host plane", "array",
                    "number", "unaligned", "scalar h"):
        assert "ok" not in seen


def test_other_arguments_give_what_the_general_path_gives(spy, monkeypatch):
    n = 333
    M, d = api.Materials(I.materials(2)), batch(n)
    x = torch.rand(n, 3, device="cuda").t()  # not contiguous: the general path copies it
    for fn in (lambda: api.eval_backward(M, d, x, True),
               lambda: api.eval_l2_backward(M, d, x, deterministic=True),
               lambda: api.eval_backward_ext(M, d, x, True, True)):
        assert same(monkeypatch, fn) == "ok"
    for fn in (lambda: api.eval_backward(M, d, x.cpu(), True),
               lambda: api.eval_backward(M, d, None, True),
               lambda: api.sample(M, d, d["u0"].cpu()),
               lambda: api.eval(M, d, stream="no stream"),
               lambda: api.eval(M, None),
               lambda: api.eval_l2_backward(M, d, x, torch.ones(n), True)):
        assert same(monkeypatch, fn) != "ok"
    assert spy.took == 0
    M.close()
    for name, fn in ops(M, d, n).items():
        assert same(monkeypatch, fn) != "ok", name


def test_parameter_updates(spy, monkeypatch):
    M = api.Materials(I.materials(2))
    P = {8: api.default_params(M.descs).cuda(), 15: api.default_params_ext(M.descs).cuda()}
    for cols, p in P.items():
        put, get = (M.set_params, M.get_params) if cols == 8 else \
            (M.set_params_ext, M.get_params_ext)

        def update(q):
            put(P[cols] * 0.5)
            put(q)
            return get()

        plain = [p * 0.9, torch.nn.Parameter(p * 0.9), (p * 0.9).requires_grad_()]
        for q in plain:
            before = spy.left
            assert same(monkeypatch, lambda: update(q)) == "ok"
            assert spy.left == before
        other = [(p * 0.9).double(), (p * 0.9).cpu(), (p * 0.9).t().contiguous().t(),
                 (p * 0.9).as_subclass(Sub)]
        for q in other:
            assert same(monkeypatch, lambda: update(q)) == "ok"
        for q in (p[:1], p[:, :1], p[0], p.cpu().numpy(), None):
            assert same(monkeypatch, lambda: update(q)) != "ok"


def test_autograd_takes_the_native_path(spy):
    n = 777
    M, d = api.Materials(I.materials(2)), batch(n)
    p = api.default_params(M.descs).cuda().requires_grad_()
    f, st = api.bysdf(p, M, d, deterministic=True)
    f.sum().backward()
    assert spy.took == 3 and spy.left == 0
    want = api.eval_backward(M, d, torch.ones(3, n, device="cuda"), deterministic=True)
    assert torch.equal(p.grad, want)
