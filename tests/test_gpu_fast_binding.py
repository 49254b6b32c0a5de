"""Native part of the binding: the same results and the same errors as the Python code, which takes every call that is out of the ordinary."""
import dataclasses
import types

import pytest
import torch

from paper_2311_12023_b200 import binding, inputs

pytestmark = pytest.mark.gpu
CFG = inputs.QuantConfig(3, 64, 8, 64, 32)


def python_only(monkeypatch):
    monkeypatch.setattr(binding, "_fast", types.SimpleNamespace(linear=lambda *a: None, encode=lambda *a: None))


def make(N=256, K=192, M=5, r=16):
    g = torch.Generator(device="cuda").manual_seed(3)
    b = lambda *s: torch.randn(*s, generator=g, device="cuda").to(torch.bfloat16)
    W = torch.randn(N, K, generator=g, device="cuda") * 0.02
    q = binding.encode(W, CFG)
    return W, q, b(N, r), b(r, K), b(M, K), b(M, N), binding.alloc_workspace(q, r, M)


@pytest.mark.parametrize("M", [1, 5, 40, 300])
@pytest.mark.parametrize("rank", [True, False])
def test_same_results(monkeypatch, M, rank):
    W, q, L1, L2, X, dY, ws = make(M=M)
    f = (L1, L2) if rank else (None, None)
    got = binding._fast.linear(False, q, *f, X, None, ws), binding._fast.linear(True, q, *f, dY, None, ws)
    params = tuple(None if t is None else torch.nn.Parameter(t) for t in f)
    given = torch.empty_like(got[0])
    assert binding.linear_fwd(q, *params, X, out=given, workspace=ws) is given and torch.equal(given, got[0])
    parts = binding._fast.encode(W, CFG, None)
    python_only(monkeypatch)
    assert torch.equal(got[0], binding.linear_fwd(q, *f, X, workspace=ws)) and torch.equal(got[1], binding.linear_bwd_input(q, *f, dY, workspace=ws))
    p = binding.encode(W, CFG)
    for a, b in zip(parts, (p.codes, p.scale_codes, p.scale2)):
        assert a.dtype == b.dtype and a.shape == b.shape and torch.equal(a, b)


def test_unusual_calls_go_to_the_python_code():
    W, q, L1, L2, X, dY, ws = make()
    fast = binding._fast

    class Tagged(torch.Tensor):
        pass

    ok = (q, L1, L2, X, None, ws)
    assert isinstance(fast.linear(False, *ok), torch.Tensor)
    bad = [(q, L1, L2, X.as_subclass(Tagged), None, ws), (q, L1, L2, X.float(), None, ws), (q, L1, L2, X.t(), None, ws), (q, L1, L2, X[0], None, ws),
           (q, L1, L2, X.cpu(), None, ws), (q, L1, L2, X, None, None), (q, L1, None, X, None, ws), (q, None, L2, X, None, ws), (q, L1[:, :8], L2, X, None, ws),
           (q, L1.float(), L2, X, None, ws), (q, L1, L2, dY, None, ws), (q, L1, L2, X, [1], ws), (None, L1, L2, X, None, ws), (q, L1, L2, None, None, ws),
           (dataclasses.replace(q, cfg=None), L1, L2, X, None, ws), (dataclasses.replace(q, N=2.0), L1, L2, X, None, ws)]
    for args in bad:
        assert fast.linear(False, *args) is None
    for args in [(W.double(), CFG, None), (W.t(), CFG, None), (W.cpu(), CFG, None), (W, None, None), (W, inputs.QuantConfig(3, 64, 4, 64, 32), None),
                 (W, inputs.QuantConfig(5, 64, 8, 64, 32), None), (W.as_subclass(Tagged), CFG, None)]:
        assert fast.encode(*args) is None
    with torch.overrides.TorchFunctionMode():
        assert fast.linear(False, *ok) is None
    assert type(binding.linear_fwd(q, L1, L2, X.as_subclass(Tagged), workspace=ws)) is torch.Tensor


def test_same_errors(monkeypatch):
    W, q, L1, L2, X, dY, ws = make()
    calls = [lambda: binding.linear_fwd(q, L1, L2, X[:0], workspace=ws), lambda: binding.linear_fwd(q, L1, L2, X, workspace=ws[:64]),
             lambda: binding.linear_fwd(q, L1, L2, X, workspace=ws[1:]), lambda: binding.encode(W, CFG, workspace=ws[:4]),
             lambda: binding.linear_fwd(q, L1, L2, dY, workspace=ws), lambda: binding.linear_bwd_input(q, L1[:, :8], L2, dY, workspace=ws),
             lambda: binding.encode(W.double(), CFG), lambda: binding.encode(W, inputs.QuantConfig(5, 64, 8, 64, 32))]

    def seen():
        out = []
        for c in calls:
            with pytest.raises((binding.LqloraError, AssertionError)) as e:
                c()
            out.append((e.type, getattr(e.value, "status", None), str(e.value) if e.type is binding.LqloraError else None))
        return out

    native = seen()
    python_only(monkeypatch)
    assert native == seen()
