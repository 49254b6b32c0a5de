"""Native part of the binding on the host: a module that is missing, does not load or was compiled against another torch is not used and not
required; the Python code takes the calls."""
import sys
import types

import pytest
import torch

import paper_2311_12023_b200 as package
from paper_2311_12023_b200 import build, inputs

CFG = inputs.QuantConfig(3, 64, 8, 64, 32)


@pytest.fixture
def binding(monkeypatch):
    build.build()
    from paper_2311_12023_b200 import binding as b
    monkeypatch.setattr(b, "_fast", None)
    monkeypatch.delattr(package, "_fast", raising=False)
    return b


def calls_go_to_the_python_code(b):
    """All three refuse host tensors by their own assertions."""
    x = torch.zeros(2, 64, dtype=torch.bfloat16)
    q = types.SimpleNamespace(N=64, K=64, cfg=CFG)
    for call in (lambda: b.encode(torch.zeros(4, 64), CFG), lambda: b.linear_fwd(q, None, None, x), lambda: b.linear_bwd_input(q, None, None, x)):
        with pytest.raises(AssertionError):
            call()


def test_calls_without_the_module(binding, monkeypatch):
    monkeypatch.setitem(sys.modules, "paper_2311_12023_b200._fast", None)
    with pytest.warns(RuntimeWarning, match="native part"):
        calls_go_to_the_python_code(binding)


def test_module_of_another_torch_is_not_used(binding, monkeypatch):
    def refuse(*args):
        raise RuntimeError("used")

    other = types.SimpleNamespace(built_for="torch 1.0.0 python 2.7", setup=refuse, linear=refuse, encode=refuse)
    monkeypatch.setitem(sys.modules, "paper_2311_12023_b200._fast", other)
    monkeypatch.setattr(package, "_fast", other, raising=False)
    with pytest.warns(RuntimeWarning, match="torch 1.0.0"):
        calls_go_to_the_python_code(binding)


def test_module_of_this_torch_is_used(binding, recwarn):
    calls_go_to_the_python_code(binding)
    assert type(binding._fast) is types.ModuleType and binding._fast.built_for == build.built_for()
    assert not [w for w in recwarn if "native part" in str(w.message)]


def test_module_is_rebuilt_for_another_torch(binding, monkeypatch):
    assert not build.fast_stale()
    monkeypatch.setattr(torch, "__version__", "9.9.9")
    assert build.fast_stale()
