"""When the native marshalling module is used: only where it was compiled against the running
torch and interpreter; otherwise the calls are left to the binding's Python path, with a warning."""

import sys
import types

import numpy as np
import pytest
import torch

import paper_1607_04245_gb300 as fem
from paper_1607_04245_gb300 import binding, build as fem_build

NAME = "paper_1607_04245_gb300._marshal"


@pytest.fixture()
def fresh(monkeypatch):
    """The binding as before its first call."""
    fem_build.build()
    monkeypatch.setattr(binding, "_native", None)
    monkeypatch.delattr(fem, "_marshal", raising=False)
    return monkeypatch


def test_the_built_module_is_used(fresh):
    m = binding.native()
    assert m.__name__ == NAME and m.built_for == fem_build.marshal_stamp()
    assert torch.__version__ in m.built_for


def _absent(mp):
    mp.setitem(sys.modules, NAME, None)  # import raises ImportError


def _stale(mp):
    m = types.ModuleType(NAME)
    m.built_for = "torch 1.0 abi 0 python x"
    m.init = lambda *a: pytest.fail("a stale module was bound")
    mp.setitem(sys.modules, NAME, m)


def _unmarked(mp):
    m = types.ModuleType(NAME)
    m.init = lambda *a: pytest.fail("a module of unknown origin was bound")
    mp.setitem(sys.modules, NAME, m)


@pytest.mark.parametrize("how", [_absent, _stale, _unmarked])
def test_otherwise_calls_are_declined(fresh, how):
    how(fresh)
    with pytest.warns(RuntimeWarning, match="marshalled in Python"):
        m = binding.native()
    assert m.laplacian(1, 2, 3) is None and m.node2cell() is None
    assert binding.native() is m
    with pytest.raises(ValueError):  # the Python path's own check answers
        fem.fem_integrate_laplacian(torch.zeros(2, 3, dtype=torch.float64), torch.zeros(3, 1, dtype=torch.int32),
                                    torch.zeros(3), torch.zeros(1, 1), None, np.ones(1))


def test_rebuilt_when_the_running_torch_differs(fresh):
    assert fem_build._marshal_is_current()
    calls = []
    fresh.setattr(fem_build, "marshal_stamp", lambda: "torch 9.9 abi 1 python y")
    fresh.setattr(fem_build, "_build_marshal", lambda: calls.append(1))
    assert not fem_build._marshal_is_current()
    fem_build.build()
    assert calls == [1]


@pytest.mark.gpu
def test_the_python_path_gives_the_same(fresh):
    import workloads
    from gpu_util import device_arrays, residual

    case = workloads.laplacian_cube_case(6 * 5 ** 3)
    c, d = device_arrays(case, "mixed")
    ref = residual(c, d, "mixed")
    fresh.setattr(binding, "_native", None)
    _absent(fresh)
    with pytest.warns(RuntimeWarning):
        got = residual(c, d, "mixed")
    assert torch.equal(got, ref)


@pytest.mark.gpu
def test_what_is_no_stream_is_refused():
    """An object that is no torch stream is refused as the Python path refuses it, whatever its attributes."""
    import workloads
    from gpu_util import device_arrays, residual

    case = workloads.laplacian_cube_case(6 * 5 ** 3)
    c, d = device_arrays(case, "mixed")
    other = types.SimpleNamespace(cuda_stream=torch.cuda.current_stream().cuda_stream)
    with pytest.raises(TypeError):
        residual(c, d, "mixed", stream=other)
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    r = residual(c, d, "mixed", stream=s)
    s.synchronize()
    assert torch.equal(r, residual(c, d, "mixed", stream=torch.cuda.current_stream().cuda_stream))
