"""Workspaces of the PCG solves: the binding's count of the smallest accepted one is the
library's, and a device without room for the full one gets that one."""

import ctypes

import numpy as np
import pytest
import torch

import paper_1607_04245_gb300 as fem
from paper_1607_04245_gb300 import binding, build as fem_build

ERR_ARG, ERR_OOM = -1, -4
SIZES = [(2, 50, 36), (2, 30011, 15200), (3, 7, 12), (3, 3001, 700), (3, 30001, 5800), (3, 120000, 22000)]


@pytest.fixture(scope="module", autouse=True)
def _built():
    fem_build.build()


def _status(name, dim, C, V, work_bytes, refined, prec):
    """The call with arrays that are never read: a workspace of enough bytes fails for its address alone."""
    P, f = ctypes.c_void_p, getattr(binding.lib(), name)
    table = np.full(4 * 3, 0.1)
    t = table.ctypes.data_as(P)
    coefs = [P(256)] * (2 if "elasticity" in name else 1)
    head = [dim, C, V, P(256), P(256), *coefs, 4, t, t, P(256), P(256), P(256), None, P(256)]
    out = [None] * (3 if refined else 2)
    nums = [5, 5, 1e-4, 1e-8] if refined else [5, 1e-8]
    return f(*head, *nums, P(1), work_bytes, *out, prec, None)


@pytest.mark.parametrize("dim,C,V", SIZES)
@pytest.mark.parametrize("name", ["fem_pcg_laplacian", "fem_pcg_elasticity"])
@pytest.mark.parametrize("prec", ["fp64", "mixed", "fp32", "fp64_df"])
def test_least_bytes_of_a_solve(name, dim, C, V, prec):
    p = binding.precision(prec)
    nc = 1 if name == "fem_pcg_laplacian" else dim
    least = binding._pcg_least_bytes(dim, C, V, nc, binding.value_dtype(p).itemsize)
    assert _status(name, dim, C, V, least - 1, False, p) == ERR_OOM
    assert _status(name, dim, C, V, least, False, p) == ERR_ARG
    assert least <= getattr(binding.lib(), name + "_work_bytes" if nc > 1 else "fem_pcg_work_bytes")(dim, C, V, p)


@pytest.mark.parametrize("dim,C,V", SIZES)
@pytest.mark.parametrize("name", ["fem_pcg_laplacian_refined", "fem_pcg_elasticity_refined"])
def test_least_bytes_of_a_refined_solve(name, dim, C, V):
    nc = 1 if "laplacian" in name else dim
    least = binding._refined_least_bytes(dim, C, V, 4, nc)
    assert _status(name, dim, C, V, least - 1, True, 0) == ERR_OOM
    assert _status(name, dim, C, V, least, True, 0) == ERR_ARG


def _limit(monkeypatch, limit):
    """torch.empty of more than `limit` bytes of uint8 raises as a full device does."""
    real, asked = torch.empty, []

    def empty(*a, **k):
        if k.get("dtype") is torch.uint8:
            asked.append(a[0])
            if a[0] > limit:
                raise torch.OutOfMemoryError("out of memory")
        return real(*a, **k)

    monkeypatch.setattr(torch, "empty", empty)
    return asked


def test_falls_back_to_the_least(monkeypatch):
    asked = _limit(monkeypatch, 1000)
    assert binding._pcg_work(5000, 700, "cpu").numel() == 700 and asked == [5000, 700]
    assert binding._pcg_work(900, 700, "cpu").numel() == 900
    with pytest.raises(torch.OutOfMemoryError):
        binding._pcg_work(5000, 2000, "cpu")
    with pytest.raises(torch.OutOfMemoryError):
        binding._pcg_work(2000, 2000, "cpu")


@pytest.mark.gpu
@pytest.mark.parametrize("name,prec", [("fem_pcg_laplacian", "fp64"), ("fem_pcg_laplacian", "mixed"),
                                       ("fem_pcg_elasticity", "mixed"), ("fem_pcg_laplacian_refined", "fp64"),
                                       ("fem_pcg_elasticity_refined", "fp64")])
def test_a_full_device_still_solves(name, prec, monkeypatch):
    from test_gpu_solver_forms import _mesh, _problem

    p = _problem(_mesh(3, 3001), "laplacian" if "laplacian" in name else "elasticity", prec)
    nc, nq = (1 if "laplacian" in name else 3), len(p["rule"][1])
    least = (binding._refined_least_bytes(3, p["C"], p["V"], nq, nc) if "refined" in name else
             binding._pcg_least_bytes(3, p["C"], p["V"], nc, binding.value_dtype(prec).itemsize))
    args = (*p["mesh"], *p["coef"], *p["rule"], *p["lists"])
    kw = {"rtol": 1e-6} if "refined" in name else {"rtol": 1e-6, "prec": prec}
    f = getattr(fem, name)
    ref = f(*args, p["x0"].clone(), b=p["b"], work=torch.empty(least, dtype=torch.uint8, device="cuda"), **kw)
    asked = _limit(monkeypatch, least)
    got = f(*args, p["x0"].clone(), b=p["b"], **kw)
    assert len(asked) == 2 and asked[1] == least
    assert torch.equal(got[0], ref[0]) and got[1:] == ref[1:]
