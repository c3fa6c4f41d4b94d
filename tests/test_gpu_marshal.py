"""The native marshalling module against the binding's own Python path: the same results bit
for bit, the same errors. The Python path is reached by giving the quadrature weights as a list,
which the module leaves to it."""

import numpy as np
import pytest
import torch

import paper_1607_04245_gb300 as fem
import workloads
from gpu_util import to_dev

pytestmark = pytest.mark.gpu

F1 = "for (int i = 0; i < DIM; ++i) f1[i] = (T(1) + u[0] * u[0]) * grad_u[i];"


def _inputs(dim, prec, C=999):
    n = workloads.meshes.smallest_square_for(C) if dim == 2 else workloads.smallest_cube_for(C)
    mesh = workloads.square_mesh(n) if dim == 2 else workloads.cube_mesh(n)
    mesh = workloads.first_cells(mesh, C)
    rng = np.random.default_rng(dim)
    rule = workloads.rule_for_dim(dim)
    dt = fem.value_dtype(prec)
    V, nq = mesh.n_verts, rule.n_q
    d = {k: to_dev(rng.uniform(0.5, 1.5, s), dt) for k, s in
         {"u": (V,), "U": (2, V), "ue": (dim, V), "a": (V,), "K": (nq, C), "lam": (nq, C), "mu": (nq, C),
          "adj": (dim + 1, C), "elem": ((dim + 1) * dim, C)}.items()}
    d.update(coords=to_dev(mesh.coords, torch.float64), conn=to_dev(mesh.conn, torch.int32), V=V, C=C, dim=dim,
             qp=rule.points, qw=rule.weights, prec=prec)
    d["ptr"], d["idx"] = fem.fem_build_node2cell(d["conn"], V)
    return d


def _calls(d):
    """name -> call(keyword replacements): each entry point that goes through the module."""
    m = lambda k: (k.get("coords", d["coords"]), k.get("conn", d["conn"]))
    q = lambda k: (k.get("qp", d["qp"]), k.get("qw", d["qw"]))
    o = lambda k: {"prec": k.get("prec", d["prec"]), "out": k.get("out"), "stream": k.get("stream")}
    n = lambda k: {"prec": k.get("prec", d["prec"]), "stream": k.get("stream")}
    g = lambda k, name: k.get(name, d[name])
    calls = {
        "laplacian": lambda **k: fem.fem_integrate_laplacian(*m(k), g(k, "u"), g(k, "K"), *q(k), **o(k)),
        "fields": lambda **k: fem.fem_integrate_laplacian_fields(*m(k), g(k, "U"), g(k, "K"), *q(k), **o(k)),
        "elasticity": lambda **k: fem.fem_integrate_elasticity(*m(k), g(k, "ue"), g(k, "lam"), g(k, "mu"), *q(k), **o(k)),
        "reaction": lambda **k: fem.fem_integrate_reaction_diffusion(*m(k), g(k, "u"), g(k, "a"), *q(k), c=g(k, "K"),
                                                                     drift=0.5, **o(k)),
        "pointwise": lambda **k: fem.fem_integrate_pointwise(*m(k), g(k, "u"), None, *q(k), f1=F1, **o(k)),
        "adjoint": lambda **k: fem.fem_adjoint_laplacian(*m(k), g(k, "u"), g(k, "K"), *q(k), g(k, "adj"), g(k, "ptr"),
                                                         g(k, "idx"), **n(k)),
    }
    if d["prec"] != "fp64_df":
        geom = fem.fem_precompute_geometry(d["coords"], d["conn"], prec=d["prec"])
        calls["geometry"] = lambda **k: fem.fem_integrate_laplacian_geom(k.get("conn", d["conn"]), d["V"], g(k, "u"),
                                                                         g(k, "K"), *q(k), geom, **o(k))
    else:
        for name in ("fields", "reaction", "pointwise"):
            del calls[name]
    return calls


def _flat(r):
    return list(r) if isinstance(r, tuple) else [r]


@pytest.mark.parametrize("dim", [2, 3])
@pytest.mark.parametrize("prec", ["mixed", "fp32", "fp64", "fp64_df"])
def test_equals_python_path(dim, prec):
    d = _inputs(dim, prec)
    calls = _calls(d)
    if prec == "fp32":
        del calls["pointwise"]
    for name, call in calls.items():
        fast, slow = call(), call(qw=list(d["qw"]))
        for a, b in zip(_flat(fast), _flat(slow)):
            assert torch.equal(a, b) and a.dtype == b.dtype, name
        if name != "adjoint":
            buf = torch.full_like(fast, 3.0)
            assert call(out=buf) is buf and torch.equal(buf, fast), name
        for stream in (torch.cuda.current_stream(), torch.cuda.current_stream().cuda_stream):
            assert torch.equal(_flat(call(stream=stream))[0], _flat(fast)[0]), name
        code = {"fp64": 0, "mixed": 1, "fp32": 2, "fp64_df": 3}[prec]
        assert torch.equal(_flat(call(prec=code))[0], _flat(fast)[0]), name


@pytest.mark.parametrize("prec", ["mixed", "fp64"])
def test_lists_and_gather(prec):
    d = _inputs(3, prec)
    work = torch.empty(fem.binding.lib().fem_node2cell_work_size(d["V"]), dtype=torch.int32, device="cuda")
    ptr, idx = fem.fem_build_node2cell(d["conn"], d["V"], work=work.view(1, -1))  # the Python path
    assert torch.equal(ptr, d["ptr"]) and torch.equal(idx, d["idx"])
    a = fem.fem_gather_nodes(d["elem"], ptr, idx, d["V"], 3, prec=prec)
    b = fem.fem_gather_nodes(d["elem"], ptr, idx, np.int64(d["V"]), 3, prec=prec)  # the Python path
    assert torch.equal(a, b)


def test_runs_on_the_current_stream():
    d = _inputs(3, "mixed")
    ref = _calls(d)["laplacian"]()
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    g = torch.cuda.CUDAGraph()
    out = torch.empty_like(ref)
    torch.cuda.synchronize()
    with torch.cuda.graph(g, stream=s):  # captured: the call went to the capturing stream
        _calls(d)["laplacian"](out=out)
    out.zero_()
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(out, ref)


@pytest.mark.parametrize("bad", ["dtype", "shape", "cpu", "stride", "none", "int64 conn", "rule", "points", "precision",
                                 "weights", "out", "number"])
def test_refusals_are_those_of_the_python_path(bad):
    d = _inputs(3, "mixed")
    replace = {
        "dtype": {"u": d["u"].double()}, "shape": {"u": d["u"][:-1]}, "cpu": {"u": d["u"].cpu()},
        "stride": {"K": torch.stack([d["K"], d["K"]], dim=2)[:, :, 0]}, "none": {"u": None},
        "int64 conn": {"conn": d["conn"].long()}, "rule": {"qw": d["qw"][:3]}, "points": {"qp": d["qp"][:, :2]},
        "precision": {"prec": "half"}, "weights": {"qw": np.full(4, np.nan)},
        "out": {"out": torch.empty((4, 998), dtype=torch.float32, device="cuda")}, "number": {"coords": 3.0},
    }[bad]
    call = _calls(d)["laplacian"]
    seen = []
    for extra in ({}, {"qw": list(replace.get("qw", d["qw"]))}):
        with pytest.raises((ValueError, KeyError, AttributeError, TypeError, fem.FemError)) as e:
            call(**{**replace, **extra})
        seen.append((e.type, str(e.value)))
    assert seen[0] == seen[1]


def test_float32_tables_and_tensors_are_converted():
    d = _inputs(3, "mixed")
    ref = _calls(d)["laplacian"]()
    got = _calls(d)["laplacian"](qw=torch.from_numpy(d["qw"]), qp=None)
    assert torch.equal(got, ref)
    got = _calls(d)["laplacian"](qw=np.asfortranarray(d["qw"]), qp=np.asfortranarray(d["qp"]))
    assert torch.equal(got, ref)
