"""The two forms of the PCG solves against each other: with a full workspace the operator is
assembled and the loop runs in one kernel; one byte less and the solve runs in element form
(which double-float, and float64 in 2D and on larger meshes, always take; for the Laplacian a
full workspace then holds the residual's factors, and the solves with and without them have the
same bits).
Sizes at the edges of what the assembled form distinguishes: slices of 32 rows (V around
multiples of 32), one CTA or several, vector entries in registers or in memory, a matrix that
fits shared memory or does not, and rows at and past the longest that is assembled (64).

Tolerance: after `ITERS` iterations from the same start the two forms' iterates differ by
rounding alone. One application sums at most 64 products of relative error 3 eps, an iteration
adds some ten operations per entry, and the two divisions of an iteration amplify errors of the
inner products by at most a few units at these first iterations: 64 * 3 * ITERS * 10 eps
< 1e4 eps of the largest entry, i.e. 1e4 * 1.1e-16 ~ 1e-12 in float64 and 1e4 * 6e-8 ~ 6e-4 in
float32."""

import numpy as np
import pytest
import torch

import paper_1607_04245_gb300 as fem
import workloads
from gpu_util import to_dev

pytestmark = pytest.mark.gpu

ITERS = 5
TOL = {"fp64": 1e-12, "mixed": 6e-4, "fp32": 6e-4}


def _mesh(dim, cells):
    n = workloads.meshes.smallest_square_for(cells) if dim == 2 else workloads.smallest_cube_for(cells)
    m = workloads.square_mesh(n, jitter=0.2, seed=5) if dim == 2 else workloads.cube_mesh(n, jitter=0.15, seed=5)
    return m if m.n_cells == cells else workloads.first_cells(m, cells)


def _problem(mesh, physics, prec, seed=0):
    rng = np.random.default_rng(seed)
    dim, V = mesh.dim, mesh.n_verts
    rule = workloads.rule_for_dim(dim)
    dt = fem.value_dtype(prec)
    x = mesh.coords
    fixed = np.any((np.abs(x) < 1e-14) | (np.abs(x - x.max(axis=1, keepdims=True)) < 1e-14), axis=0)
    shape = (V,) if physics == "laplacian" else (dim, V)
    x0 = np.where(fixed, rng.uniform(-1, 1, shape), rng.uniform(-0.1, 0.1, shape))
    b = np.where(fixed, 0.0, rng.uniform(-1, 1, shape) / V)
    if physics == "laplacian":
        coef = (rng.lognormal(0.0, 1.0, (rule.n_q, mesh.n_cells)),)
    else:
        coef = workloads.lame_from_young_poisson(rng.lognormal(0.0, 0.5, (rule.n_q, mesh.n_cells)),
                                                 rng.uniform(0.2, 0.45, (rule.n_q, mesh.n_cells)))
    coords, conn = to_dev(mesh.coords, torch.float64), to_dev(mesh.conn, torch.int32)
    ptr, idx = fem.fem_build_node2cell(conn, V)
    return {"mesh": (coords, conn), "coef": tuple(to_dev(c, dt) for c in coef), "rule": (rule.points, rule.weights),
            "lists": (ptr, idx, to_dev(fixed.astype(np.uint8), torch.uint8)), "x0": to_dev(x0, dt),
            "b": to_dev(b, dt), "dim": dim, "V": V, "C": mesh.n_cells, "prec": prec, "physics": physics}


def _work_bytes(p):
    f = "fem_pcg_work_bytes" if p["physics"] == "laplacian" else "fem_pcg_elasticity_work_bytes"
    return int(getattr(fem.binding.lib(), f)(p["dim"], p["C"], p["V"], fem.precision(p["prec"])))


def _solve(p, nbytes, max_iter=ITERS, rtol=0.0, b="b"):
    f = fem.fem_pcg_laplacian if p["physics"] == "laplacian" else fem.fem_pcg_elasticity
    return f(*p["mesh"], *p["coef"], *p["rule"], *p["lists"], p["x0"].clone(), b=p[b] if b else None, max_iter=max_iter,
             rtol=rtol, work=torch.empty(nbytes, dtype=torch.uint8, device="cuda"), prec=p["prec"])


def _element_form_bytes(p):
    """The workspace that holds the element vectors, six vectors, the partial sums and the scalars."""
    a256 = lambda n: (n + 255) // 256 * 256
    vs = 8 if p["prec"] in ("fp64", "fp64_df") else 4
    nc = 1 if p["physics"] == "laplacian" else p["dim"]
    return a256((p["dim"] + 1) * nc * p["C"] * vs) + 6 * a256(nc * p["V"] * vs) + a256(3 * 1024 * 8) + 256


def _compare(p, **kw):
    full = _work_bytes(p)
    assert full > _element_form_bytes(p)
    xa, ia, ra = _solve(p, full, **kw)
    xe, ie, re = _solve(p, full - 1, **kw)
    xm, im, rm = _solve(p, _element_form_bytes(p), **kw)
    assert torch.equal(xe, xm) and (ie, re) == (im, rm)  # the smaller workspace is enough for the element form
    # CG ends after as many iterations as there are unknowns: then rounding alone says when r.r is 0
    unknowns = int((p["lists"][2] == 0).sum()) * (1 if p["physics"] == "laplacian" else p["dim"])
    assert ia == ie or unknowns <= ITERS
    scale = float(xe.abs().max())
    err = float((xa.double() - xe.double()).abs().max()) / scale
    assert err <= TOL[p["prec"]], err
    assert fem.fem_device_error() == 0
    again = _solve(p, full, **kw)[0]
    assert torch.equal(xa, again)
    fixed = p["lists"][2].bool()
    assert torch.equal(xa[..., fixed], p["x0"][..., fixed])  # Dirichlet values are kept


# cells: tiny meshes; slices of 32 rows at their edges; one CTA (512 rows) and more; a few
# slices per CTA; ragged counts
@pytest.mark.parametrize("prec", ["fp64", "fp32", "mixed"])
@pytest.mark.parametrize("physics,dim,cells", [
    ("laplacian", 2, 2), ("laplacian", 2, 50), ("laplacian", 2, 961), ("laplacian", 2, 2047), ("laplacian", 2, 30011),
    ("laplacian", 3, 6), ("laplacian", 3, 163), ("laplacian", 3, 2058), ("laplacian", 3, 20577),
    ("elasticity", 2, 3), ("elasticity", 2, 1117), ("elasticity", 2, 25001),
    ("elasticity", 3, 7), ("elasticity", 3, 3001), ("elasticity", 3, 24001)])
def test_assembled_equals_element_form(physics, dim, cells, prec):
    if prec == "fp64" and (dim == 2 or (physics == "elasticity" and cells * dim > 30000)):
        pytest.skip("float64 has the element form alone")
    _compare(_problem(_mesh(dim, cells), physics, prec))


@pytest.mark.parametrize("physics,dim,prec", [("elasticity", 2, "fp64"), ("elasticity", 3, "fp64_df")])
def test_element_form_alone(physics, dim, prec):
    p = _problem(_mesh(dim, 2001), physics, prec)
    assert _work_bytes(p) == _element_form_bytes(p)
    x, it, _ = _solve(p, _work_bytes(p))
    assert it == ITERS and bool(torch.isfinite(x).all())
    with pytest.raises(fem.FemError):
        _solve(p, _work_bytes(p) - 1)


# every SM with several slices per warp: entries still in registers (64^3 x 6 tets), and past that
@pytest.mark.parametrize("physics,dim,cells", [("laplacian", 3, 1572864), ("laplacian", 2, 721801),
                                               ("elasticity", 2, 220001), ("elasticity", 3, 584001)])
def test_large_meshes(physics, dim, cells):
    _compare(_problem(_mesh(dim, cells), physics, "mixed"))


@pytest.mark.parametrize("physics,cells", [("laplacian", 30000), ("elasticity", 10000)])
def test_float64_in_memory(physics, cells):
    """Vertices in no cell: more rows than stay in registers."""
    m = _mesh(3, cells)
    coords = np.concatenate([m.coords, np.zeros((3, 700001))], axis=1)
    _compare(_problem(workloads.Mesh(3, coords, m.conn), physics, "fp64"))


# the factored residual against the residual kernel: the same bits. One warp of cells and its
# edges, ragged counts, either side of the float64 form's assembled sizes and of its kernel's
# integer columns (60,000 cells)
@pytest.mark.parametrize("prec", ["fp64", "fp64_df"])
@pytest.mark.parametrize("dim,cells", [(2, 2), (2, 31), (2, 33), (2, 2047), (2, 30011), (2, 60002), (3, 7), (3, 129),
                                       (3, 3001), (3, 30000), (3, 30001), (3, 60003), (3, 150000)])
def test_factored_solve_bit_for_bit(dim, cells, prec):
    if prec == "fp64" and dim == 3 and cells <= 30000:
        pytest.skip("assembled")
    p = _problem(_mesh(dim, cells), "laplacian", prec)
    full = _work_bytes(p)
    assert full == _element_form_bytes(p) + (dim * dim + 1) * cells * 8 // 256 * 256 + (
        256 if (dim * dim + 1) * cells * 8 % 256 else 0)
    for kw in ({}, {"max_iter": 60, "rtol": 1e-10}):
        xf, it, res = _solve(p, full, **kw)
        xe, ie, re = _solve(p, full - 1, **kw)
        assert torch.equal(xf, xe) and (it, res) == (ie, re)
    with pytest.raises(fem.FemError):
        _solve(p, _element_form_bytes(p) - 1)


def test_no_load_and_no_iterations():
    p = _problem(_mesh(3, 2058), "laplacian", "fp64")
    _compare(p, b=None)
    x, it, _ = _solve(p, _work_bytes(p), max_iter=0)
    assert it == 0 and torch.equal(x, p["x0"])


def _fan(k):
    """A disk of k triangles around vertex 0: row 0 has k neighbours."""
    t = 2 * np.pi * np.arange(k) / k
    coords = np.concatenate([[[0.01], [0.02]], np.stack([np.cos(t), np.sin(t)])], axis=1)
    i = np.arange(k)
    conn = np.stack([np.zeros(k), 1 + i, 1 + (i + 1) % k]).astype(np.int32)
    return workloads.Mesh(2, np.ascontiguousarray(coords), conn)


@pytest.mark.parametrize("physics", ["laplacian", "elasticity"])
@pytest.mark.parametrize("k", [63, 64, 65, 200])
def test_long_rows(k, physics):
    """Rows of up to 64 neighbours are assembled; a mesh with a longer one is solved in element form."""
    mesh = _fan(k)
    p = _problem(mesh, physics, "mixed")
    fixed = np.zeros(mesh.n_verts, dtype=np.uint8)
    fixed[1:4] = 1
    p["lists"] = (*p["lists"][:2], to_dev(fixed, torch.uint8))
    full = _work_bytes(p)
    xa, ia, _ = _solve(p, full)
    xe, ie, _ = _solve(p, full - 1)
    assert ia == ie
    assert float((xa - xe).abs().max()) <= TOL["mixed"] * float(xe.abs().max())
    if k > 64:
        assert torch.equal(xa, xe)


def test_slivers_are_assembled_in_float64():
    """Cells that the mixed form's shape test rejects enter the matrix through float64."""
    mesh = _mesh(3, 3000)
    coords = mesh.coords.copy()
    coords[2] *= 1e-3  # flat cells: every one fails the shape test
    p = _problem(workloads.Mesh(3, coords, mesh.conn), "laplacian", "mixed")
    _compare(p)


def test_bad_mesh_is_reported():
    mesh = _mesh(3, 3000)
    conn = mesh.conn.copy()
    conn[1, 17] = conn[2, 17]  # a repeated vertex
    p = _problem(workloads.Mesh(3, mesh.coords, conn), "laplacian", "fp64")
    _solve(p, _work_bytes(p))
    assert fem.fem_device_error() == -5
