"""Cell counts that are no multiple of four, and misaligned rows: the float32 forms' kernels
with cells 32 apart and the one-cell kernels, against the general path (any rule, one cell per
thread). The general path is reached with the workloads' rule plus one point of weight zero: the
same integral from the same values, and every sum has one term 0 more, so that the same
arithmetic gives the same result up to the compiler's contraction of products into FMAs.

Tolerance: each entry is a sum of at most 64 products; a contraction saves one rounding of each,
so the largest difference is below 64 * 2^-24 = 4e-6 of the largest entry in float32 and
64 * 2^-53 < 1e-14 in float64, times the condition of the cells' gradients on these meshes
(edges over heights, at most 4): 2e-5 and 5e-14. Outputs lie in a larger buffer whose margins
must stay untouched."""

import numpy as np
import pytest
import torch

import paper_1607_04245_gb300 as fem
import workloads
from gpu_util import to_dev

pytestmark = pytest.mark.gpu

TOL = {"mixed": 2e-5, "fp32": 2e-5, "fp64": 5e-14}
# a warp's 32, 64 and 128 cells and their edges, odd and 2 mod 4, and past one wave of CTAs
SIZES = [1, 2, 3, 31, 33, 62, 63, 65, 127, 129, 255, 257, 1022, 4099, 300001]
MARGIN = 256


def _inputs(dim, C, prec, seed=0):
    n = workloads.meshes.smallest_square_for(C) if dim == 2 else workloads.smallest_cube_for(C)
    mesh = workloads.square_mesh(n, seed=seed) if dim == 2 else workloads.cube_mesh(n, seed=seed)
    mesh = workloads.first_cells(mesh, C)
    rng = np.random.default_rng(seed + C)
    rule = workloads.rule_for_dim(dim)
    nq, V, dt = rule.n_q, mesh.n_verts, fem.value_dtype(prec)
    dev = lambda a: to_dev(a, dt)
    d = {"mesh": (to_dev(mesh.coords, torch.float64), to_dev(mesh.conn, torch.int32)), "V": V, "dim": dim, "C": C,
         "rule": (rule.points, rule.weights), "prec": prec, "u": dev(rng.uniform(-1, 1, V)),
         "U": dev(rng.uniform(-1, 1, (3, V))), "ue": dev(rng.normal(0, 1e-2, (dim, V))),
         "a": dev(rng.lognormal(0, 0.5, V)), "K": dev(rng.lognormal(0, 1, (nq, C))),
         "c": dev(rng.uniform(0.5, 2, (nq, C))), "adj": dev(rng.uniform(-1, 1, (dim + 1, C)))}
    lam, mu = workloads.lame_from_young_poisson(rng.lognormal(0, 0.5, (nq, C)), rng.uniform(0.2, 0.45, (nq, C)))
    d["lam"], d["mu"] = dev(lam), dev(mu)
    return d


def _general(d):
    """The same problem with a fifth (fourth) point of weight zero: the kernels for any rule."""
    p, w = d["rule"]
    g = dict(d, rule=(np.concatenate([p, p[:1]]), np.concatenate([w, [0.0]])))
    for k in ("K", "c", "lam", "mu"):
        g[k] = torch.cat([d[k], d[k][:1]]).contiguous()
    return g


def _out(shape, dt, shift=0):
    """A buffer of `shape` with margins of a sentinel, `shift` elements off 16-byte alignment."""
    n = int(np.prod(shape))
    flat = torch.full((n + 2 * MARGIN,), 7.0, dtype=dt, device="cuda")
    return flat, flat[MARGIN + shift:MARGIN + shift + n].view(shape)


def _run(op, d, out=None):
    m, r, prec, dim = d["mesh"], d["rule"], d["prec"], d["dim"]
    if op == "laplacian":
        return fem.fem_integrate_laplacian(*m, d["u"], d["K"], *r, out=out, prec=prec)
    if op == "fields":
        return fem.fem_integrate_laplacian_fields(*m, d["U"], d["K"], *r, out=out, prec=prec)
    if op == "elasticity":
        return fem.fem_integrate_elasticity(*m, d["ue"], d["lam"], d["mu"], *r, out=out, prec=prec)
    if op == "reaction":
        return fem.fem_integrate_reaction_diffusion(*m, d["u"], d["a"], *r, c=d["c"], drift=0.7, out=out, prec=prec)
    if op == "geometry":
        geom = fem.fem_precompute_geometry(*m, prec=prec)
        return fem.fem_integrate_laplacian_geom(m[1], d["V"], d["u"], d["K"], *r, geom, out=out, prec=prec)
    raise AssertionError(op)


def _shape(op, d):
    nb = d["dim"] + 1
    return {"fields": (3, nb, d["C"]), "elasticity": (nb * d["dim"], d["C"])}.get(op, (nb, d["C"]))


def _close(x, ref, prec):
    scale = float(ref.abs().max())
    err = float((x.double() - ref.double()).abs().max()) / scale
    assert err <= TOL[prec], err


@pytest.mark.parametrize("C", SIZES)
@pytest.mark.parametrize("dim", [2, 3])
@pytest.mark.parametrize("prec", ["mixed", "fp32", "fp64"])
@pytest.mark.parametrize("op", ["laplacian", "fields", "elasticity", "reaction", "geometry"])
def test_ragged_equals_general_path(op, prec, dim, C):
    d = _inputs(dim, C, prec)
    flat, out = _out(_shape(op, d), fem.value_dtype(prec))
    _run(op, d, out)
    ref = _run(op, _general(d))
    _close(out, ref, prec)
    lo, hi = flat[:MARGIN], flat[MARGIN + out.numel():]
    assert bool((lo == 7.0).all()) and bool((hi == 7.0).all())
    assert fem.fem_device_error() == 0


@pytest.mark.parametrize("dim", [2, 3])
@pytest.mark.parametrize("op", ["laplacian", "fields", "elasticity", "reaction", "geometry"])
@pytest.mark.parametrize("prec", ["mixed", "fp64"])
def test_misaligned_rows(op, prec, dim):
    d = _inputs(dim, 4096, prec)
    mis = {}
    for k in ("K", "c", "lam", "mu"):
        _, v = _out(d[k].shape, d[k].dtype, shift=1)
        v.copy_(d[k])
        mis[k] = v
    flat, out = _out(_shape(op, d), fem.value_dtype(prec), shift=1)
    _run(op, dict(d, **mis), out)
    _close(out, _run(op, _general(d)), prec)
    assert bool((flat[:MARGIN] == 7.0).all()) and bool((flat[MARGIN + 1 + out.numel():] == 7.0).all())


@pytest.mark.parametrize("C", [1, 33, 63, 65, 4099, 300001])
@pytest.mark.parametrize("dim", [2, 3])
@pytest.mark.parametrize("prec", ["mixed", "fp32", "fp64"])
def test_ragged_adjoint(prec, dim, C):
    d = _inputs(dim, C, prec)
    g = _general(d)
    ptr, idx = fem.fem_build_node2cell(d["mesh"][1], d["V"])
    nq = dim + 1
    flat, dK = _out((nq, C), fem.value_dtype(prec))
    _, du = fem.fem_adjoint_laplacian(*d["mesh"], d["u"], d["K"], *d["rule"], d["adj"], ptr, idx, dK=dK, prec=prec)
    dKg, dug = fem.fem_adjoint_laplacian(*g["mesh"], g["u"], g["K"], *g["rule"], g["adj"], ptr, idx, prec=prec)
    _close(dK, dKg[:nq], prec)
    _close(du, dug, prec)
    assert bool((flat[:MARGIN] == 7.0).all()) and bool((flat[MARGIN + dK.numel():] == 7.0).all())


@pytest.mark.parametrize("op", ["laplacian", "fields", "elasticity", "reaction"])
@pytest.mark.parametrize("C", [65, 999])
def test_ragged_slivers(op, C):
    """Cells that the mixed form recomputes in float64, at the ends of ragged tiles."""
    d = _inputs(3, C, "mixed")
    d["mesh"][0][2] *= 1e-3
    flat, out = _out(_shape(op, d), torch.float32)
    _run(op, d, out)
    ref = _run(op, _general(d))
    assert float((out - ref).abs().max()) <= TOL["mixed"] * float(ref.abs().max())
    assert bool((flat[:MARGIN] == 7.0).all()) and bool((flat[MARGIN + out.numel():] == 7.0).all())


@pytest.mark.parametrize("where", [0, 31, 62, 63, 64])
def test_ragged_bad_ids_are_reported(where):
    d = _inputs(3, 65, "mixed")
    fem.fem_device_error()
    d["mesh"][1][2, where] = d["V"] + 5
    _run("laplacian", d)
    assert fem.fem_device_error() == -5
