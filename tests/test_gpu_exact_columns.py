"""Float64 kernels over many cells take the Jacobian columns by integer operations
(csrc/fem_cell.cuh, exact_differences) and over few cells by subtraction. Both give the same bits, so
a call over all cells and calls over 15,000 cells each must agree bit for bit: no tolerance."""

import numpy as np
import pytest
import torch

import paper_1607_04245_gb300 as fem
import workloads
from gpu_util import to_dev

pytestmark = pytest.mark.gpu

PART, PARTS = 15000, 5  # 15,000 cells: subtraction; 75,000: integer operations


def _coords(kind, base, rng):
    X = base.copy()
    if kind == "far":  # all of one binade, few bits left for the edges
        X = X + 1e6
    elif kind == "centred":  # both signs in a cell, many binades, exact zeros
        X = X - 0.5
    elif kind == "binades":  # neighbouring vertices up to 40 binades apart
        X = np.ldexp(X, rng.integers(-20, 20, X.shape))
    elif kind == "edge":  # the 9 and 10 binade border, -0, subnormals and the ends of the range
        pick = rng.integers(0, 8, X.shape)
        vals = [0.0, -0.0, 2.0 ** -9, -(2.0 ** -10), 1.0, np.nextafter(1.0, 2.0), -np.nextafter(2.0, 1.0), 5e-324]
        X = np.where(rng.uniform(size=X.shape) < 0.5, np.array(vals)[pick], X)
    elif kind == "tiny":
        X = X * 1e-60
    return X


@pytest.mark.parametrize("kind", ["plain", "far", "centred", "binades", "edge", "tiny"])
@pytest.mark.parametrize("dim", [2, 3])
def test_columns_bit_for_bit(dim, kind):
    C = PART * PARTS
    n = workloads.meshes.smallest_square_for(C) if dim == 2 else workloads.smallest_cube_for(C)
    mesh = workloads.first_cells(workloads.square_mesh(n) if dim == 2 else workloads.cube_mesh(n), C)
    rng = np.random.default_rng(dim)
    coords = to_dev(_coords(kind, mesh.coords, rng), torch.float64)
    conn = to_dev(mesh.conn, torch.int32)
    rule = workloads.rule_for_dim(dim)
    pw, nq, V = (rule.points, rule.weights), rule.n_q, mesh.n_verts
    dev = lambda a: to_dev(a, torch.float64)
    u, U, ue, a = dev(rng.uniform(-1, 1, V)), dev(rng.uniform(-1, 1, (3, V))), dev(rng.uniform(-1, 1, (dim, V))), dev(
        rng.lognormal(0, 0.5, V))
    K, M, adj = dev(rng.lognormal(0, 1, (nq, C))), dev(rng.lognormal(0, 1, (nq, C))), dev(rng.uniform(-1, 1, (dim + 1, C)))

    def calls(s):
        m, k, mu, ad = (coords, conn[:, s].contiguous()), K[:, s].contiguous(), M[:, s].contiguous(), adj[:, s].contiguous()
        ptr, idx = fem.fem_build_node2cell(m[1], V)
        return [fem.fem_integrate_laplacian(*m, u, k, *pw, prec="fp64"),
                fem.fem_integrate_laplacian_fields(*m, U, k, *pw, prec="fp64").reshape(3 * (dim + 1), -1),
                fem.fem_integrate_elasticity(*m, ue, k, mu, *pw, prec="fp64").reshape(dim * (dim + 1), -1),
                fem.fem_integrate_reaction_diffusion(*m, u, a, *pw, c=k, drift=0.7, prec="fp64"),
                fem.fem_adjoint_laplacian(*m, u, k, *pw, ad, ptr, idx, prec="fp64")[0]]

    whole = calls(slice(0, C))
    for p in range(PARTS):
        s = slice(p * PART, (p + 1) * PART)
        for x, y in zip(whole, calls(s)):
            xs = x[:, s]
            same = xs.contiguous().view(torch.int64) == y.contiguous().view(torch.int64)
            assert bool((same | (xs.isnan() & y.isnan())).all())
    fem.fem_device_error()  # cells of no volume are reported, here as anywhere


@pytest.mark.parametrize("C", [33, 75000])
@pytest.mark.parametrize("constant", [False, True])
@pytest.mark.parametrize("dim", [2, 3])
def test_first_row_is_minus_the_sum(dim, constant, C):
    """r_0 = -(0 + r_1 + ... + r_d) bit for bit, the signs of zeros of a constant field included: its
    first and last operation run on the integer pipes."""
    n = workloads.meshes.smallest_square_for(C) if dim == 2 else workloads.smallest_cube_for(C)
    mesh = workloads.first_cells(workloads.square_mesh(n) if dim == 2 else workloads.cube_mesh(n), C)
    rng = np.random.default_rng(C)
    rule, V = workloads.rule_for_dim(dim), mesh.n_verts
    dev = lambda a: to_dev(a, torch.float64)
    m, pw = (dev(mesh.coords), to_dev(mesh.conn, torch.int32)), (rule.points, rule.weights)
    field = lambda *s: dev(np.full(s, 0.75) if constant else rng.uniform(-1, 1, s))
    K, M = dev(rng.lognormal(0, 1, (rule.n_q, C))), dev(rng.lognormal(0, 1, (rule.n_q, C)))
    geom = fem.fem_precompute_geometry(*m, prec="fp64")
    bits = lambda t: t.contiguous().view(torch.int64)
    for r in (fem.fem_integrate_laplacian(*m, field(V), K, *pw, prec="fp64"),
              fem.fem_integrate_laplacian_fields(*m, field(3, V), K, *pw, prec="fp64")[1],
              fem.fem_integrate_laplacian_geom(m[1], V, field(V), K, *pw, geom, prec="fp64")):
        total = torch.zeros_like(r[0])
        for j in range(dim):
            total = total + r[j + 1]
        assert torch.equal(bits(r[0]), bits(-total))
    e = fem.fem_integrate_elasticity(*m, field(dim, V), K, M, *pw, prec="fp64").view(dim + 1, dim, C)
    total = torch.zeros_like(e[0])
    for j in range(dim):
        total = total - e[j + 1]
    assert torch.equal(bits(e[0]), bits(total))
