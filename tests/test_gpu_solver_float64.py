"""Float64 PCG solves: one form, whatever the workspace holds and whatever the numbers' range.

The solves must give the same bits with a full workspace and with the smallest one that is
accepted, also where the coefficient's spread or flat cells make the iteration long (rounding
differences grow with it until the stopping test ends elsewhere), and must scale with their
data: a factor of a power of two on b and x0 changes no significand as long as the squares of
the residuals stay in float64's normal range. Both comparisons are for equal bits, so there is
no tolerance."""

import numpy as np
import pytest
import torch

import paper_1607_04245_gb300 as fem
import workloads
from gpu_util import to_dev
from test_gpu_solver_forms import _element_form_bytes, _mesh, _problem, _solve, _work_bytes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("physics,cells", [("laplacian", 3000), ("laplacian", 12000), ("laplacian", 30000),
                                           ("elasticity", 3000), ("elasticity", 10000)])
@pytest.mark.parametrize("flat", [1.0, 0.1])
def test_workspace_does_not_change_the_result(physics, cells, flat):
    for seed in range(4):
        m = _mesh(3, cells)
        coords = m.coords.copy()
        coords[2] *= flat
        p = _problem(workloads.Mesh(3, coords, m.conn), physics, "fp64", seed)
        rng = np.random.default_rng(seed + 99)
        p["coef"] = tuple(to_dev(rng.lognormal(0.0, 3.0, c.shape), torch.float64) for c in p["coef"])
        full = _solve(p, _work_bytes(p), max_iter=5000, rtol=1e-8)
        least = _solve(p, _element_form_bytes(p), max_iter=5000, rtol=1e-8)
        assert torch.equal(full[0], least[0]) and full[1:] == least[1:], (seed, full[1:], least[1:])
        assert full[2] <= 1e-8


@pytest.mark.parametrize("physics,dim,cells", [("laplacian", 3, 12000), ("laplacian", 2, 8000), ("laplacian", 3, 60000),
                                               ("elasticity", 3, 6000)])
def test_solves_scale_with_their_data(physics, dim, cells):
    p = _problem(_mesh(dim, cells), physics, "fp64")
    b, x0 = p["b"], p["x0"]
    x, it, res = _solve(p, _work_bytes(p), max_iter=2000, rtol=1e-8)
    assert res <= 1e-8
    for e in (-300, -270, 270, 300):
        p["b"], p["x0"] = b * 2.0 ** e, x0 * 2.0 ** e
        xs, its, ress = _solve(p, _work_bytes(p), max_iter=2000, rtol=1e-8)
        assert (its, ress) == (it, res), e
        assert torch.equal(xs * 2.0 ** -e, x), e
