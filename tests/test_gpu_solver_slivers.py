"""Mixed-form solves on meshes with badly shaped cells (below the shape threshold of the mixed
form): such cells are applied in float64 in every iteration, whatever the workspace. The
residual kernels do that, so a solve with a full workspace must give the bits of one with the
smallest workspace that is accepted (which runs the residual kernels); no tolerance."""

import numpy as np
import pytest
import torch

import paper_1607_04245_gb300 as fem
import workloads
from test_gpu_solver_forms import _element_form_bytes, _mesh, _problem, _solve, _work_bytes

pytestmark = pytest.mark.gpu


def _shape(coords, conn):
    """Hadamard ratio of every cell: |det| over the product of the edge lengths from vertex 0."""
    x = coords[:, conn]
    e = np.moveaxis(x[:, 1:] - x[:, :1], -1, 0)  # [C][dim][j]
    return np.abs(np.linalg.det(e)) / np.prod(np.linalg.norm(e, axis=1), axis=1)


def _sliver_mesh(dim, cells, squeeze):
    """squeeze "all": the mesh flat, most cells with it; "one": one vertex moved next to the opposite face of a cell."""
    m = _mesh(dim, cells)
    coords = m.coords.copy()
    if squeeze == "all":
        coords[dim - 1] *= 1e-3
    else:
        c = cells // 2
        v, rest = m.conn[0, c], m.conn[1:, c]
        centre = coords[:, rest].mean(axis=1)
        coords[:, v] = centre + 0.005 * (coords[:, v] - centre)
    bad = _shape(coords, m.conn) < fem.binding.lib().fem_get_mixed_threshold()
    assert bad.sum() > cells // 2 if squeeze == "all" else 1 <= bad.sum() <= 40
    return workloads.Mesh(dim, coords, m.conn)


@pytest.mark.parametrize("physics,dim,cells", [("laplacian", 2, 2047), ("laplacian", 3, 3001), ("laplacian", 3, 40001),
                                               ("elasticity", 2, 1117), ("elasticity", 3, 3001)])
@pytest.mark.parametrize("squeeze", ["one", "all"])
def test_same_bits_as_the_residual_kernels(physics, dim, cells, squeeze):
    p = _problem(_sliver_mesh(dim, cells, squeeze), physics, "mixed")
    full = _solve(p, _work_bytes(p), max_iter=30, rtol=1e-6)
    least = _solve(p, _element_form_bytes(p), max_iter=30, rtol=1e-6)
    assert full[1:] == least[1:] and torch.equal(full[0], least[0])
    assert fem.fem_device_error() == 0


@pytest.mark.parametrize("physics", ["laplacian", "elasticity"])
def test_refined_corrections(physics):
    p = _problem(_sliver_mesh(3, 3001, "one"), physics, "fp64")
    f = fem.fem_pcg_laplacian_refined if physics == "laplacian" else fem.fem_pcg_elasticity_refined
    q = "fem_pcg_refined_work_bytes" if physics == "laplacian" else "fem_pcg_elasticity_refined_work_bytes"
    need = int(getattr(fem.binding.lib(), q)(3, p["C"], p["V"], len(p["rule"][1])))
    got = [f(*p["mesh"], *p["coef"], *p["rule"], *p["lists"], p["x0"].clone(), b=p["b"], rtol=1e-10,
             work=torch.empty(n, dtype=torch.uint8, device="cuda")) for n in (need, need - 1)]
    assert got[0][1:] == got[1][1:] and torch.equal(got[0][0], got[1][0])
    assert got[0][3] <= 1e-10
