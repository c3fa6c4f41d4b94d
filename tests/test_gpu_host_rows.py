"""Float64 rows in page-locked host memory (chunks = 0): the launch's CTA edges, aligned and ragged
rows, the compiled-in rule and others; the same bits as the device entry."""

import numpy as np
import pytest
import torch

import paper_1607_04245_gb300 as fem
import workloads
from gpu_util import device_arrays
from paper_1607_04245_gb300.host import HostIntegrator

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim", [2, 3])
@pytest.mark.parametrize("n_cells", [1, 63, 64, 65, 4096, 4098, 5183, 70000])
@pytest.mark.parametrize("extra", [0, 1])
def test_same_bits_as_the_device_entry(dim, n_cells, extra):
    n = workloads.meshes.smallest_square_for(n_cells) if dim == 2 else workloads.smallest_cube_for(n_cells)
    mesh = workloads.first_cells(workloads.square_mesh(n) if dim == 2 else workloads.cube_mesh(n), n_cells)
    r = workloads.rule_for_dim(dim)
    rng = np.random.default_rng(n_cells)
    # one more point of its own weight: the rule is read at run time
    rule = workloads.QuadRule(dim, np.concatenate([r.points, np.full((extra, dim), 0.25)]),
                              np.concatenate([r.weights, np.full(extra, 0.1)]))
    case = workloads.Case("laplacian", mesh, rule, rng.uniform(-1, 1, mesh.n_verts),
                          K=rng.lognormal(0, 1, (rule.n_q, n_cells)))
    c, d = device_arrays(case, "fp64")
    ref = fem.fem_integrate_laplacian(d["coords"], d["conn"], d["u"], d["K"], rule.points, rule.weights,
                                      prec="fp64").cpu()
    hi = HostIntegrator("cuda")
    out = hi.laplacian(hi.pinned("coords", c.mesh.coords, torch.float64), hi.pinned("conn", c.mesh.conn, torch.int32),
                       hi.pinned("u", c.u, torch.float64), hi.pinned("K", c.K, torch.float64), rule.points,
                       rule.weights, prec="fp64", chunks=0)
    hi.stream.synchronize()
    assert torch.equal(out, ref) and fem.fem_device_error() == 0
