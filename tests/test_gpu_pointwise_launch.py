"""Launch shapes of the run-time compiled kernel: physics that needs local memory and registers
against the same physics without (another CTA size), and cell counts around
its CTAs' edges in both precisions against the built-in Laplacian. Tolerance: the two kernels sum
the same 4 (3) points in another order, at most 64 products of relative error eps per entry."""

import numpy as np
import pytest
import torch

import paper_1607_04245_gb300 as fem
import workloads
from gpu_util import to_dev

pytestmark = pytest.mark.gpu

TOL = {"mixed": 64 * 2.0 ** -23, "fp64": 64 * 2.0 ** -52}
PLAIN = "for (int i = 0; i < DIM; ++i) f1[i] = a[0] * grad_u[i];"
# a table indexed at run time; it contributes 0
HEAVY = ("T t[40];\nfor (int k = 0; k < 40; ++k) t[k] = u[0] + T(k);\n"
         "int at = (int)(u[0] * T(1000)); at = at < 0 ? -at : at;\nt[at % 40] += x[0];\n"
         "T s = T(0);\nfor (int k = 0; k < 40; ++k) s += t[(at + 7 * k) % 40];\n"
         "for (int i = 0; i < DIM; ++i) f1[i] = a[0] * grad_u[i] + (s - s);")


def _inputs(dim, C, prec):
    n = workloads.meshes.smallest_square_for(C) if dim == 2 else workloads.smallest_cube_for(C)
    mesh = workloads.first_cells(workloads.square_mesh(n) if dim == 2 else workloads.cube_mesh(n), C)
    rng = np.random.default_rng(C)
    rule, dt = workloads.rule_for_dim(dim), fem.value_dtype(prec)
    return (to_dev(mesh.coords, torch.float64), to_dev(mesh.conn, torch.int32),
            to_dev(rng.uniform(-1, 1, mesh.n_verts), dt), to_dev(rng.lognormal(0, 1, (rule.n_q, C)), dt),
            rule.points, rule.weights)


@pytest.mark.parametrize("dim", [2, 3])
@pytest.mark.parametrize("prec", ["mixed", "fp64"])
@pytest.mark.parametrize("C", [1, 63, 64, 65, 127, 129, 4097, 200003])
def test_edges(dim, prec, C):
    x, conn, u, K, qp, qw = _inputs(dim, C, prec)
    got = fem.fem_integrate_pointwise(x, conn, u, K[None], qp, qw, f1=PLAIN, prec=prec)
    ref = fem.fem_integrate_laplacian(x, conn, u, K, qp, qw, prec=prec)
    assert float((got - ref).abs().max()) <= TOL[prec] * float(ref.abs().max())


@pytest.mark.parametrize("dim", [2, 3])
@pytest.mark.parametrize("prec", ["mixed", "fp64"])
def test_physics_in_local_memory(dim, prec):
    x, conn, u, K, qp, qw = _inputs(dim, 30001, prec)
    a = fem.fem_integrate_pointwise(x, conn, u, K[None], qp, qw, f1=HEAVY, prec=prec)
    b = fem.fem_integrate_pointwise(x, conn, u, K[None], qp, qw, f1=PLAIN, prec=prec)
    assert float((a - b).abs().max()) <= TOL[prec] * float(b.abs().max())
