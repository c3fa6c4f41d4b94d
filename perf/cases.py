"""Timed cases of the framework's public entry points.

A case is a dict of plain values; `kind` names the call:

  residual    fem_integrate_laplacian: the element residual of the variable-coefficient Laplacian
  elasticity  fem_integrate_elasticity: the element residual of linear elasticity
  train       autograd.laplacian_residual, forward and backward: residual, dL/du, dL/dK
  request     fem_build_node2cell, then fem_adjoint_laplacian: an adjoint request on a mesh seen once
  reaction    fem_integrate_reaction_diffusion: P1 coefficient, reaction and grad a terms
  pointwise   fem_integrate_pointwise: kappa(u, x) grad u given as source text
  assembled   fem_integrate_elasticity, then fem_gather_nodes: the assembled nonlinear residual
  solve       fem_pcg_laplacian: the assembled system with Dirichlet values, to 1e-8
  refined     fem_pcg_elasticity_refined: elasticity by iterative refinement, to 1e-12

with `dim` (2 or 3), `cells` and `prec` (for `refined` the precision of the true residual).
Meshes are the first `cells` cells of a jittered structured grid of the unit square or cube
in lexicographic order; coefficients, fields and quadrature rules follow the recipes of
workloads/cases.py, drawn with torch on the device. Cell counts that are no multiple of four
are as ordinary as the others: a mesh generator returns whatever count it returns.
"""

from __future__ import annotations

import math

import torch

import paper_1607_04245_gb300 as fem
from paper_1607_04245_gb300.autograd import DeviceMesh, laplacian_residual

F64 = torch.float64

# quadrature rules of degree 2 (3 points on triangles, 4 on tetrahedra)
_A, _B = (5.0 - math.sqrt(5.0)) / 20.0, (5.0 + 3.0 * math.sqrt(5.0)) / 20.0
RULES = {
    2: ([[1 / 6, 1 / 6], [2 / 3, 1 / 6], [1 / 6, 2 / 3]], [1 / 6] * 3),
    3: ([[_A, _A, _A], [_B, _A, _A], [_A, _B, _A], [_A, _A, _B]], [1 / 24] * 4),
}
DRIFT = 1.0
# kappa(u, x) = (p0 + p1 u + p2 u^2)(1 + p3 (x_0 + 2 x_1 + 3 x_2)), times grad u
P = (1.3, -0.7, 0.45, 0.35)
NONLINEAR_F1 = (
    "T s = T(0);\nfor (int i = 0; i < DIM; ++i) s += T(i + 1) * x[i];\n"
    f"const T kappa = (T({P[0]}) + T({P[1]}) * u[0] + T({P[2]}) * u[0] * u[0]) * (T(1) + T({P[3]}) * s);\n"
    "for (int i = 0; i < DIM; ++i) f1[i] = kappa * grad_u[i];")


def listed():
    return [
        # one evaluation on a small mesh: the call's latency (the paper's 2D configuration, 64 x 64 squares)
        {"name": "residual2d_fp64_small", "kind": "residual", "dim": 2, "cells": 8192, "prec": "fp64"},
        # the benchmark's headline: one residual on 64^3 x 6 tets
        {"name": "residual3d_mixed", "kind": "residual", "dim": 3, "cells": 1572864, "prec": "mixed"},
        # the same call on a mesh of odd size, the upper end of the serving mix
        {"name": "residual3d_mixed_odd", "kind": "residual", "dim": 3, "cells": 999999, "prec": "mixed"},
        # a training step on the coefficient and the field in the default precision
        {"name": "train3d_fp64", "kind": "train", "dim": 3, "cells": 1572864, "prec": "fp64"},
        # the largest mesh of the workloads
        {"name": "elasticity2d_mixed", "kind": "elasticity", "dim": 2, "cells": 4194304, "prec": "mixed"},
        # float64-class accuracy on the float32 pipe
        {"name": "elasticity3d_df", "kind": "elasticity", "dim": 3, "cells": 2097152, "prec": "fp64_df"},
        # a served adjoint request: the mesh arrives with it, so its vertex lists are built first
        {"name": "request3d_mixed", "kind": "request", "dim": 3, "cells": 524286, "prec": "mixed"},
        # one step of a reaction-diffusion integrator on a mesh of odd size
        {"name": "reaction3d_mixed_odd", "kind": "reaction", "dim": 3, "cells": 786431, "prec": "mixed"},
        # user physics compiled at run time
        {"name": "pointwise3d_mixed", "kind": "pointwise", "dim": 3, "cells": 1572864, "prec": "mixed"},
        # the assembled residual a Newton or time stepper evaluates
        {"name": "assembled3d_mixed", "kind": "assembled", "dim": 3, "cells": 1000002, "prec": "mixed"},
        # a linear solve in the default precision on the headline mesh
        {"name": "solve3d_fp64", "kind": "solve", "dim": 3, "cells": 1572864, "prec": "fp64"},
        # a linear solve by mixed-precision refinement
        {"name": "refined3d_df", "kind": "refined", "dim": 3, "cells": 511104, "prec": "fp64_df"},
    ]


# per kind: the precisions in use and the largest drawn mesh (2D, 3D)
RANGES = {
    "residual": (("mixed", "fp64", "fp64_df", "mixed"), (4194304, 2097152)),
    "elasticity": (("mixed", "fp64", "fp64_df", "mixed"), (4194304, 2097152)),
    "train": (("mixed", "fp64"), (2000000, 1572864)),
    "request": (("mixed", "fp64"), (1000000, 1000000)),
    "reaction": (("mixed", "fp64", "mixed"), (2000000, 1572864)),
    "pointwise": (("mixed", "fp64", "mixed"), (2000000, 1572864)),
    "assembled": (("mixed", "fp64", "fp64_df", "mixed"), (2000000, 1572864)),
    "solve": (("fp64", "fp64_df"), (60000, 1200000)),
    "refined": (("fp64", "fp64_df"), (15000, 400000)),
}


def draw(rng):
    kind = rng.choice(sorted(RANGES))
    precs, most = RANGES[kind]
    dim = rng.choice((2, 3, 3))
    cells = int(round(math.exp(rng.uniform(math.log(1000), math.log(most[dim - 2])))))
    return {"kind": kind, "dim": dim, "cells": cells, "prec": rng.choice(precs)}


# ------------------------------------------------------------------ inputs


def _grid(dim, cells):
    n = max(1, int(round((cells / (2.0 if dim == 2 else 6.0)) ** (1.0 / dim))) - 1)
    while (2 * n * n if dim == 2 else 6 * n ** 3) < cells:
        n += 1
    return n


def _mesh(dim, cells, gen, dev):
    """coords [dim][V] float64, conn [dim+1][cells] int32, boundary mask [V]."""
    n = _grid(dim, cells)
    m = n + 1
    h = 1.0 / n
    ids = torch.arange(m ** dim, device=dev)
    ijk = [(ids // m ** k) % m for k in range(dim)]
    interior = torch.ones_like(ids, dtype=torch.bool)
    for c in ijk:
        interior &= (c > 0) & (c < n)
    jitter = 0.2 if dim == 2 else 0.15
    move = (torch.rand((dim, m ** dim), generator=gen, device=dev, dtype=F64) * 2 - 1) * (jitter * h)
    coords = torch.stack([c.to(F64) * h for c in ijk]) + move * interior
    per = 2 if dim == 2 else 6
    cell = torch.arange(cells, device=dev)
    box, part = cell // per, cell % per
    base = sum(((box // n ** k) % n) * m ** k for k in range(dim))
    s = [m ** k for k in range(dim)]
    if dim == 2:
        conn = torch.stack([base, torch.where(part == 0, base + s[0], base + s[0] + s[1]),
                            torch.where(part == 0, base + s[0] + s[1], base + s[1])])
    else:
        # the six paths along the axes from corner to opposite corner; odd ones swap their middle vertices
        b = torch.tensor([s[0], s[0] + s[2], s[1] + s[0], s[1], s[2], s[2] + s[1]], device=dev)
        c = torch.tensor([s[0] + s[1], s[0], s[1], s[1] + s[2], s[2] + s[0], s[2]], device=dev)
        conn = torch.stack([base, base + b[part], base + c[part], base + sum(s)])
    nv = int(conn.max()) + 1
    return coords[:, :nv].contiguous(), conn.to(torch.int32).contiguous(), ~interior[:nv]


def _lame(nq, cells, gen, dev):
    E = torch.exp(0.5 * torch.randn((nq, cells), generator=gen, device=dev, dtype=F64))
    nu = 0.2 + 0.25 * torch.rand((nq, cells), generator=gen, device=dev, dtype=F64)
    return E * nu / ((1.0 + nu) * (1.0 - 2.0 * nu)), E / (2.0 * (1.0 + nu))


def _inputs(case, seed):
    dev = torch.device("cuda")
    gen = torch.Generator(device=dev).manual_seed(int(seed))
    dim, cells, kind = case["dim"], case["cells"], case["kind"]
    qp, qw = RULES[dim]
    nq = len(qw)
    dt = F64 if case["prec"].startswith("fp64") else torch.float32
    coords, conn, edge = _mesh(dim, cells, gen, dev)
    V = coords.shape[1]
    uniform = lambda lo, hi, *shape: lo + (hi - lo) * torch.rand(shape, generator=gen, device=dev, dtype=F64)  # noqa: E731
    normal = lambda *shape: torch.randn(shape, generator=gen, device=dev, dtype=F64)  # noqa: E731
    d = {"case": dict(case), "coords": coords, "conn": conn, "qp": torch.tensor(qp, dtype=F64).numpy(),
         "qw": torch.tensor(qw, dtype=F64).numpy()}
    if kind in ("elasticity", "assembled", "refined"):
        lam, mu = _lame(nq, cells, gen, dev)
        d["lam"], d["mu"] = lam.to(dt), mu.to(dt)
    elif kind in ("residual", "train", "request", "solve"):
        d["K"] = torch.exp(normal(nq, cells)).to(dt)
    if kind in ("elasticity", "assembled"):
        d["u"] = (1e-2 * normal(dim, V)).to(dt)
    elif kind not in ("solve", "refined"):
        d["u"] = uniform(-1, 1, V).to(dt)
    if kind in ("train", "request"):
        d["lam_adj"] = uniform(-1, 1, dim + 1, cells).to(dt)
    if kind == "reaction":
        d["a"] = torch.exp(0.5 * normal(V)).to(dt)
        d["c"] = uniform(0.5, 2.0, nq, cells).to(dt)
    if kind in ("solve", "refined"):
        nc = 1 if kind == "solve" else dim
        # a linear function held on the boundary, a load inside
        g = (uniform(-1, 1, nc, 1) + uniform(-2, 2, nc, dim) @ coords) * edge
        b = uniform(-1, 1, nc, V) * ~edge / V
        d["fixed"] = edge.to(torch.uint8)
        d["x0"], d["b"] = (g[0].contiguous(), b[0].contiguous()) if kind == "solve" else (g, b)
    return d


def prepare(case, seed):
    d = _inputs(case, seed)
    V = d["coords"].shape[1]
    if case["kind"] == "train":
        d["mesh"] = DeviceMesh(d["coords"], d["conn"], d["qp"], d["qw"])
        d["u"].requires_grad_(True)
        d["K"].requires_grad_(True)
    elif case["kind"] in ("assembled", "solve", "refined"):
        d["ptr"], d["idx"] = fem.fem_build_node2cell(d["conn"], V)
    return d


# ------------------------------------------------------------------ one pass


def run(s):
    case = s["case"]
    kind, prec, dim = case["kind"], case["prec"], case["dim"]
    mesh = (s["coords"], s["conn"])
    rule = (s["qp"], s["qw"])
    if kind == "residual":
        return fem.fem_integrate_laplacian(*mesh, s["u"], s["K"], *rule, prec=prec)
    if kind == "elasticity":
        return fem.fem_integrate_elasticity(*mesh, s["u"], s["lam"], s["mu"], *rule, prec=prec)
    if kind == "train":
        r = laplacian_residual(s["u"], s["K"], s["mesh"], prec=prec)
        du, dK = torch.autograd.grad(r, (s["u"], s["K"]), s["lam_adj"])
        return {"r": r.detach(), "du": du, "dK": dK}
    if kind == "request":
        ptr, idx = fem.fem_build_node2cell(s["conn"], s["coords"].shape[1])
        dK, du = fem.fem_adjoint_laplacian(*mesh, s["u"], s["K"], *rule, s["lam_adj"], ptr, idx, prec=prec)
        return {"ptr": ptr, "idx": idx, "dK": dK, "du": du}
    if kind == "reaction":
        return fem.fem_integrate_reaction_diffusion(*mesh, s["u"], s["a"], *rule, c=s["c"], a_space=1, drift=DRIFT,
                                                    prec=prec)
    if kind == "pointwise":
        return fem.fem_integrate_pointwise(*mesh, s["u"], None, *rule, f1=NONLINEAR_F1, prec=prec)
    if kind == "assembled":
        r = fem.fem_integrate_elasticity(*mesh, s["u"], s["lam"], s["mu"], *rule, prec=prec)
        return fem.fem_gather_nodes(r, s["ptr"], s["idx"], s["coords"].shape[1], dim, prec=prec)
    x = s["x0"].clone()
    lists = (s["ptr"], s["idx"], s["fixed"])
    if kind == "solve":
        return fem.fem_pcg_laplacian(*mesh, s["K"], *rule, *lists, x, b=s["b"], max_iter=5000, rtol=1e-8, prec=prec)[0]
    return fem.fem_pcg_elasticity_refined(*mesh, s["lam"], s["mu"], *rule, *lists, x, b=s["b"], max_outer=30,
                                          max_inner=20000, rtol=1e-12, residual_prec=prec)[0]


# ------------------------------------------------------------------ work


def work(case):
    dim, C, kind = case["dim"], case["cells"], case["kind"]
    nb, nq = dim + 1, len(RULES[dim][1])
    n = _grid(dim, C)
    V = (n + 1) ** dim * C / (2 * n * n if dim == 2 else 6 * n ** 3)
    s = 8 if case["prec"].startswith("fp64") else 4
    mesh = 8 * dim * V + 4 * nb * C
    geometry = 5 if dim == 2 else 9 + 27 + 5  # columns, adjugate rows, determinant
    lap = geometry + 3 * dim + 2 * dim * dim + 2 * dim * dim + dim + 2 * nq
    el = geometry + dim * dim + 4 * dim ** 3 + 3 * dim * dim + dim * dim + 4 * nq
    if kind == "residual":
        return {"bytes": mesh + s * (V + (nq + nb) * C), "flops": lap * C}
    if kind == "elasticity":
        return {"bytes": mesh + s * (dim * V + (2 * nq + nb * dim) * C), "flops": el * C}
    if kind == "train":
        return {"bytes": mesh + s * (2 * V + (2 * nq + 2 * nb) * C), "flops": 2.5 * lap * C}
    if kind == "request":
        return {"bytes": mesh + s * (2 * V + (2 * nq + nb) * C) + 4 * (V + 1 + nb * C), "flops": 1.5 * lap * C}
    if kind == "reaction":
        return {"bytes": mesh + s * (2 * V + (nq + nb) * C), "flops": (lap + nq * 4 * nb + 4 * dim) * C}
    if kind == "pointwise":
        return {"bytes": mesh + s * (V + nb * C), "flops": (lap + nq * (4 * nb + 6 * dim + 12)) * C}
    if kind == "assembled":
        return {"bytes": mesh + s * (2 * dim * V + 2 * nq * C) + 4 * (V + 1 + nb * C), "flops": (el + nb * dim) * C}
    # the solves: what goes in and comes out, and one application of the operator
    nc = 1 if kind == "solve" else dim
    coefs = nq * (1 if kind == "solve" else 2)
    return {"bytes": mesh + 8 * (3 * nc * V + coefs * C) + 4 * (V + 1 + nb * C) + V,
            "flops": (lap if kind == "solve" else el) * C}


# ------------------------------------------------------------------ the same in 64 bits, in plain torch


def _geometry(d):
    """Basis gradients G [d+1][dim][C], |det J| [C], vertex coordinates xs [dim][d+1][C]."""
    conn = d["conn"].long()
    xs = d["coords"][:, conn]
    dim = xs.shape[0]
    e = [xs[:, j + 1] - xs[:, 0] for j in range(dim)]
    if dim == 2:
        rows = [torch.stack([e[1][1], -e[1][0]]), torch.stack([-e[0][1], e[0][0]])]
    else:
        rows = [torch.linalg.cross(e[(j + 1) % 3], e[(j + 2) % 3], dim=0) for j in range(3)]
    det = (e[0] * rows[0]).sum(0)
    G = [r / det for r in rows]
    return torch.stack([-sum(G)] + G), det.abs(), xs


def _stiffness(d, kind):
    """Element matrices [C][n][n] and the global numbers [n][C] of their rows."""
    G, adet, _ = _geometry(d)
    nb, dim, C = G.shape
    qw = torch.tensor(RULES[dim][1], dtype=F64, device=G.device)
    conn = d["conn"].long()
    if kind == "solve":
        s = (qw @ d["K"]) * adet
        return torch.einsum("bic,dic,c->cbd", G, G, s), conn
    V = d["coords"].shape[1]
    lbar, mbar = (qw @ d["lam"]) * adet, (qw @ d["mu"]) * adet
    S = torch.einsum("bkc,dlc,c->cbkdl", G, G, lbar) + torch.einsum("blc,dkc,c->cbkdl", G, G, mbar)
    diag = torch.einsum("bic,dic,c->cbd", G, G, mbar)
    for k in range(dim):
        S[:, :, k, :, k] += diag
    rows = torch.stack([conn[b] + k * V for b in range(nb) for k in range(dim)])
    return S.reshape(C, nb * dim, nb * dim), rows


def _solve(d, kind):
    """The system solved far below the entry point's tolerance: conjugate gradients in 64 bits."""
    S, rows = _stiffness(d, kind)
    b, x = d["b"].reshape(-1), d["x0"].reshape(-1).clone()
    N, V = b.numel(), d["coords"].shape[1]
    free = (d["fixed"] == 0).repeat(N // V).to(F64)
    flat = rows.reshape(-1)

    def apply(v):
        return torch.zeros(N, dtype=F64, device=v.device).index_add_(0, flat, torch.matmul(S, v[rows].t()[:, :, None])[:, :, 0].t().reshape(-1))

    D = torch.zeros(N, dtype=F64, device=b.device).index_add_(0, flat, torch.diagonal(S, dim1=1, dim2=2).t().reshape(-1))
    D = torch.where((free > 0) & (D > 0), D, torch.ones_like(D))
    for _ in range(3):  # each restart takes up the true residual
        r = (b - apply(x)) * free
        z = r / D
        p, rz = z.clone(), torch.dot(r, z)
        r0 = float(r.norm())
        if r0 == 0.0:
            break
        for it in range(4000):
            q = apply(p) * free
            alpha = rz / torch.dot(p, q)
            x += alpha * p
            r -= alpha * q
            if it % 25 == 24 and float(r.norm()) <= 1e-11 * r0:
                break
            z = r / D
            new = torch.dot(r, z)
            p = z + (new / rz) * p
            rz = new
    return x.reshape(d["x0"].shape)


def exact(case, seed):
    d = {k: v.to(F64) if isinstance(v, torch.Tensor) and v.is_floating_point() else v
         for k, v in _inputs(case, seed).items()}
    kind, dim = case["kind"], case["dim"]
    if kind in ("solve", "refined"):
        return _solve(d, kind)
    G, adet, xs = _geometry(d)
    nb, V = dim + 1, d["coords"].shape[1]
    conn = d["conn"].long()
    qp = torch.tensor(RULES[dim][0], dtype=F64, device=G.device)
    qw = torch.tensor(RULES[dim][1], dtype=F64, device=G.device)
    phi = torch.cat([1.0 - qp.sum(1, keepdim=True), qp], dim=1)  # [n_q][d+1]
    to_nodes = lambda rows: torch.zeros(V, dtype=F64, device=G.device).index_add_(0, conn.reshape(-1), rows.reshape(-1))  # noqa: E731
    if kind in ("elasticity", "assembled"):
        ue = d["u"][:, conn]  # [k][b][c]
        H = torch.einsum("kbc,bic->kic", ue, G)
        T = (qw @ d["mu"]) * adet * (H + H.transpose(0, 1))
        tr = (qw @ d["lam"]) * adet * sum(H[k, k] for k in range(dim))
        for k in range(dim):
            T[k, k] += tr
        r = torch.einsum("kic,bic->bkc", T, G)
        if kind == "elasticity":
            return r.reshape(nb * dim, -1)
        return torch.stack([to_nodes(r[:, k]) for k in range(dim)])
    ue = d["u"][conn]
    grad = torch.einsum("bc,bic->ic", ue, G)
    if kind == "reaction":
        ae = d["a"][conn]
        grad_a = torch.einsum("bc,bic->ic", ae, G)
        first = DRIFT * (grad_a * grad).sum(0)
        r = torch.zeros_like(ue)
        for q in range(len(qw)):
            f0 = d["c"][q] * (phi[q] @ ue) + first
            f1 = (phi[q] @ ae) * torch.einsum("bic,ic->bc", G, grad)
            r += qw[q] * adet * (phi[q][:, None] * f0 + f1)
        return r
    if kind == "pointwise":
        kbar = 0.0
        for q in range(len(qw)):
            uq, xq = phi[q] @ ue, torch.einsum("b,ibc->ic", phi[q], xs)
            kbar = kbar + qw[q] * (P[0] + P[1] * uq + P[2] * uq * uq) * (1 + P[3] * sum((i + 1) * xq[i] for i in range(dim)))
        return kbar * adet * torch.einsum("bic,ic->bc", G, grad)
    s = (qw @ d["K"]) * adet
    r = s * torch.einsum("bic,ic->bc", G, grad)
    if kind == "residual":
        return r
    gl = torch.einsum("bc,bic->ic", d["lam_adj"], G)
    dK = qw[:, None] * (adet * (gl * grad).sum(0))
    du = to_nodes(s * torch.einsum("bic,ic->bc", G, gl))
    if kind == "train":
        return {"r": r, "du": du, "dK": dK}
    return {"ptr": None, "idx": None, "dK": dK, "du": du}
