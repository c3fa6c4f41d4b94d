"""The bounded wait of the solves' loop kernel at its grid barrier (fem_selftest_wait runs it on
counters of its own): a wait that runs out is reported and the context stays usable."""

import time

import pytest
import torch

import paper_1607_04245_gb300 as fem
from test_gpu_solver_forms import _mesh, _problem, _solve, _work_bytes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("budget_ms", [0, 1, 20])
def test_timeout_is_reported_and_a_solve_follows(budget_ms):
    assert fem.fem_device_error() == 0
    p = _problem(_mesh(3, 20577), "laplacian", "mixed")  # several CTAs
    before = _solve(p, _work_bytes(p))
    torch.cuda.synchronize()
    t = time.perf_counter()
    fem.fem_selftest_wait(budget_ms * 1_000_000)
    torch.cuda.synchronize()
    took = time.perf_counter() - t
    assert budget_ms * 1e-3 <= took < budget_ms * 1e-3 + 1.0
    assert fem.fem_device_error() == -6 and fem.fem_device_error() == 0
    after = _solve(p, _work_bytes(p))
    assert torch.equal(before[0], after[0]) and before[1:] == after[1:]
    assert fem.fem_device_error() == 0


def test_many_at_once():
    """More calls than slots, on several streams: each runs its own wait."""
    streams = [torch.cuda.Stream() for _ in range(8)]
    for i in range(80):
        fem.fem_selftest_wait(200_000, stream=streams[i % 8])
    torch.cuda.synchronize()
    assert fem.fem_device_error() == -6 and fem.fem_device_error() == 0


def test_the_wait_is_the_loop_kernels():
    """One bounded wait in the sources, used by the loop kernel and by its self-test."""
    import os

    csrc = os.path.join(os.path.dirname(fem.__file__), "csrc")
    src = {f: open(os.path.join(csrc, f)).read() for f in os.listdir(csrc) if f.endswith((".cu", ".cuh"))}
    assert {f for f, t in src.items() if "globaltimer" in t} == {"fem_wait.cuh"}
    assert {f for f, t in src.items() if "wait_reached(" in t} == {"fem_wait.cuh", "fem_solver.cu", "fem_core.cu"}
