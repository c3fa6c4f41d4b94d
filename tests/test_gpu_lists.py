"""fem_build_node2cell against a stable sort of the connectivity on the host: lists of every
length around the shared-memory sort's limits (8 lanes per vertex, 128 entries),
vertices in no cell, several vertices per warp with the same id, scans of one tile and more, and
the larger scan whose tile sums are scanned by their own kernel."""

import numpy as np
import pytest
import torch

import paper_1607_04245_gb300 as fem

pytestmark = pytest.mark.gpu


def _check(conn, V):
    nb, C = conn.shape
    ptr, idx = fem.fem_build_node2cell(torch.from_numpy(conn).cuda(), V)
    flat = conn.T.ravel()  # entry e*nb + a at its own position
    want = np.argsort(flat, kind="stable").astype(np.int32)
    counts = np.bincount(flat, minlength=V)
    assert np.array_equal(ptr.cpu().numpy(), np.concatenate([[0], np.cumsum(counts)]))
    assert np.array_equal(idx.cpu().numpy(), want)
    assert fem.fem_device_error() == 0


@pytest.mark.parametrize("nb", [3, 4])
@pytest.mark.parametrize("C,V", [(1, 4), (31, 9), (33, 9), (257, 40), (1000, 8), (5000, 3000), (40001, 4097),
                                 (40001, 90001), (300001, 50000)])
def test_random_connectivity(nb, C, V):
    rng = np.random.default_rng(C + V + nb)
    _check(rng.integers(0, V, (nb, C)).astype(np.int32), V)


@pytest.mark.parametrize("nb", [3, 4])
@pytest.mark.parametrize("n", [1, 7, 8, 9, 31, 32, 33, 127, 128, 129, 700])
def test_one_long_list(nb, n):
    """n cells around vertex 0, whose position in the cell varies."""
    conn = np.arange(1, nb * n + 1, dtype=np.int32).reshape(n, nb)
    conn[np.arange(n), np.arange(n) % nb] = 0
    _check(np.array(conn[::-1].T, order="C"), nb * n + 1)


def test_many_tiles():
    """More than 2048 scan tiles of 4096 vertices."""
    V = 2048 * 4096 + 5
    rng = np.random.default_rng(3)
    _check(rng.integers(0, V, (3, 200001)).astype(np.int32), V)
