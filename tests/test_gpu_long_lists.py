"""Vertex-to-cell lists longer than the sort's shared memory (128 entries): hubs of many
triangles, in order and shuffled, against numpy's lists. Lengths around the merges' powers of
two, several hubs of different lengths side by side, and one long one. Integers: equality."""

import numpy as np
import pytest
import torch

import paper_1607_04245_gb300 as fem
from gpu_util import to_dev

pytestmark = pytest.mark.gpu


def _hubs(lengths):
    """Fans of triangles around one vertex each."""
    parts, at = [], 0
    for k in lengths:
        i = np.arange(k)
        parts.append(np.stack([np.zeros(k), 1 + i, 1 + (i + 1) % k]).astype(np.int32) + at)
        at += k + 1
    return np.concatenate(parts, axis=1), at


@pytest.mark.parametrize("lengths", [[127, 128, 129], [130], [255, 256, 257, 3, 40], [511, 513, 1024], [1025, 200, 2049],
                                     [20000], list(range(120, 180))])
@pytest.mark.parametrize("shuffled", [False, True])
def test_lists_of_hubs(lengths, shuffled):
    conn, V = _hubs(lengths)
    if shuffled:
        conn = conn[:, np.random.default_rng(len(lengths)).permutation(conn.shape[1])]
    C = conn.shape[1]
    flat = conn.T.reshape(-1)  # entry 3 cell + local vertex
    order = np.argsort(flat, kind="stable")
    ptr = np.concatenate([[0], np.cumsum(np.bincount(flat, minlength=V))])
    got_ptr, got_idx = fem.fem_build_node2cell(to_dev(np.ascontiguousarray(conn), torch.int32), V)
    assert np.array_equal(got_ptr.cpu().numpy(), ptr) and np.array_equal(got_idx.cpu().numpy(), order)
    assert len(order) == 3 * C and fem.fem_device_error() == 0
