"""Halo search with many overlapping parts, exact against the oracle: the nodes
of a hop are more than one step of all blocks, and steps that claim nothing
stand between steps that do (a hub reaches almost everything in two hops, a
chain behind it goes on one node per hop)."""
import numpy as np
import pytest
import torch

from oracle import xmgn_oracle as O
from tests.helpers import case
from tests.test_gpu_partition_paths import X, _check  # noqa: F401  (X is a fixture)

pytestmark = pytest.mark.gpu


def _steps(rp, col, part, P, hops):
    """Most steps that a block takes in one hop (32 nodes a step, N / 32 blocks)."""
    per_hop = np.zeros(hops + 1, np.int64)
    for pt in O.halo_partition(rp, col, part, P, hops):
        per_hop += np.bincount(pt["hop"], minlength=hops + 1)
    return int(per_hop[1:hops].max()) / (32 * -(-(len(rp) - 1) // 32))


@pytest.mark.parametrize("n,P,hops", [(100, 48, 9), (200, 28, 8), (700, 13, 12)])
def test_overlapping_parts_of_a_body(X, n, P, hops):  # noqa: F811
    xyz = case("body", n, 5)[0]
    rp, col, _, _ = O.symmetrise(O.knn(xyz, 6), n)
    assert _steps(rp, col, O.rcb(xyz, P), P, hops) > 1
    for _ in range(3):
        _check(X, xyz, rp, col.astype(np.int32), P, hops)


@pytest.mark.parametrize("n,P,tail", [(300, 20, 30), (1500, 10, 12)])
def test_hub_and_chain(X, n, P, tail):  # noqa: F811
    m = n - tail
    pairs = [(0, j) for j in range(1, m)] + [(j, j + 1) for j in range(1, n - 1)]
    e = np.unique(np.array(pairs + [(b, a) for a, b in pairs]), axis=0)
    rp = np.concatenate([[0], np.cumsum(np.bincount(e[:, 0], minlength=n))]).astype(np.int64)
    col = e[:, 1].astype(np.int32)
    part = (np.arange(n) * P // m).astype(np.int32)
    part[m:] = -1
    assert _steps(rp, col, part, P, 8) > 4
    for _ in range(3):
        _check(X, np.zeros((n, 3), np.float32), rp, col, P, 8, part)
