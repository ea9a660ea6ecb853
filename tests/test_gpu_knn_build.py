"""kNN search and symmetrisation at the edges of their ranges, bit-exact against
the oracle: every candidate-list capacity, both groupings of lanes, grids one
cell thick, far outliers (many rings), repeated points (ties by index), and rows
that pass from the shared-memory sort to the global one."""
import numpy as np
import pytest
import torch

from oracle import xmgn_oracle as O
from tests.helpers import assert_same_graph, case

pytestmark = pytest.mark.gpu


def _cloud(kind, n, k):
    rng = np.random.default_rng(n + k)
    if kind == "sphere":
        return case("sphere", n, 3)[0]
    if kind == "line":
        xyz = np.zeros((n, 3), np.float32)
        xyz[:, 1] = np.sort(rng.random(n)).astype(np.float32) ** 3
        return xyz
    if kind == "dup":  # a few sites, each many times: the copies of least index are listed by all
        return rng.integers(0, 2, (n, 3)).astype(np.float32)
    xyz = rng.random((n, 3)).astype(np.float32)
    if kind == "volume":
        xyz[:5] *= 7.0
    else:
        xyz[:, 2] = 0.5
    return xyz


def _check(xyz, k):
    from paper_2411_17164_gb300 import build, xmgn
    build.build()
    g = xmgn.build_knn(torch.from_numpy(xyz).cuda(), k, want_nbr=True)
    nbr = O.knn(xyz, k)
    np.testing.assert_array_equal(g["nbr"].cpu().numpy(), nbr)
    rp, col, _, cperm = O.symmetrise(nbr, len(xyz))
    assert_same_graph(g, rp, col, cperm)
    return np.diff(rp)


@pytest.mark.parametrize("k", [1, 3, 4, 7, 16, 17, 32])
@pytest.mark.parametrize("kind,n", [("sphere", 33), ("line", 257), ("dup", 600), ("dup", 9000), ("volume", 900),
                                    ("flat", 640)])
def test_candidate_lists_rings_and_rows(kind, n, k):
    deg = _check(_cloud(kind, n, k), k)
    if kind == "dup":
        assert deg.max() > (1040 if n > 8500 else 64)  # rows past the shared-memory sort


def test_one_lane_per_point():
    """More points than eight lanes each would fill the GPU with."""
    from paper_2411_17164_gb300 import build, xmgn
    build.build()
    n = torch.cuda.get_device_properties(0).multi_processor_count * 2048 // 8 + 3
    xyz = case("body", n, 4)[0]
    g = xmgn.build_knn(torch.from_numpy(xyz).cuda(), 6, want_nbr=True)
    nbr = O.knn_tree(xyz, 6)
    np.testing.assert_array_equal(g["nbr"].cpu().numpy(), nbr)
    rp, col, _, cperm = O.symmetrise(nbr, n)
    assert_same_graph(g, rp, col, cperm)
