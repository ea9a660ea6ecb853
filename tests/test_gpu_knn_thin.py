"""kNN of clouds whose grid is thin along one or two axes, with points far off
the others (their search takes many rings), bit-exact against the oracle: each
axis, both groupings of lanes.  A ring's rows outside the grid are not stepped
through, so every build here takes milliseconds."""
import time

import numpy as np
import pytest
import torch

from oracle import xmgn_oracle as O
from tests.helpers import assert_same_graph

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", [1, 6, 16])
@pytest.mark.parametrize("axis", [0, 1, 2])
@pytest.mark.parametrize("kind,n", [("plane", 1500), ("line", 700), ("slab", 1500), ("plane", 45000), ("line", 45000)])
def test_thin_grids_with_far_points(kind, n, axis, k):
    from paper_2411_17164_gb300 import build, xmgn
    build.build()
    rng = np.random.default_rng(10 * axis + k)
    xyz = rng.random((n, 3)).astype(np.float32) / 64
    if kind == "line":
        keep = xyz[:, axis].copy()
        xyz[:] = 0.25
        xyz[:, axis] = keep
        xyz[:4, axis] = [1.0, 1.5, 2.0, 7.5]
    else:
        xyz[:, axis] = 0.25 if kind == "plane" else rng.integers(0, 3, n) / 2048
        xyz[:3, (axis + 1) % 3] = [1.0, 1.25, 0.75]
        xyz[2:5, (axis + 2) % 3] = [2.0, 0.5, 3.0]
    t = torch.from_numpy(xyz).cuda()
    nbr = O.knn(xyz, k) if n < 2000 else O.knn_tree(xyz, k)
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    g = xmgn.build_knn(t, k, want_nbr=True)
    assert time.perf_counter() - t0 < 5.0
    np.testing.assert_array_equal(g["nbr"].cpu().numpy(), nbr)
    rp, col, _, cperm = O.symmetrise(nbr, n)
    assert_same_graph(g, rp, col, cperm)
