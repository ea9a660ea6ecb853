"""Partitioner paths against the oracle at the sizes where they can go wrong:
more segments than a shared-memory histogram holds, coordinate ties decided by
the id digits, one node per part, ids past one 8192-id block, no halo, halos
that cover everything, and rows longer than the eight- and sixteen-edge steps.
Every comparison is exact."""
import numpy as np
import pytest
import torch

from oracle import xmgn_oracle as O
from tests.helpers import case

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def X():
    from paper_2411_17164_gb300 import build, xmgn
    build.build()
    return xmgn


def _cloud(kind, n):
    if kind == "lattice":  # equal coordinates on every axis, in an order that is not the coordinate order
        side = int(round(n ** (1 / 3)))
        g = np.stack(np.meshgrid(*[np.arange(side)] * 3, indexing="ij"), -1).reshape(-1, 3)
        return (g[np.random.default_rng(1).permutation(len(g))] / 64.0).astype(np.float32)
    if kind == "plane":    # one axis constant, another with few values
        r = np.random.default_rng(2)
        return np.stack([r.integers(0, 3, n) / 8, np.full(n, 0.25), r.random(n)], 1).astype(np.float32)
    return case("body", n, 5)[0]


def _check(X, xyz, rp, col, P, hops, part_in=None):
    g = dict(n=len(xyz), E=len(col), row_ptr=torch.from_numpy(rp).cuda(), col=torch.from_numpy(col).cuda())
    pin = None if part_in is None else torch.from_numpy(part_in).cuda()
    b = X.partition_halo(g, torch.from_numpy(xyz).cuda(), P, hops, part_in=pin)
    part = O.rcb(xyz, P) if part_in is None else part_in
    np.testing.assert_array_equal(b["part"].cpu().numpy(), part)
    gid, hop, brp, bcol, recv, perm = (b[k].cpu().numpy() for k in ("gid", "hop", "row_ptr", "col", "recv", "csc_perm"))
    for p, pt in enumerate(O.halo_partition(rp, col, part, P, hops)):
        n0, n1, e0, e1 = b["node_ptr"][p], b["node_ptr"][p + 1], b["edge_ptr"][p], b["edge_ptr"][p + 1]
        np.testing.assert_array_equal(gid[n0:n1], pt["gid"])
        np.testing.assert_array_equal(hop[n0:n1], pt["hop"])
        assert b["inner_cnt"][p] == pt["n_inner"]
        np.testing.assert_array_equal(brp[n0:n1 + 1] - e0, pt["row_ptr"])
        np.testing.assert_array_equal(bcol[e0:e1] - n0, pt["col"])
    np.testing.assert_array_equal(recv, np.repeat(np.arange(len(gid)), np.diff(brp)))
    assert np.all(bcol[perm] == recv) and np.all(recv[perm] == bcol)


@pytest.mark.parametrize("kind,n,P,hops", [("lattice", 1000, 7, 2), ("plane", 1500, 13, 1), ("body", 2001, 100, 1),
                                           ("body", 90, 90, 1), ("body", 8225, 3, 0), ("body", 700, 2, 40)])
def test_bisection_and_halos(X, kind, n, P, hops):
    xyz = _cloud(kind, n)
    rp, col, _, _ = O.symmetrise(O.knn(xyz, 6), len(xyz))
    _check(X, xyz, rp, col.astype(np.int32), P, hops)


def test_rows_longer_than_one_step(X):
    """A ring with three hubs joined to every 2nd, 3rd and 40th node: rows of 2 to 600 edges; nodes of no part."""
    n = 1200
    s, t = [], []
    for i in range(n):
        s += [i, (i + 1) % n]
        t += [(i + 1) % n, i]
    for hub, step in ((0, 2), (601, 3), (1111, 40)):
        for j in range(0, n, step):
            if j != hub:
                s += [hub, j]
                t += [j, hub]
    e = np.unique(np.stack([s, t], 1), axis=0)
    rp = np.concatenate([[0], np.cumsum(np.bincount(e[:, 0], minlength=n))]).astype(np.int64)
    part = (np.arange(n) // 300).astype(np.int32)
    part[200:260] = -1
    _check(X, np.zeros((n, 3), np.float32), rp, e[:, 1].astype(np.int32), 4, 2, part)
