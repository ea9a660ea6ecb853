"""Coordinates off the lattice (too large, infinite, NaN; one or all of them):
refused with XMGN_ERR_RANGE, no output array written, and the next build of a
valid cloud is right."""
import ctypes as C

import numpy as np
import pytest
import torch

from oracle import xmgn_oracle as O
from tests.helpers import assert_same_graph, case, oracle_graph

pytestmark = pytest.mark.gpu
N, K, MARK = 2000, 6, -77
BAD = {"far": 8.0, "inf": -np.inf, "nan": np.nan}


@pytest.fixture(scope="module")
def X():
    from paper_2411_17164_gb300 import build, xmgn
    build.build()
    return xmgn


def _cloud(bad, where):
    xyz = case("sphere", N, 9)[0].copy()
    if where == "one":
        xyz[N - 1, 2] = BAD[bad]
    elif where == "all":
        xyz[:] = BAD[bad]
    return torch.from_numpy(xyz).cuda()


def _full(n, dtype=torch.int32):
    return torch.full((n,), MARK, dtype=dtype, device="cuda")


def _call_knn(X, xyz, levels):
    L, P, wsb, E = X.lib(), lambda t: C.c_void_p(t.data_ptr()), C.c_size_t(), C.c_int64(MARK)
    slots = K * len(levels) + (3 if len(levels) > 1 else 0)
    outs = [_full(N * slots), _full(N + 1, torch.int64)] + [_full(2 * N * slots) for _ in range(3)]
    if len(levels) > 1:
        hs = (C.c_int64 * len(levels))(*levels)
        assert L.xmgn_build_multiscale_ws(N, len(levels), K, 3, C.byref(wsb)) == 0
        ws = torch.empty(wsb.value, dtype=torch.uint8, device="cuda")
        rc = L.xmgn_build_multiscale(P(xyz), N, hs, len(levels), K, 3, X.DEFAULT_SCALE, P(ws), ws.numel(),
                                     *map(P, outs), 2 * N * slots, C.byref(E), None)
    else:
        assert L.xmgn_build_knn_ws(N, K, C.byref(wsb)) == 0
        ws = torch.empty(wsb.value, dtype=torch.uint8, device="cuda")
        rc = L.xmgn_build_knn(P(xyz), N, K, X.DEFAULT_SCALE, P(ws), ws.numel(), *map(P, outs), 2 * N * slots,
                              C.byref(E), None)
    torch.cuda.synchronize()
    return rc, E.value, outs


@pytest.mark.parametrize("levels", [[N], [200, 700, N]])
@pytest.mark.parametrize("bad", list(BAD))
@pytest.mark.parametrize("where", ["one", "all"])
def test_build_is_refused_and_writes_nothing(X, bad, where, levels):
    torch.cuda.synchronize()
    rc, e, outs = _call_knn(X, _cloud(bad, where), levels)
    assert rc == 2 and e == MARK
    for t in outs:
        assert bool((t == MARK).all())
    good = _cloud(bad, "none")
    _, rp, col, cperm = oracle_graph(good.cpu().numpy())
    assert_same_graph(X.build_knn(good, K), rp, col, cperm)


@pytest.mark.parametrize("parts", [1, 7])
@pytest.mark.parametrize("where", ["one", "all"])
def test_bisection_is_refused_and_writes_nothing(X, where, parts):
    good = _cloud("nan", "none")
    g = X.build_knn(good, K)
    L, P, wsb = X.lib(), lambda t: C.c_void_p(t.data_ptr()), C.c_size_t()
    assert L.xmgn_partition_halo_ws(N, g["E"], parts, C.byref(wsb)) == 0
    ws, part, xyz = torch.empty(wsb.value, dtype=torch.uint8, device="cuda"), _full(N), _cloud("nan", where)
    ptrs = [(C.c_int64 * (parts + 1))(*[MARK] * (parts + 1)) for _ in range(3)]
    torch.cuda.synchronize()
    rc = L.xmgn_partition_halo(P(g["row_ptr"]), P(g["col"]), N, g["E"], P(xyz), X.DEFAULT_SCALE, parts, 2, None, P(ws),
                               ws.numel(), P(part), *ptrs, None, None, None, None, None, None, 0, 0, None)
    torch.cuda.synchronize()
    assert rc == 2
    assert bool((part == MARK).all()) and all(v == MARK for p in ptrs for v in p)
    b = X.partition_halo(g, good, parts, 2)
    np.testing.assert_array_equal(b["part"].cpu().numpy(), O.rcb(good.cpu().numpy(), parts))
