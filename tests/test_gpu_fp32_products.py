"""FP32 products at the edges of their tiles, against the FP64 oracle: widths
that fill no whole 64- or 128-wide tile, row counts that end inside a tile, and
a parameter vector at an address that 16-byte loads cannot take (the general
kernels).  Tolerance: fp32 sums of at most 3H + n terms, relative L2 <= 1e-5
(eps 6e-8 times the root of the longest chain, about 40, with a margin of 4)."""
import numpy as np
import pytest
import torch

from oracle import xmgn_oracle as O
from paper_2411_17164_gb300 import synth
from tests.helpers import case, oracle_graph, rel_l2

pytestmark = pytest.mark.gpu
TOL = 1e-5


@pytest.mark.parametrize("H,n,off", [(32, 130, 0), (96, 257, 0), (160, 500, 0), (128, 640, 1), (320, 300, 0)])
def test_fp32_products_at_tile_edges(H, n, off):
    from paper_2411_17164_gb300 import build, xmgn
    build.build()
    xyz, nin = case("sphere", n, 11)
    _, rp, col, _ = oracle_graph(xyz)
    params = synth.init_params(H, 2, 6, 4, 13, perturb_ln=True)
    tgt = synth.fourier_targets(xyz, 3)
    lo, go, yo = O.loss_and_grad(params.astype(np.float64), (H, 2, 6, 4), rp, col, nin, xyz, tgt)
    g = xmgn.build_knn(torch.from_numpy(xyz).cuda(), 6)
    tp = torch.zeros(len(params) + off, device="cuda")[off:]
    tp.copy_(torch.from_numpy(params))
    ni, xz, tt = (torch.from_numpy(a).cuda() for a in (nin, xyz, tgt))
    m = xmgn.Model(H, 2, g, dtype="fp32", n_norm=n)
    y, loss, dp = torch.zeros((n, 4), device="cuda"), torch.zeros((), device="cuda"), torch.zeros_like(tp)
    m.forward(tp, ni, xz, targets=tt, y=y, loss=loss)
    m.backward(tp, ni, xz, tt, dp)
    torch.cuda.synchronize()
    xmgn.check_device()
    assert rel_l2(y.cpu().numpy(), yo) <= TOL
    assert rel_l2(dp.cpu().numpy(), go) <= TOL
    assert abs(float(loss) - lo) <= TOL * abs(lo)
