"""grad_W with at most 128 output channels on wide column tiles: channels of
one, part of one and two 64-row atoms, columns that end inside a tile, in its
second half and on its edge, one split (dequantized in the epilogue) and many,
the implicit im2col operand; against a 64-bit product of the dequantized codes
(max |g - r| / max(|r|, 1e-3 ||r_row||_inf) <= 1e-3).  The cases of wide tiles ask
the library whether they took them; the others are shapes that the rule leaves
to 128-column tiles."""
import numpy as np
import pytest

import oracle as orc
from paper_2010_14298_gb300 import workloads as wl
from test_gpu_pair import _product, _rel

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _grad_w(n, c, d, kind, bits):
    from paper_2010_14298_gb300 import fqt
    g = wl.rng(7 + n)
    dH = torch.from_numpy(wl.random_grad(g, n, c)).cuda()
    X = torch.from_numpy(g.uniform(-1, 1, (n, d)).astype(np.float32)).cuda()
    qx = fqt.quantize_act(X, 8)
    _, q1 = fqt.quantize_grad(dH, kind, bits, 0, seed=3)
    ws = fqt.Workspace(n, c, d)
    _, gw = fqt.linear_backward(q1, q1, qx, None, grad_x=False, ws=ws)
    assert fqt.sync_status(ws) == 0
    plan = fqt.debug_last_plan(grad_w=True)
    assert _rel(gw, _product(orc.dequant(q1.to_numpy()).T, orc.dequant(qx.to_numpy()))) <= 1e-3
    return plan


@pytest.mark.parametrize("n,c,d", [(1411, 16, 11264), (2983, 48, 6784), (1638, 64, 12880),
                                   (2001, 80, 11264), (2443, 128, 11264), (126756, 16, 144)])
def test_grad_w_wide_tiles(n, c, d):
    plan = _grad_w(n, c, d, wl.PSQ, 8)
    assert plan["kernel"] == "wide" and plan["splits"] > 1


@pytest.mark.parametrize("n,c,d", [(23, 16, 20960), (70, 64, 20976), (150, 80, 24192),
                                   (300, 128, 30656)])
def test_grad_w_wide_tiles_one_split(n, c, d):
    plan = _grad_w(n, c, d, wl.PSQ, 8)
    assert plan["kernel"] == "wide" and plan["fused"]


@pytest.mark.parametrize("n,c,d", [(20011, 64, 576), (9000, 16, 1040), (33000, 128, 272),
                                   (9100, 80, 208), (517, 48, 16384), (60, 128, 16368)])
@pytest.mark.parametrize("kind,bits", [(wl.PSQ, 8), (wl.PTQ, 4)])
def test_grad_w_wide(n, c, d, kind, bits):
    _grad_w(n, c, d, kind, bits)


@pytest.mark.parametrize("n,h,w,c,cout,k,pad", [
    (20, 30, 56, 64, 64, 3, 1), (9, 57, 9, 128, 96, 3, 1), (40, 14, 14, 192, 32, 3, 1),
    (6, 32, 64, 64, 128, 3, 1), (90, 7, 7, 128, 64, 3, 1), (30, 19, 8, 64, 48, 2, 1),
    (12, 28, 28, 64, 80, 4, 2), (10, 31, 33, 64, 64, 2, 0), (8, 24, 24, 64, 64, 5, 2)])
def test_conv_grad_w_wide(n, h, w, c, cout, k, pad):
    _conv_grad_w(n, h, w, c, cout, k, pad)


# output rows of 5 to 64 pixels in blocks of 8 to 64 slots, images whose last
# block is partly or wholly rows of the image, one to four taps a row
@pytest.mark.parametrize("n,h,w,c,cout,k,pad", [
    (200, 9, 8, 192, 16, 2, 1), (20, 33, 33, 192, 128, 2, 1), (200, 9, 9, 64, 16, 3, 1),
    (300, 7, 7, 192, 64, 3, 0), (90, 33, 7, 128, 64, 3, 1), (130, 7, 28, 128, 112, 3, 1),
    (300, 9, 9, 64, 80, 3, 1), (20, 37, 56, 64, 64, 3, 1), (130, 9, 9, 192, 128, 3, 1),
    (13, 9, 33, 192, 16, 4, 2), (200, 9, 8, 64, 64, 4, 2), (20, 9, 33, 192, 80, 4, 2),
    (130, 9, 9, 64, 64, 5, 2), (130, 9, 9, 64, 80, 5, 2), (130, 9, 9, 64, 128, 5, 2)])
def test_conv_grad_w_wide_tiles(n, h, w, c, cout, k, pad):
    plan = _conv_grad_w(n, h, w, c, cout, k, pad)
    assert plan["kernel"] == "wide" and plan["row_taps"] == (k if k <= 4 else 0)


def _conv_grad_w(n, h, w, c, cout, k, pad):
    """Equal integer sums, and so equal results, in both layouts of X~."""
    from paper_2010_14298_gb300 import fqt
    g = wl.rng(56)
    x = g.uniform(-1, 1, (n, h, w, c)).astype(np.float32)
    X = torch.from_numpy(wl.im2col_nhwc(x, k, k, 1, pad)).cuda()
    rows = X.shape[0]
    dH = torch.from_numpy(wl.random_grad(g, rows, cout)).cuda()
    _, q1 = fqt.quantize_grad(dH, fqt.PSQ, 8, 0, seed=1)
    qx = fqt.quantize_act(X, 8)
    qi = fqt.quantize_act_conv(torch.from_numpy(x).cuda(), k, k, pad, 8)
    ws = fqt.Workspace(rows, cout, k * k * c)
    _, ge = fqt.linear_backward(q1, q1, qx, None, grad_x=False, ws=ws)
    _, gi = fqt.linear_backward(q1, q1, qi, None, grad_x=False, ws=ws)
    assert fqt.sync_status(ws) == 0
    plan = fqt.debug_last_plan(grad_w=True)
    assert _rel(ge, _product(orc.dequant(q1.to_numpy()).T, orc.dequant(qx.to_numpy()))) <= 1e-3
    assert torch.equal(gi, ge)
    return plan
