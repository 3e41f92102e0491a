"""grad_W with at most 128 output channels on wide column tiles: channels of
one, part of one and two 64-row atoms, columns that end inside a tile, in its
second half and on its edge, one split (dequantized in the epilogue) and many,
the implicit im2col operand; against a 64-bit product of the dequantized codes
(max |g - r| / max(|r|, 1e-3 ||r_row||_inf) <= 1e-3)."""
import numpy as np
import pytest

import oracle as orc
from paper_2010_14298_gb300 import workloads as wl
from test_gpu_pair import _product, _rel

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,c,d", [(20011, 64, 576), (9000, 16, 1040), (33000, 128, 272),
                                   (9100, 80, 208), (517, 48, 16384), (60, 128, 16368)])
@pytest.mark.parametrize("kind,bits", [(wl.PSQ, 8), (wl.PTQ, 4)])
def test_grad_w_wide(n, c, d, kind, bits):
    from paper_2010_14298_gb300 import fqt
    g = wl.rng(7 + n)
    dH = torch.from_numpy(wl.random_grad(g, n, c)).cuda()
    X = torch.from_numpy(g.uniform(-1, 1, (n, d)).astype(np.float32)).cuda()
    qx = fqt.quantize_act(X, 8)
    _, q1 = fqt.quantize_grad(dH, kind, bits, 0, seed=3)
    ws = fqt.Workspace(n, c, d)
    _, gw = fqt.linear_backward(q1, q1, qx, None, grad_x=False, ws=ws)
    assert fqt.sync_status(ws) == 0
    assert _rel(gw, _product(orc.dequant(q1.to_numpy()).T, orc.dequant(qx.to_numpy()))) <= 1e-3


@pytest.mark.parametrize("n,h,w,c,cout,k,pad", [
    (20, 30, 56, 64, 64, 3, 1), (9, 57, 9, 128, 96, 3, 1), (40, 14, 14, 192, 32, 3, 1),
    (6, 32, 64, 64, 128, 3, 1), (90, 7, 7, 128, 64, 3, 1), (30, 19, 8, 64, 48, 2, 1),
    (12, 28, 28, 64, 80, 4, 2), (10, 31, 33, 64, 64, 2, 0), (8, 24, 24, 64, 64, 5, 2)])
def test_conv_grad_w_wide(n, h, w, c, cout, k, pad):
    """Bit-equal sums in both layouts of X~ (codes and their column sums differ
    by the im2col padding, so the results agree to their rounding)."""
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
    assert _rel(ge, _product(orc.dequant(q1.to_numpy()).T, orc.dequant(qx.to_numpy()))) <= 1e-3
    assert _rel(gi, ge.double().cpu().numpy()) <= 1e-5
