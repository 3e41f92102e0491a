"""Contractions on CTA pairs (256 x 256 super tiles): shapes whose last super
tile, second half or second CTA is partly or wholly outside the matrix, with
and without splits of the grad_W reduction, against a 64-bit product of the
dequantized codes (max |g - r| / max(|r|, 1e-3 ||r_row||_inf) <= 1e-3)."""
import numpy as np
import pytest

import oracle as orc
from paper_2010_14298_gb300 import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _rel(g, r):
    g, r = g.double().cpu().numpy(), np.asarray(r)
    floor = 1e-3 * np.abs(r).max(axis=1, keepdims=True)
    return float((np.abs(g - r) / np.maximum(np.abs(r), np.maximum(floor, 1e-30))).max())


def _product(a, b):
    return (torch.from_numpy(np.ascontiguousarray(a)).cuda() @
            torch.from_numpy(np.ascontiguousarray(b)).cuda()).cpu().numpy()


# (rows, C, D): one wave of super tiles less than the single-CTA plan needs
@pytest.mark.parametrize("n,c,d", [(2100, 528, 4112), (2063, 1008, 4096), (4097, 512, 2320),
                                   (12500, 272, 1296)])
@pytest.mark.parametrize("kind,bits,block", [(wl.PTQ, 8, 0), (wl.PSQ, 5, 0), (wl.BHQ, 5, 16),
                                             (wl.BHQ, 4, 64), (wl.BHQ, 8, 16), (wl.BHQ, 5, 4),
                                             (wl.BHQ, 5, 8), (wl.BHQ, 5, 32)])
def test_backward_pair_edges(n, c, d, kind, bits, block):
    from paper_2010_14298_gb300 import fqt
    if block * c > 65536:
        pytest.skip("blocks of this width are refused")
    g = wl.rng(77 + n)
    dH = torch.from_numpy(wl.random_grad(g, n, c)).cuda()
    X = torch.from_numpy(g.uniform(-1, 1, (n, d)).astype(np.float32)).cuda()
    W = torch.from_numpy((0.05 * g.standard_normal((c, d))).astype(np.float32)).cuda()
    qx, qw = fqt.quantize_act(X, 8), fqt.quantize_weight(W, 8)
    q2, q1 = fqt.quantize_grad(dH, kind, bits, block, seed=3)
    ws = fqt.Workspace(n, c, d)
    gx, gw = fqt.linear_backward(q2, q1, qx, qw, ws=ws)
    assert fqt.sync_status(ws) == 0
    px, pw = fqt.debug_last_plan(), fqt.debug_last_plan(grad_w=True)
    # (the int32 form takes pairs from eight K blocks on: not of 272 columns)
    assert px["kernel"] == ("single" if c == 272 and (kind, bits) == (wl.BHQ, 8) else "pair")
    if kind == wl.BHQ:  # wide rows and large blocks leave less room for row offsets in fp32
        narrow = {528: 1, 1008: 0} if block == 32 else {1008: 1}
        assert px["form"] == (0 if bits == 8 else narrow.get(c, 2))
    if d > 4000:
        assert pw["kernel"] == "pair" and pw["fused"]
    h2, h1, hx, hw = q2.to_numpy(), q1.to_numpy(), qx.to_numpy(), qw.to_numpy()
    assert _rel(gx, _product(orc.dequant(h2), orc.dequant(hw))) <= 1e-3
    assert _rel(gw, _product(orc.dequant(h1).T, orc.dequant(hx))) <= 1e-3


@pytest.mark.parametrize("n,c,d", [(2063, 4112, 528), (2100, 1040, 1024)])
def test_forward_pair_edges(n, c, d):
    from paper_2010_14298_gb300 import fqt
    g = wl.rng(91 + n)
    X = torch.from_numpy(g.standard_normal((n, d)).astype(np.float32)).cuda()
    W = torch.from_numpy((0.05 * g.standard_normal((c, d))).astype(np.float32)).cuda()
    qx, qw = fqt.quantize_act(X, 8, row_sum=True), fqt.quantize_weight(W, 8, row_sum=True)
    ws = fqt.Workspace(n, c, d)
    H = fqt.linear_forward(qx, qw, ws=ws)
    assert fqt.sync_status(ws) == 0
    assert fqt.debug_last_plan()["kernel"] == "pair"
    assert _rel(H, _product(orc.dequant(qx.to_numpy()), orc.dequant(qw.to_numpy()).T)) <= 1e-3


@pytest.mark.parametrize("n,h,w,c,cout", [(128, 14, 14, 256, 272), (130, 9, 13, 192, 320)])
def test_conv_grad_w_pair_edges(n, h, w, c, cout):
    """The implicit im2col operand on CTA pairs: bit-equal to the explicit one."""
    from paper_2010_14298_gb300 import fqt
    g = wl.rng(55)
    x = g.uniform(-1, 1, (n, h, w, c)).astype(np.float32)
    X = torch.from_numpy(wl.im2col_nhwc(x, 3, 3, 1, 1)).cuda()
    dH = torch.from_numpy(wl.random_grad(g, n * h * w, cout)).cuda()
    _, q1 = fqt.quantize_grad(dH, fqt.PSQ, 8, 0, seed=1)
    qx = fqt.quantize_act(X, 8)
    qi = fqt.quantize_act_conv(torch.from_numpy(x).cuda(), 3, 3, 1, 8)
    ws = fqt.Workspace(n * h * w, cout, 9 * c)
    _, ge = fqt.linear_backward(q1, q1, qx, None, grad_x=False, ws=ws)
    _, gi = fqt.linear_backward(q1, q1, qi, None, grad_x=False, ws=ws)
    assert fqt.sync_status(ws) == 0
    assert fqt.debug_last_plan(grad_w=True)["kernel"] == "pair"
    assert _rel(ge, _product(orc.dequant(q1.to_numpy()).T, orc.dequant(qx.to_numpy()))) <= 1e-3
    assert torch.equal(gi, ge)


@pytest.mark.parametrize("n,c,d,kernel", [(2100, 1024, 4112, "pair"), (4100, 256, 6160, "pair"),
                                          (1638, 64, 12880, "wide"), (300, 128, 30656, "wide")])
@pytest.mark.parametrize("bits", [5, 8])
def test_shifted_codes_grad_w(n, c, d, kernel, bits):
    """The shift quantizer's wide codes (exact chunks of one to eight K blocks)."""
    from paper_2010_14298_gb300 import fqt
    g = wl.rng(3 + n)
    dH = torch.from_numpy(wl.random_grad(g, n, c)).cuda()
    X = torch.from_numpy(g.uniform(-1, 1, (n, d)).astype(np.float32)).cuda()
    qx = fqt.quantize_act(X, 8)
    qs, _ = fqt.quantize_grad(dH, fqt.SHIFT, bits, 0, seed=3, with_b1=False)
    ws = fqt.Workspace(n, c, d)
    _, gw = fqt.linear_backward(qs, None, qx, None, grad_x=False, ws=ws)
    assert fqt.sync_status(ws) == 0
    assert fqt.debug_last_plan(grad_w=True)["kernel"] == kernel
    a = qs.shift16.double() * qs.shift_scale[0].double()
    x = torch.from_numpy(orc.dequant(qx.to_numpy())).cuda()
    assert _rel(gw, (a.T @ x).cpu().numpy()) <= 1e-3
