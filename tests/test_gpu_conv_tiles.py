"""grad_X in NHWC (col2im fused) at the edges of its tiles: several small
images per tile with a last partial one, uneven last rows, one row per tile at
the widest images, one 64-wide W~ atom kept resident against the ring, several
channel tiles; against the oracle fed the GPU's codes, to the bar of the other
grad_X tests (max |g - r| / max(|r|, 1e-3 ||r_row||_inf) <= 1e-3).  The bar's
floor amplifies the fp32 rounding of the offset term y R_p: three roundings of
2^-24 |y R_p| against 1e-3 of the row stay below it while |y R_p| is up to
5.6 times the row's largest entry."""
import numpy as np
import pytest
import torch

import oracle as orc
from paper_2010_14298_gb300 import fqt
from gpu_util import grad_rel_err
from test_gpu_conv_nhwc import _operands, _oracle

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="no GPU")]


@pytest.mark.parametrize("n,h,w,cin,cout,kind,bits", [
    (7, 7, 7, 64, 64, orc.PSQ, 5), (11, 2, 3, 32, 64, orc.PSQ, 5), (2, 5, 128, 64, 64, orc.PSQ, 5),
    (2, 57, 55, 64, 64, orc.PTQ, 8), (3, 30, 9, 160, 128, orc.PSQ, 5),
    (1, 64, 64, 32, 192, orc.PTQ, 4), (160, 8, 8, 64, 64, orc.PSQ, 5)])
def test_conv_grad_x_tiles(n, h, w, cin, cout, kind, bits):
    _, _, q2, qw = _operands(n, h, w, cin, cout, kind, bits)
    ws = fqt.Workspace(n * h * w, cout, 9 * cin)
    out = fqt.conv_grad_x_nhwc(q2, qw, n, h, w, cin, ws=ws)
    assert fqt.sync_status(ws) == 0
    ref = _oracle(q2, qw, n, h, w, cin, kind)
    got = out.cpu().numpy()
    assert np.isfinite(got).all()
    assert grad_rel_err(got.reshape(-1, cin), ref.reshape(-1, cin)) <= 1e-3
