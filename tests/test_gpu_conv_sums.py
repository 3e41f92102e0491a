"""Column sums and padding sums of the implicit im2col operand of a 3 x 3, pad
1 conv at the edges of their kernels (images of two rows or columns, channel
counts at and past the shared-memory rule and past one 512-channel group):
equal to the explicit im2col operand's, integer for integer and, for grad_W,
to the fp32 rounding of its last expression."""
import numpy as np
import pytest
import torch

from paper_2010_14298_gb300 import fqt
from paper_2010_14298_gb300 import workloads as wl

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="no GPU")]


@pytest.mark.parametrize("n,h,w,c,dtype", [
    (3, 2, 2, 64, torch.float32), (2, 2, 9, 8, torch.bfloat16), (5, 11, 3, 64, torch.float32),
    (1, 14, 14, 1136, torch.float32), (1, 4, 5, 1144, torch.float32),
    (9, 7, 7, 512, torch.bfloat16)])
def test_conv_column_sums(n, h, w, c, dtype):
    g = wl.rng(5)
    x = torch.from_numpy(g.uniform(-1, 1, (n, h, w, c)).astype(np.float32)).to(dtype)
    X = torch.from_numpy(wl.im2col_nhwc(x.float().numpy(), 3, 3, 1, 1))
    ws = fqt.Workspace(n * h * w, c, 16)
    qe = fqt.quantize_act(X.cuda(), 8)
    for _ in range(2):  # the second call finds the first one's sums in the workspace
        qi = fqt.quantize_act_conv(x.cuda(), 3, 3, 1, 8, ws=ws)
        assert fqt.sync_status(ws) == 0
        assert torch.equal(qi.col_sum[:-1], qe.col_sum)


@pytest.mark.parametrize("n,h,w,cin,cout", [(3, 2, 2, 64, 16), (2, 2, 11, 64, 528),
                                            (40, 9, 5, 64, 1040), (7, 33, 64, 64, 48)])
def test_conv_padding_sums(n, h, w, cin, cout):
    g = wl.rng(6)
    x = g.uniform(-1, 1.5, (n, h, w, cin)).astype(np.float32)
    X = torch.from_numpy(wl.im2col_nhwc(x, 3, 3, 1, 1)).cuda()
    dH = torch.from_numpy(wl.random_grad(g, n * h * w, cout)).cuda()
    _, q1 = fqt.quantize_grad(dH, fqt.PTQ, 8, 0, seed=1)
    ws = fqt.Workspace(n * h * w, cout, 9 * cin)
    qx = fqt.quantize_act(X, 8, ws=ws)
    qi = fqt.quantize_act_conv(torch.from_numpy(x).cuda(), 3, 3, 1, 8, ws=ws)
    _, ge = fqt.linear_backward(q1, q1, qx, None, grad_x=False, ws=ws)
    _, gi = fqt.linear_backward(q1, q1, qi, None, grad_x=False, ws=ws)
    assert fqt.sync_status(ws) == 0
    assert torch.equal(ge, gi)


@pytest.mark.parametrize("n,h,w,cin,cout", [(5, 9, 15, 64, 256), (3, 19, 12, 64, 144),
                                            (3, 39, 6, 64, 256)])
def test_conv_grad_w_fits_its_workspace(n, h, w, cin, cout):
    """Images whose padded slots would be cut into more splits than the
    workspace of fqt_workspace_size holds: fewer splits, the same result."""
    g = wl.rng(7)
    x = g.uniform(-1, 1.5, (n, h, w, cin)).astype(np.float32)
    X = torch.from_numpy(wl.im2col_nhwc(x, 3, 3, 1, 1)).cuda()
    dH = torch.from_numpy(wl.random_grad(g, n * h * w, cout)).cuda()
    _, q1 = fqt.quantize_grad(dH, fqt.PTQ, 8, 0, seed=1)
    ws = fqt.Workspace(n * h * w, cout, 9 * cin)
    qx = fqt.quantize_act(X, 8, ws=ws)
    qi = fqt.quantize_act_conv(torch.from_numpy(x).cuda(), 3, 3, 1, 8, ws=ws)
    _, ge = fqt.linear_backward(q1, q1, qx, None, grad_x=False, ws=ws)
    _, gi = fqt.linear_backward(q1, q1, qi, None, grad_x=False, ws=ws)
    assert fqt.sync_status(ws) == 0
    assert torch.equal(ge, gi)
