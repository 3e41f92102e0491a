"""The statistics and code passes of the gradient quantizers at the edges of
their layouts (rows of one oct, odd octs, one column past and short of a slab
or a team, the widest; blocks of 4, 8, 16 with a ragged last one; units of 8
rows and column splits), and the one-pass quantizers that a workspace without
their scratch takes: codes against the oracle (PTQ, PSQ equal; BHQ within +-1
at a rounding threshold), sums equal to those of the codes."""
import numpy as np
import pytest
import torch

import oracle as orc
from paper_2010_14298_gb300 import fqt
from paper_2010_14298_gb300 import workloads as wl
from gpu_util import to_dev
from test_gpu_parity import _check_b1, _check_bhq_codes

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="no GPU")]


def _check(n, c, kind, bits, block, dtype, ws=None, seed=99):
    g = wl.rng(n * 7 + c)
    dH = wl.random_grad(g, n, c)
    if dtype == "bf16":
        dH = wl.to_bf16_values(dH)
    ws = ws or fqt.Workspace(n, c, 16)
    q2, q1 = fqt.quantize_grad(to_dev(dH, dtype), kind, bits, block, seed, ws=ws)
    assert fqt.sync_status(ws) == 0
    ref = orc.quantize_grad(dH, kind, bits, block, seed, orc.STREAM_B2, want_v=True)
    h2 = q2.to_numpy()
    assert torch.equal(q2.codes, q2.codes_from_f16())
    assert np.array_equal(h2["row_sum"], h2["codes"].astype(np.int64).sum(1))
    if kind == orc.BHQ:
        assert np.array_equal(h2["lead"], ref["lead"])
        _check_bhq_codes(h2["codes"], ref["codes"], ref["v"], seed)
        assert np.allclose(h2["inv_s"], ref["inv_s"], rtol=1e-6, atol=0)
        assert np.allclose(h2["zero"], ref["zero"], rtol=1e-5, atol=1e-4)
    else:
        assert np.array_equal(h2["codes"], ref["codes"])
        assert np.array_equal(h2["inv_s"], ref["inv_s"])
        assert np.array_equal(h2["zero"], ref["zero"])
    _check_b1(q1, dH, seed)


WIDTHS = [8, 24, 64, 72, 136, 248, 264, 336, 520, 1008, 1032, 2056, 4088]


@pytest.mark.parametrize("c", WIDTHS)
@pytest.mark.parametrize("block,dtype", [(4, "f32"), (8, "bf16"), (16, "f32"), (16, "bf16")])
def test_bhq_widths(c, block, dtype):
    _check(5 * 16 + 7, c, orc.BHQ, 5, block, dtype)


@pytest.mark.parametrize("n,c,block,dtype", [
    (33, 40, 32, "f32"), (200, 56, 128, "bf16"), (777, 72, 64, "bf16"), (129, 136, 128, "f32"),
    (300, 264, 32, "f32"), (131, 1008, 64, "bf16"), (64, 1024, 64, "f32"), (95, 2048, 32, "f32"),
    (1, 64, 32, "f32")])
def test_bhq_big_blocks(n, c, block, dtype):
    _check(n, c, orc.BHQ, 5, block, dtype)


@pytest.mark.parametrize("n,c", [(1523, 40), (700, 80), (240003, 40), (1523, 128), (1523, 200), (301, 1008),
                                 (301, 1512), (200, 2048), (70, 4096)])
@pytest.mark.parametrize("block", [4, 8, 16, 32, 64, 128])
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_bhq_passes_equal_the_one_pass_quantizer(n, c, block, dtype):
    """A workspace without the passes' scratch takes the one-pass quantizers:
    every output equal, whichever kernels serve the shape."""
    if block * c > 65536:
        pytest.skip("blocks of this width are refused")
    always = c >= 64 and not c & (c - 1) and (block == 16 or (dtype == "f32" and block < 16))
    if always:
        pytest.skip("these shapes refuse the smaller workspace")
    x = to_dev(wl.random_grad(wl.rng(n + c + block), n, c), dtype)
    small = fqt.Workspace(1, 16, 16)
    small.nbytes = 256 + 32768  # the header and the range partials
    a2, a1 = fqt.quantize_grad(x, orc.BHQ, 8, block, 5, ws=fqt.Workspace(n, c, 16))
    b2, b1 = fqt.quantize_grad(x, orc.BHQ, 8, block, 5, ws=small)
    for f in ("codes", "inv_s", "zero", "row_sum", "lead", "hz", "hr"):
        assert torch.equal(getattr(a2, f), getattr(b2, f)), f
    for f in ("codes", "inv_s", "zero", "col_sum"):
        assert torch.equal(getattr(a1, f), getattr(b1, f)), f


@pytest.mark.parametrize("c", WIDTHS + [8192, 8200])
@pytest.mark.parametrize("kind,bits,dtype", [(orc.PTQ, 8, "f32"), (orc.PSQ, 8, "bf16"),
                                             (orc.PSQ, 4, "f32")])
def test_affine_widths(c, kind, bits, dtype):
    _check(61, c, kind, bits, 0, dtype)


@pytest.mark.parametrize("n,c,kind,block", [(1, 64, orc.BHQ, 4), (3, 128, orc.PSQ, 0),
                                            (9000, 80, orc.BHQ, 8), (9000, 80, orc.PTQ, 0)])
def test_row_counts(n, c, kind, block):
    _check(n, c, kind, 5, block, "f32")


@pytest.mark.parametrize("n,c,block,dtype", [(1523, 16, 2, "bf16"), (1100, 8, 2, "f32"),
                                             (2500, 8, 2, "bf16")])
def test_more_blocks_than_threads_per_unit(n, c, block, dtype):
    """Narrow rows: a staged unit of k_quant2 holds up to 1024 blocks, more than
    its CTA has threads."""
    _check(n, c, orc.BHQ, 5, block, dtype)


@pytest.mark.parametrize("c,kind,block", [(336, orc.PSQ, 0), (1008, orc.BHQ, 16)])
def test_small_workspace_takes_the_one_pass_quantizer(c, kind, block):
    ws = fqt.Workspace(1, 16, 16)
    ws.nbytes = 256 + 32768  # the header and the range partials
    _check(200, c, kind, 5, block, "f32", ws)


@pytest.mark.parametrize("rows,cols", [(5, 8), (67, 16), (200, 64), (33, 128), (70, 256),
                                       (41, 768), (9, 8192), (50, 24), (50, 1104)])
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_forward_row_sums(rows, cols, dtype):
    g = wl.rng(rows + cols)
    X = g.standard_normal((rows, cols)).astype(np.float32)
    X = wl.to_bf16_values(X) if dtype == "bf16" else X
    q = fqt.quantize_act(to_dev(X, dtype), 8, row_sum=True)
    codes = q.to_numpy()["codes"].astype(np.int64)
    assert np.array_equal(codes, orc.quantize_fwd(X, 8)["codes"])
    assert np.array_equal(q.row_sum.cpu().numpy(), codes.sum(1))
    assert np.array_equal(q.col_sum.cpu().numpy(), codes.sum(0))


@pytest.mark.parametrize("n", [3, 6, 37, 515, 3001])
@pytest.mark.parametrize("c,rows,dtype", [(64, "equal", "f32"), (64, "outliers", "bf16"),
                                          (64, "lognormal", "f32"), (128, "outliers", "f32")])
def test_adaptive_group_sizes(n, c, rows, dtype):
    """Groups of one to four rows side by side, larger ones alone, in one call."""
    g = wl.rng(n + c)
    dH = wl.random_grad(g, n, c, {"equal": 0.0, "outliers": 0.3, "lognormal": 2.0}[rows],
                        0.05 if rows == "outliers" else 0.0)
    if dtype == "bf16":
        dH = wl.to_bf16_values(dH)
    q2, q1 = fqt.quantize_grad(to_dev(dH, dtype), orc.BHQ, 5, 0, 11)
    ref = orc.quantize_grad(dH, orc.BHQ, 5, 0, 11, orc.STREAM_B2, want_v=True)
    h2 = q2.to_numpy()
    assert np.array_equal(h2["perm"], ref["perm"])
    _check_bhq_codes(h2["codes"], ref["codes"], ref["v"], 11)
    assert np.array_equal(h2["row_sum"], h2["codes"].astype(np.int64).sum(1))
    assert np.allclose(h2["zero"], ref["zero"], rtol=1e-5, atol=1e-4)
    _check_b1(q1, dH, 11)


@pytest.mark.parametrize("n,c,d", [(130, 16, 16), (3000, 24, 40), (777, 136, 200), (9001, 72, 24),
                                   (40000, 16, 48), (60001, 336, 56)])
def test_grad_w_reduction_shapes(n, c, d):
    """Splits that do not divide into their groups, row lengths off a vector."""
    g = wl.rng(n)
    c, d = (c + 15) // 16 * 16, (d + 15) // 16 * 16
    dH = to_dev(wl.random_grad(g, n, c), "f32")
    X = to_dev(g.uniform(-1, 1, (n, d)).astype(np.float32), "f32")
    _, q1 = fqt.quantize_grad(dH, orc.PSQ, 5, 0, 2)
    qx = fqt.quantize_act(X, 8)
    ws = fqt.Workspace(n, c, d)
    _, gw = fqt.linear_backward(q1, q1, qx, None, grad_x=False, ws=ws)
    assert fqt.sync_status(ws) == 0
    ref = (torch.from_numpy(orc.dequant(q1.to_numpy())).cuda().T.double()
           @ torch.from_numpy(orc.dequant(qx.to_numpy())).cuda().double()).cpu().numpy()
    got = gw.double().cpu().numpy()
    floor = 1e-3 * np.abs(ref).max(axis=1, keepdims=True)
    assert (np.abs(got - ref) / np.maximum(np.abs(ref), floor)).max() <= 1e-3


@pytest.mark.parametrize("n,c,kind,block,small", [
    (200, 136, orc.PTQ, 0, False), (200, 136, orc.PSQ, 0, False), (200, 136, orc.PSQ, 0, True),
    (200, 136, orc.BHQ, 16, False), (200, 136, orc.BHQ, 16, True), (200, 16, orc.BHQ, 2, False),
    (200, 64, orc.BHQ, 16, False), (200, 64, orc.BHQ, 0, False), (300, 256, orc.BHQ, 0, False),
    (200, 64, orc.SHIFT, 0, False)])
@pytest.mark.parametrize("scale", [1e-31, 1e-33, 1e-36])
def test_tiny_ranges(n, c, kind, block, small, scale):
    """Ranges whose scale B / R is far above 2^112: the codes of every kernel are
    the oracle's (adaptive groups: of Q_b1, whose rows no grouping orders)."""
    dH = (wl.random_grad(wl.rng(5), n, c, 0.0, 0.0) * np.float32(scale)).astype(np.float32)
    ws = fqt.Workspace(n, c, 16)
    if small:
        ws = fqt.Workspace(1, 16, 16)
        ws.nbytes = 256 + 32768  # the header and the range partials
    q2, q1 = fqt.quantize_grad(to_dev(dH, "f32"), kind, 5, block, 7, ws=ws)
    assert fqt.sync_status(ws) == 0
    ref = orc.quantize_grad(dH, orc.PTQ, 8, 0, 7, orc.STREAM_B1)
    assert np.array_equal(q1.to_numpy()["codes"], ref["codes"])
    if kind != orc.BHQ:
        ref = orc.quantize_grad(dH, kind, 5, block, 7, orc.STREAM_B2)
        assert np.array_equal(q2.to_numpy()["codes"], ref["codes"])
    elif block:
        ref = orc.quantize_grad(dH, kind, 5, block, 7, orc.STREAM_B2, want_v=True)
        _check_bhq_codes(q2.to_numpy()["codes"], ref["codes"], ref["v"], 7)


@pytest.mark.parametrize("n,c,block", [(50, 48, 1), (50, 64, 4), (50, 48, 16), (200, 64, 16),
                                       (77, 64, 32), (777, 64, 128), (61, 1040, 16), (200, 16, 2),
                                       (300, 64, 0), (300, 256, 0)])
@pytest.mark.parametrize("scale", [1e-37, 1e-39, 1e-43])
def test_bhq_of_subnormal_gradients(n, c, block, scale):
    """Blocks whose scales s1, s2 = O(B / lambda) overflow fp32 hold zeros, so
    that their rows of grad_X are zeros and not NaN."""
    g = wl.rng(8)
    dH = (wl.random_grad(g, n, c, 0.0, 0.0) * np.float32(scale)).astype(np.float32)
    dH[: n // 4] = 0.0
    X = to_dev(g.standard_normal((n, 32)).astype(np.float32), "f32")
    W = to_dev(g.standard_normal((c, 32)).astype(np.float32), "f32")
    ws = fqt.Workspace(n, c, 32)
    q2, q1 = fqt.quantize_grad(to_dev(dH, "f32"), orc.BHQ, 5, block, 7, ws=ws)
    gx, gw = fqt.linear_backward(q2, q1, fqt.quantize_act(X, 8), fqt.quantize_weight(W, 8), ws=ws)
    assert fqt.sync_status(ws) == 0
    for t in (q2.inv_s, q2.zero, *([] if block == 1 else [q2.hz, q2.hr])):
        assert torch.isfinite(t).all()
    codes = q2.to_numpy()["codes"].astype(np.int64)
    assert np.array_equal(q2.row_sum.cpu().numpy(), codes.sum(1))
    # |grad_X| <= c max|dH| max|W| (1 + 1 / B), with room for the transform
    bound = 4.0 * c * float(np.abs(dH).max()) * float(W.abs().max())
    assert torch.isfinite(gx).all() and float(gx.abs().max()) <= bound
    assert torch.isfinite(gw).all()
