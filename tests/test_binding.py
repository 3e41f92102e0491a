"""The native argument marshalling takes and refuses what QTensor.c_struct, the
ctypes marshalling of the other calls, takes and refuses (no GPU: every call
here is refused before the library would start a kernel)."""
import os
import subprocess
import sys
import types

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2010_14298_gb300 import fqt  # noqa: E402

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
STREAM = types.SimpleNamespace(cuda_stream=0)


def _qtensor(**fields):
    q = fqt.QTensor.empty(4, 8, fqt.PTQ, 8, device="cpu")
    for k, v in fields.items():
        setattr(q, k, v)
    return q


def _marshal(q):
    """A call that marshals q and that the library refuses (bits = 0)."""
    return fqt.native().quantize_fwd(0, torch.zeros(4, 8), 0, 4, 8, 0, q,
                                     torch.zeros(256, dtype=torch.uint8), 256, 0)


def _same_refusal(q):
    with pytest.raises(Exception) as ref:
        q.c_struct()
    with pytest.raises(ref.type):
        _marshal(q)


def test_a_whole_tensor_is_marshalled():
    _qtensor().c_struct()
    assert _marshal(_qtensor()) == 1  # FQT_EINVAL, from the library


@pytest.mark.parametrize("fields", [
    dict(codes=torch.zeros(2, 2, 8, dtype=torch.uint8)), dict(logical=(4, 8, 1)),
    dict(codes=torch.zeros(32, dtype=torch.uint8)), dict(logical=(4,)), dict(logical=())])
def test_codes_of_other_than_two_dimensions_are_refused(fields):
    _same_refusal(_qtensor(**fields))


@pytest.mark.parametrize("fields", [dict(inv_s=None), dict(zero=None),
                                    dict(codes=None, codes16=None)])
def test_missing_arrays_are_refused(fields):
    _same_refusal(_qtensor(**fields))


def test_missing_operands_and_workspaces_are_refused():
    ws = fqt.Workspace(4, 16, 16, device="cpu")
    with pytest.raises(AttributeError):  # no W~
        fqt.conv_grad_x_nhwc(_qtensor(), None, 1, 2, 2, 32, ws=ws, stream=STREAM,
                             out=torch.zeros(1, 2, 2, 32))
    ws.buf = None
    with pytest.raises(AttributeError):
        fqt.quantize_act(torch.zeros(4, 8), 0, ws=ws, out=_qtensor(), stream=STREAM)


@pytest.mark.parametrize("conv", [(), [], (1, 2, 3), tuple(range(8))])
def test_conv_geometries_are_taken(conv):
    """An empty geometry is an ordinary matrix's, a short one ends in zeros."""
    q = _qtensor(conv=conv)
    q.c_struct()
    assert _marshal(q) == 1


@pytest.mark.parametrize("conv", [tuple(range(9)), (1.5,) * 8, ("a",)])
def test_conv_geometries_that_do_not_fit_are_refused(conv):
    _same_refusal(_qtensor(conv=conv))


@pytest.mark.parametrize("samples", [False, True])
@pytest.mark.parametrize("seed", [1.9, "7", None, torch.tensor(7), torch.tensor([7])])
def test_seeds_that_are_no_integers_are_refused(seed, samples):
    """A tensor too: reading it would wait for the device."""
    dH = torch.zeros(4, 64)
    kw = dict(seed=seed, ws=fqt.Workspace(4, 64, 16, device="cpu"), stream=STREAM,
              q_b2=fqt.QTensor.empty(4, 64, fqt.PTQ, 8, device="cpu"), with_b1=False)
    with pytest.raises(TypeError):
        if samples:
            fqt.quantize_grad_samples(dH, 2, fqt.PTQ, 9, **kw)
        else:
            fqt.quantize_grad(dH, fqt.PTQ, 9, **kw)


@pytest.mark.parametrize("seed", [0, -1, 2 ** 64 - 1, 2 ** 70 + 3, True, np.int64(-5),
                                  np.uint64(2 ** 64 - 1)])
def test_integer_seeds_are_taken_modulo_2_64(seed):
    assert fqt._seed(seed) == int(seed) % 2 ** 64


def test_the_module_imports_without_torchs_cuda_bindings():
    """A PyTorch built without CUDA lacks the raw-stream functions."""
    code = ("import torch\n"
            "for n in ('_cuda_getCurrentRawStream', '_cuda_getDevice'):\n"
            "    delattr(torch._C, n)\n"
            "from paper_2010_14298_gb300 import fqt\n"
            "assert fqt.status_string(0) == 'ok'\n")
    r = subprocess.run([sys.executable, "-c", code], cwd=ROOT, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
