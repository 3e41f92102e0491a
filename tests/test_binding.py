"""The native argument marshalling takes and refuses what QTensor.c_struct, the
ctypes marshalling of the other calls, takes and refuses (no GPU: every call
here is refused before the library would start a kernel)."""
import os
import subprocess
import sys
import sysconfig
import types
from shutil import which

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2010_14298_gb300 import build, fqt  # noqa: E402

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


# --- the extension module is built for one interpreter, and can be absent ---
def test_the_extension_module_serves_the_calls_here():
    """Built by this interpreter, under a name that no other one loads."""
    assert isinstance(fqt.native(), types.ModuleType)
    assert build.PYEXT.endswith(sysconfig.get_config_var("EXT_SUFFIX"))


@pytest.fixture
def no_extension(monkeypatch, tmp_path):
    """The library is built, the extension module is not and cannot be."""
    build.build()
    monkeypatch.setattr(build, "PYEXT", str(tmp_path / "_fqt_py.so"))
    monkeypatch.setattr(build.shutil, "which",
                        lambda name, *a: None if name in ("cc", "gcc") else which(name, *a))
    monkeypatch.setenv("PATH", str(tmp_path))
    monkeypatch.setattr(fqt, "_native", None)


def test_build_leaves_a_whole_library_without_a_c_compiler(no_extension):
    with pytest.warns(RuntimeWarning):
        assert build.build() == build.LIB


def test_the_library_loads_without_the_extension_module(no_extension, monkeypatch):
    monkeypatch.setattr(fqt, "_lib", None)
    monkeypatch.setattr(build, "build", lambda *a, **k: pytest.fail("the library was rebuilt"))
    assert fqt.load(build_if_missing=False).fqt_workspace_size(4, 8, 16) > 0


def test_the_calls_are_made_through_ctypes_without_the_extension_module(no_extension):
    want = fqt.workspace_size(1000, 64, 576)
    with pytest.warns(RuntimeWarning):
        calls = fqt.native()
    assert calls.workspace_size(1000, 64, 576) == want
    assert _marshal(_qtensor()) == 1
    _same_refusal(_qtensor(logical=(4, 8, 1)))
    q, ws = _qtensor(), fqt.Workspace(4, 16, 16, device="cpu")
    with pytest.raises(fqt.FqtError) as e:  # k = 5 is not built
        fqt.conv_grad_x_nhwc(q, q, 1, 2, 2, 32, k=5, ws=ws, stream=STREAM,
                             out=torch.zeros(1, 2, 2, 32))
    assert e.value.status in (1, 2)
    with pytest.raises(fqt.FqtError) as e:  # W~ of other rows than dH's columns
        fqt.linear_backward(q, None, None, q, grad_w=False, ws=ws, stream=STREAM)
    assert e.value.status in (1, 2, 6)
