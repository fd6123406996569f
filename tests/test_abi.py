"""Host-only checks of the C-ABI boundary: the library loads, exports every symbol the header
declares, and rejects bad arguments before any launch (no GPU needed)."""
import ctypes
import os
import re

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def lib():
    from paper_2605_08565_b200 import build
    build.build()
    from paper_2605_08565_b200 import binding
    return binding.load_library()


def _declared_functions():
    text = open(os.path.join(ROOT, "include", "mxq.h")).read()
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    return sorted(set(re.findall(r"\b(mxq_[a-z0-9_]+)\s*\(", text)))


def test_every_declared_symbol_is_exported(lib):
    from paper_2605_08565_b200 import binding
    names = _declared_functions()
    assert len(names) >= 11
    for n in names:
        assert hasattr(lib, n), n
    assert sorted(binding.EXPORTS) == names


def test_version_and_status_strings(lib):
    assert lib.mxq_version() >= 100
    for s in range(0, 8):
        assert lib.mxq_status_string(s)
    assert lib.mxq_status_string(0) == b"ok"
    assert lib.mxq_global_scale_from_amax(2688.0) == 1.0
    assert lib.mxq_global_scale_from_amax(0.0) == 1.0
    assert lib.mxq_tensor_mse_workspace_bytes(10) >= 8


def test_argument_errors_are_caught_on_the_host(lib):
    # fake, 16-byte aligned "device" addresses: validation must fail before anything is launched
    X, C, S, E = 0x10000, 0x20000, 0x30000, 0x40000
    q = lib.mxq_quantize_ex
    ok_args = dict(x=X, dtype=0, n=64, B=16, fmt=1, recipe=0, g=1.0, dg=0, codes=C, scales=S, sse=E, stream=0)

    def call(**kw):
        a = dict(ok_args)
        a.update(kw)
        return q(a["x"], a["dtype"], a["n"], a["B"], a["fmt"], a["recipe"], a["g"], a["dg"], a["codes"], a["scales"],
                 a["sse"], a["stream"])

    assert call(x=0) == 1 and call(codes=0) == 1 and call(scales=0) == 1
    assert call(dtype=2) == 2 and call(fmt=3) == 2 and call(fmt=-1) == 2 and call(recipe=6) == 2
    assert call(B=3) == 3 and call(B=128) == 3 and call(n=0) == 3 and call(n=60) == 3
    assert call(x=X + 4) == 4 and call(codes=C + 8) == 4 and call(sse=E + 4) == 4
    assert call(g=0.0) == 5 and call(g=-1.0) == 5 and call(g=float("inf")) == 5 and call(g=float("nan")) == 5
    assert lib.mxq_tensor_mse(E, 4, 64, 0x50000, 0, 0, 0) == 6
    assert lib.mxq_tensor_mse(E, 4, 64, 0x50000, 0x60000, 8, 0) == 6
    assert lib.mxq_tensor_mse(0, 4, 64, 0x50000, 0x60000, 8192, 0) == 1
    assert lib.mxq_tensor_amax(0, 0, 64, E, 0, 0) == 1
    assert lib.mxq_tensor_amax(X, 5, 64, E, 0, 0) == 2
    assert lib.mxq_dequantize(C, S, 64, 16, 1, 1.0, 0, 0, 0) == 1
    assert lib.mxq_dequantize(C, S, 64, 5, 1, 1.0, X, 0, 0) == 3
    assert lib.mxq_dequantize(C, S, 64, 16, 1, 0.0, X, 0, 0) == 5
    assert lib.mxq_dequantize_ex(C, S, 64, 16, 1, 0.0, 0, X, 0, 0) == 5
    assert lib.mxq_dequantize_ex(C, S, 64, 16, 1, 0.0, E + 2, X, 0, 0) == 4     # misaligned device scale
    assert lib.mxq_dequantize_ex(C, S, 64, 16, 1, 0.0, E, 0, 0, 0) == 1
    qm = lib.mxq_quantize_mse
    assert qm(X, 0, 64, 16, 1, 0, 1.0, 0, C, S, E, 0, 0x60000, 8192, 0) == 1           # no MSE output
    assert qm(X, 0, 64, 16, 1, 0, 1.0, 0, C, S, E, 0x50000, 0, 8192, 0) == 6           # no workspace
    assert qm(X, 0, 64, 16, 1, 0, 1.0, 0, C, S, E, 0x50000, 0x60000, 4096, 0) == 6     # workspace too small
    assert qm(X, 0, 60, 16, 1, 0, 1.0, 0, C, S, E, 0x50000, 0x60000, 8192, 0) == 3
    assert qm(X, 0, 64, 16, 1, 0, 1.0, 0, C, S, E, 0x50004, 0x60000, 8192, 0) == 4


def test_binding_refuses_cpu_tensors():
    import torch
    from paper_2605_08565_b200 import binding
    x = torch.zeros(64)
    with pytest.raises(binding.MxqError):
        binding.quantize(x, 16, binding.MXQ_SF_UE4M3, binding.MXQ_ABSMAX)


def test_native_calls_hand_on_what_they_do_not_know(lib):
    """The extension module answers -1 to anything but contiguous CUDA tensors (or None), ints and floats, and the library's status
    otherwise; the binding then raises what its ctypes call raises."""
    import torch

    from paper_2605_08565_b200 import binding
    native = binding._native

    class Stream:
        cuda_stream = 0
    s = Stream()
    x = torch.zeros(64)
    assert native.quantize_ex(x, 64, 16, 1, 0, 1.0, None, x, x, None, s) == -1       # a CPU tensor
    assert native.segment_mse(None, 1, 1, 1, None, s) == 1                           # the library: a pointer is missing
    assert native.segment_mse(None, 1, 1, 1.0, None, s) == -1
    assert native.segment_mse(None, -1, 1, 1, None, s) == -1
    assert native.segment_mse(None, 1, 1, 1, None, None) == -1                       # no tensor to take the stream from
    assert native.segment_mse(None, 1, 1, 1) == -1
    assert native.segment_mse(object(), 1, 1, 1, None, s) == -1
    with pytest.raises(binding.MxqError, match="CUDA tensors only"):
        binding.mxq_quantize_ex(x, 64, 16, 1, 0, 1.0, None, x, x, None)
    with pytest.raises(binding.MxqError, match="status 1"):
        binding.mxq_segment_mse(None, 1, 1, 1, None, stream=s)
    with pytest.raises(binding.MxqError, match="status 2"):
        binding.mxq_set_option(7, 1)
    assert binding.mxq_get_option(binding.MXQ_OPT_BRUTE_PRUNE) == 0


def test_only_the_static_mse_keeps_a_device_address(lib):
    """A device address kept on the host outlives the context that it belongs to.  The library keeps one per device, that of the scratch
    array of mxq_tensor_mse_static(); the slots of the tensor abs-max are handed to their kernel by number."""
    import subprocess
    from paper_2605_08565_b200 import binding
    names = subprocess.run(["nm", "-C", binding.LIB_PATH], capture_output=True, text=True, check=True).stdout.splitlines()
    kept = [n for n in names if n.endswith("of_device")]
    assert len(kept) == 1 and "launch_tensor_mse_static" in kept[0], kept


def test_the_binding_works_without_the_extension_module(lib, tmp_path, monkeypatch):
    """The extension only unpacks arguments: a package without it loads, warns once and answers through ctypes; a build in which it
    fails still delivers the library."""
    import shutil
    import subprocess
    import sys
    from paper_2605_08565_b200 import binding, build
    copy = tmp_path / "paper_2605_08565_b200"
    copy.mkdir()
    for f in os.listdir(os.path.dirname(binding.__file__)):
        if f.endswith(".py"):
            shutil.copy(os.path.join(os.path.dirname(binding.__file__), f), copy)
    code = """
import warnings
import torch
from paper_2605_08565_b200 import binding
with warnings.catch_warnings(record=True) as w:
    warnings.simplefilter("always")
    binding.load_library()
    binding.load_library()
assert len(w) == 1 and "_native" in str(w[0].message), [str(x.message) for x in w]
def refused(f, text):
    try:
        f()
    except binding.MxqError as e:
        assert text in str(e), e
    else:
        raise AssertionError(text)
class Stream:
    cuda_stream = 0
x = torch.zeros(64)
refused(lambda: binding.mxq_quantize_ex(x, 64, 16, 1, 0, 1.0, None, x, x, None), "CUDA tensors only")
refused(lambda: binding.mxq_segment_mse(None, 1, 1, 1, None, stream=Stream()), "status 1")
refused(lambda: binding.mxq_set_option(7, 1), "status 2")
binding.mxq_set_option(binding.MXQ_OPT_BRUTE_PRUNE, 1)
assert binding.mxq_get_option(binding.MXQ_OPT_BRUTE_PRUNE) == 1
"""
    r = subprocess.run([sys.executable, "-c", code], cwd=tmp_path, env=dict(os.environ, MXQ_LIB=binding.LIB_PATH), capture_output=True, text=True)
    assert r.returncode == 0, r.stderr

    def fails(*args):
        raise RuntimeError("no compiler")
    monkeypatch.setattr(build, "build_native", fails)
    with pytest.warns(RuntimeWarning, match="no compiler"):
        assert build.build() == build.LIB


def test_the_extension_module_is_of_this_torch_and_python(lib, monkeypatch):
    """The module was compiled against the layout of torch's tensors: its file name carries both versions, and under another torch the
    one that is there is neither loaded nor taken for built."""
    import sysconfig
    import torch
    from paper_2605_08565_b200 import binding, build
    here = build.native_path()
    assert os.path.exists(here) and torch.__version__ in here and here.endswith(sysconfig.get_config_var("EXT_SUFFIX"))
    assert binding._native.__file__ == here
    monkeypatch.setattr(torch, "__version__", "0.0.1")
    assert build.native_path() != here and not os.path.exists(build.native_path())
    with pytest.raises(ImportError):
        binding._import_native()
