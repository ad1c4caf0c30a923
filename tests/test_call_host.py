"""The CPython entry (csrc/hif8_call.cpp) against the same calls through ctypes, on the CPU: argument errors are found
before anything touches a device, so status codes and exceptions can be compared without one."""
import ctypes
import os
import shutil
import subprocess
import sys
import sysconfig

import pytest

import paper_2409_16626_b200 as H
from paper_2409_16626_b200 import _hif8_call as call
from paper_2409_16626_b200 import binding


class Buffer:
    """Something with a data_ptr(), as a tensor."""

    def __init__(self, address):
        self.address = address

    def data_ptr(self):
        return self.address


class Stream:
    cuda_stream = 0


A, B = Buffer(0x10000), Buffer(0x20000)
ENTRIES = ["hif8_encode", "hif8_decode", "hif8_amax", "hif8_amax_scale_encode", "hif8_amax_scale_encode_static", "hif8_fake_quant",
           "hif8_gemm", "hif8_gemm_ex", "hif8_gemm_channel_scaled", "hif8_channel_amax_scale_encode", "hif8_delayed_scale_encode",
           "hif8_encode_transpose", "hif8_encode_from_amax", "hif8_als_update", "hif8_check_finite"]
CASES = [  # refused for their arguments (n = 0 and empty products: accepted without a launch)
    ("hif8_encode", (A, 7, B, 16, 0, 0, 0, 0, 0)), ("hif8_encode", (A, 0, B, 16, 127, 0, 0, 0, 0)), ("hif8_encode", (None, 0, B, 16, 0, 0, 0, 0, 0)),
    ("hif8_encode", (A, 0, B, 0, 0, 0, 0, 0, 0)), ("hif8_encode", (A, 0, A, 16, 0, 0, 0, 0, Stream())), ("hif8_encode", (A, 0, B, 16, 0, 9, 0, 0, 0)),
    ("hif8_encode", (A, 0, B, 16, 0, 0, 64, 2**64 - 1, 0)), ("hif8_decode", (A, B, 1, 16, -127, 0)), ("hif8_decode", (A, None, 1, 16, 0, 0)),
    ("hif8_decode", (0x10000, 0x10008, 1, 16, 0, 0)), ("hif8_gemm", (A, 16, B, 16, 1, A, 16, 1, 4, 4, 15, None, None, None, 0, 0)),
    ("hif8_gemm", (A, 16, B, 16, True, A, 16, 1, 0, 4, 16, None, None, None, 0, 0)), ("hif8_gemm", (A, 16, B, 16, 1, A, 16, 1, 4, 4, 16, None, None, None, 0, 0)),
    ("hif8_gemm_ex", (A, 16, 0, B, 16, 1, A, 16, 1, 4, 4, 16, None, None, None, 0, Buffer(8), 256, 0)),
    ("hif8_gemm_channel_scaled", (A, 16, B, 16, 1, A, 16, 1, 4, 4, 16, None, None, None, 0, 0)),
    ("hif8_channel_amax_scale_encode", (A, 1, B, -1, 4, 0, 14, 0, 0, 0, None, None, None, 0)),
    ("hif8_delayed_scale_encode", (A, 1, B, 4, 0, 0, 0, None, 0, 14, 0)), ("hif8_check_finite", (A, 5, 4, B, 0)), ("hif8_als_update", (None, B, 0)),
]


def through_ctypes(name, args):
    stream = args[-1] if isinstance(args[-1], int) else args[-1].cuda_stream
    return getattr(binding.lib, name)(*[binding._ptr(a) if t is ctypes.c_void_p else a for a, t in zip(args[:-1], getattr(binding.lib, name).argtypes)], stream)


@pytest.mark.parametrize("name,args", CASES)
def test_same_status(name, args):
    rc = getattr(call, name)(*args)
    assert type(rc) is int and rc == through_ctypes(name, args)


@pytest.mark.parametrize("name", ENTRIES)
def test_prototypes_agree(name):
    """As many arguments as the ctypes prototype: one less is not taken."""
    n = len(getattr(binding.lib, name).argtypes)
    assert getattr(call, name)(*[object()] * n) is None and getattr(call, name)(*[0] * (n - 1)) is None


@pytest.mark.parametrize("bad", ["x", 1.0, [1]])
def test_other_arguments_are_reported_by_ctypes(bad):
    assert call.hif8_encode(A, 0, B, bad, 0, 0, 0, 0, 0) is None
    with pytest.raises(ctypes.ArgumentError):
        H.hif8_encode(A, 0, B, bad, stream=0)
    with pytest.raises(AttributeError):
        H.hif8_encode("x", 0, B, 1, stream=0)


def test_current_stream_is_left_to_torch_before_initialisation():
    call.set_cuda_ready(False)
    assert call.hif8_encode(A, 0, B, 0, 0, 0, 0, 0, None) is None


PACKAGE = os.path.dirname(os.path.abspath(binding.__file__))


def import_elsewhere(tmp_path, files, before=""):
    """`import paper_2409_16626_b200.binding` of a copy that has only these built files, in a process of its own."""
    copy = tmp_path / "paper_2409_16626_b200"
    copy.mkdir()
    for f in ["__init__.py", "binding.py", "build.py"] + files:
        shutil.copy(os.path.join(PACKAGE, f), copy)
    code = before + "import paper_2409_16626_b200 as H, ctypes; print(H.hif8_workspace_bytes(H.WS_GEMM, 0), H.hif8_encode(65536, 7, 131072, 16, stream=0, check=False))"
    return subprocess.run([sys.executable, "-c", code], cwd=tmp_path, capture_output=True, text=True, timeout=300)


def test_entry_is_named_for_its_interpreter():
    tag = sysconfig.get_config_var("EXT_SUFFIX")
    assert os.path.basename(call.__file__) == "_hif8_call" + tag and tag != ".so" and not os.path.exists(os.path.join(PACKAGE, "_hif8_call.so"))


def test_missing_entry_says_how_to_build_it(tmp_path):
    p = import_elsewhere(tmp_path, ["libhif8.so"])
    assert p.returncode != 0 and "ImportError" in p.stderr and "paper_2409_16626_b200.build" in p.stderr


def test_import_with_a_torch_without_cuda(tmp_path):
    p = import_elsewhere(tmp_path, ["libhif8.so", os.path.basename(call.__file__)],
                         "import torch; del torch._C._cuda_getDevice, torch._C._cuda_getCurrentRawStream\n")
    assert p.returncode == 0, p.stderr
    assert p.stdout.split() == ["256", "2"]


def test_errors_and_check():
    with pytest.raises(H.Hif8Error) as e:
        H.hif8_encode(A, 7, B, 16, stream=0)
    assert e.value.status == H.hif8_encode(A, 7, B, 16, stream=0, check=False) == 2
