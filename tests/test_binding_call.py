"""The binding's argument marshalling, by csrc/pycall.c and by ctypes where that is not built, without a device: every entry point rejects
these arguments before it launches anything."""
import ctypes
import os
import subprocess
import sys

import pytest
import torch

from paper_2606_26453_b200 import build


@pytest.fixture(params=["C", "ctypes"])
def B(request, monkeypatch):
    build.build_library()
    from paper_2606_26453_b200 import binding
    lib = binding.load_library()
    from paper_2606_26453_b200 import _pycall
    assert lib.native_call is _pycall.call
    if request.param == "ctypes":
        monkeypatch.setattr(lib, "native_call", binding._ctypes_caller(lib))
    return binding


def test_arguments_arrive_in_their_places(B):
    lib, d = B.load_library(), B.dims(256, 256, 512, 8, 2)
    call = lambda name, *a: lib.native_call(lib.addresses[name], d, *a)
    assert call("moe_permute_bwd", None, 256, 256, 0) == 1                      # NULL
    assert call("moe_permute_bwd", 256, 264, 256, 0) == 4                       # misaligned
    t = torch.zeros(64, dtype=torch.uint8)
    start = -t.data_ptr() % 16
    assert call("moe_permute_bwd", 256, 256, t[start + 8:], None) == 4          # a tensor's address
    assert call("moe_permute", *[256] * 8, 8, 0) == 5                           # on the stack: workspace bytes ...
    assert call("moe_layer_fwd_bwd_host", *[256] * 14, 8, 0) == 5               # ... and the last argument but one of the longest call
    # ints, one at a time: row pitch, first column, features (a multiple of 128 that ends inside the pitch)
    for ints, status in (((512, 0, -1), 3), ((512, 0, 0), 3), ((512, 0, 64), 3), ((512, -8, 256), 2), ((512, 4, 256), 2), ((512, 264, 256), 2),
                         ((255, 0, 256), 2), ((256, 8, 256), 2), ((-512, 0, 256), 2)):
        assert call("moe_mxfp8_quantize_tokens", 256, *ints, 256, 256, 256, 0) == status, ints
    d2 = B.MoeDims(256, 200, 512, 8, 2)
    assert lib.native_call(lib.addresses["moe_permute_bwd"], d2, 256, 256, 256, 0) == 3


def test_refused_arguments(B):
    lib, d = B.load_library(), B.dims(256, 256, 512, 8, 2)
    address = lib.addresses["moe_permute_bwd"]
    with pytest.raises(ValueError, match="contiguous"):
        lib.native_call(address, d, torch.zeros(4, 4).t(), 256, 256, 0)
    for bad in (1.5, "x", object()):
        with pytest.raises((TypeError, AttributeError)):
            lib.native_call(address, d, bad, 256, 256, 0)
    with pytest.raises(TypeError):
        lib.native_call(address, b"short", 256, 256, 256, 0)
    with pytest.raises(TypeError):
        lib.native_call(address, d, *[256] * 18)
    with pytest.raises(TypeError):
        B._call("moe_permute_bwd", ctypes.byref(d), 256, 256, 256)
    with pytest.raises(ValueError):
        lib.native_call(0, d, 256)
    with pytest.raises(TypeError):
        lib.native_call((address,), d, 256, 256, 256, 0)


def test_arguments_are_counted(B):
    """A missing or surplus argument would have the callee read what happens to be in a register or on the stack as a pointer."""
    lib, d = B.load_library(), B.dims(256, 256, 512, 8, 2)
    for name in lib.addresses:
        n = len(getattr(lib, name).argtypes) - 1
        assert lib.entries[name] == (lib.addresses[name], n)
        for wrong in {0, n - 1, n + 1}:
            with pytest.raises(TypeError):
                lib.native_call(lib.entries[name], d, *[None] * wrong)
        assert lib.native_call(lib.entries[name], d, *[None] * n) != 0, name


def test_every_entry_point_fits(B):
    lib = B.load_library()
    assert all(len(getattr(lib, name).argtypes) - 1 <= 17 for name in lib.addresses)


def test_without_the_helper():
    """A build for another Python, or none at all: the binding still loads and calls."""
    code = """
import sys
sys.modules["paper_2606_26453_b200._pycall"] = None      # importing it raises ImportError
from paper_2606_26453_b200 import binding as B
lib = B.load_library()
assert lib.native_call.__module__ == B.__name__
assert lib.native_call(lib.entries["moe_permute_bwd"], B.dims(256, 256, 512, 8, 2), 256, 264, 256, 0) == 4
"""
    subprocess.run([sys.executable, "-c", code], check=True, cwd=os.path.dirname(build.PKG_DIR))


@pytest.mark.parametrize("compiler", ["/nonexistent/cc", "false"])
def test_library_is_built_without_a_c_compiler(monkeypatch, tmp_path, compiler):
    monkeypatch.setenv("CC", compiler)
    monkeypatch.setattr(build, "PYCALL_PATH", str(tmp_path / "_pycall.so"))
    monkeypatch.setattr(build, "LIB_PATH", str(tmp_path / "lib.so"))
    monkeypatch.setattr(build, "_compile", lambda path, verbose, waittest: open(path, "w").close())
    with pytest.warns(RuntimeWarning, match="was not built"):
        assert os.path.exists(build.build_library())
    with pytest.raises((OSError, RuntimeError)):
        build.build_pycall()


@pytest.mark.parametrize("name", ["moe_grouped_gemm_down_bwd", "moe_grouped_gemm_gateup_swiglu_bwd"])
def test_combined_calls_look_at_all_arguments_before_the_first_launch(B, name):
    lib, d = B.load_library(), B.dims(256, 256, 512, 8, 2)
    n = lib.entries[name][1] - 1
    for i in range(n):
        for bad, status in ((0, 1), (264, 4)):
            assert lib.native_call(lib.entries[name], d, *[bad if j == i else 256 for j in range(n)], 0) == status, (i, bad)
