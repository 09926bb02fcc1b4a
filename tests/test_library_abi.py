"""The C-ABI library loads and exports every symbol include/cake.h declares
(no compute calls: runs without a GPU)."""
import ctypes
import os
import re
import subprocess
import sys
import sysconfig

import pytest
import torch

from paper_2503_12491_b200 import binding, build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def declared_symbols():
    text = open(os.path.join(ROOT, "include", "cake.h")).read()
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    return sorted(set(re.findall(r"\b(cake_[a-z0-9_]+)\s*\(", text)))


def test_header_and_binding_list_the_same_entry_points():
    assert declared_symbols() == sorted(binding.EXPORTS)


def test_library_builds_loads_and_exports_everything():
    path = build.build()
    lib = ctypes.CDLL(path)
    for name in declared_symbols():
        assert hasattr(lib, name), name
    lib.cake_strerror.restype = ctypes.c_char_p
    lib.cake_strerror.argtypes = [ctypes.c_int32]
    assert lib.cake_strerror(0) == b"ok"
    assert b"order" in lib.cake_strerror(-7)
    lib.cake_launch_count.restype = ctypes.c_int64
    assert lib.cake_launch_count() == 0


def test_config_struct_matches_header_layout():
    # 9 int32, 3 float, int64, int32 (+pad), int64, 2 int32, float (+pad)
    assert ctypes.sizeof(binding.CakeConfig) == 88
    assert binding.CakeConfig.total_budget.offset == 48
    assert binding.CakeConfig.max_total_tokens.offset == 64
    assert binding.CakeConfig.indicator_mode.offset == 72
    assert binding.CakeConfig.alloc_mode.offset == 76
    assert binding.CakeConfig.pyramid_slope.offset == 80


@pytest.mark.parametrize("call", ["clear_unused((None,), (None,))", "clear_unused(iter([None]), iter([None]))",
                                  "clear_unused((torch.zeros(2),), ())", "clear_unused(1, 2)",
                                  "compact(0, -1, True, 0, 0, [], [], None, None, None, None)",
                                  "compact(0, 'x', True, 0, 0, [], [], None, None, None, None)",
                                  "compact_int4(0, -1, True, 32, [], [], *[None] * 9)"])
def test_arguments_the_native_marshalling_cannot_take_raise(call):
    """In a process of their own: a Python error, not the end of the process."""
    code = f"import torch; from paper_2503_12491_b200 import binding; binding.load_library(); binding._fast.{call}"
    r = subprocess.run([sys.executable, "-c", code], cwd=ROOT, capture_output=True, text=True)
    assert r.returncode == 1 and re.search(r"^(TypeError|ValueError): ", r.stderr, flags=re.M), (r.returncode, r.stderr[-300:])


def test_native_half_belongs_to_this_interpreter_and_torch(monkeypatch):
    """The file name has both; what was built for another torch is neither loaded nor taken as up to date."""
    build.build()
    path = build.binding_path()
    assert os.path.exists(path) and torch.__version__ in path and sysconfig.get_config_var("SOABI") in path
    assert binding._load_native().__file__ == path
    monkeypatch.setattr(torch, "__version__", torch.__version__ + ".other")
    assert build.binding_path() != path
    with pytest.raises(ImportError, match="build it with"):
        binding._load_native()


def test_argument_errors_need_no_gpu():
    lib = binding.load_library()
    assert lib.cake_create(None, None) == binding.CAKE_ERR_ARG
    h = ctypes.c_void_p()
    bad = binding.CakeConfig(4, 4, 3, 64, 16, 5, 0, 0, 0, 1.0, 1.0, 1.0, 512, 1, 512)   # 4 % 3 != 0
    assert lib.cake_create(ctypes.byref(bad), ctypes.byref(h)) == binding.CAKE_ERR_ARG
    small = binding.CakeConfig(4, 4, 4, 64, 16, 5, 0, 0, 0, 1.0, 1.0, 1.0, 63, 1, 512)  # B < L*S_w
    assert lib.cake_create(ctypes.byref(small), ctypes.byref(h)) == binding.CAKE_ERR_BUDGET
    even = binding.CakeConfig(4, 4, 4, 64, 16, 4, 0, 0, 0, 1.0, 1.0, 1.0, 512, 1, 512)  # even kernel
    assert lib.cake_create(ctypes.byref(even), ctypes.byref(h)) == binding.CAKE_ERR_ARG
    mode = binding.CakeConfig(4, 4, 4, 64, 16, 5, 0, 0, 0, 1.0, 1.0, 1.0, 512, 1, 512, 5)  # no such indicator
    assert lib.cake_create(ctypes.byref(mode), ctypes.byref(h)) == binding.CAKE_ERR_ARG
    alloc = binding.CakeConfig(4, 4, 4, 64, 16, 5, 0, 0, 0, 1.0, 1.0, 1.0, 512, 1, 512, 0, 3)  # no such allocation
    assert lib.cake_create(ctypes.byref(alloc), ctypes.byref(h)) == binding.CAKE_ERR_ARG
    slope = binding.CakeConfig(4, 4, 4, 64, 16, 5, 0, 0, 0, 1.0, 1.0, 1.0, 512, 1, 512, 0, 2, 1.5)
    assert lib.cake_create(ctypes.byref(slope), ctypes.byref(h)) == binding.CAKE_ERR_ARG
    assert lib.cake_begin(None, 0, None, None) == binding.CAKE_ERR_ARG
    assert lib.cake_allocate(None, 0, None) == binding.CAKE_ERR_ARG
