"""Argument arrays of the binding: what the native module packs, and what it leaves to the general path."""
import ctypes as C
import os
import re
import shutil
import struct
import subprocess
import sys

import numpy as np
import pytest
import torch

import paper_2511_02647_b200.binding as b

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def words(x, fmt):
    raw = x if isinstance(x, bytes) else bytes(x)
    return list(struct.unpack("%d%s" % (len(raw) // struct.calcsize(fmt), fmt), raw))


@pytest.mark.parametrize("n", [0, 1, 2, 64])
@pytest.mark.parametrize("kind", [list, tuple])
def test_pointers(n, kind):
    ts = kind(torch.empty(3, 4)[i % 3:] for i in range(n))
    assert words(b._ptr_array(ts), "Q") == [t.data_ptr() for t in ts]


def test_pointers_of_what_is_not_a_plain_tensor():
    t, par = torch.empty(2, 2), torch.nn.Parameter(torch.empty(3))
    assert words(b._ptr_array([None, t, par]), "Q") == [0, t.data_ptr(), par.data_ptr()]
    assert b._ptr(None) is None and b._ptr(t) == t.data_ptr() and b._ptr(par) == par.data_ptr() and b._ptr(torch.empty(0)) == 0
    for bad in (torch.empty(2, 3).t(), torch.empty(4)[::2]):
        with pytest.raises(ValueError):
            b._ptr(bad)
        with pytest.raises(ValueError):
            b._ptr_array([t, bad])
    with pytest.raises(AttributeError):
        b._ptr_array([t, 3])


@pytest.mark.parametrize("xs", [[], [0], (1, -1, 2 ** 31 - 1, -2 ** 31), np.arange(5), [np.int64(7), 3], range(4), [True, 2], [2.0, 3]])
def test_int32s(xs):
    assert words(b._i32_array(xs), "i") == [int(x) for x in xs]


def test_int32s_beyond_32_bits_wrap_as_ctypes_does():
    assert words(b._i32_array([2 ** 32 + 5, 1]), "i") == words(bytes((C.c_int32 * 2)(2 ** 32 + 5, 1)), "i")


def in_a_process(code, **env):
    return subprocess.run([sys.executable, "-c", code], cwd=ROOT, env={**os.environ, **env}, capture_output=True, text=True)


LOADED = "any('_fedattn_marshal' in x for x in open('/proc/self/maps'))"


@pytest.mark.parametrize("change,loaded", [("", True), ("torch.__version__ = torch.__version__ + '.1'", False),
                                           ("torch.version.git_version = '0' * 40", False),
                                           ("import sysconfig; sysconfig.get_config_vars()['EXT_SUFFIX'] = '.cpython-399.so'", False)])
def test_module_of_another_torch_or_python_is_not_loaded(change, loaded):
    """The module reads torch's own layouts: the one in the tree is for one torch build and one interpreter."""
    code = """
import torch
%s
try:
    import paper_2511_02647_b200
except ImportError:
    pass
print(%s)
"""
    assert in_a_process(code % (change, LOADED)).stdout.strip() == str(loaded)


def test_package_without_the_module(tmp_path):
    """A library named by FEDATTN_LIBRARY, a package folder without any build: it imports, says so, and packs the same."""
    shutil.copytree(os.path.join(ROOT, "paper_2511_02647_b200"), tmp_path / "paper_2511_02647_b200", ignore=shutil.ignore_patterns("lib"))
    code = """
import sys, warnings
sys.path.insert(0, %r)
with warnings.catch_warnings(record=True) as caught:
    warnings.simplefilter("always")
    import paper_2511_02647_b200.binding as b
import torch
t = torch.empty(3)
assert b.__file__.startswith(%r) and any("marshalling module" in str(w.message) for w in caught)
assert bytes(b._i32_array([1, -2])) == bytes((b.C.c_int32 * 2)(1, -2))
assert bytes(b._ptr_array([t, None])) == bytes((b.C.c_void_p * 2)(t.data_ptr(), None)) and b._ptr(t) == t.data_ptr()
print(b.status_string(0))
""" % (str(tmp_path), str(tmp_path))
    res = in_a_process(code, FEDATTN_LIBRARY=b.library_path())
    assert res.stdout.strip() == "ok", res.stderr


@pytest.mark.parametrize("absent", ["LIB_PATH", "module"])
def test_what_is_missing_is_built(absent, tmp_path, monkeypatch):
    """The test session and smoke() build when either file is absent, not for the library alone."""
    import paper_2511_02647_b200.build as build
    lib, module = tmp_path / "libfedattn.so", tmp_path / "module.so"
    (module if absent == "LIB_PATH" else lib).touch()
    monkeypatch.setattr(build, "LIB_PATH", str(lib))
    monkeypatch.setattr(build, "marshal_path", lambda: str(module))
    assert build.missing() == [str(lib if absent == "LIB_PATH" else module)]
    for path in ("tests/conftest.py", "__graft_entry__.py"):
        with open(os.path.join(ROOT, path)) as f:
            src = f.read()
        assert re.search(r"if \S*\.missing\(\):\n +\S*build\(\)", src) and "path.exists" not in src, path
