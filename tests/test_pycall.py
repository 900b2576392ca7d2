"""The marshalling extension behind the binding's launching calls: what it takes for an address, a workspace size and a descriptor, seen from
refusals that need no GPU, and from several threads."""
import ctypes
import importlib.machinery
import os
import subprocess
import sys
import sysconfig
import threading

import pytest
import torch

from paper_2609_33916_b200 import binding as mb
from paper_2609_33916_b200 import build


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()


def _decode(desc, ws, **kw):
    q = torch.zeros(64)
    return mb.moa_decode_attn(desc, q, q, q, q, None, ws, check=False, **kw)


def test_descriptors_of_another_type_and_things_without_an_address_are_refused():
    desc = mb.make_decode_desc(1, 1, 8, 64, 0.1)
    with pytest.raises(TypeError):
        _decode(mb.make_gemm_desc(8, 8, 8), None)
    with pytest.raises(AttributeError):
        mb.moa_decode_attn(desc, "q", None, None, None)
    with pytest.raises(OverflowError):
        mb.moa_decode_attn(desc, -1, None, None, None)


@pytest.mark.parametrize("ws,ws_bytes,want", [(None, None, "MOA_ERR_WORKSPACE"), (4096, 1, "MOA_ERR_WORKSPACE")])
def test_workspace_sizes(ws, ws_bytes, want):
    desc = mb.make_desc(1, 1, 256, 64, False, 0.1)
    a = 4096
    got = mb.moa_attn_bwd(desc, a, a, a, a, a, a, a, a, a, ws, stream=0, ws_bytes=ws_bytes, check=False)
    assert got == getattr(mb, want)
    with pytest.raises(mb.MoaError):
        mb.moa_attn_bwd(desc, a, a, a, a, a, a, a, a, a, torch.zeros(8, dtype=torch.uint8), stream=0)


@pytest.mark.parametrize("count", [1, 3])
def test_fill(count):
    class Words(ctypes.Structure):
        _fields_ = [("w", ctypes.c_uint64 * 3)]

    t = torch.zeros(4)
    words = mb.fill_pointers(Words(), (t, None, 7)[:count])
    assert list(words.w) == [t.data_ptr(), 0, 7 if count == 3 else 0]
    with pytest.raises(ValueError):
        mb.fill_pointers(Words(), (1, 2, 3, 4))


def test_from_several_threads():
    desc = mb.make_decode_desc(1, 1, -1, 64, 0.1)
    got = []
    threads = [threading.Thread(target=lambda: got.extend(_decode(desc, None, stream=0) for _ in range(500))) for _ in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert got == [mb.MOA_ERR_INVALID_ARG] * 2000


def test_after_reloads_of_the_binding():
    """(In a process of its own: the reload makes new descriptor classes.)  More reloads than any fixed table would hold."""
    code = """
import importlib
from paper_2609_33916_b200 import binding as mb
for k in range(12):
    for make, call, args in ((mb.make_decode_desc, mb.moa_decode_attn, 6), (mb.make_mlp_desc, mb.moa_gated_mlp_bwd, 13)):
        desc = make(1, 1, -1, 64, 0.1) if args == 6 else make(-1, 8, 8)
        assert call(desc, *[4096] * args, ws_bytes=0, stream=0, check=False) == mb.MOA_ERR_INVALID_ARG
    importlib.reload(mb)
"""
    r = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, cwd=build.ROOT)
    assert r.returncode == 0, r.stderr[-2000:]


def test_the_module_belongs_to_one_interpreter(monkeypatch, tmp_path):
    assert build.PYCALL.endswith(sysconfig.get_config_var("EXT_SUFFIX")) and os.path.exists(build.PYCALL)
    assert importlib.machinery.EXTENSION_SUFFIXES[0] == sysconfig.get_config_var("EXT_SUFFIX")
    # an untagged one, which every interpreter would load, goes; without a compiler or headers there is none, and that is no error
    monkeypatch.setattr(build, "HERE", str(tmp_path))
    monkeypatch.setattr(build, "PYCALL", str(tmp_path / "_pycall.tag.so"))
    (tmp_path / "_pycall.so").write_bytes(b"")
    monkeypatch.setenv("CC", str(tmp_path / "none"))
    with pytest.warns(UserWarning):
        assert build.build_pycall() is None
    assert os.listdir(tmp_path) == []
    monkeypatch.delenv("CC")
    monkeypatch.setattr(sysconfig, "get_paths", lambda: {"include": str(tmp_path)})
    with pytest.warns(UserWarning):
        assert build.build_pycall() is None
    assert os.listdir(tmp_path) == []


def test_without_the_extension():
    """The same answers through ctypes (a process of its own, in which the module cannot be imported)."""
    code = """
import ctypes, sys
sys.modules["paper_2609_33916_b200._pycall"] = None
import pytest, torch
sys.path.insert(0, "tests")
import test_pycall as t
from paper_2609_33916_b200 import binding as mb
t.test_descriptors_of_another_type_and_things_without_an_address_are_refused()
t.test_workspace_sizes(None, None, "MOA_ERR_WORKSPACE")
t.test_workspace_sizes(4096, 1, "MOA_ERR_WORKSPACE")
t.test_fill(1)
t.test_fill(3)
t.test_from_several_threads()
assert mb._load() is mb._invoke_ctypes
"""
    r = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, cwd=build.ROOT)
    assert r.returncode == 0, r.stderr[-2000:]
