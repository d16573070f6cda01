"""What the native argument marshalling refuses is what the checks in Python refused: tensors off the GPU, other types, gaps,
things that are no tensors, the other call's descriptor."""
import ctypes
import decimal
import fractions
import os
import re
import runpy
import shutil
import subprocess
import sys
import sysconfig

import numpy as np
import pytest
import torch

import __graft_entry__ as entry


@pytest.fixture(scope="module")
def mv():
    entry.build()
    import paper_2505_10526_b200 as pkg
    return pkg


def test_refused_without_a_gpu(mv):
    a, c = mv.attn_desc(1, 1, 1, 1, 64, 1, 1), mv.accept_desc(1, 1, 64, 64, 1.0)
    f, i, b = torch.zeros(64), torch.zeros(64, dtype=torch.int32), torch.zeros(64, dtype=torch.bfloat16)
    with pytest.raises(ValueError, match="CUDA device"):
        mv.massv_verify_attn(a, b, b, b, b, b, i, i, b)
    with pytest.raises(ValueError, match="CUDA device"):
        mv.massv_tvd(c, f, f, f)
    with pytest.raises(ValueError, match="CUDA device"):
        mv.massv_sample_top_p(f.view(1, 64), f, i, 1.0, 0.9)
    with pytest.raises(ValueError, match="CUDA device"):
        mv.massv_kv_commit(1, 1, i, i)
    with pytest.raises(AttributeError):
        mv.massv_kv_commit(1, 1, None, 7)
    # another descriptor, and buffers of a descriptor's length that are none
    for wrong in (a, 3, None, bytes(ctypes.sizeof(c)), bytearray(ctypes.sizeof(c)), (ctypes.c_char * ctypes.sizeof(c))(), type(c)):
        with pytest.raises(TypeError):
            mv.massv_accept(wrong, b, b, i, f, f, f, i, i)
    for wrong in (c, bytes(ctypes.sizeof(a)), (ctypes.c_char * ctypes.sizeof(a))()):
        with pytest.raises(TypeError):
            mv.massv_verify_attn(wrong, b, b, b, b, b, i, i, b)


def test_a_derived_descriptor_is_one(mv):
    class Named(mv.AcceptDesc):
        _fields_ = [("name", ctypes.c_char * 16)]

    d = Named(*[getattr(mv.accept_desc(1, 1, 64, 64, 1.0), n) for n, _ in mv.AcceptDesc._fields_])
    f = torch.zeros(64)
    with pytest.raises(ValueError, match="CUDA device"):            # past the descriptor, at the first tensor
        mv.massv_tvd(d, f, f, f)


@pytest.mark.parametrize("number", ["0.75", b"0.75", fractions.Fraction(3, 4), decimal.Decimal("0.75"), np.float32(0.75), torch.tensor(0.75), 1])
def test_numbers_are_what_float_takes(mv, number):
    f, i = torch.zeros(64), torch.zeros(64, dtype=torch.int32)
    with pytest.raises(ValueError, match="CUDA device"):            # past the numbers, at the first tensor
        mv.massv_sample_top_p(f.view(1, 64), f, i, number, number)
    with pytest.raises(TypeError):
        mv.massv_sample_top_p(f.view(1, 64), f, i, None, number)


def test_the_module_goes_with_torch_and_python(mv, monkeypatch):
    """Another torch or another Python: another file, which does not exist and is stale, so that it is built and never loaded in its place."""
    from paper_2505_10526_b200 import build
    here = build.marshal_path()
    assert mv.binding._native.__file__ == here and not build._stale(here)
    assert torch.__version__ in os.path.basename(here) and here.endswith(sysconfig.get_config_var("EXT_SUFFIX"))
    for target, name, value in ((runpy, "run_path", lambda path: {"__version__": "2.99.0"}), (sysconfig, "get_config_var", lambda name: ".cpython-399-x86_64-linux-gnu.so")):
        with monkeypatch.context() as m:
            m.setattr(target, name, value)
            other = build.marshal_path()
            assert other != here and build._stale(other)
            with pytest.raises(ImportError, match="build it with"):
                mv.binding._load_marshal()


def test_the_command_a_missing_module_names(mv, tmp_path):
    """A package without its native module says what builds it, and that command works although the package cannot be imported."""
    root = os.path.dirname(os.path.dirname(mv.LIB_PATH))
    for name in ("include", "paper_2505_10526_b200"):
        shutil.copytree(os.path.join(root, name), tmp_path / name, ignore=shutil.ignore_patterns("_marshal*", "__pycache__"))
    import_it = [sys.executable, "-c", "import paper_2505_10526_b200"]
    missing = subprocess.run(import_it, cwd=tmp_path, capture_output=True, text=True)
    assert missing.returncode != 0 and "ImportError" in missing.stderr
    command = re.search("`(python .*)`", missing.stderr.strip().splitlines()[-1]).group(1).split()
    assert command[0] == "python" and os.path.samefile(command[1], tmp_path / "paper_2505_10526_b200" / "build.py")
    subprocess.run([sys.executable] + command[1:], cwd=tmp_path, check=True)
    subprocess.run(import_it, cwd=tmp_path, check=True)


@pytest.mark.gpu
def test_refused_on_the_gpu(mv):
    lens = torch.zeros((4, 2), dtype=torch.int32, device="cuda")
    with pytest.raises(ValueError, match="contiguous"):
        mv.massv_kv_commit(4, 1, lens[:, 0], lens[:, 1])
    with pytest.raises(ValueError, match="expected torch.int32, got torch.float32"):
        mv.massv_kv_commit(4, 1, lens[0].float(), lens[1])
    with pytest.raises(mv.MassvError):
        mv.massv_kv_commit(0, 1, lens[0].contiguous(), lens[1].contiguous())
