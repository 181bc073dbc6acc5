"""When the library and the native side of the binding count as up to date.  Nothing is compiled here."""
import os
import shutil
import sysconfig

import torch

from paper_2106_09236_b200 import binding as ps
from paper_2106_09236_b200 import build


def test_module_of_another_torch_or_python_is_built_again(monkeypatch):
    ps._load_native()                                    # in place, built now if need be
    assert not build.native_needs_build()
    with monkeypatch.context() as m:                     # one version a prefix of the other
        m.setattr(torch, "__version__", torch.__version__[:-1])
        assert build.native_needs_build()
    with monkeypatch.context() as m:
        m.setattr(torch._C, "_GLIBCXX_USE_CXX11_ABI", not torch._C._GLIBCXX_USE_CXX11_ABI)
        assert build.native_needs_build()
    with monkeypatch.context() as m:
        soabi = sysconfig.get_config_var("SOABI")
        m.setattr(sysconfig, "get_config_var", lambda name: "another" if name == "SOABI" else soabi)
        assert build.native_needs_build()
    assert not build.native_needs_build()


def test_missing_or_older_module_is_built_again(monkeypatch, tmp_path):
    copy = tmp_path / "psattn_torch.so"
    monkeypatch.setattr(build, "NATIVE", str(copy))
    assert build.native_needs_build()
    copy.write_bytes(b"something else")
    assert build.native_needs_build()
    copy.write_bytes(b"..." + build.native_built_for() + b"\0...")
    assert not build.native_needs_build()
    source = tmp_path / "psattn_torch.cpp"
    source.write_text("")
    os.utime(copy, (1, 1))
    monkeypatch.setattr(build, "NATIVE_SOURCE", str(source))
    assert build.native_needs_build()


def test_library_of_other_sources_or_flags_is_built_again(monkeypatch, tmp_path):
    ps.load()
    assert not build.needs_build()
    with monkeypatch.context() as m:
        m.setattr(build, "NVCC_FLAGS", build.NVCC_FLAGS + ["-G"])
        assert build.needs_build()
    copy = tmp_path / "csrc"
    shutil.copytree(build.CSRC, copy, ignore=shutil.ignore_patterns("*.o"))
    monkeypatch.setattr(build, "CSRC", str(copy))
    assert not build.needs_build()
    with open(copy / "psattn_select.cuh", "a") as f:
        f.write("// changed\n")
    os.utime(copy / "psattn_select.cuh", (1, 1))         # older than the library, as a file put back to an earlier state
    assert build.needs_build()
