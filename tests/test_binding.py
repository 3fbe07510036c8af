"""The binding's extension module: one file per torch and Python, never another's; absent, the calls go through ctypes."""
import os
import sysconfig

import torch

from paper_2401_05391_b200 import build as b
from paper_2401_05391_b200 import segkv as sk


def test_extension_belongs_to_this_torch_and_python(monkeypatch):
    here = b.hot_path()
    assert torch.__version__ in os.path.basename(here) and here.endswith(sysconfig.get_config_var("EXT_SUFFIX"))
    monkeypatch.setattr(torch, "__version__", "0.0.0+other")
    assert b.hot_path() != here
    monkeypatch.setattr(sk, "_hot", None)
    assert sk._hot_module() is None               # built for another torch only: not loaded


def test_library_is_built_without_the_extension(monkeypatch, capsys):
    built = []
    monkeypatch.setattr(b, "_build_lib", lambda lib, *a: built.append(lib) or lib)

    def no_compiler(force=False):
        assert built == [b.LIB]                   # the library comes first
        raise OSError("no C++ compiler")

    monkeypatch.setattr(b, "build_hot", no_compiler)
    assert b.build() == b.LIB
    assert "ctypes" in capsys.readouterr().err
    assert b.build(timeline=True) == b.LIB_TIMELINE and built == [b.LIB, b.LIB_TIMELINE]
