"""The extension module belongs to one torch: it is named after its version, built with its C++ ABI, and another torch neither takes it
for built nor loads it."""
import os
import subprocess
import sys

import torch

from paper_2609_37626_b200 import build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_the_path_names_the_torch(monkeypatch):
    here = build.torch_ext_path()
    monkeypatch.setattr(torch, "__version__", "99.1.0+other")
    assert build.torch_ext_path() != here and "99_1_0_other" in build.torch_ext_path()


def test_another_torch_means_building_again(monkeypatch):
    build.build()
    commands = []
    monkeypatch.setattr(torch, "__version__", "99.1.0+other")
    monkeypatch.setattr(torch, "compiled_with_cxx11_abi", lambda: False)
    monkeypatch.setattr(subprocess, "check_call", commands.append)
    monkeypatch.setattr(os, "remove", lambda f: commands.append(["rm", f]))
    build.build()
    compiled = [c for c in commands if any(str(x).endswith("splash_torch.cpp") for x in c)]
    assert len(compiled) == 1 and "-D_GLIBCXX_USE_CXX11_ABI=0" in compiled[0] and build.torch_ext_path() in compiled[0]


def test_a_module_of_another_torch_is_not_loaded():
    build.build()
    code = ("import sys; sys.path.insert(0, %r)\nimport torch; torch.__version__ = torch.torch_version.TorchVersion('99.1.0+other')\n"
            "from paper_2609_37626_b200 import binding\n"
            "try:\n    binding.splash_lse_merge\nexcept ImportError as e:\n    assert '99.1.0' in str(e), e; print('refused')\n") % ROOT
    r = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, timeout=300)
    assert "refused" in r.stdout, r.stdout + r.stderr
