"""The four-group combine kernels are built for as many blocks to an SM as leave room for what they run beside, which caps their registers.
Within that cap their loops must not spill: ptxas says so."""
import os
import re
import subprocess

import pytest

from paper_2609_37626_b200 import build


@pytest.fixture(scope="module")
def report(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("ptxas") / "merge.so")
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    r = subprocess.run([nvcc] + build.NVCC_FLAGS + ["-Xptxas", "-v", "-o", out, os.path.join(build.CSRC, "splash_merge.cu")],
                       capture_output=True, text=True, check=True)
    return r.stdout + r.stderr


def test_grouped_combine_does_not_spill(report):
    found = re.findall(r"Compiling entry function '(\S*grouped_combine_kernel\S*)'.*?(\d+) bytes spill stores, (\d+) bytes spill loads", report, re.S)
    assert len(found) >= 4
    assert all(stores == loads == "0" for _, stores, loads in found), found
