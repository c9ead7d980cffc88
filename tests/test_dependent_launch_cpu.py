"""Kernels are launched while the work in front of them on the stream still runs and wait for it on the device
(griddepcontrol.wait).  What they read behind that wait must not be read as if it had never changed: a load through the read-only path may
be moved in front of the wait, or hit what was there before.  No kernel that waits takes a const __restrict__ pointer or uses
__ldg or ld.global.nc; and no block of a kernel goes without the wait."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_37626_b200", "csrc")
FILES = sorted(os.path.basename(f) for f in glob.glob(os.path.join(CSRC, "*.cu*")))


def code(name):
    return re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())


def kernels(text):
    """(name, parameters, body) of every __global__ function."""
    for m in re.finditer(r"__global__[^;{]*?\b(\w+)\s*\(((?:[^()]|\([^()]*\))*)\)\s*\{", text):
        depth, i = 1, m.end()
        while depth:
            depth += {"{": 1, "}": -1}.get(text[i], 0)
            i += 1
        yield m.group(1), m.group(2), text[m.end():i]


@pytest.mark.parametrize("name", FILES)
def test_no_read_only_loads(name):
    text = code(name)
    assert "__ldg(" not in text and "__ldcg(" not in text and "global.nc" not in text
    for kernel, params, body in kernels(text):
        if "grid_dependency_wait()" in body or "start_plan<" in body:
            assert not re.search(r"const\s+\w+\s*\*\s*__restrict__", params), f"{name}: {kernel}"


def test_every_kernel_that_is_launched_early_waits():
    launched, waits = set(), set()
    for name in FILES:
        text = code(name)
        for m in re.finditer(r"launch_dependent\(([^;]*?),\s*dim3", text, re.S):
            launched.update(re.findall(r"\b(\w+_kernel)\b", m.group(1)))
        for kernel, _, body in kernels(text):
            if "grid_dependency_wait()" in body or "start_plan<" in body:
                waits.add(kernel)
    assert len(launched) >= 8 and launched <= waits, launched - waits


def test_no_block_of_the_page_copy_skips_the_wait():
    body = dict((k, b) for k, _, b in kernels(code("splash_migrate.cu")))["page_migrate_kernel"]
    first = body.index("grid_dependency_wait()")
    assert body[:first].count("{") == body[:first].count("}") and "if" not in body[:first], "the wait is conditional"
