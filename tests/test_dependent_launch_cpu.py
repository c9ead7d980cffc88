"""Kernels are launched while the work in front of them on the stream still runs and wait for it on the device
(griddepcontrol.wait).  No block of a kernel goes without that wait: what another grid has waited for is not in place for one that does not."""
import glob
import os
import re

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
