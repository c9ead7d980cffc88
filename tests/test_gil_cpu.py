"""The Python entry points give the GIL up for as long as they are inside the library: with a full launch queue a launch blocks, and what
it waits for may be another thread of the process.  A stand-in for the library's function (preloaded into a child process, no GPU
needed) takes 0.5 s, and another thread has to get on meanwhile.  The decode entry points want CUDA tensors: their child runs
on a GPU, and the stand-in launches nothing there either."""
import os
import subprocess
import sys
import textwrap

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

STUBS = """
#include <stddef.h>
#include <unistd.h>
#define SLOW(name) extern "C" __attribute__((visibility("default"))) int name(...) { usleep(500000); return 0; }
SLOW(splash_lse_merge) SLOW(splash_kv_page_migrate) SLOW(splash_kv_page_migrate_static) SLOW(splash_dop_pack_rows) SLOW(splash_dop_swap_outer)
SLOW(splash_dop_unpack_rows) SLOW(splash_mla_decode) SLOW(splash_mla_decode_migrating) SLOW(splash_mla_decode_sparse)
"""

CHILD = """
import sys, threading, time
sys.path.insert(0, {root!r})
import torch
from paper_2609_37626_b200 import binding as B
sys.setswitchinterval(1e-3)
class Stream: cuda_stream = 0
dev = sys.argv[2]
f32 = lambda *s: torch.zeros(s, device=dev)
i32 = lambda *s: torch.zeros(s, dtype=torch.int32, device=dev)
u8 = lambda *s: torch.zeros(s, dtype=torch.uint8, device=dev)
ws = u8(1 << 20)
pool = u8(4, 64, 576)
def decode(**kw):
    q = f32(2, 16, 576).to(torch.bfloat16)
    return B.splash_mla_decode(q, f32(4, 64, 576).to(torch.bfloat16), i32(2, 2), i32(2), softmax_scale=1.0, out=f32(2, 16, 512), lse=f32(2, 16), workspace=ws, stream=Stream, **kw)
calls = dict(
    merge=lambda: B.splash_lse_merge(f32(2, 3, 8), f32(2, 3), f32(3, 8), f32(3), Stream),
    migrate=lambda: B.splash_kv_page_migrate(pool, pool, i32(1), i32(1), i32(4), workspace=ws, stream=Stream),
    migrate_static=lambda: B.splash_kv_page_migrate_static(pool, pool, i32(1), i32(1), i32(4), stream=Stream),
    pack=lambda: B.splash_dop_pack_rows(f32(3, 2, 8), None, i32(3), f32(3, 2, 8), Stream),
    swap=lambda: B.splash_dop_swap_outer(f32(3, 2, 8), f32(2, 3, 8), Stream),
    unpack=lambda: B.splash_dop_unpack_rows(f32(3, 8), i32(3), f32(3, 8), Stream),
    decode=lambda: decode(),
    decode_migrating=lambda: decode(migrate_job=B.make_migrate_job(pool, pool, i32(1), i32(1), i32(4), workspace=ws)),
    sparse=lambda: B.splash_mla_decode_sparse(f32(2, 16, 576).to(torch.bfloat16), u8(4, 64, 656), i32(2, 2), i32(2), i32(2, 8), i32(2), softmax_scale=1.0,
                                              out=f32(2, 16, 512), lse=f32(2, 16), workspace=ws, stream=Stream))
state = dict(inside=False, ticks=0, stop=False)
def tick():
    while not state["stop"]:
        if state["inside"]: state["ticks"] += 1
        time.sleep(0.01)
t = threading.Thread(target=tick); t.start()
call = calls[sys.argv[1]]
t0 = time.time(); state["inside"] = True
call()
state["inside"] = False; took = time.time() - t0
state["stop"] = True; t.join()
print("took", took, "ticks", state["ticks"])
assert took >= 0.45, "the stand-in was not called"
assert state["ticks"] >= 10, "no other thread ran while the call was inside the library"
"""


def run(tmp_path, call, device):
    from paper_2609_37626_b200 import build
    build.build()
    stub = tmp_path / "stub.cpp"
    stub.write_text(STUBS)
    lib = str(tmp_path / "libstub.so")
    subprocess.check_call([os.environ.get("CXX", "g++"), "-shared", "-fPIC", "-o", lib, str(stub)])
    child = tmp_path / "child.py"
    child.write_text(textwrap.dedent(CHILD.format(root=ROOT)))
    r = subprocess.run([sys.executable, str(child), call, device], env=dict(os.environ, LD_PRELOAD=lib), capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr


@pytest.mark.parametrize("call", ["merge", "migrate", "migrate_static", "pack", "swap", "unpack"])
def test_other_threads_run_meanwhile(tmp_path, call):
    run(tmp_path, call, "cpu")


@pytest.mark.gpu
@pytest.mark.parametrize("call", ["decode", "decode_migrating", "sparse"])
def test_other_threads_run_meanwhile_decode(tmp_path, call):
    run(tmp_path, call, "cuda")
