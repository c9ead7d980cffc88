"""What the combine kernels merge: requests cut into one piece a tile (less work than workers), into counts around the loads that a
thread has in flight (four, eight, twelve, sixteen) and the four groups' share of them, with an earlier request's end in the first worker
or not, few rows and many, behind every kernel family."""
import numpy as np
import pytest

from paper_2609_37626_b200 import workloads as W
from _util import compare, gpu_run, oracle_run

pytestmark = pytest.mark.gpu

FAMILIES = [(0, 1), (0, 16), (0, 32), (0, 64), (0, 128), (1, 16), (1, 32), (1, 64), (1, 128)]      # kv_dtype, heads


@pytest.mark.parametrize("kv_dtype,H", FAMILIES)
@pytest.mark.parametrize("lens", [[65], [64 * 5], [64 * 33 + 1], [100, 64 * 17, 3], [64 * 150, 0, 129, 64 * 9], [9000] * 2 + [1] * 7])
def test_few_requests(kv_dtype, H, lens):
    w = W.make_workload("pieces", 9300 + H + sum(lens), lens, H=H, kv_dtype=kv_dtype)
    compare(*gpu_run(w), *oracle_run(w), kv_dtype=kv_dtype)


@pytest.mark.parametrize("kv_dtype,H", [(0, 16), (0, 128), (1, 16), (1, 128)])
def test_many_requests_and_a_long_one(kv_dtype, H):
    """More requests than a quarter of the workers: nearly all in four pieces at most, one in many; and a batch of empty requests
    whose work costs less than there are workers."""
    rng = np.random.default_rng(H)
    lens = rng.integers(1, 500, size=40)
    lens[7], lens[20] = 64 * 60, 0
    few = np.zeros(40, np.int64)
    few[[5, 30]] = 700, 64 * 11
    for x in (lens, few):
        w = W.make_workload("pieces", 9400 + H, x, H=H, kv_dtype=kv_dtype)
        compare(*gpu_run(w), *oracle_run(w), kv_dtype=kv_dtype)


@pytest.mark.parametrize("kv_dtype,H", [(0, 16), (0, 32), (0, 128), (1, 16), (1, 128)])
@pytest.mark.parametrize("lens", [[64 * 7], [300, 700, 64, 1000], [64 * 20, 0, 1]])
def test_the_planner_makes_no_difference(kv_dtype, H, lens):
    """Less work than workers: the plan kernel (validation mode runs it) leaves workers without a piece between those with one, the
    plan that a decode kernel makes for itself does not; the same pieces, merged in the same order."""
    from paper_2609_37626_b200 import binding
    w = W.make_workload("planner", 9450 + H + sum(lens), lens, H=H, kv_dtype=kv_dtype)
    w.block_table = np.pad(w.block_table, ((0, 0), (0, 8)), constant_values=-1)      # wide enough for requests to be cut
    a, b = gpu_run(w), gpu_run(w, flags=binding.SPLASH_FLAG_VALIDATE)
    assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])
