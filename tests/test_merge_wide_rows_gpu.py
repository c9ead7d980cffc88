"""The merge of few rows of more than 512 values takes several blocks a row: the cases of the usual widths at the edges of a block's 512 columns."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("parts", [1, 5, 129])
@pytest.mark.parametrize("rows", [3, 700])
@pytest.mark.parametrize("d_v", [508, 516, 1024, 1540])
def test_wide_rows(parts, rows, d_v):
    import test_merge_widths_gpu
    test_merge_widths_gpu.test_parts_and_rows(parts, rows, d_v)


@pytest.mark.parametrize("parts", [2, 129])
@pytest.mark.parametrize("rows", [500, 1184, 1185])
@pytest.mark.parametrize("d_v", [1540, 2048])
def test_rows_that_fill_the_chip(parts, rows, d_v):
    """Around eight rows for each of 148 SMs a row goes from a few blocks, some of several times 512 columns, to one."""
    import test_merge_widths_gpu
    test_merge_widths_gpu.test_parts_and_rows(parts, rows, d_v)
