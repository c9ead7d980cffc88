"""What the Python form of splash_dop_unpack_rows takes: rows of one shape, dense each; rows without elements are dense whatever their strides
say."""
import pytest
import torch

from paper_2609_37626_b200 import binding, build


class Stream:
    cuda_stream = 0


@pytest.fixture(scope="module", autouse=True)
def built():
    build.build()


@pytest.mark.parametrize("out", [torch.empty(5, 0, 7), torch.empty(5, 4, 7)[:, :0], torch.empty(5, 4, 14)[:, :0, ::2], torch.empty(5, 7, 4)[..., :0].transpose(1, 2)])
def test_rows_without_elements(out):
    recv = torch.empty((3,) + tuple(out.shape[1:]))
    assert binding.splash_dop_unpack_rows(recv, torch.zeros(3, dtype=torch.int32), out, Stream) is out


@pytest.mark.parametrize("recv,out", [(torch.empty(3, 4), torch.empty(5, 5)), (torch.empty(3, 4), torch.empty(5, 8)[:, ::2]), (torch.empty(3, 2, 4), torch.empty(5, 4, 2).transpose(1, 2)),
                                      (torch.empty(3, 4), torch.empty(5, 4, 1))])
def test_other_rows_are_refused(recv, out):
    with pytest.raises(AssertionError):
        binding.splash_dop_unpack_rows(recv, torch.zeros(3, dtype=torch.int32), out, Stream)
