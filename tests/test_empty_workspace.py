"""A call of no tokens needs no more scratch than the workspace header."""
import pytest
import torch

from paper_2510_27258_gb300 import build


@pytest.fixture(scope="module")
def hla():
    build.build()
    from paper_2510_27258_gb300 import hla as m
    return m


@pytest.mark.parametrize("d,dv", [(16, 128), (64, 64), (128, 128)])
@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("size", ["ahla_workspace_bytes", "hla2_backward_workspace_bytes"])
def test_empty_call_workspace(hla, size, dtype, d, dv):
    assert getattr(hla, size)(2, 4, 0, d, dv, 64, dtype) == 256
