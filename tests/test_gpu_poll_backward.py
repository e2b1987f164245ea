"""The error word after a backward is that call's, whatever the workspace held before."""
import pytest
import torch

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.fixture(scope="module")
def hla():
    from paper_2510_27258_gb300 import build
    build.build()
    from paper_2510_27258_gb300 import hla as binding
    return binding


@pytest.mark.parametrize("d,dtype", [(32, torch.float32), (64, torch.float32), (32, torch.bfloat16),
                                     (64, torch.bfloat16), (128, torch.bfloat16)])
@pytest.mark.parametrize("n", [20, 200])
@pytest.mark.parametrize("normalized", [False, True])
def test_poll(hla, d, dtype, n, normalized):
    t = torch.ones((1, 2, n, d), dtype=dtype, device=DEV)
    size = hla.hla2_backward_workspace_bytes(1, 2, n, d, d, 64, dtype)
    ws = torch.full((size,), 255, dtype=torch.uint8, device=DEV)
    hla.hla2_backward(t, t, t, t, normalized=normalized, workspace=ws)
    assert hla.hla_poll_error(ws) == hla.HLA_OK
