"""More than 65535 heads (a grid's second and third dimension end there): the first and last heads' results are
those of a call with these heads alone."""
import pytest
import torch

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
H = 65536 + 3


@pytest.fixture(scope="module")
def hla():
    from paper_2510_27258_gb300 import build
    build.build()
    from paper_2510_27258_gb300 import hla as binding
    return binding


def _tokens(n, d, dtype, count):
    g = torch.Generator(device=DEV)
    g.manual_seed(n)
    return [torch.randn((1, H, n, d), generator=g, device=DEV).mul_(0.2).to(dtype) for _ in range(count)]


def _ends(x):
    return torch.cat([x[:, :2], x[:, -2:]], 1).contiguous()


def _same(call, t):
    some = call(*map(_ends, t))
    for a, b in zip(call(*t), some):
        assert torch.equal(_ends(a), b)


@pytest.mark.parametrize("n", [2, 70])
@pytest.mark.parametrize("masked", [True, False])
def test_forward(hla, n, masked):
    def call(q, k, v):
        st = torch.empty((1, q.shape[1], hla.hla2_state_floats(16, 16)), device=DEV)
        out = hla.hla2_forward(q, k, v, masked=masked, normalized=True, eps=9.0, state_out=st)
        return out, st, hla.hla2_forward(q, k, v, masked=masked, state_in=st)

    _same(call, _tokens(n, 16, torch.float32, 3))


@pytest.mark.parametrize("n", [2, 70])
def test_ahla(hla, n):
    def call(q, k, v):
        st = torch.empty((1, q.shape[1], hla.ahla_state_floats(16, 16)), device=DEV)
        return hla.ahla_forward(q, k, v, state_out=st), st, hla.ahla_forward(q, k, v, state_in=st)

    _same(call, _tokens(n, 16, torch.float32, 3))


@pytest.mark.parametrize("n,d,dtype", [(2, 16, torch.float32), (70, 16, torch.float32), (3, 128, torch.bfloat16)])
def test_backward(hla, n, d, dtype):
    _same(hla.hla2_backward, _tokens(n, d, dtype, 4))
