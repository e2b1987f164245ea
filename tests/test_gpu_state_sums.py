"""C and m of a final state: sums of the tensor cores over groups of tiles.  Up to 32 heads every head has
eight groups, so its C and m do not depend, to the bit, on the heads beside it; and every entry is within what
one fp32 addition with truncation (2^-23 of the sum of magnitudes) per 16 tokens of a group and per group allows."""
import pytest
import torch

import hla_inputs

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.fixture(scope="module")
def hla():
    from paper_2510_27258_gb300 import build
    build.build()
    from paper_2510_27258_gb300 import hla as binding
    return binding


def _final(hla, q, k, v):
    """C [B, H, d, dv] and m [B, H, d] of the final state"""
    (B, H, n, d), dv = q.shape, v.shape[-1]
    st = torch.empty((B, H, hla.hla2_state_floats(d, dv)), device=DEV)
    ws = hla.alloc_workspace(hla.hla2_workspace_bytes(B, H, n, d, dv, 128, torch.bfloat16), DEV)
    hla.hla2_forward(q, k, v, state_out=st, workspace=ws)
    assert hla.hla_poll_error(ws) == hla.HLA_OK
    C = st[..., d * d:d * d + d * dv].reshape(B, H, d, dv)
    return C, st[..., d * d + d * dv:d * d + d * dv + d]


def _tokens(H, n, d, dv):
    return [hla_inputs.as_torch(x, "bf16", DEV) for x in hla_inputs.make_qkv(1, H, n, d, dv, seed=H + n, dtype="bf16")]


@pytest.mark.parametrize("heads,n,d", [(32, 1999, 128), (31, 4000, 64), (20, 1024, 128)])
def test_other_heads_do_not_matter(hla, heads, n, d):
    t = _tokens(heads, n, d, d)
    C, m = _final(hla, *t)
    for h in (0, heads - 1):
        C1, m1 = _final(hla, *(x[:, h:h + 1].contiguous() for x in t))
        assert torch.equal(C[:, h:h + 1], C1) and torch.equal(m[:, h:h + 1], m1)


@pytest.mark.parametrize("heads", [1, 19, 20, 32, 50, 51, 64, 77, 85, 86, 128, 129, 200])
@pytest.mark.parametrize("n,d,dv", [(90, 128, 128), (640, 64, 128), (2500, 64, 64)])
def test_sums(hla, heads, n, d, dv):
    """every number of groups a block and a head, groups without tiles"""
    q, k, v = _tokens(heads, n, d, dv)
    C, m = _final(hla, q, k, v)
    tiles = -(-n // 128)
    groups = min(8, max(1, 256 // heads), tiles)
    bound = (8 * -(-tiles // groups) + groups) * 2.0 ** -23
    Q, V = q.double(), v.double()
    assert ((C - Q.mT @ V).abs() <= bound * (Q.abs().mT @ V.abs())).all()
    assert ((m - Q.sum(-2)).abs() <= bound * Q.abs().sum(-2)).all()
