"""Decode steps whose last query or key feature is infinite: sums over a head's rows take those rows alone, so
what is infinite stays infinite where a term of zero times infinity would make NaN of it."""
import pytest
import torch

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
INF = float("inf")


@pytest.fixture(scope="module")
def hla():
    from paper_2510_27258_gb300 import build
    build.build()
    from paper_2510_27258_gb300 import hla as binding
    return binding


@pytest.mark.parametrize("heads", [1, 3, 70, 201])
@pytest.mark.parametrize("d,dv", [(16, 16), (32, 32), (64, 16), (16, 128), (64, 64)])
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
def test_step(hla, heads, d, dv, dtype):
    ones = lambda *s: torch.ones((1, heads) + s, dtype=dtype, device=DEV)  # noqa: E731
    hot = ones(d)
    hot[..., -1] = INF
    # every entry positive: q^T P', q^T E' and q^T D' are infinite, with no difference of infinities in them
    out = hla.ahla_step(hot, ones(d), ones(dv), torch.ones((1, heads, hla.ahla_state_floats(d, dv)), device=DEV))
    assert (out == INF).all()
    out = hla.hla2_step_sde(hot, ones(d), ones(dv), torch.ones((1, heads, hla.hla2_sde_state_floats(d, dv)), device=DEV))
    assert (out == INF).all()
    out = hla.hla2_step(hot, ones(d), ones(dv), torch.ones((1, heads, hla.hla2_state_floats(d, dv)), device=DEV),
                        masked=False)
    assert (out == INF).all()
    # k^T C is infinite, so every entry of G' = G + k (k^T C) is
    st = torch.ones((1, heads, hla.hla2_state_floats(d, dv)), device=DEV)
    hla.hla2_step(ones(d), hot, ones(dv), st)
    at = d * d + d * dv + d
    assert (st[..., at:at + d * dv] == INF).all()
