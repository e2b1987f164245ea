"""A token that is not finite reaches the rows that depend on it and no other: every row that does not is, bit for
bit, what it is without that token.  (A masked entry that is multiplied as a zero would make NaN of it.)"""
import numpy as np
import pytest
import torch

import hla_inputs

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
N = 150
BAD = [float("nan"), float("inf")]


@pytest.fixture(scope="module")
def hla():
    from paper_2510_27258_gb300 import build
    build.build()
    from paper_2510_27258_gb300 import hla as binding
    return binding


def _tokens(d, dv, dtype):
    q, k, v = hla_inputs.make_qkv(1, 2, N, d, dv, seed=d + dv, dtype=dtype)
    g = hla_inputs.round_to(np.random.default_rng(dv).standard_normal((1, 2, N, dv)), dtype)
    return {name: hla_inputs.as_torch(x, dtype, DEV) for name, x in zip("qkvg", (q, k, v, g))}


def _planted(t, which, j, value):
    bad = dict(t)
    bad[which] = t[which].clone()
    bad[which][0, 1, j, 3] = value
    return bad


def _check(clean, bad, untouched, hit):
    """head 0 as before; of head 1 the rows in `untouched` as before, row `hit` not"""
    assert torch.equal(clean[:, 0], bad[:, 0])
    assert torch.equal(clean[0, 1, untouched], bad[0, 1, untouched])
    if hit is not None:
        assert not torch.isfinite(bad[0, 1, hit]).all()


SIZES = [(16, 16, "f32"), (32, 32, "f32"), (64, 64, "f32"), (128, 128, "f32"), (16, 64, "f32"), (32, 32, "bf16")]


@pytest.mark.parametrize("d,dv,dtype", SIZES)
@pytest.mark.parametrize("which", "qkv")
@pytest.mark.parametrize("j", [5, 50, 100, 149])
@pytest.mark.parametrize("value", BAD)
@pytest.mark.parametrize("kind", ["masked", "unmasked", "ahla"])
def test_forward(hla, d, dv, dtype, which, j, value, kind):
    def call(t, normalized, state):
        if kind == "ahla":
            st = torch.ones((1, 2, hla.ahla_state_floats(d, dv)), device=DEV) if state else None
            return hla.ahla_forward(t["q"], t["k"], t["v"], normalized=normalized, eps=1.0, state_in=st)
        st = torch.ones((1, 2, hla.hla2_state_floats(d, dv)), device=DEV) if state else None
        return hla.hla2_forward(t["q"], t["k"], t["v"], masked=kind == "masked", normalized=normalized, eps=1.0,
                                state_in=st)

    t = _tokens(d, dv, dtype)
    bad = _planted(t, which, j, value)
    for normalized in (False, True):
        for state in (False, True):
            _check(call(t, normalized, state), call(bad, normalized, state), slice(0, j), j)


# gradients of the plain output: the rows of dq, dk, dv that do not depend on token j, as (before j, after j), and
# whether row j has to be hit
DEPENDS = {"q": [(0, 0, 1), (0, 1, 1), (0, 1, 1)], "k": [(1, 0, 1), (1, 1, 1), (1, 0, 1)],
           "v": [(1, 0, 1), (0, 1, 1), (1, 1, 0)], "g": [(0, 1, 1), (0, 1, 1), (0, 1, 1)]}


def check_backward(hla, d, dv, dtype, which, j, value):
    t = _tokens(d, dv, dtype)
    bad = _planted(t, which, j, value)
    clean, got = (hla.hla2_backward(*(x[name] for name in "qkvg")) for x in (t, bad))
    for a, b, (before, after, hit) in zip(clean, got, DEPENDS[which]):
        rows = [i for i in range(N) if (i < j and before) or (i > j and after) or (i == j and not hit)]
        _check(a, b, rows, j if hit else None)


@pytest.mark.parametrize("d,dv,dtype", SIZES)
@pytest.mark.parametrize("which", "qkvg")
@pytest.mark.parametrize("j", [5, 50, 100, 149])
@pytest.mark.parametrize("value", BAD)
def test_backward(hla, d, dv, dtype, which, j, value):
    check_backward(hla, d, dv, dtype, which, j, value)


@pytest.mark.parametrize("d,dv", [(128, 128), (64, 128), (128, 64)])
@pytest.mark.parametrize("which", "qkvg")
@pytest.mark.parametrize("j", [0, 5, 100, 127, 128, 149])
@pytest.mark.parametrize("value", BAD)
def test_backward_tiles(hla, d, dv, which, j, value):
    """bf16 tokens with a head size of 128: tiles of 128 tokens on the tensor cores"""
    check_backward(hla, d, dv, "bf16", which, j, value)
