"""Decode steps of few heads (several blocks per head) against the fp64 oracle, at the head counts
where the number of blocks per head changes and at every column split.  Bars: 1e-4 of the row norm for
the output of fp32 tokens, 1e-5 of the largest entry for the updated state (one rank-one update of fp32
values: a few roundings of 2^-24 of the terms, here below 2^-20 of the largest)."""
import numpy as np
import pytest
import torch

import hla_inputs
import oracle
from parity import TOL, rowerr

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
SIZES = [(128, 128), (64, 64), (128, 64), (64, 128), (128, 16), (64, 16), (16, 16), (32, 128)]


@pytest.fixture(scope="module")
def hla():
    from paper_2510_27258_gb300 import build
    build.build()
    from paper_2510_27258_gb300 import hla as binding
    return binding


def _flat(x):
    return x.reshape((-1,) + x.shape[2:])


@pytest.mark.parametrize("heads", [1, 8, 9, 32, 33, 65, 201, 600])
@pytest.mark.parametrize("d,dv", SIZES)
@pytest.mark.parametrize("kind", ["masked", "unmasked", "sde", "ahla"])
def test_step(hla, heads, d, dv, kind):
    pq, pk, pv = (_flat(x) for x in hla_inputs.make_qkv(1, heads, 30, d, dv, seed=heads, dtype="f32"))
    q, k, v = (_flat(x) for x in hla_inputs.make_qkv(1, heads, 1, d, dv, seed=heads + 1, dtype="f32"))
    masked = kind != "unmasked"
    serial = oracle.ahla_serial if kind == "ahla" else lambda *a, **kw: oracle.hla2_serial(*a, masked=masked, **kw)
    st0 = serial(pq, pk, pv, return_state=True)[1].astype(np.float32)
    t = [hla_inputs.as_torch(x.reshape(1, heads, -1), "f32", DEV) for x in (q, k, v)]
    for normalized in (False, True):
        eps = 1.0 if normalized else hla_inputs.EPS
        ref, rst = serial(q, k, v, normalized=normalized, eps=eps, state_in=st0, return_state=True)
        if kind == "sde":
            st = torch.from_numpy(oracle.hla2_state_to_sde(st0, d, dv).astype(np.float32)).to(DEV).reshape(1, heads, -1)
            out = hla.hla2_step_sde(*t, st, normalized=normalized, eps=eps)
            rst = oracle.hla2_state_to_sde(rst, d, dv)
        else:
            st = torch.from_numpy(st0).to(DEV).reshape(1, heads, -1)
            if kind == "ahla":
                out = hla.ahla_step(*t, st, normalized=normalized, eps=eps)
            else:
                out = hla.hla2_step(*t, st, masked=masked, normalized=normalized, eps=eps)
        torch.cuda.synchronize()
        if normalized:  # near a zero of den + eps fp32 has no such bar: there the state alone is checked
            den = serial(q, k, v, state_in=st0, return_den=True)[1].reshape(-1)
            well = np.abs(den + eps) > 0.1
        else:
            well = np.ones(heads, bool)
        assert rowerr(_flat(out.cpu().numpy())[well], ref.reshape(heads, dv)[well]) < TOL["f32"]
        got = st.reshape(heads, -1).cpu().numpy()
        if kind == "unmasked":  # G and h are left as they were
            n = d * d + d * dv + d
            assert np.array_equal(got[:, n:], st0[:, n:])
            got, rst = got[:, :n], rst[:, :n]
        assert np.abs(got - rst).max() <= 1e-5 * np.abs(rst).max()
