"""Decode steps on both sides of the head counts where the kernel or the number of blocks per head changes, against
the fp64 oracle for the first and last heads.  Bars as in tests/test_gpu_step_split.py."""
import numpy as np
import pytest
import torch

import hla_inputs
import oracle
from parity import TOL, rowerr

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.fixture(scope="module")
def hla():
    from paper_2510_27258_gb300 import build
    build.build()
    from paper_2510_27258_gb300 import hla as binding
    return binding


CASES = [("ahla", h, 128, 128) for h in (64, 65, 180, 181, 1999, 2000)] + \
        [("ahla", h, *s) for h in (250, 1250, 1251) for s in ((64, 128), (128, 64))] + \
        [("ahla", h, *s) for h in (250, 3000) for s in ((32, 128), (128, 32), (128, 16))] + \
        [("unmasked", h, *s) for h in (8, 32) for s in ((128, 128), (128, 32), (128, 16), (32, 128))]


@pytest.mark.parametrize("kind,heads,d,dv", CASES)
@pytest.mark.parametrize("normalized", [False, True])
def test_step(hla, kind, heads, d, dv, normalized):
    serial = oracle.ahla_serial if kind == "ahla" else lambda *a, **kw: oracle.hla2_serial(*a, masked=False, **kw)
    size = (hla.ahla_state_floats if kind == "ahla" else hla.hla2_state_floats)(d, dv)
    q, k, v = (x[0, :, :1] for x in hla_inputs.make_qkv(1, heads, 1, d, dv, seed=heads, dtype="f32"))
    q, k = np.abs(q), np.abs(k)
    st0 = np.abs(np.random.default_rng(heads).standard_normal((heads, size))).astype(np.float32)
    if kind == "unmasked":  # S is symmetric
        S = st0[:, :d * d].reshape(heads, d, d)
        S += S.transpose(0, 2, 1).copy()
    t = [hla_inputs.as_torch(x[None, :, 0], "f32", DEV) for x in (q, k, v)]
    st = torch.from_numpy(st0).to(DEV).reshape(1, heads, -1)
    if kind == "ahla":
        out = hla.ahla_step(*t, st, normalized=normalized, eps=1.0)
    else:
        out = hla.hla2_step(*t, st, masked=False, normalized=normalized, eps=1.0)
    some = [0, 1, heads // 2, heads - 2, heads - 1]
    ref, rst = serial(q[some], k[some], v[some], normalized=normalized, eps=1.0, state_in=st0[some], return_state=True)
    assert rowerr(out[0, some].cpu().numpy(), ref[:, 0]) < TOL["f32"]
    n = size if kind == "ahla" else d * d + d * dv + d  # unmasked: G and h are left as they were
    assert np.abs(st[0, some, :n].cpu().numpy() - rst[:, :n]).max() <= 1e-5 * np.abs(rst).max()
