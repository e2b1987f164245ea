"""Up to 64 tokens at head sizes up to 32 with a state in or out: one launch, against the fp64 oracle at the edges of
its chunk, for every kind of state, in place too.  Bars as in tests/test_gpu_hla2.py."""
import numpy as np
import pytest
import torch

import hla_inputs
import oracle
from parity import TOL, check_normalized, rowerr

DEV = "cuda:0"


@pytest.fixture(scope="module")
def hla():
    from paper_2510_27258_gb300 import build
    build.build()
    from paper_2510_27258_gb300 import hla as binding
    return binding


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("masked", [True, False])
def test_launches(hla, dtype, masked):
    def launches(n, d, dv, si, so):
        return hla.hla2_forward_path(1, 4, n, d, dv, masked=masked, dtype=dtype, has_state_in=si, has_state_out=so)[1]

    for n in (1, 16, 64):
        for si, so in ((True, True), (False, True), (True, False), (False, False)):
            assert launches(n, 16, 32, si, so) == 1
    assert launches(65, 32, 32, True, True) > 1
    assert launches(1, 32, 128, True, True) > 1
    assert launches(0, 32, 32, True, True) > 1


def _flat(x):
    return x.reshape((-1,) + x.shape[2:])


@pytest.mark.gpu
@pytest.mark.parametrize("n", [1, 2, 31, 32, 33, 63, 64])
@pytest.mark.parametrize("d,dv", [(16, 16), (16, 32), (32, 16), (32, 32)])
@pytest.mark.parametrize("masked", [True, False])
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_forward(hla, n, d, dv, masked, dtype):
    B, H = 1, 5
    pq, pk, pv = (_flat(x) for x in hla_inputs.make_qkv(B, H, 40, d, dv, seed=n, dtype=dtype))
    st0 = oracle.hla2_serial(pq, pk, pv, masked=masked, return_state=True)[1].astype(np.float32)
    q, k, v = hla_inputs.make_qkv(B, H, n, d, dv, seed=n + 1, dtype=dtype)
    t = [hla_inputs.as_torch(x, dtype, DEV) for x in (q, k, v)]
    f = [_flat(x) for x in (q, k, v)]
    for start in (None, st0):
        ref, den, rst = oracle.hla2_serial(*f, masked=masked, state_in=start, return_state=True, return_den=True)
        given = None if start is None else torch.from_numpy(st0).to(DEV).reshape(B, H, -1)
        kept = torch.empty((B, H, st0.shape[1]), device=DEV) if given is None else given.clone()
        num = hla.hla2_forward(*t, masked=masked, state_in=given, state_out=kept)
        o = hla.hla2_forward(*t, masked=masked, normalized=True, eps=hla_inputs.EPS, state_in=given, state_out=kept)
        if given is not None:
            last = hla.hla2_forward(*t, masked=masked, state_in=given)  # no state wanted
            assert torch.equal(last, num)
            kept = given
            hla.hla2_forward(*t, masked=masked, state_in=kept, state_out=kept)
        torch.cuda.synchronize()
        num, o = (_flat(x.float().cpu().numpy()) for x in (num, o))
        assert rowerr(num, ref) < TOL[dtype]
        check_normalized(o, num, ref, den, hla_inputs.EPS, TOL[dtype])
        got, want = oracle.split_state2(kept.reshape(B * H, -1).cpu().numpy(), d, dv), oracle.split_state2(rst, d, dv)
        for name in ("S", "C", "m", "G", "h"):
            scale = max(np.abs(want[name]).max(), np.abs(want["S"]).max() * np.abs(want["C"]).max(), 1.0)
            assert np.abs(got[name] - want[name]).max() <= 2e-5 * scale, name
