"""The 64-token chunk kernels on the CUDA cores at the edges of their tiles: lengths around a chunk,
every padded head size, ragged mixes of d and dv, states in and out, against the fp64 oracle.  Bars as
in tests/test_gpu_hla2.py: 1e-4 of the row norm for fp32 tokens, states 2e-5 of max(|part|, |S||C|)."""
import numpy as np
import pytest
import torch

import hla_inputs
import oracle
from parity import TOL, check_normalized, rowerr

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
LENGTHS = [1, 63, 64, 65, 128, 577]
SIZES = [(16, 16), (32, 16), (16, 128), (64, 32), (64, 64), (128, 128)]


@pytest.fixture(scope="module")
def hla():
    from paper_2510_27258_gb300 import build
    build.build()
    from paper_2510_27258_gb300 import hla as binding
    return binding


def _flat(x):
    return x.reshape((-1,) + x.shape[2:])


def _gpu(*xs):
    return [hla_inputs.as_torch(x, "f32", DEV) for x in xs]


@pytest.mark.parametrize("n", LENGTHS)
@pytest.mark.parametrize("d,dv", SIZES)
@pytest.mark.parametrize("masked", [True, False])
def test_forward(hla, n, d, dv, masked):
    """Outputs, plain and normalised, and from a state, with the final state written where the state came from."""
    B, H = 1, 3
    pq, pk, pv = (_flat(x) for x in hla_inputs.make_qkv(B, H, 40, d, dv, seed=n, dtype="f32"))
    st0 = oracle.hla2_serial(pq, pk, pv, masked=masked, return_state=True)[1].astype(np.float32)
    q, k, v = hla_inputs.make_qkv(B, H, n, d, dv, seed=n + 1, dtype="f32")
    t = _gpu(q, k, v)
    num = hla.hla2_forward(*t, masked=masked)
    o = hla.hla2_forward(*t, masked=masked, normalized=True, eps=hla_inputs.EPS)
    st = torch.from_numpy(st0).to(DEV).reshape(B, H, -1)
    cont = hla.hla2_forward(*t, masked=masked, state_in=st, state_out=st)
    torch.cuda.synchronize()
    ref, den = oracle.hla2_serial(_flat(q), _flat(k), _flat(v), masked=masked, return_den=True)
    assert rowerr(_flat(num.cpu().numpy()), ref) < TOL["f32"]
    check_normalized(_flat(o.cpu().numpy()), _flat(num.cpu().numpy()), ref, den, hla_inputs.EPS, TOL["f32"])
    ref, rst = oracle.hla2_serial(_flat(q), _flat(k), _flat(v), masked=masked, state_in=st0, return_state=True)
    assert rowerr(_flat(cont.cpu().numpy()), ref) < TOL["f32"]
    got, want = oracle.split_state2(st.reshape(B * H, -1).cpu().numpy(), d, dv), oracle.split_state2(rst, d, dv)
    for name in ("S", "C", "m", "G", "h"):
        scale = max(np.abs(want[name]).max(), np.abs(want["S"]).max() * np.abs(want["C"]).max(), 1.0)
        assert np.abs(got[name] - want[name]).max() <= 2e-5 * scale, name


def test_forward_overlapping_states(hla):
    """state_out one head behind state_in in the same buffer."""
    B, H, n, d = 1, 4, 130, 32
    pq, pk, pv = (_flat(x) for x in hla_inputs.make_qkv(B, H, 40, d, d, seed=1, dtype="f32"))
    st0 = oracle.hla2_serial(pq, pk, pv, return_state=True)[1].astype(np.float32)
    q, k, v = hla_inputs.make_qkv(B, H, n, d, d, seed=2, dtype="f32")
    buf = torch.zeros((H + 1, st0.shape[1]), dtype=torch.float32, device=DEV)
    buf[1:] = torch.from_numpy(st0).to(DEV)
    out = hla.hla2_forward(*_gpu(q, k, v), state_in=buf[1:], state_out=buf[:H])
    torch.cuda.synchronize()
    ref, rst = oracle.hla2_serial(_flat(q), _flat(k), _flat(v), state_in=st0, return_state=True)
    assert rowerr(_flat(out.cpu().numpy()), ref) < TOL["f32"]
    assert np.abs(buf[:H].cpu().numpy() - rst).max() <= 1e-4 * np.abs(rst).max()


@pytest.mark.parametrize("n", LENGTHS)
@pytest.mark.parametrize("d,dv", SIZES)
def test_ahla(hla, n, d, dv):
    """AHLA outputs, plain and normalised, and from a state, with the final state written where the state came from."""
    B, H = 1, 3
    pq, pk, pv = (_flat(x) for x in hla_inputs.make_qkv(B, H, 40, d, dv, seed=n, dtype="f32"))
    st0 = oracle.ahla_serial(pq, pk, pv, return_state=True)[1].astype(np.float32)
    q, k, v = hla_inputs.make_qkv(B, H, n, d, dv, seed=n + 1, dtype="f32")
    t = _gpu(q, k, v)
    num = hla.ahla_forward(*t)
    o = hla.ahla_forward(*t, normalized=True, eps=hla_inputs.EPS)
    st = torch.from_numpy(st0).to(DEV).reshape(B, H, -1)
    cont = hla.ahla_forward(*t, state_in=st, state_out=st)
    torch.cuda.synchronize()
    ref, den = oracle.ahla_serial(_flat(q), _flat(k), _flat(v), return_den=True)
    assert rowerr(_flat(num.cpu().numpy()), ref) < TOL["f32"]
    check_normalized(_flat(o.cpu().numpy()), _flat(num.cpu().numpy()), ref, den, hla_inputs.EPS, TOL["f32"])
    ref, rst = oracle.ahla_serial(_flat(q), _flat(k), _flat(v), state_in=st0, return_state=True)
    assert rowerr(_flat(cont.cpu().numpy()), ref) < TOL["f32"]
    assert np.abs(st.reshape(B * H, -1).cpu().numpy() - rst).max() <= 2e-5 * np.abs(rst).max()


@pytest.mark.parametrize("n", LENGTHS)
@pytest.mark.parametrize("d,dv", SIZES)
@pytest.mark.parametrize("normalized", [False, True])
def test_backward(hla, n, d, dv, normalized):
    """Gradients; the normalised output with eps such that den + eps >= 1 on every row."""
    B, H = 1, 2
    q, k, v = hla_inputs.make_qkv(B, H, n, d, dv, seed=n, dtype="f32")
    g = hla_inputs.round_to(np.random.default_rng(n).standard_normal((B, H, n, dv)), "f32")
    den = oracle.hla2_serial(_flat(q), _flat(k), _flat(v), return_den=True)[1]
    eps = 1.0 + max(0.0, -float(den.min()))
    got = hla.hla2_backward(*_gpu(q, k, v, g), normalized=normalized, eps=eps)
    torch.cuda.synchronize()
    ref = oracle.hla2_backward(_flat(q), _flat(k), _flat(v), _flat(g), normalized=normalized, eps=eps, nthreads=8)
    for name, a, b in zip(("dq", "dk", "dv"), got, ref):
        assert rowerr(_flat(a.cpu().numpy()), b) < TOL["f32"], name
