"""Gradients written over the tokens that they are of: bit for bit those of a call with outputs of their own, on every
path of the backward (called through the C entry point; the Python wrapper makes its own outputs)."""
import ctypes

import numpy as np
import pytest
import torch

import hla_inputs

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
DTYPES = {"f32": torch.float32, "bf16": torch.bfloat16}


@pytest.fixture(scope="module")
def hla():
    from paper_2510_27258_gb300 import build
    build.build()
    from paper_2510_27258_gb300 import hla as binding
    return binding


def _call(hla, t, outs, normalized):
    B, H, n, d = t[0].shape
    ws = hla.alloc_workspace(hla.hla2_backward_workspace_bytes(B, H, n, d, d, 64, t[0].dtype), DEV)
    code = hla.lib().hla2_backward(*(x.data_ptr() for x in t + outs), int(t[0].dtype == torch.bfloat16), B, H, n, d, d,
                                   int(normalized), ctypes.c_float(1.0), 64, ws.data_ptr(), ws.numel(), None)
    assert code == hla.HLA_OK
    torch.cuda.synchronize()
    return [x.clone() for x in outs]


@pytest.mark.parametrize("d,dtype", [(32, "f32"), (64, "f32"), (128, "f32"), (32, "bf16"), (64, "bf16"), (128, "bf16")])
@pytest.mark.parametrize("normalized", [False, True])
@pytest.mark.parametrize("over", [(0, None, None), (1, 0, None), (None, None, 3), (0, 1, 2), (3, 2, 0)])
def test_over_tokens(hla, d, dtype, normalized, over):
    """over: for dq, dk, dv the token array (0 q, 1 k, 2 v, 3 dout) that it lies over"""
    B, H, n = 1, 40, 400
    q, k, v = hla_inputs.make_qkv(B, H, n, d, d, seed=d, dtype=dtype)
    g = hla_inputs.round_to(np.random.default_rng(d).standard_normal((B, H, n, d)), dtype)
    tokens = [hla_inputs.as_torch(np.abs(x) if normalized and i < 2 else x, dtype, DEV)
              for i, x in enumerate((q, k, v, g))]
    want = _call(hla, tokens, [torch.empty_like(x) for x in tokens[:3]], normalized)
    t = [x.clone() for x in tokens]
    got = _call(hla, t, [torch.empty_like(tokens[0]) if o is None else t[o] for o in over], normalized)
    for a, b in zip(got, want):
        assert torch.equal(a, b)

