"""The tile-by-tile backward on the tensor cores (bf16 tokens, a head size of 128) against the fp64
oracle: one tile, its edges, several tiles, mixed head sizes, plain and normalised.  Bar: 2e-2 of the row
norm (bf16 tokens); the normalised output with eps such that den + eps >= 1 on every row."""
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


def _flat(x):
    return x.reshape((-1,) + x.shape[2:])


@pytest.mark.parametrize("n", [1, 127, 128, 129, 300, 1100])
@pytest.mark.parametrize("d,dv", [(128, 128), (64, 128), (128, 64)])
@pytest.mark.parametrize("normalized", [False, True])
def test_backward_tiles(hla, n, d, dv, normalized):
    B, H = 1, 3
    assert hla.hla2_backward_path(B, H, n, d, dv, normalized=normalized) == 1
    q, k, v = hla_inputs.make_qkv(B, H, n, d, dv, seed=n, dtype="bf16")
    g = hla_inputs.round_to(np.random.default_rng(n).standard_normal((B, H, n, dv)), "bf16")
    den = oracle.hla2_serial(_flat(q), _flat(k), _flat(v), return_den=True, nthreads=8)[1]
    eps = 1.0 + max(0.0, -float(den.min()))
    t = [hla_inputs.as_torch(x, "bf16", DEV) for x in (q, k, v, g)]
    ws = hla.alloc_workspace(hla.hla2_backward_workspace_bytes(B, H, n, d, dv, 64, torch.bfloat16), DEV)
    got = hla.hla2_backward(*t, normalized=normalized, eps=eps, workspace=ws)
    assert hla.hla_poll_error(ws) == hla.HLA_OK
    ref = oracle.hla2_backward(_flat(q), _flat(k), _flat(v), _flat(g), normalized=normalized, eps=eps, nthreads=8)
    for name, a, b in zip(("dq", "dk", "dv"), got, ref):
        assert rowerr(_flat(a.float().cpu().numpy()), b) < TOL["bf16"], name
