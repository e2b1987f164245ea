"""The tile-by-tile backward held close to the fp64 oracle: long sequences, many heads, and the normalised output
with nonnegative features and a small eps, as it is used.  What the bf16 results' rounding alone gives is known: at
most 2^-8 of a value, and over many values, their logarithms evenly spread, sqrt(3 / (8 ln 2)) 2^-7 / sqrt(12) =
1.66e-3 in the root mean square.  Before the rounding, intermediates are pairs of bf16 (2^-17 each); with every one of
them rounded so, a 64-bit evaluation of the same formulas is within 6.2e-5 = 2^-14 of a head's largest row at these
sizes.  So a row may be off by 2^-8 of itself and 2^-13 of the largest, and all rows together by a tenth more than
the rounding; without the lower half of an intermediate they would be off by about 2.2e-3."""
import numpy as np
import pytest
import torch

import hla_inputs
import oracle

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.fixture(scope="module")
def hla():
    from paper_2510_27258_gb300 import build
    build.build()
    from paper_2510_27258_gb300 import hla as binding
    return binding


@pytest.mark.parametrize("heads,n,d,dv,normalized", [
    (1, 4096, 128, 128, False), (2, 1100, 128, 128, True), (2, 1100, 64, 128, True), (2, 1100, 128, 64, False),
    (400, 40, 128, 128, True), (400, 40, 128, 128, False), (700, 130, 128, 64, False), (4, 300, 128, 128, True)])
def test_close(hla, heads, n, d, dv, normalized):
    q, k, v = hla_inputs.make_qkv(1, heads, n, d, dv, seed=n, dtype="bf16")
    if normalized:
        q, k = np.abs(q), np.abs(k)
    g = hla_inputs.round_to(np.random.default_rng(n).standard_normal((1, heads, n, dv)), "bf16")
    t = [hla_inputs.as_torch(x, "bf16", DEV) for x in (q, k, v, g)]
    assert hla.hla2_backward_path(1, heads, n, d, dv, normalized=normalized) == 1
    got = hla.hla2_backward(*t, normalized=normalized, eps=1e-6)
    some = np.unique(np.linspace(0, heads - 1, 12).astype(int))
    ref = oracle.hla2_backward(*(x[0, some] for x in (q, k, v, g)), normalized=normalized, eps=1e-6, nthreads=12)
    for name, a, b in zip(("dq", "dk", "dv"), got, ref):
        err = np.linalg.norm(a[0, some].float().cpu().numpy().astype(np.float64) - b, axis=-1)
        row = np.linalg.norm(b, axis=-1)
        assert (err <= 2.0 ** -8 * row + 2.0 ** -13 * row.max(axis=-1, keepdims=True)).all(), name
        assert np.linalg.norm(err) <= 1.1 * 1.66e-3 * np.linalg.norm(row), name
