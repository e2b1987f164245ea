"""Decode steps whose output lies over the query, key or value: the result and the state are, bit for bit, those of
a step with an output of its own, for every number of blocks per head."""
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


@pytest.mark.parametrize("heads", [1, 8, 9, 32, 64, 65, 150, 300, 700])
@pytest.mark.parametrize("d", [16, 64, 128])
@pytest.mark.parametrize("normalized", [False, True])
@pytest.mark.parametrize("kind", ["hla2_step", "hla2_step_sde", "ahla_step"])
def test_output_over_a_token(hla, heads, d, normalized, kind):
    size = {"hla2_step": hla.hla2_state_floats, "hla2_step_sde": hla.hla2_sde_state_floats,
            "ahla_step": hla.ahla_state_floats}[kind](d, d)
    tokens = [hla_inputs.as_torch(x[:, :, 0], "f32", DEV)
              for x in hla_inputs.make_qkv(1, heads, 1, d, d, seed=heads, dtype="f32")]
    start = torch.randn((1, heads, size), generator=torch.Generator().manual_seed(heads)).to(DEV)

    def step(over):
        t, st = [x.clone() for x in tokens], start.clone()
        out = getattr(hla, kind)(*t, st, None if over is None else t[over], normalized=normalized, eps=1.0)
        return out, st

    want = step(None)
    for over in range(3):
        for a, b in zip(step(over), want):
            assert torch.equal(a, b)
