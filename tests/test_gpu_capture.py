"""Calls of several launches, each set up while the one before drains: captured in a CUDA graph and replayed, and two
at a time on two streams with a workspace each, they give bit for bit what they give alone."""
import pytest
import torch

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.fixture(scope="module")
def hla():
    from paper_2510_27258_gb300 import build
    build.build()
    from paper_2510_27258_gb300 import hla as binding
    return binding


CASES = ["forward_f32", "forward_prefill", "forward_continued", "unmasked", "ahla", "ahla_tc", "backward_f32",
         "backward_normalized", "backward_tiles", "backward_tiles_normalized", "third_order"]


def _call(hla, case, seed):
    """a function without arguments and the tensors that it writes"""
    H, n = 6, 700
    d = 128 if "tiles" in case or case in ("forward_prefill", "forward_continued", "ahla") else 32 if case == "third_order" \
        else 64
    dtype = torch.float32 if case in ("forward_f32", "unmasked", "backward_f32", "third_order") else torch.bfloat16
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    q, k, v, w = (torch.randn((1, H, n, d), generator=g, device=DEV).mul_(0.1).to(dtype) for _ in range(4))
    norm = "normalized" in case
    if norm:
        q, k = q.abs(), k.abs()
    if case.startswith("backward"):
        ws = hla.alloc_workspace(hla.hla2_backward_workspace_bytes(1, H, n, d, d, 64, dtype), DEV)
        return lambda: hla.hla2_backward(q, k, v, w, normalized=norm, eps=1e-3, workspace=ws)
    out = torch.empty_like(v)
    if case == "third_order":
        ws = hla.alloc_workspace(hla.hla3_workspace_bytes(1, H, n, d, d, 32, dtype), DEV)
        return lambda: (hla.hla3_forward(q, k, v, out, workspace=ws),)
    if case.startswith("ahla"):
        st = None if case == "ahla_tc" else torch.empty((1, H, hla.ahla_state_floats(d, d)), device=DEV)
        ws = hla.alloc_workspace(hla.ahla_workspace_bytes(1, H, n, d, d, 64, dtype), DEV)
        return lambda: (hla.ahla_forward(q, k, v, out, state_out=st, workspace=ws),) + (() if st is None else (st,))
    st = torch.empty((1, H, hla.hla2_state_floats(d, d)), device=DEV) if case != "unmasked" else None
    st0 = torch.full_like(st, 0.01) if case == "forward_continued" else None
    ws = hla.alloc_workspace(hla.hla2_workspace_bytes(1, H, n, d, d, 128, dtype), DEV)
    return lambda: (hla.hla2_forward(q, k, v, out, masked=case != "unmasked", state_in=st0, state_out=st, workspace=ws),) \
        + (() if st is None else (st,))


@pytest.mark.parametrize("case", CASES)
def test_replay(hla, case):
    call = _call(hla, case, 1)
    want = [x.clone() for x in call()]
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        outs = call()
    for _ in range(3):
        for x in outs:
            x.zero_()
        graph.replay()
        torch.cuda.synchronize()
        for a, b in zip(outs, want):
            assert torch.equal(a, b)


@pytest.mark.parametrize("case", CASES)
@pytest.mark.parametrize("other", ["forward_prefill", "backward_tiles_normalized"])
def test_two_streams(hla, case, other):
    calls = [_call(hla, case, 1), _call(hla, other, 2)]
    want = [[x.clone() for x in call()] for call in calls]
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    torch.cuda.synchronize()
    got = [[], []]
    for _ in range(5):
        for i, call in enumerate(calls):
            with torch.cuda.stream(streams[i]):
                got[i] = call()
    torch.cuda.synchronize()
    for a, b in zip(got, want):
        for x, y in zip(a, b):
            assert torch.equal(x, y)
