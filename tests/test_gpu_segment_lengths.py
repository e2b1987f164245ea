"""How the fused forward cuts heads into segments.  A cut rounds outputs once more, so heads that occupy
half the SMs are not cut, and fewer heads are cut into 2 to 8 tiles by the schedule model that is restated
here: the outputs have to be, bit for bit, those of the length that it gives."""
import heapq

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


def length(heads, tiles, sms):
    def span(L):
        free, last = [0.0] * sms, 0.0
        for g in range(-(-tiles // L)):
            li = min(L, tiles - g * L)
            for _ in range(heads):
                t = heapq.heappop(free)
                end = t + 5.5 * li + (2.1 * li + 7.0 if g else 2.0) + (4.7 + 5.6 * g if t == 0.0 else 0.0)
                heapq.heappush(free, end)
                last = max(last, end)
        return last

    if 2 * heads >= sms:
        return tiles
    return min(tiles, min(range(2, max(2, min(8, tiles)) + 1), key=lambda L: (span(L), L)))


@pytest.mark.parametrize("heads,n,d,normalized,state", [
    (32, 1999, 128, False, True), (64, 2048, 128, False, False), (80, 600, 64, True, False),
    (160, 1024, 128, True, False), (128, 700, 64, False, True), (24, 1500, 64, False, False),
    (12, 700, 64, True, False), (75, 900, 128, True, False), (76, 900, 128, True, False), (4, 200, 64, False, False)])
def test_length(hla, monkeypatch, heads, n, d, normalized, state):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    q, k, v = (hla_inputs.as_torch(x, "bf16", DEV)
               for x in hla_inputs.make_qkv(1, heads, n, d, d, seed=heads, dtype="bf16"))

    def call():
        st = torch.empty((1, heads, hla.hla2_state_floats(d, d)), device=DEV) if state else None
        out = hla.hla2_forward(q, k, v, normalized=normalized, eps=1.0, state_out=st)
        return [out] + ([st] if state else [])

    chosen = call()
    monkeypatch.setenv("HLA_FUSED_SEGMENT_TILES", str(length(heads, -(-n // 128), sms)))
    for a, b in zip(chosen, call()):
        assert torch.equal(a, b)
