"""The library keeps a bounded number of encoded tensor maps and replaces the oldest ones.  A call must not lose a map it has
just found to the next one it encodes: 600 calls of the backward pass on one x and ever new gradient buffers of the same
contents (the cache holds 256) give the same gradients every time (GPU required)."""
import pytest
import torch

import dsmoe_inputs as gi
import paper_2404_05567_b200 as dm
from harness import Layer

pytestmark = pytest.mark.gpu


def test_maps_found_in_a_call_survive_the_maps_encoded_after_them():
    s = gi.LayerSpec("map_cache", T=40, d=128, H=64, E=4, dtype="bf16", router_gain=4.0)
    L = Layer(s)
    scores = torch.softmax(torch.arange(s.T * s.E, device="cuda").reshape(s.T, s.E) % 7 * 0.3, dim=1).float().contiguous()
    row = torch.linspace(-1, 1, s.d, device="cuda").bfloat16()
    rows = row.repeat(s.T + 600, 1).contiguous()            # every window of T rows holds the same values at another address
    first = None
    for i in range(600):
        dS = torch.zeros((s.T, s.E), device="cuda")
        dA = torch.zeros((s.T, s.E * s.H), device="cuda", dtype=torch.bfloat16)
        dm.dsmoe_dense_backward(L.desc, L.x_d, None, L.W2_d, L.packed, scores, None, rows[i:i + s.T], dS, dA, L.ws, L.dev_status)
        if first is None:
            first = dS, dA
        assert torch.equal(dS, first[0]) and torch.equal(dA, first[1]), i
