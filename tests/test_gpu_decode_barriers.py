"""A decode call prepares its grid barriers itself: calls on workspaces filled with any bytes, replays of one captured call with
plain calls on the same workspace in between, and calls on two streams with a workspace each all give the bits of a plain
call (GPU required)."""
import pytest
import torch

import dsmoe_inputs as gi
import paper_2404_05567_b200 as dm
from harness import Layer

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T", [1, 7, 8, 37, 128])
def test_decode_calls_on_any_workspace_contents_and_replayed(T):
    s = gi.LayerSpec(f"bar{T}", T=T, d=512, H=256, E=16, dtype="bf16", mode=gi.MODE_TOPK, K=3, router_gain=4.0)
    L = Layer(s)
    want = L.forward().clone()

    def call(x, out, ws):
        dm.dsmoe_layer_forward(L.desc, x, L.Wr_d, L.br_d, None, None, L.packed, out, None, None, ws, L.dev_status)

    for fill in (0, 255, 1, 85):
        L.ws.fill_(fill)
        assert torch.equal(L.forward(), want), fill
    g = torch.Generator(device="cuda").manual_seed(T)
    L.ws.copy_(torch.randint(0, 256, L.ws.shape, generator=g, device="cuda", dtype=torch.uint8))
    assert torch.equal(L.forward(), want)

    x, out = L.x_d.clone(), torch.empty_like(want)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        call(x, out, L.ws)
    other = Layer(s, batch="y")
    want_other = other.forward().clone()
    for i in range(40):
        x.copy_(L.x_d if i % 2 else other.x_d)
        graph.replay()
        if i % 5 == 0:
            call(L.x_d, L.out, L.ws)                       # a plain call on the same workspace in between
        assert torch.equal(out, want if i % 2 else want_other), i
    torch.cuda.synchronize()
    assert int(L.dev_status.item()) == 0

    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    ws = [L.ws, torch.empty_like(L.ws)]
    outs = [[torch.empty_like(want) for _ in range(20)] for _ in streams]
    torch.cuda.synchronize()
    for i in range(20):
        for k, st in enumerate(streams):
            with torch.cuda.stream(st):
                call(L.x_d if (i + k) % 2 else other.x_d, outs[k][i], ws[k])
    torch.cuda.synchronize()
    for k in range(2):
        for i in range(20):
            assert torch.equal(outs[k][i], want if (i + k) % 2 else want_other), (k, i)
