"""Calls that follow one another on a stream without a wait, alternating between two inputs over one workspace: every
kernel may be set up while its predecessor still runs, so none may read or write early.  The outputs are those of
the same calls with a wait after each (GPU required)."""
import pytest
import torch

import dsmoe_inputs as gi
import paper_2404_05567_b200 as dm
from harness import Layer

pytestmark = pytest.mark.gpu

CASES = [
    dict(T=64, d=256, H=512, E=8, dtype="f32", mode=gi.MODE_TOPK, K=2),
    dict(T=300, d=512, H=256, E=8, dtype="f32", mode=gi.MODE_THRESHOLD, eps=0.1),
    dict(T=129, d=256, H=128, E=8, dtype="bf16", mode=gi.MODE_TOPK, K=3),
    dict(T=300, d=512, H=256, E=32, dtype="bf16", mode=gi.MODE_TOPK, K=4),
    dict(T=4099, d=256, H=128, E=16, dtype="bf16", mode=gi.MODE_TOPK, K=3),          # more than one wave of aggregating blocks
    dict(T=513, d=256, H=128, E=16, dtype="bf16", mode=gi.MODE_THRESHOLD_TOPK, eps=0.03),
    dict(T=2000, d=512, H=1024, E=2, dtype="bf16", mode=gi.MODE_TOPK, K=2, fuse_combine=1),
    dict(T=700, d=256, H=128, E=8, dtype="bf16", mode=gi.MODE_ALL),
    dict(T=16, d=512, H=256, E=16, dtype="bf16", mode=gi.MODE_TOPK, K=4),
]


@pytest.mark.parametrize("case", CASES, ids=[f"{c['dtype']}-T{c['T']}-{c['mode']}" for c in CASES])
def test_calls_without_a_wait_between_them(case):
    L = Layer(gi.LayerSpec(f"b2b{CASES.index(case)}", router_gain=4.0, **case))
    xs = [L.x_d, L.x_d.flip(0).contiguous()]
    waited = []
    for x in xs:
        L.x_d = x
        L.forward()
        waited.append((L.out.clone(), L.mask.clone(), L.counts.clone()))
    outs = [(torch.empty_like(L.out), torch.empty_like(L.mask), torch.zeros_like(L.counts)) for _ in range(20)]
    for i, (out, mask, counts) in enumerate(outs):
        dm.dsmoe_layer_forward(L.desc, xs[i % 2], L.Wr_d, L.br_d, L.W1_d, L.W2_d, L.packed, out, mask, counts, L.ws, L.dev_status)
    torch.cuda.synchronize()
    assert int(L.dev_status.item()) == 0
    for i, got in enumerate(outs):
        for a, b in zip(got, waited[i % 2]):
            assert torch.equal(a, b), i
