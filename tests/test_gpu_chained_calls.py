"""Every chained entry point, not only dsmoe_layer_forward: calls that follow one another on a stream without a wait, alternating
between two inputs over one workspace, and the same calls captured into a graph and replayed, give the bits of the same calls
with a wait after each (GPU required)."""
import numpy as np
import pytest
import torch

import dsmoe_inputs as gi
import paper_2404_05567_b200 as dm
from harness import Layer, to_dev
from test_gpu_moa import _moa_case

pytestmark = pytest.mark.gpu


def _pair(t):
    return [t, t.flip(0).contiguous()]


def _layer(**kw):
    L = Layer(gi.LayerSpec("chained", router_gain=4.0, **kw))

    def run(x):
        out, mask, counts = torch.empty_like(L.out), torch.empty_like(L.mask), torch.zeros_like(L.counts)
        dm.dsmoe_layer_forward(L.desc, x, L.Wr_d, L.br_d, L.W1_d, L.W2_d, L.packed, out, mask, counts, L.ws, L.dev_status)
        return out, mask, counts
    return _pair(L.x_d), run, L.dev_status


def _stages(**kw):
    """router, selection, statistics, grouping, experts, aggregation, each through its own entry point"""
    L = Layer(gi.LayerSpec("chained_stages", router_gain=4.0, **kw))
    s, W, A = L.s, dm.width(L.desc), dm.amax(L.desc)
    ws = torch.empty(dm.dsmoe_workspace_size(L.desc), dtype=torch.uint8, device="cuda")

    def run(x):
        i32 = lambda *shape: torch.full(shape, -1, dtype=torch.int32, device="cuda")
        scores, mask = torch.empty((s.T, s.E), device="cuda"), torch.empty(s.T, dtype=torch.int64, device="cuda")
        k_t, counts, offsets, row_token, token_rows = i32(s.T), i32(s.E), i32(s.E + 1), i32(A), i32(s.T, W)
        row_gate, stats = torch.zeros(A, device="cuda"), torch.zeros(4096, dtype=torch.uint8, device="cuda")
        xp, yp = (torch.zeros((A, s.d), dtype=L.native, device="cuda") for _ in range(2))
        out = torch.empty_like(L.out)
        dm.dsmoe_router(L.desc, x, L.Wr_d, L.br_d, scores)
        dm.dsmoe_select(L.desc, scores, mask, k_t, counts, offsets, ws)
        dm.dsmoe_stats(L.desc, scores, mask, stats)
        dm.dsmoe_permute(L.desc, x, scores, mask, offsets, row_token, row_gate, token_rows, xp, ws)
        dm.dsmoe_expert_mlp(L.desc, xp, L.W1_d, L.W2_d, L.packed, offsets, yp, ws, L.dev_status)
        dm.dsmoe_combine(L.desc, yp, row_gate, token_rows, k_t, out)
        return scores, mask, k_t, counts, offsets, stats, row_token, row_gate, token_rows, out
    return _pair(L.x_d), run, L.dev_status


def _training(pack, **kw):
    L = Layer(gi.LayerSpec("chained_training", mode=gi.MODE_ALL, router_gain=4.0, **kw), pack=pack)
    s = L.s
    g = torch.Generator(device="cuda").manual_seed(1)
    dO = torch.randn((s.T, s.d), generator=g, device="cuda").to(L.native)
    ws = torch.empty(dm.dsmoe_workspace_size(L.desc), dtype=torch.uint8, device="cuda")

    def run(x):
        scores, loss, grad, dS = (torch.empty(sh, device="cuda") for sh in ((s.T, s.E), (3,), (s.T, s.E), (s.T, s.E)))
        dA = torch.empty((s.T, s.E * s.H), dtype=L.native, device="cuda")
        dm.dsmoe_router(L.desc, x, L.Wr_d, L.br_d, scores)
        dm.dsmoe_mi_loss(L.desc, scores, loss, grad, ws)
        dm.dsmoe_dense_backward(L.desc, x, L.W1_d, L.W2_d, L.packed, scores, None, dO, dS, dA, ws, L.dev_status)
        return scores, loss, grad, dS, dA
    return _pair(L.x_d), run, L.dev_status


def _moa(T, d, E, nh, dh, n_seq, L, order, **sel):
    s, x, Wr, br, Wq, Wo, Kc, Vc, seq, pos = _moa_case("chained_moa", T, d, E, nh, dh, n_seq, L, "decode" if T == n_seq else "mixed",
                                                       gi.MODE_TOPK, **sel)
    if order == "round":
        seq = (np.arange(T) % n_seq).astype(np.int32)
    elif order == "sorted":
        seq = np.sort(seq)
    desc = dm.make_desc(T, d, nh * dh, E, dm.BF16, gi.MODE_TOPK, K=s.K)
    packed = torch.empty(dm.dsmoe_packed_size(desc), dtype=torch.uint8, device="cuda")
    dm.dsmoe_pack_weights(desc, to_dev(Wq), to_dev(Wo), packed)
    ws = torch.empty(dm.dsmoe_workspace_size_packed(desc), dtype=torch.uint8, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    Wr_d, br_d, K_d, V_d, seq_d, pos_d, x_d = (to_dev(a) for a in (Wr, br, Kc, Vc, seq, pos, x))

    def run(x):
        out, mask = torch.empty((T, d), dtype=torch.bfloat16, device="cuda"), torch.empty(T, dtype=torch.int64, device="cuda")
        counts = torch.zeros(64, dtype=torch.int32, device="cuda")
        dm.dsmoe_moa_forward(desc, nh, 0.1, K_d, V_d, seq_d, pos_d, x, Wr_d, br_d, packed, out, mask, counts, ws, status)
        return out, mask, counts
    return _pair(x_d), run, status


CALLS = {
    "layer_plain": lambda: _layer(T=200, d=256, H=128, E=8, dtype="f32", mode=gi.MODE_TOPK, K=2),
    "layer_grouped": lambda: _layer(T=300, d=512, H=256, E=32, dtype="bf16", mode=gi.MODE_TOPK, K=4),
    "layer_fused_sum": lambda: _layer(T=700, d=512, H=256, E=4, dtype="bf16", mode=gi.MODE_TOPK, K=2, fuse_combine=1),
    "layer_threshold_topk": lambda: _layer(T=513, d=256, H=128, E=16, dtype="bf16", mode=gi.MODE_THRESHOLD_TOPK, eps=0.03),
    "layer_dense": lambda: _layer(T=700, d=256, H=128, E=8, dtype="bf16", mode=gi.MODE_ALL),
    # either side of the number of tokens beyond which the aggregation is launched the ordinary way (d 256 to 128 tokens is layer_f32.cu's)
    "layer_plain_wide_128": lambda: _layer(T=128, d=520, H=128, E=8, dtype="f32", mode=gi.MODE_TOPK, K=2),
    "layer_plain_wide_129": lambda: _layer(T=129, d=520, H=128, E=8, dtype="f32", mode=gi.MODE_TOPK, K=2),
    "layer_plain_128": lambda: _layer(T=128, d=256, H=128, E=8, dtype="f32", mode=gi.MODE_TOPK, K=2),
    "layer_plain_129": lambda: _layer(T=129, d=256, H=128, E=8, dtype="f32", mode=gi.MODE_TOPK, K=2),
    "layer_grouped_129": lambda: _layer(T=129, d=512, H=256, E=32, dtype="bf16", mode=gi.MODE_TOPK, K=4, fuse_combine=0),
    "stages_f32": lambda: _stages(T=77, d=136, H=72, E=5, dtype="f32", mode=gi.MODE_TOPK, K=2),
    "stages_bf16": lambda: _stages(T=517, d=256, H=128, E=33, dtype="bf16", mode=gi.MODE_THRESHOLD, eps=0.02),
    "stages_threshold_topk": lambda: _stages(T=300, d=128, H=64, E=16, dtype="bf16", mode=gi.MODE_THRESHOLD_TOPK, eps=0.05),
    "training_packed": lambda: _training(True, T=700, d=512, H=256, E=16, dtype="bf16"),
    "training_plain": lambda: _training(False, T=40, d=128, H=72, E=6, dtype="f32"),
    "moa_decode": lambda: _moa(5, 512, 8, 2, 64, 5, 700, "", K=3),
    "moa_decode_short": lambda: _moa(9, 512, 8, 2, 64, 9, 80, "", K=3),
    "moa_prompts": lambda: _moa(203, 512, 8, 2, 64, 2, 300, "sorted", K=5),
    "moa_prompts_dense": lambda: _moa(4701, 1024, 8, 2, 64, 3, 300, "sorted", K=4),
    "moa_mixed": lambda: _moa(700, 256, 8, 2, 64, 5, 90, "round", K=5),
    "moa_mixed_long": lambda: _moa(1100, 256, 8, 4, 64, 5, 600, "round", K=5),
    "moa_mixed_dense_long": lambda: _moa(4701, 1024, 8, 2, 64, 7, 600, "round", K=4),
    "moa_plain": lambda: _moa(60, 256, 8, 2, 32, 3, 50, "sorted", K=2),
}


@pytest.mark.parametrize("name", CALLS)
def test_calls_without_a_wait_and_replayed_from_a_graph(name):
    inputs, run, status = CALLS[name]()
    want = []
    for x in inputs:
        want.append([t.clone() for t in run(x)])
        torch.cuda.synchronize()
    got = [run(inputs[i % 2]) for i in range(10)]
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    for i, outs in enumerate(got):
        for a, b in zip(outs, want[i % 2]):
            assert torch.equal(a, b), i

    # captured: behind a join of two streams (two predecessors), then one after the other
    x, other, side = inputs[0].clone(), torch.zeros(1000, device="cuda"), torch.cuda.Stream()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(side):
            other.add_(1.0)
        x2 = x.flip(0).contiguous()
        torch.cuda.current_stream().wait_stream(side)
        first = run(x)
        second = run(x2)
    for k in range(6):
        x.copy_(inputs[k % 2])
        graph.replay()
        torch.cuda.synchronize()
        for outs, at in ((first, k % 2), (second, 1 - k % 2)):
            for a, b in zip(outs, want[at]):
                assert torch.equal(a, b), k
    assert int(status.item()) == 0
    del graph
