"""The three launches of the attention layer for a few decoding tokens against the oracle, where their work is cut: token counts at the
edges of the projections' columns (16, 32, 64), caches shorter than a unit of keys, as long as one, and cut over many CTAs, tokens
that share a sequence, see one key or select nothing, experts whose reduction is one or two blocks, every head width (GPU required)."""
import math

import numpy as np
import pytest
import torch

import dsmoe_inputs as gi
import paper_2404_05567_b200 as dm
from harness import TOL_BF16, to_dev
from test_gpu_moa import _moa_case, _run

pytestmark = pytest.mark.gpu

CASES = [
    # name, T, d, E, n_head, d_head, n_seq, L, layout, mode, selection
    ("one_token_long", 1, 512, 8, 4, 128, 1, 5000, "full", gi.MODE_TOPK, dict(K=5)),          # one token's keys over every CTA
    ("one_token_short", 1, 128, 5, 1, 64, 1, 9, "full", gi.MODE_TOPK, dict(K=2)),             # less than a unit; experts not by fours
    ("edge_16", 16, 320, 16, 2, 64, 16, 16, "decode", gi.MODE_TOPK, dict(K=6)),
    ("edge_17", 17, 256, 8, 4, 96, 17, 17, "decode", gi.MODE_TOPK, dict(K=5)),
    ("edge_33", 33, 1024, 8, 4, 96, 33, 700, "decode", gi.MODE_ALL, dict()),
    ("edge_64", 64, 2048, 16, 2, 64, 64, 300, "decode", gi.MODE_TOPK, dict(K=6)),
    ("shared_sequences", 30, 256, 4, 2, 128, 7, 129, "mixed", gi.MODE_TOPK, dict(K=3)),
    ("nothing_selected", 40, 256, 16, 2, 64, 40, 90, "mixed", gi.MODE_THRESHOLD, dict(eps=0.3)),
    ("wide_groups", 12, 192, 3, 8, 128, 12, 40, "mixed", gi.MODE_ALL, dict()),                # a cluster of four over three blocks
]


@pytest.mark.parametrize("case", CASES, ids=[c[0] for c in CASES])
def test_moa_decode(case):
    name, T, d, E, nh, dh, n_seq, L, layout, mode, sel = case
    s, x, Wr, br, Wq, Wo, Kc, Vc, seq, pos = _moa_case(name, T, d, E, nh, dh, n_seq, L, layout, mode, **sel)
    if name == "nothing_selected":
        seq = np.arange(T, dtype=np.int32)
    e, er = _run(s, x, Wr, br, Wq, Wo, Kc, Vc, seq, pos, nh, 1.0 / math.sqrt(dh))
    assert er <= TOL_BF16, (e, er)


def test_steps_that_change_positions_and_cache_in_place():
    """Steps without a wait in between, each behind kernels that move the positions on, hand tokens other sequences and write new keys and
    values into the same buffers: the bits of the same steps on buffers of their own with a wait after each."""
    T, d, E, nh, dh, L, steps = 24, 256, 8, 4, 128, 200, 10
    s, x, Wr, br, Wq, Wo, Kc, Vc, seq, pos = _moa_case("in_place", T, d, E, nh, dh, T, L, "decode", gi.MODE_TOPK, K=5)
    desc = dm.make_desc(T, d, nh * dh, E, dm.BF16, dm.SELECT_TOPK, K=5)
    packed = torch.empty(dm.dsmoe_packed_size(desc), dtype=torch.uint8, device="cuda")
    dm.dsmoe_pack_weights(desc, to_dev(Wq), to_dev(Wo), packed)
    ws = torch.empty(dm.dsmoe_workspace_size_packed(desc), dtype=torch.uint8, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    x_d, Wr_d, br_d, K_d, V_d = (to_dev(a) for a in (x, Wr, br, Kc, Vc))
    seq_d, pos_d = to_dev(seq), torch.full((T,), 90, dtype=torch.int32, device="cuda") + torch.arange(T, device="cuda", dtype=torch.int32)
    g = torch.Generator(device="cuda").manual_seed(3)
    new = torch.randn((steps, 2, T, nh, dh), generator=g, device="cuda").bfloat16()
    every = torch.arange(T, device="cuda")

    def run(wait):
        K, V, q, p, outs = K_d.clone(), V_d.clone(), seq_d.clone(), pos_d.clone(), []
        for i in range(steps):
            q.copy_(q.roll(1))
            p.add_(7)
            K[every, :, p.long()], V[every, :, p.long()] = new[i, 0], new[i, 1]
            out = torch.empty((T, d), dtype=torch.bfloat16, device="cuda")
            args = [t.clone() for t in (K, V, q, p)] if wait else (K, V, q, p)
            if wait:
                torch.cuda.synchronize()
            dm.dsmoe_moa_forward(desc, nh, 0.09, *args, x_d, Wr_d, br_d, packed, out, None, None, ws, status)
            if wait:
                torch.cuda.synchronize()
            outs.append(out)
        torch.cuda.synchronize()
        return outs

    for a, b in zip(run(True), run(False)):
        assert torch.equal(a, b)
    assert int(status.item()) == 0
