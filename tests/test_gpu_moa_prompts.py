"""Attention of prompts in tiles of up to 128 rows (csrc/moa.cu, moa_attention_umma_kernel) against the oracle: the head widths, 1 to 16 rows a
token (tiles that 128 rows do and do not fill), caches that end inside a block of 64 keys, tiles of two sequences, in order and not, and of
many, values that are not finite (GPU required)."""
import math

import numpy as np
import pytest
import torch

import dsmoe_inputs as gi
import paper_2404_05567_b200 as dm
from harness import TOL_BF16, desc_of, to_dev
from test_gpu_moa import _moa_case, _run

pytestmark = pytest.mark.gpu

CASES = [
    # T, d, E, n_head, d_head, n_seq, L, layout, mode, selection
    (960, 256, 8, 4, 128, 2, 480, "prefill", gi.MODE_TOPK, dict(K=5)),          # 24 tokens a tile, a sequence's end inside one
    (1001, 256, 8, 4, 96, 7, 150, "prefill", gi.MODE_TOPK, dict(K=5)),
    (1300, 256, 16, 2, 64, 1, 1300, "prefill", gi.MODE_TOPK, dict(K=6)),        # 16 tokens a tile: 96 rows
    (152, 256, 16, 8, 64, 1, 193, "full", gi.MODE_ALL, dict()),                 # 8 tokens of 16 rows
    (4800, 64, 4, 4, 64, 3, 1600, "prefill", gi.MODE_TOPK, dict(K=1)),          # 128 tokens of one row
    (1600, 128, 8, 4, 96, 5, 130, "mixed", gi.MODE_TOPK, dict(K=3)),            # every tile of many sequences
    (1600, 128, 8, 4, 128, 5, 600, "mixed", gi.MODE_THRESHOLD, dict(eps=0.2)),  # ... left to the key-splitting kernel; tokens of no expert
]


@pytest.mark.parametrize("case", CASES, ids=lambda c: "x".join(map(str, c[:7])))
def test_prompts(case):
    T, d, E, nh, dh, n_seq, L, layout, mode, sel = case
    s, *rest = _moa_case(f"uprompt{T}x{dh}x{L}", T, d, E, nh, dh, n_seq, L, layout, mode, **sel)
    e, er = _run(s, *rest, nh, 1.0 / math.sqrt(dh), sample=60)
    assert er <= TOL_BF16, (e, er)


# Two sequences out of order with a cache beyond 512 positions: a group of four 16-row tiles with a token whose sequence is neither its
# first's nor its last's is the key-splitting kernel's, also inside a tile of 128 rows that holds no third sequence.
# T, d, E, n_head, d_head, mode, selection
OUT_OF_ORDER = [
    (1200, 128, 8, 4, 128, gi.MODE_THRESHOLD, dict(eps=0.1)),
    (1000, 128, 8, 4, 128, gi.MODE_TOPK, dict(K=5)),
    (1000, 128, 8, 4, 128, gi.MODE_TOPK, dict(K=5, fuse_combine=1)),
    (1003, 128, 8, 4, 96, gi.MODE_TOPK, dict(K=5, fuse_combine=2)),
    (1201, 128, 8, 4, 96, gi.MODE_THRESHOLD, dict(eps=0.15)),
    (1250, 128, 16, 2, 64, gi.MODE_TOPK, dict(K=6)),
    (1200, 128, 4, 4, 64, gi.MODE_ALL, dict()),
    (1000, 128, 9, 4, 64, gi.MODE_TOPK, dict(K=9)),                             # three groups of four tokens a tile
    # the dense output projection
    (2369, 2048, 8, 4, 128, gi.MODE_TOPK, dict(K=5)),
    (2433, 2048, 8, 4, 96, gi.MODE_TOPK, dict(K=5)),
    (4700, 1024, 8, 2, 64, gi.MODE_TOPK, dict(K=4)),
]


@pytest.mark.parametrize("order", ["random", "one_inside_a_group"])
@pytest.mark.parametrize("case", OUT_OF_ORDER, ids=lambda c: f"T{c[0]}-{c[3]}x{c[4]}-m{c[5]}" + "".join(f"-{k}{v}" for k, v in c[6].items()))
def test_two_sequences_out_of_order_in_a_long_cache(case, order):
    T, d, E, nh, dh, mode, sel = case
    s, x, Wr, br, Wq, Wo, Kc, Vc, seq, pos = _moa_case(f"uorder{T}x{dh}", T, d, E, nh, dh, 2, 600, "mixed", mode, **sel)
    if order == "one_inside_a_group":                      # A A B A ... | ... B, tile by tile
        W = s.K if mode == gi.MODE_TOPK else E
        group = 4 * (16 // W)
        tile = group * (128 // (group * W))
        at = np.arange(T) % tile
        seq = ((at == 2) | (at >= group)).astype(np.int32)
    e, er = _run(s, x, Wr, br, Wq, Wo, Kc, Vc, seq, pos, nh, 1.0 / math.sqrt(dh))
    assert er <= TOL_BF16, (e, er)


def test_negative_scale():
    s, *rest = _moa_case("uneg", 960, 256, 8, 4, 128, 2, 480, "prefill", gi.MODE_TOPK, K=5)
    e, er = _run(s, *rest, 4, -0.05, sample=40)
    assert er <= TOL_BF16, (e, er)


@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
def test_a_value_that_is_not_finite_stays_with_the_tokens_near_it(bad):
    s, x, Wr, br, Wq, Wo, Kc, Vc, seq, pos = _moa_case("unan", 960, 256, 8, 4, 128, 2, 480, "prefill", gi.MODE_TOPK, K=5)
    desc, V = desc_of(s.replace(out_fp32=1)), to_dev(Vc)
    packed = torch.empty(dm.dsmoe_packed_size(desc), dtype=torch.uint8, device="cuda")
    dm.dsmoe_pack_weights(desc, to_dev(Wq), to_dev(Wo), packed)
    ws = torch.empty(dm.dsmoe_workspace_size_packed(desc), dtype=torch.uint8, device="cuda")
    args = [to_dev(a) for a in (seq, pos, x, Wr, br)]
    outs = []
    for v in (None, bad):
        if v is not None:
            V[1, :, 300, 5] = v                              # seen from position 300 of the second sequence on
        out = torch.empty((s.T, s.d), dtype=torch.float32, device="cuda")
        dm.dsmoe_moa_forward(desc, 4, 0.088, to_dev(Kc), V, *args, packed, out, None, None, ws, None)
        outs.append(out)
    torch.cuda.synchronize()
    # tiles of 16 rows are 3 tokens: none before position 297 shares one with a token that sees the value
    assert torch.isfinite(outs[1][:480 + 297]).all() and not torch.isfinite(outs[1][480 + 300:]).all(dim=1).any()
    rms = outs[0].square().mean(dim=1).sqrt()
    assert ((outs[1] - outs[0])[:480 + 297].abs().amax(dim=1) <= TOL_BF16 * rms[:480 + 297]).all()
