"""The three launches of the attention layer for a few decoding tokens against the oracle, where their work is cut: token counts at the
edges of the projections' columns (16, 32, 64), caches shorter than a unit of keys, as long as one, and cut over many CTAs, tokens
that share a sequence, see one key or select nothing, experts whose reduction is one or two blocks, every head width (GPU required)."""
import math

import numpy as np
import pytest

import dsmoe_inputs as gi
from harness import TOL_BF16
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
