"""The fp32 layer of three launches against the oracle where its work is cut: one pass of rows and two, as many tokens as a CTA has threads,
reductions below, at and beyond a piece of 256 and of the largest length, ragged columns, few tiles and many, experts not by fours, empty
experts, tokens that select nothing, every expert (GPU required)."""
import pytest

import dsmoe_inputs as gi
from harness import TOL_F32, layer_parity

pytestmark = pytest.mark.gpu

CASES = [
    ("one", 1, 8, 8, 1, gi.MODE_TOPK, dict(K=1)),
    ("rows_31", 31, 264, 72, 5, gi.MODE_TOPK, dict(K=5)),
    ("tokens_512", 512, 128, 136, 32, gi.MODE_TOPK, dict(K=2)),             # as many as a CTA has threads
    ("two_passes", 96, 72, 264, 2, gi.MODE_THRESHOLD, dict(eps=0.001)),     # nearly every token selects both experts
    ("longest", 30, 512, 1024, 3, gi.MODE_ALL, dict()),
    ("many_tiles", 70, 136, 1016, 32, gi.MODE_TOPK, dict(K=3)),
    ("nothing", 90, 256, 256, 16, gi.MODE_THRESHOLD, dict(eps=0.4)),
    ("at_least_one", 90, 504, 40, 18, gi.MODE_THRESHOLD, dict(eps=0.9, min_k=1)),
]


@pytest.mark.parametrize("case", CASES, ids=[c[0] for c in CASES])
def test_layer_f32(case):
    name, T, d, H, E, mode, sel = case
    r = layer_parity(gi.LayerSpec("lf32_" + name, T=T, d=d, H=H, E=E, dtype="f32", mode=mode, router_gain=4.0, **sel))
    assert r["err_rows"] <= TOL_F32, (r["err_rows"], r["err"])
