"""The grouped layer's launch where it finds its rows in the selection words itself (csrc/mlp_grouped.cu), against the oracle: chunks of 32
tokens that are full, short and without a row, tokens without an expert, all selection rules, row tiles on both sides of 128, the largest
token count (GPU required)."""
import pytest

import dsmoe_inputs as gi
import paper_2404_05567_b200 as dm
from harness import TOL_BF16, layer_parity

pytestmark = pytest.mark.gpu

# T, d, H, E, mode, K, eps, min_k
CASES = [
    (1024, 1024, 64, 16, dm.SELECT_TOPK, 4, 0.0, 0),
    (993, 1088, 320, 3, dm.SELECT_TOPK, 3, 0.0, 0),             # every token in every expert, a last chunk of one token
    (768, 1024, 64, 32, dm.SELECT_THRESHOLD, 0, 1.3, 0),        # tokens without an expert
    (384, 1088, 128, 64, dm.SELECT_THRESHOLD, 0, 0.9, 1),
    (384, 1024, 64, 33, dm.SELECT_THRESHOLD_TOPK, 0, 0.9, 0),
    (129, 2048, 576, 8, dm.SELECT_TOPK, 8, 0.0, 0),             # row tiles of 128 and of 1
    (2048, 64, 64, 32, dm.SELECT_TOPK, 5, 0.0, 0),              # two chunks a lane
    (2047, 128, 64, 5, dm.SELECT_THRESHOLD, 0, 1.1, 0),
    (1025, 1024, 64, 32, dm.SELECT_THRESHOLD_TOPK, 0, 0.9, 0),
    (1024, 4096, 64, 64, dm.SELECT_TOPK, 2, 0.0, 0),            # routers of every kind zero the counters: this one multiplies in fp32,
    (1024, 512, 64, 48, dm.SELECT_TOPK, 2, 0.0, 0),             # tensor cores, and below
    (160, 256, 64, 9, dm.SELECT_TOPK, 2, 0.0, 0),
    (160, 256, 64, 17, dm.SELECT_THRESHOLD, 0, 1e9, 0),         # nothing selected
]


@pytest.mark.parametrize("T,d,H,E,mode,K,eps,min_k", CASES, ids=["x".join(map(str, c[:4])) + f"-m{c[4]}" for c in CASES])
def test_rows_from_selection_words(T, d, H, E, mode, K, eps, min_k):
    s = gi.LayerSpec(f"fold{T}x{d}x{H}x{E}-{mode}", T=T, d=d, H=H, E=E, dtype="bf16", mode=mode, K=K, eps=eps,
                     eps_normalized=1 if eps else 0, min_k=min_k, router_gain=4.0)
    r = layer_parity(s, sample=40)
    assert r["err_rows"] <= TOL_BF16, (r["err_rows"], r["err"])
    L = r["layer"]
    first = L.forward().clone()
    for _ in range(3):
        assert (L.forward() == first).all()
