"""The decode kernel's router by groups of tokens against the oracle where the groups change: the first and last token counts of groups of
2 and of 4, a last group that is not full, expert counts whose rows of the router's weights do and do not fill a warp (GPU required)."""
import pytest
import torch

import dsmoe_inputs as gi
from harness import TOL_BF16, Layer, layer_parity

pytestmark = pytest.mark.gpu

CASES = [(37, 2112, 32), (38, 2112, 32), (39, 256, 64), (73, 192, 5), (74, 2112, 48), (75, 2112, 33), (77, 3072, 8), (128, 2112, 64)]


@pytest.mark.parametrize("T,d,E", CASES, ids=[f"T{T}-d{d}-E{E}" for T, d, E in CASES])
def test_router_by_groups(T, d, E):
    r = layer_parity(gi.LayerSpec(f"groups{T}x{d}x{E}", T=T, d=d, H=128, E=E, dtype="bf16", mode=gi.MODE_TOPK, K=3, router_gain=4.0))
    assert r["err_rows"] <= TOL_BF16, (r["err_rows"], r["err"])
    L = r["layer"]
    first = L.forward().clone()
    for _ in range(3):                                     # the counters are zeroed by every call, the slices' order is fixed
        assert (L.forward() == first).all()


@pytest.mark.parametrize("T,d", [(38, 64), (65, 256), (74, 256)])
def test_counters_stay_in_their_place(T, d):
    """The counters of the groups, zeroed by every call, are followed in the workspace by what belongs to another entry point."""
    L = Layer(gi.LayerSpec(f"place{T}", T=T, d=d, H=128, E=8, dtype="bf16", mode=gi.MODE_TOPK, K=3, router_gain=4.0))
    up = lambda n: (n + 255) // 256 * 256
    # scores, mask, k_t, counts, offsets, chunk counts, the batch's K, barriers; then 64 counters a column range of 256
    at = up(T * 8 * 4) + up(T * 8) + up(T * 4) + up(64 * 4) + up(65 * 4) + up((T + 31) // 32 * 8 * 4) + 256 + 256
    L.ws.fill_(0x5a)
    L.forward()
    counters = L.ws[at:at + 256].view(torch.int32)
    assert (counters[:(T + 1) // 2] != 0x5a5a5a5a).all()       # they are there
    assert (L.ws[at + 256:at + 512] == 0x5a).all()


# many wide experts are grouped by expert beyond 80 (d up to 1536) and 96 tokens: both sides of each line
WIDE = [(80, 1536, 1024, 32), (81, 1536, 1024, 32), (96, 2048, 512, 64), (97, 2048, 512, 64), (128, 64, 2048, 33)]


@pytest.mark.parametrize("mode", [gi.MODE_TOPK, gi.MODE_THRESHOLD], ids=["topk", "threshold"])
@pytest.mark.parametrize("T,d,H,E", WIDE, ids=[f"T{T}-d{d}-H{H}-E{E}" for T, d, H, E in WIDE])
def test_many_wide_experts(T, d, H, E, mode):
    sel = dict(K=3) if mode == gi.MODE_TOPK else dict(eps=1.0, eps_normalized=1)
    r = layer_parity(gi.LayerSpec(f"wide{T}x{d}x{H}x{E}-{mode}", T=T, d=d, H=H, E=E, dtype="bf16", mode=mode, router_gain=4.0, **sel), sample=24)
    assert r["err_rows"] <= TOL_BF16, (r["err_rows"], r["err"])
    L = r["layer"]
    first = L.forward().clone()
    assert (L.forward() == first).all()
