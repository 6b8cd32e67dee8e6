"""One to seven tokens (few_tokens_kernel) against the oracle where its work is cut: fewer reduction blocks than warps, experts not a
multiple of four, runs of hidden units that cross an expert's end, more of them than one chunk holds, several passes over a CTA's
columns, fewer columns than CTAs, nothing selected; the same calls with weights that are aligned to 16 bytes only, which small_layer_kernel
takes; and tokens that are not numbers (GPU required)."""
import pytest
import torch

import dsmoe_inputs as gi
import paper_2404_05567_b200 as dm
from harness import TOL_BF16, Layer, layer_parity

pytestmark = pytest.mark.gpu

CASES = [
    dict(T=1, d=64, H=64, E=3, mode=gi.MODE_TOPK, K=1),                                        # one block, 64 columns for 148 CTAs
    dict(T=2, d=320, H=192, E=5, mode=gi.MODE_TOPK, K=2),
    dict(T=3, d=1088, H=448, E=13, mode=gi.MODE_THRESHOLD, eps=1.1, eps_normalized=1),
    dict(T=5, d=2048, H=256, E=32, mode=gi.MODE_THRESHOLD, eps=0.9, eps_normalized=1),
    dict(T=7, d=6144, H=64, E=8, mode=gi.MODE_TOPK, K=3),                                      # three passes over 42 columns
    dict(T=6, d=128, H=1408, E=64, mode=gi.MODE_ALL),                                          # 609 hidden units a CTA, 128 at a time
    dict(T=4, d=512, H=128, E=16, mode=gi.MODE_THRESHOLD, eps=0.999, out_fp32=1),              # nothing selected
    dict(T=7, d=512, H=128, E=16, mode=gi.MODE_THRESHOLD, eps=0.5, min_k=1),
]


@pytest.mark.parametrize("packed_at", [0, 16])
@pytest.mark.parametrize("case", CASES, ids=lambda c: f"T{c['T']}-d{c['d']}-H{c['H']}-E{c['E']}")
def test_a_handful_of_tokens(case, packed_at):
    r = layer_parity(gi.LayerSpec(f"few{CASES.index(case)}", dtype="bf16", router_gain=4.0, **case), packed_at=packed_at)
    assert r["layer"].packed.data_ptr() % 32 == packed_at
    assert r["err_rows"] <= TOL_BF16        # the tolerance of every bf16 layer test
    assert r["zero_tokens"] == (case["T"] if case.get("eps") == 0.999 else 0)


def test_weights_aligned_to_16_bytes_only():
    L = Layer(gi.LayerSpec("few_unaligned", T=3, d=512, H=256, E=8, dtype="bf16", mode=gi.MODE_TOPK, K=2))
    a = L.forward(out_fp32=True)
    buf = torch.empty(L.packed.numel() + 48, dtype=torch.uint8, device="cuda")
    at = (16 - buf.data_ptr()) % 32
    L.packed = buf[at:at + L.packed.numel()]
    assert L.packed.data_ptr() % 32 == 16
    dm.dsmoe_pack_weights(L.desc, L.W1_d, L.W2_d, L.packed)
    b = L.forward(out_fp32=True)                   # another kernel: sums in another order, hidden activations rounded to bf16 (2^-9) alike
    assert (a - b).norm() <= 2e-3 * a.norm()


def test_a_token_that_is_not_a_number():
    """Its scores are no numbers and exceed no threshold: it selects nothing and its row is zeros (Eq. 1 with an empty selection, as
    with more than 128 tokens).  The other tokens do not see it."""
    L = Layer(gi.LayerSpec("few_nan", T=5, d=512, H=256, E=8, dtype="bf16", mode=gi.MODE_THRESHOLD, eps=0.5, eps_normalized=1))
    plain = L.forward(out_fp32=True).clone()
    L.x_d = L.x_d.clone()
    L.x_d[2] = float("nan")
    out = L.forward(out_fp32=True)
    others = [0, 1, 3, 4]
    assert int(L.mask[2]) == 0 and not out[2].any()
    # (fewer experts may be selected: the sums over them then run in another order)
    assert (out[others] - plain[others]).norm() <= 1e-5 * plain[others].norm()
