"""The router whose clusters take 32 tokens (csrc/router_cluster.cu): the first and last token counts it takes, a last group of one token,
every padding of the experts, reductions that do not divide among its warps; its error against 64 bits, no larger than the FMA kernel's
(GPU required)."""
import numpy as np
import pytest
import torch

import dsmoe_inputs as gi
import test_gpu_grouped_layer
import paper_2404_05567_b200 as dm
from harness import TOL_BF16, layer_parity

pytestmark = pytest.mark.gpu

SHAPES = [(129, 256, 17), (161, 320, 64), (160, 2112, 33), (256, 2048, 5), (130, 6144, 1), (257, 1024, 32), (384, 1088, 48), (385, 1024, 31),
          (768, 1088, 20), (1024, 2048, 16), (993, 1088, 7)]


@pytest.mark.parametrize("sel", [dict(mode=gi.MODE_TOPK, K=3), dict(mode=gi.MODE_THRESHOLD, eps=0.05)], ids=["topk", "threshold"])
@pytest.mark.parametrize("shape", SHAPES, ids=["x".join(map(str, s)) for s in SHAPES])
def test_layer(shape, sel):
    T, d, E = shape
    sel = {**sel, "K": min(3, E)} if "K" in sel else sel
    s = gi.LayerSpec(f"cluster{T}x{d}x{E}", T=T, d=d, H=64, E=E, dtype="bf16", router_gain=4.0, **sel)
    r = layer_parity(s, sample=24)
    assert r["err_rows"] <= TOL_BF16, (r["err_rows"], r["err"])
    L = r["layer"]
    first = L.forward().clone()
    assert (L.forward() == first).all()


# up to 128 tokens most layers route for themselves: Threshold-TopK, whose K comes from the batch, does not
FIRST = [(65, 2048, 16), (65, 256, 17), (97, 320, 64), (97, 2112, 5), (128, 1088, 33)]


@pytest.mark.parametrize("shape", FIRST, ids=["x".join(map(str, s)) for s in FIRST])
def test_first_token_counts(shape):
    T, d, E = shape
    s = gi.LayerSpec(f"cluster{T}x{d}x{E}", T=T, d=d, H=64, E=E, dtype="bf16", router_gain=4.0, mode=gi.MODE_THRESHOLD_TOPK, eps=0.9, eps_normalized=1)
    r = layer_parity(s, sample=24)
    assert r["err_rows"] <= TOL_BF16, (r["err_rows"], r["err"])


SCORED = [(65, 2048, 16), (128, 256, 64), (129, 2048, 8), (256, 6144, 16), (256, 1024, 33), (768, 2112, 32), (384, 6144, 64)]
DRAWS = 12


def _errors(T, d, E):
    """How far the layer's scores and the FMA kernel's are from 64 bits, for each draw of tokens and weights; logits of four spreads."""
    desc = dm.make_desc(T, d, 64, E, dm.BF16, dm.SELECT_THRESHOLD_TOPK, 0.9, 1)
    # a hidden width that the tensor-core paths do not take leaves the scores to the FMA kernel
    plain = dm.make_desc(T, d, 72, E, dm.BF16, dm.SELECT_THRESHOLD_TOPK, 0.9, 1)
    packed = torch.zeros(dm.dsmoe_packed_size(desc), dtype=torch.uint8, device="cuda")
    ws = torch.empty(dm.dsmoe_workspace_size_packed(desc), dtype=torch.uint8, device="cuda")
    out, fma = torch.empty((T, d), dtype=torch.bfloat16, device="cuda"), torch.empty((T, E), device="cuda")
    errors = []
    for seed in range(DRAWS):
        g = torch.Generator(device="cuda").manual_seed(seed)
        x = torch.randn((T, d), generator=g, device="cuda").bfloat16()
        Wr = torch.randn((d, E), generator=g, device="cuda") * ((0.905, 1.56, 4.0, 0.3)[seed % 4] / d ** 0.5)
        exact = torch.softmax(x.double() @ Wr.double(), dim=1)
        dm.dsmoe_layer_forward(desc, x, Wr, None, None, None, packed, out, None, None, ws, None)
        dm.dsmoe_router(plain, x, Wr, None, fma)
        got = ws[:4 * T * E].view(torch.float32).view(T, E)      # the workspace begins with the layer's scores
        errors.append([float((v.double() - exact).norm() / exact.norm()) for v in (got, fma)])
    return np.array(errors)


def test_no_farther_from_64_bits_than_the_fma_kernel():
    """On average over all shapes, and at each shape as far as its draws can tell: the errors are rounding by chance, a single draw's two
    differ by up to 1.2 times, so the mean of log(error / error) may lie above zero by three times its own standard deviation."""
    means = []
    for shape in SCORED:
        ratio = np.log(np.divide(*_errors(*shape).T))
        means.append(ratio.mean())
        assert means[-1] <= 3 * ratio.std(ddof=1) / DRAWS ** 0.5, (shape, ratio)
    assert np.mean(means) < 0, means


PART = [(200, 2048, 64, 16, 3), (700, 1024, 64, 32, 4), (384, 1024, 64, 64, 2), (1000, 1024, 128, 8, 2)]


@pytest.mark.parametrize("sms", [16, 72])
def test_on_a_part_of_the_gpu(sms, monkeypatch):
    """Clusters of eight on a stream that owns some of the SMs."""
    monkeypatch.setattr(test_gpu_grouped_layer, "PART", PART)
    test_gpu_grouped_layer.test_on_a_part_of_the_gpu(sms)


@pytest.mark.parametrize("shape", PART, ids=lambda s: f"T{s[0]}-d{s[1]}-H{s[2]}-E{s[3]}")
def test_two_streams_with_a_workspace_each(shape):
    test_gpu_grouped_layer.test_two_streams_with_a_workspace_each(shape)
