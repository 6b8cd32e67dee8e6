"""The router whose clusters take 32 tokens (csrc/router_cluster.cu): the first and last token counts it takes, a last group of one token,
every padding of the experts, reductions that do not divide among its warps; its error against 64 bits beside the FMA kernel's (GPU
required)."""
import pytest
import torch

import dsmoe_inputs as gi
import test_gpu_grouped_layer
import paper_2404_05567_b200 as dm
from harness import TOL_BF16, Layer, desc_of, layer_parity, to_dev

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


@pytest.mark.parametrize("shape", [(129, 2048, 8), (256, 6144, 16), (768, 2112, 32), (384, 6144, 64)], ids=lambda s: "x".join(map(str, s)))
def test_no_farther_from_64_bits_than_the_fma_kernel(shape):
    T, d, E = shape
    s = gi.LayerSpec(f"cluster64_{T}x{d}x{E}", T=T, d=d, H=64, E=E, dtype="bf16", mode=gi.MODE_TOPK, K=min(3, E), router_gain=4.0)
    L = Layer(s)
    L.forward()
    torch.cuda.synchronize()
    x, (Wr, br) = gi.tokens(s), gi.router(s)
    exact = torch.softmax(to_dev(x).double() @ to_dev(Wr).double() + (to_dev(br).double() if br is not None else 0), dim=1)
    fma = torch.empty(T, E, dtype=torch.float32, device="cuda")
    # a hidden width that the tensor-core paths do not take leaves the scores to the FMA kernel
    dm.dsmoe_router(desc_of(s.replace(H=72)), to_dev(x), to_dev(Wr), to_dev(br), fma)
    got = L.ws[:4 * T * E].view(torch.float32).view(T, E)        # the workspace begins with the layer's scores
    err = [float((v.double() - exact).norm() / exact.norm()) for v in (got, fma)]
    assert err[0] <= 1.05 * err[1], err


PART = [(200, 2048, 64, 16, 3), (700, 1024, 64, 32, 4), (384, 1024, 64, 64, 2), (1000, 1024, 128, 8, 2)]


@pytest.mark.parametrize("sms", [16, 72])
def test_on_a_part_of_the_gpu(sms, monkeypatch):
    """Clusters of eight on a stream that owns some of the SMs."""
    monkeypatch.setattr(test_gpu_grouped_layer, "PART", PART)
    test_gpu_grouped_layer.test_on_a_part_of_the_gpu(sms)


@pytest.mark.parametrize("shape", PART, ids=lambda s: f"T{s[0]}-d{s[1]}-H{s[2]}-E{s[3]}")
def test_two_streams_with_a_workspace_each(shape):
    test_gpu_grouped_layer.test_two_streams_with_a_workspace_each(shape)
