"""The tensor-core router (bf16, more than 256 tokens): scores against the oracle over its cluster sizes (4, 2 and 1 CTAs per row
tile), ring and accumulator lengths (1 to 64 blocks of 64), expert counts on both sides of 32 and tokens with a mean; its
error against 64 bits beside the FMA kernel's; and what is left behind when a wait runs out (GPU required)."""
import numpy as np
import pytest
import torch

import dsmoe_inputs as gi
import oracle
import paper_2404_05567_b200 as dm
from harness import TOL_BF16, Layer, desc_of, layer_parity, to_dev
from paper_2404_05567_b200 import binding, build as dm_build

pytestmark = pytest.mark.gpu


def _spec(T, d, E, H=64, **kw):
    return gi.LayerSpec(f"router{T}x{d}x{E}", T=T, d=d, H=H, E=E, dtype="bf16", router_gain=4.0, **kw)


def _scores(s, x, Wr, br):
    out = torch.full((s.T, s.E), -1.0, dtype=torch.float32, device="cuda")
    dm.dsmoe_router(desc_of(s), to_dev(x), to_dev(Wr), to_dev(br), out)
    return out


# T, d, E: 1, 3 and 11 blocks (one CTA per row tile), 8 to 64 (4 CTAs; 2 from 38 row tiles on, 1 from 75 on); E on both sides of
# 32, and the FMA kernel where 64 experts' two accumulators would run over too many blocks (4096 wide)
SHAPES = [(257, 64, 1), (300, 192, 8), (257, 704, 33), (300, 704, 32), (300, 512, 48), (257, 2048, 64), (300, 4096, 32),
          (300, 4096, 64), (8190, 2048, 32), (8190, 2048, 48), (4900, 4096, 8), (9601, 512, 32), (9601, 704, 64), (9601, 2048, 8)]


@pytest.mark.parametrize("mean", [0.0, 0.75], ids=["centred", "mean"])
@pytest.mark.parametrize("shape", SHAPES, ids=["x".join(map(str, s)) for s in SHAPES])
def test_scores(shape, mean):
    s = _spec(*shape)
    x, (Wr, br) = gi.tokens(s), gi.router(s)
    if mean:
        x = (to_dev(x).float() + mean).bfloat16().view(torch.int16).cpu().numpy().view(np.uint16)
    got, ref = _scores(s, x, Wr, br).cpu().numpy(), oracle.router_scores(x, Wr, br)
    assert np.all(np.abs(got - ref) <= 1e-6 + 1e-5 * ref)


@pytest.mark.parametrize("sel", [dict(mode=gi.MODE_TOPK, K=3), dict(mode=gi.MODE_THRESHOLD, eps=0.05), dict(mode=gi.MODE_ALL)],
                         ids=["topk", "threshold", "all"])
@pytest.mark.parametrize("shape", [(257, 704, 33), (300, 4096, 32), (9601, 512, 32)], ids=lambda s: "x".join(map(str, s)))
def test_selection_and_counts_of_a_layer(shape, sel):
    assert layer_parity(_spec(*shape, **sel), sample=24)["err_rows"] <= TOL_BF16


@pytest.mark.parametrize("shape", [(300, 2048, 8), (8190, 2048, 64), (8190, 4096, 32), (16384, 6144, 16)],
                         ids=lambda s: "x".join(map(str, s)))
def test_no_farther_from_64_bits_than_the_fma_kernel(shape):
    s = _spec(*shape)
    x, (Wr, br) = gi.tokens(s), gi.router(s)
    exact = torch.softmax(to_dev(x).double() @ to_dev(Wr).double() + (to_dev(br).double() if br is not None else 0), dim=1)
    # a hidden width that the tensor-core paths do not take leaves the scores to the FMA kernel
    err = [float((_scores(t, x, Wr, br).double() - exact).norm() / exact.norm()) for t in (s, s.replace(H=72))]
    assert err[0] <= 1.05 * err[1], err


def test_a_wait_that_runs_out_is_seen(monkeypatch):
    """One rank of every cluster reports an expired wait (a build of the kernel for this test; nothing hangs, every wait still
    ends): the tokens' scores are NaN for all its ranks, a layer call selects nothing for them, writes zeros and reports it."""
    lib = dm_build.build_variant("give_up", "router_umma.cu", ["-DDSMOE_TEST_GIVE_UP_RANK=1"])
    s = _spec(300, 512, 16, mode=gi.MODE_TOPK, K=3)                              # clusters of four
    L = Layer(s)
    plain = _scores(s, L.x, L.Wr, L.br)
    assert bool(torch.isfinite(plain).all())
    alone = _spec(300, 192, 16)                                                  # one CTA per row tile: there is no rank 1
    x1, (Wr1, br1) = gi.tokens(alone), gi.router(alone)
    want1 = _scores(alone, x1, Wr1, br1)
    monkeypatch.setattr(binding, "LIB_PATH", lib)
    monkeypatch.setattr(binding, "_lib", None)
    assert bool(torch.isnan(_scores(s, L.x, L.Wr, L.br)).all())
    assert torch.equal(_scores(alone, x1, Wr1, br1), want1)
    L.out.fill_(7.0)
    L.mask.fill_(-1)
    dm.dsmoe_layer_forward(L.desc, L.x_d, L.Wr_d, L.br_d, None, None, L.packed, L.out, L.mask, L.counts, L.ws, L.dev_status)
    torch.cuda.synchronize()
    assert int(L.dev_status.item()) == 5                                         # DSMOE_ERR_TIMEOUT
    assert not L.mask.any() and not L.counts[:s.E].any() and not L.out.any()
