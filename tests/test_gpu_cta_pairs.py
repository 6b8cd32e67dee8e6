"""The tensor-core GEMM kernel as CTA pairs (tcgen05 .cta_group::2: two CTAs share one 256-row tile), forced on every
launch whose shapes allow it -- the library itself pairs only where that was measured faster -- and compared with
the oracle on the grouped path with both aggregation modes, the dense forward, ragged column tiles, tiles whose
second half lies past the rows, and the backward pass (GPU required)."""
import os

import pytest
import torch

import dsmoe_inputs as gi
import paper_2404_05567_b200 as dm
from harness import TOL_BF16, layer_parity, np_f32
from test_gpu_training import _backward_case

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def pairs_forced():
    old = os.environ.get("DSMOE_GEMM_PAIR")
    os.environ["DSMOE_GEMM_PAIR"] = "1"
    yield
    if old is None:
        del os.environ["DSMOE_GEMM_PAIR"]
    else:
        os.environ["DSMOE_GEMM_PAIR"] = old


PAIRED = [
    dict(T=2048, d=512, H=256, E=32, mode=gi.MODE_TOPK, K=6, fuse_combine=1),
    dict(T=2048, d=512, H=256, E=32, mode=gi.MODE_TOPK, K=6, fuse_combine=2),
    dict(T=300, d=448, H=320, E=8, mode=gi.MODE_TOPK, K=3, fuse_combine=1),        # ragged column tiles, 1 to 2 row tiles per expert
    dict(T=300, d=448, H=320, E=8, mode=gi.MODE_TOPK, K=3, fuse_combine=2),
    dict(T=1000, d=256, H=128, E=32, mode=gi.MODE_THRESHOLD, eps=0.7, eps_normalized=1, zipf_s=1.1, fuse_combine=1),   # empty and tiny experts
    dict(T=700, d=256, H=64, E=64, mode=gi.MODE_TOPK, K=64, fuse_combine=2),
    dict(T=260, d=320, H=192, E=8, mode=gi.MODE_ALL),                               # dense: 260 rows = one pair tile + 4 rows
    dict(T=1500, d=256, H=448, E=16, mode=gi.MODE_ALL, out_fp32=1),
    dict(T=513, d=128, H=128, E=16, mode=gi.MODE_THRESHOLD_TOPK, eps=0.03),
]


@pytest.mark.parametrize("case", PAIRED, ids=[str(i) for i in range(len(PAIRED))])
def test_layer_with_cta_pairs(case):
    s = gi.LayerSpec(f"pair{PAIRED.index(case)}", dtype="bf16", router_gain=4.0, **case)
    r = layer_parity(s)
    assert r["err_rows"] <= TOL_BF16, (r["err_rows"], r["err"])
    L = r["layer"]
    a = np_f32(L.forward()).copy()
    b = np_f32(L.forward())
    assert (a == b).all()                          # ordered sums: bit-identical from run to run


def test_full_size_prefill_with_cta_pairs():
    r = layer_parity(gi.spec("c3"), sample=256)
    assert r["err_rows"] <= TOL_BF16 and r["err"] <= TOL_BF16, (r["err_rows"], r["err"])


@pytest.mark.parametrize("masked", [False, True], ids=["dense", "masked"])
def test_backward_with_cta_pairs(masked):
    s = gi.LayerSpec("pair_bwd", T=517, d=256, H=448, E=16, dtype="bf16", router_gain=4.0)
    e_s, e_a = _backward_case(s, True, masked)
    assert e_s <= TOL_BF16 and e_a <= TOL_BF16, (e_s, e_a)


@pytest.mark.parametrize("d,E,H", [(1472, 4, 192), (1536, 5, 192), (1536, 4, 256), (256, 16, 448), (256, 16, 512)],
                         ids=lambda v: str(v))
def test_the_librarys_choice_on_both_sides_of_its_lines(d, E, H, monkeypatch):
    """Dense launches: the up-projection and the gradients pair from a reduction of 1536 on, the down-projection from 1024 or 8192.  Single
    CTAs, pairs and the library's choice give the same bits."""
    g = torch.Generator(device="cuda").manual_seed(d)
    T = 300
    randn = lambda *shape, std=1.0: (torch.randn(shape, generator=g, device="cuda") * std).bfloat16()
    x, dO, W1, W2 = randn(T, d), randn(T, d), randn(E, d, H, std=0.02), randn(E, H, d, std=0.02)
    Wr = torch.randn((d, E), generator=g, device="cuda") * 0.02
    desc = dm.make_desc(T, d, H, E, dm.BF16, dm.SELECT_ALL)
    packed = torch.empty(dm.dsmoe_packed_size(desc), dtype=torch.uint8, device="cuda")
    dm.dsmoe_pack_weights(desc, W1, W2, packed)
    ws = torch.empty(dm.dsmoe_workspace_size(desc), dtype=torch.uint8, device="cuda")
    status, scores = torch.zeros(1, dtype=torch.int32, device="cuda"), torch.empty((T, E), device="cuda")
    dm.dsmoe_router(desc, x, Wr, None, scores)

    def run():
        out, dS, dA = torch.empty_like(x), torch.empty((T, E), device="cuda"), torch.empty((T, E * H), dtype=torch.bfloat16, device="cuda")
        dm.dsmoe_layer_forward(desc, x, Wr, None, None, None, packed, out, None, None, ws, status)
        dm.dsmoe_dense_backward(desc, x, None, W2, packed, scores, None, dO, dS, dA, ws, status)
        torch.cuda.synchronize()
        assert int(status.item()) == 0
        return out, dS, dA

    pairs = run()
    for other in ("0", ""):
        monkeypatch.setenv("DSMOE_GEMM_PAIR", other)
        for a, b in zip(pairs, run()):
            assert torch.equal(a, b), other
