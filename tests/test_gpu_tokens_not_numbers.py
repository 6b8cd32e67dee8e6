"""Tokens whose scores are not numbers under a top-K selection: every expert selects them (a score that is no number is beaten by none), more than
the K rows that a token has.  They get NaN, or an error is reported; nothing is written past the workspace, and the other tokens' outputs
are those of a call without them (GPU required)."""
import math

import pytest
import torch

import dsmoe_inputs as gi
import paper_2404_05567_b200 as dm
from harness import Layer, to_dev
from test_gpu_moa import _moa_case

pytestmark = pytest.mark.gpu


def _bad_tokens(x, tokens):
    y = x.clone()
    y[tokens, 3] = float("nan")
    return y


def _others(T, tokens):
    return [t for t in range(T) if t not in tokens]


def _guarded(nbytes):
    return torch.full((nbytes + 65536,), 0x5a, dtype=torch.uint8, device="cuda")


@pytest.mark.parametrize("T,d,H,E,K", [(40, 72, 64, 8, 2), (30, 504, 1016, 32, 1), (64, 256, 512, 8, 3)], ids=lambda v: str(v))
def test_fp32_layer(T, d, H, E, K):
    L = Layer(gi.LayerSpec(f"nan32_{T}", T=T, d=d, H=H, E=E, dtype="f32", mode=gi.MODE_TOPK, K=K, router_gain=4.0))
    clean, nbytes = L.forward().clone(), L.ws.numel()
    bad, buf = [0, 17, T - 1], _guarded(nbytes)
    L.ws, L.x_d = buf[:nbytes], _bad_tokens(L.x_d, [0, 17, T - 1])
    out = L.forward()
    assert (buf[nbytes:] == 0x5a).all()
    assert torch.equal(out[_others(T, bad)], clean[_others(T, bad)]) and out[bad].isnan().all()
    assert all(int(L.mask[t]) == 2 ** E - 1 for t in bad)
    assert L.counts[:E].tolist() == [int(((L.mask >> e) & 1).sum()) for e in range(E)]


@pytest.mark.parametrize("ragged", [False, True], ids=["alike", "ragged"])
@pytest.mark.parametrize("T,E,K,dh", [(8, 8, 3, 128), (20, 16, 1, 64), (33, 16, 6, 96)], ids=lambda v: str(v))
def test_decoding_attention(T, E, K, dh, ragged):
    """Few enough pairs of tokens and heads that several CTAs share each one's keys and leave parts of K rows."""
    d, nh, L = 1024, 2, 400
    s, x, Wr, br, Wq, Wo, Kc, Vc, seq, pos = _moa_case(f"nanmoa{T}", T, d, E, nh, dh, T, L, "decode", gi.MODE_TOPK, K=K)
    if not ragged:
        pos[:] = L - 1
    desc = dm.make_desc(T, d, nh * dh, E, dm.BF16, dm.SELECT_TOPK, K=K, out_fp32=1)
    packed = torch.empty(dm.dsmoe_packed_size(desc), dtype=torch.uint8, device="cuda")
    dm.dsmoe_pack_weights(desc, to_dev(Wq), to_dev(Wo), packed)
    nbytes, status = dm.dsmoe_workspace_size_packed(desc), torch.zeros(1, dtype=torch.int32, device="cuda")
    args = [to_dev(a) for a in (Kc, Vc, seq, pos)]
    Wr_d, br_d, x_d = to_dev(Wr), to_dev(br), to_dev(x)

    def run(x_d):
        buf, out = _guarded(nbytes), torch.empty((T, d), device="cuda")
        dm.dsmoe_moa_forward(desc, nh, 1 / math.sqrt(dh), *args, x_d, Wr_d, br_d, packed, out, None, None, buf[:nbytes], status)
        torch.cuda.synchronize()
        assert (buf[nbytes:] == 0x5a).all()
        return out

    bad = [2, T - 1]
    clean, out = run(x_d), run(_bad_tokens(x_d, bad))
    assert int(status.item()) == 0
    assert torch.equal(out[_others(T, bad)], clean[_others(T, bad)]) and out[bad].isnan().all()


@pytest.mark.parametrize("T,E,K", [(200, 8, 2), (300, 33, 3), (1500, 16, 1)], ids=lambda v: str(v))
def test_rows_from_selection_words(T, E, K):
    """Grouped by expert there are then more rows than T * K: the experts whose segments end beyond are reported and count as empty."""
    L = Layer(gi.LayerSpec(f"nanfold{T}", T=T, d=128, H=64, E=E, dtype="bf16", mode=gi.MODE_TOPK, K=K, router_gain=4.0))
    clean, mask, nbytes, x = L.forward().clone(), L.mask.clone(), L.ws.numel(), L.x_d
    t = T // 2
    buf = _guarded(nbytes)
    L.ws, L.x_d = buf[:nbytes], _bad_tokens(x, [t])
    with pytest.raises(AssertionError, match="device status 1"):
        L.forward()
    assert (buf[nbytes:] == 0x5a).all() and int(L.mask[t]) == 2 ** E - 1
    ends = L.counts[:E].cumsum(0)
    lost = sum(1 << e for e in range(E) if int(ends[e]) > T * K)
    kept = [i for i in _others(T, [t]) if int(mask[i]) & lost == 0]
    assert len(kept) > T // 2
    assert torch.equal(L.out[kept], clean[kept])
    L.dev_status.zero_()
    L.x_d = x
    assert torch.equal(L.forward(), clean)
