"""Tokens whose scores are not numbers under a top-K selection: every expert selects them (a score that is no number is beaten by none), more than
the K rows that a token has.  They get NaN, or an error is reported; nothing is written past the workspace, and the other tokens' outputs
are those of a call without them (GPU required)."""
import pytest
import torch

import dsmoe_inputs as gi
from harness import Layer

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
