"""Parity of the mixture-of-attention-heads layer (Eq. 7-8) with the CPU oracle (GPU required): the GPU decides the
selection on its own scores (checked against the oracle's as for the feed-forward layer), the oracle evaluates Eq. 8
on the GPU's selection.  Shapes follow Table `tab:model_arch` (n_head x d_head = 2 x 64, 4 x 96, 4 x 128 per expert, 8
or 16 experts), with prefill-like batches of several sequences and decode-like batches of one token per sequence."""
import math

import numpy as np
import pytest
import torch

import dsmoe_inputs as gi
import oracle
import paper_2404_05567_b200 as dm
from harness import TOL_BF16, check_mask_against_oracle, desc_of, record, rel_err, rel_err_rows, to_dev, to_np

pytestmark = pytest.mark.gpu


def _moa_case(name, T, d, E, n_head, dh, n_seq, L, layout, mode, **sel):
    """layout 'prefill': the T tokens are n_seq sequences of T / n_seq tokens at positions 0, 1, ...; 'decode': one
    new token per sequence (T == n_seq) at seeded positions; 'mixed': seeded sequences and positions; 'full': seeded
    sequences, every token at the cache's last position."""
    H = n_head * dh
    s = gi.LayerSpec(name, T=T, d=d, H=H, E=E, dtype="bf16", mode=mode, router_gain=4.0, **sel)
    x = gi.tokens(s)
    Wr, br = gi.router(s)
    Wq, Wo = gi.experts(s)                                   # [E, d, H], [E, H, d]: same shapes as the expert MLPs' weights
    Kc = gi.normal(s.seed, f"{name}.K", (n_seq, n_head, L, dh), 1.0, "bf16")
    Vc = gi.normal(s.seed, f"{name}.V", (n_seq, n_head, L, dh), 1.0, "bf16")
    u = gi.uniform(s.seed, f"{name}.pos", T)
    if layout == "prefill":
        per = T // n_seq
        seq = (np.arange(T) // per).astype(np.int32)
        pos = (np.arange(T) % per).astype(np.int32)
    elif layout == "decode":
        seq = np.arange(T, dtype=np.int32)
        pos = np.minimum((u * L).astype(np.int32), L - 1)
        pos[0], pos[-1] = L - 1, 0
    else:
        seq = np.minimum((gi.uniform(s.seed, f"{name}.seq", T) * n_seq).astype(np.int32), n_seq - 1)
        pos = np.minimum((u * L).astype(np.int32), L - 1)
        if layout == "full":                                 # every token sees the whole cache
            pos[:] = L - 1
    return s, x, Wr, br, Wq, Wo, Kc, Vc, seq, pos


def _run(s, x, Wr, br, Wq, Wo, Kc, Vc, seq, pos, n_head, scale, sample=None, use_seq=True):
    desc = desc_of(s.replace(out_fp32=1))
    x_d, Wr_d, br_d = to_dev(x), to_dev(Wr), to_dev(br)
    packed = torch.empty(dm.dsmoe_packed_size(desc), dtype=torch.uint8, device="cuda")
    dm.dsmoe_pack_weights(desc, to_dev(Wq), to_dev(Wo), packed)
    ws = torch.empty(dm.dsmoe_workspace_size_packed(desc), dtype=torch.uint8, device="cuda")
    out = torch.empty((s.T, s.d), dtype=torch.float32, device="cuda")
    mask = torch.zeros(s.T, dtype=torch.int64, device="cuda")
    counts = torch.zeros(64, dtype=torch.int32, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    K_d, V_d, seq_d, pos_d = to_dev(Kc), to_dev(Vc), to_dev(seq) if use_seq else None, to_dev(pos)
    dm.dsmoe_moa_forward(desc, n_head, scale, K_d, V_d, seq_d, pos_d, x_d, Wr_d, br_d, packed, out, mask, counts, ws, status)
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    first = out.cpu().numpy().copy()
    dm.dsmoe_moa_forward(desc, n_head, scale, K_d, V_d, seq_d, pos_d, x_d, Wr_d, br_d, packed, out, mask, counts, ws, status)
    torch.cuda.synchronize()
    got = out.cpu().numpy()
    assert np.array_equal(first, got)                        # bit-identical from run to run
    mask_gpu = to_np(mask).view(np.uint64)
    S = oracle.router_scores(x, Wr, br)
    mask_ref, _ = oracle.select(S, s.mode, s.eps, s.eps_normalized, s.K, s.min_k)
    flips, near = check_mask_against_oracle(s, S, mask_gpu, mask_ref)
    ids = None if sample is None or sample >= s.T else gi.sample_tokens(s, sample)
    ref = oracle.moa_layer(x, Wq, Wo, Kc, Vc, S, mask_gpu, pos, n_head, scale, tok_seq=seq if use_seq else None, token_ids=ids)
    g = got if ids is None else got[ids]
    e, er = rel_err(g, ref), rel_err_rows(g, ref)
    record("moa_parity", name=s.name, T=s.T, d=s.d, E=s.E, n_head=n_head, d_head=s.H // n_head, L=int(Kc.shape[2]),
           n_seq=int(Kc.shape[0]), mode=s.mode, tokens_compared=int(ref.shape[0]), err_global=e, err_per_token=er,
           flips=flips, near_threshold=near, A=int(to_np(counts)[:s.E].sum()))
    return e, er


MOA = [
    # name, T, d, E, n_head, d_head, n_seq, L, layout, mode, selection
    ("moa_1b_prefill", 512, 2048, 16, 2, 64, 4, 128, "prefill", gi.MODE_TOPK, dict(K=6)),
    ("moa_3b_prefill", 384, 3072, 8, 4, 96, 3, 128, "prefill", gi.MODE_TOPK, dict(K=5)),
    ("moa_6b_prefill", 512, 4096, 8, 4, 128, 2, 256, "prefill", gi.MODE_THRESHOLD, dict(eps=0.08)),
    ("moa_6b_decode", 32, 4096, 8, 4, 128, 32, 700, "decode", gi.MODE_THRESHOLD, dict(eps=0.08)),
    ("moa_1b_decode", 5, 2048, 16, 2, 64, 5, 333, "decode", gi.MODE_TOPK, dict(K=3)),
    ("moa_all", 300, 256, 8, 2, 32, 7, 61, "mixed", gi.MODE_ALL, dict()),                       # the dense form the paper runs at inference
    ("moa_one_token", 1, 512, 4, 2, 64, 1, 1, "decode", gi.MODE_ALL, dict()),                   # a single key
    ("moa_empty_rows", 260, 256, 16, 2, 64, 3, 50, "mixed", gi.MODE_THRESHOLD, dict(eps=0.3)),  # tokens that select nothing
    ("moa_wide_head", 200, 512, 4, 1, 256, 2, 90, "mixed", gi.MODE_TOPK, dict(K=2)),
    ("moa_ttk", 513, 256, 8, 4, 32, 4, 140, "mixed", gi.MODE_THRESHOLD_TOPK, dict(eps=0.03)),
    ("moa_many_experts", 70, 256, 40, 2, 64, 2, 50, "mixed", gi.MODE_ALL, dict()),               # 40 rows per token: three row tiles
    ("moa_many_experts_topk", 600, 256, 24, 2, 64, 3, 90, "mixed", gi.MODE_TOPK, dict(K=20)),      # 20 rows per token: two row tiles
    ("moa_full_cache", 300, 1024, 8, 4, 64, 6, 200, "full", gi.MODE_TOPK, dict(K=4)),
    ("moa_full_cache_6b", 64, 4096, 8, 4, 128, 8, 1000, "full", gi.MODE_TOPK, dict(K=5)),
]


@pytest.mark.parametrize("case", MOA, ids=[c[0] for c in MOA])
def test_moa_layer(case):
    name, T, d, E, nh, dh, n_seq, L, layout, mode, sel = case
    s, *rest = _moa_case(name, T, d, E, nh, dh, n_seq, L, layout, mode, **sel)
    e, er = _run(s, *rest, nh, 1.0 / math.sqrt(dh))
    assert er <= TOL_BF16, (e, er)
    # The whole-output form of the bar is asserted where the rows are of one scale.  A token at cache position p
    # averages p + 1 value vectors, so its row is about sqrt((L + 1) / (p + 1)) times larger than that of a token that
    # sees the whole cache: with positions spread over the cache the early tokens' rounding alone exceeds a bar
    # relative to the whole output's RMS (measured: 2.1e-2 to 2.7e-2 there, against 0.8e-2 to 1.3e-2 per token).
    if layout == "full":
        assert e <= TOL_BF16, (e, er)


def test_moa_without_sequence_list_and_with_scale_one():
    s, x, Wr, br, Wq, Wo, Kc, Vc, seq, pos = _moa_case("moa_one_seq", 130, 256, 8, 2, 64, 1, 130, "prefill", gi.MODE_TOPK, K=3)
    e, er = _run(s, x, Wr, br, Wq, Wo, Kc, Vc, seq, pos, 2, 1.0, use_seq=False)
    assert er <= TOL_BF16, (e, er)


def test_moa_fused_and_separate_aggregation():
    for fuse in (1, 2):
        s, *rest = _moa_case(f"moa_fuse{fuse}", 700, 512, 8, 4, 64, 5, 140, "prefill", gi.MODE_TOPK, K=4, fuse_combine=fuse)
        e, er = _run(s, *rest, 4, 0.125)
        assert er <= TOL_BF16, (fuse, e, er)


def test_moa_paper_6b_shape_on_sampled_tokens():
    """DS-MoE-6B's attention layer (8 experts of 4 heads of 128, model width 4096) on 32 sequences of 256 tokens,
    the sequence length of the paper's input-throughput setting; the oracle evaluates 256 seeded tokens."""
    s, *rest = _moa_case("moa_6b_full", 8192, 4096, 8, 4, 128, 32, 256, "prefill", gi.MODE_TOPK, K=5)
    e, er = _run(s, *rest, 4, 1.0 / math.sqrt(128), sample=256)
    assert er <= TOL_BF16, (e, er)


def test_moa_rejects_what_it_does_not_support():
    desc = dm.make_desc(64, 256, 96, 4, dm.BF16, dm.SELECT_ALL)            # H = 96 is not a multiple of 64
    z = torch.zeros(16, dtype=torch.uint8, device="cuda")
    K = torch.zeros((1, 2, 8, 48), dtype=torch.bfloat16, device="cuda")
    with pytest.raises(dm.DsmoeError) as ei:
        dm.dsmoe_moa_forward(desc, 2, 1.0, K, K, None, z, z, z, None, z, z, None, None, z)
    assert ei.value.code in (1, 2)


def test_moa_plain_attention_kernel_on_a_common_head_width(monkeypatch):
    """Head widths 64, 96 and 128 normally take the tensor-core attention kernel; the plain one (other widths) is run on
    such a shape too, through the library's switch for it."""
    monkeypatch.setenv("DSMOE_MOA_PLAIN", "1")
    s, *rest = _moa_case("moa_plain", 200, 512, 8, 2, 64, 3, 77, "mixed", gi.MODE_TOPK, K=3)
    e, er = _run(s, *rest, 2, 0.125)
    assert er <= TOL_BF16, (e, er)


# Many tokens per sequence: tiles that share their copies of the keys, grouped output projection (few row tiles) and the dense
# one (row tiles enough to cover the SMs: 148 of 128 rows x 256 columns).  Ragged token counts, CTAs whose tokens belong to
# several sequences, caches around the 64-key blocks, more than 16 rows per token, every head width.
PROMPTS = [
    ("prompt_grouped", 77, 512, 8, 2, 64, 3, 65, "mixed", gi.MODE_TOPK, dict(K=3)),
    ("prompt_grouped_thr", 203, 512, 8, 2, 96, 7, 640, "mixed", gi.MODE_THRESHOLD, dict(eps=0.2)),       # some tokens select nothing
    ("prompt_one_row", 130, 256, 4, 2, 128, 2, 129, "prefill", gi.MODE_TOPK, dict(K=1)),                 # 16 tokens a tile
    ("prompt_two_row_tiles", 90, 256, 20, 2, 64, 4, 64, "mixed", gi.MODE_ALL, dict()),
    ("prompt_dense", 4701, 1024, 8, 2, 64, 3, 300, "mixed", gi.MODE_TOPK, dict(K=4)),
    ("prompt_dense_96", 4640, 1024, 8, 4, 96, 16, 290, "prefill", gi.MODE_TOPK, dict(K=5)),
    ("prompt_dense_128", 2369, 2048, 8, 1, 128, 1, 2400, "prefill", gi.MODE_TOPK, dict(K=7)),
    ("prompt_dense_all", 4609, 1024, 20, 2, 64, 11, 63, "mixed", gi.MODE_ALL, dict()),
]


@pytest.mark.parametrize("case", PROMPTS, ids=[c[0] for c in PROMPTS])
def test_moa_prompts(case):
    name, T, d, E, nh, dh, n_seq, L, layout, mode, sel = case
    s, *rest = _moa_case(name, T, d, E, nh, dh, n_seq, L, layout, mode, **sel)
    e, er = _run(s, *rest, nh, 1.0 / math.sqrt(dh), sample=200)
    assert er <= TOL_BF16, (e, er)


# One case per attention kernel: tiles that share their keys, decoding tokens (long and short caches), the plain kernel; of more tokens than
# the decoding one takes, the key-splitting and the tile-per-warp form; tiles of 128 rows with the key-splitting kernel behind them
CLAMPED = [("clamp_prompt", 40, 64, 3, 65), ("clamp_split", 12, 64, 4, 600), ("clamp_tiles", 12, 64, 4, 90), ("clamp_plain", 20, 32, 3, 33),
           ("clamp_split_80", 80, 64, 12, 600), ("clamp_tiles_80", 80, 64, 12, 90), ("clamp_tile_of_128", 3000, 64, 2, 600)]


@pytest.mark.parametrize("case", CLAMPED, ids=[c[0] for c in CLAMPED])
def test_moa_clamps_and_reports_entries_out_of_range_with_or_without_a_status_word(case):
    """tok_seq and pos entries beyond the cache count as the nearest one inside; dev_status is optional."""
    name, T, dh, n_seq, L = case
    s, x, Wr, br, Wq, Wo, Kc, Vc, seq, pos = _moa_case(name, T, 256, 8, 2, dh, n_seq, L, "mixed", gi.MODE_TOPK, K=3)
    desc = desc_of(s)
    packed = torch.empty(dm.dsmoe_packed_size(desc), dtype=torch.uint8, device="cuda")
    dm.dsmoe_pack_weights(desc, to_dev(Wq), to_dev(Wo), packed)
    ws = torch.empty(dm.dsmoe_workspace_size_packed(desc), dtype=torch.uint8, device="cuda")
    x_d, Wr_d, br_d, K_d, V_d = (to_dev(a) for a in (x, Wr, br, Kc, Vc))

    def run(seq, pos, status):
        out = torch.empty((T, 256), dtype=torch.bfloat16, device="cuda")
        dm.dsmoe_moa_forward(desc, 2, 0.2, K_d, V_d, to_dev(seq), to_dev(pos), x_d, Wr_d, br_d, packed, out, None, None, ws, status)
        torch.cuda.synchronize()
        return out

    wild_seq, wild_pos = seq.copy(), pos.copy()
    wild_seq[[1, 5]], wild_pos[[2, 7]] = (-3, n_seq + 5), (-1, L + 7)
    inside = np.clip(wild_seq, 0, n_seq - 1), np.clip(wild_pos, 0, L - 1)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    want = run(*inside, status)
    assert int(status.item()) == 0
    assert torch.equal(run(wild_seq, wild_pos, status), want)
    assert int(status.item()) == 1                                   # DSMOE_ERR_INVALID_ARG
    assert torch.equal(run(wild_seq, wild_pos, None), want)


# Groups of four tiles whose tokens share no keys (a token whose sequence is neither the group's first nor its last): with short
# caches each warp walks its own tile, with long ones the key-splitting kernel takes the group -- grouped and dense output
# projection, prompts beside decoding sequences, tokens round-robin over the sequences, one and several row tiles per token.
MIXED = [
    # name, T, d, E, n_head, d_head, n_seq, L, order, mode, selection
    ("round_robin_short", 200, 256, 8, 2, 64, 5, 90, "round", gi.MODE_TOPK, dict(K=5)),
    ("round_robin_short_128", 333, 256, 4, 2, 128, 9, 65, "round", gi.MODE_TOPK, dict(K=3)),
    ("round_robin_threshold", 300, 256, 16, 2, 96, 7, 512, "round", gi.MODE_THRESHOLD, dict(eps=0.15)),
    ("round_robin_row_tiles", 90, 256, 20, 2, 64, 3, 70, "round", gi.MODE_ALL, dict()),
    ("round_robin_long", 1600, 256, 8, 4, 64, 5, 530, "round", gi.MODE_TOPK, dict(K=5)),
    ("decode_and_prompt_long", 1031, 256, 8, 4, 128, 32, 1100, "decode_prompt", gi.MODE_TOPK, dict(K=5)),
    ("decode_and_prompt_short", 531, 256, 8, 4, 64, 20, 512, "decode_prompt", gi.MODE_TOPK, dict(K=5)),
    ("long_row_tiles", 500, 256, 20, 2, 64, 4, 700, "round", gi.MODE_ALL, dict()),
    ("round_robin_dense", 4701, 1024, 8, 2, 64, 7, 300, "round", gi.MODE_TOPK, dict(K=4)),
    ("decode_and_prompt_dense_long", 4671, 1024, 8, 4, 96, 64, 4700, "decode_prompt", gi.MODE_TOPK, dict(K=5)),
    ("round_robin_dense_long", 4640, 1024, 20, 2, 64, 11, 600, "round", gi.MODE_ALL, dict()),
]


@pytest.mark.parametrize("case", MIXED, ids=[c[0] for c in MIXED])
def test_moa_mixed_groups(case):
    name, T, d, E, nh, dh, n_seq, L, order, mode, sel = case
    s, x, Wr, br, Wq, Wo, Kc, Vc, seq, pos = _moa_case(name, T, d, E, nh, dh, n_seq, L, "mixed", mode, **sel)
    if order == "round":
        seq = (np.arange(T) % n_seq).astype(np.int32)
    else:                                          # one decoding token per sequence but the last, whose prompt is the rest
        seq = np.minimum(np.arange(T), n_seq - 1).astype(np.int32)
        pos[n_seq - 1:] = np.arange(T - n_seq + 1)
        assert pos.max() < L
    e, er = _run(s, x, Wr, br, Wq, Wo, Kc, Vc, seq, pos, nh, 1.0 / math.sqrt(dh), sample=200)
    assert er <= TOL_BF16, (e, er)
