"""Both projections of the sparse expert MLPs in one launch (fuse_combine = 0) against the two separate launches (2), which the oracle
tests cover: the same tiles, the same order of additions, so the same bits -- where the dealing out of tiles can go wrong:
one and several rounds of up tiles, incomplete ones of every kind, experts of 0, 1, 128 and 129 rows, ragged column ranges, a
reduction shorter than the ring, more tiles per CTA than one list holds (GPU required)."""
import pytest
import torch

import paper_2404_05567_b200 as dm

pytestmark = pytest.mark.gpu

CASES = [
    # T, d, H, E, mode, K, eps (normalised), out_fp32
    (129, 64, 64, 3, dm.SELECT_TOPK, 1, 0.0, 0),              # fewer tiles than CTAs, one reduction block
    (300, 320, 192, 8, dm.SELECT_TOPK, 3, 0.0, 1),            # ragged last column ranges of both projections
    (1000, 2048, 256, 32, dm.SELECT_THRESHOLD, 0, 0.9, 0),    # one round of up tiles
    (2000, 256, 1408, 64, dm.SELECT_THRESHOLD, 0, 2.5, 0),    # several rounds, few down tiles, empty experts
    (4096, 1024, 512, 32, dm.SELECT_TOPK, 6, 0.0, 0),         # several rounds, the last incomplete
    (5000, 6144, 64, 16, dm.SELECT_TOPK, 4, 0.0, 0),          # more than 32 down tiles per CTA
    (6000, 128, 6144, 16, dm.SELECT_THRESHOLD, 0, 0.9, 1),    # more than 32 up tiles per CTA, one round or two of down tiles
    (700, 512, 256, 5, dm.SELECT_THRESHOLD, 0, 1e9, 0),       # nothing selected
    (16384 + 70, 64, 64, 8, dm.SELECT_TOPK, 2, 0.0, 0),       # the counters are zeroed behind the one-block scan kernel
    (2, 64, 64, 64, dm.SELECT_THRESHOLD_TOPK, 0, 0.9, 0),     # few tokens; of one token the workspace has no room for the counters: two launches
    (1, 64, 64, 64, dm.SELECT_THRESHOLD_TOPK, 0, 0.9, 0),
]


@pytest.mark.parametrize("case", CASES, ids=lambda c: f"T{c[0]}-d{c[1]}-H{c[2]}-E{c[3]}")
def test_one_launch_equals_two(case):
    T, d, H, E, mode, K, eps, out_fp32 = case
    g = torch.Generator(device="cuda").manual_seed(T)
    randn = lambda *shape, dtype=torch.bfloat16: torch.randn(*shape, generator=g, device="cuda", dtype=dtype)
    x, Wr = randn(T, d), randn(d, E, dtype=torch.float32) * (1.5 / d ** 0.5)
    W1, W2 = randn(E, d, H) * 0.05, randn(E, H, d) * 0.05
    xs = [x, x.flip(0).contiguous(), randn(T, d)]
    want = {}
    for fuse in (2, 0):
        desc = dm.make_desc(T, d, H, E, dm.BF16, mode, eps, 1, max(K, 1), 0, out_fp32, fuse)
        packed = torch.empty(dm.dsmoe_packed_size(desc), dtype=torch.uint8, device="cuda")
        dm.dsmoe_pack_weights(desc, W1, W2, packed)
        ws = torch.full((dm.dsmoe_workspace_size_packed(desc),), 0x5a, dtype=torch.uint8, device="cuda")     # counters are not zero by chance
        status = torch.zeros(1, dtype=torch.int32, device="cuda")
        got = []
        # the first call finds the fill, every later one another input's hidden activations and counters; no waits in between
        for i in (0, 1, 2, 0, 2, 1) if fuse == 0 else (0, 1, 2):
            out = torch.full((T, d), float("nan"), dtype=torch.float32 if out_fp32 else torch.bfloat16, device="cuda")
            counts = torch.zeros(E, dtype=torch.int32, device="cuda")
            dm.dsmoe_layer_forward(desc, xs[i], Wr, None, None, None, packed, out, None, counts, ws, status)
            got.append((i, out, counts))
        torch.cuda.synchronize()
        assert int(status.item()) == 0
        for i, out, counts in got:
            if fuse == 2:
                want[i] = (out, counts)
            assert torch.equal(out, want[i][0]) and torch.equal(counts, want[i][1]), i
            if eps == 1e9:
                assert not out.any()


def test_rows_around_a_tile():
    """Experts of exactly 0, 1, 127, 128, 129 and 257 rows."""
    rows = [0, 1, 127, 128, 129, 257]
    E, d, H, T = len(rows), 128, 192, sum(rows)
    g = torch.Generator(device="cuda").manual_seed(7)
    # the first E columns of x choose the expert (their weights are scaled out of the experts' way)
    owner = torch.cat([torch.full((n,), e) for e, n in enumerate(rows)])[torch.randperm(T, generator=torch.Generator().manual_seed(3))].cuda()
    x = torch.randn(T, d, generator=g, device="cuda", dtype=torch.bfloat16)
    x[:, :E] = torch.nn.functional.one_hot(owner, E).to(x.dtype) * 4
    Wr = torch.zeros(d, E, device="cuda")
    Wr[:E] = torch.eye(E, device="cuda") * 5
    W1 = (torch.randn(E, d, H, generator=g, device="cuda") * 0.05).bfloat16()
    W2 = (torch.randn(E, H, d, generator=g, device="cuda") * 0.05).bfloat16()
    outs = []
    for fuse in (2, 0):
        desc = dm.make_desc(T, d, H, E, dm.BF16, dm.SELECT_TOPK, 0.0, 0, 1, 0, 1, fuse)
        packed = torch.empty(dm.dsmoe_packed_size(desc), dtype=torch.uint8, device="cuda")
        dm.dsmoe_pack_weights(desc, W1, W2, packed)
        ws = torch.empty(dm.dsmoe_workspace_size_packed(desc), dtype=torch.uint8, device="cuda")
        status = torch.zeros(1, dtype=torch.int32, device="cuda")
        out = torch.empty(T, d, device="cuda")
        counts = torch.zeros(E, dtype=torch.int32, device="cuda")
        dm.dsmoe_layer_forward(desc, x, Wr, None, None, None, packed, out, None, counts, ws, status)
        torch.cuda.synchronize()
        assert int(status.item()) == 0 and counts.tolist() == rows
        outs.append(out)
    assert torch.equal(outs[0], outs[1])
    # ... and the value itself, in fp32 from the same bf16 operands: h is rounded to bf16 (2^-9) before the second product
    want = torch.stack([torch.nn.functional.gelu(x[t].float() @ W1[e].float()) @ W2[e].float() for t, e in enumerate(owner.tolist())])
    gate = torch.softmax(x.float() @ Wr, dim=1).gather(1, owner[:, None])
    assert (outs[1] - gate * want).norm() <= 6e-3 * (gate * want).norm()


def test_offsets_out_of_order_are_reported():
    """A workspace whose expert offsets are overwritten during the call (here by counts_out, made to lie on them: counts that
    descend somewhere are no offsets): no tile leaves its range, the call reports DSMOE_ERR_INVALID_ARG, and the next one is whole."""
    T, d, H, E = 700, 128, 192, 8
    g = torch.Generator(device="cuda").manual_seed(11)
    x, Wr = torch.randn(T, d, generator=g, device="cuda").bfloat16(), torch.randn(d, E, generator=g, device="cuda") * 0.2
    W1, W2 = (torch.randn(E, *s, generator=g, device="cuda").bfloat16() * 0.05 for s in ((d, H), (H, d)))
    desc = dm.make_desc(T, d, H, E, dm.BF16, dm.SELECT_TOPK, 0.0, 0, 3, 0, 0, 0)
    packed = torch.empty(dm.dsmoe_packed_size(desc), dtype=torch.uint8, device="cuda")
    dm.dsmoe_pack_weights(desc, W1, W2, packed)
    ws = torch.zeros(dm.dsmoe_workspace_size_packed(desc), dtype=torch.uint8, device="cuda")
    status, out = torch.zeros(1, dtype=torch.int32, device="cuda"), torch.empty(T, d, device="cuda", dtype=torch.bfloat16)
    counts = torch.zeros(E, dtype=torch.int32, device="cuda")
    dm.dsmoe_layer_forward(desc, x, Wr, None, None, None, packed, out, None, counts, ws, status)
    want = out.clone()
    assert int(status.item()) == 0 and any(a > b for a, b in zip(counts.tolist(), counts.tolist()[1:]))
    up = lambda n: (n + 255) // 256 * 256
    at = up(T * E * 4) + up(T * 8) + up(T * 4) + up(64 * 4)          # scores, mask, k_t, counts lie before the offsets
    offsets = ws[at:at + 4 * (E + 1)].view(torch.int32)
    ends = [0] + counts.cumsum(0).tolist()
    assert offsets.tolist() == ends
    dm.dsmoe_layer_forward(desc, x, Wr, None, None, None, packed, out, None, offsets, ws, status)
    torch.cuda.synchronize()
    assert int(status.item()) == 1                                   # DSMOE_ERR_INVALID_ARG
    status.zero_()
    dm.dsmoe_layer_forward(desc, x, Wr, None, None, None, packed, out, None, counts, ws, status)
    torch.cuda.synchronize()
    assert int(status.item()) == 0 and torch.equal(out, want)


def _layer(T, d, H, E, K, seed):
    """desc, call(x, out, ws, status), x and the workspace of a top-K layer"""
    g = torch.Generator(device="cuda").manual_seed(seed)
    x, Wr = torch.randn(T, d, generator=g, device="cuda").bfloat16(), torch.randn(d, E, generator=g, device="cuda") * (1.5 / d ** 0.5)
    W1, W2 = (torch.randn(E, *s, generator=g, device="cuda").bfloat16() * 0.05 for s in ((d, H), (H, d)))
    desc = dm.make_desc(T, d, H, E, dm.BF16, dm.SELECT_TOPK, 0.0, 0, K, 0, 0, 0)
    packed = torch.empty(dm.dsmoe_packed_size(desc), dtype=torch.uint8, device="cuda")
    dm.dsmoe_pack_weights(desc, W1, W2, packed)

    def call(x, out, ws, status):
        dm.dsmoe_layer_forward(desc, x, Wr, None, None, None, packed, out, None, None, ws, status)
    return call, x, torch.full((dm.dsmoe_workspace_size_packed(desc),), 0x5a, dtype=torch.uint8, device="cuda")


# no up tile, and fewer of them than CTAs: the others begin with down tiles; several rounds
PART = [(129, 64, 64, 3, 1), (300, 512, 256, 8, 3), (4096, 1024, 512, 32, 6)]


@pytest.mark.parametrize("sms", [16, 72])
def test_on_a_part_of_the_gpu(sms):
    """A stream that owns some of the SMs: not every CTA of the launch runs at once, and the others' tiles are taken over."""
    cu = pytest.importorskip("cuda.bindings.driver")

    def ok(r):
        assert r[0] == cu.CUresult.CUDA_SUCCESS, r[0]
        return r[1] if len(r) == 2 else r[1:]
    torch.zeros(1, device="cuda")
    dev = ok(cu.cuDeviceGet(torch.cuda.current_device()))
    whole = ok(cu.cuDeviceGetDevResource(dev, cu.CUdevResourceType.CU_DEV_RESOURCE_TYPE_SM))
    groups, n, _ = ok(cu.cuDevSmResourceSplitByCount(1, whole, 0, sms))
    assert n == 1 and sms <= groups[0].sm.smCount < whole.sm.smCount
    part = ok(cu.cuGreenCtxCreate(ok(cu.cuDevResourceGenerateDesc([groups[0]], 1)), dev, cu.CUgreenCtxCreate_flags.CU_GREEN_CTX_DEFAULT_STREAM))
    raw = ok(cu.cuGreenCtxStreamCreate(part, cu.CUstream_flags.CU_STREAM_NON_BLOCKING, 0))
    stream = torch.cuda.ExternalStream(int(raw))
    try:
        for shape in PART:
            call, x, ws = _layer(*shape, seed=sms)
            status = torch.zeros(1, dtype=torch.int32, device="cuda")
            xs = [x, x.flip(0).contiguous()]
            want = [torch.empty_like(x) for _ in xs]
            for a, b in zip(xs, want):
                call(a, b, ws, status)
            got = [torch.full_like(x, float("nan")) for _ in range(6)]
            torch.cuda.synchronize()
            with torch.cuda.stream(stream):
                for i, out in enumerate(got):
                    call(xs[i % 2], out, ws, status)
            stream.synchronize()
            assert int(status.item()) == 0
            for i, out in enumerate(got):
                assert torch.equal(out, want[i % 2]), (shape, i)
    finally:
        torch.cuda.synchronize()
        ok(cu.cuStreamDestroy(raw) + (None,))
        ok(cu.cuGreenCtxDestroy(part) + (None,))


@pytest.mark.parametrize("shape", PART, ids=lambda s: f"T{s[0]}-d{s[1]}-H{s[2]}-E{s[3]}")
def test_two_streams_with_a_workspace_each(shape):
    call, x, ws = _layer(*shape, seed=3)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    xs = [x, x.flip(0).contiguous()]
    want = [torch.empty_like(x) for _ in xs]
    for a, b in zip(xs, want):
        call(a, b, ws, status)
    streams, wss = [torch.cuda.Stream(), torch.cuda.Stream()], [ws, torch.full_like(ws, 0x5a)]
    got = [[torch.full_like(x, float("nan")) for _ in range(20)] for _ in streams]
    torch.cuda.synchronize()
    for i in range(20):
        for k, st in enumerate(streams):
            with torch.cuda.stream(st):
                call(xs[(i + k) % 2], got[k][i], wss[k], status)
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    for k in range(2):
        for i in range(20):
            assert torch.equal(got[k][i], want[(i + k) % 2]), (k, i)


def test_a_workspace_for_the_running_sums_alone_is_still_enough():
    """Wide experts with many rows under top-K: with room for the tokens' sums but not for the expert outputs' rows the sum is taken inside
    the down-projection, as with fuse_combine = 1; with less the call is refused, and so is a narrower layer with as little."""
    T, d, E, K = 2048, 128, 4, 2
    g = torch.Generator(device="cuda").manual_seed(5)
    for H in (1024, 512):
        W1, W2 = (torch.randn(s, generator=g, device="cuda").bfloat16() * 0.05 for s in ((E, d, H), (E, H, d)))
        x, Wr = torch.randn((T, d), generator=g, device="cuda").bfloat16(), torch.randn((d, E), generator=g, device="cuda") * 0.1
        desc = {f: dm.make_desc(T, d, H, E, dm.BF16, dm.SELECT_TOPK, K=K, fuse_combine=f) for f in (0, 1)}
        packed = torch.empty(dm.dsmoe_packed_size(desc[0]), dtype=torch.uint8, device="cuda")
        dm.dsmoe_pack_weights(desc[0], W1, W2, packed)
        small, full = dm.dsmoe_workspace_size_packed(desc[1]), dm.dsmoe_workspace_size_packed(desc[0])
        assert small < full

        def run(f, nbytes):
            ws, out = torch.empty(nbytes, dtype=torch.uint8, device="cuda"), torch.empty((T, d), dtype=torch.bfloat16, device="cuda")
            status = torch.zeros(1, dtype=torch.int32, device="cuda")
            dm.dsmoe_layer_forward(desc[f], x, Wr, None, None, None, packed, out, None, None, ws, status)
            torch.cuda.synchronize()
            assert int(status.item()) == 0
            return out

        if H == 1024:
            assert torch.equal(run(0, small), run(1, small))
            with pytest.raises(dm.DsmoeError):
                run(0, small - 1)
        else:
            with pytest.raises(dm.DsmoeError):
                run(0, small)
        err = (run(0, full).float() - run(1, small).float()).norm() / run(1, small).float().norm()
        assert err <= 2 ** -8                                     # one rounding to bf16 of sums that differ by rounding in fp32


def test_the_other_entry_points_take_that_workspace_too():
    """dsmoe_moa_forward (sum inside, as with fuse_combine = 1), dsmoe_expert_mlp and dsmoe_dense_backward (nothing of theirs lies there):
    the bits of a call with the full workspace, or of fuse_combine = 1; with one byte less the call is refused."""
    T, d, E, K, H, nh, L = 2048, 128, 4, 2, 1024, 8, 64
    g = torch.Generator(device="cuda").manual_seed(6)
    randn = lambda *s, std=1.0: (torch.randn(s, generator=g, device="cuda") * std).bfloat16()
    x, dO, W1, W2 = randn(T, d), randn(T, d), randn(E, d, H, std=0.05), randn(E, H, d, std=0.05)
    Wr, Kc, Vc = torch.randn((d, E), generator=g, device="cuda") * 0.1, randn(2, nh, L, H // nh), randn(2, nh, L, H // nh)
    tok = torch.arange(T, device="cuda", dtype=torch.int32)
    seq, pos = tok // 1024, tok % L
    desc = {f: dm.make_desc(T, d, H, E, dm.BF16, dm.SELECT_TOPK, K=K, fuse_combine=f) for f in (0, 1)}
    packed = torch.empty(dm.dsmoe_packed_size(desc[0]), dtype=torch.uint8, device="cuda")
    dm.dsmoe_pack_weights(desc[0], W1, W2, packed)
    small, full = dm.dsmoe_workspace_size_packed(desc[1]), dm.dsmoe_workspace_size_packed(desc[0])
    assert small < full
    status, scores = torch.zeros(1, dtype=torch.int32, device="cuda"), torch.empty((T, E), device="cuda")
    dm.dsmoe_router(desc[0], x, Wr, None, scores)
    offsets = torch.arange(E + 1, device="cuda", dtype=torch.int32) * (T * K // E)
    xp = randn(T * K, d)

    def moa(f, n):
        out = torch.empty((T, d), dtype=torch.bfloat16, device="cuda")
        dm.dsmoe_moa_forward(desc[f], nh, 0.09, Kc, Vc, seq, pos, x, Wr, None, packed, out, None, None, ws[:n], status)
        return [out]

    def experts(f, n):
        yp = torch.empty((T * K, d), dtype=torch.bfloat16, device="cuda")
        dm.dsmoe_expert_mlp(desc[f], xp, None, None, packed, offsets, yp, ws[:n], status)
        return [yp]

    def backward(f, n):
        dS, dA = torch.empty((T, E), device="cuda"), torch.empty((T, E * H), dtype=torch.bfloat16, device="cuda")
        dm.dsmoe_dense_backward(desc[f], x, None, W2, packed, scores, None, dO, dS, dA, ws[:n], status)
        return [dS, dA]

    ws = torch.empty(full, dtype=torch.uint8, device="cuda")
    for call, like in ((moa, (1, small)), (experts, (0, full)), (backward, (0, full))):
        ws.fill_(0x5a)
        got = call(0, small)
        torch.cuda.synchronize()
        assert int(status.item()) == 0 and (ws[small:] == 0x5a).all()
        for a, b in zip(got, call(*like)):
            assert torch.equal(a, b), call.__name__
        with pytest.raises(dm.DsmoeError):
            call(0, small - 1)
