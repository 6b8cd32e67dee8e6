"""The work that users of this library have it do, as cases that can be timed and compared.

A case is one call (or, for training, the three calls of one step) through the public binding, on seeded synthetic
inputs that already sit on the GPU, with the weights packed once as a serving or training program keeps them:

  layer     dsmoe_layer_forward: the mixture-of-experts feed-forward layer -- decode batches, the batches between
            decode and prefill, prefill, the skewed router, the dense (all-expert) forward, fp32 layers
  training  dsmoe_router + dsmoe_mi_loss + dsmoe_dense_backward: the training side of the dense layer
  moa       dsmoe_moa_forward: the mixture-of-attention-heads layer, prompts and decoding against a key/value cache

Layer shapes are this repository's own: the benchmark configurations (d 2048 / H 1024, d 3072 / H 1536, d 4096 / H 1408,
the tiny fp32 layer) and the paper's models (32 experts, d / H = 2048/256, 3072/384, 4096/512, 5120/640, 6144/768).
"""
import math

import numpy as np
import torch

import paper_2404_05567_b200 as dm

F32, BF16 = "f32", "bf16"
_MODES = {"threshold": dm.SELECT_THRESHOLD, "topk": dm.SELECT_TOPK, "all": dm.SELECT_ALL,
          "threshold_topk": dm.SELECT_THRESHOLD_TOPK}
# Router logits are drawn with these standard deviations: 0.905 is what N(0,1) tokens and N(0, 0.02^2) router weights
# give at d = 2048, where a threshold of 0.9654 on the normalised probability keeps 35 % of the experts; 1.56 is the
# tiny fp32 layer's, where 0.8 keeps 35 %.
_LOGIT_STD, _EPS = 0.905, 0.9654
_LOGIT_STD_F32, _EPS_F32 = 1.56, 0.8


def _layer(T, d, H, E, mode, *, dtype=BF16, eps=0.0, K=0, zipf=False, fp32_out=False):
    """eps is on the normalised probability S * E, the paper's form."""
    return {"kind": "layer", "T": T, "d": d, "H": H, "E": E, "dtype": dtype, "mode": mode, "eps": eps, "K": K,
            "zipf": zipf, "fp32_out": fp32_out}


def _training(T, d, H, E):
    return {"kind": "training", "T": T, "d": d, "H": H, "E": E, "dtype": BF16, "mode": "all", "eps": 0.0, "K": 0,
            "zipf": False}


def _moa(n_seq, new_tokens, cache, d, n_head, d_head, E, K):
    """n_seq sequences with `new_tokens` new tokens each: 1 = decoding at the end of a cache of `cache` positions,
    otherwise prompts from position 0 on (cache == new_tokens)."""
    return {"kind": "moa", "T": n_seq * new_tokens, "d": d, "H": n_head * d_head, "E": E, "dtype": BF16, "mode": "topk",
            "eps": 0.0, "K": K, "zipf": False, "n_seq": n_seq, "new_tokens": new_tokens, "cache": cache,
            "n_head": n_head, "d_head": d_head}


def listed():
    named = [
        # the smallest calls: a tiny fp32 layer (the library's reference configuration), all latency
        ("fp32_t64", _layer(64, 256, 512, 8, "threshold", dtype=F32, eps=_EPS_F32)),
        # one user decoding: a single token through the decode configuration
        ("decode_t1", _layer(1, 2048, 1024, 32, "threshold", eps=_EPS)),
        # a decode batch: the configuration the benchmark's headline is quoted on
        ("decode_t32", _layer(32, 2048, 1024, 32, "threshold", eps=_EPS)),
        # a larger, odd decode batch on the paper's 3B layer
        ("decode_t100_3b", _layer(100, 3072, 384, 32, "topk", K=6)),
        # between decode and prefill: a ragged batch of continuous batching (decodes mixed with prompt chunks)
        ("batch_t300", _layer(300, 2048, 1024, 32, "threshold", eps=_EPS)),
        # prefill with wide experts, top-K
        ("prefill_wide", _layer(8192, 3072, 1536, 32, "topk", K=12)),
        # prefill on the paper's 6B layer with a ragged token count, top-K as in its speed tests
        ("prefill_6b_t7001", _layer(7001, 4096, 512, 32, "topk", K=4)),
        # a skewed router with empty experts: Zipf popularity, raw threshold 0.05 (3.2 normalised), 64 experts
        ("prefill_skewed", _layer(4096, 4096, 1408, 64, "threshold", eps=3.2, zipf=True)),
        # the dense-training forward: every expert evaluated and weighted by its score
        ("dense_t16384", _layer(16384, 2048, 1024, 32, "all")),
        # one training step of the dense layer on a ragged batch: scores, mutual-information loss, gradients
        ("training_t8190", _training(8190, 2048, 1024, 32)),
        # mixture of attention heads, the 6B attention block: 32 prompts of 256 tokens
        ("moa_prefill", _moa(32, 256, 256, 4096, 4, 128, 8, 5)),
        # ... and decoding: 32 sequences, one new token each, 2048 cached positions
        ("moa_decode", _moa(32, 1, 2048, 4096, 4, 128, 8, 5)),
    ]
    return [dict(case, name=name) for name, case in named]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


_EXPERT_SHAPES = [(2048, 256), (3072, 384), (4096, 512), (2048, 1024)]          # decode and mixed batches
_PREFILL_SHAPES = _EXPERT_SHAPES + [(3072, 1536), (5120, 640), (6144, 768)]


def draw(rng):
    kind = rng.choice(["fp32", "decode", "decode", "batch", "prefill", "prefill", "dense", "training", "moa_prefill",
                       "moa_decode"])
    if kind == "fp32":
        return _layer(_log_int(rng, 1, 300), rng.choice([128, 256, 384, 512]), rng.choice([136, 256, 512, 1024]),
                      rng.choice([4, 8, 16]), rng.choice(["threshold", "topk"]), dtype=F32, eps=_EPS_F32,
                      K=rng.choice([1, 2, 3]))
    if kind in ("decode", "batch"):
        d, H = rng.choice(_EXPERT_SHAPES)
        T = _log_int(rng, 1, 128) if kind == "decode" else _log_int(rng, 129, 2047)
        return _layer(T, d, H, 32, rng.choice(["threshold", "topk"]), eps=_EPS, K=rng.choice([4, 6]),
                      fp32_out=rng.random() < 0.15)
    if kind == "prefill":
        if rng.random() < 0.25:
            return _layer(_log_int(rng, 1024, 4096), 4096, 1408, 64, "threshold", eps=rng.choice([0.64, 3.2, 6.4]), zipf=True)
        d, H = rng.choice(_PREFILL_SHAPES)
        mode = rng.choice(["topk", "topk", "threshold", "threshold_topk"])
        return _layer(rng.randint(2048, 8192), d, H, 32, mode, eps=_EPS, K=rng.choice([4, 6, 12]))
    if kind == "dense":
        d, H = rng.choice(_EXPERT_SHAPES)
        return _layer(_log_int(rng, 129, 8192), d, H, 32, "all")
    if kind == "training":
        d, H = rng.choice(_EXPERT_SHAPES)
        return _training(_log_int(rng, 129, 8192), d, H, 32)
    d, n_head, d_head, E, K = rng.choice([(2048, 2, 64, 16, 6), (3072, 4, 96, 8, 5), (4096, 4, 128, 8, 5)])
    if kind == "moa_prefill":
        length = rng.randint(33, 400)
        return _moa(_log_int(rng, 1, 8192 // length), length, length, d, n_head, d_head, E, K)
    return _moa(_log_int(rng, 1, 64), 1, _log_int(rng, 100, 3000), d, n_head, d_head, E, K)


# ---------------------------------------------------------------- what a user's program has in hand

def _zipf_bias(E, order):
    p = np.arange(1, E + 1, dtype=np.float64) ** -1.1
    return np.log(p / p.sum())[order]


def prepare(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    c = dict(case)
    T, d, H, E = c["T"], c["d"], c["H"], c["E"]
    dt = torch.float32 if c["dtype"] == F32 else torch.bfloat16

    def normal(shape, std, dtype=dt):
        return torch.randn(shape, generator=g, device="cuda", dtype=dtype).mul_(std)

    s = {"case": c}
    s["x"] = normal((T, d), 1.0)
    std = _LOGIT_STD_F32 if c["dtype"] == F32 else _LOGIT_STD
    s["Wr"] = normal((d, E), std / math.sqrt(d), torch.float32)
    s["br"] = None
    if c["zipf"]:
        order = torch.randperm(E, generator=g, device="cuda").cpu().numpy()
        s["br"] = torch.tensor(_zipf_bias(E, order), dtype=torch.float32, device="cuda")
    W1, W2 = normal((E, d, H), 0.02), normal((E, H, d), 0.02)
    s["desc"] = dm.make_desc(T, d, H, E, dm.F32 if c["dtype"] == F32 else dm.BF16, _MODES[c["mode"]], c["eps"], 1, c["K"], 0,
                             1 if c.get("fp32_out") else 0, 0)
    s["packed"] = None
    if c["dtype"] == BF16:
        s["packed"] = torch.empty(dm.dsmoe_packed_size(s["desc"]), dtype=torch.uint8, device="cuda")
        dm.dsmoe_pack_weights(s["desc"], W1, W2, s["packed"])
    s["W1"], s["W2"] = (W1, W2) if c["dtype"] == F32 else (None, W2 if c["kind"] == "training" else None)
    nbytes = dm.dsmoe_workspace_size_packed(s["desc"]) if c["dtype"] == BF16 else dm.dsmoe_workspace_size(s["desc"])
    s["ws"] = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
    s["status"] = torch.zeros(1, dtype=torch.int32, device="cuda")
    if c["kind"] == "training":
        s["dO"] = normal((T, d), 1.0)
        s["scores"] = torch.empty((T, E), dtype=torch.float32, device="cuda")
        s["loss"] = torch.empty(3, dtype=torch.float32, device="cuda")
        s["mi_grad"] = torch.empty((T, E), dtype=torch.float32, device="cuda")
        s["dS"] = torch.empty((T, E), dtype=torch.float32, device="cuda")
        s["dA"] = torch.empty((T, E * H), dtype=dt, device="cuda")
        return s
    s["out"] = torch.empty((T, d), dtype=torch.float32 if c.get("fp32_out") else dt, device="cuda")
    s["mask"] = torch.zeros(T, dtype=torch.int64, device="cuda")
    s["counts"] = torch.zeros(E, dtype=torch.int32, device="cuda")
    if c["kind"] == "moa":
        shape = (c["n_seq"], c["n_head"], c["cache"], c["d_head"])
        s["K"], s["V"] = normal(shape, 1.0), normal(shape, 1.0)
        tok = torch.arange(T, device="cuda", dtype=torch.int32)
        s["seq"] = tok // c["new_tokens"]
        s["pos"] = tok % c["new_tokens"] if c["new_tokens"] > 1 else torch.full_like(tok, c["cache"] - 1)
    return s


def run(s):
    c, desc = s["case"], s["desc"]
    if c["kind"] == "training":
        dm.dsmoe_router(desc, s["x"], s["Wr"], s["br"], s["scores"])
        dm.dsmoe_mi_loss(desc, s["scores"], s["loss"], s["mi_grad"], s["ws"])
        dm.dsmoe_dense_backward(desc, s["x"], None, s["W2"], s["packed"], s["scores"], None, s["dO"], s["dS"], s["dA"],
                                s["ws"], s["status"])
        return {"loss": s["loss"], "mi_grad": s["mi_grad"], "dS": s["dS"], "dA": s["dA"], "scores": s["scores"]}
    if c["kind"] == "moa":
        dm.dsmoe_moa_forward(desc, c["n_head"], 1.0 / math.sqrt(c["d_head"]), s["K"], s["V"], s["seq"], s["pos"], s["x"],
                             s["Wr"], s["br"], s["packed"], s["out"], s["mask"], s["counts"], s["ws"], s["status"])
    else:
        dm.dsmoe_layer_forward(desc, s["x"], s["Wr"], s["br"], s["W1"], s["W2"], s["packed"], s["out"], s["mask"],
                               s["counts"], s["ws"], s["status"])
    return {"out": s["out"], "mask": s["mask"], "counts": s["counts"]}


# ---------------------------------------------------------------- the work of a pass

def _selected(c):
    """(assignments, experts that at least one token selects), expected over the inputs of a seed."""
    T, E = c["T"], c["E"]
    if c["mode"] == "all":
        return float(T * E), float(E)
    r = np.random.RandomState(0)
    logits = r.standard_normal((4096, E)) * (_LOGIT_STD_F32 if c["dtype"] == F32 else _LOGIT_STD)
    if c["zipf"]:
        logits = logits + _zipf_bias(E, np.arange(E))
    p = np.exp(logits)
    p /= p.sum(axis=1, keepdims=True)
    if c["mode"] == "topk":
        share = np.full(E, min(c["K"], E) / E)
    else:
        share = (p * E > c["eps"]).mean(axis=0)
        if c["mode"] == "threshold_topk":
            share = np.full(E, min(E, max(1, math.floor(share.sum() + 0.5))) / E)
    return float(T * share.sum()), float(np.sum(1.0 - (1.0 - share) ** T))


def work(case):
    c = case
    T, d, H, E = c["T"], c["d"], c["H"], c["E"]
    es = 4 if c["dtype"] == F32 else 2
    A, used = _selected(c)
    router = 2.0 * T * d * E
    if c["kind"] == "training":
        # scores, loss gradient and dS [T,E]; x, dO; both weight tensors; the gradient at the hidden activations
        return {"bytes": T * d * 2 * es + d * E * 4 + 2 * E * d * H * es + 3 * T * E * 4 + T * E * H * es,
                "flops": router + 4.0 * T * E * d * H + 2.0 * T * E * H}
    nbytes = T * d * es + T * d * (4 if c.get("fp32_out") else es) + d * E * 4 + used * 2 * d * H * es + T * 8
    flops = router + 4.0 * A * d * H
    if c["kind"] == "moa":
        seen = c["cache"] if c["new_tokens"] == 1 else (c["new_tokens"] + 1) / 2
        nbytes += 2.0 * c["n_seq"] * c["n_head"] * c["cache"] * c["d_head"] * es
        flops += 4.0 * A * H * seen
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    """About four times the distance from the same layer in float64: 5e-7 (largest element 2.8e-6) for fp32 at d = 256,
    more with longer sums; 2.4e-3 to 3.4e-3 (largest element 2.3e-2) for bf16.  A whole value that differs is a score
    within rounding of the selection's boundary."""
    if case["dtype"] == F32:
        return {"rel": 5e-6, "max": 5e-5, "differ": 1e-3}
    return {"rel": 1e-2, "max": 8e-2, "differ": 1e-3}


# ---------------------------------------------------------------- the same outputs in float64

def _up_down(x, W1, W2, gate):
    """sum over e of gate[:, e] * GeLU(x W1[e]) W2[e], only over the tokens with a gate."""
    out = torch.zeros((x.shape[0], W2.shape[2]), dtype=torch.float64, device=x.device)
    for e in range(W1.shape[0]):
        t = gate[:, e].nonzero().flatten()
        if t.numel():
            h = torch.nn.functional.gelu(x[t] @ W1[e].double())
            out.index_add_(0, t, gate[t, e:e + 1] * (h @ W2[e].double()))
    return out


def _attention(c, q, K, V, seq, pos):
    """q [n, n_head, d_head] of tokens with sequences seq and last visible positions pos."""
    o = torch.empty_like(q)
    step = max(1, (1 << 27) // (c["n_head"] * c["cache"] * c["d_head"]))
    at = torch.arange(c["cache"], device=q.device)
    for i in range(0, q.shape[0], step):
        k, v = K[seq[i:i + step]].double(), V[seq[i:i + step]].double()
        a = torch.einsum("nhd,nhld->nhl", q[i:i + step], k) / math.sqrt(c["d_head"])
        a = a.masked_fill(at[None, None, :] > pos[i:i + step, None, None], -math.inf).softmax(dim=-1)
        o[i:i + step] = torch.einsum("nhl,nhld->nhd", a, v)
    return o


def exact(case, seed):
    c, E = case, case["E"]
    s = prepare(case, seed)
    g = torch.Generator(device="cuda").manual_seed(seed)
    # the weights again, as prepare() drew them before it packed them
    dt = torch.float32 if c["dtype"] == F32 else torch.bfloat16
    torch.randn((c["T"], c["d"]), generator=g, device="cuda", dtype=dt)
    torch.randn((c["d"], E), generator=g, device="cuda", dtype=torch.float32)
    if c["zipf"]:
        torch.randperm(E, generator=g, device="cuda")
    W1 = torch.randn((E, c["d"], c["H"]), generator=g, device="cuda", dtype=dt).mul_(0.02)
    W2 = torch.randn((E, c["H"], c["d"]), generator=g, device="cuda", dtype=dt).mul_(0.02)
    x = s["x"].double()
    S = x @ s["Wr"].double()
    if s["br"] is not None:
        S = S + s["br"].double()
    S = S.softmax(dim=1)
    if c["kind"] == "training":
        m = S.mean(dim=0)
        logS, logm = S.log(), m.log()
        H_cond, H_marg = -(S * logS).sum(dim=1).mean(), -(m * logm).sum()
        # L = H(e|X) - H(e): the derivative by one score
        dL = (logm[None, :] - logS) / c["T"]
        dO = s["dO"].double()
        dS = torch.empty_like(S)
        dA = torch.empty((c["T"], E, c["H"]), dtype=torch.float64, device="cuda")
        for e in range(E):
            G = dO @ W2[e].double().T
            dS[:, e] = (torch.nn.functional.gelu(x @ W1[e].double()) * G).sum(dim=1)
            dA[:, e] = S[:, e:e + 1] * G
        return {"loss": torch.stack([H_cond - H_marg, H_marg, H_cond]), "mi_grad": dL, "dS": dS, "dA": dA.view(c["T"], -1),
                "scores": S}
    if c["mode"] == "all":
        sel = torch.ones_like(S, dtype=torch.bool)
    elif c["mode"] == "threshold":
        sel = S * E > c["eps"]
    else:
        k = c["K"]
        if c["mode"] == "threshold_topk":
            k = math.floor((S * E > c["eps"]).sum().item() / c["T"] + 0.5)
        k = min(E, max(1, k))
        sel = torch.zeros_like(S, dtype=torch.bool).scatter_(1, S.topk(k, dim=1).indices, True)
    gate = S * sel
    mask = None if E >= 64 else (sel.long() << torch.arange(E, device="cuda")).sum(dim=1)
    counts = sel.sum(dim=0).int()
    if c["kind"] == "moa":
        out = torch.zeros((c["T"], c["d"]), dtype=torch.float64, device="cuda")
        for e in range(E):
            t = sel[:, e].nonzero().flatten()
            if t.numel():
                q = (x[t] @ W1[e].double()).view(-1, c["n_head"], c["d_head"])
                o = _attention(c, q, s["K"], s["V"], s["seq"][t].long(), s["pos"][t].long())
                out.index_add_(0, t, gate[t, e:e + 1] * (o.reshape(t.numel(), -1) @ W2[e].double()))
        return {"out": out, "mask": mask, "counts": counts}
    return {"out": _up_down(x, W1, W2, gate), "mask": mask, "counts": counts}
