"""The calls whose speed this library is held to, as sizes, inputs and references.

Each case is one use of the public entry points, at a size from the workloads of
``synth/workloads.py``, from the tests, or a generic one: the whole feature path of a batch,
its single stages where a program calls them by themselves, and the fitting of the length
head.  ``listed()`` names the cases, ``draw()`` gives further ones of the same ranges,
``prepare()`` makes what a program holds before the call, ``run()`` makes the call, and
``exact()`` evaluates the same definition in plain 64-bit torch.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2608_15592_gb300 as estp

DEVICE = "cuda:0"
LAMBDA1, LAMBDA2, ALPHA = 0.7, 0.3, 1.0  # the workloads' mix (Eqs. 2-2, 2-3)
LAMBDA3 = 0.5                            # weight of the cross-entropy term (Eq. 3-3)
BIN_WIDTH = 256.0                        # spacing of the length bins' centres


# ------------------------------------------------------------------------- cases
def _features(name, dtype, B, T_lo, T_hi, V, ld, layers, Hq, Hkv, d, D, K=32):
    """Entropy of given logits, importance over `layers` layers, pooling, length head."""
    return {"name": name, "kind": "features", "dtype": dtype, "B": B, "T_lo": T_lo, "T_hi": T_hi,
            "V": V, "ld": ld, "layers": layers, "Hq": Hq, "Hkv": Hkv, "d": d, "D": D, "K": K}


def _lm_head(name, rows, D, V):
    """Entropy straight from hidden states and the output projection."""
    return {"name": name, "kind": "lm_head", "rows": rows, "D": D, "V": V}


def _attention(name, dtype, B, T_lo, T_hi, Hq, Hkv, d, n_heads=0, lse_given=False, sinks=0,
               exclude_self=False, divisor="length"):
    """One layer's importance: row normalisers (unless the prefill supplied them), column
    sums over the first n_heads of each KV group (0: all), and the closing scaling."""
    return {"name": name, "kind": "attention", "dtype": dtype, "B": B, "T_lo": T_lo, "T_hi": T_hi,
            "Hq": Hq, "Hkv": Hkv, "d": d, "n_heads": n_heads, "lse_given": lse_given,
            "sinks": sinks, "exclude_self": exclude_self, "divisor": divisor}


def _forward(name, B, T_lo, T_hi, Hq, Hkv, lse_given=False):
    """One layer's prefill attention output with the importance of the same probabilities."""
    return {"name": name, "kind": "forward", "dtype": "bf16", "B": B, "T_lo": T_lo, "T_hi": T_hi,
            "Hq": Hq, "Hkv": Hkv, "d": 128, "lse_given": lse_given, "sinks": 0}


def _head(name, B, D, K, F):
    """One training step's loss and gradients of the length head: linear (F = 0) or with a
    hidden layer of F units."""
    return {"name": name, "kind": "head", "B": B, "D": D, "K": K, "F": F}


def _misalign(name, B, T_lo, T_hi, pct):
    """Counts of high-entropy tokens of low importance and the reverse."""
    return {"name": name, "kind": "misalign", "B": B, "T_lo": T_lo, "T_hi": T_hi, "pct": pct}


def listed():
    return [
        # the smallest request: one 128-token prompt in fp32, the whole path; launches and
        # latency are what it costs
        _features("features_f32_T128", "f32", 1, 128, 128, 32000, 32000, 1, 8, 8, 64, 1024),
        # an ordinary serving batch of 16 ragged prompts with its logits in memory, importance
        # from the last four layers
        _features("features_bf16_varlen16", "bf16", 16, 256, 2048, 152064, 152064, 4, 28, 4, 128, 3584),
        # entropy without stored logits: a single short prompt (one pass over the projection) ...
        _lm_head("lm_head_37", 37, 3584, 152064),
        # ... and a batch of a few thousand tokens (a ragged number of row blocks)
        _lm_head("lm_head_4103", 4103, 4096, 128256),
        # one layer of the rollout batch: 256 prompts of 128 to 4096 tokens, 32/8 heads; the
        # largest call
        _attention("attention_rl256", "bf16", 256, 128, 4096, 32, 8, 128),
        # one layer of a long-context prompt with attention sinks, the prefill's own row
        # normalisers at hand
        _attention("attention_long32k", "bf16", 1, 32768, 32768, 28, 4, 128, lse_given=True, sinks=4),
        # many short prompts of a small model (head dim 64), half of the heads, the variant
        # without the self term and with the causal count
        _attention("attention_short_d64", "bf16", 48, 16, 300, 16, 8, 64, n_heads=8,
                   exclude_self=True, divisor="causal"),
        # fp32 activations, a few prompts of ordinary length
        _attention("attention_f32", "f32", 4, 300, 1500, 16, 4, 128),
        # the prefill's own attention of the serving batch with the importance taken along
        _forward("forward_varlen16", 16, 256, 2048, 28, 4),
        # fitting the length head on a batch of 256 pooled prompts: the linear head ...
        _head("head_loss_256", 256, 4096, 32, 0),
        # ... and the MLP predictor
        _head("mlp_loss_256", 256, 4096, 32, 1024),
        # the diagnostic over the rollout batch's signals
        _misalign("misalign_rl256", 256, 128, 4096, 40),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _span(rng, lo, hi):
    """A prompt-length range inside [lo, hi]: one fixed length or a ragged spread."""
    t_hi = _log_int(rng, lo, hi)
    t_lo = t_hi if rng.random() < 0.2 else rng.randint(lo, t_hi)
    return t_lo, t_hi


def draw(rng):
    kind = rng.choice(["features_f32", "features_bf16", "lm_head", "attention_bf16", "attention_f32",
                       "forward", "head", "mlp", "misalign"])
    if kind == "features_f32":
        Hq, Hkv = rng.choice([(8, 8), (8, 2), (4, 4)])
        V = _log_int(rng, 1000, 32000)
        t_lo, t_hi = _span(rng, 16, 256)
        case = _features("", "f32", rng.randint(1, 4), t_lo, t_hi, V, (V + 3) // 4 * 4, rng.randint(1, 2),
                         Hq, Hkv, rng.choice([64, 128]), 4 * rng.randint(64, 256))
    elif kind == "features_bf16":
        Hq, Hkv = rng.choice([(28, 4), (32, 8), (16, 16), (12, 2)])
        V = _log_int(rng, 32000, 152064)
        t_lo, t_hi = _span(rng, 32, 2048)
        case = _features("", "bf16", rng.randint(1, min(16, 20000 // t_hi)), t_lo, t_hi, V, (V + 7) // 8 * 8, rng.randint(1, 4),
                         Hq, Hkv, rng.choice([64, 128]), 8 * rng.randint(64, 512))
    elif kind == "lm_head":
        case = _lm_head("", _log_int(rng, 1, 4103), 64 * rng.randint(8, 64), _log_int(rng, 32000, 128256))
    elif kind == "attention_bf16":
        Hq, Hkv = rng.choice([(28, 4), (32, 8), (64, 8), (16, 16)])
        t_lo, t_hi = _span(rng, 16, 16384)
        # no more causal pairs than a quarter of the largest listed call
        B = rng.randint(1, max(1, min(256, int(1.5e9 / (Hq * t_hi * t_hi)), 131072 // t_hi)))
        d = 128 if rng.random() < 0.75 else 64
        case = _attention("", "bf16", B, t_lo, t_hi, Hq, Hkv, d,
                          n_heads=rng.choice([0, 0, 0, Hkv * rng.randint(1, Hq // Hkv)]),
                          lse_given=rng.random() < 0.3, sinks=rng.choice([0, 4]),
                          exclude_self=rng.random() < 0.25, divisor=rng.choice(["length", "length", "causal", "none"]))
    elif kind == "attention_f32":
        Hq, Hkv = rng.choice([(8, 8), (16, 4), (12, 2)])
        t_lo, t_hi = _span(rng, 16, 1500)
        case = _attention("", "f32", rng.randint(1, 4), t_lo, t_hi, Hq, Hkv, rng.choice([64, 128]),
                          lse_given=rng.random() < 0.3, exclude_self=rng.random() < 0.25)
    elif kind == "forward":
        Hq, Hkv = rng.choice([(28, 4), (32, 8), (16, 16)])
        t_lo, t_hi = _span(rng, 16, 4096)
        case = _forward("", rng.randint(1, max(1, min(64, 32768 // t_hi))), t_lo, t_hi, Hq, Hkv,
                        lse_given=rng.random() < 0.5)
    elif kind == "head":
        case = _head("", _log_int(rng, 1, 256), _log_int(rng, 256, 8192), rng.randint(8, 128), 0)
    elif kind == "mlp":
        case = _head("", _log_int(rng, 1, 256), _log_int(rng, 256, 4096), rng.randint(8, 64),
                     _log_int(rng, 64, 1024))
    else:
        t_lo, t_hi = _span(rng, 1, 8192)
        case = _misalign("", _log_int(rng, 1, 256), t_lo, t_hi, rng.randint(5, 50))
    del case["name"]
    return case


# ------------------------------------------------------------------------ inputs
def _dtype(case):
    return torch.bfloat16 if case["dtype"] == "bf16" else torch.float32


def _lengths(case):
    """Prompt lengths: a property of the case (the work depends on them), not of the seed."""
    rng = np.random.default_rng([case["B"], case["T_lo"], case["T_hi"]])
    return rng.integers(case["T_lo"], case["T_hi"] + 1, size=case["B"])


def _bounds(case):
    return np.concatenate([[0], np.cumsum(_lengths(case))]).astype(np.int64)


def _heads(case):
    """Selected query heads, or None for all."""
    n = case.get("n_heads", 0)
    if not n:
        return None
    rep, per = case["Hq"] // case["Hkv"], n // case["Hkv"]
    return [g * rep + i for g in range(case["Hkv"]) for i in range(per)]


def _gen(seed):
    return torch.Generator(device=DEVICE).manual_seed(int(seed))


def _normal(shape, g, dtype=torch.float32, scale=1.0):
    x = torch.empty(shape, dtype=dtype, device=DEVICE).normal_(generator=g)
    return x.mul_(scale) if scale != 1.0 else x


def _qk(case, g, sumT):
    dt = _dtype(case)
    Q = _normal((sumT, case["Hq"], case["d"]), g, dt)
    K = _normal((sumT, case["Hkv"], case["d"]), g, dt)
    if case.get("sinks"):
        cu = _bounds(case)
        idx = [t for b in range(case["B"]) for t in range(cu[b], min(cu[b] + case["sinks"], cu[b + 1]))]
        K[torch.tensor(idx, device=DEVICE)] *= 8
    return Q, K


def _logits(case, g, rows):
    """Rows of scale 0.5 to 4, in bf16 batches with a confident spike in 1 % of the rows."""
    x = torch.empty(rows, case["ld"], dtype=_dtype(case), device=DEVICE)
    sigma = torch.empty(rows, 1, device=DEVICE).uniform_(0.5, 4.0, generator=g)
    for r in range(0, rows, 4096):
        x[r:r + 4096].normal_(generator=g)
        x[r:r + 4096].mul_(sigma[r:r + 4096].to(x.dtype))
    if case["dtype"] == "bf16":
        hit = torch.rand(rows, generator=g, device=DEVICE) < 0.01
        col = torch.randint(case["V"], (rows,), generator=g, device=DEVICE)
        sel = hit.nonzero()[:, 0]
        x[sel, col[sel]] += 12.0
    return x


def _linear_head(g, K, D):
    W = _normal((K, D), g, scale=1.0 / math.sqrt(D))
    centers = (torch.arange(K, device=DEVICE, dtype=torch.float32) + 0.5) * BIN_WIDTH
    return estp.Head(W, _normal((K,), g, scale=0.1), centers)


def _clear_kink(x, W1, b1):
    """Moves the biases of hidden units that are within 1e-5 of the ReLU's kink for some
    prompt: there a rounding decides which side's derivative counts, and both are right."""
    a = x.double() @ W1.double().T
    for _ in range(100):
        near = ((a + b1.double()).abs() < 1e-5).any(dim=0)
        b1 += near * 1e-4


def _row_blocks(T):
    """Query-row blocks of a prompt, small enough for one [heads, rows, keys] block."""
    step = max(1, min(T, 2 ** 27 // max(T, 1)))
    return [(i, min(T, i + step)) for i in range(0, T, step)]


def _scores(Q, K, t0, i0, i1, heads, rep, scale, dtype):
    """Masked scores of query rows i0..i1 of the prompt at t0 against keys 0..i1, one head
    at a time: yields (head, scores)."""
    keep = torch.arange(i1, device=DEVICE)[None, :] <= torch.arange(i0, i1, device=DEVICE)[:, None]
    for h in heads:
        q = Q[t0 + i0:t0 + i1, h].to(dtype)
        k = K[t0:t0 + i1, h // rep].to(dtype)
        yield h, (q @ k.T).mul_(scale).masked_fill_(~keep, -math.inf)


def _row_normalisers(case, Q, K, dtype):
    """lse [Hq, sumT], as the prefill's attention returns it."""
    cu, rep, scale = _bounds(case), case["Hq"] // case["Hkv"], 1.0 / math.sqrt(case["d"])
    lse = torch.empty(case["Hq"], int(cu[-1]), dtype=dtype, device=DEVICE)
    for b in range(case["B"]):
        t0, T = int(cu[b]), int(cu[b + 1] - cu[b])
        for i0, i1 in _row_blocks(T):
            for h, s in _scores(Q, K, t0, i0, i1, range(case["Hq"]), rep, scale, dtype):
                lse[h, t0 + i0:t0 + i1] = torch.logsumexp(s, dim=1)
    return lse


def prepare(case, seed):
    g = _gen(seed)
    st = {"case": case}
    kind = case["kind"]
    if kind == "lm_head":
        st["hidden"] = _normal((case["rows"], case["D"]), g, torch.bfloat16)
        st["W"] = _normal((case["V"], case["D"]), g, torch.bfloat16, scale=3.0 / math.sqrt(case["D"]))
    elif kind == "head":
        B, D, K, F = case["B"], case["D"], case["K"], case["F"]
        st["pooled"] = _normal((B, D), g, scale=0.25)  # a weighted mean of hidden states
        if F:
            lin = _linear_head(g, K, F)
            W1, b1 = _normal((F, D), g, scale=math.sqrt(2.0 / D)), _normal((F,), g, scale=0.1)
            _clear_kink(st["pooled"], W1, b1)
            st["head"] = estp.MlpHead(W1, b1, lin.W, lin.bias, lin.centers)
        else:
            st["head"] = _linear_head(g, K, D)
        st["targets"] = torch.empty(B, device=DEVICE).uniform_(1.0, K * BIN_WIDTH, generator=g)
    else:
        cu = _bounds(case)
        sumT = int(cu[-1])
        st["sumT"], st["max_T"] = sumT, int(_lengths(case).max())
        st["cu"] = torch.tensor(cu, dtype=torch.int32, device=DEVICE)
        if kind == "misalign":
            st["H"] = torch.empty(sumT, device=DEVICE).uniform_(0.0, 11.0, generator=g)
            st["S"] = _normal((sumT,), g).exp_().mul_(1e-3)
        elif kind == "features":
            st["logits"] = _logits(case, g, sumT)
            st["qk"] = [_qk(case, g, sumT) for _ in range(case["layers"])]
            st["hidden"] = _normal((sumT, case["D"]), g, _dtype(case))
            st["head"] = _linear_head(g, case["K"], case["D"])
        else:
            st["Q"], st["K"] = _qk(case, g, sumT)
            if kind == "forward":
                st["V"] = _normal((sumT, case["Hkv"], case["d"]), g, torch.bfloat16)
            if case["lse_given"]:
                st["lse"] = _row_normalisers(case, st["Q"], st["K"], torch.float32)
    st["ctx"] = estp.Context(0)
    return st


# ------------------------------------------------------------------------- calls
def run(st):
    case, ctx = st["case"], st["ctx"]
    kind = case["kind"]
    if kind == "lm_head":
        return ctx.lm_head_entropy(st["hidden"], st["W"])
    if kind == "head":
        if case["F"]:
            return list(ctx.mlp_head_loss(st["pooled"], st["head"], st["targets"], LAMBDA3))
        return list(ctx.head_loss(st["pooled"], st["head"], st["targets"], LAMBDA3))
    cu, max_T, sumT = st["cu"], st["max_T"], st["sumT"]
    if kind == "misalign":
        return ctx.misalignment(st["H"], st["S"], cu, pct=case["pct"])
    if kind == "features":
        H = ctx.token_entropy(st["logits"], V=case["V"], cu_seqlens=cu)
        for n, (Q, K) in enumerate(st["qk"]):
            ctx.attn_importance(Q, K, cu, max_T, accumulate=n > 0)
        S = ctx.attn_importance_finalize(case["layers"], sumT)
        pooled, pred = ctx.pool(st["hidden"], H, S, cu, LAMBDA1, LAMBDA2, ALPHA, head=st["head"])
        return {"H": H, "S": S, "pooled": pooled, "pred": pred}
    if kind == "forward":
        O = ctx.attn_forward_importance(st["Q"], st["K"], st["V"], cu, max_T, lse=st.get("lse"))
        return {"O": O, "S": ctx.attn_importance_finalize(1, sumT)}
    lse = st.get("lse")
    out = {}
    if lse is None:
        lse = out["lse"] = ctx.attn_lse(st["Q"], st["K"], cu, max_T)
    ctx.attn_importance(st["Q"], st["K"], cu, max_T, lse=lse, heads=_heads(case),
                        exclude_self=case["exclude_self"], divisor=case["divisor"])
    out["S"] = ctx.attn_importance_finalize(1, sumT)
    return out


# -------------------------------------------------------------------------- work
def _esize(case):
    return 2 if case["dtype"] == "bf16" else 4


def work(case):
    """Each input read once and each output written once; operations of the definition
    (a multiply-add counts two)."""
    kind = case["kind"]
    if kind == "lm_head":
        r, D, V = case["rows"], case["D"], case["V"]
        return {"bytes": 2 * D * (r + V) + 4 * r, "flops": 2 * r * D * V}
    if kind == "head":
        B, D, K, F = case["B"], case["D"], case["K"], case["F"]
        n_in = B * D + B + K  # pooled, targets, centres
        weights = F * D + F + K * F + K if F else K * D + K
        # forward, weight gradient and input gradient of each layer
        flops = 6 * B * (F * D + K * F) if F else 6 * B * K * D
        return {"bytes": 4 * (n_in + 2 * weights + B * D + 1), "flops": flops}
    T = _lengths(case).astype(np.float64)
    sumT = float(T.sum())
    if kind == "misalign":
        return {"bytes": int(8 * sumT + 12 * case["B"]), "flops": int(8 * sumT)}
    es, Hq, Hkv, d = _esize(case), case["Hq"], case["Hkv"], case["d"]
    pairs = float((T * (T + 1) / 2).sum())
    qk_bytes = sumT * (Hq + Hkv) * d * es
    if kind == "features":
        D, K, V = case["D"], case["K"], case["V"]
        nbytes = (sumT * V * es + case["layers"] * qk_bytes + sumT * D * es + 8 * sumT
                  + 4 * (K * D + 2 * K + case["B"] * (D + 1)))
        flops = (case["layers"] * 2 * 2.0 * d * Hq * pairs + 4 * sumT * V + 2 * sumT * D
                 + 2 * case["B"] * K * D)
        return {"bytes": int(nbytes), "flops": int(flops)}
    if kind == "forward":
        nbytes = qk_bytes + sumT * (Hq + Hkv) * d * es + 4 * sumT
        nbytes += 4 * Hq * sumT if case["lse_given"] else 0
        passes = 2 if case["lse_given"] else 3  # row normalisers, scores, weighted values
        return {"bytes": int(nbytes), "flops": int(passes * 2.0 * d * Hq * pairs)}
    n = len(_heads(case) or range(Hq))
    nbytes = qk_bytes + 4 * Hq * sumT + 4 * sumT
    return {"bytes": int(nbytes),
            "flops": int(2.0 * d * pairs * (n if case["lse_given"] else Hq + n))}


def tolerance(case):
    """About four times the distance between this library and the 64-bit values."""
    kind = case["kind"]
    if kind == "misalign":
        return "exact"
    if kind == "forward":
        return {"rel": 1e-2}  # bf16 probabilities and output
    if kind == "lm_head":
        return {"rel": 4e-5}  # long products summed in the tensor cores' fp32 accumulators
    return {"rel": 1e-5}


# ------------------------------------------------------------------ 64-bit values
def _softmax_entropy(z):
    logp = torch.log_softmax(z, dim=1)
    return -(logp.exp() * logp).sum(dim=1)


def _exact_column_sums(case, Q, K, heads, lse=None, V=None):
    """(column sums [sumT], attention output or None), fp64."""
    cu, rep, scale = _bounds(case), case["Hq"] // case["Hkv"], 1.0 / math.sqrt(case["d"])
    sumT = int(cu[-1])
    C = torch.zeros(sumT, dtype=torch.float64, device=DEVICE)
    O = None if V is None else torch.empty(sumT, case["Hq"], case["d"], dtype=torch.float64, device=DEVICE)
    for b in range(case["B"]):
        t0, T = int(cu[b]), int(cu[b + 1] - cu[b])
        for i0, i1 in _row_blocks(T):
            for h, s in _scores(Q, K, t0, i0, i1, heads, rep, scale, torch.float64):
                norm = torch.logsumexp(s, dim=1) if lse is None else lse[h, t0 + i0:t0 + i1].double()
                p = s.sub_(norm[:, None]).exp_()
                if V is not None:
                    O[t0 + i0:t0 + i1, h] = p @ V[t0:t0 + i1, h // rep].double()
                if case.get("exclude_self"):
                    p[torch.arange(i1 - i0, device=DEVICE), torch.arange(i0, i1, device=DEVICE)] = 0.0
                C[t0:t0 + i1] += p.sum(dim=0)
    return C, O


def _exact_importance(case, C, n_terms):
    cu = _bounds(case)
    out = C / n_terms
    for b in range(case["B"]):
        t0, t1 = int(cu[b]), int(cu[b + 1])
        div = case.get("divisor", "length")
        if div == "length":
            out[t0:t1] /= t1 - t0
        elif div == "causal":
            n = torch.arange(t1 - t0, 0, -1, device=DEVICE, dtype=torch.float64)
            n -= 1.0 if case["exclude_self"] else 0.0
            out[t0:t1] = torch.where(n > 0, out[t0:t1] / n.clamp(min=1.0), torch.zeros_like(n))
    return out


def _exact_head_loss(z, targets, centers):
    """(loss, dL/dz) of the logits z [B, K]."""
    B, K = z.shape
    p_hat = torch.softmax(z, dim=1)
    c = centers.double()
    r = z.argmax(dim=1)
    rel = c[None, :] - c[r][:, None]
    dy = (p_hat * rel).sum(dim=1, keepdim=True)
    err = c[r] + dy[:, 0] - targets.double()
    i = (targets[:, None] - centers[None, :]).abs().argmin(dim=1)
    p = torch.softmax(-(torch.arange(K, device=DEVICE)[None, :] - i[:, None]).abs().double(), dim=1)
    ce = -(p * torch.log_softmax(z, dim=1)).sum(dim=1)
    loss = LAMBDA3 * ce.mean() + (1 - LAMBDA3) * (err * err).mean()
    dz = (LAMBDA3 * (p_hat - p) + (1 - LAMBDA3) * 2 * err[:, None] * p_hat * (rel - dy)) / B
    return loss.reshape(1), dz


def _exact_misalignment(case, H, S):
    cu = _bounds(case)
    counts = torch.zeros(case["B"], 3, dtype=torch.int32)
    H, S = H.cpu(), S.cpu()
    for b in range(case["B"]):
        h, s = H[cu[b]:cu[b + 1]], S[cu[b]:cu[b + 1]]
        k = case["pct"] * h.numel() // 100

        def marks(x, descending):
            m = torch.zeros(x.numel(), dtype=torch.bool)
            m[torch.sort(x, stable=True, descending=descending).indices[:k]] = True
            return m

        counts[b, 0] = k
        counts[b, 1] = int((marks(h, True) & marks(s, False)).sum())
        counts[b, 2] = int((marks(h, False) & marks(s, True)).sum())
    return counts.to(DEVICE)


def exact(case, seed):
    kind = case["kind"]
    st = prepare(case, seed)
    st.pop("ctx").close()
    if kind == "misalign":
        return _exact_misalignment(case, st["H"], st["S"])
    if kind == "lm_head":
        W = st["W"].double()
        return torch.cat([_softmax_entropy(h.double() @ W.T) for h in st["hidden"].split(1024)])
    if kind == "head":
        x, hd = st["pooled"].double(), st["head"]
        if not case["F"]:
            W = hd.W.double()
            loss, dz = _exact_head_loss(x @ W.T + hd.bias.double(), st["targets"], hd.centers)
            return [loss, dz.T @ x, dz.sum(dim=0), dz @ W]
        W1, W2 = hd.W1.double(), hd.W2.double()
        u = (x @ W1.T + hd.b1.double()).clamp_(min=0.0)
        loss, dz = _exact_head_loss(u @ W2.T + hd.b2.double(), st["targets"], hd.centers)
        du = (dz @ W2) * (u > 0)
        return [loss, du.T @ x, du.sum(dim=0), dz.T @ u, dz.sum(dim=0), du @ W1]
    if kind == "features":
        H = torch.cat([_softmax_entropy(z[:, :case["V"]].double()) for z in st["logits"].split(1024)])
        C = torch.zeros(st["sumT"], dtype=torch.float64, device=DEVICE)
        for Q, K in st["qk"]:
            C += _exact_column_sums(case, Q, K, range(case["Hq"]))[0]
        S = _exact_importance(case, C, case["layers"] * case["Hq"])
        cu, hd = _bounds(case), st["head"]
        mix = (LAMBDA1 * S + LAMBDA2 * H) / ALPHA
        pooled = torch.stack([torch.softmax(mix[cu[b]:cu[b + 1]], dim=0) @ st["hidden"][cu[b]:cu[b + 1]].double()
                              for b in range(case["B"])])
        p = torch.softmax(pooled @ hd.W.double().T + hd.bias.double(), dim=1)
        return {"H": H, "S": S, "pooled": pooled, "pred": p @ hd.centers.double()}
    if kind == "forward":
        C, O = _exact_column_sums(case, st["Q"], st["K"], range(case["Hq"]), st.get("lse"), st["V"])
        return {"O": O, "S": _exact_importance(case, C, case["Hq"])}
    heads = _heads(case) or range(case["Hq"])
    pairs = float((_lengths(case).astype(np.float64) ** 2).sum()) * case["Hq"]
    if pairs > 3.2e10:  # the rollout batch: more than about 20 seconds in 64 bits
        return None
    out = {}
    lse = st.get("lse")
    if lse is None:
        lse = out["lse"] = _row_normalisers(case, st["Q"], st["K"], torch.float64)
    C, _ = _exact_column_sums(case, st["Q"], st["K"], heads, lse)
    out["S"] = _exact_importance(case, C, len(heads))
    return out
