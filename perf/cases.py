"""The workloads by which the library's speed is measured.

Each case is one pass through a public entry point of
``paper_2602_07160_gb300.fem``, as a program calls it.  ``listed`` names them,
``draw`` gives further ones of the same ranges, ``prepare`` makes what the
caller has in hand (on the GPU, from the seed alone), ``run`` makes the pass,
``work`` counts what the pass cannot do without and ``exact`` evaluates the
definitions in 64 bits with plain torch.
"""
from __future__ import annotations

import math

import torch

from paper_2602_07160_gb300 import fem

EXACT_MAX_FLOPS = 9.0e12  # beyond this the 64-bit evaluation is left out
LARGEST_FLOPS = 8.8e12    # the longest listed read; drawn cases stay below


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
def _read(name, B, H, T, d, causal, beta=(0.05, 20.0), v="normal", const=0):
    return {"name": name, "kind": "read", "B": B, "H": H, "T": T, "d": d, "causal": causal, "beta_lo": beta[0],
            "beta_hi": beta[1], "v": v, "const": const}


def listed():
    return [
        # the smallest call: one short fp32 sequence, where the launch and one row's latency count
        {"name": "f32_tiny", "kind": "f32", "B": 1, "H": 1, "T": 64, "d": 16, "causal": True},
        # an image transformer's layer (ViT-S/16: 197 tokens, a ragged second tile; no mask)
        _read("read_vit_s", 64, 6, 197, 64, False),
        # a language model's layer at a training context, narrow heads
        _read("read_lm_d64", 8, 12, 2048, 64, True),
        # the same with wide heads at a long context: the headline read
        _read("read_lm_d128", 4, 16, 8192, 128, True),
        # the longest context, heavy-tailed values and constant channels: one sequence's prefill
        _read("read_long_student_t", 1, 32, 32768, 128, True, (1e-3, 100.0), "student_t3", 4),
        # the mixer's full layer (inner and outer gate) of a hidden-512, 4-head model at context 2K
        {"name": "gated_lm", "kind": "gated", "B": 4, "H": 4, "T": 2048, "d": 128, "causal": True},
        # one generated token against a short cache, batch 1 of a 12-head model: latency
        {"name": "decode_one", "kind": "decode", "B": 1, "H": 12, "T": 1000, "d": 64},
        # one generated token for a batch against a long cache: the cache's bytes
        {"name": "decode_long", "kind": "decode", "B": 4, "H": 16, "T": 8192, "d": 128},
        # an fp32 training step's share: the read and its gradients
        {"name": "train_f32", "kind": "train", "B": 1, "H": 4, "T": 2048, "d": 64, "causal": True},
        # the read over a gated-linear-attention prior in fp32 (the hidden-512, 4-head model's layer)
        {"name": "gla_f32", "kind": "gla", "B": 4, "H": 4, "T": 2048, "m": 64, "d": 128},
        # the same prior at a long context on the tensor cores
        {"name": "gla_tc_long", "kind": "gla_tc", "B": 4, "H": 16, "T": 8192, "m": 64, "d": 64},
        # the time-decay conditioner in front of the read's gates
        {"name": "tdc", "kind": "tdc", "B": 4, "T": 8192, "Hc": 64},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _heads(rng, limit):
    """Batch and heads with B * H <= limit."""
    H = min(rng.choice([1, 2, 4, 6, 8, 12, 16, 32]), max(1, int(limit)))
    return _log_int(rng, 1, max(1, min(64, int(limit) // H))), H


def draw(rng):
    kind = rng.choice(["read", "read", "read", "read", "gated", "decode", "decode", "f32", "train", "gla", "gla_tc",
                       "tdc"])
    if kind in ("read", "gated"):
        T, d, causal = _log_int(rng, 17, 24000), rng.choice([64, 64, 128, 128]), rng.random() < 0.7
        pairs_flops = 4.0 * T * T * d * (0.5 if causal else 1.0) * (2 if kind == "gated" else 1)
        B, H = _heads(rng, min(384, LARGEST_FLOPS / 4 / pairs_flops, 8.0e8 / (T * d)))
        c = {"kind": kind, "B": B, "H": H, "T": T, "d": d, "causal": causal}
        if kind == "read":
            heavy = rng.random() < 0.2
            c.update({"beta_lo": 1e-3 if heavy else 0.05, "beta_hi": 100.0 if heavy else 20.0,
                      "v": "student_t3" if heavy else "normal", "const": 4 if heavy else 0})
        return c
    if kind == "decode":
        T, d = _log_int(rng, 1, 32768), rng.choice([64, 128])
        B, H = _heads(rng, min(512, 6.7e7 / (T * d)))
        return {"kind": kind, "B": B, "H": H, "T": T, "d": d}
    if kind in ("f32", "train"):
        T, d, causal = _log_int(rng, 5, 2048), rng.choice([16, 32, 48, 64, 128]), rng.random() < 0.7
        B, H = _heads(rng, min(64, 4.0 * 2048 * 2048 * 64 / (T * T * d)))
        return {"kind": kind, "B": B, "H": H, "T": T, "d": d, "causal": causal}
    if kind in ("gla", "gla_tc"):
        T = _log_int(rng, 5, 8192)
        m, d = (64, 64) if kind == "gla_tc" else (rng.choice([16, 32, 64]), rng.choice([24, 32, 64, 100, 128]))
        B, H = _heads(rng, min(128, (3.4e7 if kind == "gla_tc" else 1.0e7) / (T * d)))
        return {"kind": kind, "B": B, "H": H, "T": T, "m": m, "d": d}
    return {"kind": "tdc", "B": _log_int(rng, 1, 8), "T": _log_int(rng, 5, 20000), "Hc": _log_int(rng, 8, 300)}


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _inputs(case, seed):
    """The pass's tensors on the GPU, drawn in a fixed order from one generator."""
    dev = torch.device("cuda", torch.cuda.current_device())
    g = torch.Generator(device=dev).manual_seed(int(seed))

    def normal(*shape):
        return torch.randn(shape, generator=g, device=dev)

    def log_uniform(H, d, lo, hi):
        u = torch.rand((H, d), generator=g, device=dev, dtype=torch.float64)
        return torch.exp(math.log(lo) + u * math.log(hi / lo)).float()

    kind, B, T = case["kind"], case["B"], case["T"]
    if kind == "tdc":
        # softplus rates around a decay over some tens of steps
        s = 0.05 * torch.nn.functional.softplus(normal(B, T, case["Hc"]))
        return {"s": s, "u": normal(B, T, case["Hc"])}
    H, d = case["H"], case["d"]
    if kind in ("gla", "gla_tc"):
        m = case["m"]
        return {"qf": torch.relu(normal(B, H, T, m)) + 0.05, "kf": torch.relu(normal(B, H, T, m)) + 0.05,
                "v": normal(B, H, T, d), "logdecay": -0.3 * torch.rand((B, H, T), generator=g, device=dev),
                "beta": log_uniform(H, d, 0.05, 20.0)}
    dt = torch.float32 if kind in ("f32", "train") else torch.bfloat16
    q = normal(B, H, d) if kind == "decode" else normal(B, H, T, d)
    x = {"q": q.to(dt), "k": normal(B, H, T, d).to(dt)}
    v = normal(B, H, T, d)
    if case.get("v") == "student_t3":  # t with three degrees of freedom, scaled to unit variance
        chi2 = normal(B, H, T, d).square_()
        for _ in range(2):
            chi2 += normal(B, H, T, d).square_()
        v = v.div_(chi2.div_(3.0).sqrt_()).div_(math.sqrt(3.0))
    if case.get("const"):  # channels that hold one value over the whole sequence
        v[..., :case["const"]] = v[:, :, :1, :case["const"]].clone()
    x["v"] = v.to(dt)
    x["beta"] = log_uniform(H, d, case.get("beta_lo", 0.05), case.get("beta_hi", 20.0))
    if kind == "gated":
        x["lam"] = torch.sigmoid(2.0 * normal(B, H, T, d))
        x["gate"] = torch.nn.functional.softplus(normal(B, H, T, d))
    if kind == "train":
        x["dout"] = normal(B, H, T, d)
    return x


def prepare(case, seed):
    return {"case": case, "x": _inputs(case, seed)}


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def run(state):
    case, x = state["case"], state["x"]
    kind = case["kind"]
    if kind == "read":
        return fem.fem_fwd(x["q"], x["k"], x["v"], x["beta"], causal=case["causal"])
    if kind == "gated":
        return fem.fem_fwd_gated(x["q"], x["k"], x["v"], x["beta"], x["lam"], x["gate"], causal=case["causal"])
    if kind == "decode":
        return fem.fem_decode(x["q"], x["k"], x["v"], x["beta"])
    if kind == "f32":
        return fem.fem_fwd_f32(x["q"], x["k"], x["v"], x["beta"], causal=case["causal"])
    if kind == "train":
        out, lse = fem.fem_fwd_f32(x["q"], x["k"], x["v"], x["beta"], causal=case["causal"])
        grads = fem.fem_bwd_f32(x["q"], x["k"], x["v"], x["beta"], out, lse, x["dout"], causal=case["causal"])
        return (out, lse) + tuple(grads)
    if kind == "gla":
        return fem.fem_gla_fwd(x["qf"], x["kf"], x["v"], x["logdecay"], x["beta"])
    if kind == "gla_tc":
        return fem.fem_gla_fwd_tc(x["qf"], x["kf"], x["v"], x["logdecay"], x["beta"])
    if kind == "tdc":
        return fem.fem_tdc_conv(x["s"], x["u"])
    raise ValueError(kind)


def _pairs(case):
    T = case["T"]
    return T * (T + 1) / 2 if case["causal"] else float(T) * T


def work(case):
    kind, B, T = case["kind"], case["B"], case["T"]
    if kind == "tdc":
        n = float(B * T * case["Hc"])
        return {"bytes": 12.0 * n, "flops": 2.0 * n}  # s, u in, h out; one multiply-add a step
    BH, d = B * case["H"], case["d"]
    n, rows, nb = float(BH * T * d), float(BH * T), 4.0 * case["H"] * d
    if kind == "read":  # q, k, v in, out and lse out; two contractions over the visible pairs
        return {"bytes": 10.0 * n + 4.0 * rows + nb, "flops": 4.0 * BH * _pairs(case) * d}
    if kind == "gated":  # the gates as well; the prior weights meet two banks
        return {"bytes": 18.0 * n + 4.0 * rows + nb, "flops": 6.0 * BH * _pairs(case) * d}
    if kind == "decode":
        return {"bytes": 4.0 * n + BH * (6.0 * d + 4.0) + nb, "flops": 4.0 * n}
    if kind == "f32":
        return {"bytes": 16.0 * n + 4.0 * rows + nb, "flops": 4.0 * BH * _pairs(case) * d}
    if kind == "train":  # q, k, v, dout in, out, lse and the gradients out; two contractions, then five
        return {"bytes": 32.0 * n + 4.0 * rows + 2.0 * nb, "flops": 14.0 * BH * _pairs(case) * d}
    m = case["m"]  # gla: the recurrence's state update and read, the value channels and the normaliser
    return {"bytes": rows * (8.0 * m + 8.0 * d + 8.0) + nb, "flops": 4.0 * rows * m * (d + 1)}


# ---------------------------------------------------------------------------
# the definitions in 64 bits
# ---------------------------------------------------------------------------
TILE = 128


def _lse_tiles(scores, before, within, v, beta, T, causal):
    """For every row t of [N, T]: log sum_i w_ti and, per channel, log sum_i w_ti exp(beta v_i).

    ``before(t0, t1)`` gives the log-weights [N, t1 - t0, t0] of rows t0..t1-1 on the keys before
    t0, ``within(t0, t1)`` those on the keys t0..t1-1 (causal: -inf above the diagonal).  Keys
    before the tile are contracted around the largest beta v before it; keys of the row's own tile
    are summed one by one, each row around its own largest term, so that nothing underflows that a
    row could need.  Without a mask all keys are contracted at once."""
    N, d = v.shape[0], v.shape[2]
    bv = beta[:, None, :] * v  # [N, T, d]
    num = torch.empty((N, T, d), dtype=torch.float64, device=v.device)
    den = torch.empty((N, T), dtype=torch.float64, device=v.device)
    for t0 in range(0, T, TILE):
        t1 = min(T, t0 + TILE)
        la = lz = None
        n = t0 if causal else T
        if n:
            w = scores(t0, t1) if not causal else before(t0, t1)
            top = w.amax(-1, keepdim=True)
            w = torch.exp(w - top)
            c = bv[:, :n].amax(1, keepdim=True)
            la = torch.log(torch.bmm(w, torch.exp(bv[:, :n] - c))) + c + top
            lz = torch.log(w.sum(-1)) + top[..., 0]
            del w
        if causal:
            w = within(t0, t1)
            own = torch.empty((N, t1 - t0, d), dtype=torch.float64, device=v.device)
            step = max(1, (1 << 27) // (TILE * TILE * d))
            for a in range(0, N, step):
                b = min(N, a + step)
                own[a:b] = torch.logsumexp(w[a:b, :, :, None] + bv[a:b, None, t0:t1, :], dim=2)
            lw = torch.logsumexp(w, dim=-1)
            la = own if la is None else torch.logaddexp(la, own)
            lz = lw if lz is None else torch.logaddexp(lz, lw)
        num[:, t0:t1] = la
        den[:, t0:t1] = lz
    return num, den


def _exact_softmax(q, k, v, beta, causal):
    """(out, lse) of the read with a softmax prior; q, k, v [B, H, T, d], beta [H, d], all float64."""
    B, H, T, d = v.shape
    q, k, v = (a.reshape(B * H, -1, d) for a in (q, k, v))
    bb = beta.repeat(B, 1)
    mask = torch.full((TILE, TILE), -math.inf, dtype=torch.float64, device=v.device).triu(1)

    def score(t0, t1, i0, i1):
        return torch.bmm(q[:, t0:t1], k[:, i0:i1].transpose(1, 2)) / math.sqrt(d)

    num, den = _lse_tiles(lambda a, b: score(a, b, 0, T), lambda a, b: score(a, b, 0, a),
                          lambda a, b: score(a, b, a, b) + mask[:b - a, :b - a], v, bb, T, causal)
    out = (num - den[..., None]) / bb[:, None, :]
    return out.reshape(B, H, T, d), den.reshape(B, H, T)


def _exact_gla(x):
    qf, kf, v, g, beta = (x[n].double() for n in ("qf", "kf", "v", "logdecay", "beta"))
    B, H, T, d = v.shape
    qf, kf, v = (a.reshape(B * H, T, -1) for a in (qf, kf, v))
    G = g.reshape(B * H, T).cumsum(-1)
    bb = beta.repeat(B, 1)
    mask = torch.full((TILE, TILE), -math.inf, dtype=torch.float64, device=v.device).triu(1)

    def weight(t0, t1, i0, i1):
        return torch.log(torch.bmm(qf[:, t0:t1], kf[:, i0:i1].transpose(1, 2))) + (G[:, t0:t1, None] - G[:, None, i0:i1])

    num, den = _lse_tiles(None, lambda a, b: weight(a, b, 0, a),
                          lambda a, b: weight(a, b, a, b) + mask[:b - a, :b - a], v, bb, T, True)
    out = (num - den[..., None]) / bb[:, None, :]
    return out.reshape(B, H, T, d), den.reshape(B, H, T)


def _exact_grads(x, out, lse, causal):
    """Gradients of the read: the posterior p e^x with x = beta (v - o), pair by pair."""
    q, k, v, beta, dout = (x[n].double() for n in ("q", "k", "v", "beta", "dout"))
    B, H, T, d = v.shape
    dq, dk, dv = torch.zeros_like(q), torch.zeros_like(k), torch.zeros_like(v)
    dbeta = torch.zeros_like(beta)
    rows = max(1, min(T, (1 << 25) // max(1, T * d)))
    for b in range(B):
        for h in range(H):
            bj = beta[h]
            for t0 in range(0, T, rows):
                t1 = min(T, t0 + rows)
                n = t1 if causal else T
                s = q[b, h, t0:t1] @ k[b, h, :n].T / math.sqrt(d)
                p = torch.exp(s - lse[b, h, t0:t1, None])
                if causal:
                    p = p.tril(t0)
                y = v[b, h, None, :n] - out[b, h, t0:t1, None]  # [rows, n, d]
                xx = bj * y
                go = dout[b, h, t0:t1, None] * p[..., None]
                e1 = torch.expm1(xx)
                ds = (go * e1 / bj).sum(-1) / math.sqrt(d)
                dq[b, h, t0:t1] = ds @ k[b, h, :n]
                dk[b, h, :n] += ds.T @ q[b, h, t0:t1]
                dv[b, h, :n] += (go * (e1 + 1.0)).sum(0)
                dbeta[h] += (go * (xx * (e1 + 1.0) - e1) / (bj * bj)).sum((0, 1))
    return dq, dk, dv, dbeta


def exact(case, seed):
    if work(case)["flops"] > EXACT_MAX_FLOPS:
        return None
    x, kind = _inputs(case, seed), case["kind"]
    if kind == "tdc":
        s, u = x["s"].double(), x["u"].double()
        a, h = torch.exp(-s), torch.empty_like(u)
        run_h = torch.zeros_like(u[:, 0])
        for t in range(case["T"]):
            run_h = a[:, t] * run_h + u[:, t]
            h[:, t] = run_h
        return h
    if kind in ("gla", "gla_tc"):
        return _exact_gla(x)
    q, k, v, beta = (x[n].double() for n in ("q", "k", "v", "beta"))
    if kind == "decode":
        return _exact_decode(q, k, v, beta)
    out, lse = _exact_softmax(q, k, v, beta, case["causal"])
    if kind == "gated":
        s = _exact_mean(q, k, v, lse, case["causal"])
        lam, gate = x["lam"].double(), x["gate"].double()
        return gate * ((1.0 - lam) * s + lam * out), lse
    if kind == "train":
        return (out, lse) + _exact_grads(x, out, lse, case["causal"])
    return out, lse


def _exact_decode(q, k, v, beta):
    s = torch.einsum("bhd,bhtd->bht", q, k) / math.sqrt(q.shape[-1])
    lse = torch.logsumexp(s, -1)
    out = torch.logsumexp(s[..., None] + beta[None, :, None, :] * v, dim=2)
    return (out - lse[..., None]) / beta, lse


def _exact_mean(q, k, v, lse, causal):
    """The prior mean sum_i p_t(i) v_i, tile by tile of rows."""
    B, H, T, d = v.shape
    mu = torch.empty_like(v)
    for t0 in range(0, T, TILE):
        t1 = min(T, t0 + TILE)
        n = t1 if causal else T
        p = torch.exp(q[:, :, t0:t1] @ k[:, :, :n].transpose(2, 3) / math.sqrt(d) - lse[:, :, t0:t1, None])
        mu[:, :, t0:t1] = (p.tril(t0) if causal else p) @ v[:, :, :n]
    return mu
