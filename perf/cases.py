"""Performance cases of the candidate-scoring framework.

Every case is one call (or one chain of calls) that a program scoring
candidate answers makes through the public entry points: the teacher-forced
step itself (:class:`ScoringStep`), its parts (shared-prefix attention, the
fork of the recurrent state, the LM head in its weight formats), the prefill
that comes before it (causal attention, the scan of the recurrent state) and
the hybrid decoder stack (:class:`DecoderStack`).

A case holds the batch structure as plain values: ``requests`` contexts of
``prefix_lo`` to ``prefix_hi`` tokens with ``cands`` candidates of 1 to
``len_hi`` tokens, drawn from ``shape_seed`` (so the work of a case does not
depend on the seed of its inputs), and the model dimensions the call needs.
Tensors are drawn on the GPU from the seed given to :func:`prepare`:
queries, keys, values and hidden states N(0, 1), LM-head weights N(0, 0.02^2),
unit-norm linear-attention keys, decays in [0.9, 1) and write strengths in
[0, 1).
"""
import math

import numpy as np
import torch

_SHAPES = ("requests", "prefix_lo", "prefix_hi", "cands", "len_hi", "shape_seed")


def _case(name, op, requests, prefix_lo, prefix_hi, cands, len_hi, **model):
    c = dict(name=name, op=op, requests=requests, prefix_lo=prefix_lo, prefix_hi=prefix_hi,
             cands=cands, len_hi=len_hi, shape_seed=7)
    c.update(model)
    return c


def listed():
    wide = dict(Hq=24, Hkv=4, d=256)   # heads of the multiple-choice and yes/no batches
    slim = dict(Hq=16, Hkv=2, d=256)   # heads of the hybrid and the long-context batches
    rec = dict(Hl=16, dk=128, dv=128)
    V = 151936
    return [
        # one small float32 request: an interactive call, all launches and latency
        _case("step_tiny_f32", "step", 1, 128, 128, 4, 4, dtype="f32", Hq=8, Hkv=2, d=64, D=512,
              V=8192, mode="argmax"),
        # a large batch over long contexts: the whole step (attention, LM head,
        # decision) of a throughput-bound scorer
        _case("step_long", "step", 256, 2048, 8192, 4, 12, dtype="bf16", D=2048, V=V,
              mode="argmax", **slim),
        # one long context with its answers: attention at batch 1
        _case("attend_single", "attend", 1, 6000, 6000, 4, 12, dtype="bf16", **slim),
        # a batch of multiple-choice questions: attention over short, ragged prefixes
        _case("attend_choice", "attend", 16, 200, 1200, 4, 12, dtype="bf16", **wide),
        # the prefill of the same questions
        _case("prefill_choice", "prefill", 16, 200, 1200, 4, 12, dtype="bf16", **wide),
        # the prefill of a few long contexts
        _case("prefill_long", "prefill", 16, 2048, 8192, 4, 12, dtype="bf16", **slim),
        # the prefix scan of a hybrid model's recurrent layer (ratings: 512-token contexts)
        _case("scan_hybrid", "scan", 32, 512, 512, 10, 3, dtype="bf16", rule="delta", **rec),
        # ten candidates forked from every context's recurrent state, states kept
        _case("fork_hybrid", "fork", 32, 512, 512, 10, 3, dtype="bf16", rule="delta", **rec),
        # the LM head over a small batch: the weights' stream bounds it
        _case("head_choice", "head", 16, 200, 1200, 4, 12, dtype="bf16", D=5120, V=V, lm="bf16"),
        # the LM head over a few hundred rows: the tensor cores bound it
        _case("head_rating", "head", 32, 512, 512, 10, 3, dtype="bf16", D=4096, V=V, lm="bf16"),
        # the small batch over 4-bit weights, as a memory-limited deployment runs it
        _case("head_choice_w4", "head", 16, 200, 1200, 4, 12, dtype="bf16", D=5120, V=V, lm="w4"),
        # four decoder layers (three linear, one full) over the rating batch's rows
        _case("stack_hybrid", "stack", 32, 512, 512, 10, 3, dtype="bf16", D=4096, Dff=12288,
              linear=3, full=1, rule="delta", **slim, **rec),
    ]


# --------------------------------------------------------------------------
# drawn cases: the ranges the listed ones stand for
# --------------------------------------------------------------------------
def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _batch(rng, tokens, r_hi=256, p_lo=64, p_hi=8192):
    """requests and prefix range with about ``tokens`` prefix tokens at most."""
    hi = _log(rng, p_lo, p_hi)
    lo = hi if rng.random() < 0.25 else max(1, int(hi * rng.uniform(0.2, 0.9)))
    r = _log(rng, 1, max(1, min(r_hi, tokens // hi)))
    kind = rng.choice(("choice", "yesno", "rating"))
    cands = {"choice": rng.randint(3, 5), "yesno": 2, "rating": rng.randint(5, 10)}[kind]
    len_hi = {"choice": rng.randint(4, 12), "yesno": 2, "rating": 3}[kind]
    mode = {"choice": "argmax", "yesno": "binary", "rating": "ordinal"}[kind]
    return dict(requests=r, prefix_lo=lo, prefix_hi=hi, cands=cands, len_hi=len_hi,
                shape_seed=rng.randrange(1, 1 << 20)), mode


def _heads(rng):
    Hq, Hkv = rng.choice(((8, 2), (16, 2), (24, 4), (32, 8)))
    return dict(Hq=Hq, Hkv=Hkv, d=rng.choice((64, 128, 256, 256)))


def draw(rng):
    op = rng.choice(("step", "attend", "attend", "prefill", "prefill", "scan", "fork", "head",
                     "head", "stack"))
    if op == "step" and rng.random() < 0.25:  # small float32 batches
        b, mode = _batch(rng, 4096, r_hi=8, p_hi=1024)
        return dict(b, op=op, dtype="f32", D=rng.choice((512, 1024)), V=_log(rng, 4096, 32000),
                    mode=mode, **_heads(rng))
    if op in ("step", "attend"):
        h = _heads(rng)
        b, mode = _batch(rng, 1100000 * 512 // (h["Hkv"] * h["d"]))
        c = dict(b, op=op, dtype="bf16", **h)
        if op == "step":
            c.update(D=rng.choice((1024, 2048, 4096, 5120)), mode=mode,
                     V=_log(rng, 8192, 151936))
            rows = c["requests"] * (1 + c["cands"] * c["len_hi"])
            if rows * c["D"] > 4096 * 2048:  # no more head work than the long batch
                c["requests"] = max(1, c["requests"] * 4096 * 2048 // (rows * c["D"]))
        return c
    if op == "prefill":
        h = _heads(rng)
        b, _ = _batch(rng, 60000)
        while 2.0 * h["Hq"] * h["d"] * b["requests"] * b["prefix_hi"] ** 2 > 3e12:
            b["requests"] = b["requests"] // 2
            if b["requests"] == 0:
                b["requests"], b["prefix_hi"] = 1, 4000
                b["prefix_lo"] = min(b["prefix_lo"], 4000)
        return dict(b, op=op, dtype="bf16", **h)
    rule = rng.choice(("delta", "delta", "gla"))
    if op == "scan":
        Hl = rng.choice((8, 16, 32))
        b, _ = _batch(rng, 16384 * 16 // Hl, r_hi=64, p_hi=4096)
        return dict(b, op=op, dtype="bf16", rule=rule, Hl=Hl, dk=128, dv=128)
    if op == "fork":
        Hl = rng.choice((8, 16, 32))
        b, _ = _batch(rng, 1 << 20, r_hi=512 // Hl)
        return dict(b, op=op, dtype="bf16", rule=rule, Hl=Hl, dk=128, dv=128)
    if op == "head":
        b, _ = _batch(rng, 1 << 20, r_hi=64, p_hi=1024)
        return dict(b, op=op, dtype="bf16", D=rng.choice((1024, 2048, 4096, 5120)),
                    V=_log(rng, 32000, 151936), lm=rng.choice(("bf16", "bf16", "e4m3", "w4",
                                                               "mxfp8")))
    b, _ = _batch(rng, 32768, r_hi=32, p_hi=1024)
    D = rng.choice((1024, 2048, 4096))
    return dict(b, op=op, dtype="bf16", D=D, Dff=3 * D, linear=rng.randint(0, 3),
                full=1, rule=rule, Hq=16, Hkv=2, d=256 if D == 4096 else 128, Hl=D // 256,
                dk=128, dv=128)


# --------------------------------------------------------------------------
# batch structure and inputs
# --------------------------------------------------------------------------
def _shape(case):
    """Prefix lengths, candidate counts and candidate lengths of the batch."""
    g = np.random.default_rng(case["shape_seed"])
    R, C = case["requests"], case["cands"]
    P = g.integers(case["prefix_lo"], case["prefix_hi"] + 1, size=R)
    # mostly short answers, the longest len_hi tokens (geometric, truncated)
    k = np.arange(1, case["len_hi"] + 1)
    w = 0.7 ** (k - 1) if case["len_hi"] > 3 else np.ones(len(k))
    m = g.choice(k, size=R * C, p=w / w.sum())
    return P.astype(np.int32), np.full(R, C, np.int32), m.astype(np.int32)


def _counts(case):
    P, n_cand, m = _shape(case)
    R, C = len(P), len(m)
    F = int((m - 1).sum())
    rows = np.array([1 + int((m[r * case["cands"]:(r + 1) * case["cands"]] - 1).sum())
                     for r in range(R)])
    return dict(P=P, m=m, rows=rows, R=R, C=C, F=F, N=R + F, T=int(m.sum()), S=int(P.sum()))


class _Draw:
    """Tensors drawn one after the other from one seeded generator on the GPU."""

    def __init__(self, seed, dtype):
        self.g = torch.Generator(device="cuda").manual_seed(int(seed) + 1)
        self.dt = torch.bfloat16 if dtype == "bf16" else torch.float32

    def normal(self, *shape, std=1.0, dtype=None):
        x = torch.empty(shape, device="cuda", dtype=dtype or self.dt)
        return x.normal_(0.0, std, generator=self.g)

    def uniform(self, lo, hi, *shape):
        x = torch.empty(shape, device="cuda", dtype=torch.float32)
        return x.uniform_(lo, hi, generator=self.g)

    def keys(self, *shape):
        x = self.normal(*shape, dtype=torch.float32)
        return (x / x.norm(dim=-1, keepdim=True)).to(self.dt)


def _attention_inputs(t, c, n):
    return dict(q=t.normal(n["N"], c["Hq"], c["d"]), k_pre=t.normal(n["S"], c["Hkv"], c["d"]),
                v_pre=t.normal(n["S"], c["Hkv"], c["d"]), k_cand=t.normal(n["F"], c["Hkv"], c["d"]),
                v_cand=t.normal(n["F"], c["Hkv"], c["d"]))


def _recurrent_inputs(t, c, rows):
    return dict(lq=t.normal(rows, c["Hl"], c["dk"]), lk=t.keys(rows, c["Hl"], c["dk"]),
                lv=t.normal(rows, c["Hl"], c["dv"]), alpha=t.uniform(0.9, 1.0, rows, c["Hl"]),
                beta=t.uniform(0.0, 1.0, rows, c["Hl"]))


def _stack_layers(t, c, n):
    D, Dff = c["D"], c["Dff"]
    layers = []
    for i in range(c["linear"] + c["full"]):
        full = i >= c["linear"]
        mix = ((c["Hq"] + 2 * c["Hkv"]) * c["d"] if full else
               c["Hl"] * (2 * c["dk"] + c["dv"]) + 2 * c["Hl"])
        width = c["Hq"] * c["d"] if full else c["Hl"] * c["dv"]
        w = dict(kind="full" if full else "linear",
                 g1=t.normal(D, std=0.1).add_(1.0), g2=t.normal(D, std=0.1).add_(1.0),
                 w_mix=t.normal(mix, D, std=D ** -0.5), w_o=t.normal(D, width, std=width ** -0.5),
                 w_gu=t.normal(2 * Dff, D, std=D ** -0.5), w_d=t.normal(D, Dff, std=Dff ** -0.5))
        if full:
            w.update(k_pre=t.normal(n["S"], c["Hkv"], c["d"]),
                     v_pre=t.normal(n["S"], c["Hkv"], c["d"]))
        else:
            w.update(s_prefix=t.normal(n["R"], c["Hl"], c["dk"], c["dv"],
                                       std=c["dk"] ** -0.5, dtype=torch.float32))
        layers.append(w)
    return layers


def _inputs(case, seed):
    """The batch's target ids and every tensor of the call, from the seed alone."""
    c, n = case, _counts(case)
    t = _Draw(seed, c["dtype"])
    x = dict(n=n)
    if "V" in c:
        x["ids"] = np.random.default_rng(int(seed)).integers(0, c["V"], n["T"]).astype(np.int32)
    else:
        x["ids"] = np.zeros(n["T"], np.int32)
    if c["op"] in ("step", "attend"):
        x.update(_attention_inputs(t, c, n))
    if c["op"] in ("step", "head"):
        std = 0.02 if c["dtype"] == "bf16" else c["D"] ** -0.5
        x.update(hidden=t.normal(n["N"], c["D"]), w_lm=t.normal(c["V"], c["D"], std=std))
    if c["op"] == "prefill":
        x.update(q=t.normal(n["S"], c["Hq"], c["d"]), k=t.normal(n["S"], c["Hkv"], c["d"]),
                 v=t.normal(n["S"], c["Hkv"], c["d"]))
    if c["op"] == "scan":
        x.update(_recurrent_inputs(t, c, n["S"]))
    if c["op"] == "fork":
        x.update(_recurrent_inputs(t, c, n["F"]))
        x["s_prefix"] = t.normal(n["R"], c["Hl"], c["dk"], c["dv"], std=c["dk"] ** -0.5,
                                 dtype=torch.float32)
    if c["op"] == "stack":
        x.update(layers=_stack_layers(t, c, n), x0=t.normal(n["N"], c["D"]))
    return x


def prepare(case, seed):
    from paper_2609_33874_gb300 import jet
    from paper_2609_33874_gb300 import step as S

    c, x = case, _inputs(case, seed)
    n = x["n"]
    P, n_cand, m = _shape(case)
    host = jet.jet_layout_build(P, n_cand, m, x["ids"], c.get("V", 1))
    dims = jet.make_dims(jet.DTYPE_BF16 if c["dtype"] == "bf16" else jet.DTYPE_F32,
                         **{k: c[k] for k in ("Hq", "Hkv", "d", "D", "Hl", "dk", "dv") if k in c})
    s = dict(case=c, x=x, dims=dims, jet=jet, host=host)
    dt = torch.bfloat16 if c["dtype"] == "bf16" else torch.float32

    def out(*shape, dtype=dt):
        return torch.empty(shape, device="cuda", dtype=dtype)

    if c["op"] == "step":
        s["step"] = S.ScoringStep(host, dims, jet.MODES[c["mode"]])
    elif c["op"] == "head":
        s["step"] = S.ScoringStep(host, dims, jet.DECIDE_ARGMAX, lm=c["lm"])
        pack = {"bf16": lambda w: w, "e4m3": S.quantize_lm_head, "w4": S.quantize_lm_head_w4,
                "mxfp8": S.quantize_lm_head_mxfp8}[c["lm"]]
        s["w"] = pack(x.pop("w_lm"))
    elif c["op"] == "stack":
        s["stack"] = S.DecoderStack(host, dims, x["layers"], c["Dff"], rule=c["rule"])
    else:
        s["layout"] = host.to_device()
        if c["op"] == "attend":
            s["o"] = out(n["N"], c["Hq"], c["d"])
            s["ws"] = out((jet.jet_workspace_bytes(host.sizes, dims) + 15) // 16 * 4,
                          dtype=torch.float32)
        elif c["op"] == "prefill":
            s["o"] = out(n["S"], c["Hq"], c["d"])
            s["ws"] = out((jet.jet_prefill_workspace_bytes(host.sizes, dims) + 15) // 16 * 4,
                          dtype=torch.float32)
        elif c["op"] == "scan":
            s["o"] = out(n["S"], c["Hl"], c["dv"])
            s["s"] = out(n["R"], c["Hl"], c["dk"], c["dv"], dtype=torch.float32)
        else:
            s["o"] = out(n["F"], c["Hl"], c["dv"])
            s["s"] = out(n["C"], c["Hl"], c["dk"], c["dv"], dtype=torch.float32)
    return s


def run(state):
    s = state
    c, x, jet = s["case"], s["x"], s["jet"]
    if c["op"] == "step":
        st = s["step"]
        st.run(x, x["w_lm"])
        return dict(o=st.o, tok_logprob=st.tok_logprob, cand_score=st.cand_score,
                    q_cand=st.q_cand, choice=st.choice, value=st.value)
    if c["op"] == "head":
        st = s["step"]
        st.score(x["hidden"], s["w"])
        return dict(tok_logprob=st.tok_logprob, cand_score=st.cand_score)
    if c["op"] == "stack":
        return dict(x=s["stack"].forward(x["x0"]))
    if c["op"] == "attend":
        jet.jet_prefix_attend(s["layout"], s["dims"], x["q"], x["k_pre"], x["v_pre"], x["k_cand"],
                              x["v_cand"], s["o"], s["ws"])
        return dict(o=s["o"])
    if c["op"] == "prefill":
        jet.jet_prefill_attend(s["layout"], s["dims"], x["q"], x["k"], x["v"], s["o"], s["ws"])
        return dict(o=s["o"])
    if c["op"] == "scan":
        jet.jet_prefill_state(s["layout"], s["dims"], x["lq"], x["lk"], x["lv"], x["alpha"],
                              x["beta"], s["o"], s["s"], rule=jet.RULES[c["rule"]])
        return dict(o=s["o"], s=s["s"])
    jet.jet_fork_state(s["layout"], s["dims"], x["s_prefix"], x["lq"], x["lk"], x["lv"],
                       x["alpha"], x["beta"], s["o"], s["s"], rule=jet.RULES[c["rule"]])
    return dict(o=s["o"], s=s["s"])


# --------------------------------------------------------------------------
# what a pass cannot do without
# --------------------------------------------------------------------------
def work(case):
    c, n = case, _counts(case)
    eb = 2 if c["dtype"] == "bf16" else 4
    by = fl = 0.0

    def attend():
        # prefix and candidate K/V once per request, queries in, outputs out
        b = eb * (2 * (n["S"] + n["F"]) * c["Hkv"] * c["d"] + 2 * n["N"] * c["Hq"] * c["d"])
        keys = float((n["rows"] * n["P"]).sum()) + sum(k * (k - 1) / 2.0 for k in n["m"].tolist())
        return b, 4.0 * c["Hq"] * c["d"] * keys

    def head(lm="bf16"):
        per = {"bf16": eb * c["D"], "e4m3": c["D"] + 4, "mxfp8": c["D"] + c["D"] / 32,
               "w4": c["D"] / 2 + c["D"] / 32 + 4}[lm]
        return (c["V"] * per + eb * n["N"] * c["D"] + 4 * (n["T"] + n["C"]),
                2.0 * n["N"] * c["D"] * c["V"])

    def recurrent(rows, states_in, states_out, rule):
        b = rows * c["Hl"] * ((2 * c["dk"] + 2 * c["dv"]) * eb + 8)
        b += 4.0 * (states_in + states_out) * c["Hl"] * c["dk"] * c["dv"]
        return b, (6.0 if rule == "delta" else 4.0) * rows * c["Hl"] * c["dk"] * c["dv"]

    if c["op"] == "step":
        for b, f in (attend(), head()):
            by, fl = by + b, fl + f
    elif c["op"] == "attend":
        by, fl = attend()
    elif c["op"] == "prefill":
        by = float(eb * n["S"] * c["d"] * (2 * c["Hq"] + 2 * c["Hkv"]))
        P = n["P"].astype(np.float64)
        fl = float(4.0 * c["Hq"] * c["d"] * (P * (P + 1) / 2).sum())
    elif c["op"] == "scan":
        by, fl = recurrent(n["S"], 0, n["R"], c["rule"])
    elif c["op"] == "fork":
        by, fl = recurrent(n["F"], n["R"], n["C"], c["rule"])
    elif c["op"] == "head":
        by, fl = head(c["lm"])
    else:
        D, Dff = c["D"], c["Dff"]
        by = 4.0 * n["N"] * D
        for i in range(c["linear"] + c["full"]):
            full = i >= c["linear"]
            mix = ((c["Hq"] + 2 * c["Hkv"]) * c["d"] if full else
                   c["Hl"] * (2 * c["dk"] + c["dv"]) + 2 * c["Hl"])
            width = c["Hq"] * c["d"] if full else c["Hl"] * c["dv"]
            weights = D * (mix + width + 3 * Dff)
            by += 2.0 * weights + 4.0 * D
            fl += 2.0 * n["N"] * weights
            if full:
                by += 4.0 * n["S"] * c["Hkv"] * c["d"]
                fl += attend()[1]
            else:
                by += 4.0 * n["R"] * c["Hl"] * c["dk"] * c["dv"]
                fl += recurrent(n["F"], 0, 0, c["rule"])[1]
    return dict(bytes=float(by), flops=float(fl))


def tolerance(case):
    """About four times the difference measured against :func:`exact`."""
    if case["op"] in ("attend", "prefill"):
        # bf16 probabilities and outputs
        return dict(rel=1e-2, max=0.1)
    if case["op"] == "step":
        if case["dtype"] == "f32":
            return dict(rel=1e-5, max=1e-4, differ=0.0)
        return dict(rel=1e-2, max=0.1, differ=0.01)
    if case["op"] in ("scan", "fork"):
        # float32 states; outputs rounded to bf16
        return dict(rel=8e-3, max=2e-2)
    if case["op"] == "head":
        return dict(rel=1e-5, max=1e-4)
    return dict(rel=2.5e-2, max=0.25)  # bf16 activations between a stack's operations


# --------------------------------------------------------------------------
# the same in 64 bits, in plain torch
# --------------------------------------------------------------------------
def _rows(n, cands):
    """(request, candidate or -1, t) of every query row: a request's shared row,
    then every candidate's fed tokens 1 .. m - 1."""
    rows = []
    for r in range(n["R"]):
        rows.append((r, -1, 0))
        for c in range(r * cands, (r + 1) * cands):
            rows.extend((r, c, t) for t in range(1, int(n["m"][c])))
    return rows


def _exact_attend(c, n, q, k_pre, v_pre, k_cand, v_cand):
    rows = _rows(n, c["cands"])
    g = c["Hq"] // c["Hkv"]
    o = torch.empty(n["N"], c["Hq"], c["d"], dtype=torch.float64, device="cuda")
    p0 = n0 = 0
    for r in range(n["R"]):
        P, nr = int(n["P"][r]), int(n["rows"][r])
        f0 = n0 - r
        own = rows[n0 + 1:n0 + nr]  # the fed rows in order: fed token i is row 1 + i
        mask = torch.zeros(nr, P + nr - 1, dtype=torch.bool)
        mask[:, :P] = True
        for i, (_, ci, ti) in enumerate(own):
            for j, (_, cj, tj) in enumerate(own):
                mask[1 + i, P + j] = ci == cj and tj <= ti
        k = torch.cat([k_pre[p0:p0 + P], k_cand[f0:f0 + nr - 1]]).double()
        v = torch.cat([v_pre[p0:p0 + P], v_cand[f0:f0 + nr - 1]]).double()
        qr = q[n0:n0 + nr].double().view(nr, c["Hkv"], g, c["d"])
        z = torch.einsum("nhgd,khd->hgnk", qr, k) / math.sqrt(c["d"])
        z.masked_fill_(~mask.cuda(), float("-inf"))
        p = torch.softmax(z, -1)
        o[n0:n0 + nr] = torch.einsum("hgnk,khd->nhgd", p, v).reshape(nr, c["Hq"], c["d"])
        p0, n0 = p0 + P, n0 + nr
    return o


def _exact_prefill(c, n, q, k, v):
    g = c["Hq"] // c["Hkv"]
    o = torch.empty(n["S"], c["Hq"], c["d"], dtype=torch.float64, device="cuda")
    p0 = 0
    for r in range(n["R"]):
        P = int(n["P"][r])
        kr, vr = k[p0:p0 + P].double(), v[p0:p0 + P].double()
        for a in range(0, P, 1024):
            b = min(P, a + 1024)
            qr = q[p0 + a:p0 + b].double().view(b - a, c["Hkv"], g, c["d"])
            z = torch.einsum("nhgd,khd->hgnk", qr, kr[:b]) / math.sqrt(c["d"])
            late = torch.arange(b, device="cuda")[None] > torch.arange(a, b, device="cuda")[:, None]
            p = torch.softmax(z.masked_fill_(late, float("-inf")), -1)
            o[p0 + a:p0 + b] = torch.einsum("hgnk,khd->nhgd", p, vr[:b]).reshape(
                b - a, c["Hq"], c["d"])
        p0 += P
    return o


def _update(c, s, k, v, a, b):
    """The recurrence on states s [B, H, dk, dv] for one token each."""
    a, b = a[..., None, None], b[..., None, None]
    if c["rule"] == "delta":
        v = v - torch.einsum("bhk,bhkv->bhv", k, a * s)
    return a * s + b * k[..., None] * v[..., None, :]


def _delta_or_gla(c, s, tok, x):
    """S after token tok (indices into the rows of x) and the token's output."""
    q, k, v = (x[i][tok].double() for i in ("lq", "lk", "lv"))
    s = _update(c, s, k, v, x["alpha"][tok].double(), x["beta"][tok].double())
    return s, torch.einsum("bhkv,bhk->bhv", s, q) / math.sqrt(c["dk"])


def _exact_scan(c, n, x):
    o = torch.empty(n["S"], c["Hl"], c["dv"], dtype=torch.float64, device="cuda")
    s = torch.zeros(n["R"], c["Hl"], c["dk"], c["dv"], dtype=torch.float64, device="cuda")
    order = np.argsort(-n["P"], kind="stable")  # longest first: the active ones lead
    start = np.concatenate([[0], np.cumsum(n["P"])])[:-1][order]
    start, P = torch.from_numpy(start).cuda(), n["P"][order]
    for t in range(int(P[0])):
        live = int((P > t).sum())
        s[:live], o[start[:live] + t] = _delta_or_gla(c, s[:live], start[:live] + t, x)
    out = torch.empty_like(s)
    out[torch.from_numpy(order.copy()).cuda()] = s
    return o, out


def _exact_fork(c, n, x, s_prefix, tokens):
    """Every candidate's state after its fed tokens, and the tokens' outputs;
    tokens[c] is the first fed token of candidate c."""
    o = torch.empty(n["F"], c["Hl"], c["dv"], dtype=torch.float64, device="cuda")
    req = torch.arange(n["C"], device="cuda") // c["cands"]
    s = s_prefix.double()[req]
    m, first = torch.from_numpy(n["m"]).cuda(), torch.from_numpy(tokens).cuda()
    for t in range(1, int(n["m"].max())):
        at = torch.nonzero(m > t).flatten()
        tok = first[at] + t - 1
        s[at], o[tok] = _delta_or_gla(c, s[at], tok, x)
    return o, s


def _first_fed(n):
    return np.concatenate([[0], np.cumsum(n["m"] - 1)])[:-1].astype(np.int64)


def _e2m1(x):
    """Nearest E2M1 magnitude (ties to the even code), saturating at 6, as float64."""
    grid = torch.tensor([0.0, 0.5, 1.0, 1.5, 2.0, 3.0, 4.0, 6.0], device=x.device)
    mid = (grid[1:] + grid[:-1]) / 2
    a = x.abs()
    lo = torch.bucketize(a, mid)                # ties go down ...
    hi = torch.bucketize(a, mid, right=True)    # ... or up: the even code of the two
    code = torch.where(lo % 2 == 0, lo, hi)
    return torch.copysign(grid[code].double(), x.double())


def _quantised(w, lm):
    """The values [V, D] (float64) that a weight format holds for bf16 rows w."""
    w = w.float()
    amax = w.abs().amax(1, keepdim=True)
    # tensor by tensor: torch divides by and of a number through a reciprocal
    top = torch.full_like(amax, 6.0 if lm == "w4" else 448.0)
    inv = torch.where(amax > 0, top / amax, torch.ones_like(amax))
    scale = (amax / top).double()
    if lm == "e4m3":
        code = (w * inv).clamp(-448, 448).to(torch.float8_e4m3fn)
        return code.double() * scale
    pad = -w.shape[1] % 32
    blocks = torch.nn.functional.pad(w, (0, pad)).view(w.shape[0], -1, 32)
    bmax = blocks.abs().amax(2, keepdim=True)
    if lm == "mxfp8":
        e = torch.where(bmax > 0, torch.frexp(bmax)[1] - 9, -127).clamp(-127, 127).double()
        code = (blocks.double() * torch.exp2(-e)).clamp(-448, 448).float().to(torch.float8_e4m3fn)
        return (code.double() * torch.exp2(e)).view(w.shape[0], -1)[:, :w.shape[1]]
    t = bmax * inv[..., None]
    e = torch.full_like(t, -5.0)
    for k in range(-5, 0):
        e = torch.where(t > 6.0 * 2.0 ** k, torch.full_like(t, k + 1.0), e)
    val = _e2m1(blocks * (inv[..., None] * torch.exp2(-e))) * torch.exp2(e).double()
    return val.view(w.shape[0], -1)[:, :w.shape[1]] * scale


def _exact_head(c, n, x, lm):
    h = x["hidden"]
    h = {"bf16": lambda h: h.double(), "mxfp8": lambda h: _quantised(h, "mxfp8")}.get(
        lm, lambda h: _quantised(h, "e4m3"))(h)
    lse = torch.full((n["N"],), float("-inf"), dtype=torch.float64, device="cuda")
    # the row that predicts target t of a candidate: the shared row, then its fed rows
    at = {(r, cc, t): i for i, (r, cc, t) in enumerate(_rows(n, c["cands"]))}
    row = torch.tensor([at[(k // c["cands"], k if t else -1, t)]
                        for k in range(n["C"]) for t in range(int(n["m"][k]))], device="cuda")
    ids = torch.from_numpy(x["ids"].astype(np.int64)).cuda()
    z_y = torch.empty(n["T"], dtype=torch.float64, device="cuda")
    for a in range(0, c["V"], 8192):
        w = x["w_lm"][a:a + 8192]
        w = w.double() if lm == "bf16" else _quantised(w, lm)
        z = h @ w.T
        lse = torch.logaddexp(lse, torch.logsumexp(z, 1))
        here = (ids >= a) & (ids < a + w.shape[0])
        z_y[here] = z[row[here], ids[here] - a]
    ell = z_y - lse[row]
    cand = torch.repeat_interleave(torch.arange(n["C"], device="cuda"),
                                   torch.from_numpy(n["m"].astype(np.int64)).cuda())
    s = torch.zeros(n["C"], dtype=torch.float64, device="cuda").index_add_(0, cand, ell)
    return ell, s


def _exact_stack(c, n, x):
    x_ = x["x0"].double()
    g, Hl, dk, dv = c["Hq"] // c["Hkv"], c["Hl"], c["dk"], c["dv"]
    rows = _rows(n, c["cands"])
    shared = torch.tensor([i for i, r in enumerate(rows) if r[1] < 0], device="cuda")
    fed = torch.tensor([i for i, r in enumerate(rows) if r[1] >= 0], device="cuda",
                       dtype=torch.int64)

    def norm(v, gain):
        return v * torch.rsqrt(v.square().mean(1, keepdim=True) + 1e-6) * gain.double()

    for w in x["layers"]:
        z = norm(x_, w["g1"]) @ w["w_mix"].double().T
        if w["kind"] == "full":
            qw, kw = c["Hq"] * c["d"], c["Hkv"] * c["d"]
            q = z[:, :qw].view(-1, c["Hq"], c["d"])
            k, v = (z[:, a:a + kw].view(-1, c["Hkv"], c["d"])[fed] for a in (qw, qw + kw))
            o = _exact_attend(c, n, q, w["k_pre"].double(), w["v_pre"].double(), k, v)
        else:
            q, k = (z[:, a * Hl * dk:(a + 1) * Hl * dk].view(-1, Hl, dk) for a in (0, 1))
            v = z[:, 2 * Hl * dk:2 * Hl * dk + Hl * dv].view(-1, Hl, dv)
            gates = torch.sigmoid(z[:, 2 * Hl * dk + Hl * dv:])
            k = k / torch.sqrt(k.square().sum(-1, keepdim=True) + 1e-30)
            o = torch.empty(n["N"], Hl, dv, dtype=torch.float64, device="cuda")
            o[shared] = torch.einsum("rhkv,rhk->rhv", w["s_prefix"].double(),
                                     q[shared]) / math.sqrt(dk)
            tok = dict(lq=q[fed], lk=k[fed], lv=v[fed], alpha=gates[fed, :Hl],
                       beta=gates[fed, Hl:])
            if n["F"]:
                o[fed] = _exact_fork(c, n, tok, w["s_prefix"], _first_fed(n))[0]
        x_ = x_ + o.reshape(n["N"], -1) @ w["w_o"].double().T
        y = (norm(x_, w["g2"]) @ w["w_gu"].double().T).view(n["N"], -1, 2, 64)
        y = (torch.nn.functional.silu(y[:, :, 0]) * y[:, :, 1]).reshape(n["N"], -1)
        x_ = x_ + y @ w["w_d"].double().T
    return x_


def exact(case, seed):
    c, x = case, _inputs(case, seed)
    n = x["n"]
    if c["op"] == "attend":
        return dict(o=_exact_attend(c, n, *(x[k] for k in ("q", "k_pre", "v_pre", "k_cand",
                                                           "v_cand"))))
    if c["op"] == "prefill":
        return dict(o=_exact_prefill(c, n, x["q"], x["k"], x["v"]))
    if c["op"] == "scan":
        o, s = _exact_scan(c, n, x)
        return dict(o=o, s=s)
    if c["op"] == "fork":
        o, s = _exact_fork(c, n, x, x["s_prefix"], _first_fed(n))
        return dict(o=o, s=s)
    if c["op"] == "stack":
        return dict(x=_exact_stack(c, n, x))
    ell, s = _exact_head(c, n, x, c.get("lm", "bf16"))
    if c["op"] == "head":
        return dict(tok_logprob=ell, cand_score=s)
    o = _exact_attend(c, n, *(x[k] for k in ("q", "k_pre", "v_pre", "k_cand", "v_cand")))
    q = torch.softmax(s.view(n["R"], -1), 1)
    choice = s.view(n["R"], -1).argmax(1)
    value = {"argmax": lambda: q.amax(1), "binary": lambda: q[:, 1],
             "ordinal": lambda: (q * torch.arange(q.shape[1], device="cuda")).sum(1)}[c["mode"]]()
    return dict(o=o, tok_logprob=ell, cand_score=s, q_cand=q.flatten(),
                choice=choice.to(torch.int32), value=value)
