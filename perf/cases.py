"""The calls whose speed this framework is judged by, over the sizes it is used at.

Five kinds of call, each through the package's public entry points:

  step      forward + backward of the fused head / CE / distillation loss: the
            output stage of one training step (HeadLoss.forward, .backward)
  loss      the forward alone: the validation loss of a suite
  pairwise  KL between every ordered pair of sub-models and their top-1
            agreement: the evaluation of a suite
  spec      the verify step of speculative decoding, sampling from nuclei or
            greedily: one round of a server's decode loop
  junction  Eq. 1 between neighbouring sub-models, forward or forward and backward

A case is a dict of plain values; lists (widths, weights) are comma-separated
texts.  ``listed`` gives fixed ones, ``draw`` more of the same ranges.
"""
from __future__ import annotations

import math

import torch

import paper_2608_09703_gb300 as mls

DEV = "cuda"
Z_STD = 2.5   # spread of the smallest sub-model's logits
EXTRA = 0.2   # spread of what each larger sub-model adds to them, over Z_STD


def _ints(text):
    return [int(x) for x in str(text).split(",")]


def _dtype(case):
    return torch.float32 if case["dtype"] == "fp32" else torch.bfloat16


# ------------------------------------------------------------------------- cases
def listed():
    def head(kind, name, T, d, V, dtype="bf16", **kw):
        return dict(dict(name=name, kind=kind, T=T, d=d, V=V, dtype=dtype, tau=1.0, alpha=0.5,
                         teacher=-1, w="", ignored=0.0), **kw)

    def spec(name, B, gamma, greedy, V=50304, d="1024,3072"):
        return dict(name=name, kind="spec", B=B, gamma=gamma, d=d, V=V, dtype="bf16",
                    temperature=0.4, top_p=0.9, greedy=greedy)

    return [
        # The smallest suite of the tests and the benchmark, in full precision: a
        # unit test or a toy run, where latency and the number of launches count.
        head("step", "step_tiny", 256, "128,256", 1024, "fp32"),
        # The benchmark's training step: a 3-level suite, four packed sequences of 2048 tokens.
        head("step", "step_suite3", 8192, "1024,2048,3072", 50304),
        # The largest suite of the benchmark: four levels, 128k vocabulary.
        head("step", "step_suite4", 16384, "2048,4096,6144,8192", 128256),
        # A fine-tuning micro-batch of nothing round: odd tokens and vocabulary, widths that
        # end inside a tile, the teacher in the middle, temperature and weights of its own,
        # padding tokens ignored.
        head("step", "step_ragged", 1531, "520,1032,2056", 32003, tau=2.0, alpha=0.3, teacher=1,
             w="0.5,1.0,2.0", ignored=0.1),
        # A two-level suite kept in fp32 (a debugging or reference run), one sequence of 2048.
        head("step", "step_fp32", 2048, "768,1536", 32768, "fp32"),
        # The evaluation of the benchmark's suite on one batch.
        head("pairwise", "pairwise_suite3", 8192, "1024,2048,3072", 50304),
        # The evaluation of a draft / target pair on texts of no round length, padding left out.
        head("pairwise", "pairwise_pair", 2999, "1024,3072", 49152, ignored=0.05),
        # One verify round of a full server: the largest batch and draft length of the paper.
        spec("spec_nucleus", 102, 6, False),
        # The same for a single user: the latency of interactive decoding.
        spec("spec_single", 1, 6, False),
        # Greedy verification of a half-full server.
        spec("spec_greedy", 16, 6, True),
        # Both junctions of the 3-level suite over one training batch, forward and backward.
        dict(name="junction_train", kind="junction", T=8192, d="1024,2048,3072", dtype="bf16",
             embed_first=False, backward=True),
        # The same junctions for the 714 positions of one verify round, forward only.
        dict(name="junction_decode", kind="junction", T=714, d="1024,2048,3072", dtype="bf16",
             embed_first=False, backward=False),
    ]


# No drawn case costs more than the largest listed one (step_suite4, 3.4e14 FLOPs); fp32
# products run at half the rate and their gradients move more bytes.
_MOST_FLOPS = 3.4e14


def _log_int(rng, lo, hi):
    return min(hi, max(lo, round(math.exp(rng.uniform(math.log(lo), math.log(hi))))))


def _widths(rng, M, lo, hi, unit):
    """M increasing widths, multiples of `unit` elements (rows of a multiple of 16 bytes)."""
    got = set()
    while len(got) < M:
        got.add(_log_int(rng, lo // unit, hi // unit) * unit)
    return sorted(got)


def draw(rng):
    kind = rng.choice(["step"] * 4 + ["loss"] + ["pairwise"] * 2 + ["spec"] * 3 + ["junction"] * 2)
    if kind == "junction":
        dtype = rng.choice(["bf16", "bf16", "fp32"])
        d = _widths(rng, rng.choice([2, 2, 3]), 64, 8192, 8)
        back = rng.random() < 0.6
        return dict(kind=kind, T=_log_int(rng, 1, 65536), d=",".join(map(str, d)), dtype=dtype,
                    embed_first=rng.random() < 0.3, backward=back)
    if kind == "spec":
        d = _widths(rng, 2, 128, 8192, 8)
        return dict(kind=kind, B=_log_int(rng, 1, 102), gamma=rng.randint(1, 8),
                    d=",".join(map(str, d)), V=_log_int(rng, 1000, 256000),
                    dtype=rng.choice(["bf16"] * 4 + ["fp32"]),
                    temperature=round(rng.uniform(0.3, 1.0), 3),
                    top_p=round(rng.choice([1.0, rng.uniform(0.5, 0.99), rng.uniform(0.85, 0.95)]), 3),
                    greedy=rng.random() < 0.35)
    M = rng.choice([1, 2, 2, 3, 3, 3, 4]) if kind != "pairwise" else rng.choice([2, 2, 3, 3, 4])
    dtype = rng.choice(["bf16", "bf16", "bf16", "fp32"])
    while True:
        d = _widths(rng, M, 64, 8192, 8)
        T, V = _log_int(rng, 16, 65536), _log_int(rng, 500, 256000)
        cost = (8 if kind == "step" else 2) * T * V * sum(d) * (3 if dtype == "fp32" else 1)
        # a state (weights, gradients, workspace) stays within what three of them leave room for
        if cost <= _MOST_FLOPS and V * sum(d) <= 2.7e9 and T * sum(d) <= 4e8:
            break
    teacher = -1 if rng.random() < 0.7 else rng.randrange(M)
    w = ",".join("%.2f" % rng.uniform(0.25, 2.0) for _ in d) if rng.random() < 0.3 else ""
    return dict(kind=kind, T=T, d=",".join(map(str, d)), V=V, dtype=dtype,
                tau=rng.choice([1.0, 1.0, round(rng.uniform(0.5, 3.0), 2)]),
                alpha=rng.choice([0.0, 0.3, 0.5, 0.7]), teacher=teacher, w=w,
                ignored=rng.choice([0.0, 0.05, 0.3]))


# ------------------------------------------------------------------------- inputs
def _gen(seed, k):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 8 + k)
    return g


def _suite(d, T, V, dt, seed):
    """Hidden states [T, d_m] ~ N(0, 1) and heads [V, d_m] of a nested suite: each larger
    sub-model's first channels are the smaller one's, and what it adds moves the logits by
    EXTRA of their spread, so the sub-models mostly agree, as the distilled ones do."""
    D = d[-1]
    scale = torch.empty(D, device=DEV, dtype=torch.float32)
    lo = 0
    for m, dm in enumerate(d):
        scale[lo:dm] = (Z_STD if m == 0 else EXTRA * Z_STD) / math.sqrt(dm - lo)
        lo = dm
    gH, gW = _gen(seed, 0), _gen(seed, 1)
    Hf = torch.randn(T, D, generator=gH, device=DEV, dtype=torch.float32).to(dt)
    Wf = torch.empty(V, D, device=DEV, dtype=dt)
    step = max(1, (1 << 28) // D)
    for v in range(0, V, step):
        n = min(step, V - v)
        Wf[v:v + n] = torch.randn(n, D, generator=gW, device=DEV, dtype=torch.float32) * scale
    H = [Hf[:, :dm].contiguous() for dm in d[:-1]] + [Hf]
    W = [Wf[:, :dm].contiguous() for dm in d[:-1]] + [Wf]
    return H, W


def _head_inputs(case, seed):
    d, T, V = _ints(case["d"]), case["T"], case["V"]
    H, W = _suite(d, T, V, _dtype(case), seed)
    g = _gen(seed, 2)
    y = torch.randint(0, V, (T,), generator=g, device=DEV, dtype=torch.int32)
    if case["ignored"] > 0:
        y = torch.where(torch.rand(T, generator=g, device=DEV) < case["ignored"], -1, y).to(torch.int32)
    return H, W, y


def _draw_tokens(z, temperature, top_p, g):
    """A draft model's own choice of tokens: nucleus sampling from its logits z [n, V]."""
    p, order = torch.softmax(z.float() / temperature, -1).sort(dim=-1, descending=True)
    p = torch.where(p.cumsum(-1) - p < top_p, p, 0.0)
    return order.gather(-1, torch.multinomial(p, 1, generator=g)).squeeze(-1)


def _spec_inputs(case, seed):
    d, B, gamma, V = _ints(case["d"]), case["B"], case["gamma"], case["V"]
    (Hd, Hv), (Wd, Wv) = _suite(d, B * (gamma + 1), V, _dtype(case), seed)
    Hd = Hd.view(B, gamma + 1, d[0])[:, :gamma].reshape(B * gamma, d[0]).contiguous()
    g = _gen(seed, 2)
    draft = torch.empty(B * gamma, dtype=torch.int64, device=DEV)
    step = max(1, (1 << 27) // V)
    for i in range(0, B * gamma, step):
        z = Hd[i:i + step] @ Wd.T
        draft[i:i + step] = (z.argmax(-1) if case["greedy"] else
                             _draw_tokens(z, case["temperature"], case["top_p"], g))
    u = torch.rand(B, gamma + 1, 2, generator=g, device=DEV, dtype=torch.float32)
    return Hd, Wd, Hv, Wv, draft.to(torch.int32).view(B, gamma), u


def _junction_inputs(case, seed):
    """Per junction (o, e, g): a sub-model's output, the next one's fresh embeddings, whose
    norms differ as in a trained model, and the gradient that comes back."""
    d, T, dt = _ints(case["d"]), case["T"], _dtype(case)
    gen = _gen(seed, 0)
    got = []
    for dp, dn in zip(d[:-1], d[1:]):
        o = torch.randn(T, dp, generator=gen, device=DEV) * 8
        e = torch.randn(T, dn - dp, generator=gen, device=DEV) * 0.02
        g = torch.randn(T, dn, generator=gen, device=DEV) * 1e-3
        got.append((o.to(dt), e.to(dt), g.to(dt)))
    return got


# ------------------------------------------------------------------------- passes
def prepare(case, seed):
    kind, dt = case["kind"], _dtype(case)
    s = {"kind": kind}
    if kind == "spec":
        d = _ints(case["d"])
        s["in"] = _spec_inputs(case, seed)
        s["op"] = mls.SpecVerify(case["B"], case["gamma"], case["V"], d[0], d[1], case["temperature"],
                                 case["top_p"], case["greedy"], dt, DEV)
    elif kind == "junction":
        s["in"] = _junction_inputs(case, seed)
        s["first"], s["backward"] = case["embed_first"], case["backward"]
        s["out"] = [(torch.empty_like(g), torch.empty_like(o), torch.empty_like(e))
                    for o, e, g in s["in"]]
    else:
        d = _ints(case["d"])
        s["in"] = _head_inputs(case, seed)
        s["op"] = mls.HeadLoss(d, case["T"], case["V"],
                               teacher=None if case["teacher"] < 0 else case["teacher"],
                               tau=case["tau"], alpha=case["alpha"],
                               w=[float(x) for x in case["w"].split(",")] if case["w"] else None,
                               dtype=dt, device=DEV)
    return s


def run(s):
    kind = s["kind"]
    if kind == "spec":
        n, nxt = s["op"](*s["in"])
        return {"n_accepted": n, "next_token": nxt}
    if kind == "junction":
        got = {}
        for i, ((o, e, _), (x, _, _)) in enumerate(zip(s["in"], s["out"])):
            mls.mls_junction_fwd(o, e, x, s["first"])
            got["x%d" % i] = x
        if s["backward"]:
            for i in reversed(range(len(s["in"]))):
                (o, e, g), (_, d_o, d_e) = s["in"][i], s["out"][i]
                mls.mls_junction_bwd(o, e, g, d_o, d_e, s["first"])
                got["d_o%d" % i], got["d_e%d" % i] = d_o, d_e
        return got
    op, (H, W, y) = s["op"], s["in"]
    if kind == "pairwise":
        kl, am, stats = op.pairwise(H, W, y)
        return {"tok_kl": kl, "argmax": am, "pair_stats": stats}
    got = {"loss": op.forward(H, W, y), "tok_loss": op.tok_loss, "tok_diag": op.tok_diag,
           "argmax": op.argmax, "stats": op.stats}
    if kind == "step":
        got["dH"], got["dW"] = op.backward(H, W, y)
    return got


def work(case):
    """Each input read once, each output written once; the products that the calls are defined
    by.  A training step has four of them: the logits are never stored (the forward hands only
    row statistics to the backward), so they are formed in both passes."""
    elt = 4 if case["dtype"] == "fp32" else 2
    d = _ints(case["d"])
    if case["kind"] == "junction":
        T, nxt = case["T"], sum(d[1:])  # per junction: o and e are d_next values a token, x too
        return {"bytes": T * nxt * elt * (5 if case["backward"] else 2),
                "flops": T * nxt * (9 if case["backward"] else 3)}
    V = case["V"]
    if case["kind"] == "spec":
        B, g = case["B"], case["gamma"]
        rows = [(B * (g + 1), d[1])] + ([] if case["greedy"] else [(B * g, d[0])])
        return {"bytes": sum((V + n) * dm * elt for n, dm in rows) + 4 * B * (3 * g + 4),
                "flops": sum(2 * V * n * dm for n, dm in rows)}
    T, D, M = case["T"], sum(d), len(d)
    nbytes = (T + V) * D * elt + 4 * T
    if case["kind"] == "pairwise":
        return {"bytes": nbytes + 4 * M * (M + 1) * T, "flops": 2 * T * V * D}
    nbytes += 4 * T * M * 7  # per token and sub-model: loss, three diagnostics, argmax, two statistics
    if case["kind"] == "loss":
        return {"bytes": nbytes, "flops": 2 * T * V * D}
    return {"bytes": nbytes + 4 * (T + V) * D, "flops": 8 * T * V * D}


def tolerance(case):
    """About four times the error against `exact` that was seen over the listed and some drawn cases."""
    full = case["dtype"] == "fp32"
    if case["kind"] == "spec":
        # accept / sample decisions: rounding may move one that lies within it of its threshold
        return {"rel": 0.0, "differ": 0.01}
    if case["kind"] == "junction":
        # seen 1.7e-3 (bf16 outputs; one step in the last place is 2^-8 at most)
        return {"rel": 2e-6, "max": 2e-5} if full else {"rel": 5e-3, "max": 0.016}
    if case["kind"] == "step":
        # gradients: dL/dz is rounded to bf16 (or the product's tf32) before the last products: 1e-3 to 3e-3
        return {"rel": 6e-3, "max": 0.1, "differ": 1e-3}
    # sums of fp32 statistics: 9e-6 (KL); fp32 storage takes tf32 products: 5e-4, KL 1.4e-3
    return {"rel": 6e-3, "max": 0.1, "differ": 1e-2} if full else {"rel": 4e-5, "max": 2e-3, "differ": 1e-3}


# ------------------------------------------------------------------------- in 64 bits
_EXACT_FLOPS = 8e12  # of 64-bit products: some 10 seconds


def exact(case, seed):
    kind = case["kind"]
    if kind == "spec":
        return None  # whole values only: counts and tokens
    if kind == "junction":
        return _exact_junction(case, seed)
    T, V, D = case["T"], case["V"], sum(_ints(case["d"]))
    if 2 * T * V * D > _EXACT_FLOPS:
        return None
    if kind == "pairwise":
        return _exact_pairwise(case, seed)
    return _exact_head(case, seed, kind == "step" and 6 * T * V * D <= _EXACT_FLOPS)


def _chunks(T, V):
    step = max(1, (1 << 25) // V)
    return [(t, min(T, t + step)) for t in range(0, T, step)]


def _exact_head(case, seed, grads):
    H, W, y = _head_inputs(case, seed)
    M, T, V, tau, alpha = len(H), case["T"], case["V"], case["tau"], case["alpha"]
    t = case["teacher"] if case["teacher"] >= 0 else M - 1
    w = [float(x) for x in case["w"].split(",")] if case["w"] else [1.0] * M
    f64 = dict(device=DEV, dtype=torch.float64)
    H, W = [h.double() for h in H], [x.double() for x in W]
    n = max(1, int((y >= 0).sum()))
    tok, diag, stats = torch.zeros(M, T, **f64), torch.zeros(3, M, T, **f64), torch.zeros(2, M, T, **f64)
    dH = [torch.zeros_like(h) for h in H] if grads else None
    dW = [torch.zeros_like(x) for x in W] if grads else None
    for a, b in _chunks(T, V):
        yc = y[a:b].long()
        ok = yc >= 0
        idx = yc.clamp(min=0)[:, None]
        zt = H[t][a:b] @ W[t].T
        logq = torch.log_softmax(zt / tau, -1)
        q = logq.exp()
        hq = -(q * logq).sum(-1)
        for m in range(M):
            z = zt if m == t else H[m][a:b] @ W[m].T
            lse, lset = torch.logsumexp(z, -1), torch.logsumexp(z / tau, -1)
            ce = lse - z.gather(-1, idx)[:, 0]
            ld = lset - (q * z).sum(-1) / tau
            one = ce if m == t else (1 - alpha) * ce + alpha * ld
            kl = torch.zeros_like(ld) if m == t else ld - hq
            stats[0, m, a:b], stats[1, m, a:b] = lse, lset
            for out, v in ((tok[m], one), (diag[0, m], ce), (diag[1, m], ld), (diag[2, m], kl)):
                out[a:b] = torch.where(ok, v, 0.0)
            if grads:
                G = (z - lse[:, None]).exp_()
                G.scatter_add_(-1, idx, -torch.ones_like(idx, dtype=torch.float64))
                if m != t:
                    G.mul_(1 - alpha).add_(((z / tau - lset[:, None]).exp_() - q), alpha=alpha / tau)
                G *= torch.where(ok, w[m] / n, 0.0)[:, None]
                dH[m][a:b] = G @ W[m]
                dW[m] += G.T @ H[m][a:b]
    loss = sum(w[m] * tok[m].sum() for m in range(M)) / n
    got = {"loss": loss.reshape(1), "tok_loss": tok, "tok_diag": diag, "argmax": None, "stats": stats}
    if case["kind"] == "step":
        got["dH"], got["dW"] = dH, dW
    return got


def _exact_pairwise(case, seed):
    H, W, y = _head_inputs(case, seed)
    M, T, V = len(H), case["T"], case["V"]
    W = [x.double() for x in W]
    kl = torch.zeros(M, M, T, device=DEV, dtype=torch.float64)
    same = torch.zeros(M, M, T, device=DEV, dtype=torch.float64)
    for a, b in _chunks(T, V):
        z = [H[m][a:b].double() @ W[m].T for m in range(M)]
        logp = [torch.log_softmax(x, -1) for x in z]
        top = [x.argmax(-1) for x in z]
        for i in range(M):
            p = logp[i].exp()
            for j in range(M):
                kl[i, j, a:b] = (p * (logp[i] - logp[j])).sum(-1)
                same[i, j, a:b] = (top[i] == top[j]).double()
    ok = (y >= 0).double()
    n = ok.sum().clamp(min=1)
    return {"tok_kl": kl, "argmax": None,
            "pair_stats": torch.stack([(kl * ok).sum(-1) / n, (same * ok).sum(-1) / n])}


def _exact_junction(case, seed):
    got = {}
    for i, (o, e, g) in enumerate(_junction_inputs(case, seed)):
        o, e, g = o.double(), e.double(), g.double()
        dp = o.shape[1]
        no, ne = o.norm(dim=-1, keepdim=True), e.norm(dim=-1, keepdim=True)
        s = ne / no
        got["x%d" % i] = torch.cat([e, o * s] if case["embed_first"] else [o * s, e], -1)
        if case["backward"]:
            go, ge = (g[:, -dp:], g[:, :-dp]) if case["embed_first"] else (g[:, :dp], g[:, dp:])
            dot = (go * o).sum(-1, keepdim=True)
            got["d_o%d" % i] = s * (go - o * dot / no ** 2)
            got["d_e%d" % i] = ge + s * dot * e / ne ** 2
    return got
