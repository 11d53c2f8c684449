"""The measured cases of the verifier library.

Each case is one pass through the library's public calls as a serving program
makes them: device buffers in hand, outputs preallocated, a context that the
program keeps, default options.  The listed sizes are those of the project's
workloads (five logit workloads, the scorer heads, the LM head, the validation
pool) and of its tests; `draw` spreads over the same ranges.

  route        pr_route over a whole batch of finished responses
  features     pr_token_features with offsets, then pr_aggregate_score: the
               unfused path of a program that keeps the per-token records
  decode       consecutive pr_decode_step calls of a decoding loop; requests
               end at their EOS and their slots' rows go to new requests, and
               the last step ends every live request, so that all scores are
               outputs
  lm_features  pr_lmhead_features, then pr_aggregate_score: a finished batch
               scored from hidden states, no logits in memory
  lm_decode    consecutive pr_lmhead_decode_step calls
  head         pr_head_score over the feature sequences of a batch
  quantile     pr_quantile_score over the same kind of batch
  selective    pr_selective_metrics over a validation pool
"""
import math

import numpy as np
import torch

from paper_2608_28726_gb300 import binding as B
from paper_2608_28726_gb300 import workloads as W

DEV = "cuda"
V_FULL, V_WIDE, V_TINY, V_ODD = 151936, 262144, 32000, 70001
D_MODEL = 3584
BUDGET = 2.6e9  # bytes of logits or weights of the largest pass
LEVELS = ((0, 1), (1, 10), (1, 4), (1, 2), (3, 4), (9, 10), (1, 1))  # the quantile summary's


def listed():
    return [
        # one small reply batch of an interactive user: latency and launches count
        dict(name="route_tiny", kind="route", dtype="f32", vocab=V_TINY, dist="tiny", n_req=8,
             spread="uniform", lo=16, hi=64, layout=1),
        # the headline: a batch of 64 finished responses
        dict(name="route_full", kind="route", dtype="bf16", vocab=V_FULL, dist="full", n_req=64,
             spread="uniform", lo=32, hi=256, layout=2),
        # a vocabulary that is no multiple of the vector width, so that most rows
        # start off a 16-byte boundary; ragged responses, per-token records kept
        dict(name="features_odd", kind="features", dtype="bf16", vocab=V_ODD, dist="full",
             n_req=24, spread="lognormal", lo=8, hi=1024, layout=3, topk=20),
        # wide fp32 logits with heavy tails and tied maxima
        dict(name="features_wide", kind="features", dtype="f32", vocab=V_WIDE, dist="wide",
             n_req=8, spread="uniform", lo=64, hi=512, layout=4, topk=20),
        # a decoding loop at low load: a handful of live requests
        dict(name="decode_8", kind="decode", dtype="bf16", vocab=V_FULL, dist="full", live=8,
             steps=16, layout=5),
        # a decoding loop at full load
        dict(name="decode_256", kind="decode", dtype="bf16", vocab=V_FULL, dist="full", live=256,
             steps=16, layout=6),
        # finished responses scored from their hidden states
        dict(name="lm_features", kind="lm_features", vocab=V_FULL, d=D_MODEL, n_req=10,
             spread="uniform", lo=32, hi=256, layout=7, topk=20),
        # a decoding loop that hands over hidden states
        dict(name="lm_decode_64", kind="lm_decode", vocab=V_FULL, d=D_MODEL, live=64, steps=4,
             layout=8),
        # the transformer scorer head on the headline's batch
        dict(name="head_full", kind="head", n_req=64, spread="uniform", lo=32, hi=256, layout=2,
             layers=2),
        # and on a large ragged batch
        dict(name="head_ragged", kind="head", n_req=1024, spread="lognormal", lo=8, hi=1024,
             layout=9, layers=2),
        # the quantile scorer on a ragged batch whose longest answers run to a
        # few thousand tokens
        dict(name="quantile_ragged", kind="quantile", n_req=512, spread="lognormal", lo=8,
             hi=4096, layout=12),
        # calibration of tau on a large validation pool
        dict(name="selective_pool", kind="selective", n=1 << 24, q=0.5),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges."""
    kind = rng.choice(["route", "route", "features", "features", "decode", "decode",
                       "lm_features", "lm_decode", "head", "quantile", "selective"])
    layout = rng.randrange(100, 1 << 20)
    if kind == "selective":
        return dict(kind=kind, n=_log_int(rng, 100, 1 << 24), q=round(rng.random(), 3))
    c = dict(kind=kind, layout=layout)
    if kind in ("route", "features", "lm_features", "head", "quantile"):
        c["n_req"] = _log_int(rng, 1, 1024)
        c["spread"] = rng.choice(["uniform", "lognormal"])
        top = {"head": 2048, "quantile": 4096}.get(kind, 1024)
        c["lo"] = _log_int(rng, 1, 64)
        c["hi"] = c["lo"] + _log_int(rng, 1, top - c["lo"])
    if kind in ("route", "features", "decode"):
        c["dist"] = rng.choice(["tiny", "full", "wide"])
        c["dtype"] = "bf16" if c["dist"] == "full" else "f32"
        c["vocab"] = _log_int(rng, 1000, V_WIDE)
        if rng.random() < 0.4:  # a multiple of 64, as most vocabularies are padded
            c["vocab"] = max(64, c["vocab"] // 64 * 64)
    if kind in ("lm_features", "lm_decode"):
        c["d"] = 8 * _log_int(rng, 32, 512)
        c["vocab"] = _log_int(rng, 4000, V_FULL)
    if kind in ("features", "lm_features"):
        c["topk"] = rng.randint(1, 32)
    if kind in ("decode", "lm_decode"):
        c["live"] = _log_int(rng, 1, 512 if kind == "decode" else 256)
        c["steps"] = rng.randint(4, 16) if kind == "decode" else rng.randint(2, 4)
        if kind == "decode":
            while c["live"] > 1 and c["live"] * c["steps"] * c["vocab"] * _esize(c) > BUDGET:
                c["live"] //= 2
    if kind == "head":
        c["layers"] = rng.choice([1, 2, 2, 4])
    while "n_req" in c and c["n_req"] > 1 and not _affordable(c):
        c["n_req"] = max(1, c["n_req"] * 2 // 3)
    return c


def _esize(c):
    return 2 if c["dtype"] == "bf16" else 4


def _affordable(c):
    T = _lengths(c)
    rows = int(T.sum())
    if c["kind"] in ("route", "features"):
        return rows * c["vocab"] * _esize(c) <= BUDGET
    if c["kind"] == "lm_features":
        return rows * c["vocab"] * c["d"] <= 1.5e3 * V_FULL * D_MODEL
    if c["kind"] == "head":
        return c["layers"] * (rows / 1.8e5 + float((T.astype(np.float64) ** 2).sum()) / 6e7) <= 4
    return rows <= 2.5e5


# ---- inputs -------------------------------------------------------------------------------


def _lengths(c):
    g = np.random.Generator(np.random.PCG64(c["layout"]))
    if c["spread"] == "uniform":
        return g.integers(c["lo"], c["hi"], size=c["n_req"], endpoint=True).astype(np.int64)
    mid = min(c["hi"], 128 if c["hi"] <= 1024 else 256)
    raw = np.exp(g.normal(math.log(mid), 0.8, size=c["n_req"]))
    return np.clip(np.round(raw), c["lo"], c["hi"]).astype(np.int64)


def _offsets(T):
    return np.concatenate([[0], np.cumsum(T)]).astype(np.int64)


def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _logits(c, n, g):
    """n rows of the case's distribution and their emitted tokens, drawn from
    the softmax of the stored row (Gumbel-max)."""
    V = c["vocab"]
    x = torch.empty(n, V, dtype=torch.bfloat16 if c["dtype"] == "bf16" else torch.float32,
                    device=DEV)
    chosen = torch.empty(n, dtype=torch.int32, device=DEV)
    step = max(1, (1 << 28) // V)
    for a in range(0, n, step):
        b = min(n, a + step)
        k = b - a
        r = torch.arange(k, device=DEV)
        z = torch.randn(k, V, generator=g, device=DEV)
        if c["dist"] == "wide":  # 2 t_3, the maximum copied to a second place on 10% of rows
            q = torch.zeros_like(z)
            for _ in range(3):
                q += torch.randn(k, V, generator=g, device=DEV).square_()
            z.mul_(2.0).div_(q.div_(3.0).sqrt_())
            del q
            tie = torch.rand(k, generator=g, device=DEV) < 0.1
            other = torch.randint(0, V, (k,), generator=g, device=DEV)
            top, at = z.max(dim=1)
            z[r, torch.where(tie, other, at)] = top
        else:
            if c["dist"] == "full":
                z.mul_(1.0 + 3.0 * torch.rand(k, 1, generator=g, device=DEV))
                amp = 12.0 * torch.rand(k, generator=g, device=DEV)
                amp *= torch.rand(k, generator=g, device=DEV) < 0.7
            else:
                z.mul_(2.0)
                amp = 8.0 * torch.rand(k, generator=g, device=DEV)
            at = torch.randint(0, V, (k,), generator=g, device=DEV)
            z[r, at] += amp
        x[a:b] = z
        u = torch.rand(k, V, generator=g, device=DEV).clamp_(min=1e-30).log_().neg_().log_()
        chosen[a:b] = (x[a:b].float() - u).argmax(dim=1)
        del z, u
    return x, chosen


def _hidden(c, n, g):
    h = torch.randn(n, c["d"], generator=g, device=DEV)
    h *= 0.5 + 1.5 * torch.rand(n, 1, generator=g, device=DEV)
    chosen = torch.randint(0, c["vocab"], (n,), generator=g, device=DEV, dtype=torch.int32)
    return h.bfloat16(), chosen


def _lm_weight(c, g):
    w = torch.empty(c["vocab"], c["d"], dtype=torch.bfloat16, device=DEV)
    for a in range(0, c["vocab"], 32768):
        b = min(c["vocab"], a + 32768)
        w[a:b] = torch.randn(b - a, c["d"], generator=g, device=DEV) * (2.0 / c["d"] ** 0.5)
    return w


def _records(T, g):
    """Feature records of a batch, as the verifier writes them (the slots that
    the scorer heads do not read hold noise)."""
    n = int(T.sum())
    feat = 5.0 * torch.randn(n, B.PR_NFEAT, generator=g, device=DEV)
    m = 0.02 + 0.98 * torch.rand(n, generator=g, device=DEV)
    miss = -2.0 * torch.log(torch.rand(n, generator=g, device=DEV).clamp_(min=1e-30))
    miss *= torch.rand(n, generator=g, device=DEV) < 0.5
    feat[:, B_LOGP] = torch.log(m) - miss
    feat[:, B_MAXP] = m
    feat[:, B_TOPK] = -math.log(20.0) * torch.rand(n, generator=g, device=DEV)
    lens = torch.from_numpy(T).to(DEV)
    start = torch.cumsum(lens, 0) - lens
    req = torch.repeat_interleave(torch.arange(len(T), device=DEV), lens)
    t = torch.arange(n, device=DEV) - start[req]
    feat[:, B_RHO] = (t + 1).float() / lens[req].float()
    return feat


B_LOGP, B_MAXP, B_MARGIN, B_ENT, B_TOPK, B_RHO, B_LSE, B_X1 = range(8)  # record slots


def _trace(c):
    """A decoding loop's schedule: per step the slot of each live row and
    whether its request ends there (request lengths of some hundreds of
    tokens), and the number of slots used."""
    g = np.random.Generator(np.random.PCG64(c["layout"]))
    slot = np.arange(c["live"], dtype=np.int32)
    used, slots, ends = c["live"], [], []
    for s in range(c["steps"]):
        end = g.random(c["live"]) < 1.0 / 532
        if s == c["steps"] - 1:
            end[:] = True
        slots.append(slot.copy())
        ends.append(end.astype(np.uint8))
        fresh = np.flatnonzero(end)
        if s < c["steps"] - 1:  # the next request takes an unused slot
            slot[fresh] = np.arange(used, used + fresh.size)
            used += fresh.size
    return np.stack(slots), np.stack(ends), used


class State:
    """A program's buffers and its context."""

    ctx = None

    def __del__(self):
        if self.ctx is not None:
            B.pr_ctx_destroy(self.ctx)


def _scorer(s):
    w, s.b = W.scorer(1002)
    s.w = torch.from_numpy(w).to(DEV)
    s.tau = 0.5


def _request_buffers(s, n):
    s.score = torch.zeros(n, dtype=torch.float32, device=DEV)
    s.ship = torch.zeros(n, dtype=torch.uint8, device=DEV)
    s.flags = torch.zeros(n, dtype=torch.int32, device=DEV)
    s.agg = torch.zeros(n, B.PR_NAGG, dtype=torch.float32, device=DEV)


def _row_buffers(s, n):
    s.feat = torch.empty(n, B.PR_NFEAT, dtype=torch.float32, device=DEV)
    s.top2 = torch.empty(n, 2, dtype=torch.int32, device=DEV)
    s.row_flags = torch.empty(n, dtype=torch.int32, device=DEV)


def prepare(case, seed):
    c, g, s = case, _gen(seed), State()
    s.case, kind = c, case["kind"]
    if kind == "selective":
        n = c["n"]
        s.scores = torch.sigmoid(1.5 * torch.randn(n, generator=g, device=DEV))
        s.labels = (torch.rand(n, generator=g, device=DEV) < s.scores).to(torch.uint8)
        s.scores[torch.rand(n, generator=g, device=DEV) < 0.01] = float("nan")
        s.ctx = B.pr_ctx_create(0, 1, 1)
        return s
    if kind in ("decode", "lm_decode"):
        slots, ends, used = _trace(c)
        n = c["live"] * c["steps"]
        if kind == "decode":
            x, chosen = _logits(c, n, g)
        else:
            x, chosen = _hidden(c, n, g)
            s.weight = _lm_weight(c, g)
        s.x = list(x.view(c["steps"], c["live"], -1).unbind(0))
        s.chosen = list(chosen.view(c["steps"], c["live"]).unbind(0))
        s.slot = list(torch.from_numpy(slots).to(DEV).unbind(0))
        s.eos = list(torch.from_numpy(ends).to(DEV).unbind(0))
        _scorer(s)
        _request_buffers(s, used)
        s.ctx = B.pr_ctx_create(0, 1, used)
        return s
    T = _lengths(c)
    n = int(T.sum())
    s.offsets = torch.from_numpy(_offsets(T)).to(DEV)
    _request_buffers(s, len(T))
    s.ctx = B.pr_ctx_create(0, n, len(T))
    if kind in ("route", "features"):
        s.x, s.chosen = _logits(c, n, g)
        _scorer(s)
    elif kind == "lm_features":
        s.x, s.chosen = _hidden(c, n, g)
        s.weight = _lm_weight(c, g)
        _scorer(s)
    else:
        s.records = _records(T, g)
        s.row_flags = torch.zeros(n, dtype=torch.int32, device=DEV)
        s.tau = 0.5
        if kind == "head":
            s.w = torch.from_numpy(W.head_weights(c["layers"])).to(DEV)
        else:
            s.w = torch.from_numpy(W.qmlp_weights()).to(DEV)
            s.summary = torch.zeros(len(T), B.PR_QMLP_SUMMARY, dtype=torch.float32, device=DEV)
    if kind in ("features", "lm_features"):
        _row_buffers(s, n)
    return s


def run(s):
    c = s.case
    kind = c["kind"]
    if kind == "route":
        B.pr_route(s.ctx, s.x, s.chosen, s.offsets, s.w, s.b, s.tau, score=s.score, ship=s.ship,
                   req_flags=s.flags, agg=s.agg)
        return dict(score=s.score, ship=s.ship, flags=s.flags, agg=s.agg)
    if kind in ("features", "lm_features"):
        if kind == "features":
            B.pr_token_features(s.ctx, s.x, s.chosen, c["topk"], s.offsets, s.feat, s.top2,
                                s.row_flags)
        else:
            B.pr_lmhead_features(s.ctx, s.x, s.weight, s.chosen, c["topk"], s.offsets, s.feat,
                                 s.top2, s.row_flags)
        B.pr_aggregate_score(s.ctx, s.feat, s.offsets, s.w, s.b, s.tau, s.row_flags, s.agg,
                             s.score, s.ship, s.flags)
        return dict(feat=s.feat, top2=s.top2, row_flags=s.row_flags, score=s.score, ship=s.ship,
                    flags=s.flags, agg=s.agg)
    if kind == "decode":
        for k in range(c["steps"]):
            B.pr_decode_step(s.ctx, s.x[k], s.slot[k], s.chosen[k], s.eos[k], s.w, s.b, s.tau,
                             s.score, s.ship, s.flags, s.agg)
        return dict(score=s.score, ship=s.ship, flags=s.flags, agg=s.agg)
    if kind == "lm_decode":
        for k in range(c["steps"]):
            B.pr_lmhead_decode_step(s.ctx, s.x[k], s.weight, s.slot[k], s.chosen[k], s.eos[k],
                                    s.w, s.b, s.tau, s.score, s.ship, s.flags, s.agg)
        return dict(score=s.score, ship=s.ship, flags=s.flags, agg=s.agg)
    if kind == "head":
        B.pr_head_score(s.ctx, s.records, s.offsets, s.w, c["layers"], s.tau, s.row_flags,
                        s.score, s.ship, s.flags)
        return dict(score=s.score, ship=s.ship, flags=s.flags)
    if kind == "quantile":
        B.pr_quantile_score(s.ctx, s.records, s.offsets, s.w, s.tau, s.row_flags, s.summary,
                            s.score, s.ship, s.flags)
        return dict(summary=s.summary, score=s.score, ship=s.ship, flags=s.flags)
    return B.pr_selective_metrics(s.ctx, s.scores, c["q"], s.labels)


# ---- what a pass cannot do without ------------------------------------------------------------


def work(case):
    c, kind = case, case["kind"]
    if kind == "selective":
        return {"bytes": 5.0 * c["n"], "flops": 10.0 * c["n"]}
    if kind in ("decode", "lm_decode"):
        used = _trace(c)[2]
        rows = c["live"] * c["steps"]
        # slots are read and written each step: 17 words of running state
        small = rows * (9 + 2 * 68) + used * (4 * B.PR_NAGG + 9)
        if kind == "decode":
            big = rows * c["vocab"] * _esize(c)
            return {"bytes": float(big + small), "flops": 6.0 * rows * c["vocab"]}
        big = c["steps"] * c["vocab"] * c["d"] * 2 + rows * c["d"] * 2
        return {"bytes": float(big + small), "flops": 2.0 * rows * c["vocab"] * c["d"]}
    T = _lengths(c)
    n, r = int(T.sum()), len(T)
    small = 8 * (r + 1) + r * 9
    if kind == "route":
        return {"bytes": float(n * (c["vocab"] * _esize(c) + 4) + small + 44 * r),
                "flops": 6.0 * n * c["vocab"]}
    if kind == "features":
        return {"bytes": float(n * (c["vocab"] * _esize(c) + 4 + 44) + small + 44 * r),
                "flops": 6.0 * n * c["vocab"]}
    if kind == "lm_features":
        return {"bytes": float((c["vocab"] + n) * c["d"] * 2 + n * 48 + small + 44 * r),
                "flops": 2.0 * n * c["vocab"] * c["d"]}
    if kind == "head":
        per_row = 2 * (4 * 64 + c["layers"] * (4 * 64 * 64 + 2 * 64 * 128))
        attn = c["layers"] * 2 * 2 * 64 * float((T.astype(np.float64) ** 2).sum())
        return {"bytes": float(n * 36 + 4 * W.head_param_count(c["layers"]) + small),
                "flops": n * per_row + attn}
    return {"bytes": float(n * 36 + 4 * W.qmlp_param_count() + small + r * 4 * B.PR_QMLP_SUMMARY),
            "flops": float(r * 2 * (28 * 64 + 64 * 64 + 64))}


def tolerance(case):
    """fp32 sums in another order: about four times the distance from 64 bits
    that was measured (1e-7 to 5e-7; with the LM head, whose logits are fp32
    sums of d products, 2e-6 to 8e-6, and near-ties of its top tokens may fall
    the other way)."""
    kind = case["kind"]
    if kind in ("lm_features", "lm_decode"):
        return {"rel": 3e-5, "max": 1e-3, "differ": 2e-3}
    if kind == "selective":
        return {"rel": 1e-6, "max": 1e-6}
    return {"rel": 4e-6, "max": 1e-4, "differ": 1e-3}


# ---- the same in 64 bits -----------------------------------------------------------------------


def _exact_rows(x, chosen, K):
    """The eight record slots (rho left 0) and the first two tokens of rows of
    float64 logits."""
    lse = torch.logsumexp(x, dim=1)
    p = torch.exp(x - lse[:, None])
    ent = lse - (p * torch.where(p > 0, x, torch.zeros_like(x))).sum(dim=1)
    del p
    i1 = x.argmax(dim=1)
    x1 = x.gather(1, i1[:, None])[:, 0]
    top = torch.topk(x, min(max(K, 2), x.size(1)), dim=1).values
    y = x.clone()
    y.scatter_(1, i1[:, None], float("-inf"))
    i2 = y.argmax(dim=1)
    del y
    lk = top[:, :K] - lse[:, None]
    h = (torch.exp(lk) * lk).sum(dim=1)
    rec = torch.zeros(x.size(0), B.PR_NFEAT, dtype=torch.float64, device=DEV)
    rec[:, B_LOGP] = x.gather(1, chosen.long()[:, None])[:, 0] - lse
    rec[:, B_MAXP] = torch.exp(x1 - lse)
    rec[:, B_MARGIN] = rec[:, B_MAXP] - torch.exp(top[:, 1] - lse)
    rec[:, B_ENT] = ent
    rec[:, B_TOPK] = h
    rec[:, B_LSE] = lse
    rec[:, B_X1] = x1
    return rec, torch.stack([i1, i2], dim=1)


def _exact_records(logits_of, n, V, chosen, K):
    rec, top2 = [], []
    step = max(1, (1 << 26) // V)
    for a in range(0, n, step):
        b = min(n, a + step)
        r, t = _exact_rows(logits_of(a, b), chosen[a:b], K)
        rec.append(r)
        top2.append(t)
    return torch.cat(rec), torch.cat(top2)


def _exact_pool(s, groups, rec):
    """Aggregates, scores and decisions; groups: the row indices of each request."""
    w, b = s.w.double(), float(np.float32(s.b))
    agg = torch.zeros(len(groups), B.PR_NAGG, dtype=torch.float64, device=DEV)
    for r, rows in enumerate(groups):
        v = rec[rows]
        T = v.size(0)
        cols = torch.stack([v[:, B_LOGP], v[:, B_MAXP], v[:, B_MARGIN], -v[:, B_ENT],
                            v[:, B_TOPK]], dim=1)
        agg[r, 0:10:2] = cols.mean(dim=0)
        agg[r, 1:10:2] = cols.amin(dim=0)
        agg[r, 10] = (T + 1) / (2 * T)
    score = torch.sigmoid(agg @ w + b)
    return dict(score=score, ship=(score >= s.tau).to(torch.uint8),
                flags=torch.zeros(len(groups), dtype=torch.int32, device=DEV), agg=agg)


def _exact_head(x, w, layers):
    """The transformer scorer head on one request's [T, 4] features; returns z."""
    at = 0

    def take(*shape):
        nonlocal at
        n = int(np.prod(shape))
        v = w[at:at + n].view(*shape)
        at += n
        return v

    def norm(v, gain, shift):
        v = v - v.mean(dim=1, keepdim=True)
        return v / torch.sqrt((v * v).mean(dim=1, keepdim=True) + 1e-5) * gain + shift

    D, F, T = W.HEAD_D, W.HEAD_DFF, x.size(0)
    Wi, bi = take(D, 4), take(D)
    t = torch.arange(T, dtype=torch.float64, device=DEV)[:, None]
    f = torch.exp(-torch.arange(0, D, 2, dtype=torch.float64, device=DEV) * (math.log(1e4) / D))
    pe = torch.stack([torch.sin(t * f), torch.cos(t * f)], dim=2).reshape(T, D)
    h = x @ Wi.T + bi + pe
    for _ in range(layers):
        Wq, bq, Wo, bo = take(3 * D, D), take(3 * D), take(D, D), take(D)
        g1, e1, W1, b1, W2, b2 = take(D), take(D), take(F, D), take(F), take(D, F), take(D)
        g2, e2 = take(D), take(D)
        q, k, v = ((h @ Wq.T + bq).view(T, 3, W.HEAD_HEADS, -1).permute(1, 2, 0, 3))
        o = torch.softmax(q @ k.transpose(1, 2) / math.sqrt(D // W.HEAD_HEADS), dim=2) @ v
        h = norm(h + o.permute(1, 0, 2).reshape(T, D) @ Wo.T + bo, g1, e1)
        h = norm(h + torch.relu(h @ W1.T + b1) @ W2.T + b2, g2, e2)
    wo, b = take(D), take(1)
    return h.mean(dim=0) @ wo + b[0]


def _exact_quantile(s, off):
    w = s.w.double()
    sizes = (64 * 28, 64, 64 * 64, 64, 64, 1)
    W1, b1, W2, b2, w3, b3 = torch.split(w, sizes)
    out = []
    for r in range(len(off) - 1):
        v = s.records[off[r]:off[r + 1]][:, [B_LOGP, B_MAXP, B_TOPK, B_RHO]].double()
        v = v.sort(dim=0).values
        T, cols = v.size(0), []
        for a, b in LEVELS:
            i, rem = divmod(a * (T - 1), b)
            cols.append(v[i] + rem / b * (v[min(i + 1, T - 1)] - v[i]))
        out.append(torch.stack(cols, dim=1).reshape(-1))
    q = torch.stack(out)
    h = torch.relu(q @ W1.view(64, 28).T + b1)
    z = torch.relu(h @ W2.view(64, 64).T + b2) @ w3 + b3
    return q, z


def _exact_selective(s, q):
    keep = torch.isfinite(s.scores)
    x, y = s.scores[keep].double(), s.labels[keep].double()
    n, nf, P = s.scores.numel(), x.numel(), float(y.sum())
    k = min(int(math.floor(q * n + 0.5)), nf)
    order = torch.sort(x, descending=True).indices
    x, y = x[order], y[order]
    tau = float(x[k - 1]) if k else float("inf")
    ship = x >= tau
    n_ship = int(ship.sum())
    # tie groups: their correct answers spread evenly over their ranks
    _, group, count = torch.unique_consecutive(x, return_inverse=True, return_counts=True)
    hits = torch.zeros(count.numel(), dtype=torch.float64, device=DEV).scatter_add_(0, group, y)
    shipped = torch.cumsum((hits / count)[group], 0)
    below = (count - hits).sum() - torch.cumsum(count - hits, 0)
    pairs = float((hits * (below + 0.5 * (count - hits))).sum())
    N = nf - P
    nan = float("nan")
    ranks = torch.arange(1, nf + 1, dtype=torch.float64, device=DEV)
    return dict(tau=tau, n_finite=nf, k=k, n_ship=n_ship, n_pos=int(P),
                auroc=pairs / (P * N) if P and N else nan,
                auarc=float((shipped / ranks).mean()) if nf else nan,
                acc_shipped=float(y[ship].mean()) if n_ship else nan)


def exact(case, seed):
    c, kind = case, case["kind"]
    s = prepare(case, seed)
    if kind == "selective":
        return _exact_selective(s, c["q"])
    if kind in ("decode", "lm_decode"):
        slots, _, used = _trace(c)
        x = torch.cat(s.x)
        n, chosen = x.size(0), torch.cat(s.chosen)
        slots = torch.from_numpy(slots.reshape(-1)).to(DEV)
        groups = [torch.nonzero(slots == r)[:, 0] for r in range(used)]
        w = s.weight.double() if kind == "lm_decode" else None
        rec, _ = _exact_records(
            lambda a, b: x[a:b].double() if w is None else x[a:b].double() @ w.T, n, c["vocab"],
            chosen, 20)
        return _exact_pool(s, groups, rec)
    off = _offsets(_lengths(c)).tolist()
    rows = [slice(off[r], off[r + 1]) for r in range(len(off) - 1)]
    flags = torch.zeros(len(rows), dtype=torch.int32, device=DEV)
    if kind == "head":
        w = s.w.double()
        v = s.records[:, [B_LOGP, B_MAXP, B_TOPK, B_RHO]].double()
        z = torch.stack([_exact_head(v[r], w, c["layers"]) for r in rows])
        return dict(score=torch.sigmoid(z), ship=(z >= 0).to(torch.uint8), flags=flags)
    if kind == "quantile":
        q, z = _exact_quantile(s, off)
        return dict(summary=q, score=torch.sigmoid(z), ship=(z >= 0).to(torch.uint8), flags=flags)
    w = s.weight.double() if kind == "lm_features" else None
    rec, top2 = _exact_records(
        lambda a, b: s.x[a:b].double() if w is None else s.x[a:b].double() @ w.T, s.x.size(0),
        c["vocab"], s.chosen, c.get("topk", 20))
    for r in rows:
        T = r.stop - r.start
        rec[r, B_RHO] = torch.arange(1, T + 1, dtype=torch.float64, device=DEV) / T
    out = _exact_pool(s, rows, rec)
    if kind == "route":
        return out
    out.update(feat=rec, top2=top2.int(),
               row_flags=torch.zeros(len(rec), dtype=torch.int32, device=DEV))
    return out
