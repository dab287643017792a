"""The work a user has this library do, as measurable cases.

Every case draws a seeded random FST and accepted input strings on the GPU
(the laws of ``paper_1701_03038_gb300.synth``: Zipf or uniform labels,
lognormal or uniform out-degrees, Dirichlet weights, walks that end in a
final state), keeps the handle, plan or module a program would keep, and
runs one pass through the public entry points.  ``exact`` recomputes the
floating-point results with plain torch in float64.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1701_03038_gb300 import _lib, synth
from paper_1701_03038_gb300.autograd import LogZModule
from paper_1701_03038_gb300.fst import Fst

DEV = "cuda"

# FST shapes: the workloads of synth.CONFIGS.
SMALL = dict(states=1_000, isyms=50, arcs=20_000, law="uniform", alpha=1.0)
NLP = dict(states=50_000, isyms=10_000, arcs=5_000_000, law="zipf", alpha=0.5)
LARGE = dict(states=200_000, isyms=20_000, arcs=20_000_000, law="zipf", alpha=0.5)
CRF = dict(states=100_000, isyms=5_000, arcs=2_000_000, law="zipf", alpha=0.5)
SPEECH = dict(states=1_000_000, isyms=5_000, arcs=100_000_000, law="uniform", alpha=1.0)


def listed():
    return [
        # one short sentence on a small grammar: an interactive request, all latency
        dict(name="small_viterbi", kind="sentence_viterbi", block=True, strings=1, lo=50, hi=50, **SMALL),
        dict(name="small_posteriors", kind="sentence_fb", block=True, strings=1, lo=50, hi=50, **SMALL),
        # one sentence at a time on a translation-sized transducer, host arrays in and out
        dict(name="sentence_viterbi", kind="sentence_viterbi", block=False, strings=1, lo=35, hi=35, **NLP),
        dict(name="sentence_posteriors", kind="sentence_fb", block=False, strings=1, lo=35, hi=35, **NLP),
        # a test set decoded in one call
        dict(name="batch_viterbi", kind="batch_viterbi", strings=1_000, lo=10, hi=60, **NLP),
        # one EM iteration over a corpus: expected counts, then the M-step
        dict(name="batch_em", kind="batch_em", strings=1_000, lo=10, hi=60, **NLP),
        # bulk decoding and bulk posteriors of uneven strings on a 20M-arc transducer
        dict(name="bulk_viterbi", kind="batch_viterbi", strings=4_096, lo=5, hi=200, **LARGE),
        dict(name="bulk_posteriors", kind="batch_fb", strings=4_096, lo=5, hi=200, **LARGE),
        # a gradient step of CRF / HMM style training: weights in, log Z and d log Z / d weights out
        dict(name="train_step", kind="train", strings=1_024, lo=10, hi=100, **CRF),
        # speech-like: few, long strings on a 100M-arc graph, decoded and aligned by a kept plan
        dict(name="long_strings", kind="plan", strings=64, lo=1_000, hi=1_000, **SPEECH),
        # a recogniser's confusion network decoded and scored
        dict(name="lattice", kind="lattice", strings=1, lo=30, hi=30, alternatives=3, **NLP),
        # the weight of a long observation sequence under a dense HMM, by the parallel product over time
        dict(name="hmm_product", kind="hmm", hidden=63, isyms=6, length=1_000),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["sentence_viterbi", "sentence_fb", "batch_viterbi", "batch_em", "batch_fb", "train", "plan",
                       "lattice", "hmm"])
    if kind == "hmm":
        return dict(kind=kind, hidden=_log_int(rng, 4, 96), isyms=rng.randint(2, 32), length=_log_int(rng, 10, 1_000))
    if kind.startswith("sentence") and rng.random() < 0.5:
        q = _log_int(rng, 60, 8_000)
        n = _log_int(rng, 1, 200)
        m = rng.randint(8, 200)
        return dict(kind=kind, block=True, strings=1, lo=n, hi=n, states=q, isyms=m, arcs=q * rng.randint(8, 30) + 7,
                    law=rng.choice(["uniform", "zipf"]), alpha=rng.choice([0.5, 1.0]))
    if kind == "plan":
        q = _log_int(rng, 100_000, 1_000_000)
        n = _log_int(rng, 150, 1_000)
        return dict(kind=kind, strings=rng.randint(3, 64), lo=n - n // 4, hi=n, states=q, isyms=rng.randint(4_000, 6_000),
                    arcs=q * rng.randint(60, 100), law="uniform", alpha=1.0)
    q = _log_int(rng, 5_000, 200_000)
    degree = rng.randint(15, 100)
    m = degree * rng.randint(90, 200)
    c = dict(kind=kind, states=q, isyms=m, arcs=q * degree + rng.randint(0, 999), law="zipf", alpha=rng.choice([0.5, 1.0]))
    if kind == "lattice":
        n = _log_int(rng, 5, 30)
        return dict(c, states=min(q, 50_000), arcs=min(q, 50_000) * degree + 3, strings=1, lo=n, hi=n,
                    alternatives=rng.randint(1, 3))
    if kind.startswith("sentence"):
        n = _log_int(rng, 2, 100)
        return dict(c, block=False, strings=1, lo=n, hi=n)
    if kind == "train":
        q = _log_int(rng, 5_000, 100_000)
        degree = rng.randint(5, 20)
        return dict(c, states=q, isyms=degree * rng.randint(150, 300), arcs=q * degree + 11,
                    strings=_log_int(rng, 8, 1_024), lo=10, hi=_log_int(rng, 20, 100))
    c = dict(c, strings=_log_int(rng, 2, 4_096), lo=5, hi=_log_int(rng, 20, 200))
    while c["strings"] > 1 and work(c)["bytes"] > 3.5e8:  # at most the largest listed case's work
        c["strings"] = c["strings"] * 2 // 3
    return c


# ------------------------------------------------------------- inputs
def _pick(weights, u):
    """Indices drawn in proportion to integer weights from uniforms u (integer
    sums, so that a seed gives the same inputs every time)."""
    cdf = torch.cumsum(weights, 0)
    at = (u * int(cdf[-1])).long()
    return torch.searchsorted(cdf, at, right=True).clamp_(max=weights.numel() - 1)


def _draw_fst(case, seed):
    """Arc arrays (src, dst, ilabel, olabel int32; cost, start, final float32)
    in a shuffled caller order, and the same arcs grouped by source for the
    walks: (offsets [Q+1], dst, ilabel)."""
    g = torch.Generator(device=DEV).manual_seed(int(seed) * 2 + 1)
    q, a, m = case["states"], case["arcs"], case["isyms"]
    rand = lambda n: torch.rand(n, generator=g, device=DEV)  # noqa: E731
    if case["law"] == "zipf":
        deg = (torch.exp(torch.randn(q, generator=g, device=DEV)).clamp_(max=1e4) * 2.0 ** 20).long()
        src = _pick(deg, torch.rand(a - q, generator=g, device=DEV, dtype=torch.float64))
        src = torch.cat([torch.arange(q, device=DEV), src]).to(torch.int32)  # at least one arc each
        il = _pick(2 ** 40 // torch.arange(1, m + 1, device=DEV), rand(a).double()).to(torch.int32)
    else:
        src = torch.randint(0, q, (a,), generator=g, device=DEV, dtype=torch.int32)
        il = torch.randint(0, m, (a,), generator=g, device=DEV, dtype=torch.int32)
    src = torch.sort(src).values
    dst = torch.randint(0, q, (a,), generator=g, device=DEV, dtype=torch.int32)
    ol = torch.randint(0, m, (a,), generator=g, device=DEV, dtype=torch.int32)
    # Dirichlet(1 or 1/2) over each state's arcs from exponential or squared normal draws
    if case["alpha"] == 1.0:
        w = -torch.log1p(-rand(a))
    else:
        w = torch.randn(a, generator=g, device=DEV).square_()
    w = (w * 2.0 ** 30).long().clamp_(min=1)
    tot = torch.zeros(q, dtype=torch.int64, device=DEV).index_add_(0, src, w)
    w = torch.log(tot[src].double() / w.double()).float()
    off = torch.zeros(q + 1, dtype=torch.int64, device=DEV)
    torch.cumsum(torch.bincount(src, minlength=q), 0, out=off[1:])
    start = torch.full((q,), math.inf, device=DEV)
    start[0] = 0.0
    final = torch.full((q,), math.inf, device=DEV)
    final[torch.randperm(q, generator=g, device=DEV)[:max(1, q // 10)]] = 0.0
    perm = torch.randperm(a, generator=g, device=DEV)
    walk = (off, dst, il)
    arrs = tuple(x[perm] for x in (src, dst, il, ol, w)) + (start, final)
    return arrs, walk, g


def _draw_strings(case, walk, final, g):
    """Random walks from state 0 that end in a final state: (ids int32 [N],
    offsets int64 [B+1]) on the GPU; lengths spread evenly over [lo, hi]."""
    off, dst, il = walk
    B = case["strings"]
    n = case["lo"] + torch.randperm(B, generator=g, device=DEV) * (case["hi"] - case["lo"] + 1) // B
    T = int(n.max())
    out = torch.zeros(B, T, dtype=torch.int32, device=DEV)
    todo = torch.arange(B, device=DEV)
    tries = 48 if B > 64 else 1024
    for _ in range(200):
        if todo.numel() == 0:
            break
        k = todo.numel() * tries
        lens = n[todo].repeat_interleave(tries)
        state = torch.zeros(k, dtype=torch.int64, device=DEV)
        ok = torch.ones(k, dtype=torch.bool, device=DEV)
        syms = torch.zeros(k, T, dtype=torch.int32, device=DEV)
        for t in range(T):
            deg = off[state + 1] - off[state]
            go = (lens > t) & ok
            ok &= ~(go & (deg == 0))
            go &= ok
            arc = off[state] + (torch.rand(k, generator=g, device=DEV, dtype=torch.float64) * deg).long()
            arc = torch.where(go, arc, torch.zeros_like(arc))
            syms[:, t] = torch.where(go, il[arc], torch.zeros_like(il[arc]))
            state = torch.where(go, dst[arc].long(), state)
        ok &= torch.isfinite(final[state])
        ok = ok.view(-1, tries)
        hit = ok.any(1)
        first = torch.where(ok, torch.arange(tries, device=DEV), tries).min(1).values.clamp_(max=tries - 1)
        rows = torch.arange(todo.numel(), device=DEV) * tries + first
        out[todo[hit]] = syms[rows[hit]]
        todo = todo[~hit]
    else:
        raise RuntimeError("walks that never end in a final state")
    offsets = torch.zeros(B + 1, dtype=torch.int64, device=DEV)
    torch.cumsum(n, 0, out=offsets[1:])
    keep = torch.arange(T, device=DEV)[None, :] < n[:, None]
    return out[keep].contiguous(), offsets


def _lattice(case, ids, seed):
    """A confusion network over the string: at each position its symbol and
    random alternatives."""
    rng = np.random.default_rng(int(seed) + 77)
    frm, to, lab, w = [], [], [], []
    k = case["alternatives"]
    for t, a in enumerate(ids):
        for alt in range(k):
            frm.append(t)
            to.append(t + 1)
            lab.append(int(a) if alt == 0 else int(rng.integers(0, case["isyms"])))
            w.append(math.log(0.8 if alt == 0 else 0.2 / (k - 1)))
    return (len(ids) + 1, np.array(frm, np.int32), np.array(to, np.int32), np.array(lab, np.int32),
            np.array(w, np.float32))


def _hmm(case, seed):
    rng = np.random.default_rng(int(seed))
    k, v = case["hidden"], case["isyms"]
    pi = rng.dirichlet(np.ones(k))
    trans = rng.dirichlet(np.ones(k), size=k)
    emit = rng.dirichlet(np.ones(v), size=k)
    # the FST of synth.hmm_fst: a fresh start state, then the hidden states
    p0 = (pi[:, None] * emit).reshape(-1)
    p1 = (trans[:, :, None] * emit[None]).reshape(-1)
    src = np.concatenate([np.zeros(k * v, np.int32), np.repeat(np.arange(1, k + 1), k * v)]).astype(np.int32)
    dst = np.concatenate([np.repeat(np.arange(1, k + 1), v), np.tile(np.repeat(np.arange(1, k + 1), v), k)]).astype(np.int32)
    il = np.tile(np.arange(v), k + k * k).astype(np.int32)
    w = (-np.log(np.concatenate([p0, p1]))).astype(np.float32)
    start = np.full(k + 1, np.inf, np.float32)
    start[0] = 0.0
    final = np.zeros(k + 1, np.float32)
    final[0] = np.inf
    x = rng.integers(0, v, size=case["length"]).astype(np.int32)
    return synth.FstArrays(k + 1, v, v, src, dst, il, il, w, start, final), x


def _inputs(case, seed):
    arrs, walk, g = _draw_fst(case, seed)
    ids, off = _draw_strings(case, walk, arrs[6], g)
    return arrs, ids, off


def prepare(case, seed):
    kind = case["kind"]
    if kind == "hmm":
        fa, x = _hmm(case, seed)
        return dict(kind=kind, fst=Fst.from_arrays(fa), ids=x)
    arrs, ids, off = _inputs(case, seed)
    fst = Fst(case["states"], *arrs, case["isyms"], weight_kind="cost")
    s = dict(kind=kind, fst=fst, ids=ids, off=off)
    if kind.startswith("sentence"):
        s["ids"] = ids.cpu().numpy()
        if case["block"]:
            fst.set_plain_method(_lib.PLAIN_BLOCK)
        s["buf"] = torch.empty(case["arcs"], dtype=torch.float32, pin_memory=True).numpy()
    elif kind == "lattice":
        s["lat"] = _lattice(case, ids.cpu().numpy(), seed)
    elif kind == "train":
        s["module"] = LogZModule(fst, -arrs[4])
        s["plan"] = fst.plan(ids, off, flags=_lib.PLAN_NO_VITERBI | _lib.PLAN_SINGLE_WAVE)
    elif kind == "plan":
        s["plan"] = fst.plan(ids, off)
    del arrs
    return s


def run(s):
    kind, fst = s["kind"], s["fst"]
    if kind == "sentence_viterbi":
        score, path, olab, status = fst.viterbi(s["ids"])
        return dict(score=score, path=path, olabels=olab, status=status)
    if kind == "sentence_fb":
        logz, counts, status = fst.forward_backward(s["ids"], out=s["buf"])
        return dict(logz=logz, counts=counts, status=status)
    if kind == "batch_viterbi":
        return fst.viterbi_batch(s["ids"], s["off"])
    if kind == "batch_fb":
        return fst.forward_backward_batch(s["ids"], s["off"])
    if kind == "batch_em":
        r = fst.forward_backward_batch(s["ids"], s["off"])
        r["weights"] = fst.em_update(r["counts"], pseudo_count=0.01)
        return r
    if kind == "train":
        m = s["module"]
        m.theta.grad = None
        logz = m(s["plan"])
        loss = -logz.mean()
        loss.backward()
        return dict(logz=logz.detach(), loss=loss.detach(), grad=m.theta.grad)
    if kind == "plan":
        p = s["plan"]
        p.viterbi()
        p.forward_backward()
        return dict(scores=p.scores, paths=p.paths, olabels=p.olabels, logz=p.logz, counts=p.counts, status=p.status)
    if kind == "lattice":
        score, edges, arcs, st = fst.lattice_viterbi(*s["lat"])
        logz, counts, post, st2 = fst.lattice_forward_backward(*s["lat"])
        return dict(score=score, edges=edges, arcs=arcs, status=[st, st2], logz=logz, counts=counts, edge_post=post)
    if kind == "hmm":
        logz, best, status = fst.prefix_log_z(s["ids"])
        return dict(logz=logz, best=best, status=status)
    raise ValueError(kind)


# --------------------------------------------------------------- work
def _live_arcs(case):
    """Arcs out of live states that a pass over the strings meets, expected
    under the case's laws: a walk's frontier F meets F d p_w arcs on symbol w
    and they reach Q (1 - exp(-F d p_w / Q)) states; the walk's own arc is
    always among them."""
    q, a, m = case["states"], case["arcs"], case["isyms"]
    rng = np.random.default_rng(0)
    p = np.full(m, 1.0 / m) if case["law"] == "uniform" else 1.0 / np.arange(1, m + 1)
    p = p / p.sum()
    sims, steps = 512, (case["lo"] + case["hi"]) // 2
    cdf = np.cumsum(p)
    f = np.ones(sims)
    tot = 0.0
    for _ in range(steps):
        w = np.minimum(np.searchsorted(cdf, rng.random(sims)), m - 1)
        push = np.maximum(1.0, f * (a / q) * p[w])
        tot += float(push.mean())
        f = np.maximum(1.0, q * -np.expm1(-push / q))
    return tot * case["strings"], steps * case["strings"]


def work(case):
    kind = case["kind"]
    if kind == "hmm":
        k, n = case["hidden"] + 1, case["length"]
        # a matrix-vector sweep of both semirings, and the matrices
        return dict(bytes=12 * k * k * case["isyms"] + 4 * n + 12, flops=4 * n * k * k)
    live, tokens = _live_arcs(case)
    b, a = case["strings"], case["arcs"]
    vit = dict(bytes=12 * live + 12 * tokens + 8 * b, flops=2 * live)
    # forward, backward and the posteriors of each live arc; counts of every arc out
    fb = dict(bytes=12 * live + 4 * tokens + 12 * b + 4 * a, flops=12 * live)
    if kind in ("sentence_viterbi", "batch_viterbi"):
        return vit
    if kind in ("sentence_fb", "batch_fb"):
        return fb
    if kind == "batch_em":
        return dict(bytes=fb["bytes"] + 8 * a, flops=fb["flops"] + 4 * a)
    if kind == "train":
        return dict(bytes=fb["bytes"] + 4 * a, flops=fb["flops"])
    if kind == "plan":
        return dict(bytes=vit["bytes"] + fb["bytes"], flops=vit["flops"] + fb["flops"])
    # lattice: every edge meets the live arcs of its symbol in both calls
    k = case["alternatives"]
    return dict(bytes=k * (vit["bytes"] + 12 * live) + 4 * a, flops=k * (vit["flops"] + fb["flops"]))


# -------------------------------------------------------------- exact
def _lse(val, inv, count):
    """Per-group max and log-sum-exp of val (groups inv in [0, count))."""
    mx = torch.full((count,), -math.inf, dtype=torch.float64, device=DEV).scatter_reduce_(0, inv, val, "amax")
    ref = torch.where(torch.isinf(mx), torch.zeros_like(mx), mx)
    s = torch.zeros(count, dtype=torch.float64, device=DEV).index_add_(0, inv, torch.exp(val - ref[inv]))
    return mx, ref + torch.log(s)


class _Exact:
    """Viterbi scores, log Z and expected counts of a batch in float64, over
    the states that some path reaches."""

    def __init__(self, case, arrs):
        src, dst, il, _, w, start, final = arrs
        self.q, self.a = case["states"], case["arcs"]
        key, order = torch.sort(il.long() * self.q + src.long())
        self.key, self.id = key, order
        self.dst = dst[order].long()
        self.theta = -w[order].double()
        self.final = -final.double()

    def run(self, ids, off, want_vit, want_fb, gw=None):
        q, ids = self.q, ids.long()
        n = off[1:] - off[:-1]
        B, T = n.numel(), int(n.max())
        b = torch.arange(B, device=DEV)
        st = torch.zeros(B, dtype=torch.int64, device=DEV)
        alpha = torch.zeros(B, dtype=torch.float64, device=DEV)
        vit = alpha.clone()
        best = torch.full((B,), -math.inf, dtype=torch.float64, device=DEV)
        ends_b, ends_v, steps, fronts = [], [], [], []
        for t in range(T + 1):
            end = n[b] == t
            fin = self.final[st]
            if bool(end.any()):
                if want_vit:
                    best.scatter_reduce_(0, b[end], (vit + fin)[end], "amax")
                ends_b.append(b[end])
                ends_v.append((alpha + fin)[end])
            fronts.append((b, st, alpha, torch.where(end, fin, torch.full_like(fin, -math.inf))))
            if t == T:
                break
            live = torch.nonzero(n[b] > t).view(-1)
            k = ids[off[b[live]] + t] * q + st[live]
            lo = torch.searchsorted(self.key, k)
            cnt = torch.searchsorted(self.key, k, right=True) - lo
            row = torch.repeat_interleave(torch.arange(live.numel(), device=DEV), cnt)
            arc = torch.arange(row.numel(), device=DEV) - (torch.cumsum(cnt, 0) - cnt)[row] + lo[row]
            row = live[row]
            uniq, inv = torch.unique(b[row] * q + self.dst[arc], return_inverse=True)
            if want_vit:
                vv = vit[row] + self.theta[arc]
                vit = torch.full((uniq.numel(),), -math.inf, dtype=torch.float64, device=DEV)
                vit.scatter_reduce_(0, inv, vv, "amax")
            if want_fb:
                steps.append((row, arc, inv))
                alpha = _lse(alpha[row] + self.theta[arc], inv, uniq.numel())[1]
            else:
                alpha = torch.zeros(uniq.numel(), dtype=torch.float64, device=DEV)
                fronts[-1] = None
            b, st = uniq // q, uniq % q
        if not want_fb:
            return best, None, None
        logz = _lse(torch.cat(ends_v), torch.cat(ends_b), B)[1]
        counts = torch.zeros(self.a, dtype=torch.float64, device=DEV)
        beta = fronts[T][3]
        for t in range(T - 1, -1, -1):
            bb, _, al, fin = fronts[t]
            row, arc, inv = steps[t]
            u = self.theta[arc] + beta[inv]
            g = torch.exp(al[row] + u - logz[bb[row]])
            counts.index_add_(0, self.id[arc], g if gw is None else g * gw)
            sub = _lse(u, row, al.numel())[1] if row.numel() else torch.full_like(fin, -math.inf)
            beta = torch.maximum(fin, sub)
            fronts[t + 1] = steps[t] = None
        return best, logz, counts


def _exact_lattice(case, arrs, lat):
    q, a = case["states"], case["arcs"]
    src, dst, il, _, w, start, final = arrs
    order = torch.sort(il.long()).indices
    ils, src, dst, th = il.long()[order], src.long()[order], dst.long()[order], -w[order].double()
    n, frm, to, lab, lw = lat
    neg = lambda: torch.full((q,), -math.inf, dtype=torch.float64, device=DEV)  # noqa: E731
    lo = torch.searchsorted(ils, torch.from_numpy(lab).long().to(DEV)).tolist()
    hi = torch.searchsorted(ils, torch.from_numpy(lab).long().to(DEV), right=True).tolist()
    edges = range(len(frm))
    alpha, vit = [-start.double()], [-start.double()]
    for v in range(1, n):
        val, vv, tgt = [], [], []
        for e in edges:
            if to[e] == v:
                sl = slice(lo[e], hi[e])
                val.append(alpha[frm[e]][src[sl]] + float(lw[e]) + th[sl])
                vv.append(vit[frm[e]][src[sl]] + th[sl] + float(lw[e]))
                tgt.append(dst[sl])
        tgt = torch.cat(tgt)
        alpha.append(_lse(torch.cat(val), tgt, q)[1])
        vit.append(neg().scatter_reduce_(0, tgt, torch.cat(vv), "amax"))
    fin = -final.double()
    logz = torch.logsumexp(alpha[-1] + fin, 0)
    beta = [None] * n
    beta[-1] = fin
    counts = torch.zeros(a, dtype=torch.float64, device=DEV)
    post = torch.zeros(len(frm), dtype=torch.float64, device=DEV)
    for u in range(n - 2, -1, -1):
        val, tgt = [], []
        for e in edges:
            if frm[e] == u:
                sl = slice(lo[e], hi[e])
                x = float(lw[e]) + th[sl] + beta[to[e]][dst[sl]]
                val.append(x)
                tgt.append(src[sl])
                g = torch.exp(alpha[u][src[sl]] + x - logz)
                counts.index_add_(0, order[sl], g)
                post[e] = g.sum()
        beta[u] = _lse(torch.cat(val), torch.cat(tgt), q)[1]
    return dict(score=(vit[-1] + fin).max(), edges=None, arcs=None, status=None, logz=logz, counts=counts, edge_post=post)


def _exact_hmm(fa, x):
    q = fa.num_states
    th = -fa.weight.astype(np.float64)
    mats = np.full((fa.num_isyms, q, q), -np.inf)
    mats[fa.ilabel, fa.src, fa.dst] = th
    alpha = -fa.start_weight.astype(np.float64)
    vit = alpha.copy()
    with np.errstate(divide="ignore", invalid="ignore"):
        for a in x:
            z = alpha[:, None] + mats[a]
            m = z.max(0)
            r = np.where(np.isinf(m), 0.0, m)
            alpha = r + np.log(np.exp(z - r).sum(0))
            vit = (vit[:, None] + mats[a]).max(0)
        fin = -fa.final_weight.astype(np.float64)
        z = alpha + fin
        logz = z.max() + math.log(np.exp(z - z.max()).sum())
    return dict(logz=float(logz), best=float((vit + fin).max()), status=None)


def exact(case, seed):
    kind = case["kind"]
    if kind == "hmm":
        fa, x = _hmm(case, seed)
        r = _exact_hmm(fa, x)
        return dict(logz=np.float64(r["logz"]), best=np.float64(r["best"]), status=None)
    arrs, ids, off = _inputs(case, seed)
    if kind == "lattice":
        return _exact_lattice(case, arrs, _lattice(case, ids.cpu().numpy(), seed))
    e = _Exact(case, arrs)
    vit = kind in ("sentence_viterbi", "batch_viterbi", "plan")
    fb = kind not in ("sentence_viterbi", "batch_viterbi")
    best, logz, counts = e.run(ids, off, vit, fb, gw=-1.0 / case["strings"] if kind == "train" else None)
    if kind == "sentence_viterbi":
        return dict(score=best, path=None, olabels=None, status=None)
    if kind == "sentence_fb":
        return dict(logz=logz, counts=counts, status=None)
    if kind == "batch_viterbi":
        return dict(scores=best, paths=None, olabels=None, status=None)
    if kind == "batch_fb":
        return dict(logz=logz, counts=counts, status=None)
    if kind == "batch_em":
        src = arrs[0].long()
        c = counts + 0.01
        tot = torch.zeros(case["states"], dtype=torch.float64, device=DEV).index_add_(0, src, c)
        return dict(logz=logz, counts=counts, status=None, weights=torch.log(c / tot[src]))
    if kind == "train":
        return dict(logz=logz, loss=-logz.mean(), grad=counts)
    return dict(scores=best, paths=None, olabels=None, logz=logz, counts=counts, status=None)
