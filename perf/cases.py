"""Cases of the verification library's main path, measured through its public
entry points.

One pass is one verification call over a batch of B sequences: K draft
branches of L tokens each, checked against the target model's logits.  The
shapes are those of the repository's own workloads (a 4k test vocabulary,
32k, 50k, 128k and 152k rows; K = 2..8 branches, L = 4..8 tokens, batches of
1 to 1024 sequences), plus odd sizes around them.  Inputs are seeded
synthetic logits on a draft tree: target rows are scaled normals (optionally
with a boosted head), draft rows are the target's plus normal noise, each
branch's token is drawn from its own draft distribution, branches with equal
prefixes share rows.

A call reads only the rows its walk visits, so the bytes of a pass depend on
how long the drafts survive; `work` uses the case's mean survival rate per
depth, as counted on these inputs.

Every case returns all a call writes: the tokens, the accepted lengths and
the per-depth diagnostics (target probability and importance law at the
intermediate token, residual mass, the intermediate token).  A decision whose
uniform lies within rounding of its threshold may fall either way in a
correct implementation: it moves the values after it, so a small share of the
tokens may differ.
"""
import math

import numpy as np
import torch

from paper_2410_18234_gb300 import mds

VERIFY_SEED = 1
STORAGE = {"f32": torch.float32, "bf16": torch.bfloat16}


# ------------------------------------------------------------------ cases


def _case(name, scheme, B, K, L, V, **kw):
    c = {"name": name, "scheme": scheme, "B": B, "K": K, "L": L, "V": V, "dtype": "bf16", "models": 1,
         "scale": 4.0, "sigma": 1.0, "sigma2": 1.0, "t_target": 1.0, "t_draft": 1.0, "t_draft2": 1.0,
         "boost_n": 0, "boost": 0.0, "per_seq": False, "top_k": 0, "omega0": 20, "acc_prob": 0, "entry": "device",
         "survive": 0.75}
    c.update(kw)
    return c


# the distributions of the repository's workloads
TINY = {"dtype": "f32", "scale": 3.0, "sigma": 0.7}
HEADED = {"scale": 4.0, "sigma": 1.0, "t_draft": 1.2, "boost_n": 50, "boost": 6.0}
TWO_MODELS = {"models": 2, "scale": 4.0, "sigma": 0.5, "sigma2": 1.5, "t_draft": 1.0, "t_draft2": 2.0}
PEAKED = {"scale": 5.0, "sigma": 0.8, "t_target": 0.7, "t_draft": 0.7}
SERVING = {"scale": 4.0, "per_seq": True}    # draft quality and temperature differ per sequence


def listed():
    return [
        # a handful of sequences on a test-sized vocabulary: latency and launches
        _case("tiny-single", "single", 4, 2, 4, 4096, survive=0.65, **TINY),
        # one interactive user on a large vocabulary
        _case("one-wis", "WIS", 1, 4, 4, 128256, survive=0.69, **PEAKED),
        # classical importance sampling, a mid-sized batch
        _case("llama2-32k-is", "IS", 64, 4, 5, 32000, survive=0.81, **HEADED),
        # logits that live in pinned host memory (the host entry point, copies included)
        _case("llama2-32k-wis-host", "WIS", 64, 4, 5, 32000, entry="host", survive=0.73, **HEADED),
        # two draft models, with the acceptance probability of every depth
        _case("two-models-50k-wis-acc", "WIS", 128, 2, 4, 50272, acc_prob=1, survive=0.76, **TWO_MODELS),
        # the sequential-rejection baseline on the same batch
        _case("two-models-50k-spectr", "SpecTr", 128, 2, 4, 50272, survive=0.83, **TWO_MODELS),
        # rows of an odd length in 32 bits: no aligned 16-byte units
        _case("odd-32003-f32-single", "single", 24, 3, 4, 32003, dtype="f32", survive=0.68, scale=4.0, sigma=1.0),
        # the headline batch: weighted importance sampling, its truncated
        # alphabet, and rows restricted to their ten largest logits
        _case("llama3-128k-wis", "WIS", 256, 8, 4, 128256, survive=0.81, **PEAKED),
        _case("llama3-128k-wis0", "WIS0", 256, 8, 4, 128256, survive=0.79, **PEAKED),
        _case("llama3-128k-top10-wis", "WIS", 256, 8, 4, 128256, top_k=10, survive=0.85, **PEAKED),
        # the largest batches of a serving sweep
        _case("serving-152k-single", "single", 1024, 4, 8, 151936, survive=0.73, **SERVING),
        _case("serving-152k-spectr", "SpecTr", 1024, 4, 8, 151936, survive=0.76, **SERVING),
    ]


def draw(rng):
    """A case of the same ranges: batches of 1 to 1024, rows of 4k to 152k
    logits, odd lengths among them, every scheme, both storage types."""
    scheme, top_k = rng.choice([("single", 0), ("WIS", 0), ("WIS", 0), ("WIS0", 0), ("SpecTr", 0), ("IS", 0),
                                ("WIS", 5), ("WISsort", 10), ("single", 10), ("SpecTr", 10)])
    V = int(round(math.exp(rng.uniform(math.log(4096), math.log(151936)))))
    V = V | 1 if rng.random() < 0.3 else max(4096, V // 16 * 16)
    B = int(round(math.exp(rng.uniform(0.0, math.log(1024)))))
    K, L = rng.choice([2, 2, 3, 4, 4, 8]), rng.choice([2, 3, 4, 5, 8])
    kw = dict(rng.choice([TINY, HEADED, TWO_MODELS, PEAKED, SERVING]))
    kw["dtype"] = "f32" if rng.random() < 0.25 else "bf16"
    kw["entry"] = "host" if rng.random() < 0.1 else "device"
    kw["acc_prob"] = 1 if scheme != "WIS0" and rng.random() < 0.15 else 0
    kw["omega0"] = rng.choice([10, 20, 40])
    # no more than the largest listed case: logits held, and for classical
    # importance sampling the tokens it integrates over
    held = (3e8 if kw["entry"] == "host" else 6e9) / (K * (2 * L + 1) * (4 if kw["dtype"] == "f32" else 2))
    B = max(1, min(B, int(held / V), int(6.5e6 / V) if scheme == "IS" else B))
    c = _case("", scheme, B, K, L, V, top_k=top_k, **kw)
    del c["name"]
    return c


# ------------------------------------------------------------------ inputs


def _model_ids(case):
    return [k % case["models"] for k in range(case["K"])]


def _inputs(case, seed, dev):
    """Logits, draft tokens and temperatures of the case's batch."""
    B, K, L, V = case["B"], case["K"], case["L"], case["V"]
    st = STORAGE[case["dtype"]]
    g = torch.Generator(device=dev)
    g.manual_seed(int(seed))
    mids = torch.tensor(_model_ids(case), device=dev)
    temps = torch.empty(B, 1 + K, dtype=torch.float32, device=dev)
    if case["per_seq"]:
        temps[:] = (0.5 + torch.rand(B, generator=g, device=dev))[:, None]
        sig = torch.tensor([0.3, 1.0, 2.0], device=dev)[torch.arange(B, device=dev) % 3][:, None].expand(B, K)
    else:
        temps[:, 0] = case["t_target"]
        temps[:, 1:] = torch.where(mids == 0, case["t_draft"], case["t_draft2"]).float()
        sig = torch.where(mids == 0, case["sigma"], case["sigma2"]).float()[None].expand(B, K)
    target = torch.empty(B, K, L + 1, V, dtype=st, device=dev)
    drafts = torch.empty(K, B, L, V, dtype=st, device=dev)
    tokens = torch.empty(B, K, L, dtype=torch.int32, device=dev)
    same = torch.ones(B, K, K, dtype=torch.bool, device=dev)   # branches with equal prefixes so far
    same_model = (mids[:, None] == mids[None, :])[None]
    ar = torch.arange(K, device=dev)

    def rows(x, rep):
        return torch.gather(x, 1, rep[:, :, None].expand(B, K, V))

    for j in range(L + 1):
        rep_t = torch.where(same, ar[None, None], K).amin(2)
        t32 = torch.randn(B, K, V, generator=g, device=dev).mul_(case["scale"])
        if case["boost_n"]:
            top = torch.topk(t32, case["boost_n"], dim=2).indices
            t32.scatter_add_(2, top, torch.full(top.shape, case["boost"], device=dev))
        t32 = rows(t32, rep_t)
        target[:, :, j] = t32.to(st)
        if j == L:
            break
        rep_d = torch.where(same & same_model, ar[None, None], K).amin(2)
        d = rows(t32 + sig[:, :, None] * torch.randn(B, K, V, generator=g, device=dev), rep_d).to(st)
        del t32
        drafts[:, :, j] = d.permute(1, 0, 2)
        d = d.float()
        if case["top_k"]:
            # drafts come from the restricted rows (ties: the lower id), as the caller of a top-k run draws them
            keep = _top_ids(d, case["top_k"])
            score = torch.full_like(d, -math.inf).scatter_(2, keep, torch.gather(d, 2, keep))
        else:
            score = d
        score = score / temps[:, 1:, None]
        score -= torch.rand(B, K, V, generator=g, device=dev).clamp_(1e-12).log_().neg_().log_()
        tok = score.argmax(2)
        del score, d
        tokens[:, :, j] = tok.int()
        same &= tok[:, :, None] == tok[:, None, :]
    return target, drafts, tokens, temps


def _top_ids(x, k):
    """Ids of the k largest values of each row, ties to the lower id."""
    bits = x.float().contiguous().view(torch.int32).long()
    order = torch.where(bits < 0, -(bits & 0x7fffffff), bits)
    key = order * (1 << 25) - torch.arange(x.shape[-1], device=x.device)
    return torch.topk(key, min(k, x.shape[-1]), dim=-1).indices


def prepare(case, seed):
    B, K, L, V = case["B"], case["K"], case["L"], case["V"]
    dev = torch.device("cuda", 0)
    target, drafts, tokens, temps = _inputs(case, seed, dev)
    drafts = list(drafts)
    host = case["entry"] == "host"
    if host:
        target, tokens, temps = (x.cpu().pin_memory() for x in (target, tokens, temps))
        drafts = [d.cpu().pin_memory() for d in drafts]
    # a program keeps its outputs' buffers; depths a walk does not reach stay as they are
    out = [torch.zeros(B, L + 1, dtype=torch.int32), torch.zeros(B, dtype=torch.int32), torch.zeros(B, L + 1, 4)]
    out = [x.pin_memory() if host else x.to(dev) for x in out]
    v = mds.Verifier(B, K, L, V, dtype=case["dtype"], device=0, omega0=case["omega0"], acc_prob=case["acc_prob"],
                     top_k=case["top_k"])
    d = out[2]
    results = {"tokens": out[0], "accepted": out[1], "target_prob": d[:, :, 0], "importance_prob": d[:, :, 1],
               "residual": d[:, :, 2], "intermediate": d[:, :, 3]}
    return {"call": v.verify_host if host else v.verify, "verifier": v, "scheme": case["scheme"],
            "args": (target, drafts, _model_ids(case), tokens, temps), "out": tuple(out), "results": results}


def run(state):
    state["call"](*state["args"], state["scheme"], VERIFY_SEED, out=state["out"])
    return state["results"]


def work(case):
    """The rows the walk visits, each read once: at every verified depth the
    target's and one per draft model (one draft row for single; for the
    truncated alphabet the target's only, and the drafts at Omega_0), at the
    end of a fully accepted walk the target's.  Operations: one exponential,
    a multiply-add and a comparison per logit, as four."""
    B, K, L, V, a = case["B"], case["K"], case["L"], case["V"], case["survive"]
    es = 4 if case["dtype"] == "f32" else 2
    depths = sum(a ** j for j in range(L))
    per_depth = {"single": 2, "WIS0": 1}.get(case["scheme"], 1 + case["models"])
    rows = B * (depths * per_depth + a ** L)
    io = 4 * B * (K * L + 1 + K + 5 * (L + 1) + 1)
    return {"bytes": rows * V * es + io, "flops": 4.0 * rows * V}


def tolerance(case):
    # Measured against `exact` over 64 cases of these ranges: probabilities,
    # importance laws and residual masses to at most 5e-7 (2-norm) and 3e-6
    # (one value).  Two schemes decide on ties besides.  On rows of a few
    # tokens the weighted stage's flow is often saturated exactly, and a
    # residual next to its threshold counts or not (5e-4 seen).  Omega_0 is
    # cut at equal 16-bit logits, where the candidate list may certify fewer
    # tokens (status bit MDS_ST_OMEGA0; 5e-3 seen).  Whole values: a token
    # drawn within rounding of a boundary of its distribution's running sum,
    # a few in ten thousand on broad rows.
    if case["scheme"] == "WIS0":
        return {"rel": 2e-2, "max": 0.9, "differ": 1e-2}
    if case["top_k"] and case["scheme"] in ("WIS", "WISsort"):
        return {"rel": 2e-3, "max": 0.1, "differ": 2e-3}
    return {"rel": 1e-5, "max": 1e-4, "differ": 2e-3}


# ------------------------------------------------------------------ 64-bit values


def _uniform(b, j, draw):
    """Philox4x32-10 (Salmon et al., SC'11): counter (b, j, draw, 0), key (seed, 0); word 0 as a 24-bit uniform."""
    m32 = np.uint64(0xFFFFFFFF)
    b = np.asarray(b, dtype=np.uint64)
    c = [b, np.full_like(b, j), np.full_like(b, draw), np.zeros_like(b)]
    k0, k1 = VERIFY_SEED & 0xFFFFFFFF, VERIFY_SEED >> 32
    for _ in range(10):
        p0, p1 = np.uint64(0xD2511F53) * c[0], np.uint64(0xCD9E8D57) * c[2]
        c = [(p1 >> np.uint64(32)) ^ c[1] ^ np.uint64(k0), p1 & m32, (p0 >> np.uint64(32)) ^ c[3] ^ np.uint64(k1),
             p0 & m32]
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    return (c[0] >> np.uint64(8)).astype(np.float64) * 2.0 ** -24


def _pair_flow(q, a, b, a2, b2):
    """A stage on its s free tokens: the maximum flow of the pair masses onto
    the demands max(0, q - base), first every pair in order to its own
    tokens, then along shortest paths; leftovers are split in halves.
    Returns the tokens' law and the weight of the lower token per pair."""
    s = len(q)
    base = a * b + a * b2 + b * a2
    need = np.maximum(0.0, q - base)
    eps = 1e-6 * float((q + base).sum())
    pairs = [(i, k) for i in range(s) for k in range(i + 1, s)]
    mass = {e: a[e[0]] * b[e[1]] + a[e[1]] * b[e[0]] for e in pairs}
    left = dict(mass)
    given = {(e, t): 0.0 for e in pairs for t in e}
    edge = {(u, v): (min(u, v), max(u, v)) for u in range(s) for v in range(s) if u != v}
    for e in pairs:
        for t in e:
            if left[e] > eps and need[t] > eps:
                d = min(left[e], need[t])
                given[e, t] += d
                left[e] -= d
                need[t] -= d
    for _ in range(4096):
        source = {}
        for e in pairs:
            if left[e] > eps:
                for t in e:
                    source.setdefault(t, e)
        parent, layer = {t: None for t in source}, sorted(source)
        sink = next((t for t in layer if need[t] > eps), None)
        while sink is None and layer:
            nxt = []
            for u in layer:
                for v in range(s):
                    if v not in parent and given.get((edge.get((u, v)), u), 0.0) > eps:
                        parent[v] = u
                        nxt.append(v)
            layer = sorted(nxt)
            sink = next((t for t in layer if need[t] > eps), None)
        if sink is None:
            break
        path = [sink]
        while parent[path[-1]] is not None:
            path.append(parent[path[-1]])
        path.reverse()
        hops = [(edge[u, v], u, v) for u, v in zip(path, path[1:])]
        e0 = source[path[0]]
        d = min([left[e0], need[sink]] + [given[e, u] for e, u, _ in hops])
        left[e0] -= d
        given[e0, path[0]] += d
        for e, u, v in hops:
            given[e, u] -= d
            given[e, v] += d
        need[sink] -= d
    law, low = base.copy(), {}
    for e in pairs:
        for t in e:
            law[t] += given[e, t] + 0.5 * left[e]
        low[e] = (given[e, e[0]] + 0.5 * left[e]) / mass[e] if mass[e] > 0 else 0.5
    return law, low


def _pick(om, low, x, y, u, earlier=None):
    """A stage's output for the inputs x, y: by the pair's weight inside om,
    the one inside om, otherwise a fair coin or the key order's earlier."""
    if x == y:
        return x
    where = {int(t): i for i, t in enumerate(om)}
    if x in where and y in where:
        i, k = where[x], where[y]
        w = low[min(i, k), max(i, k)]
        return x if u < (w if i < k else 1.0 - w) else y
    if x in where or y in where:
        return x if x in where else y
    if earlier is not None:
        return x if earlier(x, y) else y
    return x if u < 0.5 else y


def _stages(q, rows, X, mrow, nv, ids, j, sort_rule, s=5):
    """The pairwise weighted stages on [n, V] rows: the last stage's token and law."""
    n, V = q.shape
    law = torch.stack([rows[m][i] for i, m in enumerate(mrow[:, 0])])
    Y = X[:, 0].copy()
    for m in range(1, X.shape[1]):
        sub = np.flatnonzero(nv > m)
        if not len(sub):
            break
        ts = torch.as_tensor(sub, device=q.device)
        a, qq = law[ts], q[ts]
        b = torch.stack([rows[mrow[i, m]][i] for i in sub])
        key, order = torch.sort(qq - a * b, dim=1, descending=True, stable=True)
        om = order[:, :min(s, V)].sort(1).values
        get = lambda x: torch.gather(x, 1, om).cpu().numpy()  # noqa: E731
        oq, oa, ob = get(qq), get(a), get(b)
        rest = torch.ones_like(a).scatter_(1, om, 0.0)
        A2, B2 = (a * rest).sum(1), (b * rest).sum(1)
        new = 0.5 * (a * B2[:, None] + b * A2[:, None])
        rank = None
        if sort_rule:
            tail = order[:, min(s, V):]
            at, bt = torch.gather(a, 1, tail), torch.gather(b, 1, tail)
            after = lambda x: x.flip(1).cumsum(1).flip(1) - x  # noqa: E731
            new.scatter_(1, tail, at * bt + bt * after(at) + at * after(bt))
            rank = torch.empty_like(order).scatter_(1, order, torch.arange(V, device=q.device).expand(len(sub), V))
        A2, B2, om_h = A2.cpu().numpy(), B2.cpu().numpy(), om.cpu().numpy()
        us = _uniform(ids[sub], j, m - 1)
        vals = np.empty_like(oq)
        for r, i in enumerate(sub):
            vals[r], low = _pair_flow(oq[r], oa[r], ob[r], A2[r], B2[r])
            earlier = (lambda x, y, r=r: bool(rank[r, x] < rank[r, y])) if sort_rule else None
            Y[i] = _pick(om_h[r], low, int(Y[i]), int(X[i, m]), us[r], earlier)
        new.scatter_(1, om, torch.as_tensor(vals, device=q.device))
        law[ts] = new
    return Y, law


def _classical(q, rows, X, mrow, nv, ids, j, h=0.25):
    """Classical importance sampling: the chosen token and the law of the
    choice, by the Laplace identity 1/c = int exp(-t c) dt on a grid in ln t."""
    n, V = q.shape
    dev = q.device
    cnt = np.stack([((mrow == m) & (np.arange(X.shape[1])[None] < nv[:, None])).sum(1) for m in range(len(rows))], 1)
    rho = [q / r for r in rows]
    used = [torch.as_tensor(cnt[:, m] > 0, device=dev) for m in range(len(rows))]
    lo = min(float(r[u].min()) for r, u in zip(rho, used) if bool(u.any()))
    hi = max(float(r[u].max()) for r, u in zip(rho, used) if bool(u.any()))
    ct = torch.as_tensor(cnt, device=dev, dtype=torch.float64)
    acc = torch.zeros_like(q)
    for g in range(math.floor((-math.log(X.shape[1] * hi) - 40) / h), math.ceil(math.log(40 / lo) / h) + 1):
        t = math.exp(g * h)
        e = [torch.exp(-t * r) for r in rho]
        M = torch.stack([(p * x).sum(1) for p, x in zip(rows, e)], 1)
        for m in range(len(rows)):
            power = ct.clone()
            power[:, m] -= 1
            w = h * t * ct[:, m] * torch.where(ct[:, m] > 0, torch.prod(M ** power.clamp(min=0), 1), 0.0)
            acc.addcmul_(w[:, None].expand_as(q), e[m])
    law = q * acc
    Y = X[:, 0].copy()
    u = _uniform(ids, j, 0)
    for i in range(n):
        if nv[i] < 2:
            law[i] = rows[mrow[i, 0]][i]
            continue
        r = np.cumsum([float(rho[mrow[i, k]][i, X[i, k]]) for k in range(nv[i])])
        Y[i] = X[i, min(int(np.searchsorted(r, u[i] * r[-1], side="right")), nv[i] - 1)]
    return Y, law


def _small_alphabet(q, rows, X, mrow, nv, ids, j, M):
    """The truncated alphabet: per sequence the inner step on the target's M
    largest tokens, then keep its token or draw outside.  Returns the output
    token (-1: draw outside) and the diagnostics, and the mask to draw from."""
    n, V = q.shape
    val, idx = torch.topk(q, min(M + 1, V), dim=1)
    inside = q > val[:, M:M + 1] if M < V else torch.ones_like(q, dtype=torch.bool)
    Z, dg = np.full(n, -1), np.zeros((n, 4))
    u = {d: _uniform(ids, j, d) for d in [16, 32, 34] + list(range(X.shape[1]))}
    val, idx = val.cpu().numpy(), idx.cpu().numpy()
    for i in range(n):
        om = np.sort(idx[i][val[i] > val[i][M]]) if M < V else np.arange(V)
        dg[i, 3] = -1
        if not len(om):
            continue
        t = torch.as_tensor(om, device=q.device)
        qi = q[i, t].cpu().numpy()
        pa = qi.sum()
        qt = qi / pa
        where = {int(x): k for k, x in enumerate(om)}
        kept = [(where[int(X[i, k])], mrow[i, k]) for k in range(nv[i]) if int(X[i, k]) in where]
        sub = {m: rows[m][i, t].cpu().numpy() for m in {m for _, m in kept}}
        sub = {m: p / p.sum() for m, p in sub.items()}

        def cdf(w, uu):
            c = np.cumsum(w)
            return min(int(np.searchsorted(c, uu * c[-1], side="right")), len(w) - 1)

        if not kept:
            y = cdf(qt, u[32][i])
        else:
            y, law = kept[0][0], sub[kept[0][1]]
            for m in range(1, len(kept)):
                b = sub[kept[m][1]]
                o = np.sort(np.lexsort((np.arange(len(om)), -(qt - law * b)))[:5])
                r = np.ones(len(om), dtype=bool)
                r[o] = False
                A2, B2 = law[r].sum(), b[r].sum()
                x, low = _pair_flow(qt[o], law[o], b[o], A2, B2)
                y = _pick(o, low, y, kept[m][0], u[m - 1][i])
                law = 0.5 * (law * B2 + b * A2)
                law[o] = x
            dg[i] = qt[y], law[y], 0.0, om[y]
            if not u[16][i] < min(1.0, qt[y] / law[y] if law[y] > 0 else 1.0):
                r = np.maximum(0.0, qt - law)
                dg[i, 2] = r.sum()
                y = cdf(r if r.sum() > 0 else qt, u[32][i])
        if M >= V or u[34][i] < pa:
            Z[i] = om[y]
    return Z, dg, torch.where(inside, 0.0, q)


def _cdf(w, u):
    c = w.cumsum(1)
    t = torch.as_tensor(u, device=w.device) * c[:, -1]
    return torch.searchsorted(c, t[:, None], right=True)[:, 0].clamp(max=w.shape[1] - 1).cpu().numpy()


def exact(case, seed):
    B, K, L, V = case["B"], case["K"], case["L"], case["V"]
    if case["scheme"] == "IS" and B * V > 7e6:
        return None
    dev = torch.device("cuda", 0)
    target, drafts, tokens, temps = _inputs(case, seed, dev)
    tok_all, temps = tokens.cpu().numpy().astype(np.int64), temps.double()
    mids = np.asarray(_model_ids(case))
    diag = np.zeros((B, L + 1, 4))
    ids, valid = np.arange(B), np.ones((B, K), dtype=bool)

    def law_of(row, T):
        p = torch.softmax(row.double() / T[:, None], 1)
        if case["top_k"]:
            keep = _top_ids(row, case["top_k"])
            p = torch.zeros_like(p).scatter_(1, keep, torch.gather(p, 1, keep))
            p /= p.sum(1, keepdim=True)
        return p

    for j in range(L):
        if not len(ids):
            break
        t = torch.as_tensor(ids, device=dev)
        first = torch.as_tensor(valid.argmax(1), device=dev)
        q = law_of(target[t, first, j], temps[t, 0])
        rows = []
        for m in range(case["models"]):
            k = torch.as_tensor((valid & (mids == m)[None]).argmax(1), device=dev)
            rows.append(law_of(drafts[k, t, j], temps[t, 1 + k]))
        nv = valid.sum(1)
        order = np.argsort(~valid, axis=1, kind="stable")
        X, mrow = np.take_along_axis(tok_all[ids, :, j], order, 1), mids[order]
        n = len(ids)
        at = lambda w, y: w[torch.arange(n, device=dev), torch.as_tensor(y, device=dev)].cpu().numpy()  # noqa: E731
        first_law = lambda: torch.stack([rows[m][i] for i, m in enumerate(mrow[:, 0])])  # noqa: E731
        if case["scheme"] == "WIS0":
            Z, dg, rest = _small_alphabet(q, rows, X, mrow, nv, ids, j, case["omega0"])
            outside = _cdf(rest, _uniform(ids, j, 35))
            Z = np.where(Z < 0, outside, Z)
        elif case["scheme"] == "SpecTr":
            Z, cur, prod, dg = np.full(n, -1), q, np.ones(n), np.zeros((n, 4))
            for i in range(K):
                on = nv > i
                if not on.any():
                    break
                p = torch.stack([rows[m][r] for r, m in enumerate(mrow[:, i])])
                qx, px = at(cur, X[:, i]), at(p, X[:, i])
                if i == 0:
                    dg[:, 0], dg[:, 1], dg[:, 3] = qx, px, X[:, 0]
                ok = on & (Z < 0) & (_uniform(ids, j, 16 + i) < np.minimum(1.0, np.where(px > 0, qx / np.where(
                    px > 0, px, 1.0), 1.0)))
                Z = np.where(ok, X[:, i], Z)
                r = (cur - p).clamp(min=0.0)
                R = r.sum(1)
                go = torch.as_tensor(on, device=dev) & (R > 0)
                cur = torch.where(go[:, None], r / torch.where(R > 0, R, 1.0)[:, None], cur)
                prod = np.where(on, prod * R.cpu().numpy(), prod)
            dg[:, 2] = np.where((Z < 0) | bool(case["acc_prob"]), prod, 0.0)
            Z = np.where(Z < 0, _cdf(cur, _uniform(ids, j, 32)), Z)
        else:
            if case["scheme"] == "single":
                Y, law = X[:, 0].copy(), first_law()
            elif case["scheme"] == "IS":
                Y, law = _classical(q, rows, X, mrow, nv, ids, j)
            else:
                Y, law = _stages(q, rows, X, mrow, nv, ids, j, case["scheme"] == "WISsort")
            dg = np.zeros((n, 4))
            dg[:, 0], dg[:, 1], dg[:, 3] = at(q, Y), at(law, Y), Y
            ratio = np.where(dg[:, 1] > 0, dg[:, 0] / np.where(dg[:, 1] > 0, dg[:, 1], 1.0), 1.0)
            ok = _uniform(ids, j, 16) < np.minimum(1.0, ratio)
            r = (q - law).clamp(min=0.0)
            dg[:, 2] = np.where(~ok | bool(case["acc_prob"]), r.sum(1).cpu().numpy(), 0.0)
            Z = np.where(ok, Y, _cdf(r, _uniform(ids, j, 32)))
        diag[ids, j] = dg
        valid &= tok_all[ids, :, j] == Z[:, None]
        live = valid.any(1)
        ids, valid = ids[live], valid[live]
    diag[ids, L] = 0.0, 0.0, 1.0, -1.0   # the bonus token is drawn from the whole target row
    return {"tokens": None, "accepted": None, "target_prob": diag[:, :, 0], "importance_prob": diag[:, :, 1],
            "residual": diag[:, :, 2], "intermediate": diag[:, :, 3]}
