"""The calls this library is timed on, as a user's program makes them.

A case names a path through the public entry points of
``paper_2608_25230_gb300.fw`` and its sizes:

  exact    small rows (n <= 32): gap, swap rule over every key, exact best subset
  gap      top-k kept sets, dense and forced-weight outputs, gaps, dropped mass
  swap     the gap call, then the balancing selector inside the candidate set
  vote     the gap call, then the group vote (one kept set per KV head)
  pool     the gap call, then ES_pool at the schedule s = 4/8/16/32
  audit    the gap call, then the deployed selectors scored at that schedule
  wscore   the observation-window importance score of a whole cache
  contour  ContourKV allocation, then ragged compaction of K and V
  decode   the capped allocation, compaction into a store with room, then
           eight decode steps appended to it

Sizes, distributions and budgets are those of the workloads this repository
generates for its tests and benchmark (long rows of one KV head, GQA groups of
four rows, contour caches, exact rows with a sink), at their full sizes or a
stated share of their rows, and ragged lengths between.
"""
import math

import numpy as np
import torch

from paper_2608_25230_gb300 import fw

DEV = "cuda"
SCHED_S, SCHED_E = (4, 8, 16, 32), (24, 12, 6, 4)  # candidate-set schedule: budgets and extras
GQA_FRACS = (1 / 32, 1 / 16, 1 / 8, 1 / 4)          # budget of group g: GQA_FRACS[g % 4] * n
LONG_FRACS = (1 / 16, 1 / 8, 1 / 4, 1 / 2)          # nested budgets of long rows, the first nb of them
APPENDS = 8


def listed():
    return [
        # one prompt's worth of toy instances: the smallest call, launches and latency
        dict(name="exact_toy", path="exact", rows=256, n=20, k=5, d=64, v="f32"),
        # one model family's instances of the exact search (24 keys, 134,596 subsets a row)
        dict(name="exact_enum", path="exact", rows=36864, n=24, k=6, d=128, v="f32"),
        # eight KV heads of a 32k prompt, 512 query rows each, three nested budgets
        dict(name="gap_heads", path="gap", groups=8, R=512, n_lo=32768, n=32768, d=128, v="bf16", nb=3, budget="long"),
        # GQA groups of a ragged batch: every length its own, most of them odd
        dict(name="gap_gqa", path="gap", groups=1536, R=4, n_lo=1000, n=16384, d=128, v="bf16", nb=1, budget="gqa"),
        # the selector on ragged GQA rows of a d = 64 model
        dict(name="swap_gqa", path="swap", groups=768, R=4, n_lo=1000, n=8192, d=64, v="bf16", nb=1, budget="gqa", E=32),
        # the selector on long rows, three budgets each
        dict(name="swap_heads", path="swap", groups=4, R=128, n_lo=32768, n=32768, d=128, v="bf16", nb=3, budget="long",
             E=32),
        # one kept set per KV head, as a cache is deployed
        dict(name="vote_heads", path="vote", groups=8, R=512, n_lo=32768, n=32768, d=128, v="bf16", nb=3, budget="long"),
        # ES_pool on GQA rows
        dict(name="pool_gqa", path="pool", groups=64, R=4, n_lo=4096, n=4096, d=128, v="bf16", nb=4, budget="sched"),
        # the audit of the deployed selectors on GQA rows
        dict(name="audit_gqa", path="audit", groups=256, R=4, n_lo=4096, n=4096, d=128, v="bf16", nb=4, budget="sched"),
        # the window score of 32 layers x 8 KV heads after a 32k prefill
        dict(name="wscore_cache", path="wscore", cells=256, T=32768, d=128, w=32),
        # that cache's allocation at an eighth of its tokens, and the compaction that frees the rest
        dict(name="contour_cache", path="contour", cells=256, T=32768, d=128, frac=1 / 8),
        # a short conversation's cache, capped per cell, then eight decode steps: small kernels in a row
        dict(name="decode_small", path="decode", cells=64, T=3001, d=64, frac=1 / 8),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    path = rng.choice(("exact", "gap", "gap", "swap", "swap", "vote", "pool", "audit", "wscore", "contour", "decode"))
    if path == "exact":
        n = rng.randint(8, 24)
        k = rng.randint(2, min(6, n - 1))
        return dict(path=path, rows=_log(rng, 17, 30000), n=n, k=k, d=rng.choice((32, 64, 128)),
                    v=rng.choice(("f32", "f32", "bf16")))
    if path == "wscore":
        T = _log(rng, 500, 32768)
        return dict(path=path, cells=_log(rng, 4, min(256, 256 * 32768 // T)), T=T, d=rng.choice((64, 128)),
                    w=rng.choice((8, 16, 32, 32)))
    if path in ("contour", "decode"):
        T = _log(rng, 500, 32768)
        cells = _log(rng, 4, 256 if path == "contour" else 64)
        return dict(path=path, cells=cells, T=T, d=rng.choice((64, 128)), frac=rng.choice((1 / 16, 1 / 8, 1 / 4)))
    v, d = rng.choice((("bf16", 64), ("bf16", 128), ("bf16", 128), ("bf16", 64), ("f32", 64), ("bf16", 32)))
    if path in ("pool", "audit"):
        n = _log(rng, 300, 16384 if path == "audit" else 6000)
        R = rng.choice((1, 4, 4, 6))
        groups = _log(rng, 3, 200 if path == "audit" else 40)
        return dict(path=path, groups=groups, R=R, n_lo=max(100, n // rng.choice((1, 2))), n=n, d=d, v=v, nb=4,
                    budget="sched")
    if rng.random() < 0.5:  # a few heads, many rows each
        n = _log(rng, 1000, 32768)
        groups, R, budget, nb = rng.randint(1, 8), _log(rng, 12, 512), "long", rng.randint(1, 4)
        if path == "swap":
            R = min(R, 64)
    else:  # GQA groups
        n = _log(rng, 500, 16384)
        groups, R, budget, nb = _log(rng, 16, 768), rng.choice((1, 4, 4, 7, 8)), "gqa", 1
        if path == "swap":
            groups = min(groups, 384)
    if v == "f32" or d == 32:  # the general path: fewer rows
        groups, R = min(groups, 128), min(R, 32)
        n = min(n, 8192)
    case = dict(path=path, groups=groups, R=R, n_lo=rng.choice((n, max(40, n // 8))), n=n, d=d, v=v, nb=nb, budget=budget)
    if path == "swap":
        case["E"] = rng.choice((12, 24, 32, 32))
    return case


# ------------------------------------------------------------------ shapes
def _lengths(c):
    """Length of every group: the same for every seed, spread over [n_lo, n]."""
    g = np.arange(c["groups"], dtype=np.int64)
    span = c["n"] - c["n_lo"] + 1
    lens = c["n_lo"] + (g * 2654435761 % 4294967296) * span // 4294967296
    lens[-1] = c["n"]
    return lens.astype(np.int32)


def _budgets(c):
    """[groups][nb] budgets."""
    lens = _lengths(c)
    if c["budget"] == "sched":
        k = [[s for s in SCHED_S[:c["nb"]]] for _ in lens]
    elif c["budget"] == "gqa":
        k = [[max(1, int(round(GQA_FRACS[i % 4] * n)))] for i, n in enumerate(lens)]
    else:
        k = [[max(1, int(round(f * n))) for f in LONG_FRACS[:c["nb"]]] for n in lens]
    return np.asarray(k, np.int32)


# ----------------------------------------------------------------- prepare
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return g


def _randn(g, *shape):
    return torch.randn(*shape, generator=g, device=DEV)


def _rand(g, lo, hi, *shape):
    return torch.rand(*shape, generator=g, device=DEV).mul_(hi - lo).add_(lo)


def _small_rows(c, seed):
    """Rows of their own: Gumbel logits at a temperature of U[0.5, 3], a sink of +6, values N(0, 1)."""
    g, B, n, d = _gen(seed), c["rows"], c["n"], c["d"]
    u = torch.rand(B, n, generator=g, device=DEV, dtype=torch.float64).clamp_(1e-300, 1 - 2.0 ** -53)
    l = (-(-u.log()).log()).float() * _rand(g, 0.5, 3.0, B, 1)
    l[:, 0] += 6.0
    v = _randn(g, B, n, d)
    if c["v"] == "bf16":
        v = v.to(torch.bfloat16)
    off = torch.arange(B, device=DEV, dtype=torch.int64)
    rows = fw.Rows(rows_per_group=1, d=d, n_host=np.full(B, n, np.int32), logits=l.reshape(-1), logit_off=off * n,
                   n=torch.full((B,), n, dtype=torch.int32, device=DEV), v=v.reshape(-1), v_off=off * (n * d),
                   v_dtype=c["v"])
    return rows, torch.full((B, 1), c["k"], dtype=torch.int32, device=DEV)


def _long_rows(c, seed):
    """Groups sharing a value block: logits of a head (1.5 N(0, 1)) or of GQA rows (temperature U[0.3, 4] each), a
    sink of +8 at the first key and a recency bump; values N(0, 1)."""
    g, R, d, lens = _gen(seed), c["R"], c["d"], _lengths(c)
    tot = int(lens.sum())
    lt = torch.as_tensor(lens, device=DEV).long()
    start = torch.cumsum(lt, 0) - lt                       # first key of each group
    rlen = lt.repeat_interleave(R)                         # length of each row
    rstart = torch.cumsum(rlen, 0) - rlen                  # first logit of each row
    l = _randn(g, tot * R)
    if c["budget"] == "long":
        l.mul_(1.5)
    else:
        tau = _rand(g, 0.3, 4.0, c["groups"] * R)
        l.mul_(torch.repeat_interleave(tau, rlen, output_size=tot * R))
    back = torch.repeat_interleave(rstart + rlen - 1, rlen, output_size=tot * R) - torch.arange(tot * R, device=DEV)
    l.add_(torch.exp(back.float().mul_(-1 / 256.0)).mul_(2.0))
    del back
    l[rstart] += 8.0
    v = _randn(g, tot * d)
    if c["v"] == "bf16":
        v = v.to(torch.bfloat16)
    rows = fw.Rows(rows_per_group=R, d=d, n_host=lens, logits=l, logit_off=start * R, n=lt.to(torch.int32), v=v,
                   v_off=start * d, v_dtype=c["v"])
    kg = torch.as_tensor(_budgets(c), device=DEV)
    return rows, kg.repeat_interleave(R, 0).contiguous(), kg


def _scores(c, g):
    sigma = _rand(g, 0.5, 2.5, c["cells"], 1)
    return torch.exp(_randn(g, c["cells"], c["T"]) * sigma)


def _contour_sizes(c):
    floor = min(32, c["T"])
    total = max(c["cells"] * floor, int(round(c["cells"] * c["T"] * c["frac"])))
    return floor, total, total // c["cells"]


def prepare(c, seed):
    p = c["path"]
    if p == "exact":
        rows, k = _small_rows(c, seed)
        return dict(c=c, rows=rows, k=k, k1=k[:, 0].contiguous())
    if p in ("gap", "swap", "vote", "pool", "audit"):
        rows, k, kg = _long_rows(c, seed)
        return dict(c=c, rows=rows, k=k, kg=kg)
    g = _gen(seed)
    cells, T, d = c["cells"], c["T"], c["d"]
    if p == "wscore":
        return dict(c=c, q=_randn(g, cells, c["w"], d).to(torch.bfloat16),
                    K=torch.randn(cells, T, d, generator=g, device=DEV, dtype=torch.bfloat16))
    s = dict(c=c, scores=_scores(c, g), K=torch.randn(cells, T, d, generator=g, device=DEV, dtype=torch.bfloat16),
             V=torch.randn(cells, T, d, generator=g, device=DEV, dtype=torch.bfloat16))
    if p == "decode":  # a store with room for the cap and the appended rows
        floor, total, u = _contour_sizes(c)
        room = u + APPENDS
        s["base"] = torch.arange(cells, device=DEV, dtype=torch.int64) * room
        s["capacity"] = torch.full((cells,), room, dtype=torch.int32, device=DEV)
        s["Ks"] = torch.zeros(cells * room, d, dtype=torch.bfloat16, device=DEV)
        s["Vs"] = torch.zeros(cells * room, d, dtype=torch.bfloat16, device=DEV)
        s["status"] = torch.zeros(cells, dtype=torch.int32, device=DEV)
        s["new"] = [(torch.randn(cells, 1, d, generator=g, device=DEV, dtype=torch.bfloat16),
                     torch.randn(cells, 1, d, generator=g, device=DEV, dtype=torch.bfloat16)) for _ in range(APPENDS)]
    return s


# --------------------------------------------------------------------- run
def _outputs(out):
    return {k: v for k, v in out.items() if not k.startswith("_")}  # not the scratch


def run(s):
    c = s["c"]
    p = c["path"]
    if p in ("exact", "gap", "swap", "vote", "pool", "audit"):
        rows, k = s["rows"], s["k"]
        top = fw.dense_and_topk_gap(rows, k)
        out = dict(top=_outputs(top))
        if p == "exact":
            out["swap"] = _outputs(fw.swap_refine(rows, k, top, E=c["n"], max_swaps=32))
            out["best"] = _outputs(fw.best_subset(rows, s["k1"], k_max=c["k"]))
        elif p == "swap":
            out["swap"] = _outputs(fw.swap_refine(rows, k, top, E=c["E"], max_swaps=64))
        elif p == "vote":
            out["vote"] = _outputs(fw.group_vote(rows, s["kg"], top))
        elif p == "pool":
            out["pool"] = _outputs(fw.pool_best_subset(rows, k, top, E=SCHED_E[:c["nb"]]))
            del out["pool"]["n_cand"]  # how many subsets the search re-scored: its own work count, not a result
        elif p == "audit":
            out["audit"] = _outputs(fw.selector_audit(rows, SCHED_S[:c["nb"]], top, bits=True))
        return out
    if p == "wscore":
        return fw.window_score(s["q"], s["K"])
    floor, total, u = _contour_sizes(c)
    if p == "contour":
        a = fw.contour_alloc(s["scores"], floor=floor, total_budget=total, uniform_s=u)
        return dict(alloc=_outputs(a), kv=fw.ragged_compact(s["K"], s["V"], a["offsets"], a["kept_pos"], total))
    a = fw.contour_alloc_capped(s["scores"], floor=floor, total_budget=total, uniform_s=u, cap=u)
    fw.ragged_compact_to(s["K"], s["V"], a["offsets"], a["kept_pos"], s["base"], s["capacity"], s["Ks"], s["Vs"],
                         s["status"])
    for nk, nv in s["new"]:
        fw.ragged_append(s["Ks"], s["Vs"], s["base"], s["capacity"], a["counts"], nk, nv, s["status"])
    out = _outputs(a)
    del out["kept_pos"]  # its entries past offsets[-1] are not written; the store holds the rows it names
    return dict(alloc=out, Ks=s["Ks"], Vs=s["Vs"], status=s["status"])


# -------------------------------------------------------------------- work
def work(c):
    p = c["path"]
    if p == "exact":
        B, n, d, k = c["rows"], c["n"], c["d"], c["k"]
        eb = 4 if c["v"] == "f32" else 2
        out = 4 * (2 * d + 9) + 4 * (4 + 2 * 32) + 8 + 4 * (3 + k)
        return dict(bytes=B * (4 * n + eb * n * d + 4 + out), flops=B * (n * n * d + 4.0 * n * d))
    if p in ("gap", "swap", "vote", "pool", "audit"):
        R, d, nb, G = c["R"], c["d"], c["nb"], c["groups"]
        lens, k = _lengths(c).astype(np.float64), _budgets(c).astype(np.float64)
        words = (c["n"] + 31) // 32
        eb = 4 if c["v"] == "f32" else 2
        rows = G * R
        by = 4 * R * lens.sum() + eb * d * lens.sum() + 4.0 * rows * (d * (1 + nb) + nb * (5 + words + 1) + 3)
        fl = 2.0 * R * d * lens.sum() * 2  # the dense and the masked products
        if p == "swap":  # the pool's errors, and one round of cross products
            by += 4.0 * rows * nb * (4 + 128)
            fl += R * (3.0 * d * lens.sum() + 2.0 * d * c["E"] * k.sum())
        if p == "vote":
            by += 4.0 * (rows * (2 * nb + 1) + G * nb * (words + 1))
            fl += 2.0 * R * d * lens.sum()
        if p == "pool":
            by += 4.0 * rows * (nb * (2 + 32) + 1)
            fl += R * 3.0 * d * lens.sum() + rows * sum(float(d * (s + e) ** 2) for s, e in zip(SCHED_S, SCHED_E))
        if p == "audit":
            by += 4.0 * rows * 5 * nb * (1 + words)
            fl += rows * 2.0 * d * 5 * sum(SCHED_S[:nb])
        return dict(bytes=float(by), flops=float(fl))
    cells, T, d = c["cells"], c["T"], c["d"]
    if p == "wscore":
        return dict(bytes=cells * (2.0 * T * d + 2.0 * c["w"] * d + 4 * T + 4), flops=2.0 * cells * T * d * c["w"])
    floor, total, u = _contour_sizes(c)
    by = 4.0 * cells * T + 4.0 * total + 2 * 2 * 2.0 * total * d + 20.0 * cells
    if p == "decode":
        by += 2 * 2 * 2.0 * cells * d * APPENDS
    return dict(bytes=by, flops=2.0 * cells * T)


# --------------------------------------------------------------- tolerance
def tolerance(c):
    """Floats are fp32 sums; gaps are norms of small differences of them.  Whole numbers: bits, thresholds and
    positions follow from the inputs alone, except that a swap chain, a vote or a best set may take either side of a
    tie closer than fp32 resolves.  Measured by permuting the value columns (the same sums in another order) and
    against exact()."""
    p = c["path"]
    if p in ("contour", "decode"):  # 3e-8 from exact(): fp32 sums of T scores
        return dict(rel=1e-6, max=1e-5, differ=0.0)
    if p == "wscore":  # 2e-7: the hardware exponential
        return dict(rel=2e-6, max=2e-5)
    if p == "gap":  # up to 2e-6: fp32 sums of up to 32,768 terms
        return dict(rel=1e-5, max=2e-4, differ=0.0)
    if p == "swap":  # the same; a chain that parts at a near-tie ends close to the other, with other swaps listed
        return dict(rel=2e-5, max=1e-3, differ=5e-3)
    if p == "exact":  # 3e-8: double-float sums
        return dict(rel=1e-6, max=1e-5, differ=1e-3)
    return dict(rel=1e-5, max=2e-3, differ=1e-3)  # one flipped vote or best set in a few thousand


# ------------------------------------------------------------------- exact
def _combos(n, k):
    from itertools import combinations
    idx = torch.tensor(list(combinations(range(n), k)), device=DEV)
    ind = torch.zeros(len(idx), n, device=DEV, dtype=torch.float64)
    return ind.scatter_(1, idx, 1.0)


def _best(U, P, k):
    """min over the size-k subsets of ||sum u|| / sum p, for U [B][n][d] and P [B][n]."""
    B, n, _ = U.shape
    ind = _combos(n, k)
    i, j = torch.triu_indices(n, n, device=DEV)
    pair = ind[:, i] * ind[:, j]
    G = U @ U.transpose(1, 2)
    w = G[:, i, j] * torch.where(i == j, 1.0, 2.0).double()
    out = []
    step = max(1, 300_000_000 // len(ind))
    for a in range(0, B, step):
        es2 = (w[a:a + step] @ pair.T) / (P[a:a + step] @ ind.T).square()
        out.append(es2.min(1).values.clamp_min(0).sqrt())
    return torch.cat(out)


def _gap64(l, V, ks):
    """Rows l [R][n], values V [n][d] (fp64): the gap call's outputs at the budgets ks, and the order of the keys."""
    M = l.max(1).values
    e = torch.exp(l - M[:, None])
    Z = e.sum(1)
    p = e / Z[:, None]
    order = torch.sort(l, dim=1, descending=True, stable=True).indices
    rank = torch.empty_like(order).scatter_(1, order, torch.arange(l.shape[1], device=DEV).expand_as(order).contiguous())
    mu = p @ V
    kept = [rank < k for k in ks]
    PA = torch.stack([(p * m).sum(1) for m in kept], 1)
    PC = torch.stack([(p * ~m).sum(1) for m in kept], 1)
    mA = torch.stack([(p * m) @ V for m in kept], 1) / PA[:, :, None]
    gap = (mA - mu[:, None]).norm(dim=2)
    top = dict(o=mu, gap=gap, dropped=PC, phi=gap * PA, o_kept=mA, row_max=M, row_sum=Z)
    return top, p, rank


def _es_of(mask, p, V, mu):
    w = p * mask
    return ((w @ V) / w.sum(1, keepdim=True) - mu).norm(dim=1), (p * ~mask).sum(1)


def _topm(score, m):
    """Boolean mask of the m largest along the last axis, equal scores lower index first."""
    o = torch.sort(score, dim=-1, descending=True, stable=True).indices[..., :m]
    return torch.zeros_like(score, dtype=torch.bool).scatter_(-1, o, True)


def _audit64(l, p, V, mu, s):
    R, n = l.shape
    nan = torch.full((R,), math.nan, device=DEV, dtype=torch.float64)
    j = torch.arange(n, device=DEV)
    out = []
    if s > n:
        return torch.stack([nan] * 5, 1)
    sink = min(4, s // 2)
    out.append(((j < sink) | (j >= n - (s - sink))).expand(R, n))
    r = s // 2
    m = j >= n - r
    m = m.clone()
    m[:n - r] |= _topm(p.sum(0)[:n - r], s - r)
    out.append(m.expand(R, n))
    w = max(1, min(32, s // 2))
    vote = p[max(0, R - w):].sum(0)[:n - w]
    pooled = torch.nn.functional.max_pool1d(vote[None, None], 7, 1, 3)[0, 0]
    m = (j >= n - w).clone()
    m[:n - w] |= _topm(pooled, s - w)
    out.append(m.expand(R, n))
    for q16 in (False, True):
        P = 16 if q16 else max(2, s // 4)
        if s // P < 1 or (q16 and s < 16):
            out.append(None)
            continue
        npg = (n + P - 1) // P
        pages = torch.nn.functional.pad(l, (0, npg * P - n), value=-math.inf).view(R, npg, P).max(2).values
        out.append(_topm(pages, min(s // P, npg)).repeat_interleave(P, 1)[:, :n])
    return torch.stack([nan if m is None else _es_of(m, p, V, mu)[0] for m in out], 1)


def exact(c, seed):
    p = c["path"]
    if p == "exact":
        s = prepare(c, seed)
        B, n, d, k = c["rows"], c["n"], c["d"], c["k"]
        l, V = s["rows"].logits.view(B, n).double(), s["rows"].v.view(B, n, d).double()
        P = torch.softmax(l, 1)
        mu = torch.einsum("bn,bnd->bd", P, V)
        mask = _topm(l, k)
        w = P * mask
        PA, PC = w.sum(1), (P * ~mask).sum(1)
        mA = torch.einsum("bn,bnd->bd", w, V) / PA[:, None]
        gap = (mA - mu).norm(dim=1)
        M = l.max(1).values
        top = dict(o=mu, gap=gap[:, None], dropped=PC[:, None], phi=(gap * PA)[:, None], o_kept=mA[:, None], row_max=M,
                   row_sum=torch.exp(l - M[:, None]).sum(1))
        best = _best(P[:, :, None] * (V - mu[:, None]), P, k)
        # the swap rule's end point depends on which side of a near-tie its chain took: no 64-bit value
        return dict(top=top, swap=dict(topk_gap=gap[:, None], refined_gap=None), best=dict(best_gap=best, topk_gap=gap))
    if p in ("gap", "swap", "vote", "pool", "audit"):
        s = prepare(c, seed)
        rows, lens, ks = s["rows"], _lengths(c), _budgets(c)
        R, d = c["R"], c["d"]
        loff, voff = rows.logit_off.tolist(), rows.v_off.tolist()
        parts = []
        for g, n in enumerate(lens.tolist()):
            l = rows.logits[loff[g]:loff[g] + R * n].view(R, n).double()
            V = rows.v[voff[g]:voff[g] + n * d].view(n, d).double()
            top, P, rank = _gap64(l, V, ks[g].tolist())
            mu = top["o"]
            if p == "vote":
                G = P.sum(0)
                es = [_es_of(_topm(G, k).expand(R, n), P, V, mu) for k in ks[g].tolist()]
                top["v_gap"] = torch.stack([e for e, _ in es], 1)
                top["v_dropped"] = torch.stack([x for _, x in es], 1)
            if p == "audit":
                top["es"] = torch.stack([_audit64(l, P, V, mu, k) for k in SCHED_S[:c["nb"]]], 2)
            if p == "pool":  # the pool's masses and vectors; the search below runs over all rows at once
                err = P * (V[None] - mu[:, None]).norm(dim=2) if n * R * d < 1 << 28 else torch.stack(
                    [P[r] * (V - mu[r]).norm(dim=1) for r in range(R)])
                for b, (k, e) in enumerate(zip(SCHED_S, SCHED_E)):
                    kept = rank < k
                    e = min(e, n - k)
                    idx = torch.topk(torch.where(kept, math.inf, err), k + e, dim=1).indices
                    pk = P.gather(1, idx)
                    top["p%d" % b] = pk
                    top["u%d" % b] = pk[:, :, None] * (V[idx] - mu[:, None])
            parts.append(top)
        every = {k: torch.cat([t[k] for t in parts]) for k in parts[0]}
        top = {k: every[k] for k in ("o", "gap", "dropped", "phi", "o_kept", "row_max", "row_sum")}
        out = dict(top=top)
        if p == "swap":
            out["swap"] = dict(topk_gap=top["gap"], refined_gap=None)
        if p == "vote":
            out["vote"] = dict(gap=every["v_gap"], dropped=every["v_dropped"])
        if p == "audit":
            out["audit"] = dict(es=every["es"])
        if p == "pool":
            best = [_best(every["u%d" % b], every["p%d" % b], k) for b, k in enumerate(SCHED_S)]
            out["pool"] = dict(topk_gap=top["gap"], best_gap=torch.stack(best, 1))
        return out
    s = prepare(c, seed)
    cells, T = c["cells"], c["T"]
    if p == "wscore":
        w, lim = c["w"], T - c["w"]
        see = torch.arange(T, device=DEV)[None] <= lim + torch.arange(w, device=DEV)[:, None]
        out = []
        for q, K in zip(s["q"], s["K"]):
            a = torch.softmax((q.double() @ K.double().T / math.sqrt(c["d"])).masked_fill(~see, -math.inf), 1).sum(0)
            pre = torch.nn.functional.max_pool1d(a[None, None, :lim], 7, 1, 3)[0, 0] if lim else a[:0]
            out.append(torch.cat([pre, a[lim:]]))
        return [torch.stack(out)]
    floor, total, u = _contour_sizes(c)
    sc = s["scores"].double()
    mass = sc / sc.sum(1, keepdim=True)
    pre = sc[:, :T - floor].reshape(-1)
    K = total - cells * floor
    keep = torch.ones(cells, T, dtype=torch.bool, device=DEV)
    keep[:, :T - floor] = _topm(pre, K).view(cells, T - floor)
    tau = torch.sort(pre, descending=True).values[K - 1] if K else torch.tensor(math.inf, device=DEV)
    uni = _topm(sc, u)
    if p == "decode":  # a cell over the cap keeps its floor and its best cap - floor entries
        best = _topm(sc[:, :T - floor], u - floor)
        over = keep.sum(1) > u
        keep[over, :T - floor] = best[over]
    alloc = dict(tau=tau.reshape(1).double(), dropped_uniform=(mass * ~uni).sum(1), dropped_alloc=(mass * ~keep).sum(1))
    return dict(alloc=alloc)
