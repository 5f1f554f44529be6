"""The work that programs have this miner do, as cases that can be timed.

A case is a dict of plain values.  `listed()` names the cases, `draw(rng)` gives
one more of the same ranges, `prepare(case, seed)` makes what a program has in
hand before the call (inputs from the seed, a context), `run(state)` makes one
pass through the public entry points, `work(case)` counts what the pass cannot
do without, and `exact(case, seed)` gives the outputs that are computed numbers
in 64 bits.

Kinds of case:
  mine    one database: fim_build_bitmaps, fim_mine, fim_fetch_results
  batch   many databases: fim_mine_batched, fim_fetch_batched of all of them
  rules   association rules of mined sets: fim_rules, fim_fetch_rules
  mlp     one training step of the scheduling network

The databases have the shapes of the repository's own generators
(paper_2412_19420_gb300/datagen.py), drawn on the GPU because they are made
many times.
"""
from __future__ import annotations

import math
import types

import numpy as np
import torch

from paper_2412_19420_gb300 import datagen, fim, sched

DEV = "cuda"


def listed():
    return [
        # The smallest run of the paper's Table 1 (2,000 transactions at 1%):
        # interactive use on one small table, where launches and round trips count.
        dict(name="mine_2k_169", kind="mine", gen="zipf", n=2_000, m=169, s=1.0, mean_len=4.4, ppm=10_000,
             compact=False, host=False, learned=False),
        # The paper's largest run, 10,000 baskets of a grocer's 169 items at 1%.
        dict(name="mine_10k_169", kind="mine", gen="zipf", n=10_000, m=169, s=1.0, mean_len=4.4, ppm=10_000,
             compact=False, host=False, learned=False),
        # A small, dense table (every item in 3 of 10 rows): survey or click
        # matrices, where the search is wide at every level.
        dict(name="mine_dense_50k_60", kind="mine", gen="dense", n=50_001, m=60, density=0.3, ppm=20_000,
             compact=False, host=False, learned=False),
        # An ordinary database of odd size that starts in host memory (page-locked,
        # compact CSR) and whose result ends there.
        dict(name="mine_host_333k_701", kind="mine", gen="quest", n=333_337, m=701, avg_len=10.0, pat_len=4.0,
             n_patterns=1_400, ppm=1_000, compact=True, host=True, learned=False),
        # A large sparse database resident in HBM.
        dict(name="mine_1M_1000", kind="mine", gen="quest", n=1_000_000, m=1_000, avg_len=10.0, pat_len=4.0,
             n_patterns=2_000, ppm=1_000, compact=False, host=False, learned=False),
        # Long correlated patterns: millions of itemsets, a search many levels deep.
        dict(name="mine_planted_100k_2000", kind="mine", gen="planted", n=100_000, m=2_000, n_patterns=500, s=1.1,
             mean_len=8.0, ppm=5_000, compact=False, host=False, learned=False),
        # The same shape smaller, steered by the trained network.
        dict(name="mine_learned_20k_800", kind="mine", gen="planted", n=20_000, m=800, n_patterns=60, s=1.1,
             mean_len=8.0, ppm=5_000, compact=False, host=False, learned=True),
        # The largest single database.
        dict(name="mine_10M_5000", kind="mine", gen="quest", n=10_000_000, m=5_000, avg_len=12.0, pat_len=5.0,
             n_patterns=5_000, ppm=500, compact=False, host=False, learned=False),
        # A few databases (stores, weeks) in one call, wide CSRs.
        dict(name="batch_48", kind="batch", n_db=48, log_lo=3.0, log_hi=5.0, m_lo=64, m_hi=512, s=0.8, mean_len=6.0,
             ppm=20_000, compact=False),
        # Thousands of databases in one call, compact CSRs.
        dict(name="batch_4096", kind="batch", n_db=4_096, log_lo=3.0, log_hi=5.0, m_lo=64, m_hi=512, s=0.8,
             mean_len=6.0, ppm=20_000, compact=True),
        # Rules of a large mine's sets at 50% confidence.
        dict(name="rules_1M_1000", kind="rules", gen="quest", n=1_000_000, m=1_000, avg_len=10.0, pat_len=4.0,
             n_patterns=2_000, ppm=1_000, conf_ppm=500_000),
        # One training step of the scheduling network on a batch of traces.
        dict(name="mlp_step_4096", kind="mlp", rows=4_096, bf16=True),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["zipf", "dense", "quest", "quest", "planted", "batch", "batch", "rules", "mlp"])
    io = dict(compact=rng.random() < 0.5, host=rng.random() < 0.25, learned=False)
    if kind == "zipf":
        return dict(kind="mine", gen="zipf", n=_log_int(rng, 1_000, 100_000), m=rng.randint(60, 512),
                    s=round(rng.uniform(0.8, 1.0), 2), mean_len=round(rng.uniform(4.4, 8.0), 1),
                    ppm=rng.randint(8_000, 20_000), **io)
    if kind == "dense":
        return dict(kind="mine", gen="dense", n=_log_int(rng, 5_000, 100_000), m=rng.randint(20, 60),
                    density=round(rng.uniform(0.2, 0.3), 3), ppm=rng.randint(20_000, 40_000), **io)
    if kind == "quest":
        m = _log_int(rng, 300, 5_000)
        return dict(kind="mine", gen="quest", n=_log_int(rng, 60_000, 5_000_000), m=m,
                    avg_len=round(rng.uniform(8.0, 12.0), 1), pat_len=round(rng.uniform(4.0, 5.0), 1),
                    n_patterns=max(500, min(5_000, 2 * m)), ppm=rng.randint(700, 1_500), **io)
    if kind == "planted":
        m = rng.randint(600, 2_000)
        io.update(host=False, learned=rng.random() < 0.25)
        return dict(kind="mine", gen="planted", n=_log_int(rng, 20_000, 100_000), m=m, n_patterns=rng.randint(40, m // 4),
                    s=1.1, mean_len=8.0, ppm=5_000, **io)
    if kind == "batch":
        return dict(kind="batch", n_db=_log_int(rng, 8, 2_048), log_lo=3.0, log_hi=round(rng.uniform(4.0, 5.0), 2),
                    m_lo=64, m_hi=rng.randint(200, 512), s=0.8, mean_len=6.0, ppm=rng.randint(15_000, 30_000),
                    compact=rng.random() < 0.5)
    if kind == "rules":
        m = _log_int(rng, 300, 2_000)
        return dict(kind="rules", gen="quest", n=_log_int(rng, 60_000, 1_000_000), m=m, avg_len=10.0, pat_len=4.0,
                    n_patterns=2 * m, ppm=rng.randint(1_000, 2_000), conf_ppm=rng.randint(200_000, 800_000))
    return dict(kind="mlp", rows=_log_int(rng, 200, 8_192), bf16=rng.random() < 0.75)


# ---- databases, drawn on the GPU --------------------------------------------

def _gen(seed, salt=0):
    g = torch.Generator(device=DEV)
    g.manual_seed((int(seed) * 1_000_003 + salt) & 0x7FFFFFFFFFFFFFFF)
    return g


def _from_pairs(rows, items, n, m):
    """(indptr int64[n + 1], ids int64) of the distinct (row, item) pairs, rows
    in order, ids ascending."""
    key = torch.unique_consecutive(torch.sort(rows * m + items).values)
    r = torch.div(key, m, rounding_mode="floor")
    indptr = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    indptr[1:] = torch.cumsum(torch.bincount(r, minlength=n), 0)
    return indptr, key - r * m


def _zipf_cdf(m, s):
    w = np.arange(1, m + 1, dtype=np.float64) ** -s
    return np.cumsum(w) / w.sum()


def _lengths(g, n, mean):
    return torch.poisson(torch.full((n,), float(mean), device=DEV), generator=g).to(torch.int64)


def _zipf_pairs(g, n, m, s, mean_len):
    """Baskets of Zipf(s) items, Poisson(mean_len) draws each, at least one."""
    rows = torch.repeat_interleave(torch.arange(n, device=DEV), _lengths(g, n, mean_len).clamp(1, m))
    u = torch.rand(rows.shape[0], dtype=torch.float64, device=DEV, generator=g)
    rank = torch.searchsorted(torch.from_numpy(_zipf_cdf(m, s)).to(DEV), u).clamp(max=m - 1)
    return rows, torch.randperm(m, device=DEV, generator=g)[rank]


def _quest_pairs(g, seed, n, m, avg_len, pat_len, n_patterns):
    """Baskets filled with weighted patterns, half of a pattern's items dropped
    one by one (Agrawal and Srikant's scheme, as datagen.quest)."""
    rng = np.random.default_rng([seed, 77])
    plen = np.minimum(np.maximum(1, rng.poisson(pat_len, n_patterns)), m)
    lmax = int(plen.max())
    pats = rng.integers(0, m, (n_patterns, lmax))
    share = np.minimum(1.0, rng.exponential(0.5, n_patterns))
    off = rng.integers(0, 1 << 30, n_patterns)
    for p in range(1, n_patterns):  # part of a pattern comes from its predecessor
        k = min(int(round(share[p] * plen[p])), int(plen[p - 1]))
        pats[p, :k] = pats[p - 1, (off[p] + np.arange(k)) % plen[p - 1]]
    w = rng.exponential(1.0, n_patterns)
    cdf = torch.from_numpy(np.cumsum(w) / w.sum()).to(DEV)
    mean_keep = max(0.25, float(np.sum(w / w.sum() * (plen - (1 - 0.5 ** plen)))))
    d_pats, d_len = torch.from_numpy(pats).to(DEV), torch.from_numpy(plen).to(DEV)
    out_rows, out_items = [], []
    for r0 in range(0, n, 1 << 20):
        nr = min(n, r0 + (1 << 20)) - r0
        goal = torch.cumsum(_lengths(g, nr, avg_len).clamp(min=1), 0)
        d = int(int(goal[-1]) / mean_keep * 1.1) + 4096
        pid = torch.searchsorted(cdf, torch.rand(d, dtype=torch.float64, device=DEV, generator=g)).clamp(max=n_patterns - 1)
        length = d_len[pid]
        drop = torch.floor(-torch.log2(torch.rand(d, dtype=torch.float64, device=DEV, generator=g).clamp(min=1e-18)))
        keep = (length - drop.to(torch.int64)).clamp(min=0)
        # the kept items are a random subset of the pattern
        u = torch.rand((d, lmax), device=DEV, generator=g)
        slot = torch.arange(lmax, device=DEV)
        u = torch.where(slot[None, :] < length[:, None], u, 2.0)
        order = torch.argsort(u, dim=1, stable=True)
        items = torch.gather(d_pats[pid], 1, order)[slot[None, :] < keep[:, None]]
        # a draw belongs to the first basket whose running goal it still fits
        row = torch.searchsorted(goal, torch.cumsum(keep, 0) - keep, right=True)
        rows = torch.repeat_interleave(row, keep)
        ok = rows < nr
        out_rows.append(rows[ok] + r0)
        out_items.append(items[ok])
    return torch.cat(out_rows), torch.cat(out_items)


def _planted_pairs(g, seed, n, m, n_patterns, s, mean_len):
    """Zipf(s) baskets with patterns of 6 to 12 items in 0.5 to 3% of the rows."""
    rows, items = _zipf_pairs(g, n, m, s, mean_len)
    rng = np.random.default_rng([seed, 78])
    rr, ii = [rows], [items]
    for _ in range(n_patterns):
        pat = torch.from_numpy(rng.choice(m, size=int(rng.integers(6, 13)), replace=False)).to(DEV)
        cnt = int(round(rng.uniform(0.005, 0.03) * n))
        sel = torch.randint(0, n, (cnt,), device=DEV, generator=g)
        rr.append(sel.repeat_interleave(pat.shape[0]))
        ii.append(pat.repeat(cnt))
    return torch.cat(rr), torch.cat(ii)


def _database(case, seed):
    g = _gen(seed)
    n, m, gen = case["n"], case["m"], case["gen"]
    if gen == "zipf":
        rows, items = _zipf_pairs(g, n, m, case["s"], case["mean_len"])
    elif gen == "dense":
        rows, items = torch.nonzero(torch.rand((n, m), device=DEV, generator=g) < case["density"], as_tuple=True)
    elif gen == "quest":
        rows, items = _quest_pairs(g, seed, n, m, case["avg_len"], case["pat_len"], case["n_patterns"])
    else:
        rows, items = _planted_pairs(g, seed, n, m, case["n_patterns"], case["s"], case["mean_len"])
    return _from_pairs(rows, items, n, m)


def _typed(indptr, ids, compact):
    """The CSR as the entry points take it: int64 / int32, or (compact) uint32 /
    uint16 held in torch's int32 / int16."""
    if compact:
        return indptr.to(torch.int32), ids.to(torch.int16)
    return indptr.contiguous(), ids.to(torch.int32)


class _Ctx:
    """A context that is given back with the state that holds it."""

    def __init__(self, stream=None):
        self.h = fim.fim_create(0, stream)

    def __del__(self):
        if fim is not None and self.h:
            fim.fim_destroy(self.h)
            self.h = None


# ---- what a program has in hand ----------------------------------------------

# result buffers a program keeps: room for (sets, items of all sets)
_SETS_CAP = {"zipf": (1 << 14, 1 << 16), "dense": (1 << 17, 1 << 19), "quest": (1 << 19, 1 << 22),
             "planted": (1 << 23, 1 << 26)}


def _zeros(n, dtype, host):
    return torch.zeros(n, dtype=dtype).pin_memory() if host else torch.zeros(n, dtype=dtype, device=DEV)


def _buffers(sets, items, host):
    """(offsets, items, supports) as tensors, and as the entry points take them."""
    out = (_zeros(sets + 1, torch.int64, host), _zeros(items, torch.int32, host), _zeros(sets, torch.int32, host))
    return out, tuple(o.numpy() for o in out) if host else out

def _prepare_mine(case, seed):
    st = types.SimpleNamespace(kind="mine", ctx=_Ctx(), m=case["m"], flags=0,
                               minsup=fim.fim_minsup_from_ppm(case["n"], case["ppm"]))
    st.out, st.into = _buffers(*_SETS_CAP[case["gen"]], case["host"])
    if case["learned"]:  # the network, trained on another database of the same shape
        other = dict(case, n=20_000, m=min(case["m"], 800), n_patterns=min(case["n_patterns"], 60))
        ip, ix = _typed(*_database(other, seed + 1), False)
        x, t = sched.collect_traces(st.ctx.h, types.SimpleNamespace(indptr=ip, indices=ix, m=other["m"]), 100)
        st.weights, _ = sched.fit(st.ctx.h, x, t, steps=400, seed=0)
        fim.fim_sched_load_weights(st.ctx.h, st.weights)
        st.flags = fim.FIM_LEARNED
    ip, ix = _typed(*_database(case, seed), case["compact"])
    if case["host"]:
        ip, ix = ip.cpu().pin_memory().numpy(), ix.cpu().pin_memory().numpy()
        if case["compact"]:
            ip, ix = ip.view(np.uint32), ix.view(np.uint16)
    st.indptr, st.indices = ip, ix
    return st


def _prepare_batch(case, seed):
    rng = np.random.default_rng([seed, 79])
    D = case["n_db"]
    ns = np.floor(10.0 ** rng.uniform(case["log_lo"], case["log_hi"], D)).astype(np.int64)
    ms = rng.integers(case["m_lo"], case["m_hi"] + 1, D)
    g = _gen(seed, 5)
    N, mx = int(ns.sum()), int(ms.max())
    row0 = np.concatenate([[0], np.cumsum(ns)])
    # every database's own popularity over its own ids: one table of cdf and ids
    cdf = np.concatenate([_zipf_cdf(int(m), case["s"]) + d for d, m in enumerate(ms)])
    ids = np.concatenate([rng.permutation(int(m)) for m in ms])
    d_ns, d_row0 = torch.from_numpy(ns).to(DEV), torch.from_numpy(row0).to(DEV)
    db = torch.repeat_interleave(torch.arange(D, device=DEV), d_ns)
    rows = torch.repeat_interleave(torch.arange(N, device=DEV), _lengths(g, N, case["mean_len"]).clamp(1, case["m_lo"]))
    u = torch.rand(rows.shape[0], dtype=torch.float64, device=DEV, generator=g) * (1 - 1e-9) + db[rows]
    at = torch.searchsorted(torch.from_numpy(cdf).to(DEV), u).clamp(max=cdf.shape[0] - 1)
    del u
    indptr, items = _from_pairs(rows, torch.from_numpy(ids).to(DEV)[at], N, mx)
    del rows, at
    # each database's offsets start at 0: [n_d + 1] of them, one after another
    ptr = torch.empty(N + D, dtype=torch.int64, device=DEV)
    r = torch.arange(N, device=DEV)
    ptr[r + db] = indptr[:-1] - indptr[d_row0[:-1]][db]
    ptr[d_row0[1:] + torch.arange(D, device=DEV)] = indptr[d_row0[1:]] - indptr[d_row0[:-1]]
    cut = indptr[d_row0].cpu().numpy()
    ptr, items = _typed(ptr, items, case["compact"])
    dbs = []
    for d in range(D):
        p0 = int(row0[d]) + d
        ip, ix = ptr[p0:p0 + int(ns[d]) + 1], items[int(cut[d]):int(cut[d + 1])]
        if not case["compact"]:  # a program that holds them one by one
            ip, ix = ip.clone(), ix.clone()
        dbs.append(types.SimpleNamespace(indptr=ip, indices=ix, m=int(ms[d])))
    minsups = [fim.fim_minsup_from_ppm(int(n), case["ppm"]) for n in ns]
    torch.cuda.synchronize()
    out, into = _buffers(1 << 20, 1 << 21, False)
    return types.SimpleNamespace(kind="batch", ctx=_Ctx(), desc=fim.BatchDescriptor(dbs, minsups), out=out, into=into)


def _mlp_inputs(case, seed):
    """Traces as the miner writes them: features of order 1, a log2 work and a 0/1 label."""
    g = _gen(seed, 9)
    x = torch.rand((case["rows"], 8), device=DEV, generator=g)
    t = torch.stack([torch.rand(case["rows"], device=DEV, generator=g) * 20.0 + 4.0,
                     (torch.rand(case["rows"], device=DEV, generator=g) < 0.3).float()], 1).contiguous()
    return torch.from_numpy(datagen.mlp_init_weights(int(seed) & 0xFFFF)).to(DEV), x, t


def prepare(case, seed):
    if case["kind"] == "mine":
        return _prepare_mine(case, seed)
    if case["kind"] == "batch":
        return _prepare_batch(case, seed)
    if case["kind"] == "rules":
        st = _prepare_mine(dict(case, compact=False, host=False, learned=False), seed)
        fim.fim_build_bitmaps(st.ctx.h, st.indptr, st.indices, st.m)
        fim.fim_mine(st.ctx.h, st.minsup)
        st.kind, st.conf = "rules", case["conf_ppm"]
        N = 1 << 22
        st.out = st.into = (_zeros(N, torch.int64, False), _zeros(N, torch.int32, False),
                            _zeros(N, torch.float64, False), _zeros(N, torch.float64, False))
        return st
    p, x, t = _mlp_inputs(case, seed)
    B = case["rows"]
    first = torch.zeros((3, p.shape[0]), device=DEV)  # parameters, Adam's two moments
    first[0] = p
    stream = torch.cuda.Stream()  # the program's own work and the context's, in order
    stream.wait_stream(torch.cuda.current_stream())
    return types.SimpleNamespace(kind="mlp", stream=stream, ctx=_Ctx(stream), first=first, now=first.clone(), x=x, t=t,
                                 bf16=case["bf16"], y=torch.empty((B, 2), device=DEV),
                                 cache=torch.empty((B, 256), device=DEV), grad=torch.empty_like(p))


# ---- one pass ----------------------------------------------------------------

def run(state):
    h = state.ctx.h
    if state.kind == "mine":
        fim.fim_build_bitmaps(h, state.indptr, state.indices, state.m)
        fim.fim_mine(h, state.minsup, state.flags)
        fim.fim_fetch_results(h, state.into)
        return state.out
    if state.kind == "batch":
        fim.fim_mine_batched(h, state.desc)
        fim.fim_fetch_batched(h, fim.FIM_ALL_DBS, state.into)
        return state.out
    if state.kind == "rules":
        fim.fim_rules(h, state.conf)
        fim.fim_fetch_rules(h, state.into)
        return state.out
    s = state
    with torch.cuda.stream(s.stream):
        s.now.copy_(s.first)  # every pass is the same first step
        fim.fim_mlp_forward(h, s.now[0], s.x, s.y, s.cache, bf16=s.bf16)
        loss = fim.fim_mlp_backward(h, s.now[0], s.x, s.y, s.t, s.cache, s.grad, bf16=s.bf16)
        fim.fim_mlp_adam(h, s.now[0], s.grad, s.now[1], s.now[2], 1, 2e-3)
    return s.y, loss, s.grad, s.now


# ---- what a pass cannot do without --------------------------------------------

def work(case):
    """The CSR read once and the least a result can be written in; for the
    mines, one operation per pair of items that share a row."""
    kind = case["kind"]
    if kind == "mlp":
        B = case["rows"]
        mac = 8 * 64 + 64 * 64 + 64 * 2
        return {"bytes": 4.0 * (B * (8 + 2 + 2) + 4 * 4866), "flops": 2.0 * 3.0 * B * mac}
    if kind == "batch":
        a, b = case["log_lo"], case["log_hi"]
        rows = case["n_db"] * (10.0 ** b - 10.0 ** a) / ((b - a) * math.log(10.0))
        per = case["mean_len"]
    else:
        rows = float(case["n"])
        per = {"zipf": case.get("mean_len"), "dense": case.get("density", 0.0) * case["m"],
               "quest": case.get("avg_len"),
               "planted": case.get("mean_len", 0.0) + case.get("n_patterns", 0) * 0.0175 * 9.0}[case["gen"]]
    if kind == "rules":  # the sets come out of the mine: some 700 rules an item, 28 bytes each
        return {"bytes": 28.0 * 700.0 * case["m"], "flops": 0.0}
    off, ident = (4.0, 2.0) if case["compact"] else (8.0, 4.0)
    return {"bytes": rows * (off + per * ident), "flops": rows * per * (per - 1.0) / 2.0}


# ---- outputs in 64 bits --------------------------------------------------------

def exact(case, seed):
    """The training step in float64.  The other kinds return counts, and ratios
    of counts that only a mine of the database gives: no such values here."""
    if case["kind"] != "mlp":
        return None
    p, x, t = (v.double() for v in _mlp_inputs(case, seed))
    p.requires_grad_(True)
    parts, at = [], 0
    for shape in datagen.MLP_SHAPES:
        k = math.prod(shape)
        parts.append(p[at:at + k].view(shape))
        at += k
    w1, b1, w2, b2, w3, b3 = parts
    y = torch.relu(torch.relu(x @ w1.T + b1) @ w2.T + b2) @ w3.T + b3
    loss = (0.5 * (y[:, 0] - t[:, 0]) ** 2
            + torch.nn.functional.binary_cross_entropy_with_logits(y[:, 1], t[:, 1], reduction="none")).mean()
    loss.backward()
    grad = p.grad
    m, v = 0.1 * grad, 0.001 * grad * grad
    new = p.detach() - 2e-3 * (m / 0.1) / (torch.sqrt(v / 0.001) + 1e-8)
    return y.detach(), float(loss), grad, torch.stack([new, m, v])
