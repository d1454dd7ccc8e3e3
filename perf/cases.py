"""Cases for measuring the solver: what a program that lays out retrieval requests has it do.

A pass starts from host arrays and ends with every output of the call: new requests arrive for every
call, so a pass creates the context (or batch), solves, and takes the layout and the device tables.
What a program keeps between calls is the device workspace.  All inputs are synthetic, drawn from
the seed with the shapes of ``instances`` (RAG-shaped topical pools with a Zipf tail, the paper's
request streams, leave-one-out families).  All outputs are whole numbers.
"""

import itertools
import math

import numpy as np
import torch

from paper_2609_13692_gb300 import instances, mpt

LISTED = [
    # The smallest exact solve: 12 requests over 48 shared chunks (launches, copies and host work).
    dict(name="solve_zipf_m12", kind="solve", shape="zipf", m=12, n=48, k=5, tail_s=1.0, scale=1, tables="int64"),
    # Every request lacks one chunk of a common set: every subset of requests shares something, so
    # no split can be ruled out beforehand (few long documents that nearly all requests carry).
    dict(name="solve_leave_one_out_m20", kind="solve", shape="loo", m=20, n=20, k=19, tail_s=0.0, scale=1,
         tables="int64"),
    # Uniformly overlapping requests, an odd count: 4 to 12 of 40 chunks each.
    dict(name="solve_uniform_m23", kind="solve", shape="uniform", m=23, n=40, k=12, tail_s=0.0, scale=1,
         tables="int64"),
    # Ordinary retrieval group: 24 requests of 10 passages out of 100,000.
    dict(name="solve_rag_m24", kind="solve", shape="rag", m=24, n=100_000, pools=8, pool_size=200, k=10, tail_s=1.1,
         scale=1, tables="int64"),
    # The same with weights in bytes of cache instead of tokens: too heavy for 32-bit keys.
    dict(name="solve_rag_m24_heavy", kind="solve", shape="rag", m=24, n=100_000, pools=8, pool_size=200, k=10,
         tail_s=1.1, scale=4096, tables="int64"),
    # Deep retrieval over a million passages with the lean (int32) tables.
    dict(name="solve_rag_m26_k40_lean", kind="solve", shape="rag", m=26, n=1_000_000, pools=32, pool_size=400, k=40,
         tail_s=1.2, scale=1, tables="lean"),
    # The benchmark workload: 28 requests of 20 passages, 2^28-entry tables.
    dict(name="solve_rag_m28", kind="solve", shape="rag", m=28, n=100_000, pools=16, pool_size=300, k=20, tail_s=1.1,
         scale=1, tables="int64"),
    # Many small groups at once, the sizes of the paper's real request groups.
    dict(name="batch_20000_m8_13", kind="batch", count=20_000, m_lo=8, m_hi=13, n=100_000, k=8, scale=1),
    # Fewer, larger groups: the top of the batched range.
    dict(name="batch_1000_m14_16", kind="batch", count=1000, m_lo=14, m_hi=16, n=100_000, k=8, scale=1),
    # Agglomerative layout of a whole trace, beyond the exact recurrence.
    dict(name="greedy_m3000", kind="greedy", m=3000, k=8),
    # Serving order and finite-cache costs of one trace (10 capacities).
    dict(name="stream_m2921", kind="stream", m=2921, k=8, window=0),
    # The same for a long stream.
    dict(name="stream_m100000", kind="stream", m=100_000, k=8, window=0),
]


def listed():
    return [dict(c) for c in LISTED]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "solve", "batch", "greedy", "stream"])
    if kind == "batch":
        lo = rng.randint(2, 14)
        hi = rng.randint(lo, 16)
        most = 20_000 if hi <= 13 else 1000
        return dict(kind=kind, count=_log_int(rng, 10, most), m_lo=lo, m_hi=hi, n=_log_int(rng, 500, 200_000),
                    k=rng.randint(3, 16), scale=rng.choice([1, 1, 1, 64 if hi <= 14 else 1]))
    if kind == "greedy":
        return dict(kind=kind, m=_log_int(rng, 50, 6000), k=rng.randint(3, 20))
    if kind == "stream":
        m = _log_int(rng, 100, 100_000)
        return dict(kind=kind, m=m, k=rng.randint(3, 12), window=rng.choice([0, 0, _log_int(rng, 2, m)]))
    shape = rng.choice(["rag", "rag", "rag", "zipf", "uniform", "loo"])
    scale = rng.choice([1, 1, 1, 4096])
    c = dict(kind=kind, shape=shape, scale=scale, tables="lean" if scale == 1 and rng.random() < 0.25 else "int64")
    m = rng.randint(4, 27 if scale == 1 else 24)
    if shape == "rag":
        pools, size = rng.randint(2, 32), rng.randint(40, 400)
        n = _log_int(rng, pools * size, 1_000_000)
        return dict(c, m=m, n=n, pools=pools, pool_size=size, k=rng.randint(4, 40), tail_s=rng.choice([1.0, 1.1, 1.2]))
    m = min(m, 24)
    if shape == "zipf":
        return dict(c, m=m, n=rng.randint(32, 400), k=rng.randint(3, 8), tail_s=1.0)
    if shape == "uniform":
        n = rng.randint(20, 400)
        return dict(c, m=m, n=n, k=rng.randint(3, max(3, n // 3)), tail_s=0.0)
    return dict(c, m=m, n=m, k=m - 1, tail_s=0.0)


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------

def _instance(c, seed):
    if c["shape"] == "rag":
        inst = instances.rag_pools(c["m"], c["n"], c["pools"], c["pool_size"], c["k"], c["tail_s"], seed=seed)
    elif c["shape"] == "zipf":
        inst = instances.zipf_small(c["m"], c["n"], c["k"], c["tail_s"], seed=seed)
    elif c["shape"] == "uniform":
        rng = np.random.default_rng(seed)
        lo = max(1, c["k"] // 3)  # request sizes k / 3 .. k in a fixed order, chunks uniform
        reqs = [rng.choice(c["n"], size=lo + (7 * i) % (c["k"] - lo + 1), replace=False) for i in range(c["m"])]
        inst = instances.Instance(rng.integers(1, 100, size=c["n"], dtype=np.int64),
                                  instances.pack_requests(reqs, c["n"]))
    else:
        inst = instances.leave_one_out(c["m"])
        inst.weights = np.random.default_rng(seed).integers(1, 10, size=c["m"], dtype=np.int64)
    return inst.weights * c["scale"], inst.bits


def _weights(rng, n, mean):
    mu = math.log(mean) - 0.18
    return np.clip(np.rint(rng.lognormal(mu, 0.6, size=n)), 32, 4096).astype(np.int64)


def _distinct(rng, rows, k, one):
    """int64[rows, k]: each row k distinct ids; one(row indices) draws one id per listed row."""
    ids = one(np.repeat(np.arange(rows), k)).reshape(rows, k)
    while True:
        order = np.argsort(ids, axis=1, kind="stable")
        s = np.take_along_axis(ids, order, 1)
        again = np.zeros(ids.shape, dtype=bool)
        np.put_along_axis(again, order[:, 1:], s[:, 1:] == s[:, :-1], 1)
        r, j = np.nonzero(again)
        if not len(r):
            return ids
        ids[r, j] = one(r)


def _pool_requests(rng, rows, n, pool_of_row, pools, p_pool, k, tail_s):
    """Passages of each request: from its pool with probability p_pool, else from the tail (Zipf
    over a random ranking of all passages, or uniform when tail_s = 0)."""
    ranks = np.arange(1, n + 1, dtype=np.float64)
    cdf = np.cumsum(ranks ** -tail_s)
    cdf /= cdf[-1]
    perm = rng.permutation(n)

    def one(r):
        u = rng.random(len(r))
        tail = perm[np.minimum(np.searchsorted(cdf, rng.random(len(r)), side="right"), n - 1)]
        pool = pools[pool_of_row[r], rng.integers(0, pools.shape[1], len(r))]
        return np.where(u < p_pool, pool, tail)

    return _distinct(rng, rows, k, one)


def _prepare_batch(c, rng):
    n = c["n"]
    size = min(60, n // 4)
    pools = np.stack([rng.choice(n, size=size, replace=False) for _ in range(64)])
    ms = np.random.default_rng(c["count"]).integers(c["m_lo"], c["m_hi"] + 1, size=c["count"])  # same sizes, any seed
    inst_requests = np.concatenate([[0], np.cumsum(ms)]).astype(np.int64)
    rows = int(inst_requests[-1])
    pool_of_row = np.repeat(rng.integers(0, 64, size=c["count"]), ms)
    ids = _pool_requests(rng, rows, n, pool_of_row, pools, 0.8, c["k"], 0.0)
    offsets = np.arange(rows + 1, dtype=np.int64) * c["k"]
    weights = _weights(rng, n, 150.0) * c["scale"]
    b = mpt.mpt_batch_create(weights, inst_requests, offsets, ids.reshape(-1))
    ws = torch.empty(mpt.mpt_batch_workspace_bytes(b), dtype=torch.uint8, device="cuda")
    return dict(case=c, weights=weights, inst=inst_requests, offsets=offsets, ids=ids.reshape(-1).astype(np.int64),
                ws=ws)


def _prepare_trace(c, rng):
    """Requests in arrival order over topical pools of 40 to 60 passages with a tail (Sec. 8 streams)."""
    m, k = c["m"], c["k"]
    greedy = c["kind"] == "greedy"
    n = max(64 * k, int(m * 1.2))
    size, count = (60, max(8, m // 15)) if greedy else (40, max(8, m // 45))
    pools = np.stack([rng.choice(n, size=size, replace=False) for _ in range(count)])
    pool_of_row = rng.integers(0, len(pools), size=m)
    ids = _pool_requests(rng, m, n, pool_of_row, pools, 0.85 if greedy else 0.8, k, 0.0 if greedy else 1.0)
    return n, ids


def prepare(case, seed):
    c = dict(case)
    if c["kind"] == "solve":
        weights, bits = _instance(c, seed)
        ctx = mpt.mpt_create(weights, bits)
        mpt.mpt_set_tables(ctx, c["tables"])
        ws = torch.empty(mpt.mpt_workspace_bytes(ctx), dtype=torch.uint8, device="cuda")
        return dict(case=c, weights=weights, bits=bits, ws=ws)
    rng = np.random.default_rng(seed)
    if c["kind"] == "batch":
        return _prepare_batch(c, rng)
    n, ids = _prepare_trace(c, rng)
    weights = _weights(rng, n, 150.0 if c["kind"] == "greedy" else 750.0)
    m, k = ids.shape
    if c["kind"] == "greedy":
        offsets = np.arange(m + 1, dtype=np.int64) * k
        return dict(case=c, weights=weights, csr=mpt.to_csr((offsets, ids.reshape(-1).astype(np.int64))))
    # strings in one global order, the most frequent passage first
    count = np.bincount(ids.reshape(-1), minlength=n)
    rank = np.empty(n, dtype=np.int64)
    rank[np.lexsort((np.arange(n), -count))] = np.arange(n)
    ids = np.take_along_axis(ids, np.argsort(rank[ids], axis=1), 1)
    # the last passages of some requests did not fit their context: strings of several lengths
    keep = np.arange(k)[None, :] < rng.integers(max(1, k // 2), k + 1, size=m)[:, None]
    offsets = np.concatenate([[0], np.cumsum(keep.sum(1))]).astype(np.int64)
    flat = ids[keep].astype(np.int64)
    one = float(weights[flat].sum()) / m
    caps = [int(round(f * one)) for f in (0.25, 0.5, 0.75, 0.9, 1, 4, 16, 64, 256, 1024)]
    return dict(case=c, weights=weights, n=n, csr=(offsets, flat), caps=caps)


# ---------------------------------------------------------------------------
# One pass
# ---------------------------------------------------------------------------

def run(state):
    kind = state["case"]["kind"]
    if kind == "solve":
        tables = state["case"]["tables"]
        res = mpt.solve(state["weights"], state["bits"], workspace=state["ws"], tables=tables)
        views = mpt.mpt_tables(res.ctx) if tables == "int64" else mpt.mpt_tables32(res.ctx)
        return dict(opt=res.opt, perm_offsets=res.perm_offsets, perm_chunks=res.perm_chunks, dfs=res.dfs_order,
                    tables=list(views))
    if kind == "batch":
        b = mpt.mpt_batch_create(state["weights"], state["inst"], state["offsets"], state["ids"])
        mpt.mpt_batch_solve(b, state["ws"])
        opt, perm, dfs = mpt.mpt_batch_results(b)
        F, split, offsets = mpt.mpt_batch_tables(b)
        return dict(opt=opt, perm=perm, dfs=dfs, F=F, split=split, offsets=offsets)
    if kind == "greedy":
        g = mpt.mpt_greedy(state["weights"], state["csr"])
        total = int(state["csr"][0][-1])
        perm = np.fromiter(itertools.chain.from_iterable(g.perms), dtype=np.int64, count=total)
        return dict(cost=g.cost, savings=g.savings, lower_bound=g.lower_bound, merges=g.merges, values=g.merge_values,
                    perm=perm, dfs=g.dfs_order)
    order = mpt.mpt_serve_order(state["n"], state["csr"], window=state["case"]["window"])
    costs, unbounded = mpt.mpt_cache_costs(state["weights"], state["csr"], state["caps"], order)
    return dict(order=order, costs=costs, unbounded=unbounded)


def work(case):
    """Inputs read once and outputs written once.  How many splits have to be looked at depends on
    the requests, so no operations are stated."""
    c = case
    if c["kind"] == "solve":
        words = (c["n"] + 63) // 64
        per_subset = 20 if c["tables"] == "int64" else 8
        return {"bytes": 8 * c["n"] + 8 * c["m"] * words + per_subset * 2 ** c["m"] + 8 * c["m"] * c["k"], "flops": 0}
    if c["kind"] == "batch":
        sizes = range(c["m_lo"], c["m_hi"] + 1)
        mean_m = sum(sizes) / len(sizes)
        subsets = sum(2 ** m for m in sizes) / len(sizes)
        return {"bytes": c["count"] * (12 * subsets + (16 * c["k"] + 4) * mean_m + 8) + 8 * c["n"], "flops": 0}
    if c["kind"] == "greedy":
        return {"bytes": 16 * c["m"] * c["k"] + 20 * c["m"], "flops": 0}
    return {"bytes": 2 * 8 * c["m"] * c["k"] + 12 * c["m"], "flops": 0}


def tolerance(case):
    return "exact"  # whole numbers throughout


def exact(case, seed):
    """The recurrence of a small exact solve as plain numpy gives it (tables only)."""
    if case["kind"] != "solve" or case["m"] > 12:
        return None
    weights, bits = _instance(case, seed)
    m, N = case["m"], 1 << case["m"]
    used = np.flatnonzero(np.unpackbits(np.bitwise_or.reduce(bits).astype("<u8").view(np.uint8), bitorder="little"))
    rows = [np.unpackbits(row.astype("<u8").view(np.uint8), bitorder="little")[used].astype(bool) for row in bits]
    weights = weights[used]
    wI = np.zeros(N, dtype=np.int64)
    wI[0] = weights[np.logical_or.reduce(rows)].sum()
    for S in range(1, N):
        wI[S] = weights[np.logical_and.reduce([rows[i] for i in range(m) if S >> i & 1])].sum()
    F, split = np.zeros(N, dtype=np.int64), np.zeros(N, dtype=np.int64)
    every = np.arange(N)
    for S in range(1, N):
        low = S & -S
        if S == low:
            F[S] = wI[S]
            continue
        A = every[(every & ~S) == 0]
        A = A[((A & low) != 0) & (A != S)]
        v = F[A] + F[S ^ A]
        j = int(np.argmin(v))  # the smallest A among equals
        F[S], split[S] = v[j] - wI[S], A[j]
    tables = [F, wI, split] if case["tables"] == "int64" else [F, split]
    return dict(opt=int(F[-1]), perm_offsets=None, perm_chunks=None, dfs=None, tables=tables)
