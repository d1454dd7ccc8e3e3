"""mpt_greedy (Sec. 6.2 hierarchy, Sec. 6.3 bound) against the oracle and the paper."""

import numpy as np
import pytest

import oracle as O
from paper_2609_13692_gb300 import instances as I
from tests import oracle_pins as P

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def mpt():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2609_13692_gb300 import build as B

    B.build()
    O.build()
    from paper_2609_13692_gb300 import mpt as M

    M.load()
    return M


def _check(mpt, inst):
    reqs = [sorted(r) for r in O.request_sets(inst.weights, inst.bits)]
    got = mpt.mpt_greedy(inst.weights, reqs)
    ref = O.greedy(inst.weights, inst.bits)
    assert [tuple(x) for x in got.merges.tolist()] == [(a, b) for a, b, _ in ref["merges"]]
    assert got.merge_values.tolist() == [v for _, _, v in ref["merges"]]
    assert got.savings == ref["savings"] and got.cost == ref["cost"]
    assert got.lower_bound == O.spanning_tree_bound(inst.weights, inst.bits)
    assert got.perms == ref["perms"]
    assert got.dfs_order.tolist() == ref["dfs"]
    return got


@pytest.mark.parametrize("m", [1, 2, 3, 7, 20, 64, 150])
def test_greedy_random(mpt, m):
    inst = I.random_instance(m, 400, (0, 12), seed=100 + m, wmin=1, wmax=300, allow_empty=True)
    _check(mpt, inst)


def test_greedy_rag_and_ties(mpt):
    _check(mpt, I.config(1))
    _check(mpt, I.config(3))          # m = 24 RAG-shaped groups
    _check(mpt, I.tightness_witness())
    _check(mpt, I.leave_one_out(24))  # all ties


def test_greedy_leave_one_out_printed(mpt):
    """Sec. 6.2: greedy is exactly optimal on L_n, n = 16, 32, 64, 128 -> 64, 160, 384, 896."""
    for n, free in P.GOLDEN["greedy_on_loo"]["rows"]:
        inst = I.leave_one_out(n)
        reqs = [sorted(r) for r in O.request_sets(inst.weights, inst.bits)]
        g = mpt.mpt_greedy(inst.weights, reqs)
        assert g.cost == free
        assert O.trie_cost_sorted(inst.weights, g.perms) == free


def test_greedy_large_trace_shape(mpt):
    """m = 3000 requests of k = 8 passages (the size of the paper's NFCorpus
    trace): layout validity, Thm 6 (i) monotone merges, bound <= greedy."""
    rng = np.random.default_rng(3)
    n = 3600
    weights = rng.integers(50, 400, size=n).astype(np.int64)
    pools = [rng.choice(n, size=60, replace=False) for _ in range(200)]
    reqs = []
    for _ in range(3000):
        pool = pools[int(rng.integers(len(pools)))]
        chosen = set()
        while len(chosen) < 8:
            chosen.add(int(pool[int(rng.integers(60))]) if rng.random() < 0.85 else int(rng.integers(n)))
        reqs.append(sorted(chosen))
    g = mpt.mpt_greedy(weights, reqs)
    assert all(sorted(p) == r for p, r in zip(g.perms, reqs))
    assert sorted(g.dfs_order.tolist()) == list(range(3000))
    v = g.merge_values
    assert bool(np.all(v[:-1] >= v[1:]))
    assert g.lower_bound <= g.cost
    assert O.trie_cost_sorted(weights, g.perms) <= g.cost


def _host_greedy(weights, reqs):
    """The merges of O.greedy from a matrix of pair weights (m in the hundreds)."""
    m, n = len(reqs), len(weights)
    sig = np.zeros((m, n), dtype=np.int64)
    for i, r in enumerate(reqs):
        sig[i, r] = 1
    W = np.triu((sig * weights) @ sig.T, 1)
    W[np.tril_indices(m)] = -1
    merges = []
    for _ in range(m - 1):
        a, b = divmod(int(W.argmax()), m)  # ties: the smallest pair
        merges.append((a, b, int(W[a, b])))
        sig[a] &= sig[b]
        W[b, :] = W[:, b] = -1
        row = sig @ (sig[a] * weights)
        W[a, a + 1:] = np.where(W[a, a + 1:] >= 0, row[a + 1:], -1)
        W[:a, a] = np.where(W[:a, a] >= 0, row[:a], -1)
    return merges


def _many_round_cases():
    """Requests whose pairs tie or wait for one another: one merge per round."""
    rng = np.random.default_rng(8)
    n = 400
    w = rng.integers(1, 200, size=n).astype(np.int64)
    pools = [rng.choice(n - 1, size=20, replace=False) for _ in range(30)]
    pooled = [sorted(int(x) for x in rng.choice(pools[rng.integers(30)], size=5, replace=False)) for _ in range(500)]
    yield "pooled", w, pooled
    yield "one passage in all", w, [r + [n - 1] for r in pooled]
    yield "one passage in all, equal weights", np.full(n, 7), [r + [n - 1] for r in pooled]
    yield "nothing else", np.arange(1, 602), [[i, 600] for i in range(600)]
    yield "windows, equal weights", np.full(520, 3), [list(range(i, i + 8)) for i in range(512)]
    yield "a path, rising weights", np.arange(1, 500), [[i, i + 1] for i in range(450)]
    yield "nested", w, [list(range(1 + 3 * (i % 40))) for i in range(300)]
    for m in (32, 33, 64, 65):  # edges of the choice between rounds and one block
        yield f"m={m}", w, [r + [n - 1] * (i % 3 > 0) for i, r in enumerate(pooled[:m])]


@pytest.mark.parametrize("case", list(_many_round_cases()), ids=lambda c: c[0].replace(" ", "_"))
def test_greedy_many_rounds(mpt, case):
    _, w, reqs = case
    w = np.asarray(w, dtype=np.int64)
    g = mpt.mpt_greedy(w, reqs)
    assert list(zip(*g.merges.T.tolist(), g.merge_values.tolist())) == _host_greedy(w, reqs)
    assert all(sorted(p) == sorted(r) for p, r in zip(g.perms, reqs))
    assert O.trie_cost_sorted(w, g.perms) <= g.cost


def test_greedy_common_passage_takes_no_longer_than_its_merges(mpt):
    """3,000 requests that share one passage and nothing else: every pair ties,
    so one pair merges per round.  Some four times the time of pooled requests
    (31 times when all of it ran in rounds that scanned every row)."""
    import time

    rng = np.random.default_rng(3)
    m, n = 3000, 3600
    w = rng.integers(50, 400, size=2 * n).astype(np.int64)
    pools = [rng.choice(n, size=60, replace=False) for _ in range(200)]
    pooled = mpt.to_csr([sorted(rng.choice(pools[rng.integers(200)], size=8, replace=False).tolist()) for _ in range(m)])
    common = mpt.to_csr([[i, n] for i in range(m)])

    def seconds(reqs):
        best = 10.0
        for _ in range(4):
            t = time.perf_counter()
            mpt.mpt_greedy(w, reqs)
            best = min(best, time.perf_counter() - t)
        return best

    assert seconds(common) < 12 * seconds(pooled)
