"""The pruned recurrence (AUTO) against the full one (BLOCKED), table for table.

AUTO leaves out splits whose named part has more than one request and no
common weight; by the exchange argument in k_dp_pruned.cu that changes no
F(S) and no split(S).  The cases sit where the rule or its kernels could go
wrong: one tile bit, list lengths around the short/long limit (128), both
tile widths of the sparse kernel, requests without chunks, identical
requests, ties, a universal chunk, instances that must stay with the full
recurrence.
"""

import subprocess
import sys
from pathlib import Path

import numpy as np
import pytest

import oracle as O
from paper_2609_13692_gb300 import instances as I

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


def _from_supports(m, supports, seed, wmax=9):
    """One chunk per request set in `supports` (bit masks), weights 1..wmax."""
    w = np.random.default_rng(seed).integers(1, wmax + 1, size=len(supports)).astype(np.int64)
    reqs = [[x for x, N in enumerate(supports) if N >> i & 1] for i in range(m)]
    return I.Instance(w, I.pack_requests(reqs, len(supports)), f"supports m={m}")


def _mask(*bits):
    return sum(1 << b for b in bits)


def _cases():
    rng = np.random.default_rng(5)
    for m in range(13, 23):
        yield I.rag_pools(m, 3000, 5, 40, 8, 1.1, seed=m)
    for m in (13, 14, 17, 19):
        yield I.zipf_small(m, 60, 5, 1.0, seed=m)
        yield I.random_instance(m, 40, (0, 9), seed=m, wmin=1, wmax=3, allow_empty=True)
    yield I.leave_one_out(15)
    m = 18
    # inner parts of 6, 7 and 8 requests (2^6 .. 2^8 listed sets), alone and
    # nested in tile parts of several sizes
    for inner in (6, 7, 8):
        top = _mask(*range(6, 6 + inner))
        yield _from_supports(m, [top | _mask(0, 2, 5)], inner)
        yield _from_supports(m, [top | _mask(1), top | _mask(1, 3), _mask(0, 1, 2, 3, 4, 5), _mask(2, 17)], inner)
    # all requests inside one tile part; no shared chunk at all; identical requests
    yield _from_supports(m, [_mask(0, 1, 2), _mask(3, 4, 5), _mask(0, 5)], 1)
    yield _from_supports(m, [1 << i for i in range(m)], 2)
    yield I.Instance(np.ones(3, dtype=np.int64), I.pack_requests([[0, 1]] * 9 + [[2]] * 8, 3), "identical")
    yield I.with_common_prefix(_from_supports(m, [int(x) for x in rng.integers(1, 1 << m, 12) & rng.integers(1, 1 << m, 12)], 3, 1), 77)
    # many small sets: every tile has short lists
    pairs = [_mask(i, j) for i in range(16) for j in range(i)]
    yield _from_supports(16, pairs, 4, 2)
    # one large set among small ones: long lists beside short ones
    yield _from_supports(20, [_mask(*range(0, 20, 2)), _mask(*range(3, 20)), _mask(0, 1), _mask(1, 19)], 6)
    yield _from_supports(20, [(1 << 20) - 2, _mask(0, 1), _mask(4, 12, 13)], 7)


@pytest.mark.parametrize("inst", list(_cases()), ids=lambda inst: inst.name.replace(" ", "_")[:40])
def test_equals_the_full_recurrence(mpt, inst):
    a = mpt.solve(inst.weights, inst.bits, mode="auto")
    b = mpt.solve(inst.weights, inst.bits, mode="blocked")
    assert a.opt == b.opt
    for x, y in zip(mpt.mpt_tables(a.ctx), mpt.mpt_tables(b.ctx)):
        assert torch.equal(x, y)
    assert a.perm_chunks.tolist() == b.perm_chunks.tolist() and a.dfs_order.tolist() == b.dfs_order.tolist()
    lean = mpt.solve(inst.weights, inst.bits, tables="lean")
    F, split = mpt.mpt_tables32(lean.ctx)
    assert lean.opt == b.opt and torch.equal(split, mpt.mpt_tables(b.ctx)[2])
    assert torch.equal(F.long(), mpt.mpt_tables(b.ctx)[0])


@pytest.mark.parametrize("inst", [c for c in _cases() if c.m <= 20], ids=lambda inst: inst.name.replace(" ", "_")[:40])
def test_wide_equals_the_full_recurrence(mpt, inst):
    """The same with weights too heavy for the 32-bit keys."""
    w = inst.weights << 21
    a = mpt.solve(w, inst.bits, mode="auto")
    b = mpt.solve(w, inst.bits, mode="wide")
    assert a.opt == b.opt
    for x, y in zip(mpt.mpt_tables(a.ctx), mpt.mpt_tables(b.ctx)):
        assert torch.equal(x, y)
    assert a.perm_chunks.tolist() == b.perm_chunks.tolist() and a.dfs_order.tolist() == b.dfs_order.tolist()


def test_wide_many_members(mpt):
    """64-bit keys beyond one queue of pairs (more than 512 members per
    lowest request) and lists of more than 32 rows."""
    inst = _from_supports(24, [_mask(*range(0, 24, 2)) | _mask(1, 3, 5, 7, 9), _mask(*range(0, 12)), _mask(2, 13),
                               _mask(0, *range(12, 24)), _mask(3, 20)], 8)
    a = mpt.solve(inst.weights << 21, inst.bits)
    b = mpt.solve(inst.weights, inst.bits, mode="blocked")
    assert a.opt == b.opt << 21
    Fa, wa, sa = mpt.mpt_tables(a.ctx)
    Fb, wb, sb = mpt.mpt_tables(b.ctx)
    assert torch.equal(Fa, Fb << 21) and torch.equal(wa, wb << 21) and torch.equal(sa, sb)


@pytest.mark.parametrize("scale", [1, 1 << 21])
def test_long_lists_in_a_fresh_process(mpt, scale):
    """The first solve of a process meets a tile with a long list in step 1,
    before any launch that raises the kernels' shared-memory limits."""
    code = ("import numpy as np; from tests.test_pruned_gpu import _from_supports, _mask\n"
            "from paper_2609_13692_gb300 import mpt\n"
            "inst = _from_supports(20, [_mask(*range(0, 20, 2)), _mask(*range(3, 20)), _mask(0, 1), _mask(1, 19)], 6)\n"
            f"print(mpt.solve(inst.weights * {scale}, inst.bits).opt // {scale})")
    root = Path(__file__).resolve().parent.parent
    r = subprocess.run([sys.executable, "-c", code], cwd=root, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
    inst = _from_supports(20, [_mask(*range(0, 20, 2)), _mask(*range(3, 20)), _mask(0, 1), _mask(1, 19)], 6)
    assert int(r.stdout) == mpt.solve(inst.weights, inst.bits, mode="blocked").opt


def test_route(mpt):
    """Few shared chunks: no pair kernel.  Leave-one-out: the full one."""
    few = I.rag_pools(18, 3000, 5, 40, 8, 1.2, seed=3)
    assert mpt.mpt_get_profile(mpt.solve(few.weights, few.bits).ctx)["launches_pairs"] == 0
    loo = I.leave_one_out(16)
    p = mpt.mpt_get_profile(mpt.solve(loo.weights, loo.bits).ctx)
    assert p["launches_pairs"] == 3 and p["splits_pairs"] > 0


@pytest.mark.parametrize("inner,launches", [(7, 0), (8, 0), (10, 5)])
def test_kernels_for_long_lists(mpt, inner, launches):
    """Three sets with the same inner requests: their bounds add up to long
    lists, their lists are one of 128 members, of 256 members in 8 rows (the
    row kernel alone), of 1,024 members in 32 rows (the pair kernel too)."""
    top = _mask(*range(6, 6 + inner))
    inst = _from_supports(18, [top | _mask(0), top | _mask(0, 1), top | _mask(0, 2), _mask(3, 17)], inner)
    test_equals_the_full_recurrence(mpt, inst)
    test_wide_equals_the_full_recurrence(mpt, inst)
    r = mpt.solve(inst.weights, inst.bits, profile=True)
    assert mpt.mpt_get_profile(r.ctx)["launches_pairs"] == launches


@pytest.mark.parametrize("m", [13, 16, 17, 20])
@pytest.mark.parametrize("scale", [1, 1 << 21])
def test_tables_from_a_used_workspace(mpt, m, scale):
    """w(I) is written only in tiles with a member: what lay in the workspace
    before must not show in the tables, at one, 16 and 32 tile parts or more."""
    inst = I.rag_pools(m, 3000, 5, 40, 8, 1.1, seed=m)
    w = inst.weights * scale
    ref = mpt.solve(w, inst.bits, mode="blocked" if scale == 1 else "wide")
    for kind in ("int64", "lean") if scale == 1 else ("int64",):
        ctx = mpt.mpt_create(w, inst.bits)
        mpt.mpt_set_tables(ctx, kind)
        ws = torch.full((mpt.mpt_workspace_bytes(ctx),), 0xA5, dtype=torch.uint8, device="cuda")
        assert mpt.mpt_solve(ctx, ws) == ref.opt
        F, wI, split = mpt.mpt_tables(ref.ctx)
        if kind == "int64":
            for x, y in zip(mpt.mpt_tables(ctx), (F, wI, split)):
                assert torch.equal(x, y)
        else:
            F32, split32 = mpt.mpt_tables32(ctx)
            assert torch.equal(F32.long(), F) and torch.equal(split32, split)


@pytest.mark.parametrize("scale", [1, 1 << 21])
@pytest.mark.parametrize("inner", [5, 6])
def test_rows_counted_in_stored_order(mpt, scale, inner):
    """A list of 2^inner members in one or two rows by the natural order of the
    inner bits, and in 2^inner rows by the stored one, which has the bits of
    costlier sets in front."""
    inst = _from_supports(18, [_mask(1, 2, 3, 4, *range(12, 16)), _mask(1, 2, 3, 4, 16, 17),
                               _mask(5, *range(6, 6 + inner))], inner)
    if scale == 1:
        test_equals_the_full_recurrence(mpt, inst)
    else:
        test_wide_equals_the_full_recurrence(mpt, inst)


@pytest.mark.parametrize("scale", [1, 1 << 12])
def test_sorted_tiles(mpt, scale):
    """Enough pairs that the tiles of a layer are taken from the most work to
    the least (two launches more), tile bits and classes of several sizes."""
    top = _mask(*range(12, 20))
    inst = _from_supports(23, [top | _mask(*range(0, 8)), top | _mask(*range(1, 9)), top | _mask(0, *range(2, 9)),
                               _mask(0, 10, 21), _mask(9, 10, 11)], 23, 400)
    w = inst.weights * scale
    a, b = mpt.solve(w, inst.bits), mpt.solve(w, inst.bits, mode="blocked" if scale == 1 else "wide")
    assert a.opt == b.opt
    for x, y in zip(mpt.mpt_tables(a.ctx), mpt.mpt_tables(b.ctx)):
        assert torch.equal(x, y)
    # K1, lists (2), sort (2), tile 0, 11 layers of tiles, long ones (11), pairs, walk
    p = mpt.mpt_get_profile(mpt.solve(w, inst.bits, profile=True).ctx)
    assert p["launches_total"] == 7 + 11 + 11 + p["launches_pairs"]


@pytest.mark.parametrize("seed", [0, 1, 2])
def test_m24_equals_the_full_recurrence(mpt, seed):
    inst = I.config(3, seed=seed)
    a = mpt.solve(inst.weights, inst.bits)
    b = mpt.solve(inst.weights, inst.bits, mode="blocked")
    assert all(torch.equal(x, y) for x, y in zip(mpt.mpt_tables(a.ctx), mpt.mpt_tables(b.ctx)))


def _groups(seed):
    """Groups of 6..16 requests: pooled passages (few members), one chunk in
    every request, no shared chunk, identical requests, and nearly everything
    shared (too many members for the list)."""
    rng = np.random.default_rng(seed)
    n = 400
    out = []
    for m in list(range(6, 17)) * 2:
        pool = rng.choice(n - 20, size=40, replace=False)
        base = [[int(x) for x in rng.choice(pool, size=6, replace=False)] for _ in range(m)]
        out.append(base)
        out.append([r + [n - 1] for r in base])
        out.append([[(17 * i + j) % (n - 20) for j in range(3)] for i in range(m)])
        out.append([[1, 2, 3]] * m)
        out.append([[n - 20 + j for j in range(min(m, 12)) if j != i] for i in range(m)])
        out.append([[int(x)] if x % 3 else [] for x in rng.integers(0, 9, size=m)])
    return rng.integers(1, 30, size=n).astype(np.int64), out


@pytest.mark.parametrize("scale", [1, 1 << 12])
def test_batch_equals_single_solves(mpt, scale):
    w, groups = _groups(3)
    w = w * scale
    if scale > 1:  # 16 requests need packed keys
        groups = [g for g in groups if len(g) <= 14]
    opt, perms, orders, b = mpt.solve_batch(w, groups)
    F, split, offs = mpt.mpt_batch_tables(b)
    for i, g in enumerate(groups):
        one = mpt.solve(w, I.pack_requests(g, len(w)), mode="wide" if scale > 1 else "blocked")
        tF, _, ts = mpt.mpt_tables(one.ctx)
        assert opt[i] == one.opt and perms[i] == one.permutations() and orders[i] == one.dfs_order.tolist(), i
        assert torch.equal(F[offs[i]:offs[i + 1]], tF) and torch.equal(split[offs[i]:offs[i + 1]], ts), i


@pytest.mark.parametrize("m", [14, 15, 16])
def test_batch_members_and_rows(mpt, m):
    """From 14 requests on, groups of few members are solved by a kernel of
    their own and the others left to the row form: both kinds in one call, with
    and without heavy private and common chunks, and requests so long that the
    lists find no room."""
    rng = np.random.default_rng(m)
    w = np.concatenate([rng.integers(1, 9, size=600), np.full(m + 1, 1 << 26)]).astype(np.int64)
    loo = [[x for x in range(m) if x != i] for i in range(m)]
    groups = [loo]
    for g in range(5):
        pool = rng.choice(np.arange(m, 600), size=40 + 20 * g, replace=False)
        groups.append([sorted(rng.choice(pool, size=int(rng.integers(0, 6)), replace=False).tolist()) for _ in range(m)])
    groups += [[r + [600, 601 + i] for i, r in enumerate(g)] for g in groups[:3]]
    groups.append([[]] * m)
    for more in ([], [[sorted(rng.choice(600, size=int(rng.integers(45, 60)), replace=False).tolist()) for _ in range(m)]]):
        opt, perms, orders, b = mpt.solve_batch(w, groups + more)
        F, split, offs = mpt.mpt_batch_tables(b)
        for i, g in enumerate(groups + more):
            one = mpt.solve(w, I.pack_requests(g, len(w)), mode="blocked")
            tF, _, ts = mpt.mpt_tables(one.ctx)
            assert opt[i] == one.opt and perms[i] == one.permutations() and orders[i] == one.dfs_order.tolist(), i
            assert torch.equal(F[offs[i]:offs[i + 1]], tF) and torch.equal(split[offs[i]:offs[i + 1]], ts), i


@pytest.mark.parametrize("m", [6, 9, 11, 12, 13])
def test_batch_members_of_many_groups(mpt, m):
    """Below 14 requests the members are tried from some two thousand groups of
    one size on: one call of 2,400 against three of 800."""
    rng = np.random.default_rng(100 + m)
    w = rng.integers(1, 9, size=400).astype(np.int64)
    groups = []
    for _ in range(2400):
        pool = rng.choice(400, size=int(rng.integers(8, 60)), replace=False)
        groups.append([rng.choice(pool, size=int(rng.integers(0, 7)), replace=False).tolist() for _ in range(m)])
    opt, perms, orders, b = mpt.solve_batch(w, groups)
    F, split, _ = mpt.mpt_batch_tables(b)
    for k in range(0, 2400, 800):
        o, p, d, part = mpt.solve_batch(w, groups[k:k + 800])
        pF, ps, _ = mpt.mpt_batch_tables(part)
        assert list(o) == list(opt[k:k + 800]) and p == perms[k:k + 800] and d == orders[k:k + 800]
        assert torch.equal(pF, F[k << m:(k + 800) << m]) and torch.equal(ps, split[k << m:(k + 800) << m])


def _heavy_sets(m, size, count, seed):
    rng = np.random.default_rng(seed)
    sets = [_mask(*(int(i) for i in rng.choice(m, size=size, replace=False))) for _ in range(count)]
    pairs = [_mask(*(int(i) for i in rng.choice(m, size=2, replace=False))) for _ in range(30)]
    return _from_supports(m, sets + pairs, seed)


@pytest.mark.parametrize("m,size,count,scale", [(19, 17, 1, 1 << 12), (20, 15, 3, 1 << 12), (22, 18, 2, 1 << 12),
                                                (20, 14, 4, 1), (21, 15, 2, 1)])
def test_heavy_lists_stay_with_the_full_recurrence(mpt, m, size, count, scale):
    """A few chunks that most requests hold: lists so long that the full
    recurrence is the faster one (the pruned one took two to ten times as
    long): AUTO launches what the full form launches."""
    inst = _heavy_sets(m, size, count, m + size)
    w = inst.weights * scale
    got = [mpt.mpt_get_profile(mpt.solve(w, inst.bits, mode=mode, profile=True).ctx)
           for mode in ("auto", "wide" if scale > 1 else "blocked")]
    assert got[0]["launches_total"] == got[1]["launches_total"]
    assert got[0]["splits_pairs"] == got[1]["splits_pairs"] > 0


@pytest.mark.parametrize("scale", [1, 1 << 21])
def test_long_lists_of_a_pruned_solve_in_a_fresh_process(mpt, scale):
    """As test_long_lists_in_a_fresh_process, on an instance large enough that
    its long lists do not send it to the full recurrence."""
    sets = "_mask(*range(0, 24, 2)) | _mask(1, 3, 5, 7, 9), _mask(*range(0, 12)), _mask(2, 13), _mask(0, *range(12, 24)), _mask(3, 20)"
    code = ("import numpy as np; from tests.test_pruned_gpu import _from_supports, _mask\n"
            "from paper_2609_13692_gb300 import mpt\n"
            f"inst = _from_supports(24, [{sets}], 8)\n"
            f"r = mpt.solve(inst.weights * {scale}, inst.bits, profile=True)\n"
            "print(r.opt, mpt.mpt_get_profile(r.ctx)['launches_total'])")
    root = Path(__file__).resolve().parent.parent
    r = subprocess.run([sys.executable, "-c", code], cwd=root, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
    opt, launches = (int(x) for x in r.stdout.split())
    inst = _from_supports(24, eval(f"[{sets}]"), 8)
    full = mpt.solve(inst.weights * scale, inst.bits, mode="wide" if scale > 1 else "blocked", profile=True)
    assert opt == full.opt and launches != mpt.mpt_get_profile(full.ctx)["launches_total"]


def test_more_pairs_than_a_queue(mpt):
    """32-bit keys beyond one queue of pairs: a chunk held by 12 of the 17 tile
    requests of 29 leaves tiles of 11 requests 1,023 pairs in one group, in
    more than one round (12,376 tiles are too many to be cut into parts); another
    that shares most of them, and pairs around both."""
    inst = _from_supports(29, [_mask(*range(0, 12), 20), _mask(*range(1, 13), 21, 22), _mask(0, 13, 25), _mask(5, 28)], 29, 60)
    got = []
    for mode in ("auto", "blocked"):
        r = mpt.solve(inst.weights, inst.bits, mode=mode, tables="lean")
        got.append((r.opt, r.perm_chunks.tolist(), r.dfs_order.tolist(), *mpt.mpt_tables32(r.ctx)))
        assert (mpt.mpt_get_profile(r.ctx)["splits_pairs"] == 0) == (mode == "auto")
    assert got[0][:3] == got[1][:3]
    assert torch.equal(got[0][3], got[1][3]) and torch.equal(got[0][4], got[1][4])
