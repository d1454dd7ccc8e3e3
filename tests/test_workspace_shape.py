"""The workspace follows from an instance's shape, not from its overlaps."""

import ctypes

import numpy as np
import pytest

from paper_2609_13692_gb300 import instances as I


@pytest.fixture(scope="module")
def mpt():
    from paper_2609_13692_gb300 import build as B
    from paper_2609_13692_gb300 import mpt as M

    B.build()
    M.load()
    return M


def _one_shape(m, k=6):
    """Instances of m requests of k chunks out of 6 m: nothing shared, windows
    over a ring, pooled (few sets), leave-one-out beside private chunks, one
    chunk in nearly all."""
    n = 6 * m
    rng = np.random.default_rng(m)
    pool = rng.choice(n, size=20, replace=False)
    yield [[k * i + j for j in range(k)] for i in range(m)]
    yield [[(i * 3 + j) % n for j in range(k)] for i in range(m)]
    yield [sorted(rng.choice(pool, size=k, replace=False).tolist()) for _ in range(m)]
    yield [[j for j in range(k + 1) if j != i % (k + 1)] for i in range(m)]
    yield [([0] if i else [n - 1]) + [1 + 5 * i + j for j in range(k - 1)] for i in range(m)]


@pytest.mark.parametrize("m", [13, 16, 20])
@pytest.mark.parametrize("scale", [1, 1 << 24])
@pytest.mark.parametrize("tables", ["int64", "lean"])
def test_size_is_one_per_shape(mpt, m, scale, tables):
    if tables == "lean" and scale > 1:
        pytest.skip("lean tables need light weights")
    sizes = {"auto": set(), "blocked": set(), "wide": set()}
    for reqs in _one_shape(m):
        w = np.full(6 * m, scale, dtype=np.int64)
        if scale > 1 and len({x for r in reqs for x in r}) == 6 * m:
            continue  # nothing shared: the 32-bit keys do
        for mode in sizes:
            if mode == "blocked" and scale > 1:
                continue
            ctx = mpt.mpt_create(w, I.pack_requests(reqs, 6 * m))
            mpt.mpt_set_dp_mode(ctx, mode)
            mpt.mpt_set_tables(ctx, tables)
            sizes[mode].add(mpt.mpt_workspace_bytes(ctx))
            mpt.mpt_destroy(ctx)
    assert all(len(s) <= 1 for s in sizes.values()), sizes
    assert sizes["auto"] == sizes["wide" if scale > 1 else "blocked"]


def _without_lists(m, n, slots):
    """Bytes of the int64 workspace with 32-bit keys and tiles of 2^12, as the
    staged solves use it: inputs, tables, layout."""
    up = lambda b: (b + 255) & ~255
    tiles = [1]
    for k in range(1, m - 11):
        tiles.append(tiles[-1] * (m - 12 - k + 1) // k)
    N = 1 << m
    return sum(up(b) for b in (8 * n, 8 * m * ((n + 63) // 64), 4 * slots, 4 * slots, 32, 8 * N, 8 * N, 4 * N, 4 * N,
                               4 * N, 8 * max(tiles) << 12, 33 * 8, 8 * slots, 8 * (m + 1), 8 * slots, 4 * m, 40))


def test_staged_solves_take_a_workspace_without_lists(mpt):
    """A checkpoint holds no lists (staged solves look at every split): it is
    resumed in a workspace of the tables and buffers alone, on an instance whose
    one-shot solve needs more.  The pointer is never dereferenced."""
    m = 16
    lib = mpt.load()
    reqs = list(_one_shape(m))[2]
    ctx = mpt.mpt_create(np.ones(6 * m, dtype=np.int64), I.pack_requests(reqs, 6 * m))
    need = _without_lists(m, 6 * m, 6 * m)
    assert need < mpt.mpt_workspace_bytes(ctx)
    at, opt = ctypes.c_void_p(1 << 20), ctypes.c_int64()
    assert lib.mpt_solve_resume(ctx.handle, at, need, 1) == 0
    assert lib.mpt_solve_resume(ctx.handle, at, need - 1, 1) == 5
    assert lib.mpt_solve(ctx.handle, at, mpt.mpt_workspace_bytes(ctx) - 1, None, ctypes.byref(opt)) == 5
    mpt.mpt_destroy(ctx)


@pytest.mark.gpu
@pytest.mark.parametrize("scale", [1, 1 << 21])
def test_one_workspace_for_all_overlaps(mpt, scale):
    """Full and pruned solves of one shape one after the other in one
    workspace, sized for the first of them."""
    import torch

    m = 16
    loo = [[x for x in range(m) if x != i] for i in range(m)]
    light = [[(i * (m - 1) + j) % 230 for j in range(m - 1)] for i in range(m)]
    w = np.arange(1, 231, dtype=np.int64) * scale
    ws = None
    for reqs in (loo, light, loo, light):
        bits = I.pack_requests(reqs, 230)
        ctx = mpt.mpt_create(w, bits)
        if ws is None:
            ws = torch.empty(mpt.mpt_workspace_bytes(ctx), dtype=torch.uint8, device="cuda")
        ref = mpt.solve(w, bits, mode="blocked" if scale == 1 else "wide")
        assert mpt.mpt_solve(ctx, ws) == ref.opt
        for x, y in zip(mpt.mpt_tables(ctx), mpt.mpt_tables(ref.ctx)):
            assert torch.equal(x, y)
