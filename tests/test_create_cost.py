"""mpt_create stays cheap where nearly every chunk is shared (no GPU needed)."""

import time

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


def _seconds(mpt, w, bits):
    best = 1.0
    for _ in range(15):
        t = time.perf_counter()
        ctx = mpt.mpt_create(w, bits)
        best = min(best, time.perf_counter() - t)
        mpt.mpt_destroy(ctx)
    return best


@pytest.mark.parametrize("m", [14, 16, 20])
def test_create_with_every_chunk_shared(mpt, m):
    """8,000 chunks, each in about half of the requests, against the same
    requests each over chunks of its own sharing nothing: the same number of
    occurrences in a universe m / 2 times as large.  The sets of the shared
    chunks are looked at only until they rule the pruned form out (taking and
    sorting all of them made it some six times the time of the other)."""
    n = 8000
    rng = np.random.default_rng(m)
    shared = [np.flatnonzero(rng.random(n) < 0.5) for _ in range(m)]
    own = n // 2
    private = [np.arange(i * own, (i + 1) * own) for i in range(m)]
    t = _seconds(mpt, np.ones(n, dtype=np.int64), I.pack_requests([x.tolist() for x in shared], n))
    t0 = _seconds(mpt, np.ones(m * own, dtype=np.int64), I.pack_requests([x.tolist() for x in private], m * own))
    assert t < 3.0 * t0, (t, t0)
