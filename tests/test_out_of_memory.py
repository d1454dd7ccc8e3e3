"""Host allocations that fail inside a C entry come back as its status (no GPU
needed: each call here fails before its first CUDA call)."""

import subprocess
import sys
import textwrap

import pytest

from paper_2609_13692_gb300 import build as B

CHILD = """
import ctypes, mmap, resource
import numpy as np
from paper_2609_13692_gb300 import mpt

lib = mpt.load()
i64, i32 = ctypes.POINTER(ctypes.c_int64), ctypes.POINTER(ctypes.c_int32)
P = lambda a, t: a.ctypes.data_as(t)
m = 1 << 22
offs = np.zeros(m + 1, dtype=np.int64)       # m empty strings
ids = np.zeros(1, dtype=np.int64)
perm = np.arange(m, dtype=np.int32)
order = np.zeros(m, dtype=np.int32)
w = np.ones(1, dtype=np.int64)
caps, costs = np.zeros(1, dtype=np.int64), np.zeros(1, dtype=np.int64)
held = int(open("/proc/self/statm").read().split()[0]) * mmap.PAGESIZE
resource.setrlimit(resource.RLIMIT_AS, (held + (1 << 20), resource.RLIM_INFINITY))  # the calls want 4 MB and more
if CALL == "serve_order":
    st = lib.mpt_serve_order(1, m, P(offs, i64), P(ids, i64), P(perm, i32), 0, None, P(order, i32))
elif CALL == "cache_costs":
    st = lib.mpt_cache_costs(P(w, i64), 1, m, P(offs, i64), P(ids, i64), P(perm, i32), P(caps, i64), 1, None,
                             P(costs, i64), None)
else:
    st = lib.mpt_layout_pinned(P(w, i64), 1, m, P(offs, i64), P(ids, i64), 1, 1, None, None, None, P(costs, i64))
print("status", st)
"""


@pytest.mark.parametrize("call", ["serve_order", "cache_costs", "layout_pinned"])
def test_a_failed_host_allocation_is_a_status(call):
    """A C++ exception that left the library would end the process."""
    B.build()
    r = subprocess.run([sys.executable, "-c", f"CALL = {call!r}\n" + textwrap.dedent(CHILD)],
                       capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stderr[-500:]
    assert r.stdout.split() == ["status", "4"], r.stdout  # MPT_ERR_OUT_OF_MEMORY
