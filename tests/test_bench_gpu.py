"""bench.py's lines where a solve does not evaluate every split."""

import json
import subprocess
import sys
from pathlib import Path

import pytest

pytestmark = pytest.mark.gpu

ROOT = Path(__file__).resolve().parent.parent


def _line(*args):
    r = subprocess.run([sys.executable, "bench.py", "--steps", "3", "--warmup", "3", "--no-cpu-baseline", *args],
                       cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
    return json.loads(r.stdout.strip().splitlines()[-1])


def test_auto_reports_a_time():
    """Pruned solves (m = 24, passages of 10): seconds per solve, no split
    rate, no roofline; leave-one-out at m = 20 looks at every split."""
    line = _line("--dp-mode", "auto", "--workload", "3")
    assert line["unit"] == "s" and line["roofline"] is None and line["e2e"]["unit"] == "s"
    assert not line["higher_is_better"] and 0 < line["value"] < line["e2e"]["value"] < 0.1
    line = _line("--dp-mode", "auto", "--workload", "2")
    assert line["unit"] == "splits/s" and line["roofline"]["kernel"] == "k_dp_pairs"


def test_batch_reports_instances():
    line = _line("--mode", "batch", "--batch-size", "300")
    assert line["unit"] == "instances/s" and "splits_per_s" not in line
