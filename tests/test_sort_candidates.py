"""Candidates come back sorted by (dm_idx, t, width_idx): by comparisons below 256 of
them, by digits of a 64-bit key above, in place where no scratch can be had (host only)."""
import os
import subprocess
import sys

import numpy as np
import pytest

import paper_1107_2516_gb300 as dd
from paper_1107_2516_gb300 import build as ddbuild
from paper_1107_2516_gb300.dd import dd_sort_candidates

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module", autouse=True)
def _lib():
    ddbuild.build()
    dd.load()


def candidates(n, ndm, t0, span, nw, seed=1):
    rng = np.random.default_rng(seed)
    c = np.zeros(n, dd.CANDIDATE_DTYPE)
    c["dm_idx"], c["width_idx"] = rng.integers(0, ndm, n), rng.integers(0, nw, n)
    c["t"] = t0 + rng.integers(0, span, n)
    c["value"], c["snr"] = np.arange(n), rng.random(n)
    return c


# a key of one digit, of several 11-bit ones, of more than 63 bits (comparisons); negative times (boundary windows)
RANGES = [(4, 0, 16, 2), (2000, 0, 1 << 20, 6), (60000, -63, 1 << 30, 64), (1 << 30, -(1 << 40), 1 << 41, 64), (1, 7, 1, 1)]


@pytest.mark.parametrize("n", [0, 1, 2, 255, 256, 257, 511, 512, 513, 20000])
@pytest.mark.parametrize("ndm,t0,span,nw", RANGES)
def test_order_and_records(n, ndm, t0, span, nw):
    c = candidates(n, ndm, t0, span, nw)
    got = c.copy()
    dd_sort_candidates(got)
    want = c[np.lexsort((c["value"], c["width_idx"], c["t"], c["dm_idx"]))]
    for k in ("dm_idx", "t", "width_idx"):
        assert np.array_equal(got[k], want[k])
    # every record whole and once
    assert np.array_equal(np.sort(got["value"]), np.arange(n))
    assert np.array_equal(got, c[got["value"].astype(np.int64)])


def test_without_scratch():
    # 4 million hits with less address space left than their 256 MB of scratch
    code = f"""
import sys, resource
sys.path[:0] = [{ROOT!r}, {os.path.join(ROOT, "tests")!r}]
import numpy as np
from test_sort_candidates import candidates, dd_sort_candidates
import paper_1107_2516_gb300 as dd
dd.load()
c = candidates(1 << 22, 2000, 0, 1 << 20, 6)
size = int(open("/proc/self/statm").read().split()[0]) * 4096
resource.setrlimit(resource.RLIMIT_AS, (size + (32 << 20), resource.getrlimit(resource.RLIMIT_AS)[1]))
dd_sort_candidates(c)
for lo in range(0, len(c) - 1, 1 << 16):
    p = c[lo:lo + (1 << 16) + 1]
    key = (p["dm_idx"].astype(np.int64) << 30) | (p["t"] << 8) | p["width_idx"]
    assert np.all(np.diff(key) >= 0)
print("sorted")
"""
    r = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "sorted" in r.stdout, r.stderr[-2000:]
