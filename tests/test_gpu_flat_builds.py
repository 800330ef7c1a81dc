"""Builds and rebuilds without rounds, launched directly: in a fresh process
(the option "graph_rounds" not set) trees on both sides of every base-case
size, and updates whose rebuilt subtrees all fit shared memory, equal the
oracle's; they record no graph, a build with rounds does."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

_FRESH = r'''
import sys
import numpy as np
sys.path.insert(0, sys.argv[1])
import oracle as O
from paper_2411_09275_gb300 import inputs as I, pkd
from tests import treeutil as U
from tests.gpuutil import ids_dev, make_points, oparams, to_dev

def graphs():
    return pkd.pkd_kernel_stats("graph_builds")[0]

for d, kind in ((1, "uniform"), (2, "varden"), (3, "uniform"), (3, "dups"), (5, "uniform"), (8, "varden")):
    p = pkd.Params(d=d, phi=16, sigma_log2=3, sigma_os=8)
    # (a CTA holds about 7500 3-D points, 3400 8-D ones; the inserts add half)
    for n in (1, 16, 17, 128, 129, 256, 257, 512, 513, 2000) + ((3800,) if d <= 5 else ()):
        X = make_points(kind, n, d, 700 + n)
        ids = (np.arange(n, dtype=np.uint64) * 2654435761 % (1 << 32)).astype(np.uint32)
        g0 = graphs()
        t = pkd.Tree(to_dev(X), ids_dev(ids), p)
        assert graphs() == g0, (d, n)
        o = O.OracleTree(X, ids, oparams(p))
        U.assert_exports_equal(t.export(), o.export())
        # leaves, some of them split, and (skewed points) whole subtrees rebuilt
        Y = make_points(kind, n // 2 + 3, d, 900 + n)
        Y[: n // 4, 0] //= 64
        yid = np.setdiff1d((np.arange(len(Y) + 64, dtype=np.uint64) * 40503 + 11).astype(np.uint32), ids)[: len(Y)]
        t.insert(to_dev(Y), ids_dev(yid))
        o.insert(Y, yid)
        U.assert_exports_equal(t.export(), o.export())
        gone = np.concatenate([ids[: n // 3], yid[::2]])
        assert t.delete(ids_dev(gone)) == o.delete(gone)
        U.assert_exports_equal(t.export(), o.export())
        assert graphs() == g0, (d, n)
        t.close()
# ids 0..n-1 (their table is written slot by slot): every id is found again, at
# the sizes where the table has one chunk, a few, and just fits
for d in (1, 2, 3, 4, 6, 8):
    for n in (1, 31, 32, 33, 614, 615, 5000):
        X = I.uniform(n, d, n + d)
        p = pkd.Params(d=d)
        t, o = pkd.Tree(to_dev(X), None, p), O.OracleTree(X, None, oparams(p))
        for bad in (0, n - 1):
            try:
                t.insert(to_dev(X[:1]), ids_dev(np.array([bad], np.uint32)))
                raise AssertionError("a stored id was inserted")
            except pkd.PkdError:
                pass
        gone = np.arange(n + 5, dtype=np.uint32)[::2].copy()
        assert t.delete(ids_dev(gone)) == o.delete(gone)
        U.assert_exports_equal(t.export(), o.export())
        back = gone[gone < n][::3].copy()
        t.insert(to_dev(X[back]), ids_dev(back))
        o.insert(X[back], back)
        rest = np.arange(n, dtype=np.uint32)
        assert t.delete(ids_dev(rest)) == o.delete(rest) and t.size == 0
        t.close()
g0 = graphs()
X = I.uniform(100000, 3, 5)
p = pkd.Params(d=3)
t = pkd.Tree(to_dev(X), None, p)
assert graphs() == g0 + 1
U.assert_exports_equal(t.export(), O.OracleTree(X, None, oparams(p)).export())
# more build shapes than the graph cache holds: evicted graphs and fresh ones
pkd.pkd_set_option("base_cap", 256)
p = pkd.Params(d=2, phi=8, lam=3, sigma_log2=2, sigma_os=4)
for i in range(80):
    X = make_points("uniform", 3000 + 17 * (i % 75), 2, i)
    t = pkd.Tree(to_dev(X), None, p)
    if i % 8 == 0 or i > 74:
        U.assert_exports_equal(t.export(), O.OracleTree(X, None, oparams(p)).export())
    t.close()
print("RESULT ok")
'''


def test_builds_without_rounds_match_the_oracle():
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", _FRESH, root], capture_output=True, text=True, timeout=600)
    assert r.returncode == 0 and "RESULT ok" in r.stdout, r.stdout[-2000:] + r.stderr[-2000:]
