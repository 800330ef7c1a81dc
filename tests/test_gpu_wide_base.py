"""The base case with the SM to itself: 32 warps a CTA up to five dimensions,
in builds beside which no id table is written (forests); 16 in the others, above
five dimensions, and where a larger capacity set by the caller leaves no room for
the stacks of 32.  Trees equal the oracle's on both sides of the sizes at which a
subproblem goes to that form, with even and crowded coordinates (counting pass
and radix passes) and with children of very different sizes."""
import numpy as np
import pytest

import oracle as O
from tests import treeutil as U
from tests.gpuutil import ids_dev, knobs, make_points, oparams, to_dev

pytestmark = pytest.mark.gpu


def _check(kind, sizes, d, phi):
    from paper_2411_09275_gb300 import pkd

    X = np.concatenate([make_points(kind, n, d, n + d) for n in sizes])
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.uint64)
    if kind == "varden":
        for a, n in zip(off[:-1], sizes):
            X[int(a):int(a) + n // 16] //= 4096  # a corner that tiny children split off
    ids = (np.arange(len(X), dtype=np.uint64) * 2654435761 % (1 << 32)).astype(np.uint32)
    p = pkd.Params(d=d, phi=phi, sigma_log2=3, sigma_os=8)
    f = pkd.pkd_build_forest(to_dev(X), ids_dev(ids), off, p)
    for i in range(len(sizes)):
        a, b = int(off[i]), int(off[i + 1])
        want = O.OracleTree(X[a:b], ids[a:b], oparams(p)).export()
        U.assert_exports_equal(pkd.pkd_forest_export(f, i), want)
        t = pkd.Tree(to_dev(X[a:b]), ids_dev(ids[a:b]), p)
        U.assert_exports_equal(t.export(), want)
        t.close()
    pkd.pkd_forest_free(f)


@pytest.mark.parametrize("kind", ["uniform", "varden", "dups", "dups_big"])
@pytest.mark.parametrize("d", [1, 2, 3, 4, 5, 6])
def test_one_cta_per_sm(kind, d):
    per = 6 * d + 7  # shared memory a point, bytes
    cap = (200 * 1024 - 18200) // per // 64 * 64
    half = (112 * 1024 - 18200) // per // 64 * 64
    for phi in (1, 32):
        _check(kind, [half - 64, half + 65, (cap + half) // 2 + 1, cap - 64, cap + 65], d, phi)


@pytest.mark.parametrize("kind", ["uniform", "varden", "dups_big"])
def test_capacity_without_room_for_32_warps(kind):
    with knobs(base_cap=8256):
        _check(kind, [5000, 8255, 8256], 3, 32)
