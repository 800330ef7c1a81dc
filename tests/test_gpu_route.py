"""Batch routing by teams: a warp up to 256 batch points, a CTA up to 4096,
the sieve above; a batch of at most 4096 points queues all its rounds.  Trees
after updates equal the oracle's at the edges of those sizes, for skeletons of
1 to 10 levels, clustered batches (many points in one leaf or one subtree),
skewed ones (subtrees rebuilt, which a delete goes through too), leaves above
32 and above 1024 points, and rejected batches leave the tree as it was."""
import numpy as np
import pytest

import oracle as O
from paper_2411_09275_gb300 import inputs as I
from tests import treeutil as U
from tests.gpuutil import ids_dev, make_points, oparams, to_dev

pytestmark = pytest.mark.gpu


def _pair(kind, n, d, seed, **over):
    from paper_2411_09275_gb300 import pkd

    X = make_points(kind, n, d, seed)
    p = pkd.Params(d=d, **over)
    t, o = pkd.Tree(to_dev(X), None, p), O.OracleTree(X, None, oparams(p))
    return pkd, t, o, X


def _same(t, o):
    assert t.size == o.size
    U.assert_exports_equal(t.export(), o.export())


@pytest.mark.parametrize("m", [1, 31, 256, 257, 4096, 4097, 9000])
@pytest.mark.parametrize("kind,d,lam", [("uniform", 3, 6), ("varden", 2, 1), ("dups", 3, 3), ("uniform", 5, 10),
                                        ("varden", 8, 5), ("uniform", 1, 6)])
def test_batch_sizes(kind, d, lam, m):
    n = 30000
    pkd, t, o, X = _pair(kind, n, d, 70 + d, phi=8, lam=lam, sigma_log2=2, sigma_os=4)
    rng = np.random.default_rng(m)
    nxt = n
    for step in range(3):
        if step == 0:  # spread
            Y = make_points(kind, m, d, 71 + m)
        elif step == 1:  # skewed: subtrees leave the balance
            Y = make_points(kind, m, d, 72 + m)
            Y[:, 0] //= 512
        else:  # all at one place
            Y = np.repeat(X[:1], m, axis=0)
        yid = np.arange(nxt, nxt + m, dtype=np.uint32)
        nxt += m
        t.insert(to_dev(Y), ids_dev(yid))
        o.insert(Y, yid)
        _same(t, o)
        # random ones, then every point of one corner: subtrees shrink out of balance
        live = np.sort(o.points()[0])
        gone = rng.choice(live, min(m, len(live) // 3), replace=False).astype(np.uint32)
        assert t.delete(ids_dev(gone)) == o.delete(gone)
        _same(t, o)
        pid, pts = o.points()
        gone = pid[np.argsort(pts[:, 0], kind="stable")[:m]].astype(np.uint32)
        assert t.delete(ids_dev(gone)) == o.delete(gone)
        _same(t, o)
    t.close()


@pytest.mark.parametrize("m", [300, 3000, 20000])
def test_large_leaves(m):
    # half of the points identical: a heavy leaf of thousands of points
    pkd, t, o, X = _pair("dups_big", 6000, 3, 91, phi=40)
    Y = np.concatenate([np.repeat(X[:1], m - 100, axis=0), I.uniform(100, 3, 92)])
    yid = np.arange(6000, 6000 + m, dtype=np.uint32)
    t.insert(to_dev(Y), ids_dev(yid))
    o.insert(Y, yid)
    _same(t, o)
    gone = np.concatenate([yid[::2], np.arange(0, 6000, 5)]).astype(np.uint32)
    assert t.delete(ids_dev(gone)) == o.delete(gone)
    _same(t, o)
    t.close()


def test_rejected_and_empty_batches():
    pkd, t, o, X = _pair("uniform", 5000, 3, 95, phi=8, lam=4, sigma_log2=2, sigma_os=4)
    Y = I.uniform(5000, 3, 96)
    for m in (10, 5000):
        yid = np.arange(10000, 10000 + m, dtype=np.uint32)
        for bad in (7, 0xFFFFFFFF, yid[0]):  # stored, reserved, repeated
            z = yid.copy()
            z[m // 2] = bad
            with pytest.raises(pkd.PkdError) as e:
                t.insert(to_dev(Y[:m]), ids_dev(z))
            assert e.value.code == pkd.PKD_EINVAL
            _same(t, o)
        far = Y[:m].copy()
        far[m - 1, 2] = -1
        with pytest.raises(pkd.PkdError):
            t.insert(to_dev(far), ids_dev(yid))
        _same(t, o)
        assert t.delete(ids_dev(np.arange(20000, 20000 + m, dtype=np.uint32))) == 0
        _same(t, o)
        t.insert(to_dev(Y[:m]), ids_dev(yid))
        o.insert(Y[:m], yid)
        assert t.delete(ids_dev(np.concatenate([yid, yid[:3]]))) == o.delete(np.concatenate([yid, yid[:3]])) == m
        _same(t, o)
    t.close()


@pytest.mark.parametrize("n", [700, 6000])
def test_small_flatten_overflow_is_redone(n):
    # a subtree of up to 8192 points is flattened by one block.  At alpha = 0 the
    # insert rebuilds the root: 6000 points in leaves of at most 2 overflow the
    # smallest lists (1024 entries above the roots'), which are then redone larger
    from paper_2411_09275_gb300 import pkd as P
    from tests.gpuutil import knobs

    pkd, t, o, X = _pair("uniform", n, 3, 97, phi=2, lam=3, sigma_log2=2, sigma_os=4, alpha_num=0)
    Y = I.uniform(n // 2, 3, 98)
    Y[:, 0] //= 64
    yid = np.arange(n, n + n // 2, dtype=np.uint32)
    P.pkd_kernel_timing(True)
    try:
        with knobs(front_cap=64):
            t.insert(to_dev(Y), ids_dev(yid))
            retries = P.pkd_kernel_stats("front_retries")[0]
            o.insert(Y, yid)
            _same(t, o)
            gone = yid[: n // 3]
            assert t.delete(ids_dev(gone)) == o.delete(gone)
            _same(t, o)
    finally:
        P.pkd_kernel_timing(False)
    assert retries == (1 if n == 6000 else 0)
    t.close()
