"""Small batches into a tree far taller than usual: their routing rounds stop
when no item is left, instead of being queued for the tallest path, and trees
equal the oracle's wherever the batch goes: near the root, down the whole
path, and all over."""
import numpy as np
import pytest

import oracle as O
from tests import treeutil as U
from tests.gpuutil import ids_dev, oparams, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lam", [1, 2])
def test_small_batches_into_a_tall_tree(lam):
    # alpha = 1/2 never rebuilds an inner node: batches past the last point
    # grow one path by about two levels each
    from paper_2411_09275_gb300 import pkd

    p = pkd.Params(d=1, phi=2, lam=lam, sigma_log2=0, sigma_os=1, alpha_num=1, alpha_den=2)
    X = (np.arange(8, dtype=np.int32) * 7).reshape(8, 1)
    t, o = pkd.Tree(to_dev(X), None, p), O.OracleTree(X, None, oparams(p))
    nxt, top = 8, 100

    def insert(Y):
        nonlocal nxt
        yid = np.arange(nxt, nxt + len(Y), dtype=np.uint32)
        nxt += len(Y)
        Y = np.asarray(Y, np.int32).reshape(-1, 1)
        t.insert(to_dev(Y), ids_dev(yid))
        o.insert(Y, yid)
        return yid

    while t.height <= 260:
        insert([top + 3, top + 1, top + 2])
        top += 10
    U.assert_exports_equal(t.export(), o.export())

    def launches(call):
        a = pkd.pkd_kernel_stats("launches")[0]
        out = call()
        return out, pkd.pkd_kernel_stats("launches")[0] - a

    # the first leaf is a few levels down: a few rounds, not one for every
    # lambda levels of the tallest path (130 and more)
    ids, n = launches(lambda: insert([1]))
    assert n < 100, n
    U.assert_exports_equal(t.export(), o.export())
    (got, want), n = launches(lambda: (t.delete(ids_dev(ids)), o.delete(ids)))
    assert got == want == 1 and n < 100, n
    U.assert_exports_equal(t.export(), o.export())
    rng = np.random.default_rng(lam)
    for m in (1, 300, 4096):
        a = insert(np.full(m, top + 5))  # all past the last point
        b = insert(rng.integers(0, top, m))
        U.assert_exports_equal(t.export(), o.export())
        gone = np.concatenate([a[::2], b[::3], ids])
        assert t.delete(ids_dev(gone)) == o.delete(gone)
        U.assert_exports_equal(t.export(), o.export())
    assert t.size == o.size
    t.close()
