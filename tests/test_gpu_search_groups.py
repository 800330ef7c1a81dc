"""The cooperative searches: k-NN with 4, 8 or 32 lanes per query (chosen by
d, k and the number of queries) and 1 to 4 neighbours per lane; range count
and report with a warp per box.  Exact against the oracle at the edges of
those choices: k on both sides of every list size, batches on both sides of
the warp-per-query limit, leaves above 32 points, heavy leaves, fewer points
than k, boxes without points and boxes over the whole domain."""
import numpy as np
import pytest

import oracle as O
from paper_2411_09275_gb300 import inputs as I
from tests.gpuutil import ids_dev, make_points, oparams, to_dev

pytestmark = pytest.mark.gpu

TOP = (1 << 30) - 1


def _tree(kind, n, d, phi, seed):
    from paper_2411_09275_gb300 import pkd

    X = make_points(kind, n, d, seed)
    ids = (np.arange(n, dtype=np.uint64) * 2654435761 % (1 << 32)).astype(np.uint32)
    p = pkd.Params(d=d, phi=phi, lam=4, sigma_log2=2, sigma_os=4)
    return pkd, pkd.Tree(to_dev(X), ids_dev(ids), p), O.OracleTree(X, ids, oparams(p)), X


@pytest.mark.parametrize("kind,n,d,phi", [("uniform", 3000, 1, 32), ("dups", 2500, 3, 8), ("uniform", 3001, 4, 100),
                                          ("varden", 2999, 5, 32), ("dups_big", 1500, 8, 1), ("uniform", 7, 2, 32)])
@pytest.mark.parametrize("q", [8192, 8193])
def test_knn_list_sizes_and_batch_limit(kind, n, d, phi, q):
    pkd, t, o, X = _tree(kind, n, d, phi, 31 + d)
    Q = np.concatenate([I.uniform(300, d, 32), X, X])[:400]
    many = np.concatenate([Q, I.uniform(q - len(Q), d, 33)])
    for k in (1, 4, 5, 8, 9, 12, 13, 16, 17, 32, 33, 64, 65, 128):
        wi, wd = o.knn(Q, k)
        for boxes in (False, True):
            pkd.pkd_set_bounding_boxes(t._h, boxes)
            gi, gd = t.knn(to_dev(many if k <= 17 else Q), k)
            assert np.array_equal(gd[:len(Q)].cpu().numpy(), wd), (k, boxes)
            assert np.array_equal(gi[:len(Q)].cpu().numpy().view(np.uint32), wi), (k, boxes)
    t.close()


@pytest.mark.parametrize("kind,n,d,phi", [("uniform", 20000, 1, 32), ("varden", 30000, 2, 16), ("dups", 9000, 3, 8),
                                          ("uniform", 20001, 5, 100), ("dups_big", 3000, 8, 1), ("uniform", 5, 2, 32)])
def test_range_faces_and_leaf_order(kind, n, d, phi):
    pkd, t, o, X = _tree(kind, n, d, phi, 51 + d)
    lo, hi = I.boxes(300, d, 1 << 29, 52)
    lo2, hi2 = I.boxes(300, d, 1 << 20, 53)
    at = X[np.arange(200) % n]
    whole = np.zeros((4, d), np.int32), np.full((4, d), TOP, np.int32)
    whole[0][1, 0], whole[1][2, d - 1] = 1, TOP - 1  # one face short of the domain
    whole[0][3, 0], whole[1][3, 0] = 9, 8            # holds nothing
    lo = np.concatenate([whole[0], lo, lo2, at, np.minimum(at, 4)]).astype(np.int32)
    hi = np.concatenate([whole[1], hi, hi2, at, np.maximum(at, TOP - 4)]).astype(np.int32)
    for step in range(2):
        want = o.range_report(lo, hi)
        ex = t.export()
        for boxes in (False, True):
            pkd.pkd_set_bounding_boxes(t._h, boxes)
            cnt = t.range_count(to_dev(lo), to_dev(hi)).cpu().numpy()
            assert np.array_equal(cnt.astype(np.uint64), o.range_count(lo, hi))
            off, got = pkd.pkd_range_report(t._h, to_dev(lo), to_dev(hi))
            off, got = off.cpu().numpy(), got.cpu().numpy().view(np.uint32)
            assert np.array_equal(np.diff(off), cnt)
            for i in range(len(lo)):
                assert np.array_equal(np.sort(got[off[i]:off[i + 1]]), want[i])
            # the whole domain comes out leaf by leaf, depth first
            lf = ex["leaf_offsets"].astype(np.int64)
            for a, b in zip(lf[:-1], lf[1:]):
                assert np.array_equal(np.sort(got[a:b]), ex["leaf_ids"][a:b])
        # again on a tree whose subtrees are no longer contiguous
        Y = make_points(kind, 500, d, 54)
        yid = (np.arange(500, dtype=np.uint64) * 2654435761 + 977).astype(np.uint32)
        yid = np.setdiff1d(yid, np.concatenate([ex["leaf_ids"], [0xFFFFFFFF]]))[:400]
        t.insert(to_dev(Y[:len(yid)]), ids_dev(yid))
        o.insert(Y[:len(yid)], yid)
        gone = ex["leaf_ids"][::3].copy()
        assert t.delete(ids_dev(gone)) == o.delete(gone)
    t.close()


def test_refused_queries_write_nothing_and_offsets_bound_the_ids():
    # the search is queued behind its coordinate check: a refused call leaves
    # its outputs alone, the next call is served
    import ctypes as C

    import torch

    pkd, t, o, X = _tree("uniform", 5000, 3, 32, 61)
    Q = I.uniform(700, 3, 62)
    bad = Q.copy()
    bad[699, 2] = 1 << 30
    oi = torch.full((700, 5), -7, dtype=torch.int32, device="cuda")
    od = torch.full((700, 5), -7, dtype=torch.int64, device="cuda")
    cnt = torch.full((700,), -7, dtype=torch.int64, device="cuda")
    hi = np.maximum(Q, TOP - 5)
    for k in range(3):
        with pytest.raises(pkd.PkdError) as e:
            if k == 0:
                pkd.pkd_knn(t._h, to_dev(bad), 5, oi, od)
            elif k == 1:
                pkd.pkd_range_count(t._h, to_dev(bad), to_dev(hi), cnt)
            else:
                pkd.pkd_range_count(t._h, to_dev(Q), to_dev(-hi), cnt)
        assert e.value.code == pkd.PKD_EINVAL
    torch.cuda.synchronize()
    assert (oi == -7).all().item() and (od == -7).all().item() and (cnt == -7).all().item()
    gi, gd = t.knn(to_dev(Q), 5)
    wi, wd = o.knn(Q, 5)
    assert np.array_equal(gd.cpu().numpy(), wd) and np.array_equal(gi.cpu().numpy().view(np.uint32), wi)
    # more boxes than one block scans, and ids under offsets cut short
    q = 40000
    lo, hi = I.boxes(q, 3, 1 << 27, 63)
    off, ids = pkd.pkd_range_report(t._h, to_dev(lo), to_dev(hi))
    assert np.array_equal(off.cpu().numpy(), np.concatenate([[0], np.cumsum(o.range_count(lo, hi).astype(np.int64))]))
    n = ids.numel()
    out = torch.full((n + 64,), -7, dtype=torch.int32, device="cuda")
    gl, gh = to_dev(lo), to_dev(hi)
    for cap in (n, n // 2, 0):
        out.fill_(-7)
        r = pkd.lib().pkd_range_report_ids(t._h, pkd._dptr(gl), pkd._dptr(gh), C.c_uint64(q), pkd._dptr(off),
                                           pkd._dptr(out), C.c_uint64(cap), pkd._stream(None))
        torch.cuda.synchronize()
        assert r == pkd.PKD_OK and (out[cap:] == -7).all().item()
        if cap == n:
            assert (out[:n] == ids).all().item()
    assert np.array_equal(t.range_count(gl[:50], gh[:50]).cpu().numpy().astype(np.uint64), o.range_count(lo[:50], hi[:50]))
    t.close()


def test_refused_queries_that_overlap_write_nothing():
    # two threads on streams of their own: one call's refusal must not hide the other's
    import threading

    import torch

    pkd, t, o, X = _tree("uniform", 5000, 3, 32, 71)
    bad = to_dev(np.full((64, 3), 1 << 30, np.int32))
    outs, errors = [], []

    def calls():
        s = torch.cuda.Stream()
        with torch.cuda.stream(s):
            oi = torch.full((64, 5), -7, dtype=torch.int32, device="cuda")
            od = torch.full((64, 5), -7, dtype=torch.int64, device="cuda")
            for _ in range(200):
                try:
                    pkd.pkd_knn(t._h, bad, 5, oi, od, stream=s)
                    errors.append("a refused call was served")
                except pkd.PkdError as e:
                    if e.code != pkd.PKD_EINVAL:
                        errors.append(e.code)
            s.synchronize()
            outs.append((oi, od))

    torch.cuda.synchronize()
    threads = [threading.Thread(target=calls) for _ in range(2)]
    for th in threads:
        th.start()
    for th in threads:
        th.join()
    torch.cuda.synchronize()
    assert not errors and len(outs) == 2
    assert all((oi == -7).all().item() and (od == -7).all().item() for oi, od in outs)
    t.close()
