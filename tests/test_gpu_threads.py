"""Host threads that work on trees of their own, each on its own stream: what
one thread's call does on the library's shared state (the streams and the lock
of recorded builds, the kernels' shared-memory limits) never reaches another
thread's tree.  Trees equal the oracle's after every call."""
import threading
import time

import numpy as np
import pytest

import oracle as O
from paper_2411_09275_gb300 import inputs as I
from tests import treeutil as U
from tests.gpuutil import ids_dev, knobs, oparams, to_dev

pytestmark = pytest.mark.gpu


def _together(*bodies):
    """Run every body(stream) in a thread of its own; re-raise what one raised."""
    import torch

    torch.cuda.synchronize()
    failed = []
    start = threading.Barrier(len(bodies))

    def run(body):
        s = torch.cuda.Stream()
        try:
            with torch.cuda.stream(s):
                start.wait(60)
                body(s)
                s.synchronize()
        except BaseException as e:  # noqa: BLE001
            failed.append(e)

    threads = [threading.Thread(target=run, args=(b,)) for b in bodies]
    for th in threads:
        th.start()
    for th in threads:
        th.join(300)
    assert not any(th.is_alive() for th in threads)
    if failed:
        raise failed[0]


def test_builds_that_record_beside_updates_of_another_tree():
    # one thread builds trees of ever new sizes, so that each records its
    # graph; the other's tree is rebuilt from the root by every update
    # (alpha = 0), as one segment that runs on the direct build's second stream
    import torch

    from paper_2411_09275_gb300 import pkd

    p = pkd.Params(d=3)
    points = [I.uniform(9000 + 37 * i, 3, 9000 + i) for i in range(100)]
    p0 = pkd.Params(d=3, alpha_num=0)
    X = I.uniform(5000, 3, 3)
    Q = np.concatenate([X[::100], I.uniform(200, 3, 4)])
    o = O.OracleTree(X, None, oparams(p0))
    batches, want = [], []
    for i in range(100):
        Y = I.uniform(50 + i, 3, 7000 + i)
        yid = np.arange(5000 + 200 * i, 5000 + 200 * i + len(Y), dtype=np.uint32)
        gone = np.concatenate([yid[::2], np.arange(40 * i, 40 * i + 20, dtype=np.uint32)])
        batches.append((Y, yid, gone))
        o.insert(Y, yid)
        want.append(o.knn(Q, 5))
        assert o.delete(gone) == len(gone)
        want.append(o.knn(Q, 5))
    builds, answers = [], []
    dev_points = [to_dev(x) for x in points]
    dev_batches = [(to_dev(Y), ids_dev(yid), ids_dev(gone)) for Y, yid, gone in batches]
    gX, gQ = to_dev(X), to_dev(Q)
    updated = []

    def build(s):
        for x in dev_points:
            builds.append(pkd.Tree(x, None, p, s))

    def update(s):
        t = pkd.Tree(gX, None, p0, s)
        updated.append(t)
        for Y, yid, gone in dev_batches:
            t.insert(Y, yid, s)
            answers.append(t.knn(gQ, 5, s))
            assert t.delete(gone, s) == gone.numel()
            answers.append(t.knn(gQ, 5, s))

    _together(build, update)
    torch.cuda.synchronize()
    for x, t in zip(points, builds):
        U.assert_exports_equal(t.export(), O.OracleTree(x, None, oparams(p)).export())
        t.close()
    for (gi, gd), (wi, wd) in zip(answers, want):
        assert np.array_equal(gd.cpu().numpy(), wd) and np.array_equal(gi.cpu().numpy().view(np.uint32), wi)
    U.assert_exports_equal(updated[0].export(), o.export())
    updated[0].close()
    assert len(builds) == len(points) and len(answers) == len(want)


def test_builds_that_record_beside_exports_of_another_tree():
    # an export waits for the whole device, which CUDA forbids while a stream
    # is being recorded
    from paper_2411_09275_gb300 import pkd

    p = pkd.Params(d=2)
    points = [I.uniform(30000 + 41 * i, 2, 600 + i) for i in range(80)]
    X = I.uniform(20000, 2, 5)
    t = pkd.Tree(to_dev(X), None, p)
    dev_points = [to_dev(x) for x in points]
    builds, exports, heights = [], [], []

    def build(s):
        for x in dev_points:
            builds.append(pkd.Tree(x, None, p, s))

    def export(s):
        while len(builds) < len(points) and len(exports) < 5000:
            exports.append(t.export())
            heights.append(t.height)
            del exports[1:-1]

    _together(build, export)
    want = O.OracleTree(X, None, oparams(p)).export()
    assert len(builds) == len(points)
    for e in exports:
        U.assert_exports_equal(e, want)
    for x, b in zip(points, builds):
        U.assert_exports_equal(b.export(), O.OracleTree(x, None, oparams(p)).export())
        b.close()
    t.close()


def test_a_rebuild_that_waits_holds_up_no_other_build():
    # the insert rebuilds its tree from the root (alpha = 0), more points than
    # one CTA takes, and sleeps two seconds in front of the first round
    from paper_2411_09275_gb300 import pkd

    X, Y, Z = I.uniform(20000, 3, 11), I.uniform(100, 3, 12), I.uniform(40000, 3, 13)
    p, p0 = pkd.Params(d=3), pkd.Params(d=3, alpha_num=0)
    pkd.Tree(to_dev(Z), None, p).close()
    t, o = pkd.Tree(to_dev(X), None, p0), O.OracleTree(X, None, oparams(p0))
    gY, gZ, yid = to_dev(Y), to_dev(Z), np.arange(20000, 20100, dtype=np.uint32)
    gyid = ids_dev(yid)
    o.insert(Y, yid)
    at, built = {}, []

    def update(s):
        at["start"] = time.monotonic()
        t.insert(gY, gyid, s)
        at["update"] = time.monotonic()

    def build(s):
        time.sleep(0.5)
        built.append(pkd.Tree(gZ, None, p, s))
        at["build"] = time.monotonic()

    with knobs(pause_rounds=12000):
        _together(update, build)
    assert at["update"] - at["start"] >= 1.9  # the rebuild did sleep there
    assert at["build"] < at["update"] - 0.5
    U.assert_exports_equal(t.export(), o.export())
    U.assert_exports_equal(built[0].export(), O.OracleTree(Z, None, oparams(p)).export())
    t.close()
    built[0].close()


def test_searches_and_updates_with_different_shared_memory():
    # stacks of trees of heights about 75 and 115, and skeletons of 9 and 10
    # levels, take more than 48 KB of shared memory, each another amount
    from paper_2411_09275_gb300 import pkd

    def chain(batches):  # alpha = 1/2, always past the last point: one path grows
        p = pkd.Params(d=3, phi=2, lam=2, sigma_log2=0, sigma_os=1, alpha_num=1, alpha_den=2)
        X = np.zeros((8, 3), np.int32)
        X[:, 0] = np.arange(8) * 7
        t, o = pkd.Tree(to_dev(X), None, p), O.OracleTree(X, None, oparams(p))
        for r in range(batches):
            Y = np.zeros((3, 3), np.int32)
            Y[:, 0] = 100 + 10 * r + np.array([3, 1, 2])
            yid = np.arange(8 + 3 * r, 11 + 3 * r, dtype=np.uint32)
            t.insert(to_dev(Y), ids_dev(yid))
            o.insert(Y, yid)
        return t, o

    Q = I.uniform(9000, 3, 21)
    Q[:, 0] %= 700
    Q[:, 1:] %= 50
    gQ = to_dev(Q)
    pairs = [chain(36), chain(56)]
    assert 66 <= pairs[0][0].height < 85 and 100 < pairs[1][0].height < 126
    X = I.uniform(3000, 3, 22)
    Y, yid = I.uniform(20, 3, 23), np.arange(3000, 3020, dtype=np.uint32)
    gY, gyid = to_dev(Y), ids_dev(yid)
    wide = []
    for lam in (9, 10):
        p = pkd.Params(d=3, lam=lam, phi=8)
        wide.append((pkd.Tree(to_dev(X), None, p), O.OracleTree(X, None, oparams(p))))
    answers = []

    def search(k, wait):
        def body(s):
            time.sleep(wait)
            answers.append((k, pairs[k][0].knn(gQ, 4, s)))
        return body

    def update(k, wait):
        def body(s):
            time.sleep(wait)
            wide[k][0].insert(gY, gyid, s)
        return body

    # the larger one sleeps between the limit and its launch, the other runs meanwhile
    for small, large in ((search(0, 0.3), search(1, 0)), (update(0, 0.3), update(1, 0))):
        with knobs(pause_smem=10700):
            _together(small, large)
    for k, (gi, gd) in answers:
        wi, wd = pairs[k][1].knn(Q, 4)
        assert np.array_equal(gd.cpu().numpy(), wd) and np.array_equal(gi.cpu().numpy().view(np.uint32), wi)
    for t, o in wide:
        o.insert(Y, yid)
        U.assert_exports_equal(t.export(), o.export())
    for t, o in pairs + wide:
        t.close()


def _asker(pkd, t, q, outs, k=5):
    """A body that asks for k neighbours of q on t, its outputs marked first."""
    import torch

    def body(s):
        n = q.shape[0]
        oi = torch.full((n, k), -7, dtype=torch.int32, device="cuda")
        od = torch.full((n, k), -7, dtype=torch.int64, device="cuda")
        code = pkd.PKD_OK
        try:
            pkd.pkd_knn(t._h, q, k, oi, od, stream=s)
        except pkd.PkdError as e:
            code = e.code
        s.synchronize()
        outs.append((code, oi, od))

    return body


def test_a_refusal_stands_until_its_search_has_run():
    # a refused call sleeps between its check and its search while 40 others
    # are refused on the same tree
    from paper_2411_09275_gb300 import pkd

    t = pkd.Tree(to_dev(I.uniform(5000, 3, 31)), None, pkd.Params(d=3))
    bad = to_dev(np.full((64, 3), 1 << 30, np.int32))
    slow, others = [], []

    def refused(s):
        time.sleep(0.3)
        for _ in range(40):
            _asker(pkd, t, bad, others)(s)

    with knobs(pause_query=11500):
        _together(_asker(pkd, t, bad, slow), refused)
    assert len(slow) == 1 and len(others) == 40
    for code, oi, od in slow + others:
        assert code == pkd.PKD_EINVAL
        assert (oi == -7).all().item() and (od == -7).all().item()
    t.close()


@pytest.mark.parametrize("threads", [2, 16, 17, 40])
def test_queries_in_flight_at_once(threads):
    # every call sleeps between its check and its search, so that all are in
    # flight together: more than there are slots for refusals, too
    from paper_2411_09275_gb300 import pkd

    X, Q = I.uniform(5000, 3, 41), I.uniform(64, 3, 42)
    p = pkd.Params(d=3)
    t, o = pkd.Tree(to_dev(X), None, p), O.OracleTree(X, None, oparams(p))
    good = to_dev(Q)
    bad = to_dev(np.full((64, 3), 1 << 30, np.int32))
    wi, wd = o.knn(Q, 5)
    served, refused = [], []
    for _ in range(2):  # the slots are free again
        with knobs(pause_query=threads * 10000 + 300):
            _together(*[_asker(pkd, t, bad if i % 3 == 0 else good, refused if i % 3 == 0 else served)
                        for i in range(threads)])
    assert len(served) + len(refused) == 2 * threads
    for code, oi, od in refused:
        assert code == pkd.PKD_EINVAL
        assert (oi == -7).all().item() and (od == -7).all().item()
    for code, oi, od in served:
        assert code == pkd.PKD_OK
        assert np.array_equal(od.cpu().numpy(), wd) and np.array_equal(oi.cpu().numpy().view(np.uint32), wi)
    t.close()
