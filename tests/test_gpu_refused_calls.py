"""Calls that are refused leave nothing behind: on a stream that is being captured
nothing is launched or allocated."""
import ctypes as C

import numpy as np
import pytest

import oracle as O
from paper_2411_09275_gb300 import inputs as I
from tests import treeutil as U
from tests.gpuutil import ids_dev, oparams, to_dev

pytestmark = pytest.mark.gpu


def test_calls_on_a_capturing_stream_record_nothing():
    import torch

    from paper_2411_09275_gb300 import pkd

    cu = C.CDLL("libcuda.so.1")
    X = I.uniform(5000, 3, 3)
    p = pkd.Params(d=3)
    t, o = pkd.Tree(to_dev(X), None, p), O.OracleTree(X, None, oparams(p))
    Q, new, gone = to_dev(X[:100]), ids_dev(np.arange(5000, 5100)), np.arange(0, 5000, 7, dtype=np.uint32)
    ids = ids_dev(gone)
    oi = torch.empty((100, 5), dtype=torch.int32, device="cuda")
    od = torch.empty((100, 5), dtype=torch.int64, device="cuda")
    cnt = torch.empty(100, dtype=torch.int64, device="cuda")
    s = torch.cuda.Stream()
    calls = [lambda: pkd.pkd_batch_delete(t._h, ids, stream=s), lambda: pkd.pkd_batch_insert(t._h, Q, new, stream=s),
             lambda: pkd.pkd_knn(t._h, Q, 5, oi, od, stream=s), lambda: pkd.pkd_range_count(t._h, Q, Q, cnt, stream=s),
             lambda: pkd.pkd_range_report(t._h, Q, Q, stream=s)]
    h = C.c_void_p(s.cuda_stream)
    for k, call in enumerate(calls):
        torch.cuda.synchronize()
        before = [pkd.pkd_kernel_stats(n)[0] for n in ("launches", "allocations")]
        assert cu.cuStreamBeginCapture_v2(h, C.c_int(1)) == 0  # thread-local
        code = 0
        try:
            call()
        except pkd.PkdError as e:
            code = e.code
        graph = C.c_void_p()
        ended = cu.cuStreamEndCapture(h, C.byref(graph))
        assert code == pkd.PKD_ECUDA and ended != 0, k
        assert [pkd.pkd_kernel_stats(n)[0] for n in ("launches", "allocations")] == before, k
    assert t.delete(ids, s) == o.delete(gone) == len(gone)
    U.assert_exports_equal(t.export(), o.export())
    t.close()
