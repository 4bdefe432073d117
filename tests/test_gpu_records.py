"""GPU tests of a handle's records over runs of changing replica counts."""
import time

import numpy as np
import pytest

from paper_2407_10205_gb300 import instances as ins

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _best_us(phia, h, n):
    t = []
    for _ in range(200):
        t0 = time.perf_counter()
        phia.best(h, n)
        t.append(time.perf_counter() - t0)
    return 1e6 * float(np.median(t))


def test_few_replicas_after_many(gpu_lib):
    """A run of 16 replicas after one of 65536 on the same handle has the records of a fresh handle, goes
    on from them, and reading them costs what 16 replicas cost."""
    phia = gpu_lib
    N, R, T = 64, 16, 40
    d = ins.dense_int(N, 7, 7, 1)
    sched = phia.schedule(0.01, 0.3, 0.1, 2.0, refresh=9)
    out, us = [], []
    for many in (False, True):
        with phia.Annealer(d.k, d.kh, path=phia.PATH_TC) as A:
            if many:
                phia.anneal(A.h, sched, 65536, T, 3)
                assert len(phia.replica_results(A.h, 65536, N)[0]) == 65536
            x, v = torch.empty((R, N), device="cuda"), torch.empty((R, N), device="cuda")
            phia.init_state(A.h, R, 7, x, v)
            for t0, k in ((0, 15), (15, T - 15)):
                phia.run(A.h, sched, R, t0, k, T, 7, x, v, reset_best=(t0 == 0))
            out.append(phia.replica_results(A.h, R, N))
            us.append(_best_us(phia, A.h, N))
    for u, w in zip(*out):
        assert np.array_equal(u, w)
    assert us[1] < 1.5 * us[0] + 8.0


def test_records_that_are_gone_are_refused(gpu_lib):
    """A field call for more replicas than any run had takes new buffers: no results are left to read."""
    phia = gpu_lib
    d = ins.dense_int(64, 7, 7, 1)
    with phia.Annealer(d.k, d.kh, path=phia.PATH_TC) as A:
        phia.anneal(A.h, phia.schedule(0.01, 0.3, 0.1, 2.0), 8, 5, 3)
        phia.best(A.h, 64)
        phia.field(A.h, torch.ones((4096, 64), dtype=torch.int8, device="cuda"),
                   torch.empty((4096, 64), dtype=torch.int32, device="cuda"))
        with pytest.raises(phia.PhiaError) as e:
            phia.best(A.h, 64)
        assert e.value.code == phia.ESTATE
