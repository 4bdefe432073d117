"""GPU tests of handles used by several threads, each its own ones."""
import threading

import numpy as np
import pytest

from paper_2407_10205_gb300 import instances as ins

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _in_threads(work):
    errors = []

    def guarded(fn):
        try:
            fn()
        except Exception as e:                         # noqa: BLE001 -- reported by the test
            errors.append(e)

    th = [threading.Thread(target=guarded, args=(fn,)) for fn in work]
    for t in th:
        t.start()
    for t in th:
        t.join()
    assert not errors, errors


def test_launches_of_one_kernel_with_other_shared_memory(gpu_lib):
    """Sparse instances of 600 and of 3000 spins run one kernel with 67 and 111 KB of dynamic shared
    memory, GAHMC of 40 and 900 spins with few and many.  Runs of changing length launch every
    iteration by itself, so the two threads' launches alternate."""
    phia = gpu_lib
    sched = phia.schedule(0.01, 0.2, 0.1, 2.0, refresh=7)
    small, large = ins.erdos_renyi(600, 0.03, 127, 31, 4, 1), ins.erdos_renyi(3000, 0.01, 127, 31, 4, 2)

    def sparse(c, R, runs):
        def fn():
            s = torch.cuda.Stream()
            with phia.Annealer(h_k=c.kh, frac_bits=4, csr=(c.row_ptr, c.col, c.val), stream=s.cuda_stream) as A:
                out = None
                for k in range(runs):
                    phia.anneal(A.h, sched, R, 50 + k % 40, 3)
                    if k % 40 == 0:
                        got = phia.replica_results(A.h, R, c.n)
                        for u, w in zip(got, out or got):
                            assert np.array_equal(u, w)
                        out = got
        return fn

    def crossings(n, runs):
        d = ins.sk_pm1(n, n)

        def fn():
            s = torch.cuda.Stream()
            with phia.Annealer(d.k, d.kh, path=phia.PATH_TC, stream=s.cuda_stream) as A:
                for _ in range(runs):
                    phia.gahmc(A.h, phia.gahmc_schedule(0.01, 0.1), 4, 1, 5)
                phia.sync(A.h)
        return fn

    _in_threads([sparse(small, 32, 160), sparse(large, 256, 160)])
    _in_threads([crossings(40, 300), crossings(900, 60)])


def test_kernels_that_fill_the_gpu_run_beside_each_other(gpu_lib):
    """Handles of several kinds on streams of their own: overlapped kernels with wide and with narrow
    tiles, whose CTAs wait on each other, the cluster kernel, and a sparse gather.  Records as alone."""
    phia = gpu_lib
    sched = phia.schedule(0.005, 0.13, 0.1, 2.0, refresh=30)
    wide, narrow, cluster = ins.sk_pm1(2000, 1), ins.sk_pm1(1500, 2), ins.sk_pm1(600, 3)
    sparse = ins.erdos_renyi(3000, 0.01, 127, 31, 4, 2)

    def open_(c, stream):
        if hasattr(c, "k"):
            return phia.Annealer(c.k, c.kh, path=phia.PATH_TC, stream=stream)
        return phia.Annealer(h_k=c.kh, frac_bits=c.frac_bits, csr=(c.row_ptr, c.col, c.val), stream=stream)

    def check(c, R, T, runs):
        with open_(c, None) as A:
            phia.anneal(A.h, sched, R, T, 3)
            alone = phia.replica_results(A.h, R, c.n)

        def fn():
            s = torch.cuda.Stream()
            with open_(c, s.cuda_stream) as A:
                for _ in range(runs):
                    phia.anneal(A.h, sched, R, T, 3)
                for u, w in zip(phia.replica_results(A.h, R, c.n), alone):
                    assert np.array_equal(u, w)
        return fn

    _in_threads([check(wide, 2048, 60, 8), check(narrow, 256, 100, 10), check(cluster, 128, 200, 20),
                 check(sparse, 256, 120, 10), check(wide, 300, 100, 8)])
