"""GPU tests of what a handle's kernel choice is after the calls that change it: a tuned replica
count, an acceptance run."""
import numpy as np
import pytest

from paper_2407_10205_gb300 import instances as ins

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _kernel_of(phia, h, sched, R, T=20):
    phia.anneal(h, sched, R, T, 5)
    st = phia.stats_get(h)
    return st.tc_kernel, st.kernel_launches


@pytest.mark.parametrize("N", [150, 230, 1100, 1536, 2000])
def test_a_tuned_replica_count_leaves_others_alone(gpu_lib, N):
    """Tuned for 8192 replicas, a handle runs 64 as a fresh one does (its kernel shows in the code and the
    number of launches: 2 for the kernels that run from one launch, one more for each conversion)."""
    phia = gpu_lib
    d = ins.dense_int(N, 7, 7, N)
    sched = phia.schedule(0.01, 0.1, 0.1, 2.0, refresh=50)
    with phia.Annealer(d.k, d.kh, path=phia.PATH_TC, instance_id=3) as B:
        fresh = _kernel_of(phia, B.h, sched, 64)
    with phia.Annealer(d.k, d.kh, path=phia.PATH_TC, instance_id=3) as A:
        phia.autotune(A.h, sched, 8192, probe_iters=10)
        tuned = _kernel_of(phia, A.h, sched, 8192)
        assert _kernel_of(phia, A.h, sched, 64) == fresh
        assert _kernel_of(phia, A.h, sched, 8192) == tuned


@pytest.mark.parametrize("N", [16, 40, 64, 90, 128])
def test_autotune_after_an_acceptance_run_times_its_candidates(gpu_lib, N):
    """The tuner's time is that of the kernel it chose.  Sizes where the warp-level kernel takes half the
    time of the first candidate, which the tuner credited with it."""
    phia = gpu_lib
    R, T = 256, 2000
    d = ins.dense_int(N, 7, 7, N)
    plain = phia.schedule(0.01, 0.1, 0.1, 2.0, refresh=50)
    with phia.Annealer(d.k, d.kh, path=phia.PATH_TC) as A:
        phia.anneal(A.h, phia.schedule(0.01, 0.1, 0.1, 2.0, refresh=50, accept_test=1), R, 50, 5)
        res = phia.autotune(A.h, plain, R, probe_iters=T)
        best = min(_device_us(phia, A.h, plain, R, T) for _ in range(3))
        assert phia.stats_get(A.h).tc_kernel == res.tc_kernel
        assert best < 1.3 * res.best_us_per_iter


def _device_us(phia, h, sched, R, T):
    phia.anneal(h, sched, R, T, 5)
    return 1000.0 * phia.stats_get(h).device_ms / T


def test_a_run_goes_on_after_an_acceptance_run(gpu_lib):
    """384 spins x 16384 replicas are tuned to a per-iteration kernel; a run with the acceptance test
    takes the resident one.  The ordinary run that goes on from it keeps its records."""
    phia = gpu_lib
    N, R = 384, 16384
    d = ins.dense_int(N, 7, 7, 2)
    kw = dict(refresh=5)
    test, plain = (phia.schedule(0.01, 0.1, 0.1, 2.0, accept_test=k, **kw) for k in (1, 0))
    out = []
    for fixed in (True, False):
        o = dict(tc_kernel=phia.KERNEL_RESIDENT, coupling_mem=phia.MEM_SHARED) if fixed else {}
        with phia.Annealer(d.k, d.kh, path=phia.PATH_TC, **o) as A:
            if not fixed:
                assert phia.autotune(A.h, plain, R, probe_iters=10).tc_kernel == 2
            x, v = torch.empty((R, N), device="cuda"), torch.empty((R, N), device="cuda")
            phia.init_state(A.h, R, 7, x, v)
            phia.run(A.h, test, R, 0, 20, 30, 7, x, v)
            # backwards, so that the second piece improves few replicas and the first's records count
            phia.run(A.h, phia.schedule(0.0, 0.0, 0.1, 2.0, **kw), R, 20, 10, 30, 7, x, v, reset_best=False)
            out.append(phia.replica_results(A.h, R, N))
    assert (out[0][1] < 20).any()
    for u, w in zip(*out):
        assert np.array_equal(u, w)


def test_the_warp_kernels_tile_is_reported_as_it_is(gpu_lib):
    """It runs 8 replicas per CTA, whatever is asked for."""
    phia = gpu_lib
    sched, seen = phia.schedule(0.01, 0.1, 0.1, 2.0, refresh=50), 0
    for N in (8, 16, 24, 32, 48, 64):
        d = ins.dense_int(N, 7, 7, N)
        with phia.Annealer(d.k, d.kh, path=phia.PATH_TC, instance_id=9) as A:
            res = phia.autotune(A.h, sched, 72, probe_iters=100)
        if res.tc_kernel == 3:
            seen += 1
            assert res.tile_replicas == 8
    assert seen


@pytest.mark.parametrize("N,R,variant,form", [(2000, 4096, 0, 2), (2000, 4096, 1, 1), (2000, 4096, 11, 2), (1500, 256, 7, 3),
                                              (600, 64, 7, 4), (600, 64, 0, 4), (600, 64, 12, 2)])
def test_stats_name_the_form_that_ran(gpu_lib, N, R, variant, form):
    phia = gpu_lib
    d = ins.sk_pm1(N, 1)
    with phia.Annealer(d.k, d.kh, path=phia.PATH_TC, tc_kernel=phia.KERNEL_PER_STEP, large_variant=variant) as A:
        phia.anneal(A.h, phia.schedule(0.01, 0.1, 0.1, 2.0), R, 4, 1)
        st = phia.stats_get(A.h)
        assert (st.tc_kernel, st.large_form) == (2, form)
    d = ins.sk_pm1(300, 1)
    with phia.Annealer(d.k, d.kh, path=phia.PATH_TC) as A:
        phia.anneal(A.h, phia.schedule(0.01, 0.1, 0.1, 2.0), 64, 4, 1)
        st = phia.stats_get(A.h)
        assert (st.tc_kernel, st.large_form) in ((2, 4), (1, 0))


def test_an_autotune_that_fails_leaves_the_handle_as_it_was(gpu_lib):
    phia = gpu_lib
    d = ins.dense_int(100, 7, 7, 1)
    good, bad = phia.schedule(0.01, 0.1, 0.1, 2.0), phia.schedule(0.01, 0.1, 0.0, 2.0)
    with phia.Annealer(d.k, d.kh, path=phia.PATH_TC, tc_kernel=phia.KERNEL_PER_STEP, large_variant=1) as A:
        with pytest.raises(phia.PhiaError) as e:
            phia.autotune(A.h, bad, 32, probe_iters=10)
        assert e.value.code == phia.EINVAL
        assert _kernel_of(phia, A.h, good, 32)[0] == 2
