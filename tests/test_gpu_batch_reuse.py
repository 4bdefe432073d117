"""GPU tests of one batch used several times: what a run leaves behind (the cut into sets, tables,
times) must not reach the next one."""
import numpy as np
import pytest

from paper_2407_10205_gb300 import instances as ins

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _records(B, count, R):
    return [B.replica_results(k, R) for k in range(count)]


@pytest.mark.parametrize("mode", [1, 2])
def test_replica_counts_may_change_between_runs(gpu_lib, mode):
    """8 bytes of state per spin and replica: 64 replicas are one set of instances, 1024 and 2048
    several, cut at other places.  Sizes and densities go up and down, so that the heaviest blocks of
    a set come from all of its members."""
    phia = gpu_lib
    g = np.random.default_rng(7)
    insts = [ins.erdos_renyi(int(n), float(d), 127, 31, 4, seed=k)
             for k, (n, d) in enumerate(zip(g.integers(200, 2500, 14), g.uniform(0.004, 0.05, 14)))]
    sched = phia.schedule(0.01, 0.2, 0.1, 2.0, refresh=5)
    counts, T = (64, 2048, 64, 1024), 12
    fresh = {}
    for R in set(counts):
        with phia.Batch(insts, csr_mode=mode) as B:
            B.anneal(sched, R, T, seed=9)
            fresh[R] = _records(B, len(insts), R)
    with phia.Batch(insts, csr_mode=mode) as B:
        for R in counts:
            B.anneal(sched, R, T, seed=9)
            for a, b in zip(_records(B, len(insts), R), fresh[R]):
                for u, w in zip(a, b):
                    assert np.array_equal(u, w)


def test_device_time_leaves_out_the_host_work_of_a_first_run(gpu_lib):
    """The first run with a replica count sorts the blocks of its sets on the host (12000 of them here,
    some ms); the time that stats report is the device's, as for the second run."""
    phia = gpu_lib
    insts = [ins.erdos_renyi(3000, 0.002, 127, 31, 4, seed=k) for k in range(64)]
    sched = phia.schedule(0.01, 0.2, 0.1, 2.0)
    first, second = [], []
    for _ in range(4):
        with phia.Batch(insts) as B:
            for out in (first, second):
                B.anneal(sched, 32, 2, seed=9)
                out.append(B.stats().device_ms)
    assert min(first[1:]) < 1.5 * min(second) + 0.1


def test_small_sparse_and_dense_members_together(gpu_lib):
    """All members on resident kernels, of every size class: the records of each alone."""
    phia = gpu_lib
    insts = [ins.dense_int(60, 7, 7, 1), ins.erdos_renyi(100, 0.1, 127, 31, 4, 2), ins.dense_int(300, 7, 7, 3),
             ins.erdos_renyi(400, 0.05, 127, 31, 4, 4), ins.erdos_renyi(200, 0.05, 127, 31, 4, 5), ins.dense_int(130, 7, 7, 6)]
    sched, R, T = phia.schedule(0.01, 0.2, 0.1, 2.0, refresh=7), 45, 60
    with phia.Batch(insts, instance_ids=range(6)) as B:
        B.anneal(sched, R, T, seed=9)
        mix = _records(B, 6, R)
    for k, c in enumerate(insts):
        with phia.Batch([c], instance_ids=[k]) as A:
            A.anneal(sched, R, T, seed=9)
            for u, w in zip(mix[k], A.replica_results(0, R)):
                assert np.array_equal(u, w)


@pytest.mark.parametrize("top", [160, 161, 208, 209, 240, 256])
def test_members_of_129_to_256_spins(gpu_lib, top):
    """The kernels that a batch's launch is built for by its largest member (10, 13 or 15 warps), and the
    tcgen05 and cluster kernels above 240 spins, for both operands: the records of each alone."""
    phia = gpu_lib
    insts = [ins.dense_int(129, 7, 7, 1), ins.dense_int(top, 7, 7, 2), ins.dense_int(top, 100, 7, 3),
             ins.erdos_renyi(top, 0.1, 127, 31, 4, 4), ins.dense_int(max(129, top - 15), 100, 7, 5)]
    R, T = 45, 40
    for deriv in (0, 1):
        sched = phia.schedule(0.01, 0.2, 0.1, 2.0, refresh=7, deriv=deriv)
        with phia.Batch(insts, instance_ids=range(5)) as B:
            B.anneal(sched, R, T, seed=9)
            mix = _records(B, 5, R)
        for k, c in enumerate(insts):
            d = c if hasattr(c, "k") else c.to_dense()
            with phia.Annealer(d.k, d.kh, d.frac_bits, path=phia.PATH_TC, instance_id=k, tc_kernel=phia.KERNEL_PER_STEP,
                               large_variant=1) as A:
                phia.anneal(A.h, sched, R, T, 9)
                for u, w in zip(mix[k], phia.replica_results(A.h, R, d.n)):
                    assert np.array_equal(u, w)
