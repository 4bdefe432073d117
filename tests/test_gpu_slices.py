"""GPU tests of the sparse path's layout: slices of 32 rows, words of 32 replicas, sets of
instances that run one after the other."""
import numpy as np
import pytest

import oracle as o
from paper_2407_10205_gb300 import instances as ins

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _mask(n, keep):
    m = np.triu(np.random.default_rng(n).random((n, n)) < keep, 1)
    return m | m.T


def _to_csr(d):
    rows, cols = np.nonzero(d.k)
    rp = np.zeros(d.n + 1, dtype=np.int32)
    np.add.at(rp, rows + 1, 1)
    return ins.Csr(np.cumsum(rp).astype(np.int32), cols.astype(np.int32), d.k[rows, cols], d.kh, d.frac_bits)


# Edges of the slices (32 rows) and of the replica groups (32), rows without couplings, sums that
# leave 32 bits (the wide form), several groups per block with a ragged last one.
@pytest.mark.parametrize("N,R,kmax,hmax,keep", [
    (1, 1, 7, 7, 1.0), (31, 31, 7, 7, 0.5), (32, 32, 127, 9, 1.0), (33, 33, 7, 0, 0.1), (97, 300, 127, 1 << 23, 0.6),
    (200, 65, 127, (1 << 24) - 1, 1.0), (700, 257, 16, 7, 0.02)])
@pytest.mark.parametrize("csr_mode", [1, 2])
def test_slices_equal_the_dense_kernel(gpu_lib, N, R, kmax, hmax, keep, csr_mode):
    """The field and the update are those of the dense kernels, so the records are, bit for bit."""
    phia = gpu_lib
    T = 60
    d = ins.dense_int(N, kmax, hmax, seed=N + R)
    d = ins.Dense((d.k * _mask(N, keep)).astype(np.int8), d.kh)
    sched = phia.schedule(0.01, 0.2, 0.1, 2.0, refresh=17)
    # beside a member too large for the resident kernels, so that the gather runs
    with phia.Batch([_to_csr(d), ins.erdos_renyi(600, 0.02, 127, 31, 4, seed=1)], csr_mode=csr_mode) as B:
        B.anneal(sched, R, T, seed=3)
        a = B.replica_results(0, R)
    with phia.Annealer(d.k, d.kh, path=phia.PATH_TC, tc_kernel=phia.KERNEL_PER_STEP, large_variant=1) as A:
        phia.anneal(A.h, sched, R, T, 3)
        b = phia.replica_results(A.h, R, N)
    for u, w in zip(a, b):
        assert np.array_equal(u, w)


@pytest.mark.parametrize("N", [12300, 12600, 16384, 16390, 30000, 42000])
def test_both_offset_widths(gpu_lib, N):
    """16-bit neighbour offsets up to 16384 positions, 32-bit ones above, with x and v staged in
    shared memory or not, the spins in shared memory or not: fields and energies."""
    phia = gpu_lib
    c = ins.erdos_renyi(N, 6.0 / N, 127, 31, 4, seed=N)
    P = o.Instance(c.kh, row_ptr=c.row_ptr, col=c.col, val=c.val, frac_bits=4)
    S = ins.random_spins(5, N, seed=2)
    with phia.Annealer(h_k=c.kh, frac_bits=4, csr=(c.row_ptr, c.col, c.val), path=phia.PATH_CSR) as A:
        f = torch.empty((5, N), dtype=torch.int32, device="cuda")
        e = torch.empty(5, dtype=torch.int64, device="cuda")
        phia.field(A.h, torch.from_numpy(S).cuda(), f, e)
        torch.cuda.synchronize()
        I, E = o.field_batch(P, S)
        assert np.array_equal(f.cpu().numpy(), I) and np.array_equal(e.cpu().numpy(), E)
        phia.anneal(A.h, phia.schedule(0.01, 0.2, 0.1, 2.0), 40, 30, 3)
        be, _, _, bits = phia.replica_results(A.h, 40, N)
    B = phia.unpack_bits(bits, N)
    for r in range(0, 40, 13):
        assert o.energy_exact(P, B[r]) == be[r]


def test_several_sets_equal_each_instance_alone(gpu_lib):
    """Instances whose states together exceed L2 run in sets: same records as alone."""
    phia = gpu_lib
    R, T = 2048, 12                  # 8 bytes of state per spin and replica: 33 MB an instance
    insts = [ins.erdos_renyi(n, 0.01, 127, 31, 4, seed=n) for n in (2000, 1990, 2010, 500, 1800)]
    sched = phia.schedule(0.01, 0.2, 0.1, 2.0, refresh=5)
    for mode in (1, 2):
        with phia.Batch(insts, instance_ids=range(5), csr_mode=mode) as B:
            B.anneal(sched, R, T, seed=9)
            mix = [B.replica_results(k, R) for k in range(5)]
        for k, c in enumerate(insts):
            with phia.Batch([c], instance_ids=[k], csr_mode=mode) as A:
                A.anneal(sched, R, T, seed=9)
                alone = A.replica_results(0, R)
            for u, w in zip(mix[k], alone):
                assert np.array_equal(u, w)


# Edges of the resident kernels' sizes: 16-spin warps, the classes of 64, 128 and 256 spins, clusters
# of 2 and 4 CTAs, and the first size that gathers; replicas in one wave and in many.
@pytest.mark.parametrize("N,R", [(1, 3), (16, 40), (64, 8), (65, 33), (128, 300), (129, 17), (256, 256), (257, 9),
                                 (384, 70), (385, 5), (512, 256), (513, 40), (300, 3000)])
def test_small_sparse_handles_equal_the_gather(gpu_lib, N, R):
    """Small sparse instances run on a resident kernel where that is estimated faster: records
    (frozen at a replica's own hit where the run stops at a target) and states of runs in pieces
    are those of the gather."""
    phia = gpu_lib
    T = 50
    c = _to_csr(ins.Dense((ins.dense_int(N, 127, 9, seed=N).k * _mask(N, 0.1)).astype(np.int8),
                          ins.dense_int(N, 7, 90, seed=N).kh))
    big = ins.erdos_renyi(600, 0.02, 127, 31, 4, seed=1)
    for target, stop in ((None, False), (-40 * N, True)):
        sched = phia.schedule(0.01, 0.1, 0.1, 2.0, refresh=13, target=target, stop_at_target=stop)
        with phia.Batch([c, big]) as B:
            B.anneal(sched, R, T, seed=5)
            a = B.replica_results(0, R)
        with phia.Annealer(h_k=c.kh, csr=(c.row_ptr, c.col, c.val), path=phia.PATH_CSR) as A:
            x = torch.empty((R, N), device="cuda"); v = torch.empty((R, N), device="cuda")
            phia.init_state(A.h, R, 5, x, v)
            for t0, n in ((0, 1), (1, 2), (3, T - 3)):
                phia.run(A.h, sched, R, t0, n, T, 5, x, v, reset_best=(t0 == 0))
            b = phia.replica_results(A.h, R, N)
            torch.cuda.synchronize()
            assert phia.stats_get(A.h).path == phia.PATH_CSR
        for u, w in zip(a, b):
            assert np.array_equal(u, w)
    with phia.Annealer(c.to_dense().k, c.kh, path=phia.PATH_TC, tc_kernel=phia.KERNEL_PER_STEP, large_variant=1) as D:
        xd = torch.empty((R, N), device="cuda"); vd = torch.empty((R, N), device="cuda")
        phia.init_state(D.h, R, 5, xd, vd)
        phia.run(D.h, phia.schedule(0.01, 0.1, 0.1, 2.0, refresh=13), R, 0, T, T, 5, xd, vd)
        torch.cuda.synchronize()
        assert torch.equal(x, xd) and torch.equal(v, vd)
