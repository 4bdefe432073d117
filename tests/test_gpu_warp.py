"""GPU tests of the resident warp-level kernel (dense, N <= 256): its FP32 sums of integer
products are exact and its update does the same operations in the same order as the resident
tcgen05 kernel, so records and final states must be equal bit for bit."""
import numpy as np
import pytest

from paper_2407_10205_gb300 import instances as ins

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def run_pieces(phia, d, kern, sched, R, pieces, seed, **kw):
    """Records and final states of one run in the given pieces, and the last piece's stats."""
    N, T = d.n, sum(pieces)
    with phia.Annealer(d.k, d.kh, path=phia.PATH_TC, tc_kernel=kern, **kw) as A:
        x = torch.empty((R, N), device="cuda"); v = torch.empty((R, N), device="cuda")
        phia.init_state(A.h, R, seed, x, v)
        t0 = 0
        for k, s in enumerate(pieces):
            phia.run(A.h, sched, R, t0, s, T, seed, x, v, reset_best=(k == 0))
            t0 += s
        torch.cuda.synchronize()
        return (*phia.replica_results(A.h, R, N), x.cpu().numpy(), v.cpu().numpy()), phia.stats_get(A.h)


def assert_same(a, b):
    for u, w in zip(a, b):
        assert np.array_equal(u, w)


# Edges of the 16-spin warps, of the sizes the kernel is built for (1, 2, 4, 6, 8, 10, 13, 15, 16
# warps), ragged replicas (8 per CTA), the largest couplings and the largest fields.
@pytest.mark.parametrize("N,R,kmax,hmax", [
    (1, 5, 7, 7), (15, 1, 16, 0), (16, 8, 7, 7), (17, 9, 127, 100), (64, 33, 7, 7), (65, 7, 16, 7),
    (96, 16, 7, 7), (127, 2500, 7, 7), (129, 17, 127, 31), (160, 8, 7, 7), (161, 24, 16, 1 << 20),
    (208, 9, 7, 7), (209, 11, 7, 7), (240, 300, 127, 127), (241, 16, 7, 7),
    (256, 1300, 127, (1 << 24) - 1)])
def test_warp_kernel_equals_resident_tcgen05(gpu_lib, N, R, kmax, hmax):
    phia = gpu_lib
    d = ins.dense_int(N, kmax, hmax, seed=N + R)
    for deriv in (0, 1):
        sched = phia.schedule(0.01, 0.3, 0.1, 2.0, refresh=13, deriv=deriv)
        a, sa = run_pieces(phia, d, phia.KERNEL_RESIDENT, sched, R, [60], 4)
        b, sb = run_pieces(phia, d, 3, sched, R, [1, 2, 57], 4)
        assert sa.tc_kernel == 1 and sb.tc_kernel == 3
        assert_same(a, b)


def test_automatic_handle_after_an_acceptance_run(gpu_lib):
    """Runs with the acceptance test take the tcgen05 resident kernel; the next ordinary run of
    an automatic handle takes the kernel that it took before, with the same records."""
    phia = gpu_lib
    N, R, T = 100, 20, 40
    d = ins.dense_int(N, 7, 7, seed=3)
    plain = phia.schedule(0.01, 0.3, 0.1, 2.0, refresh=10)
    with phia.Annealer(d.k, d.kh, path=phia.PATH_TC) as A:
        phia.anneal(A.h, plain, R, T, 5)
        before, k0 = phia.replica_results(A.h, R, N), phia.stats_get(A.h).tc_kernel
        phia.anneal(A.h, phia.schedule(0.01, 0.3, 0.1, 2.0, refresh=10, accept_test=1), R, T, 5)
        assert phia.stats_get(A.h).tc_kernel == 1
        phia.anneal(A.h, plain, R, T, 5)
        assert phia.stats_get(A.h).tc_kernel == k0
        assert_same(before, phia.replica_results(A.h, R, N))
