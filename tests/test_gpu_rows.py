"""GPU tests of the sparse form with a row to a warp, which runs of large instances with few couplings
a row take from a replica count on.  A replica's run does not depend on how many run beside it, so
its records and states must equal those of 128 replicas, which take the form with a row to a lane."""
import numpy as np
import pytest

from paper_2407_10205_gb300 import instances as ins

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _star(n, seed):
    """A ring with a row that is coupled to all others."""
    g = np.random.default_rng(seed)
    pairs = {(i, (i + 1) % n): int(g.integers(1, 128)) for i in range(n)}
    pairs.update({(0, i): int(g.integers(-127, 0)) for i in range(2, n - 1)})
    rows = np.array([(i, j, k) for (i, j), k in pairs.items()] + [(j, i, k) for (i, j), k in pairs.items()])
    rows = rows[np.lexsort((rows[:, 1], rows[:, 0]))]
    rp = np.zeros(n + 1, dtype=np.int32)
    np.add.at(rp, rows[:, 0] + 1, 1)
    return ins.Csr(np.cumsum(rp).astype(np.int32), rows[:, 1].astype(np.int32), rows[:, 2].astype(np.int8),
                   g.integers(-99, 100, n).astype(np.int32), 4)


# Both sides of the size whose spins fit in shared memory, a last block of few rows, ragged replicas,
# fields that make the terms wide, one row much longer than the others.
@pytest.mark.parametrize("n,R,degree,hmax", [(20000, 256, 6, 31), (12609, 1000, 6, 31), (28928, 250, 12, 31),
                                             (30001, 256, 30, (1 << 24) - 1), (9000, 500, 0, 0)])
@pytest.mark.parametrize("mode", [0, 1])
def test_rows_to_warps_equal_rows_to_lanes(gpu_lib, n, R, degree, hmax, mode):
    phia = gpu_lib
    T, part = 25, 128
    c = ins.erdos_renyi(n, degree / n, 127, hmax, 4, seed=n) if degree else _star(n, 3)
    with phia.Annealer(h_k=c.kh, frac_bits=4, csr=(c.row_ptr, c.col, c.val), tc_kernel=mode) as A:
        phia.anneal(A.h, phia.schedule(0.01, 0.2, 0.1, 2.0, refresh=6), part, T, 3)
        target = int(np.median(phia.replica_results(A.h, part, n)[0]))
    for deriv, stop in ((0, False), (1, True)):
        sched = phia.schedule(0.01, 0.2, 0.1, 2.0, refresh=6, deriv=deriv, target=target, stop_at_target=stop)
        out = []
        for reps, pieces in ((part, (T,)), (R, (1, 2, T - 3))):
            with phia.Annealer(h_k=c.kh, frac_bits=4, csr=(c.row_ptr, c.col, c.val), tc_kernel=mode) as A:
                x, v = torch.empty((reps, n), device="cuda"), torch.empty((reps, n), device="cuda")
                phia.init_state(A.h, reps, 3, x, v)
                t0 = 0
                for k in pieces:
                    phia.run(A.h, sched, reps, t0, k, T, 3, x, v, reset_best=(t0 == 0))
                    t0 += k
                torch.cuda.synchronize()
                rec = phia.replica_results(A.h, reps, n)
                out.append([u[:part] for u in rec] + [x[:part].cpu().numpy(), v[:part].cpu().numpy()])
        for u, w in zip(*out):
            assert np.array_equal(u, w)
