"""GPU tests of the resident kernel over thread-block clusters (dense, N up to 1024 with the
e4m3 operand, 512 with bf16), which automatic handles take where its estimated time is least:
the same exact fields and the same FP32 update per replica as one launch per iteration, so
records and final states must be equal bit for bit."""
import pytest

from paper_2407_10205_gb300 import instances as ins
from test_gpu_warp import assert_same, run_pieces

pytestmark = pytest.mark.gpu


# Edges of a CTA's 128 or 192 spins, of the fragments' sizes (256, 384, 512, 768, 1024 spins) and
# of the operands; ragged replicas (8 per cluster); more clusters than the GPU holds at once.
@pytest.mark.parametrize("N,R,kmax,hmax,op", [
    (128, 8, 7, 7, 1), (129, 9, 127, 100, 2), (255, 1, 7, 7, 1), (256, 700, 16, 7, 1), (257, 33, 127, 9, 2),
    (384, 17, 16, 1 << 20, 1), (385, 8, 7, 7, 1), (512, 5, 127, (1 << 24) - 1, 2), (513, 3, 16, 7, 1),
    (768, 9, 7, (1 << 24) - 1, 1), (769, 8, 7, 7, 1), (1024, 20, 16, 0, 1)])
def test_cluster_kernel_equals_one_launch_per_iteration(gpu_lib, N, R, kmax, hmax, op):
    phia = gpu_lib
    d = ins.dense_int(N, kmax, hmax, seed=N + R)
    for deriv in (0, 1):
        sched = phia.schedule(0.01, 0.2, 0.1, 2.0, refresh=11, deriv=deriv)
        a, _ = run_pieces(phia, d, phia.KERNEL_PER_STEP, sched, R, [50], 6, operand=op, large_variant=1)
        b, st = run_pieces(phia, d, phia.KERNEL_PER_STEP, sched, R, [1, 4, 45], 6, operand=op)
        assert st.tc_kernel == 2 and st.kernel_launches <= 2   # one launch, after the counters' reset
        assert_same(a, b)


@pytest.mark.parametrize("N,op", [(200, 0), (333, 1), (400, 1)])
def test_automatic_choice_and_early_stop_agree(gpu_lib, N, op):
    """Runs that stop at a target never take the cluster kernel; the earliest hit is the same as
    with a target that does not stop the run."""
    phia = gpu_lib
    R, T = 64, 200
    d = ins.sk_pm1(N, 3)
    with phia.Annealer(d.k, d.kh, path=phia.PATH_TC, operand=op) as A:
        phia.anneal(A.h, phia.schedule(0.01, 0.2, 0.1, 2.0), R, T, 2)
        target = int(phia.stats_get(A.h).best_energy_k) + 40
        hits = []
        for stop in (False, True):
            phia.anneal(A.h, phia.schedule(0.01, 0.2, 0.1, 2.0, target=target, stop_at_target=stop), R, T, 2)
            st = phia.stats_get(A.h)
            hits.append((st.hit_step, st.hit_replica))
    assert hits[0][0] >= 0 and hits[0] == hits[1]
