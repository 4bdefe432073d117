"""GPU tests of the overlapped kernel for few replicas (tiles of 128 replicas x 32 or 64 spins,
one per CTA), which automatic handles take where its estimated time is least: the same exact
fields and the same FP32 update per replica as one launch per iteration, so records and final
states must be equal bit for bit."""
import pytest

from paper_2407_10205_gb300 import instances as ins
from test_gpu_warp import assert_same, run_pieces

pytestmark = pytest.mark.gpu


# Sizes past the cluster kernel's range: edges of the 16-spin chunks, of both widths (64 where
# 32-wide tiles are more than the SMs), ragged replica tiles, K in one stage and in many, and
# fields so large that a chunk's energy terms leave the exact range of an FP32 sum.
@pytest.mark.parametrize("N,R,kmax,hmax,op", [
    (513, 1, 127, 7, 2), (529, 130, 127, 31, 2), (1025, 129, 16, 7, 1), (1040, 128, 7, (1 << 24) - 1, 1),
    (1100, 257, 127, 1 << 20, 2), (2000, 300, 1, 0, 1), (2431, 128, 16, 100, 1), (4500, 33, 7, 7, 1)])
def test_narrow_tiles_equal_one_launch_per_iteration(gpu_lib, N, R, kmax, hmax, op):
    phia = gpu_lib
    d = ins.dense_int(N, kmax, hmax, seed=N + R)
    for deriv in (0, 1):
        sched = phia.schedule(0.01, 0.2, 0.1, 2.0, refresh=11, deriv=deriv)
        a, _ = run_pieces(phia, d, phia.KERNEL_PER_STEP, sched, R, [30], 6, operand=op, large_variant=1)
        b, st = run_pieces(phia, d, phia.KERNEL_PER_STEP, sched, R, [1, 3, 26], 6, operand=op)
        assert st.tc_kernel == 2
        assert_same(a, b)
