"""GPU test of the server's turns: requests that run get their chunks while others are admitted."""
import pytest

from paper_2407_10205_gb300 import instances as ins

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def test_a_running_request_goes_on_while_others_are_admitted(gpu_lib):
    """The first request holds the budget for some 0.2 s, so that the others queue.  When it ends they
    are admitted one after the other; the second request needs six chunks, each shorter than an
    admission, and has to end before the last of the twelve behind it has been admitted."""
    phia = gpu_lib
    sched = phia.schedule(0.02, 0.5, 0.1, 2.0, refresh=40)
    hold = ins.dense_int(200, 7, 7, 1)
    others = [ins.erdos_renyi(600, 0.2, 127, 127, 8, 10 + k) for k in range(13)]
    with phia.Server(max_inflight=16, hbm_budget_bytes=46 << 20, chunk_iters=20) as S:
        first = S.submit(hold, sched, 8192, 30000, seed=1)
        ids = [S.submit(c, sched, 32, 120, seed=2 + k, instance_id=k) for k, c in enumerate(others)]
        S.wait_all()
        st = [S.poll(i)[0] for i in ids]
        end = S.poll(first)[0].t_done_s
    assert all(s.state == 2 and s.steps_run == 120 for s in st)
    assert all(s.t_submit_s < end <= s.t_admit_s for s in st)      # the case that is meant
    assert st[0].t_done_s < st[-1].t_admit_s
