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
    with phia.Server(max_inflight=16, hbm_budget_bytes=44 << 20, chunk_iters=20) as S:
        first = S.submit(hold, sched, 8192, 30000, seed=1)
        ids = [S.submit(c, sched, 32, 120, seed=2 + k, instance_id=k) for k, c in enumerate(others)]
        S.wait_all()
        st = [S.poll(i)[0] for i in ids]
        end = S.poll(first)[0].t_done_s
    assert all(s.state == 2 and s.steps_run == 120 for s in st)
    assert all(s.t_submit_s < end <= s.t_admit_s for s in st)      # the case that is meant
    assert st[0].t_done_s < st[-1].t_admit_s


def test_large_dense_requests_in_turns_equal_the_same_alone(gpu_lib):
    """Beside other requests a large dense one runs one launch per iteration, alone all iterations of a
    chunk in one: the records are the same, whichever its chunks take."""
    phia = gpu_lib
    sched = phia.schedule(0.005, 0.13, 0.1, 2.0, refresh=30)
    insts = [ins.sk_pm1(n, n) for n in (1500, 2100, 900)]
    with phia.Server(max_inflight=3, hbm_budget_bytes=8 << 30, chunk_iters=40) as S:
        ids = [S.submit(c, sched, 300, 160, seed=5 + k, instance_id=k) for k, c in enumerate(insts)]
        S.wait_all()
        mix = [S.poll(i, want_spins=True) for i in ids]
    for k, (c, (st, spins)) in enumerate(zip(insts, mix)):
        with phia.Annealer(c.k, c.kh, path=phia.PATH_TC, instance_id=k) as A:
            alone = A.anneal(sched, 300, 160, 5 + k)
        assert st.state == 2 and st.energy_k == alone.energy_k
        assert (spins == alone.spins).all()


def test_the_budget_counts_what_a_sparse_request_takes(gpu_lib):
    """Slices pad the rows, and large instances keep their couplings twice (some 10 bytes each): a budget
    that holds the rest of the request and 5 bytes a coupling is not enough."""
    phia = gpu_lib
    n, R = 40000, 256
    c = ins.erdos_renyi(n, 100.0 / n, 127, 31, 4, 1)
    rest = 2 * R * n * 4 + n * 8 * 256 + 4 * n * 8 * 4 + 256 * (24 + n // 8) + 8 * n + (1 << 20)
    sched = phia.schedule(0.02, 0.5, 0.1, 2.0)
    with phia.Server(max_inflight=1, hbm_budget_bytes=rest + 5 * c.nnz) as S:
        with pytest.raises(phia.PhiaError) as e:
            S.submit(c, sched, R, 10, seed=1)
        assert e.value.code == phia.ENOMEM
    with phia.Server(max_inflight=1, hbm_budget_bytes=rest + 12 * c.nnz) as S:
        rid = S.submit(c, sched, R, 10, seed=1)
        S.wait_all()
        assert S.poll(rid)[0].state == 2
