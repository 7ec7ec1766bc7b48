"""Continuous batching, told by launch numbers: a request that arrives while another runs is carried by a
launch of that run.  (Admission times do not tell: two requests of one pass have different ones.)"""
import numpy as np
import pytest

from paper_2501_17913_gb300 import inputs as I
from paper_2501_17913_gb300 import serve, tjm

from test_serve_host import Clock, FakeBackend, _wl


def joined_a_running_batch(done):
    return any(b.first_launch < a.first_launch <= b.last_launch for a in done for b in done)


class OneBatchAtATime(serve.Server):
    """A server without continuous batching: admits only when nothing runs."""

    def _admit(self, now):
        if not self.active:
            super()._admit(now)


@pytest.mark.parametrize("cls,expected", [(serve.Server, True), (OneBatchAtATime, False)])
def test_launch_numbers_show_continuous_batching(cls, expected):
    clk = Clock()
    srv = cls(mem_budget=10 ** 12, backend=FakeBackend(clk), clock=clk)
    for n_steps, arrival in ((4, 0.0), (2, 0.0), (3, 1.5), (1, 20.0)):
        srv.submit(_wl(4, n_steps), arrival=arrival)
    while srv.tick():
        if not srv.active and srv.queue:
            clk.t = max(clk.t, min(q.arrival for q in srv.queue))
    done = sorted(srv.finished, key=lambda r: r.rid)
    assert len(done) == 4
    assert (done[0].first_launch, done[0].last_launch, done[1].last_launch) == (1, 4, 2)
    assert all(r.last_launch - r.first_launch + 1 == r.wl.n_steps for r in done)
    assert joined_a_running_batch(done) is expected
    srv.close()


@pytest.mark.gpu
def test_request_submitted_during_a_run_joins_it_with_the_result_it_has_alone():
    """Arrivals tied to launches, not to the clock: the second and third request come after launch 2 of the
    first one's eight or nine (one step each, the first launch also initialises)."""
    from gpu_common import lib_ready
    lib_ready()
    wls = [I.Workload('req%d' % k, I.xxx_mpo(L, 1.0, 0.3), I.noise(L, 0.2, 0.2), 0.1, n, chi, 1e-10, 5, 50 + k,
                      I.neel(L), I.z_observables(L), list(range(n + 1)))
           for k, (L, chi, n) in enumerate([(12, 8, 8), (8, 4, 3), (10, 8, 2)])]
    srv = serve.Server(precision=tjm.PREC_FP32_DEC32, steps_per_tick=1, keep_per_traj=True)
    srv.submit(wls[0])
    assert srv.tick() and srv.tick()
    for wl in wls[1:]:
        srv.submit(wl)
    done = sorted(srv.drain(), key=lambda r: r.rid)
    assert [r.first_launch for r in done] == [1, 3, 3]
    assert done[0].last_launch > max(done[1].last_launch, done[2].last_launch) and joined_a_running_batch(done)
    for r in done:
        wl = r.wl
        ctx = tjm.Context(wl.W, wl.jumps, wl.dt, wl.chi_max, wl.trunc_eps, precision=tjm.PREC_FP32_DEC32)
        alone = ctx.result(ctx.run(np.array(wl.psi0), wl.n_traj, wl.seed, wl.observables, wl.times))[2]
        assert np.array_equal(alone, r.per_traj), r.rid
        ctx.close()
    srv.close()
