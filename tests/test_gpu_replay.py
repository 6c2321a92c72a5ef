"""Step graphs kept on a handle and replayed by runs from another state, time, packet or basis:
every call keeps the number of steps, the time step and the read-out interval, so that a run
after the first replays what the first one captured (the host tests count the captures), and
equals the same run on a fresh handle, bit for bit; kd_step and kd_batch_step."""
import numpy as np
import pytest

from paper_2307_01571_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def kd():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2307_01571_gb300 import _build
    _build.build()
    from paper_2307_01571_gb300 import kd as mod
    return mod


WL = W.small(64, 128, W.GAUSS, units=W.ATOMIC, a0=0.3)


def _start(sim, k):
    """The k-th start: one momentum (the read-out windows stay), other places, spins, times,
    bases and states."""
    g, p = WL.grid, WL.packet
    pk = [p,
          W.Packet(p.p0x, p.p0y, 0.2 * g.x_max, -0.1 * g.y_max, p.sigma_p, -1, p.basis),
          p,
          W.Packet(p.p0x, p.p0y, 0.0, 0.3 * g.y_max, p.sigma_p, 1, 1 - p.basis),     # the basis alone
          W.Packet(p.p0x, p.p0y, 0.0, 0.3 * g.y_max, p.sigma_p, -1, 1 - p.basis)][k]
    sim.init_packet(pk)
    if k == 2:
        sim.set_spinor(W.random_spinor(g.nx, g.ny, 5))
    sim.set_time([0.0, 2.5, 1.7, 0.0, 7.0][k] * WL.dt)


ORDER = (0, 1, 2, 0, 2, 1, 3, 4, 3, 0, 1)


@pytest.mark.parametrize("obs_every", [0, 4])
@pytest.mark.parametrize("prec", [0, 1, 3])
def test_runs_replayed_from_other_starts(kd, prec, obs_every):
    with kd.Sim(WL.units, WL.grid, WL.field, prec) as used:
        for k in ORDER:
            _start(used, k)
            obs = used.step(WL.dt, 12, obs_every=obs_every)
            with kd.Sim(WL.units, WL.grid, WL.field, prec) as fresh:
                _start(fresh, k)
                ref = fresh.step(WL.dt, 12, obs_every=obs_every)
                assert np.array_equal(used.get_spinor(), fresh.get_spinor()), k
                assert obs == ref and used.get_time() == fresh.get_time(), k


@pytest.mark.parametrize("obs_every", [0, 4])
def test_batches_replayed_from_other_starts(kd, obs_every):
    precs = (1, 0, 1)
    sims = [kd.Sim(WL.units, WL.grid, WL.field, p) for p in precs]
    with kd.Batch(sims) as b:
        for i, k in enumerate(ORDER):
            ks = [k, ORDER[(i + 1) % len(ORDER)], ORDER[(i + 3) % len(ORDER)]]
            for s, kk in zip(sims, ks):
                _start(s, kk)
            obs = b.step([WL.dt] * 3, 12, obs_every=obs_every)
            for s, p, kk, o in zip(sims, precs, ks, obs):
                with kd.Sim(WL.units, WL.grid, WL.field, p) as fresh:
                    _start(fresh, kk)
                    ref = fresh.step(WL.dt, 12, obs_every=obs_every)
                    assert np.array_equal(s.get_spinor(), fresh.get_spinor()) and o == ref, (i, kk)
    for s in sims:
        s.close()
