"""The FP32 sweeps' compiled forms by grid size (small, both pairs per thread, large): the
default variant on either side of every line of the rule, each against the oracle and, bit for
bit, against variant 1 and a repeated run."""
import numpy as np
import pytest

import oracle
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


# two steps of FP32 rounding (2^-24 a rounding, ~20 of them a stage and point, growing as their
# square root): 5e-6 of max |psi| is ten times the FP32 form's measured 5.7e-7 after four steps
TOL = 5e-6


@pytest.mark.parametrize("nx,ny", [
    (4, 4096), (4096, 4), (4096, 16), (16, 4096),            # longest axes, fewest lines
    (128, 128), (512, 128), (512, 256), (512, 512),          # y lines at 2^16 and 2^17 points
    (2048, 64), (2048, 128), (4096, 64), (4096, 128),        # x: small / both pairs
    (64, 1024), (128, 1024), (256, 1024), (512, 1024),       # y: small / one pair / large
    (128, 2048), (256, 2048)])
def test_default_form_matches_oracle(kd, nx, ny):
    wl = W.small(nx, ny, W.GAUSS, units=W.ATOMIC, nsteps=2, a0=0.4)
    u, g, f = wl.units, wl.grid, wl.field
    psi = W.random_spinor(nx, ny, nx + 3 * ny).astype(np.complex64)
    ref = oracle.step(u, g, f, psi.astype(np.complex128), 0.0, wl.dt, 2)
    out = []
    for v in ((0, 0), (1, 1), (0, 0)):
        with kd.Sim(u, g, f, kd.KD_FP32) as sim:
            sim.sweep_variants = v
            sim.set_spinor(psi)
            sim.step(wl.dt, 2)
            out.append(sim.get_spinor())
    assert np.max(np.abs(out[0] - ref)) <= TOL * np.max(np.abs(ref))
    assert np.array_equal(out[0], out[1]) and np.array_equal(out[0], out[2])


def test_large_forms_keep_a_plane_wave(kd):
    """2048 x 2048 points (the large form on both axes, beyond the oracle): a positive-energy
    plane wave is an eigenstate of every free step, psi(n) = psi(0) exp(-i (E - v p_y) n dt)."""
    wl = W.small(2048, 2048, W.NONE, units=W.ATOMIC, nsteps=20)
    u, g, f = wl.units, wl.grid, wl.field
    kx, ky = 37, -21
    px = 2 * np.pi * kx / (g.x_max - g.x_min)
    py = 2 * np.pi * ky / (g.y_max - g.y_min)
    pix, piy = px + f.p_shift_x, py + f.p_shift_y
    spin = oracle.spinor_u(u, pix, piy, 1)
    ph = np.exp(2j * np.pi * (kx * np.arange(2048)[None, :] / 2048 + ky * np.arange(2048)[:, None] / 2048))
    psi = (ph[:, :, None] * spin).astype(np.complex64)
    with kd.Sim(u, g, f, kd.KD_FP32) as sim:
        sim.set_spinor(psi)
        sim.step(wl.dt, 20)
        got = sim.get_spinor()
    E = np.sqrt(u.mc2 ** 2 + u.c ** 2 * (pix ** 2 + piy ** 2))
    ref = psi * np.exp(-1j * (E - f.box_vy * py) * 20 * wl.dt)
    assert np.max(np.abs(got - ref)) <= 2e-5 * np.max(np.abs(ref))


def test_members_of_a_crowded_batch_equal_members_alone(kd):
    """Together the members fill the SMs (2^18 points and more), so their small column sweeps
    run wide tiles; each still equals itself run alone, bit for bit."""
    shapes = [(128, 128), (256, 128), (256, 256), (64, 512), (512, 64), (32, 32), (256, 256), (128, 256)]
    wls = [W.small(nx, ny, W.GAUSS, units=W.ATOMIC, a0=0.05 * (i + 1)).with_(precision=1)
           for i, (nx, ny) in enumerate(shapes * 2)]
    assert sum(w.points for w in wls) > 1 << 18
    alone = []
    for wl in wls:
        with kd.Sim.from_workload(wl) as sim:
            sim.init_packet(wl.packet)
            obs = sim.step(wl.dt, 30, obs_every=10)
            alone.append((sim.get_spinor(), obs))
    sims = [kd.Sim.from_workload(wl) for wl in wls]
    for s, wl in zip(sims, wls):
        s.init_packet(wl.packet)
    with kd.Batch(sims) as b:
        obs = b.step([wl.dt for wl in wls], 30, obs_every=10)
    for s, o, (ref, ref_obs) in zip(sims, obs, alone):
        assert np.array_equal(s.get_spinor(), ref) and o == ref_obs
        s.close()


@pytest.mark.parametrize("prec", ["fp32", "fp64", "dw"])
def test_runs_from_new_states_and_times_replay_the_same_steps(kd, prec):
    """The step graphs outlive a new time or packet (nothing captured depends on them): every
    run on a used handle equals the same run on a fresh one, with read-outs whose windows and
    basis change in between."""
    wl = W.small(64, 128, W.GAUSS, units=W.ATOMIC, a0=0.3)
    u, g, f = wl.units, wl.grid, wl.field
    p2 = W.Packet(1.5 * wl.packet.p0x, wl.packet.p0y, 0.1 * g.x_max, 0.2 * g.y_max, wl.packet.sigma_p, -1, 1)
    prec = {"fp32": kd.KD_FP32, "fp64": kd.KD_FP64, "dw": kd.KD_DW}[prec]

    def run(sim, k):
        if k == 2:
            sim.set_spinor(W.random_spinor(64, 128, 3))
            sim.set_time(1.7 * wl.dt)
        else:
            sim.init_packet(wl.packet if k == 0 else p2)
        obs = sim.step(wl.dt, 12, obs_every=4)
        obs += sim.step(wl.dt, 6)
        return sim.get_spinor(), obs, sim.get_time()

    with kd.Sim(u, g, f, prec) as used:
        for k in (0, 1, 0, 2, 1, 2):
            psi, obs, t = run(used, k)
            with kd.Sim(u, g, f, prec) as fresh:
                if k == 2:
                    fresh.init_packet(p2 if np.isclose(spec_basis, 1) else wl.packet)   # the read-out spec
                ref, ref_obs, ref_t = run(fresh, k)
            spec_basis = 1 if k == 1 else (0 if k == 0 else spec_basis)
            assert np.array_equal(psi, ref) and obs == ref_obs and t == ref_t


@pytest.mark.parametrize("nx,ny", [(4, 1024), (32, 1024), (16, 2048), (32, 2048), (64, 2048), (16, 4096),
                                   (2048, 32), (1024, 64), (1024, 128), (1024, 256), (256, 4096)])
def test_more_default_forms_match_oracle(kd, nx, ny):
    """Tall columns on both sides of their line, and 1024-point rows in each of their forms."""
    test_default_form_matches_oracle(kd, nx, ny)


@pytest.mark.parametrize("shapes", [
    [(512, 128), (1024, 64), (2048, 32), (2048, 64), (512, 256), (1024, 128), (8, 8)],
    [(64, 512), (128, 512), (256, 512), (64, 1024), (32, 1024), (4, 1024), (32, 2048)],
    [(128, 1024), (256, 1024), (64, 2048), (16, 4096), (64, 4096), (8, 2048)]])
@pytest.mark.parametrize("variants", [None, (0, 3), (1, 2)])
def test_long_lines_in_a_crowded_batch_equal_members_alone(kd, shapes, variants):
    """As test_members_of_a_crowded_batch_equal_members_alone, at every length and size whose
    form a crowd changes, with the default variants and others beside them."""
    wls = [W.small(nx, ny, W.GAUSS, units=W.ATOMIC, a0=0.3).with_(precision=1) for nx, ny in shapes]
    assert sum(w.points for w in wls) > 1 << 18

    def make(wl):
        sim = kd.Sim.from_workload(wl)
        if variants:
            sim.sweep_variants = variants
        sim.init_packet(wl.packet)
        return sim

    alone = []
    for wl in wls:
        with make(wl) as sim:
            alone.append((sim.step(wl.dt, 6, obs_every=3), sim.get_spinor()))
    sims = [make(wl) for wl in wls]
    with kd.Batch(sims) as b:
        obs = b.step([wl.dt for wl in wls], 6, obs_every=3)
    for s, o, (ref_obs, ref) in zip(sims, obs, alone):
        assert np.array_equal(s.get_spinor(), ref) and o == ref_obs
        s.close()
