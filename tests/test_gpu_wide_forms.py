"""The 64-bit forms' launch shapes at every axis length: the potential factors traded between
the two pairs' CTAs of a cluster (FP64, and the double-word form from 1024 points) or the two
halves of a CTA, one warp of lines per CTA, and grids with fewer lines than a CTA holds."""
import numpy as np
import pytest

import oracle
from paper_2307_01571_gb300 import workloads as W

pytestmark = pytest.mark.gpu

LENGTHS = [4, 8, 16, 32, 64, 128, 256, 512, 1024, 2048, 4096]


@pytest.fixture(scope="module")
def kd():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2307_01571_gb300 import _build
    _build.build()
    from paper_2307_01571_gb300 import kd as mod
    return mod


# three steps of O(30) roundings a point and step: 1e-13 (FP64) and 1e-12 (48 significand
# bits) of max |psi| leave an order of magnitude each
@pytest.mark.parametrize("prec,tol", [("fp64", 1e-13), ("dw", 1e-12)])
@pytest.mark.parametrize("n", LENGTHS)
@pytest.mark.parametrize("axis", ["x", "y"])
def test_every_axis_length_matches_oracle(kd, prec, tol, n, axis):
    nx, ny = (n, 8) if axis == "x" else (4, n)
    wl = W.small(nx, ny, W.GAUSS, units=W.ATOMIC, nsteps=3, a0=0.4)
    u, g, f = wl.units, wl.grid, wl.field
    psi = W.random_spinor(nx, ny, n)
    ref = oracle.step(u, g, f, psi, 0.0, wl.dt, 3)
    with kd.Sim(u, g, f, kd.KD_FP64 if prec == "fp64" else kd.KD_DW) as sim:
        sim.set_spinor(psi)
        sim.step(wl.dt, 3)
        got = sim.get_spinor()
        sim.set_spinor(psi)
        sim.set_time(0.0)
        sim.step(wl.dt, 3)
        again = sim.get_spinor()
    assert np.max(np.abs(got - ref)) <= tol * np.max(np.abs(ref))
    assert np.array_equal(got, again)
