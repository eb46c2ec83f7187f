"""Deposits into a batch whose uploads are still under way when the call
returns: several thousand tracks per simulation (copies far above the 64 KB a
driver may stage at once), a second deposit into a simulation whose first may
not have been copied yet, and the re-deposits of a pulse train.  Densities
bitwise those of single contexts."""
import numpy as np
import pytest

from paper_1610_06749_gb300 import binding as B
from paper_1610_06749_gb300 import synth

pytestmark = pytest.mark.gpu

# tracks of a simulation's deposits (a context deposits up to 8192 tracks as one sum per cell)
DEPOSITS = [(2049,), (6000,), (8192,), (3000, 5000), (1, 4000, 1), (7000,), (2500, 2500), (5000,)]


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1610_06749_gb300 import build
    build.build()
    B.lib()


@pytest.mark.parametrize("pulses", [1, 3])
def test_uploads_of_many_tracks(pulses):
    nx, ny, nz, dx, V, dt, check = 64, 40, 30, 5e-4, 200.0, 1e-10, 4
    sims = [[synth.uniform_tracks(700 + 10 * k + q, n, nx * dx, ny * dx, 8e-4) for q, n in enumerate(ns)]
            for k, ns in enumerate(DEPOSITS)]
    d = dict(nx=nx, ny=ny, nz=nz, dx_cm=dx, voltage_V=V, dt_s=dt)
    steps = 4 * check
    with B.Batch([d] * len(sims), scheme=B.IT_UPWIND) as bt:
        for k, parts in enumerate(sims):
            for t in parts:
                bt.deposit(k, t.x_cm, t.y_cm, t.let_keV_um, t.b_cm)
            if pulses > 1:
                bt.set_pulses(k, pulses, check)
        bt.run(tol=0.0, max_steps=steps, check_every=check)
        for k, parts in enumerate(sims):
            with B.Simulation(nx, ny, nz, dx, V, dt_s=dt, scheme=B.IT_UPWIND) as g:
                for t in parts:
                    g.deposit(t.x_cm, t.y_cm, t.let_keV_um, t.b_cm)
                for q in range(1, pulses):
                    g.step(check)
                    # a train re-deposits all of a simulation's tracks as one
                    cat = [np.concatenate([getattr(t, a) for t in parts])
                           for a in ("x_cm", "y_cm", "let_keV_um", "b_cm")]
                    g.deposit(*cat)
                g.step(steps - (pulses - 1) * check)
                for s in range(2):
                    assert np.array_equal(bt.density(k, s), g.density(s)), (k, s)
                assert np.allclose(bt.tallies(k).released, g.tallies().released, rtol=1e-12, atol=0)
