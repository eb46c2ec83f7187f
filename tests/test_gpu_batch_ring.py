"""Batches large enough for the TMA-staged march against the same simulations
alone, bitwise, where its tiles can go wrong: row counts that leave one, an odd
and an even number of rows in the last tile, fewer rows than a tile, widths at
which 256 threads hold a whole and a broken number of rows, the narrowest and
the widest rows, both faces, the space-charge term."""
import numpy as np
import pytest

from paper_1610_06749_gb300 import binding as B
from paper_1610_06749_gb300 import synth

pytestmark = pytest.mark.gpu

SHAPES = [(136, 143, 260), (256, 117, 180), (200, 121, 220), (244, 99, 230), (36, 301, 250), (100, 250, 200),
          (252, 7, 300), (4, 600, 280), (128, 129, 300), (64, 331, 250), (148, 147, 230), (180, 203, 140)]


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1610_06749_gb300 import build
    build.build()
    B.lib()


@pytest.mark.parametrize("bc", [B.IT_PERIODIC, B.IT_ABSORBING])
@pytest.mark.parametrize("sc", [False, True])
def test_batch_staged_march_equals_single_contexts_bitwise(bc, sc):
    sims, dx, steps = [], 5e-4, 6
    for q, (nx, ny, nz) in enumerate(SHAPES):
        tr = synth.uniform_tracks(900 + q, 6, nx * dx, ny * dx, 8e-4)
        npk = 40.0 * B.it_peak_density(tr.let_keV_um, tr.b_cm)
        sims.append((dict(nx=nx, ny=ny, nz=nz, dx_cm=dx, voltage_V=150.0 + 20 * q, n_peak_cm3=npk), tr))
    # every simulation five times: 3 GB, where staging by TMA is the faster
    with B.Batch([d for d, _ in sims] * 5, lateral_bc=bc, scheme=B.IT_UPWIND, space_charge=sc) as bt:
        for k, (_, t) in enumerate(sims * 5):
            bt.deposit(k, t.x_cm, t.y_cm, t.let_keV_um, t.b_cm)
        bt.run(tol=0.0, max_steps=steps, check_every=6)
        for k, (d, t) in enumerate(sims):
            with B.Simulation(d["nx"], d["ny"], d["nz"], d["dx_cm"], d["voltage_V"], n_peak_cm3=d["n_peak_cm3"],
                              lateral_bc=bc, scheme=B.IT_UPWIND, space_charge=sc) as g:
                g.deposit(t.x_cm, t.y_cm, t.let_keV_um, t.b_cm)
                g.step(steps)
                for s in range(2):
                    a = g.density(s)
                    assert np.array_equal(bt.density(k, s), a), (k, s)
                    assert np.array_equal(bt.density(k + 4 * len(sims), s), a), (k, s)
                a, b = bt.tallies(k), g.tallies()
                tol = 1e-6 * b.released.sum()
                assert a.steps == b.steps
                assert abs(a.recombined - b.recombined) <= tol and abs(a.f - b.f) <= 1e-6
                for name in ("collected_anode", "collected_cathode", "lost_lateral", "in_domain", "space_charge"):
                    assert np.max(np.abs(getattr(a, name) - getattr(b, name))) <= tol, (k, name)
