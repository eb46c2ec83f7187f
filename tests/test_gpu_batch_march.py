"""Batches on the march without a ring (float4 segments and single cells)
against the same simulations alone, bitwise, over grids at the edges of its
entries: fewer segments than a block of 128, just below and above it, one
plane, chunks of every fitted length, both faces, the space-charge term; and
the shapes a batch moves through as its simulations finish."""
import numpy as np
import pytest

from paper_1610_06749_gb300 import binding as B
from paper_1610_06749_gb300 import synth

pytestmark = pytest.mark.gpu

SHAPES = [(4, 4, 1), (5, 3, 7), (36, 14, 9), (64, 8, 33), (64, 9, 5), (128, 4, 70), (260, 3, 11), (127, 33, 6),
          (48, 48, 100), (33, 31, 64)]


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1610_06749_gb300 import build
    build.build()
    B.lib()


def _sims():
    out = []
    for q, (nx, ny, nz) in enumerate(SHAPES):
        dx = 5e-4
        tr = synth.uniform_tracks(700 + q, 4, nx * dx, ny * dx, 8e-4)
        npk = 40.0 * B.it_peak_density(tr.let_keV_um, tr.b_cm)     # tracks pile up on small sections
        out.append((dict(nx=nx, ny=ny, nz=nz, dx_cm=dx, voltage_V=150.0 + 20 * q, n_peak_cm3=npk), tr))
    return out


@pytest.mark.parametrize("bc", [B.IT_PERIODIC, B.IT_ABSORBING])
@pytest.mark.parametrize("sc", [False, True])
def test_batch_march_equals_single_contexts_bitwise(bc, sc):
    sims = _sims()
    steps = 12
    with B.Batch([d for d, _ in sims], lateral_bc=bc, scheme=B.IT_UPWIND, space_charge=sc) as bt:
        for k, (_, t) in enumerate(sims):
            bt.deposit(k, t.x_cm, t.y_cm, t.let_keV_um, t.b_cm)
        bt.run(tol=0.0, max_steps=steps, check_every=4)
        for k, (d, t) in enumerate(sims):
            with B.Simulation(d["nx"], d["ny"], d["nz"], d["dx_cm"], d["voltage_V"], n_peak_cm3=d["n_peak_cm3"],
                              lateral_bc=bc, scheme=B.IT_UPWIND, space_charge=sc) as g:
                g.deposit(t.x_cm, t.y_cm, t.let_keV_um, t.b_cm)
                g.step(steps)
                for s in range(2):
                    assert np.array_equal(bt.density(k, s), g.density(s)), (k, s)
                a, b = bt.tallies(k), g.tallies()
                tol = 1e-6 * b.released.sum()
                assert a.steps == b.steps
                assert abs(a.recombined - b.recombined) <= tol and abs(a.f - b.f) <= 1e-6
                for name in ("collected_anode", "collected_cathode", "lost_lateral", "in_domain", "space_charge"):
                    assert np.max(np.abs(getattr(a, name) - getattr(b, name))) <= tol, (k, name)


def test_batch_through_its_shapes_to_completion():
    # autotuned, then rebuilt as simulations finish: the same steps and
    # densities as without the autotuner
    sims = [s for s in _sims() if s[0]["nz"] > 5]
    res = []
    for tune in (False, True):
        with B.Batch([d for d, _ in sims], scheme=B.IT_UPWIND, dt_ladder=True) as bt:
            for k, (_, t) in enumerate(sims):
                bt.deposit(k, t.x_cm, t.y_cm, t.let_keV_um, t.b_cm)
            if tune:
                bt.autotune(trial_steps=4)
            bt.run(tol=1e-6, max_steps=20_000, check_every=16)
            res.append([(bt.tallies(k).steps, bt.tallies(k).f, bt.density(k, 0)) for k in range(len(sims))])
    for a, b in zip(*res):
        assert a[0] == b[0] and abs(a[1] - b[1]) <= 1e-6 and np.array_equal(a[2], b[2])
