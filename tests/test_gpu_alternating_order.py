"""The marches without a ring on states that stream from HBM, whose units run
in reverse on every other step: bitwise the staged march and the simple kernel
alone, tallies to 1e-6 of the released charge (the staged march sums up to 32
planes in plain FP32)."""
import numpy as np
import pytest

from paper_1610_06749_gb300 import binding as B
from paper_1610_06749_gb300 import synth

pytestmark = pytest.mark.gpu

DX, V = 5e-4, 200.0


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1610_06749_gb300 import build
    build.build()
    B.lib()


def _same(a, b, tol):
    assert abs(a.recombined - b.recombined) <= tol
    for name in ("collected_anode", "collected_cathode", "lost_lateral", "in_domain", "space_charge"):
        assert np.max(np.abs(getattr(a, name) - getattr(b, name))) <= tol, name


@pytest.mark.parametrize("lat", [B.IT_PERIODIC, B.IT_ABSORBING])
def test_single_direct_march(lat):
    nx, ny, nz = 224, 293, 119                      # ny is prime: no tile for the ring
    n = [(1e13 * synth.uniform01(23 + s, nx * ny * nz)).reshape(nz, ny, nx).astype(np.float32) for s in range(2)]
    res = []
    for kernel in (B.IT_KERNEL_AUTO, B.IT_KERNEL_SIMPLE):
        with B.Simulation(nx, ny, nz, DX, V, lateral_bc=lat, scheme=B.IT_UPWIND, kernel=kernel, n_peak_cm3=2e13) as g:
            g.set_density(n[0], n[1])
            g.step(5)
            res.append((g.density(0), g.density(1), g.tallies(), g.launch()))
    (p0, m0, t0, l0), (p1, m1, t1, _) = res
    assert l0["kernel"] == B.IT_KERNEL_ZMARCH and l0["stages"] == 0
    assert np.array_equal(p0, p1) and np.array_equal(m0, m1)
    _same(t0, t1, 1e-6 * t1.released.sum())


def test_batched_marches():
    # rows of more than 256 cells and of odd length: no ring for either
    sims = []
    for q, (nx, ny, nz) in enumerate([(260, 131, 120), (127, 133, 140), (300, 97, 90)]):
        tr = synth.uniform_tracks(950 + q, 6, nx * DX, ny * DX, 8e-4)
        npk = 40.0 * B.it_peak_density(tr.let_keV_um, tr.b_cm)
        sims.append((dict(nx=nx, ny=ny, nz=nz, dx_cm=DX, voltage_V=V, n_peak_cm3=npk), tr))
    assert sum(16 * d["nx"] * d["ny"] * d["nz"] for d, _ in sims) > 115e6
    with B.Batch([d for d, _ in sims], scheme=B.IT_UPWIND) as bt:
        for k, (_, t) in enumerate(sims):
            bt.deposit(k, t.x_cm, t.y_cm, t.let_keV_um, t.b_cm)
        bt.run(tol=0.0, max_steps=6, check_every=6)
        for k, (d, t) in enumerate(sims):
            with B.Simulation(d["nx"], d["ny"], d["nz"], DX, V, n_peak_cm3=d["n_peak_cm3"], scheme=B.IT_UPWIND,
                              kernel=B.IT_KERNEL_SIMPLE) as g:
                g.deposit(t.x_cm, t.y_cm, t.let_keV_um, t.b_cm)
                g.step(6)
                for s in range(2):
                    assert np.array_equal(bt.density(k, s), g.density(s)), (k, s)
                a, b = bt.tallies(k), g.tallies()
                assert a.steps == b.steps
                _same(a, b, 1e-6 * b.released.sum())
