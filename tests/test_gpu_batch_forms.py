"""Every form of a batch's step -- the march straight from L1/L2, the TMA-staged
kernel with one and with two float4 per thread, several z splits -- against
single contexts, bitwise, the form being asked for and not left to the fitted
times: row counts that leave one, an odd and an even number of rows in the last
tile, fewer rows than a tile, widths at which 256 threads hold a broken number
of rows, the narrowest and widest rows, rows that no staged form takes.  And
which form is chosen for batches that stay in L2 and that stream from HBM."""
import numpy as np
import pytest

from paper_1610_06749_gb300 import binding as B
from paper_1610_06749_gb300 import synth

pytestmark = pytest.mark.gpu

DX, V, STEPS = 5e-4, 150.0, 6
SHAPES = [(136, 43, 30), (256, 17, 20), (256, 9, 33), (200, 21, 20), (244, 19, 17), (36, 61, 20), (252, 3, 40),
          (4, 300, 24), (128, 1, 20), (64, 33, 8), (132, 14, 70), (260, 12, 20), (63, 20, 20)]


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1610_06749_gb300 import build
    build.build()
    B.lib()


def _descs(shapes):
    out = []
    for q, (nx, ny, nz) in enumerate(shapes):
        tr = synth.uniform_tracks(910 + q, 6, nx * DX, ny * DX, 8e-4)
        npk = 400.0 * B.it_peak_density(tr.let_keV_um, tr.b_cm)    # narrow sections pile up many images
        out.append((dict(nx=nx, ny=ny, nz=nz, dx_cm=DX, voltage_V=V, n_peak_cm3=npk), tr))
    return out


@pytest.fixture(scope="module")
def single(_lib):
    res = {}
    for bc in (B.IT_PERIODIC, B.IT_ABSORBING):
        for sc in (False, True):
            for k, (d, t) in enumerate(_descs(SHAPES)):
                with B.Simulation(d["nx"], d["ny"], d["nz"], DX, V, n_peak_cm3=d["n_peak_cm3"], lateral_bc=bc,
                                  scheme=B.IT_UPWIND, space_charge=sc, kernel=B.IT_KERNEL_SIMPLE) as g:
                    g.deposit(t.x_cm, t.y_cm, t.let_keV_um, t.b_cm)
                    g.step(STEPS)
                    res[bc, sc, k] = g.density(0), g.density(1), g.tallies()
    return res


@pytest.mark.parametrize("form", [(0, 1), (0, 2), (1, 1), (1, 16), (2, 1), (2, 32)], ids=lambda f: f"{f[0]}x{f[1]}")
@pytest.mark.parametrize("bc", [B.IT_PERIODIC, B.IT_ABSORBING])
@pytest.mark.parametrize("sc", [False, True])
def test_every_form_equals_single_contexts(single, form, bc, sc):
    sims = _descs(SHAPES)
    with B.Batch([d for d, _ in sims], lateral_bc=bc, scheme=B.IT_UPWIND, space_charge=sc) as bt:
        for k, (_, t) in enumerate(sims):
            bt.deposit(k, t.x_cm, t.y_cm, t.let_keV_um, t.b_cm)
        B.it_test_batch_launch(bt.h, *form)
        assert bt.launch() == {"float4_per_thread": form[0], "ctas_per_sm": form[1] if form[0] else 0}
        bt.run(tol=0.0, max_steps=STEPS, check_every=STEPS)
        for k in range(len(sims)):
            p, m, t = single[bc, sc, k]
            assert np.isfinite(p).all()
            assert np.array_equal(bt.density(k, 0), p) and np.array_equal(bt.density(k, 1), m), k
            a, tol = bt.tallies(k), 1e-6 * t.released.sum()
            assert a.steps == t.steps and abs(a.recombined - t.recombined) <= tol
            for name in ("collected_anode", "collected_cathode", "lost_lateral", "in_domain", "space_charge"):
                assert np.max(np.abs(getattr(a, name) - getattr(t, name))) <= tol, (k, name)


def test_small_batches_march_straight_and_large_ones_are_staged():
    with B.Batch([d for d, _ in _descs(SHAPES)]) as bt:
        assert bt.launch()["float4_per_thread"] == 0
    big = [(136, 143, 260), (256, 117, 180), (200, 121, 220), (244, 99, 230), (36, 301, 250), (100, 250, 200),
           (252, 7, 300), (4, 600, 280), (128, 129, 300), (64, 331, 250), (148, 147, 230), (180, 203, 140)]
    for sc in (False, True):      # the batch whose staged march is compared with single contexts
        with B.Batch([d for d, _ in _descs(big)] * 5, scheme=B.IT_UPWIND, space_charge=sc) as bt:
            assert bt.launch()["float4_per_thread"] == 2
            B.it_test_batch_launch(bt.h, 1, 4)
            assert bt.launch() == {"float4_per_thread": 1, "ctas_per_sm": 4}
            B.it_test_batch_launch(bt.h, -1)
            assert bt.launch()["float4_per_thread"] == 2
    with B.Batch([d for d, _ in _descs(SHAPES[:1])]) as bt:
        with pytest.raises(B.ItError):
            B.it_test_batch_launch(bt.h, 3, 1)
        with pytest.raises(B.ItError):
            B.it_test_batch_launch(bt.h, 2, 0)
