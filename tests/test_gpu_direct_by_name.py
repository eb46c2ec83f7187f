"""The march without a ring can be asked for by what it_get_launch reports of
it, on another context and whatever that one's automatic choice is: a shape
the autotuner has found can be kept."""
import dataclasses

import numpy as np
import pytest

from paper_1610_06749_gb300 import binding as B
from paper_1610_06749_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1610_06749_gb300 import build
    build.build()
    B.lib()


def _run(g, tr):
    g.deposit(tr.x_cm, tr.y_cm, tr.let_keV_um, tr.b_cm)
    g.step(35)
    t = g.tallies()
    return {f.name: np.asarray(getattr(t, f.name)).tolist() for f in dataclasses.fields(t)}, g.density(0), g.density(1)


@pytest.mark.parametrize("kernel", [B.IT_KERNEL_AUTO, B.IT_KERNEL_SIMPLE, B.IT_KERNEL_ZMARCH])
def test_the_reported_shape_selects_the_direct_march(kernel):
    nx, ny, nz, dx, V = 64, 48, 40, 5e-4, 200.0
    tr = synth.uniform_tracks(47, 30, nx * dx, ny * dx, 1e-3)
    npk = 40.0 * B.it_peak_density(tr.let_keV_um, tr.b_cm)      # tracks and their images may pile up
    with B.Simulation(nx, ny, nz, dx, V, n_peak_cm3=npk) as a, \
            B.Simulation(nx, ny, nz, dx, V, n_peak_cm3=npk, kernel=kernel) as b:
        shape = a.launch()
        assert shape["kernel"] == B.IT_KERNEL_ZMARCH and shape["tile_rows"] == B.IT_NO_RING and shape["stages"] == 0
        b.set_launch(**{k: shape[k] for k in ("kernel", "tile_rows", "ctas_per_sm", "stages")})
        assert b.launch() == shape
        ra, rb = _run(a, tr), _run(b, tr)
    assert ra[0]["recombined"] > 0 and ra[0] == rb[0]          # the same sums in the same order
    assert np.array_equal(ra[1], rb[1]) and np.array_equal(ra[2], rb[2])


def test_other_rows_stay_the_ring():
    with B.Simulation(64, 48, 40, 5e-4, 200.0) as g:
        for rows in (0, -2):
            g.set_launch(B.IT_KERNEL_ZMARCH, rows)
            assert g.launch()["stages"] >= 3 and g.launch()["tile_rows"] > 0
        with pytest.raises(B.ItError):       # no segments of four cells
            with B.Simulation(66, 48, 40, 5e-4, 200.0) as odd:
                odd.set_launch(B.IT_KERNEL_ZMARCH, B.IT_NO_RING)
