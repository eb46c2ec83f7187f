"""The tilted deposit from per-plane tables (few tracks) against the kernel
that evaluates every weight in every cell (tables of more than 256 MB): the
same tracks in one call and in two halves, in FP64 storage.  Both add the
same FP64 products, so they agree to the rounding of a sum of n terms,
n 2^-53 = 2.2e-13 for 2000 tracks; 1e-12 of the maximum is asked."""
import numpy as np
import pytest

from paper_1610_06749_gb300 import binding as B
from paper_1610_06749_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lat", [B.IT_PERIODIC, B.IT_ABSORBING])
def test_table_form_equals_the_general_form(lat):
    from paper_1610_06749_gb300 import build
    build.build()
    nx, ny, nz, dx, n = 61, 3, 299, 5e-4, 2000     # tables: 292 MB for all tracks, 146 MB for half
    tr = synth.uniform_tracks(17, n, nx * dx, ny * dx, 2e-4)
    th = 0.5 * np.pi * synth.uniform01(18, n)
    th[:3] = (0.0, 0.5 * np.pi, 0.5 * np.pi - 1e-5)
    res = []
    for parts in (1, 2):
        with B.Simulation(nx, ny, nz, dx, 200.0, dt_s=1e-9, lateral_bc=lat, precision=B.IT_FP64) as g:
            for q in range(parts):
                s = slice(q * n // parts, (q + 1) * n // parts)
                g.deposit_angled(tr.x_cm[s], tr.y_cm[s], tr.let_keV_um[s], tr.b_cm[s], th[s])
            res.append((g.density(0), g.density(1), g.tallies().released))
    (a, b, ra), (c, d, rc) = res
    assert np.max(np.abs(a - c)) <= 1e-12 * np.max(a) and np.array_equal(a, b) and np.array_equal(c, d)
    assert np.max(np.abs(ra - rc)) <= 1e-12 * ra[0]
