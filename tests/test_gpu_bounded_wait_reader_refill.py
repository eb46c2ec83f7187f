"""The bounded waits of the staged march's instances without a producer warp
(space charge; absorbing faces with two rows that are no pair; more than two
float4 per thread), whose slots the last reader refills: a first load that is
never issued makes them run out, the error is reported, and after a reset the
same context steps as a fresh one does."""
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


@pytest.mark.parametrize("shape,launch,sc,lat", [((64, 48, 40), (8, 2, 4, 0), True, B.IT_PERIODIC),
                                                 ((200, 14, 30), (7, 2, 4, 0), False, B.IT_ABSORBING),
                                                 ((128, 24, 30), (24, 2, 4, 0), False, B.IT_PERIODIC),
                                                 ((384, 16, 20), (8, 2, 3, 0), True, B.IT_ABSORBING)])
def test_the_waits_run_out_and_the_context_recovers(shape, launch, sc, lat):
    nx, ny, nz = shape
    dx, V = 5e-4, 200.0
    tr = synth.uniform_tracks(33, 12, nx * dx, ny * dx, 1e-3)
    kw = dict(n_peak_cm3=40.0 * B.it_peak_density(tr.let_keV_um, tr.b_cm), scheme=B.IT_UPWIND, space_charge=sc,
              lateral_bc=lat, kernel=B.IT_KERNEL_ZMARCH)
    with B.Simulation(nx, ny, nz, dx, V, **kw) as g, B.Simulation(nx, ny, nz, dx, V, **kw) as ref:
        g.set_launch(B.IT_KERNEL_ZMARCH, *launch)
        ref.set_launch(B.IT_KERNEL_ZMARCH, *launch)
        g.deposit(tr.x_cm, tr.y_cm, tr.let_keV_um, tr.b_cm)
        B.it_set_wait_limit(g.h, 1 << 20)          # about 0.5 ms at 2 GHz
        B.it_test_withhold_load(g.h, True)
        g.step(2)
        with pytest.raises(B.ItError) as e:
            g.tallies()
        assert e.value.code == B.IT_ETIMEOUT
        B.it_test_withhold_load(g.h, False)
        g.reset()
        for h in (g, ref):
            h.deposit(tr.x_cm, tr.y_cm, tr.let_keV_um, tr.b_cm)
            h.step(40)
        a, b = g.tallies(), ref.tallies()
        assert a.steps == 40 and a.recombined == b.recombined and a.f == b.f and np.isfinite(a.recombined)
        for s in range(2):
            assert np.array_equal(g.density(s), ref.density(s))
