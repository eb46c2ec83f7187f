"""The autotuner remembers its choice per kind of chamber: the space-charge
term selects other instances of the step kernel, so a chamber with it is timed
by itself, and one like it is not timed again."""
import pytest

from paper_1610_06749_gb300 import binding as B
from paper_1610_06749_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1610_06749_gb300 import build
    build.build()
    B.lib()


@pytest.mark.parametrize("order", [(False, True), (True, False)])
def test_space_charge_is_tuned_by_itself(order):
    # a grid per order, which nothing else tunes
    nx, ny, nz, dx, V = (68, 30, 22, 5e-4, 200.0) if order[0] else (76, 30, 22, 5e-4, 200.0)
    tr = synth.uniform_tracks(53, 5, nx * dx, ny * dx, 8e-4)
    for again in (False, True):
        for sc in order:
            with B.Simulation(nx, ny, nz, dx, V, space_charge=sc, n_peak_cm3=1e12) as g:
                g.deposit(tr.x_cm, tr.y_cm, tr.let_keV_um, tr.b_cm)
                us = g.autotune(trial_steps=2)
                assert us == -1.0 if again else us > 0, (sc, again)
