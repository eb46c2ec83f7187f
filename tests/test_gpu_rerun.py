"""A context that is reset, or given densities, after an odd number of steps
runs as a fresh one does: bitwise the same tallies.  The marches alternate
their direction step by step, and the sums of a step depend on it."""
import dataclasses

import numpy as np
import pytest

from paper_1610_06749_gb300 import binding as B
from paper_1610_06749_gb300 import synth

pytestmark = pytest.mark.gpu

DX, V = 5e-4, 200.0
# the staged march, on two CTAs that walk many planes each; the march without a
# ring, above the size from which its units alternate
CASES = [((64, 24, 90), (8, 2, 4, 2)), ((224, 293, 119), None)]


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1610_06749_gb300 import build
    build.build()
    B.lib()


def _fields(t):
    return {f.name: np.asarray(getattr(t, f.name)).tolist() for f in dataclasses.fields(t)}


@pytest.mark.parametrize("shape,ring", CASES, ids=["ring", "direct"])
@pytest.mark.parametrize("how", ["reset", "set_density"])
@pytest.mark.parametrize("steps", [3, 37])   # fewer and more than a captured segment
def test_a_run_after_an_odd_number_of_steps_equals_a_fresh_one(shape, ring, how, steps):
    nx, ny, nz = shape
    n = [(1e13 * synth.uniform01(41 + s, nx * ny * nz)).reshape(nz, ny, nx).astype(np.float32) for s in range(2)]
    tr = synth.uniform_tracks(43, 20, nx * DX, ny * DX, 8e-4)
    npk = 40.0 * B.it_peak_density(tr.let_keV_um, tr.b_cm)      # tracks and their images may pile up

    def go(g):
        if how == "reset":
            g.reset()
            g.deposit(tr.x_cm, tr.y_cm, tr.let_keV_um, tr.b_cm)
        else:
            g.set_density(n[0], n[1])
        g.step(steps)
        return _fields(g.tallies()), g.density(0), g.density(1)

    with B.Simulation(nx, ny, nz, DX, V, n_peak_cm3=npk, scheme=B.IT_UPWIND) as g:
        if ring:
            g.set_launch(B.IT_KERNEL_ZMARCH, *ring)
        assert (g.launch()["stages"] > 0) == bool(ring)
        first = go(g)
        second = go(g)      # the first run ended after an odd number of steps
        third = go(g)       # after an even one in all
    assert np.isfinite(first[0]["recombined"]) and first[0]["recombined"] > 0
    for other in (second, third):
        assert other[0] == first[0]
        assert np.array_equal(other[1], first[1]) and np.array_equal(other[2], first[2])
