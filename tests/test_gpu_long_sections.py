"""Deposits on sections with more rows than a launch grid has blocks in y
(65535): the released charge of one track is its ions per cm times the gap."""
import numpy as np
import pytest

from paper_1610_06749_gb300 import binding as B

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1610_06749_gb300 import build
    build.build()
    B.lib()


@pytest.mark.parametrize("nx,ny", [(1, 524_289), (1, 700_001), (700_001, 1)])
def test_one_track_on_a_long_section(nx, ny):
    dx, nz, let, b = 5e-4, 2, 10.0, 2e-3
    # away from the ends, whose images would share the window
    at = dx * (0.5 * np.array([nx, ny]) + 0.25)
    with B.Simulation(nx, ny, nz, dx, 50.0, precision=B.IT_FP64) as g:
        g.deposit([at[0]], [at[1]], [let], [b])
        t = g.tallies()
        p = g.density(0)
    want = let * 1e7 / 34.0 * nz * dx
    # the window cuts the profile at 6 b (2e-17); sums of some hundred cells in 64 bits
    assert np.allclose(t.released, want, rtol=1e-12, atol=0)
    # the cells add up to it too, and the peak lies in the track's cell
    assert np.isclose(p.sum() * dx ** 3, want, rtol=1e-12, atol=0)
    assert np.unravel_index(np.argmax(p[0]), (ny, nx)) == (ny // 2, nx // 2)
