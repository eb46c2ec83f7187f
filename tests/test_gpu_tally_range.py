"""Tallies of the FP32 marches on dense states: the products n+ n- that a block
or a thread sums add up to more than FP32 holds (3.4e38), while every product
and the 64-bit sum are finite.  One step's tallies against FP64 sums of the
FP32 products, to 1e-12 of the sum of their magnitudes (as the simple kernel's
edge test asks of ordinary states).  With space charge the march without a ring
adds four cells of a narrow section in FP32 first, two roundings deep: 2^-23."""
import numpy as np
import pytest

from paper_1610_06749_gb300 import binding as B
from paper_1610_06749_gb300 import synth

pytestmark = pytest.mark.gpu

MU, ALPHA, Q_OVER_EPS0 = (1.73, 1.87), 1.6e-6, 1.602176634e-19 / 8.8541878128e-14


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1610_06749_gb300 import build
    build.build()
    B.lib()


@pytest.mark.parametrize("shape,kernel", [((301, 17, 9), B.IT_KERNEL_SIMPLE), ((128, 1, 40), B.IT_KERNEL_SIMPLE),
                                          ((128, 1, 300), B.IT_KERNEL_AUTO), ((132, 31, 40), B.IT_KERNEL_AUTO),
                                          ((384, 8, 40), B.IT_KERNEL_ZMARCH)],
                         ids=["simple_301x17x9", "simple_128x1x40", "direct_128x1x300", "direct_132x31x40",
                              "ring_384x8x40"])
@pytest.mark.parametrize("sc", [False, True])
def test_sums_beyond_fp32(shape, kernel, sc):
    nx, ny, nz = shape
    dx, dt, f = 5e-4, 1e-15, np.float32
    n = [(1e18 * (1 + 5 * synth.uniform01(61 + s, nx * ny * nz))).reshape(nz, ny, nx).astype(f) for s in range(2)]
    rr = n[0] * n[1]
    assert np.isfinite(rr).all() and rr.astype(np.float64).sum() > 3.5e38
    with B.Simulation(nx, ny, nz, dx, 200.0, dt_s=dt, scheme=B.IT_UPWIND, kernel=kernel, space_charge=sc) as g:
        if kernel == B.IT_KERNEL_AUTO:
            assert g.launch()["stages"] == 0
        if kernel == B.IT_KERNEL_ZMARCH:
            g.set_launch(kernel, 4, 2, 4, 2)
        g.set_density(n[0], n[1])
        g.step(1)
        t = g.tallies()
    vol, tol = dx ** 3, 2.0 ** -23 if sc and kernel == B.IT_KERNEL_AUTO else 1e-12
    want = rr.astype(np.float64).sum() * float(f(ALPHA * dt)) * vol
    assert abs(t.recombined - want) <= tol * want
    for s in range(2):
        if sc:
            k = float(f(-(1.0 if s == 0 else -1.0) * dt * MU[s] * Q_OVER_EPS0)) * vol
            q = (n[s] * (n[0] - n[1])).astype(np.float64)
            assert abs(t.space_charge[s] - q.sum() * k) <= tol * np.abs(q).sum() * abs(k)
        assert np.isfinite(t.in_domain[s]) and np.isfinite(t.collected_anode[s])
