"""The z-march without a shared-memory ring (chosen for small grids) against
the TMA-staged one, bitwise, where its work split can go wrong: one segment,
one row, one plane, rows shorter and longer than a warp, segments just below
and above a block of 128, more planes than chunks, both faces, the
space-charge term.  Tallies are compared to 1e-6 of the released charge: both
kernels sum FP32 terms, the staged one up to 32 planes in plain FP32."""
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


@pytest.mark.parametrize("shape", [(4, 1, 1), (4, 3, 70), (8, 64, 1), (36, 20, 23), (124, 33, 5), (128, 4, 9),
                                   (132, 31, 40), (256, 2, 3), (384, 40, 24), (512, 5, 17)],
                         ids=lambda s: "x".join(map(str, s)))
@pytest.mark.parametrize("lat", [B.IT_PERIODIC, B.IT_ABSORBING])
@pytest.mark.parametrize("sc", [False, True])
def test_direct_march_equals_the_staged_one(shape, lat, sc):
    nx, ny, nz = shape
    dx, V = 5e-4, 200.0
    n = [(1e13 * synth.uniform01(11 + s, nx * ny * nz)).reshape(nz, ny, nx).astype(np.float32) for s in range(2)]
    res = []
    for kernel in (B.IT_KERNEL_AUTO, B.IT_KERNEL_ZMARCH):
        with B.Simulation(nx, ny, nz, dx, V, lateral_bc=lat, scheme=B.IT_UPWIND, kernel=kernel, space_charge=sc,
                          n_peak_cm3=2e13) as g:
            g.set_density(n[0], n[1])
            g.step(5)
            res.append((g.density(0), g.density(1), g.tallies(), g.launch()))
    (p0, m0, t0, l0), (p1, m1, t1, l1) = res
    assert l0["kernel"] == l1["kernel"] == B.IT_KERNEL_ZMARCH
    assert l0["stages"] == 0 and l1["stages"] >= 3
    assert np.array_equal(p0, p1) and np.array_equal(m0, m1)
    tol = 1e-6 * t1.released.sum()
    assert abs(t0.recombined - t1.recombined) <= tol
    for name in ("collected_anode", "collected_cathode", "lost_lateral", "in_domain", "space_charge"):
        assert np.max(np.abs(getattr(t0, name) - getattr(t1, name))) <= tol, name
