"""The TMA-staged z-march against the simple kernel, bitwise, over the forms
its launch shapes select: one to four float4 per thread (as vertical pairs or
not), one and two CTAs per SM, ring depths from 3 to 16, rows wider than a TMA
box, one CTA that walks many short segments, one plane, odd step counts (steps
alternate between marching up and down).  Tallies are compared to 1e-6 of the
released charge: the staged march sums up to 32 planes in plain FP32."""
import numpy as np
import pytest

from paper_1610_06749_gb300 import binding as B
from paper_1610_06749_gb300 import synth

pytestmark = pytest.mark.gpu

# nx, ny, nz, (tile rows, CTAs per SM, ring depth, grid), float4 per thread
SHAPES = [(64, 24, 9, (4, 2, 4, 0), 1), (36, 10, 7, (5, 1, 3, -1), 1), (256, 16, 9, (8, 2, 4, 0), 2),
          (256, 16, 9, (16, 1, 5, -1), 2), (200, 20, 5, (10, 2, 3, 3), 2), (200, 14, 6, (7, 2, 4, 2), 2),
          (128, 24, 5, (24, 2, 4, 1), 3), (384, 16, 4, (16, 1, 3, 2), 3), (256, 32, 6, (16, 2, 3, 2), 4),
          (256, 26, 6, (13, 2, 3, 0), 4), (512, 8, 5, (8, 1, 4, 3), 2), (32, 40, 3, (2, 2, 16, 1), 1),
          (32, 40, 3, (1, 1, 8, 2), 1), (256, 16, 1, (8, 2, 4, 1), 2), (200, 10, 40, (10, 2, 4, 3), 2)]


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1610_06749_gb300 import build
    build.build()
    B.lib()


@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "x".join(map(str, s[:3])) + "_" + "_".join(map(str, s[3])))
@pytest.mark.parametrize("lat", [B.IT_PERIODIC, B.IT_ABSORBING])
@pytest.mark.parametrize("sc", [False, True])
def test_staged_march_equals_the_simple_kernel(shape, lat, sc):
    nx, ny, nz, launch, ipt = shape
    assert -(-(nx // 4) * launch[0] // (512 if launch[1] == 1 else 256)) == ipt
    dx, V = 5e-4, 200.0
    n = [(1e13 * synth.uniform01(17 + s, nx * ny * nz)).reshape(nz, ny, nx).astype(np.float32) for s in range(2)]
    res = []
    for kernel in (B.IT_KERNEL_ZMARCH, B.IT_KERNEL_SIMPLE):
        with B.Simulation(nx, ny, nz, dx, V, lateral_bc=lat, scheme=B.IT_UPWIND, kernel=kernel, space_charge=sc,
                          n_peak_cm3=2e13) as g:
            if kernel == B.IT_KERNEL_ZMARCH:
                g.set_launch(kernel, *launch)
            g.set_density(n[0], n[1])
            a = []
            for steps in (1, 4):
                g.step(steps)
                a += [g.density(0), g.density(1)]
            res.append((a, g.tallies()))
    (a0, t0), (a1, t1) = res
    for x, y in zip(a0, a1):
        assert np.array_equal(x, y)
    tol = 1e-6 * t1.released.sum()
    assert abs(t0.recombined - t1.recombined) <= tol
    for name in ("collected_anode", "collected_cathode", "lost_lateral", "in_domain", "space_charge"):
        assert np.max(np.abs(getattr(t0, name) - getattr(t1, name))) <= tol, name
