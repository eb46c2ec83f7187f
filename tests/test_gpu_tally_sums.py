"""Tallies of sections wider than 256 cells (and no multiple of it), on every
form of the staged march and on the march without a ring: FP32 terms summed as
closely as FP64 would, to 1e-12 of the sum of their magnitudes.  The terms are
those of the state before each step (n+ n-, n (n+ - n-), the densities of the
electrode planes and absorbing sides), rounded to FP32 once where they are
products.  The sums carry the rounding error of each addition along, so what is
left is 2^-48 per addition of the at most some hundred additions of a thread."""
import numpy as np
import pytest

from paper_1610_06749_gb300 import binding as B
from paper_1610_06749_gb300 import synth

pytestmark = pytest.mark.gpu

MU, D, ALPHA, Q_OVER_EPS0 = (1.73, 1.87), (0.037, 0.037), 1.6e-6, 1.602176634e-19 / 8.8541878128e-14
# nx, ny, nz, launch shape (rows, CTAs per SM, ring depth, grid; None: the automatic choice), float4 per thread
SHAPES = [(384, 40, 24, None, 0), (260, 6, 40, (2, 1, 4, 0), 1), (384, 8, 40, (4, 1, 4, 2), 1),
          (384, 8, 70, (4, 2, 4, 2), 2), (320, 9, 35, (9, 1, 3, 0), 2), (320, 9, 35, (9, 2, 3, 1), 3),
          (384, 16, 4, (16, 1, 3, 2), 3), (288, 12, 40, (12, 2, 3, 1), 4), (320, 9, 1, (3, 2, 4, 0), 1)]


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1610_06749_gb300 import build
    build.build()
    B.lib()


def terms(n, nz, dx, V, dt, absorbing, sc):
    """(sum, sum of magnitudes) of every tally of one upwind step of the FP32 densities n."""
    f, E, vol = np.float32, V / (nz * dx), dx * dx * dx
    out = {"rec": [(n[0] * n[1]).astype(np.float64), float(f(ALPHA * dt)) * vol]}
    for s in range(2):
        c, sd = MU[s] * E * dt / dx, D[s] * dt / (dx * dx)
        wzm, wzp = f(sd + (c if s == 0 else 0.0)), f(sd + (0.0 if s == 0 else c))
        d = n[s].astype(np.float64)
        out[f"an{s}"], out[f"ca{s}"] = [d[0], float(wzp) * vol], [d[-1], float(wzm) * vol]
        if absorbing:
            out[f"lat{s}"] = [np.concatenate([x.ravel() for x in (d[:, :, 0], d[:, :, -1], d[:, 0], d[:, -1])]),
                              float(f(sd)) * vol]
        if sc:
            k = f(-(1.0 if s == 0 else -1.0) * dt * MU[s] * Q_OVER_EPS0)
            out[f"sc{s}"] = [(n[s] * (n[0] - n[1])).astype(np.float64), float(k) * vol]
    return {k: (x.sum() * w, np.abs(x).sum() * abs(w)) for k, (x, w) in out.items()}


@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "x".join(map(str, s[:3])) + "_" + str(s[4]))
@pytest.mark.parametrize("lat", [B.IT_PERIODIC, B.IT_ABSORBING])
@pytest.mark.parametrize("sc", [False, True])
def test_wide_sections_sum_as_fp64_does(shape, lat, sc):
    nx, ny, nz, launch, ipt = shape
    dx, V = 5e-4, 200.0
    n = [(1e13 * synth.uniform01(67 + s, nx * ny * nz)).reshape(nz, ny, nx).astype(np.float32) for s in range(2)]
    p = B.it_params_default(gap_cm=nz * dx, voltage_V=V, scheme=B.IT_UPWIND, n_peak_cm3=1e13, space_charge=int(sc))
    dt = 0.5 * B.it_auto_dt(p, dx)
    want = {}
    with B.Simulation(nx, ny, nz, dx, V, dt_s=dt, lateral_bc=lat, scheme=B.IT_UPWIND, space_charge=sc) as g:
        if launch:
            assert -(-(nx // 4) * launch[0] // (512 if launch[1] == 1 else 256)) == ipt
            g.set_launch(B.IT_KERNEL_ZMARCH, *launch)
        assert (g.launch()["stages"] >= 3) == bool(launch)
        g.set_density(n[0], n[1])
        for _ in range(2):          # up and down
            for k, (x, m) in terms(n, nz, dx, V, dt, lat == B.IT_ABSORBING, sc).items():
                a, b = want.get(k, (0.0, 0.0))
                want[k] = (a + x, b + m)
            g.step(1)
            n = [g.density(0), g.density(1)]
        t = g.tallies()
    got = {"rec": t.recombined}
    for s in range(2):
        got[f"an{s}"], got[f"ca{s}"] = t.collected_anode[s], t.collected_cathode[s]
        got[f"lat{s}"], got[f"sc{s}"] = t.lost_lateral[s], t.space_charge[s]
    for k, x in got.items():
        a, m = want.get(k, (0.0, 0.0))
        assert abs(x - a) <= 1e-12 * m, (k, abs(x - a) / m if m else x)
