"""The simple step kernel at the edges of its work split -- one column, one
plane, columns just below and above a block of 128, more chunks than planes,
every face, the space-charge term, both types -- against a restatement of the
update in numpy.

Densities are compared bitwise: the restatement rounds each operation as the
kernel does (a fused multiply-add as one rounding of the quad-precision
result).  Tallies are compared with FP64 sums of the restated terms, to
1e-12 of the sum of their magnitudes: the kernel's FP32 sums carry their
rounding errors along and keep about 46 bits (2^-46 = 1.4e-14 per addition).
"""
import numpy as np
import pytest

from paper_1610_06749_gb300 import binding as B
from paper_1610_06749_gb300 import synth

pytestmark = pytest.mark.gpu

SHAPES = [(1, 1, 1), (1, 1, 37), (2, 1, 5), (127, 1, 3), (128, 1, 2), (129, 1, 40), (5, 3, 1), (31, 33, 65),
          (43, 6, 400), (301, 17, 9)]
MU, D, ALPHA = (1.73, 1.87), (0.037, 0.037), 1.6e-6
Q_OVER_EPS0 = 1.602176634e-19 / 8.8541878128e-14
Q = np.longdouble


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1610_06749_gb300 import build
    build.build()
    B.lib()


def fma(a, b, c, T):
    return (Q(a) * Q(b) + Q(c)).astype(T)


def side(n, axis, step, periodic):
    out = np.roll(n, step, axis)
    if not periodic:
        at = [slice(None)] * 3
        at[axis] = 0 if step > 0 else -1
        out[tuple(at)] = 0
    return out


def restated_step(n, nz, dx, V, dt, T, periodic, sc):
    """(next densities, tallies, magnitudes) of one upwind step."""
    E, vol = V / (nz * dx), dx * dx * dx
    P, M = n
    rr = P * M
    adt = T(ALPHA * dt)
    tal = {"rec": [rr.astype(np.float64), float(adt) * vol]}
    new = []
    for s in range(2):
        c, sd = MU[s] * E * dt / dx, D[s] * dt / (dx * dx)
        wzm, wzp = T(sd + (c if s == 0 else 0.0)), T(sd + (0.0 if s == 0 else c))
        wd, a = T(sd), n[s]
        s4 = (side(a, 2, 1, periodic) + side(a, 2, -1, periodic)) + (side(a, 1, 1, periodic) + side(a, 1, -1, periodic))
        v = wd * fma(T(-4), a, s4, T)
        v = fma(wzm, side(a, 0, 1, False) - a, v, T)
        v = fma(wzp, side(a, 0, -1, False) - a, v, T)
        v = fma(-adt, rr, v, T)
        v = a + v
        d = a.astype(np.float64)
        if sc:
            k = T(-(1.0 if s == 0 else -1.0) * dt * MU[s] * Q_OVER_EPS0)
            t = a * (P - M)
            v = fma(k, t, v, T)
            tal[f"sc{s}"] = [t.astype(np.float64), float(k) * vol]
        tal[f"an{s}"], tal[f"ca{s}"] = [d[0], float(wzp) * vol], [d[-1], float(wzm) * vol]
        if not periodic:
            tal[f"lat{s}"] = [np.concatenate([x.ravel() for x in (d[:, :, 0], d[:, :, -1], d[:, 0], d[:, -1])]),
                              float(wd) * vol]
        new.append(v.astype(T))
    return new, {k: (x.sum() * f, np.abs(x).sum() * abs(f)) for k, (x, f) in tal.items()}


@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "x".join(map(str, s)))
@pytest.mark.parametrize("prec", [B.IT_FP32, B.IT_FP64])
@pytest.mark.parametrize("lat", [B.IT_PERIODIC, B.IT_ABSORBING])
@pytest.mark.parametrize("sc", [False, True])
def test_simple_step_edges_match_the_restated_update(shape, prec, lat, sc):
    if prec == B.IT_FP64 and np.finfo(Q).nmant < 112:
        pytest.skip("needs a quad-precision long double to restate a double fma")
    nx, ny, nz = shape
    T = np.float64 if prec == B.IT_FP64 else np.float32
    dx, V = 5e-4, 200.0
    n = [(1e13 * synth.uniform01(7 + s, nx * ny * nz)).reshape(nz, ny, nx).astype(T) for s in range(2)]
    p = B.it_params_default(gap_cm=nz * dx, voltage_V=V, scheme=B.IT_UPWIND, n_peak_cm3=1e13, space_charge=int(sc))
    dt = 0.5 * B.it_auto_dt(p, dx)
    want = {}
    with B.Simulation(nx, ny, nz, dx, V, dt_s=dt, precision=prec, lateral_bc=lat, scheme=B.IT_UPWIND,
                      kernel=B.IT_KERNEL_SIMPLE, space_charge=sc) as g:
        g.set_density(n[0], n[1])
        for _ in range(2):
            g.step(1)
            n, tal = restated_step(n, nz, dx, V, dt, T, lat == B.IT_PERIODIC, sc)
            for s in range(2):
                assert np.array_equal(g.density(s), n[s]), s
            for k, (x, m) in tal.items():
                a, b = want.get(k, (0.0, 0.0))
                want[k] = (a + x, b + m)
        t = g.tallies()
    got = {"rec": t.recombined}
    for s in range(2):
        got[f"an{s}"], got[f"ca{s}"] = t.collected_anode[s], t.collected_cathode[s]
        got[f"lat{s}"], got[f"sc{s}"] = t.lost_lateral[s], t.space_charge[s]
    for k, x in got.items():
        a, m = want.get(k, (0.0, 0.0))
        assert abs(x - a) <= 1e-12 * m, k
