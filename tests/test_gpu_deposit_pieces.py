"""Deposits on axes longer than a piece of the weight tables (992 cells) and on
sections of more tiles than a launch has blocks (19456): tracks whose windows
straddle the pieces' ends and the periodic face, windows longer than a piece and
than the axis, against the weights (erf(hi/b) - erf(lo/b))/2 in numpy, cell by
cell to 1e-12 of the largest (some tens of FP64 roundings of 1.1e-16)."""
import numpy as np
import pytest

from paper_1610_06749_gb300 import binding as B

pytestmark = pytest.mark.gpu

DX, W_EV = 5e-4, 34.0


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1610_06749_gb300 import build
    build.build()
    B.lib()


def weights(centre, b, n, periodic):
    from scipy.special import erf
    w, ic = int(np.ceil(6.0 * b / DX)), int(np.floor(centre / DX))
    lo = np.arange(ic - w, ic + w + 1)
    v = 0.5 * (erf(((lo + 1) * DX - centre) / b) - erf((lo * DX - centre) / b))
    out = np.zeros(n)
    keep = slice(None) if periodic else (lo >= 0) & (lo < n)
    np.add.at(out, (lo % n)[keep], v[keep])
    return out


@pytest.mark.parametrize("nx,ny", [(2000, 12), (12, 2000), (991, 993), (992, 1985), (1200, 1200)])
@pytest.mark.parametrize("bc", [B.IT_PERIODIC, B.IT_ABSORBING])
def test_pieces(nx, ny, bc):
    # cells (fractions of a cell included) of the track axes, radii in cells
    cells = [(0.1, 0.2), (nx - 0.01, ny - 0.3), (991.9, 3.3), (992.0, 991.5), (nx / 2, ny / 2), (1984.2, 1984.7),
             (5.5, 992.4)]
    tr = [(x % nx, y % ny, 10.0 + k, r) for k, (x, y) in enumerate(cells) for r in (0.7, 4.0)]
    tr += [(nx / 3, ny / 3, 5.0, 90.0), (nx / 4, ny / 5, 7.0, 400.0)]
    x, y, let, b = (np.array(v) for v in zip(*tr))
    want = np.zeros((ny, nx))
    for k in range(len(x)):
        n0 = let[k] * 1e7 / W_EV
        want += n0 * np.outer(weights(y[k] * DX, b[k] * DX, ny, bc == B.IT_PERIODIC),
                              weights(x[k] * DX, b[k] * DX, nx, bc == B.IT_PERIODIC)) / DX ** 2
    with B.Simulation(nx, ny, 1, DX, 50.0, precision=B.IT_FP64, lateral_bc=bc) as g:
        g.deposit(x * DX, y * DX, let, b * DX)
        got, t = g.density(0)[0], g.tallies()
    assert np.max(np.abs(got - want)) <= 1e-12 * want.max()
    assert np.allclose(t.released, want.sum() * DX ** 3, rtol=1e-12, atol=0)
