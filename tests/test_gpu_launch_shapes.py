"""A launch shape given together with the automatic kernel is the shape that
runs, also on grids whose automatic choice is the march without a ring."""
import pytest

from paper_1610_06749_gb300 import binding as B

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1610_06749_gb300 import build
    build.build()
    B.lib()


@pytest.mark.parametrize("asked", [dict(tile_rows=8, ctas_per_sm=2, stages=4), dict(tile_rows=4),
                                   dict(ctas_per_sm=1), dict(stages=5), dict(grid=3)],
                         ids=lambda a: "_".join(f"{k}{v}" for k, v in a.items()))
def test_a_shape_given_with_the_automatic_kernel_is_used(asked):
    # a small grid, where the march without a ring is the automatic choice
    with B.Simulation(64, 48, 40, 5e-4, 200.0) as g, \
            B.Simulation(64, 48, 40, 5e-4, 200.0, kernel=B.IT_KERNEL_ZMARCH) as ring:
        assert g.launch()["stages"] == 0
        g.set_launch(B.IT_KERNEL_AUTO, **asked)
        ring.set_launch(B.IT_KERNEL_ZMARCH, **asked)
        assert g.launch() == ring.launch()
        got = g.launch()
        for k, v in asked.items():
            assert got["ctas" if k == "grid" else k] == v
        g.set_launch(B.IT_KERNEL_AUTO)
        assert g.launch()["stages"] == 0
