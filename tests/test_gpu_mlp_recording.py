"""Training where the step cannot be recorded (made to fail by a hook, after the
step has been captured): the call goes on with single launches and gives the
same weights and losses, and the network records again afterwards."""
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


@pytest.mark.parametrize("samples,batch,epochs", [(160, 16, 2), (300, 64, 5)])
def test_a_step_that_cannot_be_recorded(samples, batch, epochs):
    members = 2
    theta = synth.mlp_init(81, members)
    u = synth.uniform01(83, 7 * samples).reshape(samples, 7)
    X, y = 2.0 * u[:, :6] - 1.0, 0.05 + 0.9 * u[:, 6]
    h = B.it_mlp_create(members, batch)
    try:
        B.it_mlp_set_data(h, X, y)
        res = []
        for refuse in (False, True, False):
            for m in range(members):
                B.it_mlp_set_params(h, m, theta[m])
            B.it_test_refuse_recording(h, refuse)
            loss = B.it_mlp_train(h, epochs, batch, 1e-3, 9)
            res.append((loss, [B.it_mlp_get_params(h, m) for m in range(members)]))
    finally:
        B.it_mlp_destroy(h)
    for loss, p in res[1:]:
        assert np.isfinite(loss).all() and np.array_equal(loss, res[0][0])
        assert all(np.array_equal(a, b) for a, b in zip(p, res[0][1]))
