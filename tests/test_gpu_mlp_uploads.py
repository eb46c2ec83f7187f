"""Training over epochs that are not waited for: the sample orders and Adam's
corrections of an epoch are uploaded while earlier epochs still run, from host
memory that must not change before it has been read.  With the losses asked
for, every epoch is waited for; the weights are bitwise the same without."""
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


# sample orders of 0.4 and 1.6 MB an epoch; a short epoch that the host runs ahead of; no recorded step
@pytest.mark.parametrize("members,samples,batch,epochs", [(5, 20_000, 512, 7), (4, 100_000, 4096, 5), (2, 64, 32, 40),
                                                          (3, 50, 64, 7)])
def test_epochs_in_flight(members, samples, batch, epochs):
    theta = synth.mlp_init(71, members)
    u = synth.uniform01(73, 7 * samples).reshape(samples, 7)
    X, y = 2.0 * u[:, :6] - 1.0, 0.05 + 0.9 * u[:, 6]
    res = []
    for wait in (True, False):
        h = B.it_mlp_create(members, batch)
        try:
            for m in range(members):
                B.it_mlp_set_params(h, m, theta[m])
            B.it_mlp_set_data(h, X, y)
            if wait:
                loss = B.it_mlp_train(h, epochs, batch, 1e-3, 5)
                assert np.isfinite(loss).all() and (loss > 0).all()
            else:
                assert B.lib().it_mlp_train(h, epochs, batch, 1e-3, 5, None) == B.IT_OK
            res.append([B.it_mlp_get_params(h, m) for m in range(members)])
        finally:
            B.it_mlp_destroy(h)
    for a, b in zip(*res):
        assert np.isfinite(a).all() and np.array_equal(a, b)
