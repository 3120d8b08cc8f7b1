"""Network passes whose activations in shared memory come to 48 KiB exactly (a width of 384 with 16 rows
per block, of 768 with 8): the logits' bits are those of smaller batches."""
import numpy as np
import pytest

from paper_2010_00180_gb300 import build, qis

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    qis.load()


@pytest.mark.parametrize("hidden,rows", [(384, 4000), (768, 2000), (400, 4000)])
def test_logits_do_not_depend_on_the_tile(hidden, rows):
    X = np.random.default_rng(880).normal(size=(rows, qis.MLP.N_FEATURES)).astype(np.float32)
    net = qis.MLP(hidden=hidden, max_sites=1, batch=rows, max_n=2, seed=hidden)
    z = net.forward(X)
    for r in (0, 1000, rows - 250):
        assert np.array_equal(z[r: r + 250], net.forward(X[r: r + 250]))
    net.loss_grad(X, (z > 0).astype(np.float32))
    net.close()
