"""Energies of given states do not read the bits above n of a state's last word."""
import numpy as np
import pytest

from paper_2010_00180_gb300 import build, inputs as I, qis

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    qis.load()


@pytest.mark.parametrize("precision", ["split_bf16", "fp64"])
@pytest.mark.parametrize("n", [2, 63, 65, 100, 127, 129])
def test_bits_above_n_are_ignored(precision, n):
    J, h = I.instance("gaussian", n, seed=870)
    bits = I.random_states(n, 5, seed=871)
    stray = bits.copy()
    stray[:, -1] |= np.uint64((1 << 64) - (1 << (n % 64)))
    ctx = qis.Context(K=1, R=1, precision=precision, max_n=n)
    ctx.create_instance(J, h)
    assert np.array_equal(ctx.energies(0, stray), ctx.energies(0, bits))
    ctx.close()
