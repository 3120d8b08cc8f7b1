"""Energies of given states and a device-side wait that runs out (the wait probe with a short bound): the
call that waited reports it, the context stays usable, and a search that timed out earlier does not stand
in the way of energies, which do not depend on it."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2010_00180_gb300 import build, inputs as I, qis

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    qis.load()


@pytest.mark.parametrize("precision", ["split_bf16", "fp64"])
@pytest.mark.parametrize("n,count", [(16, 3), (200, 300), (1100, 130)])   # one block per state, and several
def test_energies_report_a_wait_that_ran_out(precision, n, count):
    J, h = I.instance("gaussian", n, seed=875, grid_bits=20)
    bits = I.random_states(n, count, seed=876)
    ctx = qis.Context(K=4, R=2, precision=precision, max_n=n)
    ctx.create_instance(J, h)
    E = ctx.energies(0, bits)
    ctx.set_wait_limit(1_000_000, probe=True)
    with pytest.raises(qis.QISError) as e:
        ctx.energies(0, bits)
    assert e.value.name == "DEVICE_TIMEOUT"
    ctx.set_wait_limit(2_000_000_000, probe=False)
    assert np.array_equal(ctx.energies(0, bits), E)
    ctx.init_states(0, bits[:2])   # and searches run as if nothing had been
    ctx.iterate(5)
    ref = O.qi_search(J, h, 4, 5, bits[0])
    assert np.array_equal(ctx.search_list(0, 0)["E"], ref["E"][: ref["count"]])
    ctx.close()


def test_energies_after_a_search_that_timed_out():
    n, R = 200, 8
    J, h = I.instance("gaussian", n, seed=877)
    bits = I.random_states(n, R, seed=878)
    ctx = qis.Context(K=20, R=R, precision="split_bf16", max_n=n)
    ctx.create_instance(J, h)
    E = ctx.energies(0, bits)
    ctx.init_states(0, bits)
    ctx.set_wait_limit(1_000_000, probe=True)
    ctx.iterate(1)
    with pytest.raises(qis.QISError):
        ctx.synchronize()
    ctx.set_wait_limit(2_000_000_000, probe=False)
    assert np.array_equal(ctx.energies(0, bits), E)
    with pytest.raises(qis.QISError):   # the searches stay undefined until they are restarted
        ctx.synchronize()
    ctx.close()
