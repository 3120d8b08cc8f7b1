"""Single-flip searches with far more sites tied at the bound of the lowest changes of energy than the
survivor buffer holds: those that cannot enter a full list take no place in it; an error is left only
where more than the buffer holds can enter."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2010_00180_gb300 import build, inputs as I, qis

pytestmark = pytest.mark.gpu
KEYS = ("bits", "E", "stamp", "used")


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    qis.load()


def fields_only(n, low, tied):
    """Changes of energy from the state of all spins up: `low` sites with distinct small negative ones,
    n - low sites with `tied`."""
    a = np.full(n, tied)
    a[:low] = -np.arange(1, low + 1) / 16.0
    return np.zeros((n, n)), -a / 2


def search(J, h, K, cap, iters, psi0):
    ctx = qis.Context(K=K, R=1, precision="split_bf16", max_n=len(h), flips="single", survivor_cap=cap)
    ctx.create_instance(J, h)
    ctx.init_states(0, psi0)
    ctx.iterate(iters)
    out = ctx.search_list(0, 0)
    ctx.close()
    return out


# (n, K, sites below the tie, buffer, the tie): more ties than the block's 512 places or fewer, more than the
# default buffer of 2048, K+1 near what the buckets rank at once; 0.5: some equal the last kept energy
@pytest.mark.parametrize("n,K,low,cap,tied", [(300, 8, 10, 100, 8.0), (300, 8, 10, 100, 0.5), (900, 8, 9, 100, 8.0),
                                              (900, 8, 9, 100, 0.5), (1200, 200, 202, 868, 40.0), (3000, 120, 122, 0, 8.0)])
def test_ties_that_cannot_enter(n, K, low, cap, tied):
    J, h = fields_only(n, low, tied)
    psi0 = np.zeros((1, (n + 63) // 64), np.uint64)
    got = search(J, h, K, cap, 12, psi0)
    ref = O.qi_search(J, h, K, 12, psi0[0], flips=1)
    for key in KEYS:
        assert np.array_equal(got[key], ref[key][: ref["count"]]), key


def test_ties_that_can_enter_are_still_an_error():
    n, K = 300, 8
    J, h = fields_only(n, 4, -0.0625)   # 297 equal sites below the state's own energy, a list of one
    with pytest.raises(qis.QISError) as e:
        search(J, h, K, 100, 3, np.zeros((1, (n + 63) // 64), np.uint64))
    assert e.value.name == "CAPACITY"
