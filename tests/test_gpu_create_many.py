"""More instances in one creation call than a grid's second dimension counts."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2010_00180_gb300 import build, inputs as I, qis

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    qis.load()


@pytest.mark.parametrize("precision", ["fp64", "split_bf16"])
def test_seventy_thousand_instances(precision):
    cnt, n = 70000, 2
    rng = np.random.default_rng(895)
    c, h = np.round(rng.normal(size=cnt) * 2 ** 20) / 2 ** 20, np.round(rng.normal(size=(cnt, n)) * 2 ** 20) / 2 ** 20
    J = np.zeros((cnt, n, n))
    J[:, 0, 1] = J[:, 1, 0] = c
    ctx = qis.Context(K=3, R=1, precision=precision, max_n=n, max_instances=cnt)
    ids = ctx.create_instances(list(zip(J, h)))
    psi0 = np.zeros((1, 1), np.uint64)
    for i in ids:
        ctx.init_states(i, psi0)
    ctx.iterate(3)
    for i in (0, 65534, 65535, 65536, cnt - 1):
        ref = O.qi_search(J[i], h[i], 3, 3, psi0[0])
        got = ctx.search_list(i, 0)
        for key in ("bits", "E", "stamp", "used"):
            assert np.array_equal(got[key], ref[key][: ref["count"]]), (i, key)
    ctx.close()
