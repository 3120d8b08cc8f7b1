"""Edges of the fused search's rules.

More survivors than the buffer holds: the iteration is run again with a bound from the survivors at
hand. The instances hold a state (two flips from psi0 and close to it in energy) that a list which has
settled picks as its parent late, and from which every further site lowers the energy, so that the
last kept energy lets through all pairs at once.

The block size: 256 threads while every search's block is resident at once, 128 beyond that and for
small instances; equal lists on both sides of the line."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2010_00180_gb300 import build, inputs as I, qis

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    qis.load()


def hidden_descent(n):
    J = np.zeros((n, n))
    J[0, 1] = -2.5
    J[0, 6:] = J[1, 6:] = -1.0
    J = J + J.T
    rng = np.random.default_rng(830)
    a = np.concatenate([[5.0, 5.0390625], np.arange(1, 5) / 64.0, 6.0 + rng.integers(0, 1024, n - 6) / 1024.0])
    return J, -a / 2 - J.sum(axis=1)   # a_i: the change of energy when spin i of the all-up state is flipped


@pytest.mark.parametrize("precision", ["split_bf16", "fp64"])
@pytest.mark.parametrize("n,K,cap", [(60, 8, 100), (200, 8, 100), (300, 8, 0), (200, 20, 148)])
def test_settled_list_meets_many_survivors(precision, n, K, cap):
    J, h = hidden_descent(n)
    phi = I.pack_bits(np.zeros((1, n)))
    ctx = qis.Context(K=K, R=1, precision=precision, max_n=n, max_instances=1, survivor_cap=cap)
    iid = ctx.create_instance(J, h)
    ctx.init_states(iid, phi)
    ctx.iterate(40)
    got = ctx.search_list(0, 0)
    ctx.close()
    ref = O.qi_search(J, h, K, 40, phi[0])
    assert got["count"] == ref["count"]
    for key in ("bits", "E", "stamp", "used"):
        assert np.array_equal(got[key], ref[key][: ref["count"]]), key


@pytest.mark.parametrize("precision,flips,n,K", [("split_bf16", "single_pair", 150, 20), ("split_bf16", "single_pair", 128, 20),
                                                 ("split_bf16", "exchange", 130, 9), ("fp64", "single_pair", 40, 12),
                                                 ("fp64", "exchange", 33, 12)])
def test_block_size_line(precision, flips, n, K):
    torch = pytest.importorskip("torch")
    line = 4 * torch.cuda.get_device_properties(0).multi_processor_count
    J, h = I.instance("gaussian", n, seed=831)
    phi = I.random_states(n, line + 1, seed=832)
    lists = []
    for R in (line, line + 1):
        ctx = qis.Context(K=K, R=R, precision=precision, max_n=n, max_instances=1, flips=flips)
        ctx.create_instance(J, h)
        ctx.init_states(0, phi[:R])
        ctx.iterate(12)
        lists.append([ctx.search_list(0, r) for r in range(line)])
        ctx.close()
    for x, y in zip(*lists):
        assert all(np.array_equal(x[key], y[key]) for key in ("bits", "E", "stamp", "used"))
    for r in (0, line - 1):
        ref = O.qi_search(J, h, K, 12, phi[r], flips={"single_pair": 0, "exchange": 2}[flips])
        for key in ("bits", "E", "stamp", "used"):
            assert np.array_equal(lists[0][r][key], ref[key][: ref["count"]]), key
