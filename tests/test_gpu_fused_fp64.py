"""The fused search in the FP64 mode (FP32 filter, defining FP64 energies of the survivors) against
the per-kernel form, which evaluates every pair in FP64: identical lists bit for bit (states,
energies, stamps, used flags), on grids and on couplings as drawn, where energies that differ by
less than an ulp of E tie; magnitudes the filter covers, and one context whose magnitudes it does
not (the per-kernel form runs then)."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2010_00180_gb300 import build, inputs as I, qis

pytestmark = pytest.mark.gpu
KEYS = ("count", "bits", "E", "stamp", "used")


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    qis.load()


def lists(data, phis, K, R, chunks, flips):
    ctx = qis.Context(K=K, R=R, precision="fp64", max_n=max(len(h) for _, h in data), max_instances=len(data), flips=flips)
    for iid, phi in zip(ctx.create_instances(data), phis):
        ctx.init_states(iid, phi)
    for c in chunks:
        ctx.iterate(c)
    out = [ctx.search_list(k, r) for k in range(len(data)) for r in range(R)]
    out += [ctx.topk_states(k, K + 1) for k in range(len(data))]
    counts = ctx.candidate_count(), ctx.evaluated_pairs(), ctx.iterate(0, count_active=True)
    ctx.close()
    return out, counts


def both(monkeypatch, data, phis, K, R, chunks, flips="single_pair"):
    got = lists(data, phis, K, R, chunks, flips)
    monkeypatch.setenv("QIS_FUSED", "0")
    ref = lists(data, phis, K, R, [sum(chunks)], flips)
    assert got[1] == ref[1]
    for x, y in zip(got[0], ref[0]):
        for key in (k for k in KEYS if k in x):
            assert np.array_equal(x[key], y[key]), key
    return got[0]


@pytest.mark.parametrize("ens,grid,ns,K,R,chunks,flips", [
    ("gaussian", None, [2, 5], 3, 2, [4], "single_pair"),
    ("gaussian", None, [100, 64, 65], 120, 5, [1, 30, 9], "single_pair"),
    ("gaussian", 32, [128, 200], 60, 4, [25], "single_pair"),
    ("pm1", 32, [90, 150], 120, 4, [20], "single_pair"),
    ("uniform", None, [333, 1000], 200, 2, [12], "single_pair"),
    ("gaussian", None, [129, 40], 50, 4, [30], "exchange")])
def test_fused_fp64_equals_per_kernel_form(monkeypatch, ens, grid, ns, K, R, chunks, flips):
    data = [I.instance(ens, n, seed=820, inst=k, grid_bits=grid) for k, n in enumerate(ns)]
    phis = [I.random_states(n, R, seed=821, inst=k) for k, n in enumerate(ns)]
    got = both(monkeypatch, data, phis, K, R, chunks, flips)
    J, h = data[0]
    ref = O.qi_search(J, h, K, sum(chunks), phis[0][0], flips={"single_pair": 0, "exchange": 2}[flips])
    for key in KEYS[1:]:
        assert np.array_equal(got[0][key], ref[key][: ref["count"]]), key


@pytest.mark.parametrize("js,hs", [(2.0 ** -58, 2.0 ** -58), (2.0 ** 54, 1.0), (1e-9, 2.0 ** 40), (1.0, 1e17),
                                   (1e-30, 1e-30), (1e25, 1.0)])
def test_fused_fp64_magnitudes(monkeypatch, js, hs):
    """Couplings and fields scaled apart (a large common energy makes many energies tie by rounding);
    the last two lie outside the filter's range."""
    n, K, R = 70, 40, 3
    J, h = I.instance("gaussian", n, seed=822, grid_bits=None)
    both(monkeypatch, [(J * js, h * hs)], [I.random_states(n, R, seed=823)], K, R, [15])
