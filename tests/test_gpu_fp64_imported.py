"""FP64 searches that continue from imported lists whose energies, taken as given, are far larger than
any change of energy, so that many candidates round to one energy and the lowest by index enter: the
fused search against the per-kernel form, which decides every candidate in FP64, bit for bit."""
import numpy as np
import pytest

from paper_2010_00180_gb300 import build, inputs as I, qis

pytestmark = pytest.mark.gpu
KEYS = ("count", "bits", "E", "stamp", "used")


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    qis.load()


@pytest.mark.parametrize("flips,n", [("single_pair", 40), ("single_pair", 100), ("exchange", 60)])
@pytest.mark.parametrize("offset", [0.0, 3e9, 1e13, -1e15, 1e15, 1e18, -1e300])
@pytest.mark.parametrize("full", [False, True])
def test_lists_with_large_energies(monkeypatch, flips, n, offset, full):
    K = 30
    J, h = I.instance("gaussian", n, seed=860, grid_bits=None)
    s0 = np.zeros(n, np.uint8)
    s0[: n // 2] = 1
    states = [s0]
    for i in range(K if full else 0):   # exchanges of one pair: near states under either flip set
        s = s0.copy()
        s[[i % (n // 2), n - 1 - i // (n // 2)]] ^= 1
        states.append(s)
    S = 1.0 - 2.0 * np.array(states).astype(np.float64)
    E = 0.5 * np.einsum("ki,ij,kj->k", S, J, S) + S @ h + offset
    o = np.argsort(E, kind="stable")
    bits = I.pack_bits(np.array(states)[o])
    out = []
    for fused in ("1", "0"):
        monkeypatch.setenv("QIS_FUSED", fused)
        ctx = qis.Context(K=K, R=1, precision="fp64", max_n=n, flips=flips, survivor_cap=8192)
        ctx.create_instance(J, h)
        ctx.init_states(0, bits[:1])
        ctx.set_search_list(0, 0, bits, E[o])
        ctx.iterate(1)
        ctx.iterate(7)
        out.append(ctx.search_list(0, 0))
        ctx.close()
    for key in KEYS:
        assert np.array_equal(out[0][key], out[1][key]), key


def test_no_candidate_below_the_last_energy_and_a_small_buffer(monkeypatch):
    """Every candidate passes the filter, none is below the last kept energy in FP64."""
    n, K = 100, 30
    J, h = I.instance("gaussian", n, seed=861, grid_bits=None)
    states = np.zeros((K + 1, n), np.uint8)
    states[np.arange(1, K + 1), np.arange(K)] = 1
    bits = I.pack_bits(states)
    out = []
    for fused in ("1", "0"):
        monkeypatch.setenv("QIS_FUSED", fused)
        ctx = qis.Context(K=K, R=1, precision="fp64", max_n=n, survivor_cap=188)
        ctx.create_instance(J, h)
        ctx.init_states(0, bits[:1])
        ctx.set_search_list(0, 0, bits, np.full(K + 1, 1e300))
        ctx.iterate(5)
        out.append(ctx.search_list(0, 0))
        ctx.close()
    for key in KEYS:
        assert np.array_equal(out[0][key], out[1][key]), key
