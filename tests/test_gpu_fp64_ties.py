"""FP64 searches in which far more candidates than the survivor buffer holds have the changes of energy
of the last kept state, equal to it or apart by less than the FP32 filter resolves: the fused search
against the per-kernel form, whose test E' < T leaves few of them, bit for bit."""
import numpy as np
import pytest

from paper_2010_00180_gb300 import build, inputs as I, qis

pytestmark = pytest.mark.gpu
KEYS = ("count", "bits", "E", "stamp", "used")


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    qis.load()


def crowded(flips, noise):
    """Fields only: n sites whose flips cost 4 (exchanges: 2 each), or that and some 1e-9 more; the list
    is the state and K of its neighbours, unused."""
    n, K = (300, 8) if flips == "single_pair" else (40, 8)
    rng = np.random.default_rng(850)
    a = np.full(n, 4.0 if flips == "single_pair" else 2.0) + (1e-9 * rng.random(n) if noise else 0.0)
    s0 = np.zeros(n, np.uint8)
    if flips == "exchange":
        s0[: n // 2] = 1
    S = 1.0 - 2.0 * s0
    h = -a * S / 2
    if flips == "single_pair":
        near = [(i,) for i in np.argsort(a, kind="stable")[n // 2: n // 2 + K]]
    else:
        near = [(i, n - 1 - i) for i in range(K)]
    states = [s0]
    for f in near:
        s = s0.copy()
        s[list(f)] ^= 1
        states.append(s)
    E = np.array([float(np.sum(h * S))] + [float(np.sum(h * S)) + sum(a[list(f)]) for f in near])
    o = np.argsort(E, kind="stable")
    return n, K, h, np.array(states)[o], E[o]


@pytest.mark.parametrize("flips", ["single_pair", "exchange"])
@pytest.mark.parametrize("noise", [False, True])
@pytest.mark.parametrize("R", [1, 700])   # blocks of 256 and of 128 threads
def test_ties_at_the_last_kept_energy(monkeypatch, flips, noise, R):
    n, K, h, states, E = crowded(flips, noise)
    bits = I.pack_bits(states)
    out = []
    for fused in ("1", "0"):
        monkeypatch.setenv("QIS_FUSED", fused)
        ctx = qis.Context(K=K, R=R, precision="fp64", max_n=n, flips=flips, survivor_cap=230)
        ctx.create_instance(np.zeros((n, n)), h)
        ctx.init_states(0, np.repeat(bits[:1], R, axis=0))
        for r in range(R):
            ctx.set_search_list(0, r, bits, E)
        ctx.iterate(1)
        ctx.iterate(5)
        out.append([ctx.search_list(0, r) for r in (0, R - 1)])
        ctx.close()
    for x, y in zip(*out):
        for key in KEYS:
            assert np.array_equal(x[key], y[key]), key
