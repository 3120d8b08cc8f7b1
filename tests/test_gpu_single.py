"""The single-flip search kernel (every iteration of a launch in one block) against the per-kernel
form of the same searches, whose lists it must equal bit for bit: block sizes (padded n up to 1024,
4096 and beyond), more iterations than a launch holds, generators that have left the ring, ties and
outliers that put more sites into one histogram bin than the block's buffer holds, searches that
use up their states, imported lists."""
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


def lists(data, phis, K, R, chunks, prec, cap=0):
    ctx = qis.Context(K=K, R=R, precision=prec, max_n=max(len(h) for _, h in data), max_instances=len(data),
                      flips="single", survivor_cap=cap)
    for iid, phi in zip(ctx.create_instances(data), phis):
        ctx.init_states(iid, phi)
    for c in chunks:
        ctx.iterate(c)
    out = [ctx.search_list(k, r) for k in range(len(data)) for r in range(R)]
    out += [ctx.topk_states(k, K + 1) for k in range(len(data))]
    active = ctx.iterate(0, count_active=True)
    counts = ctx.candidate_count()
    ctx.close()
    return out, active, counts


def both(monkeypatch, data, phis, K, R, chunks, prec, cap=0):
    got = lists(data, phis, K, R, chunks, prec, cap)
    monkeypatch.setenv("QIS_FUSED", "0")
    ref = lists(data, phis, K, R, [sum(chunks)], prec, cap)
    monkeypatch.delenv("QIS_FUSED")
    assert got[1:] == ref[1:]
    for x, y in zip(got[0], ref[0]):
        for key in (k for k in KEYS if k in x):
            assert np.array_equal(x[key], y[key]), key
    return got[0]


@pytest.mark.parametrize("prec,ens,ns,K,R,chunks", [
    ("split_bf16", "gaussian", [2, 31], 2, 2, [3]),
    ("split_bf16", "gaussian", [64, 127, 300], 40, 5, [1, 7, 1]),
    ("pm1_fp8", "pm1", [500, 257], 120, 4, [30, 1, 9]),
    ("split_bf16", "uniform", [1025, 4096], 120, 3, [20, 2]),
    ("split_bf16", "uniform", [4097, 90], 255, 2, [25]),
    ("split_bf16", "gaussian", [90], 200, 3, [300, 5])])          # more than one launch per call
def test_single_equals_per_kernel_form(monkeypatch, prec, ens, ns, K, R, chunks):
    data = [I.instance(ens, n, seed=800, inst=k, grid_bits=20) for k, n in enumerate(ns)]   # energies exact in FP64
    phis = [I.random_states(n, R, seed=801, inst=k) for k, n in enumerate(ns)]
    got = both(monkeypatch, data, phis, K, R, chunks, prec)
    J, h = data[-1]
    ref = O.qi_search(J, h, K, sum(chunks), phis[-1][0], flips=1)
    x = got[(len(ns) - 1) * R]
    for key in KEYS[1:]:
        assert np.array_equal(x[key], ref[key][: ref["count"]]), key


def test_single_generators_out_of_the_ring(monkeypatch):
    monkeypatch.setenv("QIS_FIELD_RING", "2")
    data = [I.instance("gaussian", 200, seed=802)]
    both(monkeypatch, data, [I.random_states(200, 4, seed=803)], 60, 4, [10, 12], "split_bf16")


@pytest.mark.parametrize("what", ["outlier", "ties", "two_values"])
def test_single_crowded_bins(monkeypatch, what):
    """1500 sites: one coupling 2^30 times the others (the histogram of their changes is one bin),
    fields only of one size (every change of energy is one of two values), or of two sizes."""
    n, K, R = 1500, 120, 2
    J, h = np.zeros((n, n)), np.ones(n)
    if what == "outlier":
        J, h = I.instance("uniform", n, seed=804, grid_bits=8)
        J[3, 7] = J[7, 3] = 2.0 ** 22
    elif what == "two_values":
        h[::3] = 5.0
    both(monkeypatch, [(J, h)], [I.random_states(n, R, seed=805)], K, R, [8], "split_bf16")


def test_single_full_spectrum_and_imported_lists(monkeypatch):
    """K + 1 = 2^n: the searches end with every state used; a list imported with arrival stamps
    beyond its iteration continues as in the per-kernel form."""
    n, R = 6, 2
    J, h = I.instance("gaussian", n, seed=806)
    both(monkeypatch, [(J, h)], [I.random_states(n, R, seed=807)], 2 ** n - 1, R, [70], "split_bf16")
    n, K = 80, 30
    J, h = I.instance("gaussian", n, seed=808)
    phi = I.random_states(n, 1, seed=809)
    out = []
    for fused in ("1", "0"):
        monkeypatch.setenv("QIS_FUSED", fused)
        ctx = qis.Context(K=K, R=1, precision="split_bf16", max_n=n, flips="single")
        ctx.create_instance(J, h)
        ctx.init_states(0, phi)
        ctx.iterate(9)
        x = ctx.search_list(0, 0)
        ctx.set_search_list(0, 0, x["bits"], x["E"], x["used"], x["stamp"], t=4)
        ctx.iterate(11)
        out.append(ctx.search_list(0, 0))
        ctx.close()
    for key in KEYS:
        assert np.array_equal(out[0][key], out[1][key]), key
