"""Device memory of FP64 contexts: couplings are staged a few instances at a time, the filter's planes
and rings are left out where nothing reads them, and a context that does not fit with them is created
without (the per-kernel form)."""
import numpy as np
import pytest
import torch

from paper_2010_00180_gb300 import build, inputs as I, qis

pytestmark = pytest.mark.gpu
KEYS = ("count", "bits", "E", "stamp", "used")
GiB = 1 << 30


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    qis.load()


def taken(**cfg):
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    ctx = qis.Context(precision="fp64", **cfg)
    got = before - torch.cuda.mem_get_info()[0]
    ctx.close()
    return got


def test_couplings_are_not_held_twice():
    # 32 instances of n = 2048: 1 GiB of couplings; lists, buffers and the staging take less than a quarter
    taken(K=8, R=1, max_n=64, flips="single")   # (the CUDA context's own memory)
    assert taken(K=8, R=1, max_n=2048, max_instances=32, flips="single") < 1.25 * GiB


def test_no_filter_planes_where_the_fused_form_is_off(monkeypatch):
    # 32 instances of n = 1024, 64 searches each: 256 MiB of couplings, 16 MiB per iteration of a field ring
    monkeypatch.setenv("QIS_FUSED", "0")
    taken(K=8, R=1, max_n=64)
    assert taken(K=8, R=64, max_n=1024, max_instances=32) < 0.75 * GiB


@pytest.mark.parametrize("flips", ["single", "single_pair"])
def test_staging_in_parts(flips):
    """A batch of more couplings than the staging holds, page-locked ones among them."""
    n, cnt, K, R = 600, 70, 8, 2
    data = []
    for k in range(cnt):
        J, h = I.instance("gaussian", n, seed=890, inst=k)
        if k % 5 == 3:
            J = torch.from_numpy(J).pin_memory().numpy()
        data.append((J, h))
    phi = [I.random_states(n, R, seed=891, inst=k) for k in range(cnt)]
    ctx = qis.Context(K=K, R=R, precision="fp64", max_n=n, max_instances=cnt, flips=flips)
    for iid, p in zip(ctx.create_instances(data), phi):
        ctx.init_states(iid, p)
    for k in range(cnt):
        S = 1.0 - 2.0 * I.unpack_bits(phi[k], n).astype(np.float64)
        E = 0.5 * np.einsum("ki,ij,kj->k", S, data[k][0], S) + S @ data[k][1]
        # sums of dyadic numbers: exact in FP64 in any order
        assert np.array_equal(ctx.energies(k, phi[k]), E), k
    ctx.close()


def test_created_without_the_filter_where_memory_is_short():
    n, cnt, K, R = 1024, 32, 8, 64
    cfg = dict(K=K, R=R, precision="fp64", max_n=n, max_instances=cnt)
    J, h = I.instance("gaussian", n, seed=892, grid_bits=None)
    phi = I.random_states(n, R, seed=893)

    def lists():
        ctx = qis.Context(**cfg)
        ctx.create_instance(J, h)
        ctx.init_states(0, phi)
        ctx.iterate(4)
        out = [ctx.search_list(0, r) for r in range(0, R, 9)]
        ctx.close()
        return out

    ref = lists()
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    hold = torch.empty(free - GiB, dtype=torch.uint8, device="cuda")   # 1 GiB left: 2.6 with the filter, 0.5 without
    try:
        got = lists()
    finally:
        del hold
        torch.cuda.empty_cache()
    for x, y in zip(got, ref):
        for key in KEYS:
            assert np.array_equal(x[key], y[key]), key
