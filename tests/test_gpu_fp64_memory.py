"""Device memory of FP64 contexts: couplings are staged a few instances at a time."""
import numpy as np
import pytest
import torch

from paper_2010_00180_gb300 import build, inputs as I, qis

pytestmark = pytest.mark.gpu
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
