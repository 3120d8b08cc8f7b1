"""The warm-start network's kernels at the edges of their tiles: rows per block (4, 8, 16), the
128 columns of a warp, the 128 x 64 tiles and row parts of the weight gradients, hidden sizes
that fill a tile partly. Tolerances as for the full-size gradients. A row with a pre-activation
within FP32 rounding of zero is left out: its ReLU may fall on either side."""
import numpy as np
import pytest

from oracle import mlp_oracle as M
from paper_2010_00180_gb300 import build, inputs as I, qis

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    qis.load()


@pytest.mark.parametrize("H,rows", [(16, 1), (16, 3000), (48, 5), (128, 33), (144, 129), (256, 31), (256, 2437),
                                    (272, 4001), (528, 1300), (528, 2600), (1024, 7)])
def test_gradients_at_tile_edges(H, rows):
    net = qis.MLP(hidden=H, max_sites=1, batch=rows, max_n=2, seed=6)
    p = M.unflatten(net.get_params().astype(np.float64), 8, H)
    rng = np.random.default_rng(H + rows)
    X = rng.normal(0, 1, (rows + rows // 20 + 8, 8)).astype(np.float32)
    _, acts = M.forward(p, X)
    kink = np.any([(np.abs(a) < 2e-6 * np.abs(a).max()).any(1) for a in (acts[1], acts[3], acts[5])], axis=0)
    X = X[~kink][:rows]
    assert len(X) == rows
    y = (rng.random(rows) < 0.4).astype(np.float32)
    L, g = net.loss_grad(X, y)
    L_ref, g_ref = M.loss_and_grad(p, X, y)
    assert abs(L - L_ref) <= 1e-5 * abs(L_ref)
    o = 0
    for k in M.PARAM_ORDER:
        b = np.asarray(g_ref[k], np.float64).reshape(-1)
        a = g[o:o + b.size].astype(np.float64)
        np.testing.assert_allclose(a, b, rtol=2e-3, atol=2e-4 * max(np.abs(b).max(), 1e-12), err_msg=k)
        o += b.size
    z_ref, _ = M.forward(p, X)
    np.testing.assert_allclose(net.forward(X), z_ref, rtol=1e-4, atol=1e-4 * np.abs(z_ref).max())


@pytest.mark.parametrize("H", [64, 256, 640])
def test_logits_do_not_depend_on_the_tile(H):
    """A row's logit has the same bits in a batch of any size (any rows per block)."""
    rows = 4500
    net = qis.MLP(hidden=H, max_sites=1, batch=rows, max_n=2, seed=7)
    X = np.random.default_rng(1).normal(0, 1, (rows, 8)).astype(np.float32)
    z = net.forward(X)
    for m in (1, 6, 1000):
        assert np.array_equal(net.forward(X[:m]), z[:m])


@pytest.mark.parametrize("n,R", [(31, 1), (64, 9), (97, 8), (300, 33)])
def test_proposed_states_are_the_stream_draws(n, R):
    """Half words and groups of eight searches: search 0 is sign(z), every other bit compares its
    SplitMix64 draw with sigmoid(z) in FP64; a second instance's call follows without a wait."""
    def mix(key, c):
        return I.splitmix64(np.uint64(key), c)

    seed, ids = 9, (0, 1)
    net = qis.MLP(hidden=64, max_sites=1, batch=n, max_n=n, seed=8)
    ctx = qis.Context(K=3, R=R, precision="split_bf16", max_n=n, max_instances=2, seed=seed)
    data = [I.instance("gaussian", n, seed=10, inst=k) for k in ids]
    ctx.create_instances(data)
    for k in ids:
        ctx.init_states_learned(k, net)
    for k in ids:
        z = net.forward(net.features(*data[k])).astype(np.float64)
        key = mix(int(mix(int(mix(int(mix(seed, 0)) ^ k, 0)) ^ 3, 0)) ^ 5, 0)
        p = 1.0 / (1.0 + np.exp(-z))
        for r in range(R):
            u = (mix(key, np.arange(r * n, r * n + n)) >> np.uint64(11)).astype(np.float64) * 2.0 ** -53
            sig = (z < 0) if r == 0 else ~(u < p)
            safe = np.abs(u - p) > 1e-12 if r else np.ones(n, bool)   # exp() of the device and of numpy
            got = I.unpack_bits(ctx.search_list(k, r)["bits"][0], n)[0].astype(bool)
            assert np.array_equal(got[safe], sig[safe])
    ctx.close()
