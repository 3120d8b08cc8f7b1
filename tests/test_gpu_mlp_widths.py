"""Wide networks. Passes whose activations in shared memory come to 48 KiB exactly (a width of 384 with 16
rows per block, of 768 with 8): the logits' bits are those of smaller batches. Widths above 512, where a
warp takes all rows of a block: logits and gradients against the FP64 oracle (tolerances of the other
widths' tests), logits' bits independent of the batch."""
import numpy as np
import pytest

from oracle import mlp_oracle as M
from paper_2010_00180_gb300 import build, qis

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    qis.load()


@pytest.mark.parametrize("hidden,rows", [(384, 4000), (768, 2000), (400, 4000), (528, 4000), (1024, 4000)])
def test_logits_do_not_depend_on_the_tile(hidden, rows):
    X = np.random.default_rng(880).normal(size=(rows, qis.MLP.N_FEATURES)).astype(np.float32)
    net = qis.MLP(hidden=hidden, max_sites=1, batch=rows, max_n=2, seed=hidden)
    z = net.forward(X)
    for r in (0, 1000, rows - 250):
        assert np.array_equal(z[r: r + 250], net.forward(X[r: r + 250]))
    net.loss_grad(X, (z > 0).astype(np.float32))
    net.close()


@pytest.mark.parametrize("H,rows", [(528, 3), (528, 3000), (640, 609), (880, 2800), (896, 2801), (1024, 608), (1024, 1001)])
def test_wide_networks_against_the_oracle(H, rows):
    net = qis.MLP(hidden=H, max_sites=1, batch=rows, max_n=2, seed=6)
    p = M.unflatten(net.get_params().astype(np.float64), 8, H)
    rng = np.random.default_rng(H + rows)
    X = rng.normal(0, 1, (rows + rows // 10 + 8, 8)).astype(np.float32)
    _, acts = M.forward(p, X)   # (rows at a kink of a ReLU are left out)
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
        np.testing.assert_allclose(g[o:o + b.size], b, rtol=2e-3, atol=2e-4 * max(np.abs(b).max(), 1e-12), err_msg=k)
        o += b.size
    z_ref, _ = M.forward(p, X)
    np.testing.assert_allclose(net.forward(X), z_ref, rtol=1e-4, atol=1e-4 * np.abs(z_ref).max())
    net.close()
