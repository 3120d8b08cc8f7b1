"""Candidate counts across qis_clear_instances: those of removed instances stay in the totals, the next
instances' start at zero."""
import pytest

from paper_2010_00180_gb300 import build, inputs as I, qis

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    qis.load()


def run(ctx, ns, R, seed, iters):
    data = [I.instance("gaussian", n, seed=seed, inst=k) for k, n in enumerate(ns)]
    for k, (iid, n) in enumerate(zip(ctx.create_instances(data), ns)):
        ctx.init_states(iid, I.random_states(n, R, seed=seed + 1, inst=k))
    ctx.iterate(iters)


@pytest.mark.parametrize("precision", ["split_bf16", "fp64"])
@pytest.mark.parametrize("flips", ["single_pair", "exchange", "single"])
@pytest.mark.parametrize("R", [1, 130])
def test_counts_of_removed_instances_stay(precision, flips, R):
    sets = [([8, 70], 850, 5), ([33], 860, 7), ([16, 9, 40], 870, 3)]
    alone = []
    for ns, seed, iters in sets:
        ctx = qis.Context(K=12, R=R, precision=precision, max_n=70, max_instances=3, flips=flips)
        run(ctx, ns, R, seed, iters)
        alone.append(ctx.candidate_count())
        ctx.close()
    ctx = qis.Context(K=12, R=R, precision=precision, max_n=70, max_instances=3, flips=flips)
    ctx.clear_instances()   # nothing there yet
    total = (0, 0)
    for (ns, seed, iters), c in zip(sets, alone):
        run(ctx, ns, R, seed, iters)
        total = tuple(a + b for a, b in zip(total, c))
        assert tuple(ctx.candidate_count()) == total
        ctx.clear_instances()
        assert tuple(ctx.candidate_count()) == total
        ctx.clear_instances()
        assert tuple(ctx.candidate_count()) == total
    assert total[0] + total[1] > 0
    ctx.close()
