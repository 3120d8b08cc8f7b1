"""The Alg. 4 merge in runs of consecutive searches merged side by side, against the oracle's merge of
the searches in turn: many equal energies (couplings of +-1, the same state found by several searches,
equal initial states), counts of searches around the line at which runs are used and that do not
divide evenly, lists that are not full."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2010_00180_gb300 import build, inputs as I, qis

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    qis.load()


@pytest.mark.parametrize("ens,precision", [("pm1", "pm1_fp8"), ("gaussian", "split_bf16")])
@pytest.mark.parametrize("n,K,R,iters", [(8, 6, 11, 5), (8, 6, 12, 5), (10, 30, 13, 3), (6, 40, 26, 8), (70, 9, 65, 6),
                                         (130, 120, 17, 4)])
def test_runs_equal_the_merge_in_turn(ens, precision, n, K, R, iters):
    data = [I.instance(ens, n, seed=840, inst=k) for k in range(2)]
    ctx = qis.Context(K=K, R=R, precision=precision, max_n=n, max_instances=2)
    phis = []
    for k, (iid, (J, h)) in enumerate(zip(ctx.create_instances(data), data)):
        phi = I.random_states(n, R, seed=841, inst=k)
        phi[R // 2] = phi[1]   # (equal lists: every state of one is a copy)
        ctx.init_states(iid, phi)
        phis.append(phi)
    ctx.iterate(iters)
    for k, (J, h) in enumerate(data):
        seen, entries = set(), []
        for r in range(R):
            ref = O.qi_search(J, h, K, iters, phis[k][r])
            for p in range(ref["count"]):
                entries.append((ref["E"][p], r, p, ref["bits"][p].tobytes()))
        want = []
        for E, r, p, x in sorted(entries):
            if x not in seen and len(want) < K + 1:
                seen.add(x)
                want.append((E, x, (r << 32) | p))
        got = ctx.topk_states(k, K + 1)
        assert [x.tobytes() for x in got["bits"][: len(want)]] == [x for _, x, _ in want]
        assert np.array_equal(got["E"][: len(want)], [E for E, _, _ in want])
        assert got["src"].tolist() == [s for _, _, s in want]
        assert len(got["E"]) == len(want)
    ctx.close()
