"""Energies from scratch on the tensor cores (Eq. 1) at the edges of their tiles: 64 rows, 64-column
steps, the extra column that holds the fields (its own step when n is a multiple of 64), 1024-column
segments, 128 states; every number of digits; couplings that no 58-bit integer holds exactly.

On a grid the energy is exact. Otherwise every coupling is within 2^-59 of the largest power of two
above |J|, |h| of its integer, and the sum is rounded to FP64 once or twice: the bound below."""
import math

import numpy as np
import pytest

from paper_2010_00180_gb300 import build, inputs as I, qis

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    qis.load()


def exact_energy(J, h, s):
    iu, ju = np.triu_indices(len(h), 1)
    return math.fsum(np.concatenate([J[iu, ju] * s[iu] * s[ju], h * s]))


def energies(J, h, bits, precision):
    ctx = qis.Context(K=1, R=1, precision=precision, max_n=len(h))
    ctx.create_instance(J, h)
    E = ctx.energies(0, bits)
    ctx.close()
    return E


@pytest.mark.parametrize("precision,ens", [("split_bf16", "gaussian"), ("fp64", "gaussian"), ("pm1_fp8", "pm1"),
                                           ("split_bf16", "unrounded"), ("fp64", "unrounded")])
@pytest.mark.parametrize("n,count", [(2, 3), (63, 1), (64, 128), (65, 129), (127, 5), (128, 127), (192, 300),
                                     (1023, 4), (1024, 3), (1025, 2), (2111, 2)])
def test_energies_equal_exact_sums(precision, ens, n, count):
    J, h = I.instance("gaussian" if ens == "unrounded" else ens, n, seed=n, grid_bits=None if ens == "unrounded" else 30)
    bits = I.random_states(n, count, seed=n + 1)
    S = 1.0 - 2.0 * I.unpack_bits(bits, n).astype(np.float64)
    E = energies(J, h, bits, precision)
    for k in sorted({0, count // 2, count - 1}):
        ref = exact_energy(J, h, S[k])
        top = 2.0 ** math.frexp(max(np.abs(J).max(), np.abs(h).max()))[1]
        tol = 0.0 if ens != "unrounded" else n * (n + 1) / 2 * top * 2.0 ** -59 + 2.0 ** -52 * abs(ref)
        assert abs(E[k] - ref) <= tol, (k, E[k], ref)


@pytest.mark.parametrize("scale", [2.0 ** -900, 1e-12, 3e9, 2.0 ** 600])
def test_energies_of_extreme_magnitudes(scale):
    """The integers' exponent follows the largest coupling; fields far larger than the couplings."""
    n = 70
    J, h = I.instance("gaussian", n, seed=3, grid_bits=None)
    J, h = J * scale, h * scale * 1000.0
    bits = I.random_states(n, 9, seed=4)
    S = 1.0 - 2.0 * I.unpack_bits(bits, n).astype(np.float64)
    E = energies(J, h, bits, "fp64")
    top = 2.0 ** math.frexp(np.abs(h).max())[1]
    for k in range(9):
        ref = exact_energy(J, h, S[k])
        assert abs(E[k] - ref) <= n * (n + 1) / 2 * top * 2.0 ** -59 + 2.0 ** -52 * abs(ref)


def test_merged_and_initial_energies_of_mixed_sizes():
    """Instances of different sizes and digit counts in one launch: every merged list's energies
    equal those of qis_energies, and the initial energies those of the states."""
    K, R = 140, 3
    data = [I.instance("gaussian", 64, seed=1), I.instance("pm1", 200, seed=2), I.instance("gaussian", 129, seed=3, grid_bits=None)]
    ctx = qis.Context(K=K, R=R, precision="split_bf16", max_n=200, max_instances=3)
    ctx.create_instances(data)
    phis = [I.random_states(len(h), R, seed=5 + k) for k, (_, h) in enumerate(data)]
    for k in range(3):
        ctx.init_states(k, phis[k])
    for k, (J, h) in enumerate(data):   # the searches' energies are those of the couplings on the grid 2^-q
        q = ctx.instance_info(k)[0]
        Jg, hg = (np.rint(x * 2.0 ** q) * 2.0 ** -q for x in (J, h))
        S = 1.0 - 2.0 * I.unpack_bits(phis[k], len(h)).astype(np.float64)
        for r in range(R):
            assert ctx.search_list(k, r)["E"][0] == exact_energy(Jg, hg, S[r])
    ctx.iterate(9)
    for k, top in enumerate(ctx.topk_states_all(K + 1)):
        assert np.array_equal(top["E"], ctx.energies(k, top["bits"]))
        assert np.array_equal(top["E"], ctx.topk_states(k, K + 1)["E"])
    ctx.close()
