"""Large FP64 Phi with a model whose entries have decayed over many decades: the
kernel that keeps the rows in FP64 takes over from the float pairs, with the same
bits for both forms of the rows and for a resumed solve."""
import numpy as np
import pytest

import oracle
from paper_2307_03276_gb300 import cpapr, synth

pytestmark = pytest.mark.gpu
# 684 tiles of 1024 nonzeros (at least 608); the pairs' launches take 512 nonzeros a tile
DIMS, RANK, NNZ = (3000, 2000, 100), 20, 700_000
PI = [cpapr.CPAPR_PI_FUSED, cpapr.CPAPR_PI_MATERIALISED]


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_2307_03276_gb300 import build
    build.build()
    oracle.build()


@pytest.fixture(scope="module")
def tensor():
    rng = np.random.default_rng(31)
    idx = np.stack([np.minimum((rng.random(NNZ) ** 2 * d).astype(np.int64), d - 1) for d in DIMS])
    return idx, rng.integers(1, 6, NNZ).astype(np.float64)


def late_model(seed, decades):
    """Each factor row uses a few components; the others are `decades` decades down."""
    rng = np.random.default_rng(seed)
    fs = []
    for d in DIMS:
        A = 10.0 ** rng.uniform(-decades, -decades / 2, (d, RANK))
        use = rng.random((d, RANK)) < 0.2
        A[use] = rng.random(int(use.sum()))
        A[np.arange(d), rng.integers(0, 3, d)] += 0.5
        fs.append(A)
    return fs


@pytest.mark.parametrize("pi_mode", PI)
def test_phi_leaves_the_pairs_and_returns(tensor, pi_mode):
    idx, vals = tensor
    early, late = synth.random_factors(DIMS, RANK, 5), late_model(6, 60)
    lam = np.ones(RANK)
    with cpapr.Tensor(DIMS, idx, vals, RANK, pi_mode=pi_mode) as t:
        for fs, tile in ((early, 512), (late, 1024), (early, 512)):
            t.set_model(lam, fs)
            for n in (2, 0):
                want = oracle.phi(DIMS, idx, vals, fs, fs[n], n)
                got = t.phi(n)
                assert t.info().tile_nnz[n] == tile, n
                assert np.all(np.abs(got - want) <= 1e-12 * want), n
            ll = oracle.loglik(DIMS, idx, vals, lam, fs)
            assert abs(t.loglik() - ll) <= 1e-11 * abs(ll)
    # always on the pairs where the caller says so
    with cpapr.Tensor(DIMS, idx, vals, RANK, pi_mode=pi_mode, fp64_dot=cpapr.CPAPR_DOT_FP32_PIPE) as t:
        t.set_model(lam, late)
        got = t.phi(0)
        assert t.info().tile_nnz[0] == 512
        want = oracle.phi(DIMS, idx, vals, late, late[0], 0)
        assert np.all(np.abs(got - want) <= 1e-12 * want)


@pytest.mark.parametrize("decades", [30, 45, 60])
def test_solves_keep_their_bits(tensor, decades):
    """Fused and materialised, stopped and not, with modes on either kernel."""
    idx, vals = tensor
    fs = late_model(7, decades)
    lam = np.full(RANK, 50.0)
    ends = []
    for pm in PI:
        with cpapr.Tensor(DIMS, idx, vals, RANK, pi_mode=pm) as t:
            t.set_model(lam, fs)
            r = t.mu_solve(1e-4, 4, 2, trace=True)
            ends.append((r, cpapr.cpapr_get_state(t.ctx)))
        with cpapr.Tensor(DIMS, idx, vals, RANK, pi_mode=pm) as t:
            t.set_model(lam, fs)
            t.mu_solve(1e-4, 2, 2)
            state = cpapr.cpapr_get_state(t.ctx)
            r = t.mu_solve(1e-4, 2, 2)
            ends.append((r, cpapr.cpapr_get_state(t.ctx)))
        with cpapr.Tensor(DIMS, idx, vals, RANK, pi_mode=pm) as t:
            cpapr.cpapr_set_state(t.ctx, state)
            r = t.mu_solve(1e-4, 2, 2)
            ends.append((r, cpapr.cpapr_get_state(t.ctx)))
    for r, s in ends[1:]:
        assert np.array_equal(s["lambda"], ends[0][1]["lambda"])
        for a, b in zip(s["factors"] + s["phi_prev"], ends[0][1]["factors"] + ends[0][1]["phi_prev"]):
            assert np.array_equal(a, b)
    for k in (0, 3):  # the log-likelihood sums the rows in one order per form
        assert ends[k][0]["loglik"] == ends[k + 1][0]["loglik"] == ends[k + 2][0]["loglik"]
