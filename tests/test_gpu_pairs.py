"""The FP64 form's Phi on float-pair Khatri-Rao rows (fp64_dot = the FP32 pipe)
at the edges of the pairs' ranges, against the FP64 oracle at the FP64 bound:
every Phi entry is a sum of non-negative v pi whose relative errors are below
1e-12 (v 3e-13, pi a few 1e-15 or FP64)."""
import numpy as np
import pytest

import oracle
from paper_2307_03276_gb300 import cpapr, synth

pytestmark = pytest.mark.gpu
PIPE = cpapr.CPAPR_DOT_FP32_PIPE


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_2307_03276_gb300 import build
    build.build()
    oracle.build()


def max_rel(got, want):
    nz = want != 0
    e = np.zeros_like(want)
    e[nz] = np.abs(got[nz] - want[nz]) / np.abs(want[nz])
    e[~nz] = np.abs(got[~nz]) > 0
    return float(e.max(initial=0.0))


def tensor(dims, nnz, seed):
    rng = np.random.default_rng(seed)
    idx = np.stack([np.minimum((rng.random(nnz) ** 3 * d).astype(np.int64), d - 1) for d in dims])
    return idx, rng.integers(1, 6, nnz).astype(np.float64)


def spread(dims, rank, decades, seed):
    """Factor entries over `decades` decades below 1, with zeros and 1e9 among them."""
    rng = np.random.default_rng(seed)
    fs = [10.0 ** rng.uniform(-decades, 0.5, (d, rank)) for d in dims]
    for A in fs:
        A[rng.random(A.shape) < 0.05] = 0.0
    fs[0][rng.random(fs[0].shape) < 0.01] = 1e9
    return fs


# padded ranks 2 to 128; runs of one nonzero and rows over several tiles; rows of
# pairs, of escapes (products below 2^-140 of the largest) and of both
@pytest.mark.parametrize("dims,nnz,rank", [((7, 5), 40, 1), ((60, 50, 40), 1, 3), ((60, 50, 40), 3001, 8),
                                           ((300, 20, 10), 5003, 10), ((40, 30, 20, 10), 4000, 33),
                                           ((12, 11, 10, 9, 8), 3000, 16), ((9, 8, 7, 6, 5, 4), 2000, 128)])
@pytest.mark.parametrize("decades", [1, 25, 50])
def test_pair_ranges_match_oracle(dims, nnz, rank, decades):
    idx, vals = tensor(dims, nnz, 3)
    fs = spread(dims, rank, decades, 4)
    lam = np.linspace(0.5, 1.5, rank)
    got = {}
    for pm in (cpapr.CPAPR_PI_FUSED, cpapr.CPAPR_PI_MATERIALISED):
        with cpapr.Tensor(dims, idx, vals, rank, fp64_dot=PIPE, pi_mode=pm) as t:
            t.set_model(lam, fs)
            got[pm] = [t.phi(n) for n in range(len(dims))]
            ll = t.loglik()
        want = oracle.loglik(dims, idx, vals, lam, fs)
        assert ll == want or abs(ll - want) <= 1e-11 * abs(want)
    for n in range(len(dims)):
        want = oracle.phi(dims, idx, vals, fs, fs[n] * lam, n)
        assert np.array_equal(*[g[n] for g in got.values()]), n
        assert max_rel(got[cpapr.CPAPR_PI_FUSED][n], want) <= 1e-12, n


def test_entries_above_the_factor_exponent():
    """A column without mass keeps its entries through a normalisation: they
    exceed the exponent the pairs assume afterwards and take the FP64 path."""
    dims, rank = (50, 40, 30), 6
    idx, vals = tensor(dims, 4000, 9)
    fs = synth.random_factors(dims, rank, 8)
    for A in fs:
        A[:, 2] *= 1e12
    lam = np.ones(rank)
    lam[2] = 0.0
    ref = oracle.mu_solve(dims, idx, vals, lam, fs, tol=1e-4, max_outer=2, max_inner=4)
    with cpapr.Tensor(dims, idx, vals, rank, fp64_dot=PIPE) as t:
        t.set_model(lam, fs)
        r = t.mu_solve(tol=1e-4, max_outer=2, max_inner=4)
        lam_g, fs_g = t.get_model()
    assert r["total_inner"] == ref["total_inner"]
    np.testing.assert_allclose(lam_g, ref["lambda"], rtol=1e-10)
    for A, Ar in zip(fs_g, ref["factors"]):
        np.testing.assert_allclose(A, Ar, rtol=1e-9, atol=1e-14 * Ar[:, [0, 1, 3, 4, 5]].max())
    assert abs(r["loglik"] - ref["loglik"][-1]) <= 1e-11 * abs(ref["loglik"][-1])


@pytest.mark.parametrize("nnz", [608 * 1024 - 1024, 608 * 1024 - 1023, 1368 * 1024 + 1])
def test_pair_tiles_at_the_dispatch_edges(nnz):
    """Just below and at 608 tiles (FP64 dot, pairs), and where the pair launch takes larger tiles."""
    dims, rank = (3000, 2000, 100), 20
    idx, vals = tensor(dims, nnz, 11)
    fs = synth.random_factors(dims, rank, 12)
    lam = np.ones(rank)
    with cpapr.Tensor(dims, idx, vals, rank) as t:
        t.set_model(lam, fs)
        n = 2
        assert max_rel(t.phi(n), oracle.phi(dims, idx, vals, fs, fs[n] * lam, n)) <= 1e-12
        assert max_rel(t.mttkrp(n), oracle.mttkrp(dims, idx, vals, fs, n)) <= 1e-12
