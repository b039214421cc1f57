"""The FP64 form on float pairs keeps the FP64 range: results near its top, and sums
far below the largest products, against the oracle at the FP64 bound (1e-12)."""
import numpy as np
import pytest

import oracle
from paper_2307_03276_gb300 import cpapr

pytestmark = pytest.mark.gpu
PI = [cpapr.CPAPR_PI_FUSED, cpapr.CPAPR_PI_MATERIALISED]


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_2307_03276_gb300 import build
    build.build()
    oracle.build()


def tensor(dims, nnz, seed):
    rng = np.random.default_rng(seed)
    idx = np.stack([np.minimum((rng.random(nnz) ** 2 * d).astype(np.int64), d - 1) for d in dims])
    return rng, idx, rng.integers(1, 6, nnz).astype(np.float64)


def check(got, want):
    assert np.all(np.isfinite(want))
    assert np.all(np.abs(got - want) <= 1e-12 * want)


@pytest.mark.parametrize("pi_mode", PI)
def test_results_near_the_top_of_the_range(pi_mode):
    dims, rank = (50, 40, 30), 8
    rng, idx, vals = tensor(dims, 3000, 1)
    fs = [0.5 + 0.5 * rng.random((d, rank)) for d in dims]
    vals[idx[0] % 3 == 0] *= 1e300  # sums up to some 1e302, below 1.8e308
    with cpapr.Tensor(dims, idx, vals, rank, fp64_dot=cpapr.CPAPR_DOT_FP32_PIPE, pi_mode=pi_mode) as t:
        t.set_model(np.ones(rank), fs)
        check(t.phi(0), oracle.phi(dims, idx, vals, fs, fs[0], 0))


@pytest.mark.parametrize("pi_mode", PI)
def test_sums_far_below_the_largest_products(pi_mode):
    """Six modes whose largest products are near 2^500, and rows of products near 1e-225."""
    dims, rank = (60, 20, 20, 20, 20, 20), 8
    rng, idx, vals = tensor(dims, 3000, 2)
    fs = [0.5 + 0.5 * rng.random((d, rank)) for d in dims]
    small = idx[0] % 2 == 0  # mode-0 rows whose nonzeros meet small factor rows only
    for m in range(1, 6):
        idx[m] = np.where(small, idx[m] % 10, 10 + idx[m] % 10)
        fs[m][:10] *= 1e-45
        fs[m][10:] *= 1e30
    with cpapr.Tensor(dims, idx, vals, rank, fp64_dot=cpapr.CPAPR_DOT_FP32_PIPE, pi_mode=pi_mode) as t:
        t.set_model(np.ones(rank), fs)
        want = oracle.phi(dims, idx, vals, fs, fs[0], 0)
        assert 0 < want[::2][want[::2] > 0].min() < 1e-200
        check(t.phi(0), want)


@pytest.mark.parametrize("pi_mode", PI)
def test_counts_at_the_edges_of_the_quotients_range(pi_mode):
    """Counts from 2^-20 up to 2^30 take the FP32 quotient, all others FP64."""
    dims, rank = (50, 40, 30), 8
    rng, idx, vals = tensor(dims, 3000, 3)
    fs = [0.5 + 0.5 * rng.random((d, rank)) for d in dims]
    edge = np.array([2.0 ** -20, np.nextafter(2.0 ** -20, 0), np.nextafter(2.0 ** 30, 0), 2.0 ** 30, 2.0 ** 30 - 1, 2.0 ** 31])
    vals[:] = edge[rng.integers(0, edge.size, vals.size)]
    vals[::11] = 0.0
    with cpapr.Tensor(dims, idx, vals, rank, fp64_dot=cpapr.CPAPR_DOT_FP32_PIPE, pi_mode=pi_mode) as t:
        t.set_model(np.ones(rank), fs)
        for n in range(3):
            check(t.phi(n), oracle.phi(dims, idx, vals, fs, fs[n], n))
