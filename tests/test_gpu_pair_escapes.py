"""Elements outside the float pairs' window, of every kind and with every other kind in
one product, against the FP64 oracle at the FP64 bound (1e-12 per entry); both
forms of the Khatri-Rao rows give the same bits."""
import numpy as np
import pytest

import oracle
from paper_2307_03276_gb300 import cpapr

pytestmark = pytest.mark.gpu

# zero; the factors' top; their smallest pair (2^-160 under a top of 1) and its
# neighbours; entries whose products are at the window's lower edge (2^-140), or far
# below it; entries above the exponent of a normalised factor
KINDS = [0.0, 1.0, np.nextafter(1.0, 0), 0.3, 2.0 ** -70, 2.0 ** -70 * 1.5, 2.0 ** -139, 2.0 ** -140,
         np.nextafter(2.0 ** -140, 0), 2.0 ** -160, np.nextafter(2.0 ** -160, 0), 2.0 ** -160 * 1.7, 1e-80, 1e-150,
         np.nextafter(1.0, 2), 1.5, 1e9]


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_2307_03276_gb300 import build
    build.build()
    oracle.build()


@pytest.mark.parametrize("nmodes", [2, 3, 4, 6])
@pytest.mark.parametrize("rank", [3, 16])
@pytest.mark.parametrize("resumed", [False, True])
def test_products_of_every_kind(nmodes, rank, resumed):
    rng = np.random.default_rng(10 * nmodes + rank)
    dims = (400,) + (60, 50, 40, 30, 20)[:nmodes - 1]
    nnz = 4000
    idx = np.stack([rng.integers(0, d, nnz) for d in dims]).astype(np.int64)
    vals = rng.integers(1, 6, nnz).astype(np.float64)
    kinds = np.array(KINDS)
    fs = [kinds[rng.integers(0, kinds.size, (d, rank))] for d in dims]
    # rows of one kind each, so that whole columns of a row are small
    for A in fs[1:]:
        A[::3] = kinds[rng.integers(0, kinds.size, rank)]
    fs[0] = rng.random((dims[0], rank))
    lam = np.ones(rank)
    got = {}
    for pm in (cpapr.CPAPR_PI_FUSED, cpapr.CPAPR_PI_MATERIALISED):
        with cpapr.Tensor(dims, idx, vals, rank, fp64_dot=cpapr.CPAPR_DOT_FP32_PIPE, pi_mode=pm) as t:
            if resumed:  # exponents of normalised factors: entries above 1 have no pair
                cpapr.cpapr_set_state(t.ctx, {"lambda": lam, "factors": fs, "outer_done": 1})
            else:        # exponents measured: the largest entry's
                t.set_model(lam, fs)
            got[pm] = t.phi(0)
            ll = t.loglik()
        want = oracle.loglik(dims, idx, vals, lam, fs)
        assert ll == want or abs(ll - want) <= 1e-11 * abs(want)
    want = oracle.phi(dims, idx, vals, fs, fs[0], 0)
    assert np.array_equal(*got.values())
    nz = want > 0
    assert np.all(np.abs(got[pm][nz] - want[nz]) <= 1e-12 * want[nz])
    assert np.all(got[pm][~nz] == 0)
