"""FP32 Phi and MTTKRP tiles (direct.cuh) where their windows, runs and tiles
end, against the FP64 oracle at the FP32 bound of the parity tests (1e-5 per
entry: sums of non-negative terms with a few dozen roundings of 6e-8 each)."""
import numpy as np
import pytest

import oracle
from paper_2307_03276_gb300 import cpapr, synth

pytestmark = pytest.mark.gpu
TOL = 1e-5


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_2307_03276_gb300 import build
    build.build()
    oracle.build()


def max_rel(got, want):
    return float(np.max(np.abs(got - want) / np.maximum(np.abs(want), 1e-300), initial=0.0))


def tensor(dims, nnz, seed):
    """Cubed coordinates: rows of one nonzero, of a few, and of hundreds."""
    rng = np.random.default_rng(seed)
    idx = np.stack([np.minimum((rng.random(nnz) ** 3 * d).astype(np.int64), d - 1) for d in dims])
    return idx, rng.integers(1, 6, nnz).astype(np.float64)


@pytest.mark.parametrize("dims", [(300, 7), (60, 50, 40), (40, 30, 20, 10), (12, 11, 10, 9, 8), (9, 8, 7, 6, 5, 4)])
@pytest.mark.parametrize("nnz,rank,tile", [(1, 1, 0), (3, 4, 0), (5, 8, 0), (130, 3, 64), (1021, 16, 64), (2049, 10, 128),
                                           (4099, 32, 320), (3000, 33, 0), (2500, 128, 0)])
def test_direct_tiles_match_oracle(dims, nnz, rank, tile):
    idx, vals = tensor(dims, nnz, nnz + rank)
    fs = synth.random_factors(dims, rank, 5)
    lam = np.linspace(0.5, 1.5, rank)
    for pm in (cpapr.CPAPR_PI_FUSED, cpapr.CPAPR_PI_MATERIALISED):
        with cpapr.Tensor(dims, idx, vals, rank, precision=cpapr.CPAPR_FP32, pi_mode=pm, tile_nnz=tile) as t:
            t.set_model(lam, fs)
            for n in range(len(dims)):
                assert max_rel(t.phi(n), oracle.phi(dims, idx, vals, fs, fs[n] * lam, n)) <= TOL, (pm, n)
                assert max_rel(t.mttkrp(n), oracle.mttkrp(dims, idx, vals, fs, n)) <= TOL, (pm, n)


@pytest.mark.parametrize("pi_mode", [cpapr.CPAPR_PI_FUSED, cpapr.CPAPR_PI_MATERIALISED])
def test_an_infinite_product_stays_in_its_row(pi_mode):
    """Factor entries whose FP32 product overflows make their own nonzero's row
    infinite or NaN; every other row, its neighbours in a window included, is right."""
    dims, rank = (500, 40, 30), 8
    idx, vals = tensor(dims, 3000, 2)
    idx[0] = np.random.default_rng(3).integers(0, 500, 3000)  # about six nonzeros a row
    fs = synth.random_factors(dims, rank, 6)
    fs[1][7, 2] = fs[2][5, 2] = 1e30
    hit = np.unique(idx[0][(idx[1] == 7) & (idx[2] == 5)])
    if hit.size == 0:
        idx[1][0], idx[2][0] = 7, 5
        hit = idx[0][:1]
    want = oracle.phi(dims, idx, vals, fs, fs[0], 0)
    keep = np.setdiff1d(np.unique(idx[0]), hit)
    with cpapr.Tensor(dims, idx, vals, rank, precision=cpapr.CPAPR_FP32, pi_mode=pi_mode) as t:
        t.set_model(np.ones(rank), fs)
        assert max_rel(t.phi(0)[keep], want[keep]) <= TOL
