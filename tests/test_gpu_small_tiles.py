"""Automatic tile sizes of small tensors, and the batched solver's larger
tiles made of several of them (FP64), against the FP64 oracle."""
import numpy as np
import pytest

import oracle
from paper_2307_03276_gb300 import cpapr, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_2307_03276_gb300 import build
    build.build()
    oracle.build()


def heavy_row_tensor(nnz, seed, dims=(40, 3000, 200)):
    """Half of the nonzeros in one row of mode 0 (cut by many tiles), the rest uniform."""
    rng = np.random.default_rng(seed)
    i0 = np.where(rng.random(nnz) < 0.5, 17, rng.integers(0, dims[0], nnz))
    idx = np.stack([i0] + [rng.integers(0, d, nnz) for d in dims[1:]]).astype(np.int64)
    return dims, idx, rng.integers(1, 5, nnz).astype(np.float64)


def max_rel(got, want):
    return float(np.max(np.abs(got - want) / np.maximum(np.abs(want), 1e-300), initial=0.0))


# (nonzeros, expected tile): FP64 takes the smallest power of two >= 64 with
# fewer than 608 tiles, FP32 with fewer than 152
@pytest.mark.parametrize("precision,nnz,tile", [
    (cpapr.CPAPR_FP64, 1, 64), (cpapr.CPAPR_FP64, 63, 64), (cpapr.CPAPR_FP64, 64 * 607, 64),
    (cpapr.CPAPR_FP64, 64 * 607 + 1, 128), (cpapr.CPAPR_FP64, 128 * 607 + 1, 256),
    (cpapr.CPAPR_FP32, 1, 64), (cpapr.CPAPR_FP32, 64 * 151, 64), (cpapr.CPAPR_FP32, 64 * 151 + 1, 128)])
def test_small_tiles_match_oracle(precision, nnz, tile):
    dims, idx, vals = heavy_row_tensor(nnz, nnz)
    fs = synth.random_factors(dims, 10, 3)
    lam = np.linspace(0.5, 1.5, 10)
    # every Phi entry is a sum of non-negative terms: the FP64 and FP32 bounds of the parity tests
    tol = 1e-12 if precision == cpapr.CPAPR_FP64 else 1e-5
    with cpapr.Tensor(dims, idx, vals, 10, precision=precision) as t:
        t.set_model(lam, fs)
        assert t.info().tile_nnz[0] == tile
        for n in range(3):
            assert max_rel(t.phi(n), oracle.phi(dims, idx, vals, fs, fs[n] * lam, n)) <= tol, n


@pytest.mark.parametrize("nnz", [65, 5000, 40_000])
def test_batch_of_coarse_tiles_matches_oracle(nnz):
    """FP64: the batched solver takes 2^k of a small tensor's tiles as one;
    rows that span several of the larger tiles, of the smaller ones only, or none."""
    tensors = [heavy_row_tensor(nnz, 7), heavy_row_tensor(nnz // 3, 8)]
    ctxs = []
    for d, i, v in tensors:
        t = cpapr.Tensor(d, i, v, 8)
        t.set_model(np.ones(8), synth.random_factors(d, 8, 5))
        ctxs.append(t)
    res = cpapr.cpapr_batch_mu_solve([t.ctx for t in ctxs], 1e-4, 2, 3)
    for t, (d, i, v), r in zip(ctxs, tensors, res):
        ref = oracle.mu_solve(d, i, v, np.ones(8), synth.random_factors(d, 8, 5), tol=1e-4, max_outer=2, max_inner=3)
        lam, fs = t.get_model()
        assert r["total_inner"] == ref["total_inner"]
        np.testing.assert_allclose(lam, ref["lambda"], rtol=1e-10)
        for a, b in zip(fs, ref["factors"]):
            np.testing.assert_allclose(a, b, rtol=1e-9, atol=1e-14 * b.max())
        assert abs(r["loglik"] - ref["loglik"][-1]) <= 1e-11 * abs(ref["loglik"][-1])
        t.close()
