"""The direct FP32 Phi's tiles where their number crosses one wave of blocks (1216), with
the log-likelihood, MTTKRP and the batched solver on tiles of their own."""
import numpy as np
import pytest

import oracle
from paper_2307_03276_gb300 import cpapr, synth

pytestmark = pytest.mark.gpu
WAVE = 1216


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_2307_03276_gb300 import build
    build.build()
    oracle.build()


def tensor(dims, nnz, seed):
    rng = np.random.default_rng(seed)
    idx = np.stack([np.minimum((rng.random(nnz) ** 3 * d).astype(np.int64), d - 1) for d in dims])
    return idx, rng.integers(1, 6, nnz).astype(np.float64)


def close(got, want, tol):
    assert np.all(np.abs(got - want) <= tol * np.abs(want))


# (dims, nonzeros, rank, tile): the smallest tile of at most a wave, from 256 on (from 64 on at
# padded rank 64)
@pytest.mark.parametrize("dims,nnz,rank,tile", [
    ((500, 400, 300), WAVE * 1024, 4, 1024), ((500, 400, 300), WAVE * 1024 + 1, 4, 2048),
    ((300, 200, 100, 50), WAVE * 1024 + 1, 8, 2048), ((300, 200, 100, 50), 700_000, 10, 1024),
    ((500, 400, 300), WAVE * 256 + 1, 33, 512), ((500, 400, 300), WAVE * 256, 16, 256), ((500, 400, 300), 5000, 70, 64)])
def test_tiles_of_one_wave_match_oracle(dims, nnz, rank, tile):
    idx, vals = tensor(dims, nnz, nnz % 1000 + rank)
    fs = synth.random_factors(dims, rank, 5)
    lam = np.linspace(0.5, 1.5, rank)
    with cpapr.Tensor(dims, idx, vals, rank, precision=cpapr.CPAPR_FP32) as t:
        t.set_model(lam, fs)
        n = len(dims) - 1
        assert t.info().tile_nnz[n] == tile
        close(t.phi(n), oracle.phi(dims, idx, vals, fs, fs[n] * lam, n), 1e-5)
        close(t.mttkrp(n), oracle.mttkrp(dims, idx, vals, fs, n), 1e-5)
        ll = oracle.loglik(dims, idx, vals, lam, fs)
        assert abs(t.loglik() - ll) <= 1e-5 * abs(ll)


def test_batched_and_lone_solves_agree():
    """The batched solver takes larger tiles: the same sums in another order."""
    dims, rank = (300, 200, 100), 8
    idx, vals = tensor(dims, 900_000, 3)
    fs = synth.random_factors(dims, rank, 6)
    out = []
    for batched in (False, True):
        with cpapr.Tensor(dims, idx, vals, rank, precision=cpapr.CPAPR_FP32) as t:
            t.set_model(np.ones(rank), fs)
            if batched:
                cpapr.cpapr_batch_mu_solve([t.ctx], 1e-4, 1, 1)
            else:
                t.mu_solve(1e-4, 1, 1)
            out.append(cpapr.cpapr_get_state(t.ctx))
    close(out[0]["phi_prev"][0], out[1]["phi_prev"][0], 1e-5)
    for a, b in zip(out[0]["factors"], out[1]["factors"]):
        close(a, b, 1e-5)
