"""FP32 sums and quotients beyond the float range are infinite, whatever path the
row takes (one run, several runs of a tile, several tiles, staged or direct
tiles); every entry within the range is right (the FP32 bound of the parity
tests, 1e-5)."""
import numpy as np
import pytest

import oracle
from paper_2307_03276_gb300 import cpapr

pytestmark = pytest.mark.gpu
TOL, TOP = 1e-5, float(np.finfo(np.float32).max)


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_2307_03276_gb300 import build
    build.build()
    oracle.build()


def tensor(dims, nnz, seed):
    """Rows of a few nonzeros, and one (mode 0, row 3) of a third of them all."""
    rng = np.random.default_rng(seed)
    idx = np.stack([rng.integers(0, d, nnz) for d in dims]).astype(np.int64)
    idx[0, ::3] = 3
    return idx, rng.integers(1, 6, nnz).astype(np.float64)


def check(got, want, over=None):
    """over: entries whose terms overflow by themselves (else: those whose sum does)."""
    fits = want < TOP * (1 - TOL) if over is None else ~over
    over = want > TOP * (1 + TOL) if over is None else over
    assert over.any() and fits.any()
    assert np.all(np.isposinf(got[over]))
    err = np.abs(got[fits] - want[fits]) / np.maximum(np.abs(want[fits]), 1e-300)
    assert float(err.max()) <= TOL


@pytest.mark.parametrize("dims", [(900, 40), (900, 40, 30), (900, 40, 30, 20)])
@pytest.mark.parametrize("rank", [3, 16, 64])
@pytest.mark.parametrize("tile", [0, 64])
@pytest.mark.parametrize("pi_mode", [cpapr.CPAPR_PI_FUSED, cpapr.CPAPR_PI_MATERIALISED])
def test_overflowing_sums_are_infinite(dims, rank, tile, pi_mode):
    idx, vals = tensor(dims, 3000, 4)
    rng = np.random.default_rng(rank)
    fs = [0.5 + 0.5 * rng.random((d, rank)) for d in dims]
    # products stay below 2e38; the sums of a few of them do not
    fs[1][::2] *= 2e38
    with cpapr.Tensor(dims, idx, vals, rank, precision=cpapr.CPAPR_FP32, tile_nnz=tile, pi_mode=pi_mode) as t:
        t.set_model(np.ones(rank), fs)
        check(t.mttkrp(0), oracle.mttkrp(dims, idx, vals, fs, 0))
    # quotients x / eps of 1e10 each (no B: the model is 0 there), times products up to 1e29
    fs[1][::2] *= 1e29 / 2e38
    with cpapr.Tensor(dims, idx, vals, rank, precision=cpapr.CPAPR_FP32, tile_nnz=tile, pi_mode=pi_mode) as t:
        t.set_model(np.ones(rank), fs)
        B = np.zeros_like(fs[0])
        check(t.phi(0, B=B), oracle.phi(dims, idx, vals, fs, B, 0))


@pytest.mark.parametrize("rank", [3, 16, 64])
def test_an_overflowing_quotient_is_infinite(rank):
    """x / max(s, eps) = 1e39 from a divisor whose reciprocal is a float."""
    dims = (900, 40, 30)
    idx, vals = tensor(dims, 3000, 5)
    vals[idx[0] % 2 == 0] = 1e10
    fs = [0.5 + 0.5 * np.random.default_rng(rank).random((d, rank)) for d in dims]
    B = np.zeros_like(fs[0])
    with cpapr.Tensor(dims, idx, vals, rank, precision=cpapr.CPAPR_FP32, eps=1e-29) as t:
        t.set_model(np.ones(rank), fs)
        want = oracle.phi(dims, idx, vals, fs, B, 0, eps=1e-29)
        quotient = np.broadcast_to(np.arange(900)[:, None] % 2 == 0, want.shape) & (want > 0)
        check(t.phi(0, B=B), want, quotient)
