"""A solve on float pairs resumed from a checkpoint gives the bits of the solve that
did not stop, also where Khatri-Rao elements lie at the edge of the pairs' window
(which depends on the exponents the factors are scaled by)."""
import numpy as np
import pytest

from paper_2307_03276_gb300 import cpapr

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_2307_03276_gb300 import build
    build.build()


@pytest.mark.parametrize("pi_mode", [cpapr.CPAPR_PI_FUSED, cpapr.CPAPR_PI_MATERIALISED])
@pytest.mark.parametrize("stop", [0, 1, 2])
def test_resume_is_bit_identical_at_the_windows_edge(pi_mode, stop):
    dims, rank, nnz = (300, 200, 100), 8, 4000
    rng = np.random.default_rng(17)
    idx = np.stack([np.minimum((rng.random(nnz) ** 2 * d).astype(np.int64), d - 1) for d in dims])
    vals = rng.integers(1, 6, nnz).astype(np.float64)
    fs = [10.0 ** rng.uniform(-40, 0, (d, rank)) for d in dims]
    lam = np.full(rank, 100.0)
    opt = dict(fp64_dot=cpapr.CPAPR_DOT_FP32_PIPE, pi_mode=pi_mode)
    with cpapr.Tensor(dims, idx, vals, rank, **opt) as t:
        t.set_model(lam, fs)
        t.mu_solve(1e-4, stop, 2)
        state = cpapr.cpapr_get_state(t.ctx)
        r1 = t.mu_solve(1e-4, 2, 2)
        a = cpapr.cpapr_get_state(t.ctx)
    with cpapr.Tensor(dims, idx, vals, rank, **opt) as u:
        cpapr.cpapr_set_state(u.ctx, state)
        r2 = u.mu_solve(1e-4, 2, 2)
        b = cpapr.cpapr_get_state(u.ctx)
    assert r1 == r2
    assert np.array_equal(a["lambda"], b["lambda"])
    for x, y in zip(a["factors"] + a["phi_prev"], b["factors"] + b["phi_prev"]):
        assert np.array_equal(x, y)


@pytest.mark.parametrize("pi_mode", [cpapr.CPAPR_PI_FUSED, cpapr.CPAPR_PI_MATERIALISED])
def test_resume_after_a_batched_solve_is_bit_identical(pi_mode):
    """The batched solver leaves a context's pairs as mu_solve does."""
    dims, rank, nnz = (300, 200, 100), 8, 4000
    rng = np.random.default_rng(17)
    idx = np.stack([np.minimum((rng.random(nnz) ** 2 * d).astype(np.int64), d - 1) for d in dims])
    vals = rng.integers(1, 6, nnz).astype(np.float64)
    fs = [10.0 ** rng.uniform(-40, 0, (d, rank)) for d in dims]
    opt = dict(fp64_dot=cpapr.CPAPR_DOT_FP32_PIPE, pi_mode=pi_mode)
    ends = []
    with cpapr.Tensor(dims, idx, vals, rank, **opt) as t:
        t.set_model(np.full(rank, 100.0), fs)
        cpapr.cpapr_batch_mu_solve([t.ctx], 1e-4, 1, 2)
        state = cpapr.cpapr_get_state(t.ctx)
        r1 = t.mu_solve(1e-4, 2, 2)
        ends.append(cpapr.cpapr_get_state(t.ctx))
    with cpapr.Tensor(dims, idx, vals, rank, **opt) as u:
        cpapr.cpapr_set_state(u.ctx, state)
        r2 = u.mu_solve(1e-4, 2, 2)
        ends.append(cpapr.cpapr_get_state(u.ctx))
    assert r1 == r2
    for x, y in zip(ends[0]["factors"] + ends[0]["phi_prev"], ends[1]["factors"] + ends[1]["phi_prev"]):
        assert np.array_equal(x, y)
