"""A context without the memory for its factors as float pairs still works: the
FP64 kernels that need none take over (within 1e-12 of the oracle)."""
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


@pytest.mark.parametrize("pi_mode", [cpapr.CPAPR_PI_FUSED, cpapr.CPAPR_PI_MATERIALISED])
def test_no_room_for_the_pairs_is_not_an_error(monkeypatch, pi_mode):
    T = synth.random_tensor((60, 50, 40), 5000, 12, 7)
    fs = synth.random_factors(T.dims, 12, 8)
    opt = dict(fp64_dot=cpapr.CPAPR_DOT_FP32_PIPE, pi_mode=pi_mode)
    with cpapr.Tensor(T.dims, T.idx, T.vals, 12, **opt) as t:
        full = t.info().device_bytes
    pairs = sum(-(-d * 16 * 8 // 256) * 256 for d in T.dims) + 256
    worked = 0
    for k in range(1, 100):
        monkeypatch.setenv("CPAPR_FAULT_ALLOC_AT", str(k))
        try:
            t = cpapr.Tensor(T.dims, T.idx, T.vals, 12, **opt)
        except cpapr.CpaprError as e:
            assert e.status == 4 and "injected" in str(e)
            continue
        finally:
            monkeypatch.delenv("CPAPR_FAULT_ALLOC_AT")
        with t:
            if t.info().device_bytes == full:  # past the last allocation
                break
            worked += 1
            assert t.info().device_bytes == full - pairs
            t.set_model(np.ones(12), fs)
            for n in range(3):
                want = oracle.phi(T.dims, T.idx, T.vals, fs, fs[n], n)
                assert np.all(np.abs(t.phi(n) - want) <= 1e-12 * want)
            ref = oracle.mu_solve(T.dims, T.idx, T.vals, np.ones(12), fs, tol=1e-4, max_outer=2, max_inner=3)
            assert t.mu_solve(1e-4, 2, 3)["total_inner"] == ref["total_inner"]
    assert worked == 1 and k < 99
