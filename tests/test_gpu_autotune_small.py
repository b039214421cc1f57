"""The autotuner's candidates where the built-in choice lies outside the large tiles,
and lanes that Phi does not read."""
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


@pytest.mark.parametrize("precision,tol", [(cpapr.CPAPR_FP64, 1e-12), (cpapr.CPAPR_FP32, 1e-5)])
def test_a_small_tensor_keeps_small_tiles(precision, tol):
    """1e4 nonzeros: ten tiles of 1024 take over twice as long as 64-nonzero ones."""
    T = synth.generate(synth.C1)
    fs = synth.random_factors(T.dims, T.rank, 4)
    lam = np.ones(T.rank)
    with cpapr.Tensor(T.dims, T.idx, T.vals, T.rank, precision=precision, autotune=1) as t:
        info = t.info()
        t.set_model(lam, fs)
        for n in range(T.nmodes):
            assert info.tile_nnz[n] < 1024
            want = oracle.phi(T.dims, T.idx, T.vals, fs, fs[n], n)
            assert np.all(np.abs(t.phi(n) - want) <= tol * np.abs(want))


@pytest.mark.parametrize("opt", [dict(precision=cpapr.CPAPR_FP32), dict(fp64_dot=cpapr.CPAPR_DOT_FP32_PIPE)])
def test_lanes_phi_does_not_read_are_not_tuned(opt):
    """FP32 Phi and the float pairs keep lanes of their own (16 ranks per lane, which
    the pairs do not take, may still win in FP64)."""
    T = synth.random_tensor((300, 200, 100), 50_000, 32, 5)
    with cpapr.Tensor(T.dims, T.idx, T.vals, 32, **opt) as t:
        built_in = list(t.info().rank_lanes[:3])
    with cpapr.Tensor(T.dims, T.idx, T.vals, 32, autotune=1, **opt) as t:
        for lanes, own in zip(t.info().rank_lanes[:3], built_in):
            assert lanes == own or (32 // lanes > 8 and "fp64_dot" in opt)
