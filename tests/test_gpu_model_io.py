"""Models and outputs through host, pinned, device and misaligned device
buffers, and the error cases of cpapr_set_model."""
import ctypes

import numpy as np
import pytest

from paper_2307_03276_gb300 import cpapr, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_2307_03276_gb300 import build
    build.build()


DIMS = (30, 20, 10)


def context(rank, precision):
    T = synth.random_tensor(DIMS, 900, rank, 40 + rank)
    return cpapr.Tensor(T.dims, T.idx, T.vals, rank, precision=precision)


@pytest.mark.parametrize("precision", [cpapr.CPAPR_FP64, cpapr.CPAPR_FP32])
@pytest.mark.parametrize("rank", [1, 3, 8, 33, 128])
def test_model_round_trip_from_every_kind_of_memory(precision, rank):
    import torch
    fs = synth.random_factors(DIMS, rank, 3)
    lam = np.linspace(0.5, 2.0, rank)

    def misaligned(a):  # a device copy that starts 4 bytes off an 8-byte boundary
        raw = torch.zeros(a.size * 8 + 8, dtype=torch.uint8, device="cuda")
        raw[4:4 + a.size * 8] = torch.from_numpy(np.ascontiguousarray(a).view(np.uint8).reshape(-1)).cuda()
        return raw, raw.data_ptr() + 4

    with context(rank, precision) as t:
        t.set_model(lam, fs)
        want = [t.phi(n) for n in range(3)]
        for kind in ("host", "pinned", "device", "mixed", "misaligned"):
            t.set_model(np.ones(rank), [np.ones_like(A) for A in fs])
            if kind == "misaligned":
                keep = [misaligned(A) for A in [lam] + fs]
                torch.cuda.synchronize()
                arr = (ctypes.c_void_p * 3)(*[k[1] for k in keep[1:]])
                assert cpapr.load().cpapr_set_model(t.ctx, keep[0][1], arr) == 0
            else:
                conv = {"host": lambda a, m: a, "pinned": lambda a, m: torch.from_numpy(a).pin_memory(),
                        "device": lambda a, m: torch.from_numpy(a).cuda(),
                        "mixed": lambda a, m: torch.from_numpy(a).cuda() if m % 2 else a}[kind]
                args = conv(lam, 1), [conv(A, m) for m, A in enumerate(fs)]
                torch.cuda.synchronize()
                t.set_model(*args)
            lg, fg = t.get_model()
            assert np.array_equal(lg, lam), kind
            for A, B in zip(fs, fg):
                assert np.array_equal(A, B), kind  # FP32 returns the FP64 masters
            for n in range(3):
                out = torch.zeros((DIMS[n], rank), dtype=torch.float64, device="cuda")
                torch.cuda.synchronize()
                assert np.array_equal(t.phi(n), want[n]), kind
                assert np.array_equal(t.phi(n, out=out).cpu().numpy(), want[n]), kind


@pytest.mark.parametrize("precision", [cpapr.CPAPR_FP64, cpapr.CPAPR_FP32])
@pytest.mark.parametrize("bad", [-1.0, np.nan, np.inf])
def test_bad_lambda_leaves_the_model_and_bad_factors_drop_it(precision, bad):
    rank = 5
    fs = synth.random_factors(DIMS, rank, 3)
    lam = np.ones(rank)
    with context(rank, precision) as t:
        t.set_model(lam, fs)
        wrong = lam.copy()
        wrong[4] = bad
        with pytest.raises(cpapr.CpaprError) as e:
            t.set_model(wrong, [A * 2 for A in fs])
        assert e.value.status == 3
        for A, B in zip(fs, t.get_model()[1]):
            assert np.array_equal(A, B)
        wf = [A.copy() for A in fs]
        wf[1][19, 4] = bad
        with pytest.raises(cpapr.CpaprError) as e:
            t.set_model(lam, wf)
        assert e.value.status == 3
        with pytest.raises(cpapr.CpaprError) as e:
            t.phi(0)
        assert e.value.status == 7


def test_many_contexts_come_and_go():
    """More contexts than a block of page-locked slots holds, destroyed in another order."""
    ts = [context(2, cpapr.CPAPR_FP64) for _ in range(70)]
    for t in ts:
        t.init_random(1)
    want = ts[0].loglik()
    for k in list(range(0, 70, 2)) + list(range(1, 69, 2)):
        ts[k].close()
    assert ts[69].loglik() == want
    ts[69].close()
    with context(2, cpapr.CPAPR_FP64) as t:
        t.init_random(1)
        assert t.loglik() == want
