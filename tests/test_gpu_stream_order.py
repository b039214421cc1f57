"""Device inputs written by work still queued on the default stream when the call
is made: the context's own stream has to read them after it."""
import numpy as np
import pytest

from paper_2307_03276_gb300 import cpapr, synth

pytestmark = pytest.mark.gpu
DIMS, RANK, NNZ = (3000, 200, 100), 7, 20_000
SPIN = 200_000_000  # cycles of a busy kernel in front of the writes: about a tenth of a second


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_2307_03276_gb300 import build
    build.build()


def late(torch, a):
    """A device buffer of ones whose real contents, a, are queued behind a busy kernel."""
    src = torch.from_numpy(np.ascontiguousarray(a)).cuda()
    dst = torch.ones_like(src)
    return src, dst


@pytest.mark.parametrize("precision", [cpapr.CPAPR_FP64, cpapr.CPAPR_FP32])
@pytest.mark.parametrize("lam_on", ["host", "device"])
def test_inputs_queued_on_the_default_stream_are_complete(precision, lam_on):
    import torch
    T = synth.random_tensor(DIMS, NNZ, RANK, 12)
    fs = [np.ascontiguousarray(A) for A in synth.random_factors(DIMS, RANK, 3)]
    lam = np.linspace(0.5, 2.0, RANK)
    Bm = fs[1] * 1.25
    with cpapr.Tensor(DIMS, T.idx, T.vals, RANK, precision=precision) as t:
        t.set_model(lam, fs)
        want, want_b = t.phi(0), t.phi(1, B=Bm)
        t.set_model(np.ones(RANK), [np.ones_like(A) for A in fs])
        bufs = [late(torch, a) for a in [lam] + fs]
        torch.cuda.synchronize()
        torch.cuda._sleep(SPIN)
        for src, dst in bufs:
            dst.copy_(src)
        t.set_model(lam if lam_on == "host" else bufs[0][1], [d for _, d in bufs[1:]])
        lg, fg = t.get_model()
        assert np.array_equal(lg, lam)
        for A, G in zip(fs, fg):
            assert np.array_equal(A, G)
        assert np.array_equal(t.phi(0), want)
        src, dst = late(torch, Bm)
        torch.cuda.synchronize()
        torch.cuda._sleep(SPIN)
        dst.copy_(src)
        assert np.array_equal(t.phi(1, B=dst), want_b)


def test_a_tensor_queued_on_the_default_stream_is_complete():
    import torch
    T = synth.random_tensor(DIMS, NNZ, RANK, 13)
    fs = synth.random_factors(DIMS, RANK, 4)
    with cpapr.Tensor(DIMS, T.idx, T.vals, RANK) as t:
        t.set_model(np.ones(RANK), fs)
        want = t.phi(0)
    idx = [late(torch, np.asarray(r, dtype=np.int64)) for r in T.idx]
    vals = late(torch, T.vals)
    torch.cuda.synchronize()
    torch.cuda._sleep(SPIN)
    for src, dst in idx + [vals]:
        dst.copy_(src)
    with cpapr.Tensor(DIMS, [d for _, d in idx], vals[1], RANK) as t:
        t.set_model(np.ones(RANK), fs)
        assert np.array_equal(t.phi(0), want)
