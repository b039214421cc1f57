"""cpapr_phi_noalloc accepts a mode whenever some tiles of its launches leave room
in the fixed scratch: at padded rank 128 the float-pair launches take 512
nonzeros a tile (14.6 MB of partial rows here), the mode's others 1024 (7.3 MB)."""
import numpy as np
import pytest

from paper_2307_03276_gb300 import cpapr, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_2307_03276_gb300 import build
    build.build()


@pytest.mark.parametrize("pi_mode", [cpapr.CPAPR_PI_FUSED, cpapr.CPAPR_PI_MATERIALISED])
def test_scratch_fits_with_the_modes_larger_tiles(pi_mode):
    import torch
    nnz, dims, rank = 3_650_000, (4000, 3000, 500), 70
    assert 2 * -(-nnz // 1024) * 128 * 8 <= 8 << 20 < 2 * -(-nnz // 512) * 128 * 8
    rng = np.random.default_rng(21)
    idx = np.stack([np.minimum((rng.random(nnz) ** 3 * d).astype(np.int64), d - 1) for d in dims])
    vals = rng.integers(1, 6, nnz).astype(np.float64)
    with cpapr.Tensor(dims, idx, vals, rank, pi_mode=pi_mode) as t:
        t.set_model(np.ones(rank), synth.random_factors(dims, rank, 3))
        for n in (0, 2):
            want = t.phi(n)
            out = torch.full((dims[n], rank), float("nan"), dtype=torch.float64, device="cuda")
            torch.cuda.synchronize()
            cpapr.cpapr_phi_noalloc(t.ctx, n, out)
            # the same terms in another order of partial sums: each within 1e-12 of the exact sum
            got = out.cpu().numpy()
            assert np.all(np.abs(got - want) <= 2e-12 * np.abs(want)), n
