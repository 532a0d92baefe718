"""How long the float32 chains of the adjoint's sums are, against the FP64 oracle."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import nufft as O

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2408_02367_gb300 import build
    build.build()
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


@pytest.mark.parametrize("bins", [(4, 4, 4), (4, 4, 8)])
def test_equal_samples_sum_in_short_chains(bins):
    """64 positions with 4096 equal samples each, in chunks of up to 512: every grid point adds the
    same value again and again, so a chain of N additions drifts by its rounding in one direction.
    The chains run in numpy (float32, partial sums of eight, then of those) and taken through the
    oracle's remaining steps give a relative L2 error of 7.8e-6 to 8.6e-6 with N = 512 and 4.1e-6 to
    4.2e-6 with N = 256 over three seeds; the bound of 6e-6 leaves the weights' and the FFT's own
    1.2e-6 room beside the second.  The oracle takes each position once, with 4096 times its value."""
    from paper_2408_02367_gb300 import op
    rng = np.random.default_rng(3)
    n, W, sigma, P, R = (24, 20, 28), 4, 1.25, 64, 4096
    om = rng.uniform(-2.8, 2.8, (P, 3)).astype(np.float32)
    V = np.array([[0.7 + 0.2j, -0.3 + 0.9j]], np.complex64)
    S = np.ones((2,) + n, np.complex64)
    r = (rng.standard_normal(P) + 1j * rng.standard_normal(P)).astype(np.complex64)
    coils = np.array([0, 1], np.int32)
    A = op.make_operator(np.repeat(om, R, 0), np.zeros(P * R, np.int64), n, W, sigma, V, S, max_batch=2,
                         tuning={"spread_bins": bins, "spread_chunk": 512})
    y = torch.from_numpy(np.repeat(r, R)).cuda().repeat(2, 1).contiguous()
    a = A.adjoint(y, torch.from_numpy(coils).cuda()).cpu().numpy()
    ref = O.gridding_adjoint(O.Geometry(n, W, sigma), np.stack([r, r]).astype(np.complex128) * R, S, V, om,
                             np.zeros(P, np.int64), coils)
    assert np.linalg.norm(a - ref) <= 6e-6 * np.linalg.norm(ref)
    assert A.status() == 0
