"""Which axis-3 kernels a plan without a tuning stages, and that it gives the same bits either way."""
import pytest

torch = pytest.importorskip("torch")

from paper_2408_02367_gb300 import synth
from tests.test_gpu_parity import make_case, t

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2408_02367_gb300 import build
    build.build()
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


@pytest.mark.parametrize("n3,sigma,K,mask", [
    (48, 1.25, 5, 0), (64, 1.25, 2, 0), (64, 1.25, 3, 2), (76, 1.25, 5, 1), (48, 2.0, 8, 0), (48, 2.0, 5, 1),
    (80, 1.25, 5, 2), (80, 1.25, 1, 2), (96, 1.25, 5, 3), (96, 1.25, 2, 1), (96, 1.25, 12, 2), (128, 1.25, 8, 3), (64, 2.0, 6, 2),
    (160, 1.25, 5, 3), (100, 2.0, 5, 2), (200, 1.25, 1, 3), (124, 2.0, 5, 3), (204, 1.25, 5, 2)])
def test_staged_kernels_of_a_plan_without_a_tuning(n3, sigma, K, mask):
    """Both sides of every line of the rule (axis-3 grids of 60, 80, 96, 100, 120, 128, 160, 200, 250 and 256
    points): the reported choice, and the bits of the plans that stage none and both."""
    from paper_2408_02367_gb300 import op
    n = (6, 9, n3)
    c = make_case(n, 4, sigma, K, 2, 2 * K, 1, 80, [1, 0])
    make = lambda tuning: op.make_operator(c["omega"], c["frame"], n, 4, sigma, c["V"], c["S"], 2, tuning=tuning)  # noqa: E731
    A = make(None)
    assert A.tuning["fft_staged"] == mask
    x, ci = t(c["x"]), t(c["coils"])
    r = t(synth.random_complex((2, A.J), 7))
    y, a = A.forward(x, ci), A.adjoint(r, ci)
    for staged in (0, 3):
        B = make(dict(A.tuning, fft_staged=staged))
        assert torch.equal(B.forward(x, ci), y) and torch.equal(B.adjoint(r, ci), a)
        assert B.status() == 0
    assert A.status() == 0
