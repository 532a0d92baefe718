"""The tuning that a plan reports."""
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


@pytest.mark.parametrize("n,W,sigma,K", [((40, 36, 44), 4, 1.25, 5), ((16, 12, 20), 6, 2.0, 3), ((12, 13, 40), 3, 1.5, 1)])
@pytest.mark.parametrize("tuning", [None, {}, {"spread_bins": (4, 4, 4), "spread_chunk": 64, "spread_coils": 1},
                                    {"interp_tiled": 1, "fft_staged": 3, "spread_chunk": 1024}])
def test_a_plan_with_the_reported_tuning_is_the_same_plan(n, W, sigma, K, tuning):
    """Same facts (units, subproblems, incidences, memory), same report, equal bits both ways."""
    from paper_2408_02367_gb300 import op
    c = make_case(n, W, sigma, K, 3, 2 * K + 4, 1, 700, [2, 0, 1])
    make = lambda tn: op.make_operator(c["omega"], c["frame"], n, W, sigma, c["V"], c["S"], 3, tuning=tn)  # noqa: E731
    A = make(tuning)
    B = make(A.tuning)
    assert B.tuning == A.tuning and B.info() == A.info()
    x, ci = t(c["x"]), t(c["coils"])
    r = t(synth.random_complex((3, A.J), 5))
    assert torch.equal(A.forward(x, ci), B.forward(x, ci))
    assert torch.equal(A.adjoint(r, ci), B.adjoint(r, ci))
    assert A.status() == 0 and B.status() == 0
