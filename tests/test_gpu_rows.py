"""The row interpolation (interp.cu) against the FP64 oracle: every width, one channel (the tap
kernel) to more than a launch's group of channels, windows that wrap on every side, grids of 2 W
points, a pair of coils and a single one, and the same kernel in a batched call.  Tolerance:
FP32_BOUND of test_gpu_parity."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import nufft as O
from tests.test_gpu_parity import FP32_BOUND, assert_close, make_case, t

pytestmark = pytest.mark.gpu
ROWS = {"interp_tiled": 0, "interp_threads": 256}


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2408_02367_gb300 import build
    build.build()
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


@pytest.mark.parametrize("K", [1, 5, 9])
@pytest.mark.parametrize("W,sigma,n", [(2, 1.25, (2, 13, 20)), (3, 2.0, (3, 8, 11)), (4, 1.25, (13, 6, 21)),
                                       (5, 2.0, (5, 9, 8)), (6, 2.0, (6, 7, 12)), (7, 2.0, (7, 8, 9)), (8, 2.0, (8, 9, 10))])
def test_row_interpolation_matches_oracle(W, sigma, n, K):
    from paper_2408_02367_gb300 import op
    c = make_case(n, W, sigma, K, 3, 2 * K, 1, 150, [2, 0, 1])
    geo = O.Geometry(c["n"], W, sigma)
    A = op.make_operator(c["omega"], c["frame"], n, W, sigma, c["V"], c["S"], max_batch=3, tuning=ROWS)
    y = A.forward(t(c["x"]), t(c["coils"]))
    assert_close(y.cpu().numpy(), O.gridding_forward(geo, c["x"], c["S"], c["V"], c["omega"], c["frame"], c["coils"]),
                 FP32_BOUND, f"W={W} M={geo.M} K={K} rows")
    if K > 1:
        part = A.forward(t(c["x"]), t(c["coils"]), k0=0, nk=1)
        A.forward(t(c["x"]), t(c["coils"]), out=part, accumulate=True, k0=1, nk=K - 1)
        assert_close(part.cpu().numpy(), y.cpu().numpy(), FP32_BOUND, "channel subsets")
    assert A.status() == 0


@pytest.mark.parametrize("W,sigma,n,K", [(4, 1.25, (38, 51, 64), 5), (6, 2.0, (24, 32, 40), 5), (4, 1.25, (38, 51, 64), 1),
                                         (6, 2.0, (24, 32, 40), 1)])
def test_batched_row_interpolation_equals_single_calls(W, sigma, n, K):
    """Two plans, three items in one launch per stage: each item's bits are its single call's, one
    channel (the tap kernel) included."""
    from paper_2408_02367_gb300 import op
    c = make_case(n, W, sigma, K, 3, 10, 1, 150, [2, 0, 1])
    plans = [op.make_operator(c["omega"], c["frame"], n, W, sigma, c["V"], c["S"], max_batch=3, tuning=ROWS)
             for _ in range(2)]
    x = t(c["x"])
    items = [(A, x, t(np.array(cs, np.int32)), None) for A, cs in zip(plans + plans[:1], ([2, 0], [1], [1]))]
    n0 = op.launch_count()
    ys = op.forward_batched(items)
    assert op.launch_count() - n0 == 4
    for (A, _, ci, _), y in zip(items, ys):
        assert torch.equal(y, A.forward(x, ci))
    assert all(A.status() == 0 for A in plans)


def _runs_tiled(A, x, ci):
    """Whether a forward runs the tiled interpolation: its test hook withholds a tile's row, so that
    the call reports a timeout (after 2 ms); the row kernels have no such wait."""
    A.set_wait_test(0, timeout_ns=2_000_000)
    A.forward(x, ci)
    timed_out = A.status() == 4
    A.set_wait_test(-1, timeout_ns=0)
    return timed_out


@pytest.mark.parametrize("tuning,tiled", [(None, True), ({"interp_tiled": 1}, True), ({"interp_tiled": 0}, False),
                                          ({"fft_staged": 3}, False), ({"interp_tiled": 1, "interp_run": 2}, True)])
def test_a_tuning_says_which_interpolation_runs(tuning, tiled):
    """interp_tiled = 0, also by default in a tuning, is the row kernel, 1 the tiled one; a plan without
    a tuning chooses (five channels at W = 4: the tiled one).  The plan reports what it runs."""
    from paper_2408_02367_gb300 import op
    c = make_case((20, 18, 16), 4, 1.25, 5, 2, 10, 1, 150, [1, 0])
    A = op.make_operator(c["omega"], c["frame"], c["n"], 4, 1.25, c["V"], c["S"], max_batch=2, tuning=tuning)
    assert A.tuning["interp_tiled"] == int(tiled)
    assert _runs_tiled(A, t(c["x"]), t(c["coils"])) == tiled
    assert A.status() == 0


@pytest.mark.parametrize("W,K,tiled", [(2, 3, True), (2, 4, False), (3, 7, True), (3, 8, False), (4, 1, True), (4, 7, True),
                                       (4, 8, False), (5, 1, False), (5, 2, True), (6, 1, False), (6, 8, True), (8, 1, False),
                                       (8, 2, True), (4, 9, False)])
def test_plans_without_a_tuning_take_the_faster_interpolation(W, K, tiled, max_batch=2, n=(16, 14, 18)):
    """Both sides of every line of the rule; the call agrees with the oracle either way, and a plan with
    the reported tuning gives equal bits."""
    from paper_2408_02367_gb300 import op
    sigma = 1.25 if W <= 4 else 2.0
    c = make_case(n, W, sigma, K, 2, 2 * K, 1, 120, [1, 0])
    coils = c["coils"][:max_batch]
    A = op.make_operator(c["omega"], c["frame"], n, W, sigma, c["V"], c["S"], max_batch=max_batch)
    x, ci = t(c["x"]), t(coils)
    y = A.forward(x, ci)
    assert_close(y.cpu().numpy(), O.gridding_forward(O.Geometry(n, W, sigma), c["x"], c["S"], c["V"], c["omega"],
                                                     c["frame"], coils), FP32_BOUND, f"W={W} K={K}")
    B = op.make_operator(c["omega"], c["frame"], n, W, sigma, c["V"], c["S"], max_batch=max_batch, tuning=A.tuning)
    assert torch.equal(B.forward(x, ci), y) and B.tuning == A.tuning
    assert _runs_tiled(A, x, ci) == tiled
    assert A.status() == 0 and B.status() == 0


@pytest.mark.parametrize("W,n,tiled", [(4, (16, 14, 18), True), (5, (16, 14, 18), True), (6, (16, 14, 18), True),
                                       (7, (16, 14, 18), True), (8, (16, 14, 18), False), (8, (32, 30, 32), False),
                                       (8, (32, 32, 32), True)])
def test_one_channel_plans_of_one_coil(W, n, tiled):
    """As above for plans whose calls have one coil (as the density compensation's)."""
    test_plans_without_a_tuning_take_the_faster_interpolation(W, 1, tiled, max_batch=1, n=n)
