"""Calls of several host threads and streams that share the library: each gives what it gives alone."""
import threading

import numpy as np
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


def _plan(n, K, maxB=1, **kw):
    from paper_2408_02367_gb300 import op
    c = make_case(n, 4, 1.25, K, 2, 2 * K, 1, 60, [1])
    return op.make_operator(c["omega"], c["frame"], n, 4, 1.25, c["V"], c["S"], max_batch=maxB, **kw), t(c["x"])


def test_staged_kernels_of_two_threads_keep_their_shared_memory():
    """One and five channels on an axis-3 grid of 160 points run the same staged axis-3 kernels with
    different amounts of shared memory: two threads that call them at the same time are never refused
    a launch, and every result is the one the thread had alone."""
    ci = torch.tensor([1], dtype=torch.int32, device="cuda")
    work = []
    for K in (1, 5):
        A, x = _plan((16, 16, 128), K, tuning={"fft_staged": 3})
        y = A.forward(x, ci)
        work.append((A, x, y, A.adjoint(y, ci)))
    torch.cuda.synchronize()
    errors = []

    def loop(A, x, y, a):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                y2, a2 = torch.empty_like(y), torch.empty_like(a)
                for _ in range(3000):
                    A.forward(x, ci, out=y2)
                    A.adjoint(y, ci, out=a2)
                torch.cuda.current_stream().synchronize()
                assert torch.equal(y, y2) and torch.equal(a, a2)
        except BaseException as e:      # a thread's failure is the test's
            errors.append(e)

    threads = [threading.Thread(target=loop, args=w) for w in work]
    for th in threads:
        th.start()
    for th in threads:
        th.join()
    assert not errors, errors
    assert all(w[0].status() == 0 for w in work)


def _items(plans, B):
    ci = torch.arange(B, dtype=torch.int32, device="cuda")
    return [(A, x, ci, torch.empty((B, A.J), dtype=torch.complex64, device="cuda")) for A, x in plans]


def _adjoints(items):
    return [(A, y, c, torch.empty_like(x), False) for A, x, c, y in items]


def test_batch_beside_the_capture_of_another():
    """A batch past 2^25 grid values (128 x 96 x 96 images on 160 x 120 x 120 grids, four items of
    two coils on two plans) is captured; before the capture ends, batches of other plans, a large one and one that never
    takes the fused form (W = 4 and 6 mixed), run on another stream.  None of them fails, and the eager
    results and the replay's are the single calls'."""
    from paper_2408_02367_gb300 import op
    n = (128, 96, 96)
    plans = [_plan(n, 5, 2) for _ in range(4)]
    assert 2 * 4 * 5 * int(np.prod(plans[0][0].grid)) > 2 ** 25
    c6 = make_case((24, 24, 24), 6, 2.0, 5, 2, 10, 1, 60, [1])
    small = (op.make_operator(c6["omega"], c6["frame"], (24, 24, 24), 6, 2.0, c6["V"], c6["S"], max_batch=1), t(c6["x"]))
    captured, eager = _items(plans[:2], 2) + _items(plans[:2], 2), _items(plans[2:], 2) + _items(plans[2:], 2)
    mixed = _items(plans[2:3], 1) + _items([small], 1)
    back, eager_back = _adjoints(captured), _adjoints(eager)
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, capture_error_mode="thread_local"):
        op.forward_batched(captured)
        op.adjoint_batched(back)
        with torch.cuda.stream(side):
            op.forward_batched(eager)
            op.adjoint_batched(eager_back)
            op.forward_batched(mixed)
    side.synchronize()
    for A, x, c, y in eager + mixed:
        assert torch.equal(y, A.forward(x, c))
    for A, y, c, a, _ in eager_back:
        assert torch.equal(a, A.adjoint(y, c))
    g.replay()
    torch.cuda.synchronize()
    for A, x, c, y in captured:
        assert torch.equal(y, A.forward(x, c))
    for A, y, c, a, _ in back:
        assert torch.equal(a, A.adjoint(y, c))
    assert all(A.status() == 0 for A, _ in plans + [small])


def test_large_batch_on_a_stream_of_another_priority():
    """The same results, item after item on the caller's stream."""
    from paper_2408_02367_gb300 import op
    plans = [_plan((128, 96, 96), 5, 2) for _ in range(2)]
    items = _items(plans, 2) + _items(plans, 2)
    torch.cuda.synchronize()
    st = torch.cuda.Stream(priority=-1)
    with torch.cuda.stream(st):
        op.forward_batched(items)
    st.synchronize()
    for A, x, c, y in items:
        assert torch.equal(y, A.forward(x, c))
