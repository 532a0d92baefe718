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
