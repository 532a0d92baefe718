"""The kernels at the edges of their shapes, against the FP64 oracle: the spread's units (every
width, one and several channel groups, grids shorter than a unit and not a multiple of one, chunks
down to 32 incidences), the tiled interpolation (every width, tiles that wrap on every side), every
two-pass FFT length, the strided passes' tensor-load kernel and the large batches' route, and the
dictionary's last, partly filled tile.

Tolerance: FP32_BOUND of test_gpu_parity (2e-5 relative L2, 10 times that per element), and equal
bits where the same arithmetic runs in another kernel or minibatch.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import dm as DM
from oracle import nufft as O
from paper_2408_02367_gb300 import synth
from tests.test_gpu_parity import FP32_BOUND, assert_close, make_case, t

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2408_02367_gb300 import build
    build.build()
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


@pytest.mark.parametrize("W,sigma,n,K,chunk", [
    (2, 1.25, (2, 3, 30), 1, 32), (2, 2.0, (8, 9, 20), 5, 64), (3, 1.5, (6, 5, 9), 8, 32), (3, 2.0, (7, 9, 12), 2, 512),
    (4, 1.25, (17, 15, 9), 5, 32), (4, 2.0, (4, 6, 23), 7, 32), (5, 2.0, (9, 7, 11), 5, 32), (5, 1.5, (10, 12, 21), 1, 64),
    (6, 2.0, (13, 9, 7), 8, 32), (6, 2.0, (6, 7, 25), 3, 64), (7, 2.0, (9, 11, 8), 4, 32), (8, 2.0, (8, 9, 13), 6, 32),
    (8, 2.0, (9, 8, 12), 11, 64)])
@pytest.mark.parametrize("seg", [4, 8])
def test_spread_units_match_oracle(W, sigma, n, K, chunk, seg):
    """Three coils (a pair and a single): the adjoint against the oracle, and each coil's own call
    giving the same bits as the same coil repeated in a pair."""
    from paper_2408_02367_gb300 import op
    c = make_case(n, W, sigma, K, 3, 2 * K, 1, 150, [2, 0, 1])
    geo = O.Geometry(c["n"], W, sigma)
    A = op.make_operator(c["omega"], c["frame"], n, W, sigma, c["V"], c["S"], max_batch=3,
                         tuning={"spread_bins": (4, 4, seg), "spread_chunk": chunk})
    r = synth.random_complex((3, A.J), 3)
    a = A.adjoint(t(r), t(c["coils"]))
    assert_close(a.cpu().numpy(), O.gridding_adjoint(geo, r, c["S"], c["V"], c["omega"], c["frame"], c["coils"]),
                 FP32_BOUND, f"W={W} M={geo.M} K={K} adjoint")
    one = A.adjoint(t(r[:1]), t(c["coils"][:1]))
    pair = A.adjoint(t(np.concatenate([r[:1], np.zeros_like(r[:1])])), t(c["coils"][:2]))
    assert torch.equal(one + 0.0, pair + 0.0)          # (the second coil adds zeros; -0 + 0 = 0)
    assert torch.equal(A.adjoint(t(r), t(c["coils"])), a)
    assert A.status() == 0


@pytest.mark.parametrize("W,sigma,n,K", [
    (2, 1.25, (13, 14, 21), 8), (3, 2.0, (8, 11, 9), 5), (4, 1.25, (13, 26, 15), 5), (4, 2.0, (9, 8, 12), 1),
    (5, 2.0, (8, 10, 9), 7), (6, 2.0, (8, 9, 17), 5), (6, 2.0, (12, 8, 8), 8), (7, 2.0, (8, 9, 8), 7),
    (7, 2.0, (9, 8, 8), 8), (8, 2.0, (8, 9, 10), 6), (8, 2.0, (9, 8, 8), 7)])
def test_tiled_interpolation_widths_match_oracle(W, sigma, n, K):
    """Grids of 16 points and a little more along an axis (every tile wraps), and the sizes past which
    a tile no longer fits the shared memory (W=7 K=8, W=8 K=7: the row kernel); a channel subset added
    onto the rest gives the whole."""
    from paper_2408_02367_gb300 import op
    c = make_case(n, W, sigma, K, 2, 2 * K, 1, 200, [1, 0])
    geo = O.Geometry(c["n"], W, sigma)
    A = op.make_operator(c["omega"], c["frame"], n, W, sigma, c["V"], c["S"], max_batch=2)
    ci = t(c["coils"])
    y = A.forward(t(c["x"]), ci)
    assert min(geo.M) >= 16
    assert_close(y.cpu().numpy(), O.gridding_forward(geo, c["x"], c["S"], c["V"], c["omega"], c["frame"], c["coils"]),
                 FP32_BOUND, f"W={W} M={geo.M} K={K} forward")
    if K > 1:
        part = A.forward(t(c["x"]), ci, k0=0, nk=1)
        A.forward(t(c["x"]), ci, out=part, accumulate=True, k0=1, nk=K - 1)
        assert_close(part.cpu().numpy(), y.cpu().numpy(), FP32_BOUND, "channel subsets")
    assert A.status() == 0


LENGTHS = (20, 24, 30, 32, 36, 40, 48, 50, 54, 60, 64, 72, 80, 90, 96, 100, 108, 120, 128, 144, 150, 160, 162, 180, 192,
           200, 216, 240, 250, 256, 270, 288, 300, 320)


@pytest.mark.parametrize("L", LENGTHS)
def test_every_two_pass_length_matches_oracle(L):
    """Length L along axis 1 (strided) and axis 3 (fused), forward and adjoint, staged and direct."""
    from paper_2408_02367_gb300 import op
    n1 = int(L / 1.25)
    for n in ((n1, 6, 8), (8, 6, n1)):
        c = make_case(n, 4, 1.25, 2, 2, 4, 1, 100, [1, 0])
        geo = O.Geometry(c["n"], 4, 1.25)
        assert L in geo.M
        y_ref = O.gridding_forward(geo, c["x"], c["S"], c["V"], c["omega"], c["frame"], c["coils"])
        r = synth.random_complex(y_ref.shape, 5)
        a_ref = O.gridding_adjoint(geo, r, c["S"], c["V"], c["omega"], c["frame"], c["coils"])
        for staged in (0, 3):
            A = op.make_operator(c["omega"], c["frame"], n, 4, 1.25, c["V"], c["S"], max_batch=2,
                                 tuning={"fft_staged": staged})
            assert_close(A.forward(t(c["x"]), t(c["coils"])).cpu().numpy(), y_ref, FP32_BOUND, f"L={L} forward")
            assert_close(A.adjoint(t(r), t(c["coils"])).cpu().numpy(), a_ref, FP32_BOUND, f"L={L} adjoint")
            assert A.status() == 0


@pytest.mark.parametrize("n", [(128, 128, 96), (96, 64, 128)])
def test_tensor_load_passes_and_large_batches_equal_the_direct_kernels(n):
    """Strided passes with enough units for the tensor-load kernel (its last column block partly off
    the grid's end at K = 1), against a batch of the same item small enough for the direct kernels:
    equal bits; and a batch past 2^25 grid values (each plan's own kernels on worker streams), with
    two plans adding into one image in item order."""
    from paper_2408_02367_gb300 import op
    for K in (5, 1):
        c = make_case(n, 4, 1.25, K, 4, 10, 1, 300, [3, 1])
        A = op.make_operator(c["omega"], c["frame"], n, 4, 1.25, c["V"], c["S"], max_batch=4)
        A2 = op.make_operator(c["omega"], c["frame"], n, 4, 1.25, c["V"], c["S"], max_batch=4)
        x, ci, one = t(c["x"]), t(c["coils"]), t(c["coils"][:1])
        y1 = A.forward(x, one)
        y2 = op.forward_batched([(A2, x, one, None)])[0]
        assert torch.equal(y1, y2)
        assert torch.equal(A.adjoint(y1, one), op.adjoint_batched([(A2, y1, one, None, False)])[0])
    G = int(np.prod(A.grid))
    big = t(np.array([0, 1, 2, 3], np.int32))
    c = make_case(n, 4, 1.25, 5, 4, 10, 1, 300, [3, 1])
    A = op.make_operator(c["omega"], c["frame"], n, 4, 1.25, c["V"], c["S"], max_batch=4)
    A2 = op.make_operator(c["omega"], c["frame"], n, 4, 1.25, c["V"], c["S"], max_batch=4)
    assert 2 * 4 * 5 * G > 2 ** 25
    x = t(c["x"])
    ys = op.forward_batched([(A, x, big, None), (A2, x, big, None)])
    assert torch.equal(ys[0], A.forward(x, big)) and torch.equal(ys[0], ys[1])
    acc = torch.zeros_like(x)
    op.adjoint_batched([(A, ys[0], big, acc, True), (A2, ys[1], big, acc, True)])
    ref = A.adjoint(ys[0], big)
    assert torch.equal(acc, ref + ref)
    assert A.status() == 0 and A2.status() == 0


@pytest.mark.parametrize("P", [1, 31, 33, 64, 65, 129, 200])
def test_matching_dictionaries_around_a_tile(P):
    """Atoms that fill one, two or three 64-atom tiles partly: one tile leaves an epilogue buffer
    without work, an odd number of tiles alternates the buffers from step to step."""
    from paper_2408_02367_gb300 import dm
    rng = np.random.default_rng(P)
    atoms = (rng.standard_normal((P, 4)) + 1j * rng.standard_normal((P, 4))).astype(np.complex64)
    x, _, _ = synth.dm_volume(atoms, 152 * 256 + 300, noise=0.0, seed=P)     # more than one step per CTA
    M = dm.DictionaryMatcher(t(atoms), max_vox=x.shape[1])
    idx, pd = M.match(t(x))
    ref_idx, ref_pd = DM.dictionary_match(x, atoms)
    assert np.array_equal(idx.cpu().numpy(), ref_idx)
    assert np.max(np.abs(pd.cpu().numpy() - ref_pd) / np.abs(ref_pd)) < 2e-5
    assert M.status() == 0
