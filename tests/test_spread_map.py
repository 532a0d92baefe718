"""The integer maps of the spread's units and the interpolation's tiles, enumerated on the CPU from
the header that the plan and the kernels compile (csrc/spread_map.cuh): every width, axes from the
shortest (2 W points) on, cut last units, and every first tap."""
import ctypes
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2408_02367_gb300", "csrc")
WIDTHS = range(2, 9)


@pytest.fixture(scope="module")
def so(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    lib = tmp_path_factory.mktemp("smap") / "libsmap.so"
    r = subprocess.run([cxx, "-std=c++17", "-O1", "-shared", "-fPIC", "-I", CSRC,
                        os.path.join(ROOT, "tests", "spread_map_shim.cpp"), "-o", str(lib)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return ctypes.CDLL(str(lib))


def meets(so, W, M, edge, axis3, m):
    buf = (ctypes.c_int * 64)()
    n = so.smap_unit_meets(W, M, edge, int(axis3), m, buf)
    return [(buf[2 * i], buf[2 * i + 1]) for i in range(n)]


def axis_lengths(W):
    return [M for M in (4, 6, 8, 10, 12, 14, 16, 18, 20, 24, 30, 36, 50) if M >= 2 * W]


@pytest.mark.parametrize("W", WIDTHS)
def test_units_of_axes_1_and_2_cover_every_window_once(so, W):
    """The taps at the positions of the units that a window meets are its W taps, each at its own grid
    point, each once (positions past the end of a cut last unit are off the grid and not stored);
    k fits the incidence's 8 bits."""
    for M in axis_lengths(W):
        for m in range(M):
            got = []
            for u, k in meets(so, W, M, 4, False, m):
                assert 0 <= u < -(-M // 4) and 0 <= k < 256
                for x in range(4):
                    tap = so.smap_unit_tap(W, k, x)
                    if 0 <= tap < W and 4 * u + x < M:
                        got.append((4 * u + x, tap))
            assert sorted(got) == sorted(((m + t) % M, t) for t in range(W)), (W, M, m)


@pytest.mark.parametrize("seg", [16, 32])
@pytest.mark.parametrize("W", WIDTHS)
def test_units_of_axis_3_cover_every_window_once(so, W, seg):
    """The same for the planes, two pieces of one unit included: position x of a piece with plane r has
    tap x - r + W - 1.  Planes stay within the seg + W - 1 that the plan's table has room for, and the
    positions that a plane reaches lie in the blocks that spread_block_lo and _hi name."""
    for M in axis_lengths(W) + [seg, seg + 2, seg + W - 1 + (seg + W - 1) % 2, 2 * seg + 4]:
        if M < 2 * W:
            continue
        two = 0
        for m in range(M):
            got, units = [], []
            for u, r in meets(so, W, M, seg, True, m):
                points = min(seg, M - seg * u)
                assert points > 0 and 0 <= r <= points + W - 2 < seg + W - 1
                units.append(u)
                lo, hi = so.smap_block_lo(r, W), so.smap_block_hi(r, points)
                reached = [x for x in range(points) if 0 <= x - r + W - 1 < W]
                assert lo == reached[0] // 4 and hi == reached[-1] // 4, (W, M, m, u, r)
                got += [(seg * u + x, x - r + W - 1) for x in reached]
            two += len(units) != len(set(units))
            assert sorted(got) == sorted(((m + t) % M, t) for t in range(W)), (W, M, m)
        if M < min(seg, M) + W - 1 and M <= seg:
            assert two > 0          # a window that wraps meets the only unit twice


@pytest.mark.parametrize("W", WIDTHS)
def test_windows_lie_in_their_tile(so, W):
    """For every window start of a tile (relative to the tile's first point less W / 2, up to the edge):
    the window's points lie in the tile's copy on every axis, its start is the flat index of its
    first point less axis 3's extra one, and rows start and end on even points (16 bytes of complex
    values)."""
    edge = [so.smap_tile_edge(W, a) for a in range(3)]
    pts = [so.smap_tile_points(W, a) for a in range(3)]
    before = [so.smap_tile_before(W, a) for a in range(3)]
    assert edge[1:] == [8, 8] and edge[0] in (4, 8) and pts[2] % 2 == 0 and before[2] % 2 == 0
    assert max(pts) <= 16           # an axis of 16 points: the copy wraps around it at most once
    for a in range(3):
        extra = before[a] - W // 2
        assert extra in ((0, 1) if a == 2 else (0,))
        for e in range(edge[a] + 1):
            assert extra + e + W <= pts[a]
    starts = {}
    for e1 in range(edge[0] + 1):
        for e2 in range(edge[1] + 1):
            for e3 in range(edge[2] + 1):
                s = so.smap_tile_start(W, e1, e2, e3)
                assert s == (e1 * pts[1] + e2) * pts[2] + e3
                assert starts.setdefault(s, (e1, e2, e3)) == (e1, e2, e3)
