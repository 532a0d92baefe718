// Host build of paper_2408_02367_gb300/csrc/spread_map.cuh for the CPU tests in
// test_spread_map.py: the arithmetic that the plan and the kernels compile, not a
// restatement of it.  Nothing here runs on a GPU.
#include "spread_map.cuh"

using namespace sdp::imap;

extern "C" {

// out[2 i ..] = unit, k of the pieces of the window of first tap m; returns their number
int smap_unit_meets(int W, int M, int edge, int axis3, int m, int* out) {
    int n = 0;
    unit_meets(W, M, edge, axis3 != 0, m, [&](int unit, int k) {
        out[2 * n] = unit;
        out[2 * n + 1] = k;
        ++n;
    });
    return n;
}
int smap_unit_tap(int W, int k, int x) { return unit_tap(W, k, x); }
int smap_block_lo(int r0, int W) { return spread_block_lo(r0, W); }
int smap_block_hi(int r1, int seg) { return spread_block_hi(r1, seg); }
int smap_tile_edge(int W, int axis) { return tile_edge(W, axis); }
int smap_tile_before(int W, int axis) { return tile_before(W, axis); }
int smap_tile_points(int W, int axis) { return tile_points(W, axis); }
int smap_tile_start(int W, int e1, int e2, int e3) { return tile_start(W, e1, e2, e3); }

}  // extern "C"
