// Integer maps of the spread's units (spread_impl.cuh), of the interpolation's tiles
// (interp_tiles.cu) and of the plan tables that feed both (api.cu).  Kept in one place,
// compiled into the plan and the kernels and, for the tests, into a host library that
// enumerates them over widths, short axes and cut last units.
#pragma once

#if !defined(SDP_MAP)
#if defined(__CUDACC__)
#define SDP_MAP __host__ __device__ __forceinline__
#else
#define SDP_MAP inline
#endif
#endif

namespace sdp {
namespace imap {

// ---------------- units met by a window ----------------
// Along an axis of M points cut into units of `edge`, a window has the taps m, m + 1, ..,
// m + W - 1 (mod M).  f(unit, k) is called for every piece of it that lies in one unit:
//   - axes 1 and 2 (edge 4), once per unit: unit_tap(W, k, x) is the tap at position x;
//   - axis 3, k the plane r at which the window starts: position x has tap x - r + W - 1.  On
//     an axis shorter than edge + W - 1 points a window can meet a unit in two pieces, the
//     second's plane one grid length further.
template <class F>
inline void unit_meets(int W, int M, int edge, bool axis3, int m, F&& f) {
    for (int t = 0; t < W; ++t) {
        const int u = (m + t) % M / edge;
        bool seen = false;
        for (int s = 0; s < t; ++s) seen = seen || (m + s) % M / edge == u;
        if (seen) continue;
        int d = u * edge - m;   // tap of the unit's first position, wrapped
        d += d < 0 ? M : 0;
        if (axis3) {
            const int points = M - u * edge < edge ? M - u * edge : edge;
            const int top = points + W - 2;   // last plane with a window in the unit
            int r = m - u * edge + W - 1;
            r += r < 0 ? M : 0;
            r -= r >= M ? M : 0;
            for (; r <= top; r += M) f(u, r);
        } else if (W == 2) {   // a 4-point axis: the window may meet the unit in two pieces
            int k = 0;
            for (int x = 0; x < 4; ++x) {
                const int tap = (d + x) % M;
                k |= (tap < 2 ? tap + 1 : 0) << (2 * x);
            }
            f(u, k);
        } else {               // M >= 2 W >= W + 3: one piece
            f(u, (d < W ? d : d - M) + 3);
        }
    }
}

// Tap at position x (0 .. 3) of a unit along axis 1 or 2; outside [0, W): none.
SDP_MAP int unit_tap(int W, int k, int x) { return W == 2 ? ((k >> (2 * x)) & 3) - 1 : x + k - 3; }

// First and last block of four positions of a unit (seg points) that planes r0 .. r1 reach.
SDP_MAP int spread_block_lo(int r0, int W) { return r0 < W - 1 ? 0 : (r0 - (W - 1)) >> 2; }
SDP_MAP int spread_block_hi(int r1, int seg) { return (r1 < seg - 1 ? r1 : seg - 1) >> 2; }

// ---------------- interpolation tiles ----------------
// Tile edges in grid points: 8 along axes 2 and 3, and along axis 1 up to W = 5; from W = 6 on 4
// (interp_tiles.cu).
constexpr int kTileEdge = 8;
SDP_MAP constexpr int tile_edge(int W, int axis) { return axis == 0 && W >= 6 ? 4 : kTileEdge; }

// Points before a tile's own along an axis, W / 2, along axis 3 made even (16-byte rows); and the
// points that are copied, the tile with the margins of its windows, along axis 3 even too.
SDP_MAP constexpr int tile_before(int W, int axis) { return axis == 2 ? (W / 2 + 1) & ~1 : W / 2; }
SDP_MAP constexpr int tile_points(int W, int axis) {
    return axis == 2 ? (kTileEdge + W + tile_before(W, 2) - W / 2 + 1) & ~1 : tile_edge(W, axis) + W;
}

// Point of the tile at which a window starts whose first tap along axis d is e_d + the tile's first
// point - W / 2, 0 <= e_d <= tile_edge(W, d), without axis 3's extra point before.
SDP_MAP constexpr int tile_start(int W, int e1, int e2, int e3) {
    return (e1 * tile_points(W, 1) + e2) * tile_points(W, 2) + e3;
}

}  // namespace imap
}  // namespace sdp
