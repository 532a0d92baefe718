// Adjoint spreading (kernel template, included by the spread_*.cu translation
// units and batch_sp.cu) with the conjugate subspace weights (gridding step A5):
//
//   H_{b,k}[m mod M] = sum_j phi(g_j1 - m1) phi(g_j2 - m2) phi(g_j3 - m3) conj(V[t_j, k]) r_b[j]
//
// the first step of A_c^H, which Algorithm 1 of StoDIP needs for
// loss.backward() (Sec. 2.1, Eq. 3).  conj(V[t_j, k]) r_b[j] folds the
// temporal subspace into the spread, so only K channel grids are formed.
//
// Owner-computes units with a sliding window.  The grid is cut into units of
// 4 x 4 columns by `seg` points along axis 3.  The plan lists, per unit, every
// sample whose W^3 window touches it (the incidences), in order of the plane r
// at which the window starts along axis 3 (r = window start - lo3 + W - 1, so
// 0 <= r <= seg + W - 2), split into chunks of bounded length (the
// subproblems).  A CTA is ONE warp that takes one subproblem for NC coils.
// Lanes l and l + 16 own column ((l % 16) / 4, l % 4) of the unit, of which
// they keep only the W grid points that the current plane's windows cover, NK
// channels each, in a ring of registers: the warp runs all incidences of plane
// r (along axis 3 no multiply-add falls outside a window, and an incidence is
// met once per unit, not once per 4 points), then the oldest position is
// final, is written out, and the ring turns by one.  Ring slots are
// compile-time indices: the code has one copy per ring phase.
//   - two coils: half-warp h holds coil h, a ring of W positions;
//   - one coil: half-warp 0 holds the first half of the window's positions and
//     half-warp 1 the rest; as the ring turns, the oldest position of half-warp
//     1 moves to half-warp 0.
// Both sum every grid point over its incidences in the same order, so a coil's
// result does not depend on the minibatch it is in, bit for bit.
//
// What bounds it is the staging: its gathers read one cache line per lane, and
// without the multiply-adds the kernel takes the same time.  So the split is the
// one with the fewest incidences: with W = 4, 3.1 (seg + 3) / seg incidences per
// sample against 5.4 for 4 x 4 x 4 bins of fixed registers (344 us by default, 227
// tuned, at 128^3, two coils, five channels, against 190), and an incidence carries
// its sample's index and frame, so a round waits for two round trips (182 us; the
// sums by pairs, spread_together() below, are not hidden behind them: 197).
//
// Incidences are staged 32 at a time in shared memory: the 16 products of
// axis-1 and axis-2 weights (zero outside the window), the W axis-3 weights, and
// c_k = conj(V[t, k]) r_b for the warp's coils, one record of an odd number of
// 16-byte units per incidence, so the 16-byte stores of a quarter-warp fall on
// distinct banks.
// Finished positions are gathered four at a time in shared memory, a dense box
// of 4 x 4 columns by 4 points by NK channels per coil, which one thread sends
// to the grid (channel-interleaved, [b][i1][i2][i3][kk]) with one tensor store
// (cp.async.bulk.tensor); the edges of the grid are cut off by the tensor map.
// (The warp's own 16-byte stores, and a bulk copy per column, each cost 600 to
// 800 instructions per box: the bulk copies of a warp's lanes are issued one
// after the other.)  Calls on some of the plan's channels, plans of more than 8,
// and partial sums are stored by the warp.
// Finishing a unit:
//   - one chunk: the runs go straight into the grid;
//   - several chunks (the dense k-space centre): a chunk covers a range of
//     planes, so it writes partial sums of the blocks of four positions its
//     windows reach only; the last chunks to finish a block (device-scope counters
//     per block, no waiting) sum its partials in a fixed order and store it.  (One
//     counter per unit left a single warp summing a hundred whole partial tiles of
//     the k-space centre, 0.2 ms of the 128^3 spread.)
// Every grid point is written exactly once by plain stores: no zero fill of
// the grid, no atomics on it, and the result is bitwise repeatable.
#pragma once

#include "sdp_internal.cuh"
#include "spread_map.cuh"
#include "tma.cuh"

namespace sdp {
namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kCols = 16;   // columns of a unit (4 x 4)

__device__ __forceinline__ unsigned long long pack2(float x, float y) {
    unsigned long long r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(x), "f"(y));
    return r;
}

// A warp's shared memory for width W, NK channels and NC coils, in 16-byte units: 32 records
// of an odd stride, then the finished positions.
template <int W, int NK, int NC>
struct SpreadDims {
    static constexpr int kSlots = NC == 2 ? W : (W + 1) / 2;    // ring slots of a lane
    static constexpr int kCoef = (NK + 1) / 2;                  // a coil's coefficients
    static constexpr int kW3 = (kSlots + 3) / 4;                // a half-warp's axis-3 weights
    static constexpr int kOfsW3 = NC * kCoef;
    static constexpr int kOfsW12 = kOfsW3 + (NC == 2 ? 1 : 2) * kW3;
    static constexpr int kRec = (kOfsW12 + 4) | 1;
    static constexpr int kRun = 2 * NK;                         // a column's four positions
    static constexpr int kOut = NC * kCols * kRun;
    static constexpr int kAll = 32 * kRec + kOut;
};

// The weights of a unit's four positions along axis 1 or 2 from the W weights of a window, the taps
// of imap::unit_tap: v[u] = w[u + k - 3], 0 outside the window, k in [0, W + 2].  A barrel shift of the
// zero-padded window (compile-time indices keep it in registers).  W = 2, whose windows can
// meet a unit of a 4-point axis in two pieces: two bits of k per position, 1 + the tap.
template <int W>
__device__ __forceinline__ void window_at(const float* w, int k, float (&v)[4]) {
    if constexpr (W == 2) {
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int t = (k >> (2 * u)) & 3;
            v[u] = t == 1 ? w[0] : (t == 2 ? w[1] : 0.f);
        }
        return;
    }
    constexpr int N = W + 6;
    float c[N];
#pragma unroll
    for (int i = 0; i < N; ++i) c[i] = (i >= 3 && i < 3 + W) ? w[i - 3] : 0.f;
    int len = N;
#pragma unroll
    for (int s = 8; s >= 1; s >>= 1) {
        if (s <= W + 2) {
            const int nl = 3 + s;
            const bool sh = (k & s) != 0;
#pragma unroll
            for (int i = 0; i < nl; ++i) {
                const float far = i + s < len ? c[i + s] : 0.f;
                c[i] = sh ? far : (i < len ? c[i] : 0.f);
            }
            len = nl;
        }
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) v[u] = c[u];
}

// Incidences of a plane whose products are summed before they are added to the ring.  A chunk at the
// k-space centre adds up to 512 of them to one float32 value per point; two at a time halve that
// chain, at half as many instructions again (a multiply, a multiply-add and an add for two
// multiply-adds).  Error of the adjoint against 64 bits at 128^3, two coils, five channels: 1.47e-6
// one at a time, 1.12e-6 by pairs (4 x 4 x 4 bins of fixed registers, two chains per chunk, had
// 1.23e-6), for 182 -> 197 us; of eight volumes of 24^3 to 70 x 88 x 74 it falls by 11%.  Wider
// windows are bound by their multiply-adds (29 x 36 x 25, W = 6: 18% more time by pairs, for an
// error that is 0.6% smaller) and keep the single chain.
__host__ __device__ constexpr int spread_together(int W) { return W <= 5 ? 2 : 1; }

// acc += sum over g of wt[g][a] v[g] (its first or second value): the products of the G incidences
// are summed first, then added to the running sum once.
template <int G, int N>
__device__ __forceinline__ void add_products(unsigned long long& acc, const unsigned long long (&wt)[G][N],
                                             const ulonglong2 (&v)[G], int a, bool second) {
    if (G == 1) {
        asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc) : "l"(wt[0][a]), "l"(second ? v[0].y : v[0].x));
        return;
    }
    unsigned long long t;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(t) : "l"(wt[0][a]), "l"(second ? v[0].y : v[0].x));
#pragma unroll
    for (int g = 1; g < G; ++g)
        asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(t) : "l"(wt[g][a]), "l"(second ? v[g].y : v[g].x));
    asm("add.rn.f32x2 %0, %0, %1;" : "+l"(acc) : "l"(t));
}

// G incidences into the ring, the lane's positions starting at ring slot P: position a goes
// to slot (P + a) mod kSlots with weight w phi3(a), w = phi1 phi2 of the lane's column.
// `coef`, `w3` and `w12` point at the first record's values of the half-warp's coil, positions and column.
template <int P, int G, int W, int NK, int NC>
__device__ __forceinline__ void spread_add(unsigned long long (&acc)[SpreadDims<W, NK, NC>::kSlots][NK],
                                           const float4* coef, const float4* w3, const float* w12) {
    using D = SpreadDims<W, NK, NC>;
    constexpr int NS = D::kSlots, R = D::kRec;
    unsigned long long wt[G][4 * D::kW3];
#pragma unroll
    for (int g = 0; g < G; ++g) {
        const float w = w12[4 * R * g];
#pragma unroll
        for (int q = 0; q < D::kW3; ++q) {
            const float4 v = w3[R * g + q];
            const float wa = w * v.x, wb = w * v.y, wc = w * v.z, wd = w * v.w;
            wt[g][4 * q] = pack2(wa, wa);
            wt[g][4 * q + 1] = pack2(wb, wb);
            wt[g][4 * q + 2] = pack2(wc, wc);
            wt[g][4 * q + 3] = pack2(wd, wd);
        }
    }
    // acc += sum over g of ((w1 w2) w3) c, both components at once, two coefficients per load
#pragma unroll
    for (int m = 0; m < NK; m += 2) {
        ulonglong2 v[G];
#pragma unroll
        for (int g = 0; g < G; ++g) v[g] = *reinterpret_cast<const ulonglong2*>(coef + R * g + m / 2);
#pragma unroll
        for (int a = 0; a < NS; ++a) {
            add_products<G>(acc[(P + a) % NS][m], wt, v, a, false);
            if (m + 1 < NK) add_products<G>(acc[(P + a) % NS][m + 1 < NK ? m + 1 : m], wt, v, a, true);
        }
    }
}

// The staged incidences [i, e) of one plane.  coef, w3 and w12 point at record 0's
// values for the lane.
template <int P, int W, int NK, int NC>
__device__ __forceinline__ void spread_run(unsigned long long (&acc)[SpreadDims<W, NK, NC>::kSlots][NK],
                                           const float4* coef, const float4* w3, const float* w12, int i, int e) {
    constexpr int R = SpreadDims<W, NK, NC>::kRec;
    coef += i * R;
    w3 += i * R;
    w12 += i * (4 * R);
    constexpr int G = spread_together(W);
    int n = e - i;
#pragma unroll 1
    for (; n > 1; n -= 2) {
        if constexpr (G == 2) {
            spread_add<P, 2, W, NK, NC>(acc, coef, w3, w12);
        } else {
            spread_add<P, 1, W, NK, NC>(acc, coef, w3, w12);
            spread_add<P, 1, W, NK, NC>(acc, coef + R, w3 + R, w12 + 4 * R);
        }
        coef += 2 * R;
        w3 += 2 * R;
        w12 += 8 * R;
    }
    if (n > 0) spread_add<P, 1, W, NK, NC>(acc, coef, w3, w12);
}

template <int P, int W, int NK, int NC>
__device__ __forceinline__ void spread_plane(int ph, unsigned long long (&acc)[SpreadDims<W, NK, NC>::kSlots][NK],
                                             const float4* coef, const float4* w3, const float* w12, int i, int e) {
    if constexpr (P + 1 < SpreadDims<W, NK, NC>::kSlots) {
        if (ph == P)
            spread_run<P, W, NK, NC>(acc, coef, w3, w12, i, e);
        else
            spread_plane<P + 1, W, NK, NC>(ph, acc, coef, w3, w12, i, e);
    } else {
        spread_run<P, W, NK, NC>(acc, coef, w3, w12, i, e);
    }
}

// The position in ring slot P is final: its values into `out` (null: a position outside the
// unit), and the slot takes the next position (new, or half-warp 1's oldest).
template <int P, int W, int NK, int NC>
__device__ __forceinline__ void spread_take(int ph, unsigned long long (&acc)[SpreadDims<W, NK, NC>::kSlots][NK],
                                            unsigned long long* out, int h) {
    if constexpr (P + 1 < SpreadDims<W, NK, NC>::kSlots) {
        if (ph != P) {
            spread_take<P + 1, W, NK, NC>(ph, acc, out, h);
            return;
        }
    }
    if (out && (NC == 2 || h == 0)) {
#pragma unroll
        for (int q = 0; q < NK; ++q) out[q] = acc[P][q];
    }
#pragma unroll
    for (int q = 0; q < NK; ++q) {
        if constexpr (NC == 2) {
            acc[P][q] = 0ull;
        } else {
            const unsigned long long up = __shfl_down_sync(kFull, acc[P][q], 16);
            acc[P][q] = h == 0 ? up : 0ull;
        }
    }
}

// Where a unit's columns go: value q of position x of column (c1, c2) of coil slot s at
// p[s cs + c1 s1 + c2 s2 + x nk + q], for c1 < n1, c2 < n2.
// (A coil's grid has fewer than 2^31 values, so the strides within it fit 32 bits.)
struct SpreadDst {
    float2* p;
    long long cs;
    int s1, s2;
    int n1, n2, nk;
};

// The runs of positions [x0, x0 + np) of every column of nc coils from `tr` (column slot
// cl = 16 s + c at tr[cl RUN ..], RUN 8-byte values).  With all channels of the destination in the group a
// column's run is contiguous, and consecutive lanes store consecutive 16-byte pieces of
// the runs (16-byte aligned: row lengths, segments, x0 and np are even); otherwise 8 bytes
// at a time.
template <int NK, int RUN>
__device__ __forceinline__ void spread_store(const float2* tr, const SpreadDst& d, int nc, int x0, int np, int lane) {
    if (d.nk == NK) {
        const int per = np * NK / 2;
        const int tot = nc * kCols * per;
        float2* g = d.p + (long long)x0 * NK;
        if (np == 4) {
            constexpr int kPer = 2 * NK;
            for (int e = lane; e < nc * kCols * kPer; e += 32) {
                const int cl = e / kPer, j = e - cl * kPer;
                const int c1 = (cl >> 2) & 3, c2 = cl & 3;
                const float2 a = tr[cl * RUN + 2 * j], b = tr[cl * RUN + 2 * j + 1];
                if (c1 < d.n1 && c2 < d.n2)
                    *reinterpret_cast<float4*>(g + (cl >> 4) * d.cs + c1 * d.s1 + c2 * d.s2 + 2 * j) =
                        make_float4(a.x, a.y, b.x, b.y);
            }
        } else {
            for (int e = lane; e < tot; e += 32) {
                const int cl = e / per, j = e - cl * per;
                const int c1 = (cl >> 2) & 3, c2 = cl & 3;
                const float2 a = tr[cl * RUN + 2 * j], b = tr[cl * RUN + 2 * j + 1];
                if (c1 < d.n1 && c2 < d.n2)
                    *reinterpret_cast<float4*>(g + (cl >> 4) * d.cs + c1 * d.s1 + c2 * d.s2 + 2 * j) =
                        make_float4(a.x, a.y, b.x, b.y);
            }
        }
    } else {
        const int per = np * NK, tot = nc * kCols * per;
        for (int e = lane; e < tot; e += 32) {
            const int cl = e / per, r = e - cl * per;
            const int c1 = (cl >> 2) & 3, c2 = cl & 3;
            const int x = r / NK, q = r - x * NK;
            if (c1 < d.n1 && c2 < d.n2)
                d.p[(cl >> 4) * d.cs + c1 * d.s1 + c2 * d.s2 + (long long)(x0 + x) * d.nk + q] = tr[cl * RUN + r];
        }
    }
}

// One warp's subproblem `sub` for coils NC * by .. NC * by + NC - 1 (those below B), with
// SpreadDims::kAll 16-byte units of shared memory `rec`.
template <int W, int NK, int NC>
__device__ __forceinline__ void spread_body(const SpreadArgs& a, int kofs, int B, int sub, int by, float4* rec,
                                            const CUtensorMap* map) {
    using D = SpreadDims<W, NK, NC>;
    constexpr int NW = 3 * W;
    constexpr int NS = D::kSlots;
    // record of an incidence: [coil][k] conj(V[t, k]) r_b, the axis-3 weights (per half-warp
    // with one coil), [column] phi1 phi2 (0 outside the window)
    float4* out4 = rec + 32 * D::kRec;          // [column slot][kRun]: four finished positions
    float2* tr = reinterpret_cast<float2*>(out4);
    const Geo& g = a.g;
    const int lane = threadIdx.x;
    const int h = lane >> 4;     // the lane's incidence slot in a step
    const int col = lane & 15;
    const SubProb sp = a.subs[sub];
    const int b0 = by * NC;                 // first coil of the warp
    const int nc = min(NC, B - b0);         // its coils (the last warp of an odd batch has one)
    const int bin3 = sp.bin % a.nb3;
    const int bt = sp.bin / a.nb3;
    const int bin2 = bt % a.nb2;
    const int bin1 = bt / a.nb2;
    const int lo1 = bin1 * 4, lo2 = bin2 * 4, lo3 = bin3 * a.seg;
    const int M1 = g.M[0], M2 = g.M[1], M3 = g.M[2];
    const int seg = min(a.seg, M3 - lo3);   // positions of this unit
    const int nk = a.nk;

    SpreadDst grid;
    grid.s2 = M3 * nk;
    grid.s1 = M2 * grid.s2;
    grid.cs = (long long)M1 * grid.s1;
    grid.p = a.grids + b0 * grid.cs + (((long long)lo1 * M2 + lo2) * M3 + lo3) * nk + kofs;
    grid.n1 = M1 - lo1;
    grid.n2 = M2 - lo2;
    grid.nk = nk;

    const int cs = NC == 2 ? lane : col;   // this lane's column slot
    const bool mapped = NK == nk && a.use_map;
    // four finished positions from x0 of the unit, all columns of the warp's coils, from `box`
    // (one thread)
    auto send = [&](const float4* box, int x0, bool same) {
        for (int c = 0; c < nc; ++c)
            tma::tensor_store_4d(map, box + (same ? 0 : c * kCols * D::kRun), (lo3 + x0) * NK, lo2, lo1,
                                 a.coil0 + b0 + c);
    };
    if (sp.count == 0) {   // no window reaches the unit: zeros (a chunked unit has no empty chunk)
        if (mapped) {
            for (int e = lane; e < kCols * D::kRun; e += 32) out4[e] = make_float4(0.f, 0.f, 0.f, 0.f);
            tma::fence_async();
            __syncwarp();
            if (lane == 0) {
                for (int x0 = 0; x0 < seg; x0 += 4) send(out4, x0, true);
                tma::bulk_wait_read();
            }
        } else if ((NC == 2 ? h < nc : h == 0) && (col >> 2) < grid.n1 && (col & 3) < grid.n2) {
            float2* gcol = grid.p + (NC == 2 ? h : 0) * grid.cs + (col >> 2) * grid.s1 + (col & 3) * grid.s2;
            for (int e = 0; e < seg * NK; ++e) gcol[(long long)(e / NK) * nk + e % NK] = make_float2(0.f, 0.f);
        }
        return;
    }

    SpreadDst dst = grid;
    const bool whole = sp.nchunks == 1, bulk = whole && mapped;
    if (!whole) {
        dst.p = a.partials + ((long long)b0 * a.slots_per_b + sp.slot + sp.chunk) * a.slot_elems +
                (long long)kofs * kCols * a.seg;
        dst.cs = a.slots_per_b * a.slot_elems;
        dst.s2 = a.seg * NK;
        dst.s1 = 4 * dst.s2;
        dst.n1 = dst.n2 = 4;
        dst.nk = NK;
    }

    // the ring: positions x NK channels as packed (Re, Im) pairs
    unsigned long long acc[NS][NK];
#pragma unroll
    for (int p = 0; p < NS; ++p)
#pragma unroll
        for (int q = 0; q < NK; ++q) acc[p][q] = 0ull;

    // Current plane, its ring phase cur mod kSlots, and the last position to finish.  A chunk starts
    // and ends on whole blocks of four positions.
    int cur = 0, last_pos = seg - 1;
    if (!whole) {
        cur = sp.r0 < W - 1 ? sp.r0 : 4 * imap::spread_block_lo(sp.r0, W) + W - 1;
        last_pos = min(last_pos, sp.r1 | 3);   // the last position of block imap::spread_block_hi(r1)
    }
    int ph = cur % NS;
    // the position that plane `cur` finishes is cur - (W - 1); then the next plane
    auto finish_plane = [&] {
        const int pos = cur - (W - 1);
        const bool in = pos >= 0 && pos < seg;
        unsigned long long* out = nullptr;
        if (in) {
            out = reinterpret_cast<unsigned long long*>(tr + cs * (2 * D::kRun) + (pos & 3) * NK);
            if (bulk && (pos & 3) == 0) {
                if (lane == 0) tma::bulk_wait_read();   // the last box has been read
                __syncwarp();
            }
        }
        spread_take<0, W, NK, NC>(ph, acc, out, h);
        if (in && ((pos & 3) == 3 || pos == seg - 1)) {
            if (bulk) {
                tma::fence_async();
                __syncwarp();
                if (lane == 0) send(out4, pos & ~3, false);
            } else {
                __syncwarp();
                spread_store<NK, 2 * D::kRun>(tr, dst, nc, pos & ~3, (pos & 3) + 1, lane);
                __syncwarp();
            }
        }
        ++cur;
        ph = ph + 1 == NS ? 0 : ph + 1;
    };

    const float sc = a.scale ? __ldg(a.scale) : 1.f;
    const int kv = a.k0 + kofs;   // first channel of V of this group
    const int4* incs = a.inc + sp.start;
    for (int base = 0; base < sp.count; base += 32) {
        const int n = min(32, sp.count - base);
        int rel = -1;   // the plane of staged incidence `lane` (-1: none)
        if (lane < n) {
            const int4 in = __ldg(incs + base + lane);
            rel = in.y >> 16;
            const int s = in.x, orig = in.z, t = in.w;
            const float* ws = a.wts + (long long)s * NW;
            // the sample's 3W weights (3W floats from a multiple of 3W: 16-byte loads when
            // 3W is a multiple of 4, 8-byte loads when even)
            float wl[NW];
            if constexpr (NW % 4 == 0) {
#pragma unroll
                for (int q = 0; q < NW; q += 4) {
                    const float4 v = __ldg(reinterpret_cast<const float4*>(ws + q));
                    wl[q] = v.x;
                    wl[q + 1] = v.y;
                    wl[q + 2] = v.z;
                    wl[q + 3] = v.w;
                }
            } else if constexpr (NW % 2 == 0) {
#pragma unroll
                for (int q = 0; q < NW; q += 2) {
                    const float2 v = __ldg(reinterpret_cast<const float2*>(ws + q));
                    wl[q] = v.x;
                    wl[q + 1] = v.y;
                }
            } else {
#pragma unroll
                for (int q = 0; q < NW; ++q) wl[q] = __ldg(ws + q);
            }
            float v1[4], v2[4];
            window_at<W>(wl, in.y & 255, v1);
            window_at<W>(wl + W, (in.y >> 8) & 255, v2);
            float4* mine = rec + lane * D::kRec;
#pragma unroll
            for (int x = 0; x < 4; ++x)
                mine[D::kOfsW12 + x] = make_float4(v1[x] * v2[0], v1[x] * v2[1], v1[x] * v2[2], v1[x] * v2[3]);
#pragma unroll
            for (int q = 0; q < (NC == 2 ? 1 : 2) * D::kW3; ++q) {
                float wq[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int slot = 4 * (q % D::kW3) + u, o = q / D::kW3 * NS + slot;   // window position
                    wq[u] = slot < NS && o < W ? wl[2 * W + (o < W ? o : 0)] : 0.f;
                }
                mine[D::kOfsW3 + q] = make_float4(wq[0], wq[1], wq[2], wq[3]);
            }
            float2 vq[NK];
            load_v_row<NK>(a.V + (long long)t * a.vstride + kv, kv % 2 == 0, vq);
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                float2 r = make_float2(0.f, 0.f);   // a missing second coil spreads zeros and is not stored
                if (c < nc) {
                    r = __ldg(a.y + (long long)(b0 + c) * g.J + orig);
                    r.x *= sc;
                    r.y *= sc;
                }
                float2 cv[2 * D::kCoef];
#pragma unroll
                for (int q = 0; q < NK; ++q)
                    cv[q] = make_float2(vq[q].x * r.x + vq[q].y * r.y, vq[q].x * r.y - vq[q].y * r.x);
                if (2 * D::kCoef > NK) cv[2 * D::kCoef - 1] = make_float2(0.f, 0.f);
#pragma unroll
                for (int q = 0; q < D::kCoef; ++q)
                    mine[c * D::kCoef + q] = make_float4(cv[2 * q].x, cv[2 * q].y, cv[2 * q + 1].x, cv[2 * q + 1].y);
            }
        }
        __syncwarp();
        // the staged planes in turn (the plan orders a unit's incidences by plane)
        for (int i = 0; i < n;) {
            const int r = __shfl_sync(kFull, rel, i);
            const unsigned diff = __ballot_sync(kFull, rel != r) & (kFull << i);
            const int e = diff ? __ffs(diff) - 1 : 32;   // lanes >= n hold -1, so e <= n
            while (cur < r) finish_plane();
            spread_plane<0, W, NK, NC>(ph, acc, rec + (NC == 2 ? h * D::kCoef : 0),
                                       rec + D::kOfsW3 + (NC == 2 ? 0 : h * D::kW3),
                                       reinterpret_cast<const float*>(rec + D::kOfsW12) + col, i, e);
            i = e;
        }
        __syncwarp();
    }
    while (cur <= last_pos + W - 1) finish_plane();
    if (bulk && lane == 0) tma::bulk_wait_read();   // before the warp's shared memory goes away
    if (whole) return;

    // The chunk's partial blocks are in its slot.  Lane q counts block q, which the chunks
    // [c0, c1) reach: the last of every kGroup of them to arrive sums the group's partials
    // (into the grid if the group is all of them, else into its first chunk's slot), the last
    // group to be summed sums the groups.  So the centre's hundred partials of a block are
    // added in two short chains by several warps, in a fixed order.
    constexpr int kGroup = 8;
    __threadfence();
    __syncwarp();
    const int nblk = (seg + 3) >> 2;
    const long long first_counter = (long long)b0 * a.ngroups + a.group;
    int* unit_count = a.counters + (first_counter * a.nbins + sp.bin) * a.nblk;
    int* group_count = a.group_counters + (first_counter * a.slots_per_b + sp.slot) * a.nblk;
    int c0 = 0, c1 = 0;
    bool mine = false;
    if (lane < nblk) {
        const int2 rg = __ldg(a.ranges + (long long)sp.multi * a.nblk + lane);
        c0 = rg.x;
        c1 = rg.y;
        if (sp.chunk >= c0 && sp.chunk < c1) {
            const int g0 = c0 + (sp.chunk - c0) / kGroup * kGroup;
            mine = atomicAdd(group_count + g0 * a.nblk + lane, 1) == min(kGroup, c1 - g0) - 1;
        }
    }
    unsigned todo = __ballot_sync(kFull, mine);
    if (!todo) return;
    __threadfence();
    for (; todo; todo &= todo - 1) {
        const int q = __ffs(todo) - 1;
        const int ca = __shfl_sync(kFull, c0, q), cb = __shfl_sync(kFull, c1, q);
        const int per = min(4, seg - 4 * q) * NK / 2, tot = nc * kCols * per;
        constexpr int kPieces = NC * NK;   // 16-byte pieces of a block per lane
        float4 sum[kPieces];
        float4* src[kPieces];              // the lane's pieces in the unit's first slot
#pragma unroll
        for (int m = 0; m < kPieces; ++m) {
            const int e = min(lane + 32 * m, tot - 1);
            const int cl = e / per, j = e - cl * per;
            src[m] = reinterpret_cast<float4*>(
                         a.partials + ((long long)(b0 + (cl >> 4)) * a.slots_per_b + sp.slot) * a.slot_elems +
                         (long long)kofs * kCols * a.seg + ((cl & 15) * a.seg + 4 * q) * NK) + j;
        }
        const long long slot4 = a.slot_elems / 2;
        auto add_up = [&](int first, int end, int step) {
#pragma unroll
            for (int m = 0; m < kPieces; ++m) sum[m] = make_float4(0.f, 0.f, 0.f, 0.f);
            for (int ch = first; ch < end; ch += step) {
                const long long o = ch * slot4;
#pragma unroll
                for (int m = 0; m < kPieces; ++m) {
                    const float4 v = __ldcg(src[m] + o);
                    sum[m].x += v.x;
                    sum[m].y += v.y;
                    sum[m].z += v.z;
                    sum[m].w += v.w;
                }
            }
        };
        const int g0 = ca + (sp.chunk - ca) / kGroup * kGroup;
        add_up(g0, min(g0 + kGroup, cb), 1);
        if (lane == 0) group_count[g0 * a.nblk + q] = 0;
        if (cb - ca > kGroup) {
#pragma unroll
            for (int m = 0; m < kPieces; ++m)
                if (lane + 32 * m < tot) src[m][g0 * slot4] = sum[m];
            __threadfence();
            __syncwarp();
            int last = 0;
            if (lane == 0) last = atomicAdd(unit_count + q, 1) == (cb - ca + kGroup - 1) / kGroup - 1;
            if (!__shfl_sync(kFull, last, 0)) continue;
            __threadfence();
            add_up(ca, cb, kGroup);
            if (lane == 0) unit_count[q] = 0;
        }
#pragma unroll
        for (int m = 0; m < kPieces; ++m) {
            const int e = lane + 32 * m;
            if (e >= tot) continue;
            const int cl = e / per, j = e - cl * per;
            const int k1 = (cl >> 2) & 3, k2 = cl & 3;
            if (k1 >= grid.n1 || k2 >= grid.n2) continue;
            float2* o = grid.p + (cl >> 4) * grid.cs + k1 * grid.s1 + k2 * grid.s2 + (long long)4 * q * nk;
            if (nk == NK) {
                *reinterpret_cast<float4*>(o + 2 * j) = sum[m];
            } else {
                const int x0 = 2 * j / NK, q0 = 2 * j - x0 * NK, x1 = (2 * j + 1) / NK, q1 = 2 * j + 1 - x1 * NK;
                o[(long long)x0 * nk + q0] = make_float2(sum[m].x, sum[m].y);
                o[(long long)x1 * nk + q1] = make_float2(sum[m].z, sum[m].w);
            }
        }
    }
}

// Resident warps per SM the registers are bounded for: the ring's pairs plus about 50.  (With the sums
// by pairs a ring of 32, W = 4 with 8 channels, spills 524 bytes at 16 warps and 60 at 12: 8 coils of
// 96^3 1058 us and 895.)
template <int W, int NK, int NC>
constexpr int spread_warps() {
    constexpr int n = SpreadDims<W, NK, NC>::kSlots * NK;
    return n <= 12 ? 24 : (n <= 20 ? 20 : (n <= (spread_together(W) == 2 ? 30 : 32) ? 16 : (n <= 42 ? 12 : (n <= 48 ? 10 : 8))));
}

template <int W, int NK, int NC>
__global__ void __launch_bounds__(32, (spread_warps<W, NK, NC>())) spread_kernel(SpreadArgs a, const __grid_constant__ CUtensorMap map, int kofs, int B) {
    __shared__ __align__(128) float4 rec[SpreadDims<W, NK, NC>::kAll];
    spread_body<W, NK, NC>(a, kofs, B, (int)blockIdx.x, (int)blockIdx.y, rec, &map);
}

template <int W, int NK>
cudaError_t launch_wk(const SpreadArgs& a, const CUtensorMap& map, int kofs, int nsub, int B, int coils, cudaStream_t st) {
    if (coils != 1 && B >= 2) {
        dim3 grid((unsigned)nsub, (unsigned)((B + 1) / 2));
        spread_kernel<W, NK, 2><<<grid, 32, 0, st>>>(a, map, kofs, B);
    } else {
        dim3 grid((unsigned)nsub, (unsigned)B);
        spread_kernel<W, NK, 1><<<grid, 32, 0, st>>>(a, map, kofs, B);
    }
    return cudaGetLastError();
}

// Channels run in groups of at most 8 (one launch each, exact group size).
template <int W>
cudaError_t launch_spread_width(SpreadArgs a, const CUtensorMap& map, int nsub, int B, int coils, cudaStream_t st) {
    a.ngroups = (a.nk + 7) / 8;
    for (int gi = 0; gi < a.ngroups; ++gi) {
        const int kofs = gi * 8;
        const int ng = a.nk - kofs < 8 ? a.nk - kofs : 8;
        a.group = gi;
        cudaError_t e;
        switch (ng) {
            case 1: e = launch_wk<W, 1>(a, map, kofs, nsub, B, coils, st); break;
            case 2: e = launch_wk<W, 2>(a, map, kofs, nsub, B, coils, st); break;
            case 3: e = launch_wk<W, 3>(a, map, kofs, nsub, B, coils, st); break;
            case 4: e = launch_wk<W, 4>(a, map, kofs, nsub, B, coils, st); break;
            case 5: e = launch_wk<W, 5>(a, map, kofs, nsub, B, coils, st); break;
            case 6: e = launch_wk<W, 6>(a, map, kofs, nsub, B, coils, st); break;
            case 7: e = launch_wk<W, 7>(a, map, kofs, nsub, B, coils, st); break;
            default: e = launch_wk<W, 8>(a, map, kofs, nsub, B, coils, st); break;
        }
        if (e != cudaSuccess) return e;
        if (gi > 0) note_launches(1);   // the stage counts its first launch
    }
    return cudaSuccess;
}

}  // namespace
}  // namespace sdp
