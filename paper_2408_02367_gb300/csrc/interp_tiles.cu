// Forward interpolation with the subspace contraction (gridding step A3, the
// same operation as interp.cu), from shared-memory tiles:
//
//   y_b[j] = sum_k V[t_j, k] sum_{W^3 taps} phi(g1 - m1) phi(g2 - m2) phi(g3 - m3) U_{b,k}[m mod M]
//
// for the per-coil operator A_c of StoDIP (Sec. 2 Eq. 1, Sec. 2.1 Eq. 3).
//
// The plan orders the samples by tile of 8 x 8 x 8 grid points (4 x 8 x 8 from W = 6
// on; the tile of the sample's own coordinate) and lists work items, heaviest first: each
// non-empty tile, a dense one cut into pieces of at most 512 samples (the
// k-space centre's tiles hold thousands, which one CTA would serialise).
// A sample of tile t has its window start m0 = ceil(g - W/2) in
// [e t - W/2, e t + e - W/2] (integer division) along an axis of tile edge e, so
// its taps lie in the e + W points from e t - W/2.  Persistent CTAs walk the
// (work item, coil) units; a CTA copies the unit's points x nk channels of the
// channel-interleaved grid ([b][i1][i2][i3][kk], wrapped periodically) into
// shared memory, completing on an mbarrier whose wait is bounded: one tensor load
// (cp.async.bulk.tensor) where the points do not wrap around the grid, else (and
// for calls on some of the plan's channels) a bulk copy per row, two where the row
// wraps along axis 3.  (Row copies alone were a third of the kernel's
// instructions: the copies of a warp's lanes are issued one after the other.)
// Rows start on an even point and have an even length, so that every piece is
// 16-byte aligned.  Then it interpolates every sample of the item from shared
// memory: the scattered, latency-bound gathers of the row kernel become one
// coalesced copy per tile and coil plus shared loads.
//
// What bounds it is latency, the tiles' and the samples' loads (128^3, two coils, five
// channels, 182 us: issue 39%, 6.4 warps per issue wait on global loads and 3.2 on
// shared, 36% of warp slots filled, the shared memory of three CTAs), so everything
// that depends on the sample alone is made by the plan (index in y, frame, start of the
// window in the tile, the 3W weights), and the warp does little besides the window sums:
//   - W <= 4: a warp takes two samples, one per half-warp.  Lane (a2, a3) of a
//     half-warp owns the axis-2/axis-3 tap pair: over the W axis-1 taps it
//     accumulates phi1(a1) U_k for its tap's nk channels (shared loads at
//     compile-time offsets from one address), contracts them with V[t, k] and
//     scales by phi2(a2) phi3(a3); the half-warp sums its lanes, real and
//     imaginary parts side by side.
//   - W >= 5 (W^2 > 16 tap pairs): a warp takes one sample.  Lane l owns entry l
//     (and l + 32, ...) of a row's W nk contiguous values, i.e. one axis-3 tap and
//     channel, and walks the W^2 rows of the window.
// The next samples' records and weights are loaded while the current ones are
// interpolated, and a unit's first ones while its tile is on its way.  Widths 2 to 8 and up
// to 8 channels per call; other calls use interp.cu.
#include <type_traits>

#include "batch.cuh"
#include "index_map.cuh"
#include "interp_impl.cuh"
#include "spread_map.cuh"
#include "tma.cuh"

namespace sdp {
namespace {

// Tile edges in grid points (the plan's sample order): 8 along axes 2 and 3, and along axis 1 up to
// W = 5; from W = 6 on 4, so that a tile with its margin leaves room for a second CTA on the SM up
// to 6 channels (125 KB and 90 KB at W = 6, K = 5: 4 coils of 32^3 on the 64^3 grid, 114 us with
// 8 points, 89 with 4).
constexpr int kTile = imap::kTileEdge;

template <int W, int NK>
struct TileDims {
    static constexpr int E1 = imap::tile_edge(W, 0), H1 = imap::tile_points(W, 0);   // tile plus window margin, axis 1
    static constexpr int H = imap::tile_points(W, 1);          // and axis 2
    static constexpr int LO3 = imap::tile_before(W, 2);        // axis-3 points before the tile: W / 2, made even
    static constexpr int OFF3 = LO3 - W / 2;
    static constexpr int H3 = imap::tile_points(W, 2);         // axis-3 points of a row, even
    static constexpr int ROW = H3 * NK;   // complex values of one (h1, h2) row
    static constexpr int PLANE = H * ROW;
    static constexpr int SIZE = H1 * PLANE;
    static constexpr int BYTES = SIZE * 8;
    static constexpr int SLOT = (BYTES + 127) & ~127;          // tensor loads want 128-byte aligned boxes
    static constexpr int SMEM = SLOT + 16;   // the tile and the copies' mbarrier
    static_assert(SMEM <= 227 * 1024, "every tile of up to 8 channels fits");
    // threads per CTA: 24 warps per SM in 3 or more, 2 or 1 CTAs, by the tile's size.  (One CTA
    // with a ring of three tiles, loading warps and no barrier per tile was slower, 229 us against
    // 187 on the 128^3 workload: every warp goes through every unit, and half of the tiles hold
    // fewer than 64 samples.)
    static constexpr int NT = SMEM <= 75 * 1024 ? 256 : (SMEM <= 113 * 1024 ? 384 : 768);
    static constexpr int NWARP = NT / 32;
    // resident CTAs the registers are bounded for (40 warps per SM where the tiles are small: one
    // channel at W = 4, 491,520 samples, 56 us unbounded, 51 bounded)
    static constexpr int fit = 225 * 1024 / SMEM;
    static constexpr int most = W <= 4 ? 5 : 4;
    static constexpr int CTAS = NT == 256 ? (fit < 3 ? 3 : (fit > most ? most : fit)) : (NT == 384 ? 2 : 1);
};

// A thread's share of y[j] for the sum over a group of 16 or 32 lanes: lanes with the top
// bit hold the imaginary part afterwards, the others the real part, complete in the
// group's lanes 0 and TOP.
template <int TOP>
__device__ __forceinline__ float lane_sum(float sx, float sy, int lane) {
    const bool hi = (lane & TOP) != 0;
    float v = (hi ? sy : sx) + __shfl_xor_sync(kFullI, hi ? sx : sy, TOP);
#pragma unroll
    for (int o = TOP / 2; o > 0; o >>= 1) v += __shfl_xor_sync(kFullI, v, o);
    return v;
}

__device__ __forceinline__ void put1(float* dst, float v, int accumulate) { *dst = accumulate ? *dst + v : v; }

// One lane's part of the interpolation of the samples [start, start + count) of one coil, W <= 4:
// a sample per half-warp.  The constructor issues the first samples' loads (before the tile
// has landed), run() interpolates from the tile.
template <int W, int NK>
struct HalfSamples {
    using D = TileDims<W, NK>;
    static constexpr int NWARP = D::NWARP;
    const int4* rec;
    const float* wts;
    const float2* V;
    float2* yb;
    int vstride, count, half, q0;
    bool aligned;        // V rows read 16 bytes at a time
    imap::TileLane tl;
    int4 rn, rn2;        // the records run two steps ahead, the weights and V rows one
    float w1n[W], w23n;
    float2 vn[NK];

    __device__ __forceinline__ int sample(int q) const {
        const int si = min(2 * q, count - 1) + half;
        return si < count ? si : count - 1;   // a half without a sample repeats the last one
    }

    __device__ __forceinline__ void fetch(int q, const int4& r) {
        const float* ws = wts + sample(q) * (3 * W);
        if constexpr (W == 4) {   // 48 bytes per sample: the axis-1 weights are one aligned 16-byte load
            const float4 v = __ldg(reinterpret_cast<const float4*>(ws));
            w1n[0] = v.x;
            w1n[1] = v.y;
            w1n[2] = v.z;
            w1n[3] = v.w;
        } else {
#pragma unroll
            for (int i = 0; i < W; ++i) w1n[i] = __ldg(ws + i);
        }
        w23n = __ldg(ws + W + tl.a2) * __ldg(ws + 2 * W + tl.a3);
        load_v_row<NK>(V + r.y * vstride, aligned, vn);
    }

    __device__ __forceinline__ HalfSamples(const InterpTiles& a, const int4& td, int b)
        : rec(a.srec + td.y), wts(a.wts + (long long)td.y * (3 * W)), V(a.V + a.k0), yb(a.y + (long long)b * a.g.J),
          vstride(a.vstride), count(td.z), half((threadIdx.x >> 4) & 1), q0(threadIdx.x >> 5), aligned(a.k0 % 2 == 0),
          tl(imap::tile_lane_map(threadIdx.x & 15, W)) {
        rn = __ldg(rec + sample(q0));   // a warp without a pair loads the last sample's
        rn2 = __ldg(rec + sample(q0 + NWARP));
        fetch(q0, rn);
    }

    __device__ __forceinline__ void run(const float2* sg, int accumulate) {
        const int lane = threadIdx.x & 31, l16 = lane & 15;
        const unsigned long long* mine =
            reinterpret_cast<const unsigned long long*>(sg) + (tl.a2 * D::H3 + tl.a3 + D::OFF3) * NK;
        // a warp takes the sample pairs q = warp, warp + NWARP, ...
        for (int q = q0; 2 * q < count; q += NWARP) {
            const int4 r = rn;
            float w1[W];
            float2 vk[NK];
#pragma unroll
            for (int i = 0; i < W; ++i) w1[i] = w1n[i];
#pragma unroll
            for (int k = 0; k < NK; ++k) vk[k] = vn[k];
            const float w23 = tl.act ? w23n : 0.f;   // idle lanes repeat tap (0, 0) with zero weight
            rn = rn2;
            if (2 * (q + NWARP) < count) {
                fetch(q + NWARP, rn);
                rn2 = __ldg(rec + sample(q + 2 * NWARP));
            }
            const unsigned long long* base = mine + r.z * NK;
            unsigned long long acc[NK];
#pragma unroll
            for (int k = 0; k < NK; ++k) acc[k] = 0ull;
#pragma unroll
            for (int a1 = 0; a1 < W; ++a1) {
                const unsigned long long wa = pk2(w1[a1], w1[a1]);
#pragma unroll
                for (int k = 0; k < NK; ++k) acc[k] = fma2(wa, base[a1 * D::PLANE + k], acc[k]);
            }
            float sx = 0.f, sy = 0.f;
#pragma unroll
            for (int k = 0; k < NK; ++k) {
                const float2 v = vk[k];
                const float2 u = upk2(acc[k]);
                sx = fmaf(v.x, u.x, sx);
                sx = fmaf(-v.y, u.y, sx);
                sy = fmaf(v.x, u.y, sy);
                sy = fmaf(v.y, u.x, sy);
            }
            const float v = lane_sum<8>(sx * w23, sy * w23, lane);
            if ((l16 & 7) == 0 && 2 * q + half < count)
                put1(reinterpret_cast<float*>(yb + r.x) + (l16 >> 3), v, accumulate);
        }
    }
};

// The same for W >= 5: a sample per warp.
template <int W, int NK>
struct RowSamples {
    using D = TileDims<W, NK>;
    static constexpr int NWARP = D::NWARP;
    static constexpr int N = W * NK, NI = (N + 31) / 32;   // entries of a row, per lane
    const int4* rec;
    const float* wts;
    const float2* V;
    float2* yb;
    int vstride, count;
    int ent[NI];         // the lane's entries (idle lanes repeat the last one with a zero coefficient)
    int4 rn, rn2;
    float wn[2 * W], w3n[NI];
    float2 vn[NI];

    __device__ __forceinline__ void fetch(int s, const int4& r) {
        const float* ws = wts + s * (3 * W);
        if constexpr (W % 2 == 0) {
#pragma unroll
            for (int i = 0; i < 2 * W; i += 2) {
                const float2 v = __ldg(reinterpret_cast<const float2*>(ws + i));
                wn[i] = v.x;
                wn[i + 1] = v.y;
            }
        } else {
#pragma unroll
            for (int i = 0; i < 2 * W; ++i) wn[i] = __ldg(ws + i);
        }
#pragma unroll
        for (int i = 0; i < NI; ++i) {
            const int a3 = ent[i] / NK;
            w3n[i] = __ldg(ws + 2 * W + a3);
            vn[i] = __ldg(V + r.y * vstride + (ent[i] - a3 * NK));
        }
    }

    __device__ __forceinline__ RowSamples(const InterpTiles& a, const int4& td, int b)
        : rec(a.srec + td.y), wts(a.wts + (long long)td.y * (3 * W)), V(a.V + a.k0), yb(a.y + (long long)b * a.g.J),
          vstride(a.vstride), count(td.z) {
        const int n = count, lane = threadIdx.x & 31, s0 = min((int)threadIdx.x >> 5, n - 1);
#pragma unroll
        for (int i = 0; i < NI; ++i) ent[i] = min(lane + 32 * i, N - 1);
        rn = __ldg(rec + s0);
        rn2 = __ldg(rec + min(s0 + NWARP, n - 1));
        fetch(s0, rn);
    }

    __device__ __forceinline__ void run(const float2* sg, int accumulate) {
        const int lane = threadIdx.x & 31;
        const unsigned long long* mine = reinterpret_cast<const unsigned long long*>(sg) + D::OFF3 * NK;
        for (int s = threadIdx.x >> 5; s < count; s += NWARP) {
            const int4 r = rn;
            float w[2 * W], w3[NI];
            float2 vk[NI];
#pragma unroll
            for (int i = 0; i < 2 * W; ++i) w[i] = wn[i];
#pragma unroll
            for (int i = 0; i < NI; ++i) {
                w3[i] = lane + 32 * i < N ? w3n[i] : 0.f;
                vk[i] = vn[i];
            }
            rn = rn2;
            if (s + NWARP < count) {
                fetch(s + NWARP, rn);
                rn2 = __ldg(rec + min(s + 2 * NWARP, count - 1));
            }
            float sx = 0.f, sy = 0.f;
            unsigned long long w2[W];   // (w, w) pairs, made once per sample
#pragma unroll
            for (int a2 = 0; a2 < W; ++a2) w2[a2] = pk2(w[W + a2], w[W + a2]);
#pragma unroll
            for (int i = 0; i < NI; ++i) {
                const unsigned long long* base = mine + r.z * NK + ent[i];
                unsigned long long acc = 0ull;
#pragma unroll
                for (int a1 = 0; a1 < W; ++a1) {
                    unsigned long long t = 0ull;
#pragma unroll
                    for (int a2 = 0; a2 < W; ++a2)
                        t = fma2(w2[a2], base[a1 * D::PLANE + a2 * D::ROW], t);
                    acc = fma2(pk2(w[a1], w[a1]), t, acc);
                }
                const float2 u = upk2(acc);
                const float cx = w3[i] * vk[i].x, cy = w3[i] * vk[i].y;
                sx = fmaf(cx, u.x, sx);
                sx = fmaf(-cy, u.y, sx);
                sy = fmaf(cx, u.y, sy);
                sy = fmaf(cy, u.x, sy);
            }
            const float v = lane_sum<16>(sx, sy, lane);
            if ((lane & 15) == 0) put1(reinterpret_cast<float*>(yb + r.x) + (lane >> 4), v, accumulate);
        }
    }
};

template <int W, int NK>
using TileSamples = typename std::conditional<(W <= 4), HalfSamples<W, NK>, RowSamples<W, NK>>::type;

// Copies the tile of work item td = (flattened tile index, first sample, sample count, -) of
// coil b into sg, completing on bar.
template <int W, int NK, bool TEST>
__device__ __forceinline__ void tile_copy(const InterpTiles& a, const CUtensorMap* map, const int4& td, int b,
                                          float2* sg, uint64_t* bar, int withhold_row) {
    using D = TileDims<W, NK>;
    constexpr int H = D::H, H3 = D::H3;
    const int M1 = a.g.M[0], M2 = a.g.M[1], M3 = a.g.M[2];
    const int t3 = td.x % a.nt3, t12 = td.x / a.nt3;
    const int t2 = t12 % a.nt2, t1 = t12 / a.nt2;
    const int lo1 = t1 * D::E1 - W / 2, lo2 = t2 * kTile - W / 2;
    // a row's H3 points along axis 3 start at p0 and run la points before they wrap
    // around the grid (la = H3 unless the tile crosses the grid's end along axis 3)
    const int p0 = wrap1(t3 * kTile - D::LO3, M3);
    const int la = M3 - p0 < H3 ? M3 - p0 : H3;
    const int t = threadIdx.x;
    if (t == 0) tma::mbar_expect_tx(bar, (uint32_t)D::BYTES);
    if (!TEST && a.use_map && la == H3 && lo1 >= 0 && lo1 + D::H1 <= M1 && lo2 >= 0 && lo2 + H <= M2) {
        if (t == 0) tma::tensor_load_4d(map, sg, p0 * NK, lo2, lo1, a.coil0 + b, bar);
        return;
    }
    __syncthreads();   // the expected bytes are registered before any copy lands
    const float2* gb = a.grids + (long long)b * ((long long)M1 * M2 * M3 * NK);
    // rows dealt out over the warps first: a warp's copies go one after the other
    for (int r = (t & 31) * D::NWARP + (t >> 5); r < D::H1 * H; r += D::NT) {
        if (TEST && r == withhold_row) continue;   // the wait test hook: this row never lands
        const int h1 = r / H, h2 = r - h1 * H;
        const float2* src = gb + ((long long)wrap1(lo1 + h1, M1) * M2 + wrap1(lo2 + h2, M2)) * M3 * NK;
        float2* dst = sg + r * D::ROW;
        tma::bulk_g2s(dst, src + (long long)p0 * NK, (uint32_t)(la * NK * 8), bar);
        if (la < H3) tma::bulk_g2s(dst + la * NK, src, (uint32_t)((H3 - la) * NK * 8), bar);
    }
}

// One plan's units: work item u / B of coil u mod B (the coils of an item are neighbours: its
// records stay in L2).
struct PlanUnits {
    const InterpTiles& a;
    const CUtensorMap* map;
    __device__ __forceinline__ const InterpTiles& plan(int) const { return a; }
    __device__ __forceinline__ const CUtensorMap* tensor_map(int) const { return map; }
    __device__ __forceinline__ int4 unit(int u, int& b, int& i) const {
        const int q = u / a.B;
        b = u - q * a.B;
        i = 0;
        return __ldg(a.tiles + q);
    }
};

__device__ __forceinline__ int mv_find_item(const MvUnits& u, long long unit) {
    int i = 0;
    while (i + 1 < u.n && unit >= u.start[i + 1]) ++i;
    return i;
}

// The units of every item of a batched call; u.start: prefix sums of work items times coils.
struct BatchUnits {
    const MvArgs& a;
    const MvUnits& u;
    __device__ __forceinline__ InterpTiles plan(int i) const {
        const MvItem& it = a.it[i];
        return InterpTiles{it.g, it.itiles, it.n_itiles, it.nt2, it.nt3, it.srec, it.wts, it.Vp, it.vstride, it.bufA,
                           it.B, 0, it.y, 0, it.status, it.coil0, 1};   // batched calls take all channels
    }
    __device__ __forceinline__ const CUtensorMap* tensor_map(int i) const { return &a.it[i].tile_map; }
    __device__ __forceinline__ int4 unit(int w, int& b, int& i) const {
        i = mv_find_item(u, w);
        const MvItem& it = a.it[i];
        const int local = (int)(w - u.start[i]), q = local / it.B;
        b = local - q * it.B;
        return __ldg(it.itiles + q);
    }
};

// A tile per CTA: copy, wait, interpolate, unit after unit.
template <int W, int NK, bool TEST, class Units>
__device__ __forceinline__ void tile_loop(const Units& units, int nunits, float2* sg, int withhold_row,
                                          unsigned long long wait_ns) {
    using D = TileDims<W, NK>;
    static_assert(D::ROW % 2 == 0 && D::LO3 % 2 == 0, "16-byte row pieces");
    uint64_t* bar = reinterpret_cast<uint64_t*>(reinterpret_cast<unsigned char*>(sg) + D::SLOT);
    if (threadIdx.x == 0) {
        tma::mbar_init(bar, 1);
        tma::fence_init();
    }
    uint32_t phase = 0;
    int b, i, nb = 0, ni = 0;
    int4 next = units.unit(min((int)blockIdx.x, nunits - 1), nb, ni);
    for (int u = blockIdx.x; u < nunits; u += gridDim.x) {
        const int4 td = next;
        b = nb;
        i = ni;
        next = units.unit(min(u + (int)gridDim.x, nunits - 1), nb, ni);
        const InterpTiles& t = units.plan(i);
        __syncthreads();   // the last unit's readers are done
        tile_copy<W, NK, TEST>(t, units.tensor_map(i), td, b, sg, bar, u == 0 ? withhold_row : -1);
        TileSamples<W, NK> samples(t, td, b);
        const bool landed = __syncthreads_and(tma::mbar_wait(bar, phase, t.status, wait_ns)) != 0;
        if (!landed) {
            // a copy did not complete within the wait's bound (status holds
            // SDP_ERR_TIMEOUT): give the copies in flight one more bounded wait, leave
            tma::mbar_wait(bar, phase, nullptr, wait_ns);
            return;
        }
        phase ^= 1u;
        samples.run(sg, t.accumulate);
    }
}

// TEST: the instantiation that honours the wait test hook (withhold_row, wait_ns);
// the other ignores both, so the hook costs the production kernel nothing.
template <int W, int NK, bool TEST>
__global__ void __launch_bounds__(TileDims<W, NK>::NT, TileDims<W, NK>::CTAS) interp_tiles_kernel(const __grid_constant__ InterpTiles a,
                                                                           const __grid_constant__ CUtensorMap map,
                                                                           int withhold_row,
                                                                           unsigned long long wait_ns) {
    extern __shared__ __align__(128) float2 sg[];   // [h1][h2][h3][k], then the copies' mbarrier
    tile_loop<W, NK, TEST>(PlanUnits{a, &map}, a.ntiles * a.B, sg, TEST ? withhold_row : -1,
                             TEST ? wait_ns : tma::kWaitNs);
}

// Several plans in one launch (the batched forward's interpolation).
template <int W, int NK>
__global__ void __launch_bounds__(TileDims<W, NK>::NT, TileDims<W, NK>::CTAS) mv_interp_tiles_kernel(const __grid_constant__ MvArgs a,
                                                                              const __grid_constant__ MvUnits u) {
    extern __shared__ __align__(128) float2 sg[];   // [h1][h2][h3][k], then the copies' mbarrier
    tile_loop<W, NK, false>(BatchUnits{a, u}, (int)u.start[u.n], sg, -1, tma::kWaitNs);
}

// Persistent grid: the CTAs that are resident at once, or fewer for little work.
template <class K>
cudaError_t tiles_grid(K kernel, int bytes, int threads, long long nwork, ResidentCtas& resident, unsigned& grid) {
    long long nres = 0;
    const cudaError_t e = resident.get(kernel, bytes, threads, nres);
    grid = (unsigned)(nwork < nres ? nwork : nres);
    return e;
}

template <int W, int NK>
cudaError_t launch_mv_tiles_k(const MvArgs& a, const MvUnits& u, cudaStream_t st) {
    using D = TileDims<W, NK>;
    static ResidentCtas resident;
    unsigned grid = 0;
    if (u.start[u.n] > 0x3fffffffLL) return cudaErrorInvalidConfiguration;
    const cudaError_t e = tiles_grid(mv_interp_tiles_kernel<W, NK>, D::SMEM, D::NT, u.start[u.n], resident, grid);
    if (e != cudaSuccess) return e;
    mv_interp_tiles_kernel<W, NK><<<grid, D::NT, D::SMEM, st>>>(a, u);
    return cudaGetLastError();
}

template <int W, int NK>
cudaError_t launch_tiles_k(const InterpTiles& a, const CUtensorMap& map, int withhold_row, unsigned long long wait_ns, cudaStream_t st) {
    using D = TileDims<W, NK>;
    const long long nunits = (long long)a.ntiles * a.B;
    if (nunits > 0x3fffffffLL) return cudaErrorInvalidConfiguration;
    unsigned grid = 0;
    if (withhold_row >= 0 || wait_ns != tma::kWaitNs) {
        static ResidentCtas resident_t;
        const cudaError_t e = tiles_grid(interp_tiles_kernel<W, NK, true>, D::SMEM, D::NT, nunits, resident_t, grid);
        if (e != cudaSuccess) return e;
        interp_tiles_kernel<W, NK, true><<<grid, D::NT, D::SMEM, st>>>(a, map, withhold_row, wait_ns);
    } else {
        static ResidentCtas resident;
        const cudaError_t e = tiles_grid(interp_tiles_kernel<W, NK, false>, D::SMEM, D::NT, nunits, resident, grid);
        if (e != cudaSuccess) return e;
        interp_tiles_kernel<W, NK, false><<<grid, D::NT, D::SMEM, st>>>(a, map, -1, tma::kWaitNs);
    }
    return cudaGetLastError();
}

// f(W, NK) as compile-time constants, for widths 2 .. 8 and 1 .. 8 channels.
template <int W, class F>
cudaError_t with_channels(int nk, F&& f) {
    using std::integral_constant;
    const integral_constant<int, W> w{};
    switch (nk) {
        case 1: return f(w, integral_constant<int, 1>{});
        case 2: return f(w, integral_constant<int, 2>{});
        case 3: return f(w, integral_constant<int, 3>{});
        case 4: return f(w, integral_constant<int, 4>{});
        case 5: return f(w, integral_constant<int, 5>{});
        case 6: return f(w, integral_constant<int, 6>{});
        case 7: return f(w, integral_constant<int, 7>{});
        case 8: return f(w, integral_constant<int, 8>{});
        default: return cudaErrorInvalidValue;
    }
}

template <class F>
cudaError_t with_tile(int W, int nk, F&& f) {
    switch (W) {
        case 2: return with_channels<2>(nk, f);
        case 3: return with_channels<3>(nk, f);
        case 4: return with_channels<4>(nk, f);
        case 5: return with_channels<5>(nk, f);
        case 6: return with_channels<6>(nk, f);
        case 7: return with_channels<7>(nk, f);
        case 8: return with_channels<8>(nk, f);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace

bool interp_tiles_supported(int W, int nk) { return W >= 2 && W <= 8 && nk >= 1 && nk <= 8; }

// Tiled over row time, geometric mean over 24^3, 48^3 and 80^3 images with 1 to 8 coils.  One
// channel: 0.78 at W = 4, but from W = 5 on the lanes of a row of W values mostly idle: 1.5 at W = 5,
// 1.4 at 6, 1.1 at 7, 1.4 at 8.  A plan for one coil a call is another matter, as the row kernel's
// gathers then serve one coil only.  Tiled and row us there, 16^3 with 371 thousand samples, 40^3 with
// 102 thousand, 90^3 with a million:
//   W = 5: 106 and 129, 37 and 39, 307 and 379     W = 6: 135 and 180, 47 and 55, 381 and 530
//   W = 7: 174 and 299, 57 and 90, 473 and 1030    W = 8: 221 and 188, 71 and 70, 612 and 756
// (W = 8 between them: 238 and 225 on a grid of 48^3 points, 297 and 311 on 80^3, 131 and 135 on 128^3.)
// Eight channels up to W = 4 put a point's values on the same banks as its neighbours': 1.4 at W = 2,
// 1.9 at 3, 2.1 at 4 (seven: 0.85 at W = 4).  At W = 2 a tile is copied for few taps: 0.86 and 0.89
// with two and three channels, 1.13, 1.01, 1.13 and 1.20 with four to seven.  The bits of a coil's
// samples do not depend on its minibatch, so the line is drawn by the most coils of the plan's calls,
// not by those of a call.
bool interp_tiles_faster(int W, int nk, int max_batch, long long points) {
    if (nk == 1) return W <= 4 || (max_batch == 1 && (W <= 7 || points >= 64LL * 64 * 64));
    return W >= 5 || nk <= (W == 2 ? 3 : 7);
}

cudaError_t launch_mv_interp_tiles(const MvArgs& a, const MvUnits& u, int W, int K, cudaStream_t st) {
    if (u.start[u.n] == 0) return cudaSuccess;
    // widths of the batched path (mv_width_supported)
    auto f = [&](auto w, auto k) { return launch_mv_tiles_k<decltype(w)::value, decltype(k)::value>(a, u, st); };
    return W == 4 ? with_channels<4>(K, f) : (W == 6 ? with_channels<6>(K, f) : cudaErrorInvalidValue);
}

cudaError_t launch_interp_tiles(const InterpTiles& a, const CUtensorMap& map, int nk, int withhold_row, long long wait_ns, cudaStream_t st) {
    if (a.ntiles == 0 || a.B == 0) return cudaSuccess;
    const unsigned long long wn = wait_ns > 0 ? (unsigned long long)wait_ns : tma::kWaitNs;
    return with_tile(a.g.W, nk, [&](auto w, auto k) {
        return launch_tiles_k<decltype(w)::value, decltype(k)::value>(a, map, withhold_row, wn, st);
    });
}

}  // namespace sdp
