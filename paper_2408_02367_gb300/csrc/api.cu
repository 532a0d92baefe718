// C ABI of the subspace multicoil NUFFT operator (declared in include/stodip_op.h):
// plan construction on the host (grid sizes, Kaiser-Bessel beta and
// deapodisation, FFT factorisation and twiddles, grid coordinates, bin sort,
// spread incidence lists), and the launch sequences of the forward operator
// A_c and its adjoint (StoDIP Sec. 2 Eq. 1, Sec. 2.1 Eq. 3, Algorithm 1).
#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <mutex>
#include <new>
#include <vector>

#include "batch.cuh"
#include "sdp_internal.cuh"
#include "spread_map.cuh"

using namespace sdp;

namespace {

constexpr double kPi = 3.14159265358979323846;
std::atomic<long long> g_launches{0};

struct ProfRec {
    int stage;
    cudaEvent_t a, b;
};

}  // namespace

void sdp::note_launches(long long n) { g_launches.fetch_add(n, std::memory_order_relaxed); }

constexpr int kTiledByRule = 2;   // a plan without a tuning: interp_tiles_faster()

struct sdp_plan_s {
    int dev = 0;
    Geo geo{};
    int64_t n[3] = {0, 0, 0};
    int64_t M[3] = {0, 0, 0};
    double sigma = 0, beta = 0;
    int maxB = 0;
    uint32_t flags = 0;
    FftAxis ax[3]{};
    int bs[3] = {0, 0, 0};    // the tuning's spread_bins
    int seg = 0;              // points of a spread unit along axis 3 (4 x 4 columns)
    int nu[3] = {0, 0, 0};    // spread units per axis
    int spread_chunk = 0;
    int fft_lines = 0, fft_cols = 0;   // the tuning's, reported back
    int interp_threads = 0;   // resolved CTA size of the interpolation kernel
    int spread_coils = 0;     // coils per spread warp: 0 = two where they fit, 1 = one
    int interp_run = 1;       // consecutive samples per interpolation warp run
    int interp_coils = 0;     // coils per interpolation sweep over the samples: 0 = all
    int interp_tiled = kTiledByRule;   // the interpolation where both have a kernel: 1 tiled (interp_tiles.cu), 0 rows
    int nt[3] = {0, 0, 0};    // interpolation tiles per axis
    int n_itiles = 0;         // tiled interpolation work items
    int wait_test_row = -1;   // test hook (sdp_plan_set_wait_test): a tile row the first CTA withholds
    long long wait_test_ns = 0;   // and the limit of the tiled kernel's waits (0: one second)
    int nunits = 0;
    int nsub = 0;
    long long ninc = 0;
    long long slots_per_b = 0;
    // device memory
    int4* wstart = nullptr;  // sorted samples: first tap per axis, in [0, M), and index in y (row kernels)
    int* tframe = nullptr;
    float* wts = nullptr;    // [J][3W] Kaiser-Bessel weights of the sorted samples
    float2* V = nullptr;
    float2* S = nullptr;
    float* dinv = nullptr;   // [N1 | N2 | N3]
    float2* tw = nullptr;    // [M1 | M2 | M3]
    int4* inc = nullptr;     // spread incidences (SpreadArgs::inc)
    float2* Vp = nullptr;    // V with rows of an even number of values (16-byte aligned)
    int4* srec = nullptr;    // sorted samples: index in y, frame, window start in the interpolation tile, 0
    SubProb* subs = nullptr;
    int4* itiles = nullptr;  // tiled interpolation work items (flat tile index, first sample, count, 0), heaviest first
    float2* partials = nullptr;
    int2* ranges = nullptr;  // chunks that reach each block of the multi-chunk units
    int* counters = nullptr;
    int* group_counters = nullptr;
    int* status = nullptr;
    double* loss_partials = nullptr;
    unsigned int* loss_counter = nullptr;
    double* tv_part = nullptr;
    unsigned int* tv_counter = nullptr;
    // Grid workspaces, channel-interleaved: a call with nk channels holds
    // [b][i1][i2][i3][kk] (kk fastest), so the W x nk values one row of a
    // Kaiser-Bessel window touches along axis 3 are one contiguous run.
    CUtensorMap grid_map{}, tile_map{};   // of bufA with all channels (K <= 8): the spread's and the interpolation's boxes
    int has_map = 0;
    StridedMaps fft_maps[4];   // inputs of the strided passes with all channels: forward axis 2, axis 1, inverse axis 1, axis 2
    int has_fft_map[2] = {0, 0};   // per axis: the axis has a two-pass length
    float2* bufA = nullptr;
    float2* bufB = nullptr;
    size_t workspace_bytes = 0;
    size_t total_bytes = 0;
    std::vector<void*> allocs;
    // batched calls: the stream of this plan's items beside those of other plans, and its ends
    cudaStream_t own = nullptr;
    cudaEvent_t forked = nullptr, joined = nullptr;
    // profiling
    bool prof = false;
    std::vector<ProfRec> prof_used;
    std::vector<ProfRec> prof_free;
    double prof_ms[kNumStages] = {0};
    long long prof_n[kNumStages] = {0};
};

namespace {

bool smooth235(long long m) {
    for (int p : {2, 3, 5})
        while (m % p == 0) m /= p;
    return m == 1;
}

long long grid_len(long long n, double sigma, int W) {
    long long m = std::max((long long)std::ceil(sigma * (double)n), 2LL * W);
    while ((m % 2) || !smooth235(m)) ++m;
    return m;
}

// Grid points of a spread unit along axis 3 (spread_impl.cuh): four times the depth of the spread
// bins, a tuning's or {8, 4, 4}.  A window meets (seg + W - 1) / seg units along axis 3,
// and longer units leave fewer warps to balance.  Spread of 2 coils on the 160^3 grid (W = 4,
// K = 5, 491,520 samples): 8 points 204 us, 16 points 190, 32 points 195; of 4 coils on 120^3:
// 293, 299, 322; one coil at W = 6 on 150 x 128 x 180: 131, 112, 105.
int spread_segment(const int bins[3]) { return 4 * bins[2]; }

// Upper bound of a spread subproblem's incidences, whatever the tuning asks for.  The k-space
// centre's units hold thousands: a long chunk is the last one running on a small problem, a
// short one costs partial sums.  128^3 workload (1.8 million incidences): 256 211 us, 512 190;
// 24^3, W = 6 (319 thousand): 128 87 us, 256 81, 512 92.
long long spread_chunk_cap(long long ninc) { return std::min(512LL, std::max(64LL, ninc / 1400)); }

constexpr int kDefaultBins[3] = {8, 4, 4};   // of a plan without a tuning

double i0(double x) { return std::cyl_bessel_i(0.0, x); }

// Continuous Fourier transform of the normalised Kaiser-Bessel window.
double kb_ft(double xi, int W, double beta) {
    const double z2 = beta * beta - (kPi * W * xi) * (kPi * W * xi);
    const double z = std::sqrt(std::fabs(z2));
    double v;
    if (z == 0.0)
        v = 1.0;
    else if (z2 > 0)
        v = std::sinh(z) / z;
    else
        v = std::sin(z) / z;
    return W * v / i0(beta);
}

template <typename T>
int dev_alloc(sdp_plan_s* p, T** ptr, size_t count) {
    *ptr = nullptr;
    if (count == 0) count = 1;
    void* q = nullptr;
    if (cudaMalloc(&q, count * sizeof(T)) != cudaSuccess) {
        cudaGetLastError();
        return SDP_ERR_OOM;
    }
    p->allocs.push_back(q);
    p->total_bytes += count * sizeof(T);
    *ptr = static_cast<T*>(q);
    return SDP_OK;
}

void free_plan(sdp_plan_s* p) {
    if (!p) return;
    cudaDeviceSynchronize();
    for (void* q : p->allocs) cudaFree(q);
    if (p->own) cudaStreamDestroy(p->own);
    if (p->forked) cudaEventDestroy(p->forked);
    if (p->joined) cudaEventDestroy(p->joined);
    for (auto& r : p->prof_used) {
        cudaEventDestroy(r.a);
        cudaEventDestroy(r.b);
    }
    for (auto& r : p->prof_free) {
        cudaEventDestroy(r.a);
        cudaEventDestroy(r.b);
    }
    delete p;
}

#define SDP_TRY(expr)                      \
    do {                                   \
        int _rc = (expr);                  \
        if (_rc != SDP_OK) return _rc;     \
    } while (0)

#define SDP_CUDA(expr)                     \
    do {                                   \
        if ((expr) != cudaSuccess) {       \
            cudaGetLastError();            \
            return SDP_ERR_CUDA;           \
        }                                  \
    } while (0)

// Grid coordinate of one axis, bit-for-bit the definition of the oracle:
// g = omega * (M / 2 pi) in float64, wrapped into [0, M), rounded to float32,
// a float32 equal to M becomes 0.  (Built with -ffp-contract=off.)
float grid_coord(float omega, long long M) {
    const double m = (double)M;
    const double s = m / (2.0 * kPi);
    double g = (double)omega * s;
    if (g < 0.0) g = g + m;
    if (g >= m) g = g - m;
    float g32 = (float)g;
    if (g32 >= (float)m) g32 = 0.0f;
    return g32;
}

int build_plan(sdp_plan_s* p, const sdp_plan_desc* d, const sdp_tuning* tn, cudaStream_t st) {
    const int W = d->width;
    const int K = d->K;
    const long long J = d->J;
    for (int a = 0; a < 3; ++a) {
        p->n[a] = d->n[a];
        p->M[a] = grid_len(d->n[a], d->oversamp, W);
        if (p->M[a] > (1 << 14)) return SDP_ERR_UNSUPPORTED;
    }
    const long long G = p->M[0] * p->M[1] * p->M[2];
    const long long nvox = p->n[0] * p->n[1] * p->n[2];
    // one coil's channel-interleaved grid [M1][M2][M3][K] is indexed with 32-bit offsets
    if (G * K >= (1LL << 31) || nvox >= (1LL << 31)) return SDP_ERR_UNSUPPORTED;
    p->sigma = d->oversamp;
    const double arg = (W / d->oversamp) * (W / d->oversamp) * (d->oversamp - 0.5) * (d->oversamp - 0.5) - 0.8;
    if (!(arg > 0)) return SDP_ERR_UNSUPPORTED;
    p->beta = kPi * std::sqrt(arg);
    p->maxB = d->max_batch;
    p->flags = d->flags;
    Geo& g = p->geo;
    for (int a = 0; a < 3; ++a) {
        g.N[a] = (int)p->n[a];
        g.M[a] = (int)p->M[a];
    }
    g.W = W;
    g.K = K;
    g.T = d->T;
    g.C = d->C;
    g.J = (int)J;
    g.beta = (float)p->beta;
    g.inv_i0_beta = (float)(1.0 / i0(p->beta));
    g.halfW = (float)(0.5 * W);
    for (int a = 0; a < 3; ++a) {
        if (!fft_factor(g.M[a], &p->ax[a])) return SDP_ERR_UNSUPPORTED;
        p->ax[a].generic = tn ? tn->fft_engine : 0;
        p->ax[a].staged = tn ? tn->fft_staged : fft2_staged_default(g.N[2], g.M[2], K);
    }
    p->fft_lines = tn ? tn->fft_lines : 0;
    p->fft_cols = tn ? tn->fft_cols : 0;
    // interpolation CTA size: the 1024-thread kernel is built for W <= 4 only
    const int ithreads = tn ? tn->interp_threads : 0;
    if (ithreads == 1024 && W > 4) return SDP_ERR_UNSUPPORTED;
    p->interp_threads = ithreads ? ithreads : 256;
    p->spread_coils = tn ? tn->spread_coils : 0;
    p->interp_run = (tn && tn->interp_run) ? tn->interp_run : 1;
    p->interp_coils = tn ? tn->interp_coils : 0;
    p->interp_tiled = tn ? tn->interp_tiled : kTiledByRule;

    // ---- host tables ----
    std::vector<float> dinv(p->n[0] + p->n[1] + p->n[2]);
    {
        size_t o = 0;
        for (int a = 0; a < 3; ++a)
            for (long long i = 0; i < p->n[a]; ++i) {
                const double nc = (double)(i - p->n[a] / 2);
                // times (-1)^n: the grids hold frequency m at index m + M/2.  The samples' dense
                // centre and most of their windows then lie inside the grid, where a tile is one
                // box, instead of on its corners, where every window wraps around.
                const double sign = (i - p->n[a] / 2) % 2 ? -1.0 : 1.0;
                dinv[o++] = (float)(sign / kb_ft(nc / (double)p->M[a], W, p->beta));
            }
    }
    std::vector<float2> tw;
    for (int a = 0; a < 3; ++a) {
        std::vector<float2> t = fft_twiddles(g.M[a]);
        tw.insert(tw.end(), t.begin(), t.end());
    }

    // ---- trajectory -> grid coordinates, frames ----
    std::vector<float> traj((size_t)J * 3);
    SDP_CUDA(cudaMemcpyAsync(traj.data(), d->traj, traj.size() * sizeof(float), cudaMemcpyDeviceToHost, st));
    SDP_CUDA(cudaStreamSynchronize(st));
    std::vector<int> frame((size_t)J);
    for (int t = 0; t < d->T; ++t)
        for (long long j = d->frame_offsets[t]; j < d->frame_offsets[t + 1]; ++j) frame[j] = t;
    std::vector<float> gc((size_t)J * 3);
    for (long long j = 0; j < J; ++j) {
        const float* om = &traj[(size_t)j * 3];
        if (!(std::fabs(om[0]) <= (float)kPi + 1e-6f && std::fabs(om[1]) <= (float)kPi + 1e-6f &&
              std::fabs(om[2]) <= (float)kPi + 1e-6f))
            return SDP_ERR_INVALID_ARG;
        for (int a = 0; a < 3; ++a) gc[(size_t)j * 3 + a] = grid_coord(om[a], p->M[a]);
    }

    // ---- spread units: 4 x 4 columns by seg points (spread_impl.cuh) ----
    for (int a = 0; a < 3; ++a) p->bs[a] = tn ? tn->spread_bins[a] : kDefaultBins[a];
    p->seg = spread_segment(p->bs);
    const int ue[3] = {4, 4, p->seg};
    for (int a = 0; a < 3; ++a) p->nu[a] = (int)((p->M[a] + ue[a] - 1) / ue[a]);
    const long long nunits = (long long)p->nu[0] * p->nu[1] * p->nu[2];
    if (nunits >= (1LL << 31)) return SDP_ERR_UNSUPPORTED;
    p->nunits = (int)nunits;

    // window start of each sample, and its sort key: samples are ordered by interpolation
    // tile (the tiled interpolation takes a tile's samples as
    // one range), then by 4^3 cell within the tile, both of the sample's own coordinate
    const float halfW = (float)(0.5 * W);
    int edge[3];
    for (int a = 0; a < 3; ++a) edge[a] = imap::tile_edge(W, a);
    constexpr int kCell = 4;
    long long BPT = 1;   // cells per tile
    for (int a = 0; a < 3; ++a) {
        p->nt[a] = (int)((p->M[a] + edge[a] - 1) / edge[a]);
        BPT *= edge[a] / kCell;
    }
    const long long ntiles = (long long)p->nt[0] * p->nt[1] * p->nt[2];
    const long long nkeys = ntiles * BPT;
    // Positions are on the shifted grid (index m + M/2 for frequency m).  m0: first tap, in
    // [0, M); estart: the window's start within the sample's tile.
    std::vector<int> m0((size_t)J * 3), estart((size_t)J);
    std::vector<long long> skey((size_t)J);
    for (long long j = 0; j < J; ++j) {
        long long ti = 0, li = 0;
        int e[3];
        for (int a = 0; a < 3; ++a) {
            const float gv = gc[(size_t)j * 3 + a];
            const float tt = gv - halfW;
            const int M = (int)p->M[a], c0 = (int)gv;   // gv < M
            const int sh = c0 + M / 2 < M ? M / 2 : M / 2 - M, c = c0 + sh;
            const int first = (int)std::ceil(tt) + sh;
            m0[(size_t)j * 3 + a] = first < 0 ? first + M : first;
            e[a] = first - (c / edge[a] * edge[a] - W / 2);
            if (e[a] < 0 || e[a] > edge[a]) return SDP_ERR_UNSUPPORTED;   // cannot happen: the window lies in the tile
            ti = ti * p->nt[a] + c / edge[a];
            li = li * (edge[a] / kCell) + c % edge[a] / kCell;
        }
        estart[(size_t)j] = imap::tile_start(W, e[0], e[1], e[2]);
        skey[j] = ti * BPT + li;
    }
    // stable counting sort of samples by key
    std::vector<long long> cnt((size_t)nkeys + 1, 0);
    for (long long j = 0; j < J; ++j) cnt[(size_t)skey[j] + 1]++;
    for (long long b = 0; b < nkeys; ++b) cnt[(size_t)b + 1] += cnt[(size_t)b];
    std::vector<int> perm((size_t)J);   // sorted position -> original sample
    {
        std::vector<long long> cur(cnt.begin(), cnt.end() - 1);
        for (long long j = 0; j < J; ++j) perm[(size_t)cur[(size_t)skey[j]]++] = (int)j;
    }
    // the tiled interpolation's work items (flattened tile index, first sorted sample,
    // count), heaviest first: every non-empty tile, a dense one (the k-space centre holds
    // tiles of thousands of samples) cut into near-equal pieces of at most kTileItem
    // samples, each of which copies the tile's grid once per coil
    // (a small problem's into shorter ones, so that there are a few per resident CTA)
    const long long kTileItem = std::min(512LL, std::max(128LL, J * p->maxB / 2048));
    std::vector<int4> itiles;
    for (long long t = 0; t < ntiles; ++t) {
        const long long c0 = cnt[(size_t)(t * BPT)], c1 = cnt[(size_t)((t + 1) * BPT)];
        const long long n = c1 - c0, parts = (n + kTileItem - 1) / kTileItem;
        for (long long q = 0; q < parts; ++q) {
            const long long a = c0 + n * q / parts, b = c0 + n * (q + 1) / parts;
            itiles.push_back(make_int4((int)t, (int)a, (int)(b - a), 0));
        }
    }
    std::stable_sort(itiles.begin(), itiles.end(), [](const int4& a, const int4& b) { return a.z > b.z; });
    p->n_itiles = (int)itiles.size();
    std::vector<float4> pts((size_t)J);
    std::vector<int> tf((size_t)J);
    for (long long s = 0; s < J; ++s) {
        const int j = perm[s];
        pts[s] = make_float4(gc[(size_t)j * 3], gc[(size_t)j * 3 + 1], gc[(size_t)j * 3 + 2], 0.f);
        tf[s] = frame[j];
    }

    // incidences: (unit, sorted sample) for every unit a window touches, in order of unit,
    // then plane (the window's start relative to the unit), then sample.  Along axis 3 a window
    // on a grid shorter than seg + W - 1 points can meet a unit in two pieces: two incidences,
    // the second's plane one grid length further.  Everything depends on the window's first tap
    // along each axis, so it is tabulated per tap: the units met and, for the spread kernel,
    // window_k (axes 1 and 2) or the plane (axis 3).
    const int M3 = (int)p->M[2], seg = p->seg, nplanes = seg + W - 1;
    auto seg_points = [&](int u3) { return std::min(seg, M3 - u3 * seg); };
    struct Meet {
        int unit, k;
    };
    std::vector<Meet> meets[3];
    std::vector<int> meet0[3];   // meets of first tap m: [meet0[m], meet0[m + 1])
    for (int a = 0; a < 3; ++a) {
        const int M = (int)p->M[a], edge = ue[a];
        meet0[a].push_back(0);
        for (int m = 0; m < M; ++m) {
            imap::unit_meets(W, M, edge, a == 2, m, [&](int unit, int k) { meets[a].push_back({unit, k}); });
            meet0[a].push_back((int)meets[a].size());
        }
    }
    // calls f(unit * nplanes + plane, k) for every incidence of sample j
    auto each_incidence = [&](int j, auto&& f) {
        const int* mm = &m0[(size_t)j * 3];
        const Meet *x = &meets[0][(size_t)meet0[0][(size_t)mm[0]]], *xe = &meets[0][0] + meet0[0][(size_t)mm[0] + 1];
        const Meet *y0 = &meets[1][(size_t)meet0[1][(size_t)mm[1]]], *ye = &meets[1][0] + meet0[1][(size_t)mm[1] + 1];
        const Meet *z0 = &meets[2][(size_t)meet0[2][(size_t)mm[2]]], *ze = &meets[2][0] + meet0[2][(size_t)mm[2] + 1];
        for (; x < xe; ++x)
            for (const Meet* y = y0; y < ye; ++y) {
                const long long c = ((long long)x->unit * p->nu[1] + y->unit) * p->nu[2];
                for (const Meet* z = z0; z < ze; ++z) f((c + z->unit) * nplanes + z->k, x->k | y->k << 8 | z->k << 16);
            }
    };
    std::vector<unsigned> first((size_t)nunits * nplanes + 1, 0);   // first incidence of (unit, plane)
    long long ninc = 0;
    for (long long s = 0; s < J; ++s)
        each_incidence(perm[(size_t)s], [&](long long q, int) {
            ++first[(size_t)q + 1];
            ++ninc;
        });
    if (ninc >= (1LL << 31)) return SDP_ERR_UNSUPPORTED;
    for (size_t q = 0; q + 1 < first.size(); ++q) first[q + 1] += first[q];
    p->ninc = ninc;
    std::vector<int4> inc((size_t)std::max(ninc, 1LL), make_int4(0, 0, 0, 0));
    {
        std::vector<unsigned> cur(first.begin(), first.end() - 1);
        for (long long s = 0; s < J; ++s)
            each_incidence(perm[(size_t)s], [&](long long q, int k) {
                inc[cur[(size_t)q]++] = make_int4((int)s, k, perm[(size_t)s], frame[(size_t)perm[(size_t)s]]);
            });
    }
    std::vector<int4> srec((size_t)J), wstart((size_t)J);
    for (long long s = 0; s < J; ++s) {
        const int j = perm[(size_t)s];
        srec[(size_t)s] = make_int4(j, frame[(size_t)j], estart[(size_t)j], 0);
        wstart[(size_t)s] = make_int4(m0[(size_t)j * 3], m0[(size_t)j * 3 + 1], m0[(size_t)j * 3 + 2], j);
    }
    // subproblems: every unit (empty ones too, they write zeros), chunks of at most kChunk
    long long kChunk = 512;
    if (tn)
        kChunk = tn->spread_chunk;
    else if (const char* ev = std::getenv("SDP_SPREAD_CHUNK"))
        kChunk = std::min(65536LL, std::max(32LL, std::atoll(ev)));
    p->spread_chunk = (int)kChunk;
    kChunk = std::min(kChunk, spread_chunk_cap(ninc));
    std::vector<SubProb> subs;
    std::vector<int2> ranges;   // [multi-chunk unit][block of four positions]: the chunks [x, y) that reach it
    const int nblk = seg / 4;
    int multi = 0;
    long long slots = 0;
    for (long long b = 0; b < nunits; ++b) {
        const long long c0 = first[(size_t)(b * nplanes)], n = first[(size_t)((b + 1) * nplanes)] - c0;
        const int nch = (int)std::max(1LL, (n + kChunk - 1) / kChunk);
        const int u3 = (int)(b % p->nu[2]), top = seg_points(u3) + W - 2;
        if (nch > 1) ranges.resize((size_t)(multi + 1) * nblk, make_int2(0, 0));
        auto of = [&](const int4& e) { return e.y >> 16; };
        // a chunk's planes run on to the next chunk's first, so that together they cover the unit
        for (int ch = 0; ch < nch; ++ch) {
            SubProb sp;
            sp.bin = (int)b;
            sp.start = (int)(c0 + n * ch / nch);
            sp.count = (int)(c0 + n * (ch + 1) / nch) - sp.start;
            sp.chunk = ch;
            sp.nchunks = nch;
            sp.slot = nch > 1 ? (int)slots : 0;
            sp.r0 = ch == 0 ? 0 : of(inc[(size_t)sp.start]);
            sp.r1 = ch == nch - 1 ? top : std::max(of(inc[(size_t)(sp.start + sp.count - 1)]),
                                                   of(inc[(size_t)(sp.start + sp.count)]) - 1);
            sp.multi = multi;
            if (nch > 1)
                for (int q = imap::spread_block_lo(sp.r0, W); q <= imap::spread_block_hi(sp.r1, seg_points(u3)); ++q) {
                    int2& rg = ranges[(size_t)multi * nblk + q];
                    if (rg.y == 0) rg.x = ch;
                    rg.y = ch + 1;
                }
            subs.push_back(sp);
        }
        if (nch > 1) {
            slots += nch;
            ++multi;
        }
    }
    // heaviest subproblems first
    std::stable_sort(subs.begin(), subs.end(), [](const SubProb& a, const SubProb& b) { return a.count > b.count; });
    p->nsub = (int)subs.size();
    p->slots_per_b = slots;

    // ---- device memory ----
    const size_t Kz = (size_t)K;
    SDP_TRY(dev_alloc(p, &p->wstart, (size_t)J));
    SDP_TRY(dev_alloc(p, &p->tframe, (size_t)J));
    SDP_TRY(dev_alloc(p, &p->wts, (size_t)J * 3 * W));
    SDP_TRY(dev_alloc(p, &p->V, (size_t)d->T * Kz));
    const size_t Kp = (Kz + 1) & ~(size_t)1;
    SDP_TRY(dev_alloc(p, &p->Vp, (size_t)d->T * Kp));
    if (d->flags & SDP_FLAG_BORROW_MAPS)
        p->S = const_cast<float2*>(static_cast<const float2*>(d->coil_maps));   // read only, caller-owned
    else
        SDP_TRY(dev_alloc(p, &p->S, (size_t)d->C * nvox));
    SDP_TRY(dev_alloc(p, &p->dinv, dinv.size()));
    SDP_TRY(dev_alloc(p, &p->tw, tw.size()));
    SDP_TRY(dev_alloc(p, &p->inc, inc.size()));
    SDP_TRY(dev_alloc(p, &p->srec, (size_t)J));
    SDP_TRY(dev_alloc(p, &p->subs, subs.size()));
    SDP_TRY(dev_alloc(p, &p->itiles, std::max<size_t>(itiles.size(), 1)));
    const size_t P = (size_t)16 * p->seg;   // grid points of a unit
    SDP_TRY(dev_alloc(p, &p->partials, (size_t)std::max(slots, 1LL) * P * Kz * p->maxB));
    const size_t ncount = (size_t)nunits * (p->seg / 4) * p->maxB * ((K + 7) / 8);
    SDP_TRY(dev_alloc(p, &p->ranges, ranges.size()));
    const size_t gcount = (size_t)std::max(slots, 1LL) * (p->seg / 4) * p->maxB * ((K + 7) / 8);
    SDP_TRY(dev_alloc(p, &p->counters, ncount));
    SDP_TRY(dev_alloc(p, &p->group_counters, gcount));
    SDP_TRY(dev_alloc(p, &p->status, 1));
    SDP_TRY(dev_alloc(p, &p->loss_partials, (size_t)residual_loss_partials(p->maxB, J)));
    SDP_TRY(dev_alloc(p, &p->loss_counter, 1));
    SDP_TRY(dev_alloc(p, &p->tv_part, (size_t)tv_partials(K, (int)p->n[0], (int)p->n[1], (int)p->n[2])));
    SDP_TRY(dev_alloc(p, &p->tv_counter, 1));
    const size_t before = p->total_bytes;
    const size_t gridA = (size_t)std::max<long long>(G, p->n[0] * p->n[1] * p->M[2]);
    const size_t gridB = (size_t)(p->n[0] * p->M[1] * p->M[2]);
    SDP_TRY(dev_alloc(p, &p->bufA, gridA * Kz * p->maxB));
    SDP_TRY(dev_alloc(p, &p->bufB, gridB * Kz * p->maxB));
    p->workspace_bytes = p->total_bytes - before;

    if (K <= 8) {
        SDP_TRY(grid_tensor_map(&p->grid_map, p->bufA, K, p->M, p->maxB, 4, 4, 4));
        // (the tiled interpolation needs 16 points per axis, the largest box)
        if (p->M[0] >= 16 && p->M[1] >= 16 && p->M[2] >= 16)
            SDP_TRY(grid_tensor_map(&p->tile_map, p->bufA, K, p->M, p->maxB, imap::tile_points(W, 0),
                                    imap::tile_points(W, 1), imap::tile_points(W, 2)));
        p->has_map = 1;
    }
    {
        const long long N1 = p->n[0], N2 = p->n[1], M1 = p->M[0], M2 = p->M[1], in2 = p->M[2] * K, in1 = M2 * in2;
        if (fft2_supported((int)M2)) {
            SDP_TRY(strided_tensor_maps(&p->fft_maps[0], p->bufA, (int)M2, (int)N2, 1, in2, p->maxB * N1));
            SDP_TRY(strided_tensor_maps(&p->fft_maps[3], p->bufB, (int)M2, (int)M2, 0, in2, p->maxB * N1));
            p->has_fft_map[1] = 1;
        }
        if (fft2_supported((int)M1)) {
            SDP_TRY(strided_tensor_maps(&p->fft_maps[1], p->bufB, (int)M1, (int)N1, 1, in1, p->maxB));
            SDP_TRY(strided_tensor_maps(&p->fft_maps[2], p->bufA, (int)M1, (int)M1, 0, in1, p->maxB));
            p->has_fft_map[0] = 1;
        }
    }
    SDP_CUDA(cudaMemcpyAsync(p->tframe, tf.data(), tf.size() * sizeof(int), cudaMemcpyHostToDevice, st));
    SDP_CUDA(cudaMemcpyAsync(p->V, d->V, (size_t)d->T * Kz * sizeof(float2), cudaMemcpyDeviceToDevice, st));
    SDP_CUDA(cudaMemsetAsync(p->Vp, 0, (size_t)d->T * Kp * sizeof(float2), st));
    SDP_CUDA(cudaMemcpy2DAsync(p->Vp, Kp * sizeof(float2), d->V, Kz * sizeof(float2), Kz * sizeof(float2), d->T,
                               cudaMemcpyDeviceToDevice, st));
    if (!(d->flags & SDP_FLAG_BORROW_MAPS))
        SDP_CUDA(cudaMemcpyAsync(p->S, d->coil_maps, (size_t)d->C * nvox * sizeof(float2), cudaMemcpyDeviceToDevice,
                                 st));
    SDP_CUDA(cudaMemcpyAsync(p->dinv, dinv.data(), dinv.size() * sizeof(float), cudaMemcpyHostToDevice, st));
    SDP_CUDA(cudaMemcpyAsync(p->tw, tw.data(), tw.size() * sizeof(float2), cudaMemcpyHostToDevice, st));
    SDP_CUDA(cudaMemcpyAsync(p->inc, inc.data(), inc.size() * sizeof(int4), cudaMemcpyHostToDevice, st));
    SDP_CUDA(cudaMemcpyAsync(p->srec, srec.data(), srec.size() * sizeof(int4), cudaMemcpyHostToDevice, st));
    if (!ranges.empty())
        SDP_CUDA(cudaMemcpyAsync(p->ranges, ranges.data(), ranges.size() * sizeof(int2), cudaMemcpyHostToDevice, st));
    SDP_CUDA(cudaMemcpyAsync(p->subs, subs.data(), subs.size() * sizeof(SubProb), cudaMemcpyHostToDevice, st));
    if (!itiles.empty())
        SDP_CUDA(cudaMemcpyAsync(p->itiles, itiles.data(), itiles.size() * sizeof(int4), cudaMemcpyHostToDevice, st));
    SDP_CUDA(cudaMemsetAsync(p->counters, 0, ncount * sizeof(int), st));
    SDP_CUDA(cudaMemsetAsync(p->group_counters, 0, gcount * sizeof(int), st));
    SDP_CUDA(cudaMemsetAsync(p->status, 0, sizeof(int), st));
    SDP_CUDA(cudaMemsetAsync(p->loss_counter, 0, sizeof(unsigned int), st));
    SDP_CUDA(cudaMemsetAsync(p->tv_counter, 0, sizeof(unsigned int), st));
    // the weights are made from the coordinates, whose place the window starts then take
    static_assert(sizeof(float4) == sizeof(int4), "one table after the other");
    SDP_CUDA(cudaMemcpyAsync(p->wstart, pts.data(), pts.size() * sizeof(float4), cudaMemcpyHostToDevice, st));
    SDP_CUDA(launch_kb_weights(g, reinterpret_cast<const float4*>(p->wstart), p->wts, st));
    SDP_CUDA(cudaMemcpyAsync(p->wstart, wstart.data(), wstart.size() * sizeof(int4), cudaMemcpyHostToDevice, st));
    SDP_CUDA(cudaStreamSynchronize(st));
    size_t o = 0;
    for (int a = 0; a < 3; ++a) {
        p->ax[a].tw = p->tw + o;
        o += (size_t)g.M[a];
    }
    return SDP_OK;
}

// ---- profiling hooks ----
int prof_begin(sdp_plan_s* p, cudaStream_t st, ProfRec* rec) {
    if (!p->prof) return SDP_OK;
    if (p->prof_free.empty()) {
        ProfRec r;
        if (cudaEventCreate(&r.a) != cudaSuccess || cudaEventCreate(&r.b) != cudaSuccess) {
            cudaGetLastError();
            return SDP_ERR_CUDA;
        }
        p->prof_free.push_back(r);
    }
    *rec = p->prof_free.back();
    p->prof_free.pop_back();
    SDP_CUDA(cudaEventRecord(rec->a, st));
    return SDP_OK;
}

int prof_end(sdp_plan_s* p, cudaStream_t st, ProfRec* rec, int stage) {
    if (!p->prof) return SDP_OK;
    rec->stage = stage;
    SDP_CUDA(cudaEventRecord(rec->b, st));
    p->prof_used.push_back(*rec);
    return SDP_OK;
}

template <typename F>
int run(sdp_plan_s* p, int stage, cudaStream_t st, F&& f) {
    ProfRec rec{};
    SDP_TRY(prof_begin(p, st, &rec));
    const cudaError_t e = f();
    g_launches.fetch_add(1, std::memory_order_relaxed);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return SDP_ERR_CUDA;
    }
    return prof_end(p, st, &rec, stage);
}

const float* dinv_axis(const sdp_plan_s* p, int a) {
    size_t o = 0;
    for (int q = 0; q < a; ++q) o += (size_t)p->n[q];
    return p->dinv + o;
}

int check_call(const sdp_plan_s* p, const void* in, const int32_t* coil_idx, int B, int k0, int nk,
               const void* out) {
    if (!p || !in || !coil_idx || !out) return SDP_ERR_INVALID_ARG;
    if (B < 1 || B > p->maxB) return SDP_ERR_INVALID_ARG;
    if (k0 < 0 || nk < 1 || k0 + nk > p->geo.K) return SDP_ERR_INVALID_ARG;
    return SDP_OK;
}

SpreadArgs spread_args(const sdp_plan_s* p, const float2* y, const float* scale, int k0, int nk, int coil_off) {
    SpreadArgs a{};
    a.g = p->geo;
    a.seg = p->seg;
    a.nb1 = p->nu[0];
    a.nb2 = p->nu[1];
    a.nb3 = p->nu[2];
    a.subs = p->subs;
    a.inc = p->inc;
    a.wts = p->wts;
    a.V = p->Vp;
    a.vstride = (p->geo.K + 1) & ~1;
    a.y = y;
    a.scale = scale;
    a.k0 = k0;
    a.nk = nk;
    a.grids = p->bufA;
    a.slots_per_b = p->slots_per_b;
    a.slot_elems = (long long)p->geo.K * 16 * p->seg;
    a.partials = p->partials + (size_t)coil_off * (size_t)p->slots_per_b * (size_t)a.slot_elems;
    a.ranges = p->ranges;
    a.nblk = p->seg / 4;
    a.counters = p->counters + (size_t)coil_off * (size_t)p->nunits * a.nblk;
    a.group_counters = p->group_counters + (size_t)coil_off * (size_t)p->slots_per_b * a.nblk;
    a.nbins = p->nunits;
    a.coil0 = coil_off;
    // the map describes grids of all channels (G >= N1 N2 M3, so they follow one another)
    a.use_map = p->has_map && nk == p->geo.K;
    a.ngroups = 1;
    a.group = 0;
    return a;
}

// Whether step A3 of a call with nk channels runs the tiled interpolation: the plan
// asks for it, a kernel exists for the width and channel count, and every grid axis
// has at least 16 points (a tile with its margin then wraps around it at most once).
bool plan_interp_tiled(const sdp_plan_s* p, int nk) {
    const Geo& g = p->geo;
    const bool wanted = p->interp_tiled == kTiledByRule ? interp_tiles_faster(g.W, nk, p->maxB, p->M[0] * p->M[1] * p->M[2])
                                                        : p->interp_tiled != 0;
    return wanted && interp_tiles_supported(g.W, nk) && g.M[0] >= 16 && g.M[1] >= 16 && g.M[2] >= 16;
}

// Step A3 of the plan: the tiled interpolation where the plan asks for it and a kernel
// exists for the width and channel count, else the row kernel.
cudaError_t plan_interp(const sdp_plan_s* p, const float2* grids, int B, int k0, int nk, float2* y, int accumulate,
                        cudaStream_t st) {
    const Geo& g = p->geo;
    if (plan_interp_tiled(p, nk)) {
        InterpTiles a{g, p->itiles, p->n_itiles, p->nt[1], p->nt[2], p->srec, p->wts, p->Vp, (g.K + 1) & ~1, grids, B, k0,
                      y, accumulate,
                      p->status, 0, p->has_map && nk == g.K};
        return launch_interp_tiles(a, p->tile_map, nk, p->wait_test_row, p->wait_test_ns, st);
    }
    return launch_interp(g, p->interp_threads, p->interp_run, p->interp_coils, p->wstart, p->tframe, p->wts, p->V, grids,
                         B, k0, nk, y, accumulate, st);
}

// The tensor maps of strided pass `i` along `axis` for a call on nk channels, if it has any.
const StridedMaps* pass_maps(const sdp_plan_s* p, int i, int axis, int nk) {
    return p->has_fft_map[axis] && nk == p->geo.K ? &p->fft_maps[i] : nullptr;
}

int forward_impl(sdp_plan_s* p, const void* x, const int32_t* coil_idx, int B, int k0, int nk, void* y,
                 int accumulate, cudaStream_t st) {
    SDP_TRY(check_call(p, x, coil_idx, B, k0, nk, y));
    const Geo& g = p->geo;
    const long long N1 = g.N[0], N2 = g.N[1];
    const long long M1 = g.M[0], M2 = g.M[1], M3 = g.M[2];
    const float2* xs = static_cast<const float2*>(x);
    SDP_TRY(run(p, ST_FWD_FFT3, st, [&] {
        return launch_fwd_prologue_fft3(g, p->ax[2], xs, p->S, coil_idx, B, k0, nk, dinv_axis(p, 0),
                                        dinv_axis(p, 1), dinv_axis(p, 2), p->bufA, p->status, st);
    }));
    SDP_TRY(run(p, ST_FWD_FFT2, st, [&] {
        return launch_fft_strided(p->ax[1], 0, p->bufA, p->bufB, (int)N2, 1, (int)M2, 0, M3 * nk, B * N1,
                                  pass_maps(p, 0, 1, nk), p->status, st);
    }));
    SDP_TRY(run(p, ST_FWD_FFT1, st, [&] {
        return launch_fft_strided(p->ax[0], 0, p->bufB, p->bufA, (int)N1, 1, (int)M1, 0, M2 * M3 * nk, B,
                                  pass_maps(p, 1, 0, nk), p->status, st);
    }));
    SDP_TRY(run(p, ST_INTERP, st, [&] {
        return plan_interp(p, p->bufA, B, k0, nk, static_cast<float2*>(y), accumulate, st);
    }));
    return SDP_OK;
}

int adjoint_impl(sdp_plan_s* p, const void* y, const int32_t* coil_idx, int B, int k0, int nk, void* out,
                 int accumulate, const float* scale, cudaStream_t st) {
    SDP_TRY(check_call(p, y, coil_idx, B, k0, nk, out));
    const Geo& g = p->geo;
    const long long N1 = g.N[0], N2 = g.N[1];
    const long long M1 = g.M[0], M2 = g.M[1], M3 = g.M[2];
    SDP_TRY(run(p, ST_SPREAD, st, [&] {
        return launch_spread(spread_args(p, static_cast<const float2*>(y), scale, k0, nk, 0), p->grid_map, p->nsub, B,
                             p->spread_coils, st);
    }));
    SDP_TRY(run(p, ST_ADJ_FFT1, st, [&] {
        return launch_fft_strided(p->ax[0], 1, p->bufA, p->bufB, (int)M1, 0, (int)N1, 1, M2 * M3 * nk, B,
                                  pass_maps(p, 2, 0, nk), p->status, st);
    }));
    SDP_TRY(run(p, ST_ADJ_FFT2, st, [&] {
        return launch_fft_strided(p->ax[1], 1, p->bufB, p->bufA, (int)M2, 0, (int)N2, 1, M3 * nk, B * N1,
                                  pass_maps(p, 3, 1, nk), p->status, st);
    }));
    SDP_TRY(run(p, ST_ADJ_FFT3, st, [&] {
        return launch_adj_fft3_epilogue(g, p->ax[2], p->bufA, p->S, coil_idx, B, k0, nk, dinv_axis(p, 0),
                                        dinv_axis(p, 1), dinv_axis(p, 2), static_cast<float2*>(out), accumulate,
                                        p->status, st);
    }));
    return SDP_OK;
}

// ---- batched calls in one launch per stage (batch.cu) ----

// Whether the items can share launches: the same kernel width, channel count,
// spread bin shape and interpolation kernel (CTA size, tiled or not); one
// channel group (K <= 8 and K <= 32 / W); every grid length served by the
// two-pass FFT.
bool fused_eligible(const sdp_work* items, int n) {
    if (n < 1) return false;
    const sdp_plan_s* p0 = items[0].plan;
    for (int i = 0; i < n; ++i) {
        const sdp_plan_s* p = items[i].plan;
        if (p->geo.W != p0->geo.W || p->geo.K != p0->geo.K ||
            p->interp_threads != p0->interp_threads || p->interp_coils != p0->interp_coils ||
            plan_interp_tiled(p, p->geo.K) != plan_interp_tiled(p0, p0->geo.K))
            return false;
        if (p->geo.K > 8 || p->geo.K > 32 / p->geo.W || !mv_width_supported(p->geo.W)) return false;
        for (int a = 0; a < 3; ++a)
            if (p->ax[a].generic || !mv_length_supported(p->geo.M[a])) return false;
    }
    return true;
}

// Grid values (coils x channels x grid points) of a batch, and the most of them that take one
// launch per stage.  Up to there a batch is four launches on the caller's own stream, whatever its
// number of items; that is what a caller of many small items gets, and not always the least time: the
// batched kernels pay for their generality (any length and plan per unit).  Forward + adjoint in one
// launch per stage against each plan's own kernels on the plans' streams: four volumes on 48^3 grids
// (2.2 M values) 390 us and 351, two on 80^3 (5 M) 323 and 261, two on 120^3 (17 M) 573 and 435; eight
// items of one plan on 80^3, which cannot overlap (20 M), 1034 and 1343.  Larger batches gain more
// from their own kernels, 10% of half a millisecond and up: the four volumes of 64^3 to
// 128 x 128 x 96 (166 M) with loss 4724 us and 4129.
constexpr long long kFusedMost = 1LL << 25;
long long batch_values(const sdp_work* items, int n) {
    long long v = 0;
    for (int i = 0; i < n; ++i) {
        const sdp_plan_s* p = items[i].plan;
        v += (long long)items[i].B * p->geo.K * p->M[0] * p->M[1] * p->M[2];
    }
    return v;
}

// One wave: items whose plans have room for all their coils at once.  Fills
// the launch descriptors and runs the four stages of one direction.
int run_wave(const sdp_work* items, const std::vector<int>& idx, const std::vector<int>& coil_off, bool adjoint,
             cudaStream_t st) {
    MvArgs a;
    std::memset(&a, 0, sizeof(a));
    const int n = (int)idx.size();
    const sdp_plan_s* p0 = items[idx[0]].plan;
    const bool tiled = plan_interp_tiled(p0, p0->geo.K);   // the plans agree (fused_eligible)
    for (int q = 0; q < n; ++q) {
        const sdp_work& w = items[idx[q]];
        sdp_plan_s* p = w.plan;
        const Geo& g = p->geo;
        MvItem& it = a.it[q];
        const long long N1 = g.N[0], N2 = g.N[1];
        const long long M1 = g.M[0], M2 = g.M[1], M3 = g.M[2];
        const long long K = g.K;
        const size_t gridA = (size_t)std::max<long long>(M1 * M2 * M3, N1 * N2 * M3);
        const size_t gridB = (size_t)(N1 * M2 * M3);
        it.g = g;
        for (int d = 0; d < 3; ++d) {
            it.L[d] = g.M[d];
            it.tw[d] = p->ax[d].tw;
            it.d[d] = dinv_axis(p, d);
        }
        it.S = p->S;
        it.coil_idx = w.coil_idx;
        it.B = w.B;
        it.accumulate = w.accumulate ? 1 : 0;
        it.status = p->status;
        it.bufA = p->bufA + (size_t)coil_off[q] * gridA * K;
        it.bufB = p->bufB + (size_t)coil_off[q] * gridB * K;
        it.wstart = p->wstart;
        it.tframe = p->tframe;
        it.wts = p->wts;
        it.V = p->V;
        if (adjoint) {
            it.x = static_cast<float2*>(w.out);
            it.pass[0] = MvPass{it.bufA, it.bufB, (int)M1, 0, (int)N1, 1, M2 * M3 * K};
            it.pass[1] = MvPass{it.bufB, it.bufA, (int)M2, 0, (int)N2, 1, M3 * K};
        } else {
            it.x = const_cast<float2*>(static_cast<const float2*>(w.in));
            it.y = static_cast<float2*>(w.out);
            it.pass[1] = MvPass{it.bufA, it.bufB, (int)N2, 1, (int)M2, 0, M3 * K};
            it.pass[0] = MvPass{it.bufB, it.bufA, (int)N1, 1, (int)M1, 0, M2 * M3 * K};
        }
        it.sa = spread_args(p, adjoint ? static_cast<const float2*>(w.in) : nullptr, nullptr, 0, g.K, coil_off[q]);
        it.sa.grids = it.bufA;
        it.grid_map = p->grid_map;
        it.tile_map = p->tile_map;
        it.coil0 = coil_off[q];
        it.nsub = p->nsub;
        it.spread_pairs = (p->spread_coils != 1 && w.B >= 2) ? 1 : 0;
        it.interp_coils = p->interp_coils > 0 && p->interp_coils < w.B ? p->interp_coils : w.B;
        it.srec = p->srec;
        it.Vp = p->Vp;
        it.vstride = (g.K + 1) & ~1;
        it.itiles = p->itiles;
        it.n_itiles = p->n_itiles;
        it.nt2 = p->nt[1];
        it.nt3 = p->nt[2];
    }
    // units of each stage
    auto units = [&](auto count) {
        MvUnits u;
        u.n = n;
        u.start[0] = 0;
        for (int q = 0; q < n; ++q) u.start[q + 1] = u.start[q] + count(a.it[q]);
        return u;
    };
    auto ceil_div = [](long long x, long long y) { return (x + y - 1) / y; };
    const MvUnits u_fused_fwd = units([&](const MvItem& it) {
        return ceil_div((long long)it.g.N[0] * it.g.N[1] * it.g.K, mv_fused_lines(it.L[2])) * it.B;
    });
    const MvUnits u_fused_adj = units([&](const MvItem& it) {
        return ceil_div((long long)it.g.N[0] * it.g.N[1] * it.g.K, mv_fused_lines(it.L[2]));
    });
    auto u_strided = [&](int axis) {
        return units([&](const MvItem& it) {
            const long long outer = axis == 1 ? (long long)it.B * it.g.N[0] : (long long)it.B;
            return ceil_div(it.pass[axis].inner, mv_strided_cols(it.L[axis])) * outer;
        });
    };
    // stage timing (sdp_profile_*) is recorded on the first item's plan
    sdp_plan_s* pf = items[idx[0]].plan;
    if (!adjoint) {
        const MvUnits u2 = u_strided(1), u1 = u_strided(0);
        const MvUnits us = tiled ? units([&](const MvItem& it) { return (long long)it.n_itiles * it.B; })
                                 : units([&](const MvItem& it) { return (long long)it.g.J; });
        SDP_TRY(run(pf, ST_FWD_FFT3, st, [&] { return launch_mv_prologue(a, u_fused_fwd, st); }));
        SDP_TRY(run(pf, ST_FWD_FFT2, st, [&] { return launch_mv_strided(a, u2, 1, 0, st); }));
        SDP_TRY(run(pf, ST_FWD_FFT1, st, [&] { return launch_mv_strided(a, u1, 0, 0, st); }));
        SDP_TRY(run(pf, ST_INTERP, st, [&] {
            return tiled ? launch_mv_interp_tiles(a, us, p0->geo.W, p0->geo.K, st)
                         : launch_mv_interp(a, us, p0->geo.W, p0->interp_threads, st);
        }));
    } else {
        const MvUnits u1 = u_strided(0), u2 = u_strided(1);
        const MvUnits usp = units([&](const MvItem& it) {
            return (long long)it.nsub * (it.spread_pairs ? (it.B + 1) / 2 : it.B);
        });
        SDP_TRY(run(pf, ST_SPREAD, st, [&] { return launch_mv_spread(a, usp, p0->geo.W, p0->geo.K, st); }));
        SDP_TRY(run(pf, ST_ADJ_FFT1, st, [&] { return launch_mv_strided(a, u1, 0, 1, st); }));
        SDP_TRY(run(pf, ST_ADJ_FFT2, st, [&] { return launch_mv_strided(a, u2, 1, 1, st); }));
        SDP_TRY(run(pf, ST_ADJ_FFT3, st, [&] { return launch_mv_epilogue(a, u_fused_adj, st); }));
    }
    return SDP_OK;
}

// Bytes an item writes: y [B][J] (forward) or out [K][N1][N2][N3] (adjoint).
std::pair<uintptr_t, uintptr_t> out_range(const sdp_work& w, bool adjoint) {
    const sdp_plan_s* p = w.plan;
    const size_t n = adjoint ? (size_t)p->geo.K * p->n[0] * p->n[1] * p->n[2] : (size_t)w.B * p->geo.J;
    const uintptr_t a = reinterpret_cast<uintptr_t>(w.out);
    return {a, a + n * sizeof(float2)};
}

// Items in order; an item joins the current wave while its plan has room for
// its coils there (items of one plan take consecutive coil slices of the
// plan's workspace) and its output does not overlap the output of an item
// already in the wave (two items adding into one image must not run in the
// same launch), else the wave is run and a new one starts.
int run_batched_fused(const sdp_work* items, int n, bool adjoint, cudaStream_t st) {
    std::vector<int> idx, off;
    std::vector<std::pair<const sdp_plan_s*, int>> used;   // coils taken per plan in the wave
    for (int i = 0; i < n; ++i) {
        const sdp_plan_s* p = items[i].plan;
        int* u = nullptr;
        for (auto& e : used)
            if (e.first == p) u = &e.second;
        const int have = u ? *u : 0;
        const auto ri = out_range(items[i], adjoint);
        bool overlap = false;
        for (int q : idx) {
            const auto rq = out_range(items[q], adjoint);
            overlap |= ri.first < rq.second && rq.first < ri.second;
        }
        if ((int)idx.size() == kMaxMvItems || have + items[i].B > p->maxB || overlap) {
            SDP_TRY(run_wave(items, idx, off, adjoint, st));
            idx.clear();
            off.clear();
            used.clear();
            u = nullptr;
        }
        if (!u) {
            used.emplace_back(p, 0);
            u = &used.back().second;
        }
        idx.push_back(i);
        off.push_back(*u);
        *u += items[i].B;
    }
    if (!idx.empty()) SDP_TRY(run_wave(items, idx, off, adjoint, st));
    return SDP_OK;
}

std::mutex g_batch_mu;   // batched calls of several host threads enqueue one after the other

int run_batched(const sdp_work* items, int n, bool adjoint, cudaStream_t st) {
    if (n < 0 || (n > 0 && !items)) return SDP_ERR_INVALID_ARG;
    for (int i = 0; i < n; ++i) {
        const sdp_work& w = items[i];
        if (!w.plan) return SDP_ERR_INVALID_ARG;
        SDP_TRY(check_call(w.plan, w.in, w.coil_idx, w.B, 0, w.plan->geo.K, w.out));
    }
    if (n == 0) return SDP_OK;
    const bool eligible = fused_eligible(items, n) && !std::getenv("SDP_BATCH_STREAMS");
    if (eligible && batch_values(items, n) <= kFusedMost) return run_batched_fused(items, n, adjoint, st);
    auto run_one = [&](const sdp_work& w, cudaStream_t s) {
        return adjoint ? adjoint_impl(w.plan, w.in, w.coil_idx, w.B, 0, w.plan->geo.K, w.out, w.accumulate ? 1 : 0,
                                      nullptr, s)
                       : forward_impl(w.plan, w.in, w.coil_idx, w.B, 0, w.plan->geo.K, w.out, 0, s);
    };
    std::vector<sdp_plan_s*> plans;
    for (int i = 0; i < n; ++i)
        if (std::find(plans.begin(), plans.end(), items[i].plan) == plans.end()) plans.push_back(items[i].plan);
    // outputs of different plans that overlap (two adjoints adding into one image) keep item order
    bool ordered = plans.size() == 1;   // one plan: nothing to overlap in time
    for (int i = 0; i < n && !ordered; ++i)
        for (int q = 0; q < i && !ordered; ++q) {
            const auto ri = out_range(items[i], adjoint), rq = out_range(items[q], adjoint);
            ordered = items[i].plan != items[q].plan && ri.first < rq.second && rq.first < ri.second;
        }
    // the plans' streams have the default priority: a batch that could take one launch per stage
    // keeps the priority of the caller's stream
    int priority = 0;
    if (eligible) SDP_CUDA(cudaStreamGetPriority(st, &priority));
    if (ordered || priority != 0) {
        for (int i = 0; i < n; ++i) SDP_TRY(run_one(items[i], st));
        return SDP_OK;
    }
    // Every plan's items on the plan's own stream, forked from and joined back to the caller's.  No
    // stream is shared with the calls of other plans: they neither queue behind this batch nor meet
    // a stream that a capture of it holds.
    std::lock_guard<std::mutex> lk(g_batch_mu);
    const cudaEvent_t fork = plans[0]->forked;
    SDP_CUDA(cudaEventRecord(fork, st));
    for (sdp_plan_s* p : plans) SDP_CUDA(cudaStreamWaitEvent(p->own, fork, 0));
    int rc = SDP_OK;
    for (int i = 0; i < n && rc == SDP_OK; ++i) rc = run_one(items[i], items[i].plan->own);
    // always join the plans' streams back, also after a failed launch
    for (sdp_plan_s* p : plans) {
        if (cudaEventRecord(p->joined, p->own) != cudaSuccess || cudaStreamWaitEvent(st, p->joined, 0) != cudaSuccess) {
            cudaGetLastError();
            rc = rc == SDP_OK ? SDP_ERR_CUDA : rc;
        }
    }
    return rc;
}

}  // namespace

extern "C" {

int sdp_forward_batched(const sdp_work* items, int32_t n, void* stream) {
    return run_batched(items, n, false, static_cast<cudaStream_t>(stream));
}

int sdp_adjoint_batched(const sdp_work* items, int32_t n, void* stream) {
    return run_batched(items, n, true, static_cast<cudaStream_t>(stream));
}

int sdp_plan_create(sdp_plan_t* out, const sdp_plan_desc* d, void* stream) {
    return sdp_plan_create_tuned(out, d, nullptr, stream);
}

int sdp_plan_create_tuned(sdp_plan_t* out, const sdp_plan_desc* d, const sdp_tuning* tn, void* stream) {
    if (!out) return SDP_ERR_INVALID_ARG;
    *out = nullptr;
    if (tn) {
        if (tn->spread_chunk < 32 || tn->spread_chunk > 65536 || tn->fft_engine < 0 || tn->fft_engine > 1 ||
            (tn->fft_lines != 0 && tn->fft_lines != 8 && tn->fft_lines != 4) ||
            (tn->fft_cols != 0 && tn->fft_cols != 32 && tn->fft_cols != 8) ||
            (tn->interp_threads != 0 && tn->interp_threads != 256 && tn->interp_threads != 1024) ||
            tn->spread_coils < 0 || tn->spread_coils > 2 ||
            (tn->interp_run != 0 && tn->interp_run != 1 && tn->interp_run != 2 && tn->interp_run != 4 &&
             tn->interp_run != 8) ||
            tn->interp_coils < 0 || tn->interp_coils > kMaxBatch || tn->fft_staged < 0 || tn->fft_staged > 3 ||
            tn->interp_tiled < 0 || tn->interp_tiled > 1)
            return SDP_ERR_INVALID_ARG;
        const int32_t* sb = tn->spread_bins;
        if (!((sb[0] == 8 || sb[0] == 4) && sb[1] == 4 && (sb[2] == 8 || sb[2] == 4))) return SDP_ERR_UNSUPPORTED;
    }
    if (!d || !d->traj || !d->V || !d->coil_maps || !d->frame_offsets) return SDP_ERR_INVALID_ARG;
    for (int a = 0; a < 3; ++a)
        if (d->n[a] < 2) return SDP_ERR_INVALID_ARG;
    if (!(d->oversamp >= 1.0 && d->oversamp <= 4.0)) return SDP_ERR_INVALID_ARG;
    if (d->width < 2 || d->width > kMaxWidth) return SDP_ERR_UNSUPPORTED;
    if (d->K < 1 || d->K > kMaxK) return SDP_ERR_UNSUPPORTED;
    if (d->T < 1 || d->C < 1 || d->J < 1 || d->J >= (1LL << 31)) return SDP_ERR_INVALID_ARG;
    if (d->max_batch < 1 || d->max_batch > kMaxBatch) return SDP_ERR_INVALID_ARG;
    if (d->flags & ~(uint32_t)SDP_FLAG_BORROW_MAPS) return SDP_ERR_INVALID_ARG;
    if ((d->flags & SDP_FLAG_BORROW_MAPS) && (reinterpret_cast<uintptr_t>(d->coil_maps) % alignof(float2)))
        return SDP_ERR_INVALID_ARG;
    if (d->frame_offsets[0] != 0 || d->frame_offsets[d->T] != d->J) return SDP_ERR_INVALID_ARG;
    for (int t = 0; t < d->T; ++t)
        if (d->frame_offsets[t + 1] < d->frame_offsets[t]) return SDP_ERR_INVALID_ARG;
    // size limits, on the host before any device call: grid lengths up to 2^14, and one coil's
    // channel-interleaved grid and one image indexed with 32-bit offsets
    {
        long long G = 1, nvox = 1;
        for (int a = 0; a < 3; ++a) {
            const long long m = grid_len(d->n[a], d->oversamp, d->width);
            if (m > (1 << 14)) return SDP_ERR_UNSUPPORTED;
            G *= m;
            nvox *= d->n[a];
        }
        if (G * d->K >= (1LL << 31) || nvox >= (1LL << 31)) return SDP_ERR_UNSUPPORTED;
    }
    sdp_plan_s* p = new (std::nothrow) sdp_plan_s();
    if (!p) return SDP_ERR_OOM;
    if (cudaGetDevice(&p->dev) != cudaSuccess) {
        cudaGetLastError();
        delete p;
        return SDP_ERR_CUDA;
    }
    int rc = build_plan(p, d, tn, static_cast<cudaStream_t>(stream));
    if (rc == SDP_OK && (cudaStreamCreateWithFlags(&p->own, cudaStreamNonBlocking) != cudaSuccess ||
                         cudaEventCreateWithFlags(&p->forked, cudaEventDisableTiming) != cudaSuccess ||
                         cudaEventCreateWithFlags(&p->joined, cudaEventDisableTiming) != cudaSuccess)) {
        cudaGetLastError();
        rc = SDP_ERR_CUDA;
    }
    if (rc != SDP_OK) {
        free_plan(p);
        return rc;
    }
    *out = p;
    return SDP_OK;
}

void sdp_plan_destroy(sdp_plan_t p) { free_plan(p); }

int sdp_forward(sdp_plan_t p, const void* x, const int32_t* coil_idx, int32_t B, void* y, void* stream) {
    if (!p) return SDP_ERR_INVALID_ARG;
    return forward_impl(p, x, coil_idx, B, 0, p->geo.K, y, 0, static_cast<cudaStream_t>(stream));
}

int sdp_adjoint(sdp_plan_t p, const void* y, const int32_t* coil_idx, int32_t B, void* out, int32_t accumulate,
                void* stream) {
    if (!p) return SDP_ERR_INVALID_ARG;
    return adjoint_impl(p, y, coil_idx, B, 0, p->geo.K, out, accumulate ? 1 : 0, nullptr,
                        static_cast<cudaStream_t>(stream));
}

int sdp_adjoint_scaled(sdp_plan_t p, const void* y, const int32_t* coil_idx, int32_t B, const float* scale,
                       void* out, int32_t accumulate, void* stream) {
    if (!p || !scale) return SDP_ERR_INVALID_ARG;
    return adjoint_impl(p, y, coil_idx, B, 0, p->geo.K, out, accumulate ? 1 : 0, scale,
                        static_cast<cudaStream_t>(stream));
}

int sdp_residual_loss_weighted(sdp_plan_t p, const void* yhat, const void* y_meas, int32_t n_meas_rows,
                               const int32_t* meas_idx, int32_t B, const float* dcf, void* r2, float* loss,
                               void* stream) {
    if (!p || !yhat || !y_meas || !meas_idx || !r2 || !loss) return SDP_ERR_INVALID_ARG;
    if (B < 1 || B > p->maxB || n_meas_rows < 1) return SDP_ERR_INVALID_ARG;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    return run(p, ST_LOSS, st, [&] {
        return launch_residual_loss(static_cast<const float2*>(yhat), static_cast<const float2*>(y_meas), meas_idx,
                                    dcf, B, (long long)p->geo.J, n_meas_rows, static_cast<float2*>(r2),
                                    p->loss_partials, p->loss_counter, loss, p->status, st);
    });
}

int sdp_tv_value(sdp_plan_t p, const void* x, float eps, float lambda, float* value, void* stream) {
    if (!p || !x || !value || !(eps > 0.f)) return SDP_ERR_INVALID_ARG;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    return run(p, ST_TV, st, [&] {
        return launch_tv_value(p->geo, static_cast<const float2*>(x), eps, lambda, p->tv_part, p->tv_counter, value,
                               st);
    });
}

int sdp_tv_grad(sdp_plan_t p, const void* x, float eps, float lambda, const float* scale, void* out,
                int32_t accumulate, void* stream) {
    if (!p || !x || !out || !(eps > 0.f)) return SDP_ERR_INVALID_ARG;
    if (x == out) return SDP_ERR_INVALID_ARG;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    return run(p, ST_TV, st, [&] {
        return launch_tv_grad(p->geo, static_cast<const float2*>(x), eps, lambda, scale, static_cast<float2*>(out),
                              accumulate ? 1 : 0, st);
    });
}

int sdp_gram_samples(sdp_plan_t p, const void* y, int32_t B, void* out, void* stream) {
    if (!p || !y || !out || B < 1 || B > p->maxB) return SDP_ERR_INVALID_ARG;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const Geo& g = p->geo;
    SDP_TRY(run(p, ST_SPREAD, st, [&] {
        return launch_spread(spread_args(p, static_cast<const float2*>(y), nullptr, 0, g.K, 0), p->grid_map, p->nsub, B,
                             p->spread_coils, st);
    }));
    return run(p, ST_INTERP, st, [&] {
        return plan_interp(p, p->bufA, B, 0, g.K, static_cast<float2*>(out), 0, st);
    });
}

int sdp_residual_loss(sdp_plan_t p, const void* yhat, const void* y_meas, int32_t n_meas_rows,
                      const int32_t* meas_idx, int32_t B, void* r2, float* loss, void* stream) {
    return sdp_residual_loss_weighted(p, yhat, y_meas, n_meas_rows, meas_idx, B, nullptr, r2, loss, stream);
}

int sdp_forward_channels(sdp_plan_t p, const void* x, const int32_t* coil_idx, int32_t B, int32_t k0, int32_t nk,
                         void* y, int32_t accumulate, void* stream) {
    return forward_impl(p, x, coil_idx, B, k0, nk, y, accumulate ? 1 : 0, static_cast<cudaStream_t>(stream));
}

int sdp_adjoint_channels(sdp_plan_t p, const void* y, const int32_t* coil_idx, int32_t B, int32_t k0, int32_t nk,
                         void* out, int32_t accumulate, void* stream) {
    return adjoint_impl(p, y, coil_idx, B, k0, nk, out, accumulate ? 1 : 0, nullptr, static_cast<cudaStream_t>(stream));
}

int sdp_status(sdp_plan_t p, void* stream) {
    if (!p) return SDP_ERR_INVALID_ARG;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (cudaStreamSynchronize(st) != cudaSuccess) {
        cudaGetLastError();
        return SDP_ERR_CUDA;
    }
    int v = 0;
    if (cudaMemcpy(&v, p->status, sizeof(int), cudaMemcpyDeviceToHost) != cudaSuccess ||
        cudaMemset(p->status, 0, sizeof(int)) != cudaSuccess) {
        cudaGetLastError();
        return SDP_ERR_CUDA;
    }
    return v;
}

int sdp_plan_info(sdp_plan_t p, int64_t* out, int32_t cap) {
    if (!p || !out || cap < 0) return SDP_ERR_INVALID_ARG;
    const int64_t v[16] = {p->M[0],        p->M[1],     p->M[2],   p->geo.J,
                           p->geo.K,       p->maxB,     4,         4,
                           p->seg,         p->nunits,   p->nsub,   p->ninc,
                           (int64_t)p->workspace_bytes, (int64_t)p->total_bytes, p->geo.W, p->geo.C};
    for (int i = 0; i < cap && i < 16; ++i) out[i] = v[i];
    return SDP_OK;
}

int sdp_plan_tuning(sdp_plan_t p, sdp_tuning* out) {
    if (!p || !out) return SDP_ERR_INVALID_ARG;
    *out = sdp_tuning{};
    for (int a = 0; a < 3; ++a) out->spread_bins[a] = p->bs[a];
    out->spread_chunk = p->spread_chunk;
    out->fft_engine = p->ax[0].generic;
    out->fft_lines = p->fft_lines;
    out->fft_cols = p->fft_cols;
    out->interp_threads = p->interp_threads;
    out->spread_coils = p->spread_coils;
    out->interp_run = p->interp_run;
    out->interp_coils = p->interp_coils;
    out->fft_staged = p->ax[2].staged;
    // (more than 8 channels: the row kernel for a call on all of them, whatever this says)
    out->interp_tiled = p->interp_tiled == kTiledByRule
                            ? (p->geo.K > 8 || interp_tiles_faster(p->geo.W, p->geo.K, p->maxB, p->M[0] * p->M[1] * p->M[2]) ? 1 : 0)
                            : p->interp_tiled;
    return SDP_OK;
}

double sdp_plan_beta(sdp_plan_t p) { return p ? p->beta : -1.0; }

size_t sdp_workspace_bytes(sdp_plan_t p) { return p ? p->workspace_bytes : 0; }

size_t sdp_workspace_bytes_for(sdp_plan_t p, int32_t maxB) {
    if (!p || maxB < 1 || maxB > kMaxBatch) return 0;
    const long long G = p->M[0] * p->M[1] * p->M[2];
    const size_t gridA = (size_t)std::max<long long>(G, p->n[0] * p->n[1] * p->M[2]);
    const size_t gridB = (size_t)(p->n[0] * p->M[1] * p->M[2]);
    return (gridA + gridB) * (size_t)p->geo.K * (size_t)maxB * sizeof(float2);
}

int sdp_plan_set_wait_test(sdp_plan_t p, int32_t withhold_row, int64_t timeout_ns) {
    if (!p) return SDP_ERR_INVALID_ARG;
    const int W = p->geo.W;
    const int rows = imap::tile_points(W, 0) * imap::tile_points(W, 1);
    if (withhold_row < -1 || withhold_row >= rows) return SDP_ERR_INVALID_ARG;
    if (timeout_ns != 0 && (timeout_ns < 1000 || timeout_ns > 10000000000LL)) return SDP_ERR_INVALID_ARG;
    p->wait_test_row = withhold_row;
    p->wait_test_ns = timeout_ns;
    return SDP_OK;
}

int64_t sdp_launch_count(void) { return g_launches.load(); }

int sdp_profile_enable(sdp_plan_t p, int32_t enable) {
    if (!p) return SDP_ERR_INVALID_ARG;
    p->prof = enable != 0;
    return SDP_OK;
}

int sdp_profile_read(sdp_plan_t p, double* ms, int64_t* launches, int32_t cap) {
    if (!p) return -SDP_ERR_INVALID_ARG;
    for (auto& r : p->prof_used) {
        if (cudaEventSynchronize(r.b) != cudaSuccess) {
            cudaGetLastError();
            return -SDP_ERR_CUDA;
        }
        float t = 0.f;
        if (cudaEventElapsedTime(&t, r.a, r.b) != cudaSuccess) {
            cudaGetLastError();
            return -SDP_ERR_CUDA;
        }
        p->prof_ms[r.stage] += t;
        p->prof_n[r.stage] += 1;
        p->prof_free.push_back(r);
    }
    p->prof_used.clear();
    const int n = cap < kNumStages ? cap : kNumStages;
    for (int s = 0; s < n; ++s) {
        if (ms) ms[s] = p->prof_ms[s];
        if (launches) launches[s] = p->prof_n[s];
        p->prof_ms[s] = 0;
        p->prof_n[s] = 0;
    }
    return n;
}

int64_t sdp_grid_size(int64_t n, double oversamp, int32_t width) {
    if (n < 1 || width < 2 || width > kMaxWidth || !(oversamp >= 1.0 && oversamp <= 4.0)) return -1;
    return grid_len(n, oversamp, width);
}

double sdp_kb_beta(int32_t width, double oversamp) {
    const double arg = (width / oversamp) * (width / oversamp) * (oversamp - 0.5) * (oversamp - 0.5) - 0.8;
    return arg > 0 ? kPi * std::sqrt(arg) : -1.0;
}

const char* sdp_strerror(int s) {
    switch (s) {
        case SDP_OK: return "ok";
        case SDP_ERR_INVALID_ARG: return "invalid argument";
        case SDP_ERR_OOM: return "device out of memory";
        case SDP_ERR_CUDA: return "CUDA runtime error";
        case SDP_ERR_TIMEOUT: return "bounded device wait timed out";
        case SDP_ERR_BOUNDS: return "device-side index out of range (coil index)";
        case SDP_ERR_UNSUPPORTED: return "unsupported parameters";
        default: return "unknown status";
    }
}

}  // extern "C"
