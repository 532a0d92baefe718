// Internal definitions shared by the kernels and the C ABI of the subspace
// multicoil NUFFT operator.  Not part of the public interface.
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <vector>

#include "../../include/stodip_op.h"

namespace sdp {

constexpr int kMaxRadixStages = 12;
constexpr int kMaxWidth = 8;
constexpr int kMaxK = 16;
constexpr int kMaxBatch = 64;
constexpr int kNumStages = 10;  // profiling stages, see stodip_op.h

enum Stage {
    ST_FWD_FFT3 = 0,
    ST_FWD_FFT2 = 1,
    ST_FWD_FFT1 = 2,
    ST_INTERP = 3,
    ST_SPREAD = 4,
    ST_ADJ_FFT1 = 5,
    ST_ADJ_FFT2 = 6,
    ST_ADJ_FFT3 = 7,
    ST_LOSS = 8,
    ST_TV = 9,
};

// One axis of the 3D FFT: length L = prod(radix[0..nst)), twiddles
// tw[m] = exp(-2 pi i m / L) in float32 (computed in float64 on the host).
struct FftAxis {
    int L;
    int nst;
    int radix[kMaxRadixStages];
    const float2* tw;
    int generic;   // 1: always the Stockham kernels (a plan's tuning), 0: two-pass where available
    int staged;    // fused axis-3 kernels staged by bulk copies where supported: bit 0 prologue, bit 1 epilogue
};

// A spread subproblem: one chunk of the incidence list of one output unit (4 x 4 columns by
// `seg` points along axis 3; unit index ((c1 * nb2) + c2) * nb3 + segment).
struct SubProb {
    int bin;       // flattened unit index
    int start;     // first incidence
    int count;     // incidences in this chunk
    int chunk;     // chunk number within the unit
    int nchunks;   // chunks of this unit (1 = write the grid directly)
    int slot;      // partial slot of chunk 0 of this unit (multi-chunk units)
    int r0, r1;    // planes of this chunk (multi-chunk units: together they cover every plane of the unit)
    int multi;     // number of this multi-chunk unit (its row of SpreadArgs::ranges)
};

// Shared view of a plan passed to the kernel launchers.
struct Geo {
    int N[3];
    int M[3];
    int W;
    int K;
    int T;
    int C;
    int J;
    float beta;
    float inv_i0_beta;
    float halfW;
};

// Arguments of the spread kernels (spread_impl.cuh) for one plan and call.
struct SpreadArgs {
    Geo g;
    int seg;             // grid points of a unit along axis 3 (a multiple of 4)
    int nb1, nb2, nb3;   // units per axis
    const SubProb* subs;
    const int4* inc;     // incidences: sorted sample, window_at k of axes 1 and 2 and plane (8, 8, 16 bits), index in y, frame
    const float* wts;
    const float2* V;     // [T][vstride]
    int vstride;
    const float2* y;
    const float* scale;
    int k0, nk;
    float2* grids;
    float2* partials;
    long long slots_per_b;
    long long slot_elems;
    const int2* ranges;  // [multi-chunk unit][nblk]: chunks [x, y) whose windows reach the block
    int* counters;       // [coil][group][unit][nblk]
    int* group_counters; // [coil][group][slot][nblk]
    int nbins;           // units
    int nblk;            // blocks of four positions per unit
    int coil0;     // coil of `grids` in the plan's grid workspace
    int use_map;   // 1: the call's grids have the layout of the plan's tensor map
    int ngroups;   // channel groups of this call (counters are per group)
    int group;
};

// Tensor maps of a strided FFT pass's input [outer][n_in][inner] (fft2_strided_impl.cuh): two boxes
// of rows[i] rows by kTmaCols columns, from row src0 to FFT position 0 and from src1 to dst1.
constexpr int kTmaCols = 16;
struct StridedMaps {
    CUtensorMap map[2];
    int rows[2];
    int src0, src1, dst1;
};
int strided_tensor_maps(StridedMaps* m, void* base, int L, int n_in, int in_centred, long long inner, long long outer);

// The NK values of a row of V from an even (`aligned`: 16-byte loads) or odd channel on.
#if defined(__CUDACC__)
template <int NK>
__device__ __forceinline__ void load_v_row(const float2* __restrict__ row, bool aligned, float2 (&v)[NK]) {
    if (NK > 1 && aligned) {
#pragma unroll
        for (int k = 0; k + 1 < NK; k += 2) {
            const float4 q = __ldg(reinterpret_cast<const float4*>(row + k));
            v[k] = make_float2(q.x, q.y);
            v[k + 1] = make_float2(q.z, q.w);
        }
        if (NK % 2) v[NK - 1] = __ldg(row + NK - 1);
    } else {
#pragma unroll
        for (int k = 0; k < NK; ++k) v[k] = __ldg(row + k);
    }
}
#endif

// Launch helpers (each returns cudaError_t of the launch).  `pr` may be null.
cudaError_t launch_fwd_prologue_fft3(const Geo& g, const FftAxis& ax, const float2* x, const float2* S,
                                     const int* coil_idx, int B, int k0, int nk, const float* dinv1,
                                     const float* dinv2, const float* dinv3, float2* out, int* status,
                                     cudaStream_t st);
cudaError_t launch_fft_strided(const FftAxis& ax, int inverse, const float2* in, float2* out, int n_in,
                               int in_centred, int n_out, int out_centred, long long inner, long long outer,
                               const StridedMaps* maps, int* status, cudaStream_t st);
cudaError_t launch_adj_fft3_epilogue(const Geo& g, const FftAxis& ax, const float2* in, const float2* S,
                                     const int* coil_idx, int B, int k0, int nk, const float* dinv1,
                                     const float* dinv2, const float* dinv3, float2* out, int accumulate,
                                     int* status, cudaStream_t st);
// Kaiser-Bessel weights of every (sorted) sample: wts[s][d][a] = phi(g_d - (m0_d + a)),
// m0_d = ceil(g_d - W/2) in float32; computed once per plan.
cudaError_t launch_kb_weights(const Geo& g, const float4* pts, float* wts, cudaStream_t st);
// Tiled interpolation (interp_tiles.cu): samples ordered by tiles of imap::tile_edge() grid
// points per axis; `tiles` lists work items (flattened tile index over nt1 x nt2 x nt3, first sample,
// count, 0), a dense tile's samples split over several items; `srec` holds each sorted
// sample's index in y, its frame and its window's start in the tile, imap::tile_start().
bool interp_tiles_supported(int W, int nk);
bool interp_tiles_faster(int W, int nk, int max_batch, long long points);   // than the row kernel: the choice of a plan without a tuning
struct InterpTiles {
    Geo g;
    const int4* tiles;
    int ntiles, nt2, nt3;
    const int4* srec;
    const float* wts;
    const float2* V;   // [T][vstride]
    int vstride;
    const float2* grids;
    int B, k0;
    float2* y;
    int accumulate;
    int* status;
    int coil0;       // coil of `grids` in the plan's grid workspace
    int use_map;     // 1: the grids have the layout of the plan's tensor map (all channels)
};
cudaError_t launch_interp_tiles(const InterpTiles& a, const CUtensorMap& map, int nk, int withhold_row, long long wait_ns, cudaStream_t st);
// wstart: first tap of every sorted sample per axis, in [0, M), and its index in y.
cudaError_t launch_interp(const Geo& g, int threads, int run, int cblock, const int4* wstart, const int* tframe,
                          const float* wts,
                          const float2* V, const float2* grids, int B, int k0, int nk, float2* y, int accumulate,
                          cudaStream_t st);
// Tensor map of the plan's grid workspace, [coil][M1][M2][M3 K] complex values, with boxes of
// b1 x b2 columns by b3 points (even) of all K <= 8 channels.
int grid_tensor_map(CUtensorMap* map, void* base, int K, const int64_t M[3], int coils, int b1, int b2, int b3);
// Adjoint spread of a.nk channels and B coils over the plan's nsub subproblems; `a` without
// its channel group fields, which the launcher fills.  coils: 1 = one coil per warp, else
// two where they fit.
cudaError_t launch_spread(const SpreadArgs& a, const CUtensorMap& map, int nsub, int B, int coils, cudaStream_t st);
long long residual_loss_partials(int maxB, long long J);
cudaError_t launch_residual_loss(const float2* yhat, const float2* ymeas, const int* meas_idx, const float* dcf, int B,
                                 long long J, int nrows, float2* r2, double* partials, unsigned int* counter,
                                 float* loss, int* status, cudaStream_t st);

// Two-pass register FFT kernels (fft2.cu) for the specialised lengths; they
// return cudaErrorNotSupported for any other length (the Stockham kernels of
// fft.cu then run instead).
bool fft2_supported(int L);
cudaError_t launch_fft2_strided(const FftAxis& ax, int inverse, const float2* in, float2* out, int n_in,
                                int in_centred, int n_out, int out_centred, long long inner, long long outer,
                                const StridedMaps* maps, int* status, cudaStream_t st);
cudaError_t launch_fft2_fwd_prologue(const Geo& g, const FftAxis& ax, const float2* x, const float2* S,
                                     const int* coil_idx, int B, int k0, int nk, const float* dinv1,
                                     const float* dinv2, const float* dinv3, float2* out, int* status,
                                     cudaStream_t st);
// Adjoint axis-3 FFT + epilogue with bulk-copy staged inputs (fft2_staged.cu).
bool fft2_epilogue_staged_ok(const Geo& g, const FftAxis& ax, const float2* in, const float2* S, int nk);
cudaError_t launch_fft2_epilogue_staged(const Geo& g, const FftAxis& ax, const float2* in, const float2* S,
                                        const int* coil_idx, int B, int k0, int nk, const float* dinv1,
                                        const float* dinv2, const float* dinv3, float2* out, int accumulate,
                                        int* status, cudaStream_t st);
// The axis-3 kernels that a plan without a tuning stages, as FftAxis::staged (fft2_staged.cu).
int fft2_staged_default(int N3, int L, int K);
// Forward prologue + axis-3 FFT with bulk-copy staged inputs (fft2_staged.cu).
bool fft2_prologue_staged_ok(const Geo& g, const FftAxis& ax, const float2* x, const float2* S, int nk);
cudaError_t launch_fft2_prologue_staged(const Geo& g, const FftAxis& ax, const float2* x, const float2* S,
                                        const int* coil_idx, int B, int k0, int nk, const float* dinv1,
                                        const float* dinv2, const float* dinv3, float2* out, int* status,
                                        cudaStream_t st);
cudaError_t launch_fft2_adj_epilogue(const Geo& g, const FftAxis& ax, const float2* in, const float2* S,
                                     const int* coil_idx, int B, int k0, int nk, const float* dinv1,
                                     const float* dinv2, const float* dinv3, float2* out, int accumulate,
                                     int* status, cudaStream_t st);

// Total variation of the image (tv.cu).
long long tv_partials(int K, int N1, int N2, int N3);

// Count kernel launches made outside the plan's run() wrapper (sdp_launch_count).
void note_launches(long long n);
cudaError_t launch_tv_value(const Geo& g, const float2* x, float eps, float lambda, double* partials,
                            unsigned int* counter, float* out, cudaStream_t st);
cudaError_t launch_tv_grad(const Geo& g, const float2* x, float eps, float lambda, const float* scale, float2* out,
                           int accumulate, cudaStream_t st);

// Host helpers.
bool fft_factor(int L, FftAxis* ax);
std::vector<float2> fft_twiddles(int L);

}  // namespace sdp
