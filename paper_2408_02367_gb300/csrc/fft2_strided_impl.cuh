// The strided two-pass register FFT kernel over one plan (axis 1 or 2 of steps A2 / A6; the
// body is in fft2_impl.cuh) and its launch, instantiated per direction in fft2_fwd.cu and
// fft2_inv.cu.
#pragma once

#include "fft2_impl.cuh"
#include "tma.cuh"

namespace sdp {
namespace {

// Resident CTAs the registers are bounded for: 48 warps per SM with 32 columns and a factor of 15
// or more (at 44 registers instead of 40 the 512-thread CTAs of length 160 fit twice instead of
// three times, and axis 1 at 128^3 takes 129 us instead of 111); the other shapes are left to the
// compiler (bounded the same way, length 120 takes 5% more, length 250 with a bound of one CTA 60%).
template <int A, int B, int NLT>
constexpr int strided_ctas() {
    constexpr int f = A > B ? A : B;
    return NLT == 32 && f >= 15 ? 48 / f : 0;
}

template <int A, int B, int NLT, bool INV>
__global__ void __launch_bounds__(NLT*(A > B ? A : B), (strided_ctas<A, B, NLT>())) fft2_strided_kernel(const float2* __restrict__ in,
                                                                         float2* __restrict__ out,
                                                                         const float2* __restrict__ twg, int n_in,
                                                                         int in_centred, int n_out, int out_centred,
                                                                         long long inner, long long ncolblk) {
    __shared__ float2 tw[A * B];
    __shared__ float2 Y[A * B * NLT];
    fft2_strided_body<A, B, NLT, INV>(tw, Y, in, out, twg, n_in, in_centred, n_out, out_centred, inner, ncolblk,
                                      (long long)blockIdx.x);
}

// The same pass with its input fetched by tensor loads: persistent CTAs walk the (column block,
// outer line) units; a unit's rows land in shared memory at their FFT positions (two boxes: for a
// centred input the rows from n_in / 2 on at position 0, those before at the end, the zeros
// between written once; else two halves), and the next unit's boxes are on their way while the
// second half of this one's transform runs.  No register holds a load in flight and no address
// or row test is computed per element on the way in.  The arithmetic per line is
// fft2_strided_body's.
//
// What bounds the direct kernel at the long lengths is latency: at 250 two 400-thread CTAs fit an
// SM.  Columns per CTA: 16 (row segments of 128 bytes).
template <int A, int B>
struct TmaPass {
    static constexpr int L = A * B, NC = kTmaCols, threads = NC * (A > B ? A : B);
    static constexpr int smem = (2 * L * NC + L) * 8 + 16;   // X, Y, twiddles, the mbarrier
    // resident CTAs the registers are bounded for: 40 warps up to a factor of 16, then 32, 25 at 25,
    // and no more than the shared memory holds (from length 180 on that is fewer, but for 200, 216 and
    // 250: bounded for five CTAs of which three fit, length 240 spilled, and its four passes over
    // 192^2 x 80 images, 2 coils, 5 channels, took 540 us against 470)
    static constexpr int f = A > B ? A : B, most = f <= 16 ? 80 / f : (f <= 20 ? 64 / f : 2);
    static constexpr int fit = 227 * 1024 / (smem + 1024), ctas = most < fit ? most : fit;
};

template <int A, int B, bool INV>
__global__ void __launch_bounds__(TmaPass<A, B>::threads, TmaPass<A, B>::ctas) fft2_strided_tma_kernel(
    const __grid_constant__ StridedMaps maps, float2* __restrict__ out, const float2* __restrict__ twg, int n_out,
    int out_centred, long long inner, int ncolblk, int nunits, int* status) {
    using P = TmaPass<A, B>;
    constexpr int L = P::L, NC = P::NC;
    extern __shared__ __align__(128) unsigned char smem[];
    float2* X = reinterpret_cast<float2*>(smem);
    float2* Y = X + L * NC;
    float2* tw = Y + L * NC;
    uint64_t* bar = reinterpret_cast<uint64_t*>(tw + L);
    const int tid = threadIdx.x;
    for (int i = tid; i < L; i += P::threads) tw[i] = twg[i];
    for (int i = maps.rows[0] * NC + tid; i < maps.dst1 * NC; i += P::threads) X[i] = make_float2(0.f, 0.f);
    if (tid == 0) {
        tma::mbar_init(bar, 1);
        tma::fence_init();
    }
    __syncthreads();
    auto issue = [&](int u) {   // thread 0
        const int o = u / ncolblk, c0 = (u - o * ncolblk) * NC;
        tma::mbar_expect_tx(bar, (uint32_t)((maps.rows[0] + maps.rows[1]) * NC * 8));
        tma::tensor_load_3d(&maps.map[0], X, c0, maps.src0, o, bar);
        tma::tensor_load_3d(&maps.map[1], X + maps.dst1 * NC, c0, maps.src1, o, bar);
    };
    if (tid == 0 && (int)blockIdx.x < nunits) issue(blockIdx.x);
    uint32_t phase = 0;
    const int c1 = tid % NC, f1 = tid / NC;   // column, and pass 1's b or pass 2's q1
    const int h = out_centred ? n_out / 2 : 0;
    for (int u = blockIdx.x; u < nunits; u += gridDim.x) {
        const bool ok = tma::mbar_wait(bar, phase, status);
        if (!__syncthreads_and(ok)) {
            // the boxes did not land within the limit: one more bounded wait, leave
            tma::mbar_wait(bar, phase, nullptr);
            return;
        }
        phase ^= 1u;
        if (tid < NC * B) {
            float2 x[A];
            StaticFor<0, A>::run([&](auto ac) {
                constexpr int a = decltype(ac)::value;
                x[a] = X[(B * a + f1) * NC + c1];
            });
            RegDft<A, INV>::run(x);
            StaticFor<0, A>::run([&](auto qc) {
                constexpr int q1 = decltype(qc)::value;
                Y[(q1 * B + f1) * NC + c1] = q1 == 0 ? x[q1] : cmul(x[q1], twiddle(tw, f1 * q1, INV));
            });
        }
        __syncthreads();
        if (tid == 0 && u + (int)gridDim.x < nunits) issue(u + gridDim.x);   // X has been read
        if (tid < NC * A) {
            float2 z[B];
            StaticFor<0, B>::run([&](auto bc) {
                constexpr int b = decltype(bc)::value;
                z[b] = Y[(f1 * B + b) * NC + c1];
            });
            RegDft<B, INV>::run(z);
            const int o = u / ncolblk, c0 = (u - o * ncolblk) * NC;
            float2* dst = out + (long long)o * n_out * inner + c0 + c1;
            const bool in = c0 + c1 < inner;
            StaticFor<0, B>::run([&](auto qc) {
                constexpr int q2 = decltype(qc)::value;
                int row = f1 + A * q2 + h;   // output row whose FFT index is q1 + A q2
                if (row >= L) row -= L;
                if (row < n_out && in) dst[(long long)row * inner] = z[q2];
            });
        }
        __syncthreads();   // Y is free
    }
}

// Launches the tensor-load kernel; cudaErrorNotSupported where it does not apply (no maps for the
// call, a length with none) or does not pay (fewer than two units per resident CTA).
template <bool INV>
cudaError_t launch_strided_tma(const FftAxis& ax, const StridedMaps& maps, float2* out, int n_out, int out_centred,
                               long long inner, long long outer, int* status, cudaStream_t st) {
    cudaError_t err = cudaErrorNotSupported;
    with_strided_shape(ax.L, [&](auto sh) {
        using S = decltype(sh);
        using P = TmaPass<S::a, S::b>;
        static ResidentCtas resident;
        auto kern = fft2_strided_tma_kernel<S::a, S::b, INV>;
        long long grid = 0;
        const cudaError_t e = resident.get(kern, P::smem, P::threads, grid);
        if (e != cudaSuccess) {
            cudaGetLastError();   // the direct kernel takes the call
            return;
        }
        const long long ncolblk = (inner + P::NC - 1) / P::NC, nunits = ncolblk * outer;
        if (nunits < 2 * grid || nunits > 0x3fffffffLL) return;
        kern<<<(unsigned)grid, P::threads, P::smem, st>>>(maps, out, ax.tw, n_out, out_centred, inner, (int)ncolblk,
                                                          (int)nunits, status);
        err = cudaGetLastError();
    });
    return err;
}

template <bool INV>
cudaError_t launch_strided(const FftAxis& ax, const float2* in, float2* out, int n_in, int in_centred, int n_out,
                           int out_centred, long long inner, long long outer, cudaStream_t st) {
    cudaError_t err = cudaErrorNotSupported;
    with_strided_shape(ax.L, [&](auto sh) {
        using S = decltype(sh);
        const long long ncolblk = (inner + S::nl - 1) / S::nl;
        const long long nblk = ncolblk * outer;
        if (nblk <= 0) {
            err = cudaSuccess;
            return;
        }
        if (nblk > 0x7fffffffLL) {
            err = cudaErrorInvalidConfiguration;
            return;
        }
        fft2_strided_kernel<S::a, S::b, S::nl, INV><<<(unsigned)nblk, S::threads, 0, st>>>(
            in, out, ax.tw, n_in, in_centred, n_out, out_centred, inner, ncolblk);
        err = cudaGetLastError();
    });
    return err;
}

}  // namespace
}  // namespace sdp
