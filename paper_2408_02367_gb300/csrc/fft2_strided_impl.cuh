// The strided two-pass register FFT kernel over one plan (axis 1 or 2 of steps A2 / A6; the
// body is in fft2_impl.cuh) and its launch, instantiated per direction in fft2_fwd.cu and
// fft2_inv.cu.
#pragma once

#include "fft2_impl.cuh"

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
