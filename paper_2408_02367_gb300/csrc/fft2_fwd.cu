// Strided two-pass FFT passes, forward (fft2_strided_impl.cuh).
#include "fft2_strided_impl.cuh"

namespace sdp {

cudaError_t launch_fft2_strided_fwd(const FftAxis& ax, const float2* in, float2* out, int n_in, int in_centred,
                                    int n_out, int out_centred, long long inner, long long outer,
                                    const StridedMaps* maps,
                                    int* status, cudaStream_t st) {
    if (maps) {
        const cudaError_t e =
            launch_strided_tma<false>(ax, *maps, out, n_out, out_centred, inner, outer, status, st);
        if (e != cudaErrorNotSupported) return e;
    }
    return launch_strided<false>(ax, in, out, n_in, in_centred, n_out, out_centred, inner, outer, st);
}

}  // namespace sdp
