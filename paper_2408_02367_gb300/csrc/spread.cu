// Adjoint spreading: the dispatch over kernel widths and widths 2 and 3.  The
// kernel itself is in spread_impl.cuh; the other widths are instantiated in
// translation units of their own (spread_w45.cu, spread_w67.cu, spread_w8.cu).
#include "spread_impl.cuh"

namespace sdp {

cudaError_t launch_spread_w45(const SpreadArgs& a, const CUtensorMap& map, int nsub, int B, int coils,
                              cudaStream_t st);
cudaError_t launch_spread_w67(const SpreadArgs& a, const CUtensorMap& map, int nsub, int B, int coils,
                              cudaStream_t st);
cudaError_t launch_spread_w8(const SpreadArgs& a, const CUtensorMap& map, int nsub, int B, int coils,
                             cudaStream_t st);

int grid_tensor_map(CUtensorMap* map, void* base, int K, const int64_t M[3], int coils, int b1, int b2, int b3) {
    // the encoder comes from the driver the runtime has loaded: nothing to link against
    void* fn = nullptr;
    cudaDriverEntryPointQueryResult found;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &found) != cudaSuccess ||
        found != cudaDriverEntryPointSuccess || !fn) {
        cudaGetLastError();
        return SDP_ERR_CUDA;
    }
    using Encode = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
    const cuuint64_t row = (cuuint64_t)M[2] * K;   // 8-byte values; M[2] is even, so every stride is a multiple of 16 bytes
    const cuuint64_t dims[4] = {row, (cuuint64_t)M[1], (cuuint64_t)M[0], (cuuint64_t)coils};
    const cuuint64_t strides[3] = {row * 8, row * 8 * M[1], row * 8 * M[1] * M[0]};
    const cuuint32_t box[4] = {(cuuint32_t)(b3 * K), (cuuint32_t)b2, (cuuint32_t)b1, 1}, step[4] = {1, 1, 1, 1};
    const CUresult rc = reinterpret_cast<Encode>(fn)(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT64, 4, base, dims, strides, box,
                                                     step, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                                                     CU_TENSOR_MAP_L2_PROMOTION_NONE,
                                                     CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return rc == CUDA_SUCCESS ? SDP_OK : SDP_ERR_CUDA;
}

cudaError_t launch_spread(const SpreadArgs& a, const CUtensorMap& map, int nsub, int B, int coils,
                          cudaStream_t st) {
    switch (a.g.W) {
        case 2: return launch_spread_width<2>(a, map, nsub, B, coils, st);
        case 3: return launch_spread_width<3>(a, map, nsub, B, coils, st);
        case 4:
        case 5: return launch_spread_w45(a, map, nsub, B, coils, st);
        case 6:
        case 7: return launch_spread_w67(a, map, nsub, B, coils, st);
        case 8: return launch_spread_w8(a, map, nsub, B, coils, st);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace sdp
