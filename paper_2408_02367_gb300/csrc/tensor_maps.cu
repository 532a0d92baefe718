// Tensor maps (cuTensorMapEncodeTiled) of the plan's grid workspaces, made on the host when a plan
// is created: the boxes of the spread's stores, of the interpolation's tiles and of the strided
// FFT passes' inputs.  All hold complex64 values as 8-byte elements.
#include <algorithm>

#include "sdp_internal.cuh"

namespace sdp {
namespace {

int encode(CUtensorMap* map, void* base, int rank, const cuuint64_t* dims, const cuuint64_t* strides,
           const cuuint32_t* box) {
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
    const cuuint32_t step[4] = {1, 1, 1, 1};
    const CUresult rc = reinterpret_cast<Encode>(fn)(
        map, CU_TENSOR_MAP_DATA_TYPE_FLOAT64, (cuuint32_t)rank, base, dims, strides, box, step,
        CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_NONE,
        CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return rc == CUDA_SUCCESS ? SDP_OK : SDP_ERR_CUDA;
}

}  // namespace

int grid_tensor_map(CUtensorMap* map, void* base, int K, const int64_t M[3], int coils, int b1, int b2, int b3) {
    const cuuint64_t row = (cuuint64_t)M[2] * K;   // M[2] is even, so every stride is a multiple of 16 bytes
    const cuuint64_t dims[4] = {row, (cuuint64_t)M[1], (cuuint64_t)M[0], (cuuint64_t)coils};
    const cuuint64_t strides[3] = {row * 8, row * 8 * M[1], row * 8 * M[1] * M[0]};
    const cuuint32_t box[4] = {(cuuint32_t)(b3 * K), (cuuint32_t)b2, (cuuint32_t)b1, 1};
    return encode(map, base, 4, dims, strides, box);
}

int strided_tensor_maps(StridedMaps* m, void* base, int L, int n_in, int in_centred, long long inner, long long outer) {
    // rows to FFT positions: centred, rows from n_in / 2 on at 0 and those before at the end;
    // else the two halves in order (L is even)
    const int h = n_in / 2;
    m->rows[0] = in_centred ? n_in - h : h;
    m->rows[1] = in_centred ? h : n_in - h;
    m->src0 = in_centred ? h : 0;
    m->src1 = in_centred ? 0 : h;
    m->dst1 = in_centred ? L - h : h;
    const cuuint64_t dims[3] = {(cuuint64_t)inner, (cuuint64_t)n_in, (cuuint64_t)outer};
    const cuuint64_t strides[2] = {(cuuint64_t)inner * 8, (cuuint64_t)inner * 8 * n_in};
    for (int i = 0; i < 2; ++i) {
        const cuuint32_t box[3] = {kTmaCols, (cuuint32_t)m->rows[i], 1};
        const int rc = encode(&m->map[i], base, 3, dims, strides, box);
        if (rc != SDP_OK) return rc;
    }
    return SDP_OK;
}

}  // namespace sdp
