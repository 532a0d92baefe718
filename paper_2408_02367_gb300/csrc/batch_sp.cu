// Spread of several plans in one launch (the batched adjoint's first stage; see
// batch.cu for the layout of a batched launch).  One warp per (subproblem, coil
// pair or coil) of every item, running the single-plan spread's body
// (spread_impl.cuh) on that item's plan.  Kernel widths 4 and 6, one channel
// group (K <= 32 / W).
#include "batch.cuh"
#include "spread_impl.cuh"

namespace sdp {
namespace {

__device__ __forceinline__ int find_item(const MvUnits& u, long long unit) {
    int i = 0;
    while (i + 1 < u.n && unit >= u.start[i + 1]) ++i;
    return i;
}

// u.start holds the prefix sums of nsub * (coil groups) per item.
template <int W, int NK>
__global__ void __launch_bounds__(32, (spread_warps<W, NK, 2>())) mv_spread_kernel(const __grid_constant__ MvArgs a, const MvUnits u) {
    __shared__ __align__(128) float4 rec[SpreadDims<W, NK, 2>::kAll];   // the larger of the two
    static_assert(SpreadDims<W, NK, 2>::kAll >= SpreadDims<W, NK, 1>::kAll, "shared memory of one coil");
    const long long unit = blockIdx.x;
    const int i = find_item(u, unit);
    const MvItem& it = a.it[i];
    const long long local = unit - u.start[i];
    const int sub = (int)(local % it.nsub);
    const int by = (int)(local / it.nsub);
    if (it.spread_pairs)
        spread_body<W, NK, 2>(it.sa, 0, it.B, sub, by, rec, &it.grid_map);
    else
        spread_body<W, NK, 1>(it.sa, 0, it.B, sub, by, rec, &it.grid_map);
}

// One channel group of at most 32 / W channels (the batched path's eligibility).
template <int W, int NK>
cudaError_t launch_mv_spread_k(const MvArgs& a, const MvUnits& u, cudaStream_t st) {
    if constexpr (NK <= 32 / W) {
        mv_spread_kernel<W, NK><<<(unsigned)u.start[u.n], 32, 0, st>>>(a, u);
        return cudaGetLastError();
    } else {
        return cudaErrorInvalidValue;
    }
}

template <int W>
cudaError_t launch_mv_spread_w(const MvArgs& a, const MvUnits& u, int K, cudaStream_t st) {
    switch (K) {
        case 1: return launch_mv_spread_k<W, 1>(a, u, st);
        case 2: return launch_mv_spread_k<W, 2>(a, u, st);
        case 3: return launch_mv_spread_k<W, 3>(a, u, st);
        case 4: return launch_mv_spread_k<W, 4>(a, u, st);
        case 5: return launch_mv_spread_k<W, 5>(a, u, st);
        case 6: return launch_mv_spread_k<W, 6>(a, u, st);
        case 7: return launch_mv_spread_k<W, 7>(a, u, st);
        case 8: return launch_mv_spread_k<W, 8>(a, u, st);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace

cudaError_t launch_mv_spread(const MvArgs& a, const MvUnits& u, int W, int K, cudaStream_t st) {
    if (u.start[u.n] == 0) return cudaSuccess;
    if (u.start[u.n] > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
    switch (W) {
        case 4: return launch_mv_spread_w<4>(a, u, K, st);
        case 6: return launch_mv_spread_w<6>(a, u, K, st);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace sdp
