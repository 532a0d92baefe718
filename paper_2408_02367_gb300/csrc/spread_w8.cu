// Adjoint spreading, width 8 (the kernel is in spread_impl.cuh).
#include "spread_impl.cuh"

namespace sdp {

cudaError_t launch_spread_w8(const SpreadArgs& a, const CUtensorMap& map, int nsub, int B, int coils,
                             cudaStream_t st) {
    return launch_spread_width<8>(a, map, nsub, B, coils, st);
}

}  // namespace sdp
