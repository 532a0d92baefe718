// Adjoint spreading, widths 6 and 7 (the kernel is in spread_impl.cuh).
#include "spread_impl.cuh"

namespace sdp {

cudaError_t launch_spread_w67(const SpreadArgs& a, const CUtensorMap& map, int nsub, int B, int coils,
                              cudaStream_t st) {
    return a.g.W == 6 ? launch_spread_width<6>(a, map, nsub, B, coils, st) : launch_spread_width<7>(a, map, nsub, B, coils, st);
}

}  // namespace sdp
