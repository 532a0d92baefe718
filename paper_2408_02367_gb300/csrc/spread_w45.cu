// Adjoint spreading, widths 4 and 5 (the kernel is in spread_impl.cuh).
#include "spread_impl.cuh"

namespace sdp {

cudaError_t launch_spread_w45(const SpreadArgs& a, const CUtensorMap& map, int nsub, int B, int coils,
                              cudaStream_t st) {
    return a.g.W == 4 ? launch_spread_width<4>(a, map, nsub, B, coils, st) : launch_spread_width<5>(a, map, nsub, B, coils, st);
}

}  // namespace sdp
