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
