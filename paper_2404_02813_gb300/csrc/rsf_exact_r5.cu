// rsf_exact_r5.cu -- the exact arithmetic at radii 5 to 8 (see rsf_exact.cuh).
#include "rsf_exact.cuh"

namespace rsf {
namespace tiled {
cudaError_t prepare_exact_r5(int R) {
    switch (R) {
        case 5: return prepare_exact_r<5>();
        case 6: return prepare_exact_r<6>();
        case 7: return prepare_exact_r<7>();
        case 8: return prepare_exact_r<8>();
        default: return cudaErrorInvalidValue;
    }
}
cudaError_t launch_exact_r5(const TiledGroup &g, int parity, Profiler *prof, cudaStream_t s) {
    switch (g.taps.R) {
        case 5: return launch_exact_r<5>(g, parity, prof, s);
        case 6: return launch_exact_r<6>(g, parity, prof, s);
        case 7: return launch_exact_r<7>(g, parity, prof, s);
        case 8: return launch_exact_r<8>(g, parity, prof, s);
        default: return cudaErrorInvalidValue;
    }
}
}  // namespace tiled
}  // namespace rsf
