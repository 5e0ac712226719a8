// rsf_exact_r9.cu -- the exact arithmetic at radii 9 to 12 (see rsf_exact.cuh).
#include "rsf_exact.cuh"

namespace rsf {
namespace tiled {
cudaError_t prepare_exact_r9(int R) {
    switch (R) {
        case 9: return prepare_exact_r<9>();
        case 10: return prepare_exact_r<10>();
        case 11: return prepare_exact_r<11>();
        case 12: return prepare_exact_r<12>();
        default: return cudaErrorInvalidValue;
    }
}
cudaError_t launch_exact_r9(const TiledGroup &g, int parity, Profiler *prof, cudaStream_t s) {
    switch (g.taps.R) {
        case 9: return launch_exact_r<9>(g, parity, prof, s);
        case 10: return launch_exact_r<10>(g, parity, prof, s);
        case 11: return launch_exact_r<11>(g, parity, prof, s);
        case 12: return launch_exact_r<12>(g, parity, prof, s);
        default: return cudaErrorInvalidValue;
    }
}
}  // namespace tiled
}  // namespace rsf
