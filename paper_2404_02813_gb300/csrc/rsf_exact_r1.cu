// rsf_exact_r1.cu -- the exact arithmetic at radii 1 to 4 (see rsf_exact.cuh).
#include "rsf_exact.cuh"

namespace rsf {
namespace tiled {
cudaError_t prepare_exact_r1(int R) {
    switch (R) {
        case 1: return prepare_exact_r<1>();
        case 2: return prepare_exact_r<2>();
        case 3: return prepare_exact_r<3>();
        case 4: return prepare_exact_r<4>();
        default: return cudaErrorInvalidValue;
    }
}
cudaError_t launch_exact_r1(const TiledGroup &g, int parity, Profiler *prof, cudaStream_t s) {
    switch (g.taps.R) {
        case 1: return launch_exact_r<1>(g, parity, prof, s);
        case 2: return launch_exact_r<2>(g, parity, prof, s);
        case 3: return launch_exact_r<3>(g, parity, prof, s);
        case 4: return launch_exact_r<4>(g, parity, prof, s);
        default: return cudaErrorInvalidValue;
    }
}
}  // namespace tiled
}  // namespace rsf
