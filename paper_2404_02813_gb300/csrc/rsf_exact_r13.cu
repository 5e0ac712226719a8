// rsf_exact_r13.cu -- the exact arithmetic at radii 13 to 16 (see rsf_exact.cuh).
#include "rsf_exact.cuh"

namespace rsf {
namespace tiled {
cudaError_t prepare_exact_r13(int R) {
    switch (R) {
        case 13: return prepare_exact_r<13>();
        case 14: return prepare_exact_r<14>();
        case 15: return prepare_exact_r<15>();
        case 16: return prepare_exact_r<16>();
        default: return cudaErrorInvalidValue;
    }
}
cudaError_t launch_exact_r13(const TiledGroup &g, int parity, Profiler *prof, cudaStream_t s) {
    switch (g.taps.R) {
        case 13: return launch_exact_r<13>(g, parity, prof, s);
        case 14: return launch_exact_r<14>(g, parity, prof, s);
        case 15: return launch_exact_r<15>(g, parity, prof, s);
        case 16: return launch_exact_r<16>(g, parity, prof, s);
        default: return cudaErrorInvalidValue;
    }
}
}  // namespace tiled
}  // namespace rsf
