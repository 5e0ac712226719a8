// rsf_tiled_update_img32.cu -- the update kernel for float images (see rsf_tiled_update.cuh).
#include "rsf_tiled_update.cuh"

namespace rsf {
namespace tiled {
cudaError_t prepare_update_img32(int R) { return prepare_update<float>(R); }
cudaError_t launch_update_img32(const TiledGroup &g, int parity, Profiler *prof, cudaStream_t s) {
    return launch_update<float>(g, parity, prof, s);
}
}  // namespace tiled
}  // namespace rsf
