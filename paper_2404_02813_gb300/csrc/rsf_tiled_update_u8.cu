// rsf_tiled_update_u8.cu -- the update kernel for uint8_t images (see rsf_tiled_update.cuh).
#include "rsf_tiled_update.cuh"

namespace rsf {
namespace tiled {
cudaError_t prepare_update_u8(int R) { return prepare_update<uint8_t>(R); }
cudaError_t launch_update_u8(const TiledGroup &g, int parity, Profiler *prof, cudaStream_t s) {
    return launch_update<uint8_t>(g, parity, prof, s);
}
}  // namespace tiled
}  // namespace rsf
