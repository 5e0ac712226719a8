// rsf_tiled_update_u16.cu -- the update kernel for uint16_t images (see rsf_tiled_update.cuh).
#include "rsf_tiled_update.cuh"

namespace rsf {
namespace tiled {
cudaError_t prepare_update_u16(int R) { return prepare_update<uint16_t>(R); }
cudaError_t launch_update_u16(const TiledGroup &g, int parity, Profiler *prof, cudaStream_t s) {
    return launch_update<uint16_t>(g, parity, prof, s);
}
}  // namespace tiled
}  // namespace rsf
