// rsf_tiled_update.cuh -- launch and set-up of the update kernel of the tiled
// iteration (k_tb_z of rsf_tiled.cuh) for one image type.  Every storage type and
// both force forms share it; each image type is a translation unit of its own
// (rsf_tiled_update_*.cu), so that they compile side by side.
#pragma once

#include "rsf_tiled.cuh"

namespace rsf {
namespace tiled {

template <int R, class ImgT>
cudaError_t launch_update_r(const TiledGroup &g, int parity, Profiler *prof, cudaStream_t s) {
    GroupArgs G{g.bricks, g.starts[3], g.nb, parity, g.err, g.fault_tx};
    ProfScope ps(prof, KID_TB_Z);
    Taps t = g.taps;
    if (R == 0) {  // the Eq. (15) form: one unit tap, no convolution of (a, b)
        t.R = 0;
        t.g[0] = 1.f;
    }
    if (g.dump)
        launch_next(g.overlap, k_tb_z<R, ImgT, true>, g.ncta[3], TBZ<R>::THREADS, TBZ<R>::bytes, s, G, tap_pairs(t));
    else
        launch_next(g.overlap, k_tb_z<R, ImgT>, g.ncta[3], TBZ<R>::THREADS, TBZ<R>::bytes, s, G, tap_pairs(t));
    return cudaGetLastError();
}
template <int R, class ImgT>
cudaError_t prepare_update_r() {
    const cudaError_t e = prepare_kernel(k_tb_z<R, ImgT, false>, TBZ<R>::bytes);
    if (e != cudaSuccess) return e;
    return prepare_kernel(k_tb_z<R, ImgT, true>, TBZ<R>::bytes);
}

template <class ImgT>
cudaError_t prepare_update(int R) {
    switch (R) {
        case 0: return prepare_update_r<0, ImgT>();
        case 2: return prepare_update_r<2, ImgT>();
        case 3: return prepare_update_r<3, ImgT>();
        case 4: return prepare_update_r<4, ImgT>();
        case 5: return prepare_update_r<5, ImgT>();
        case 6: return prepare_update_r<6, ImgT>();
        case 8: return prepare_update_r<8, ImgT>();
        case 10: return prepare_update_r<10, ImgT>();
        case 12: return prepare_update_r<12, ImgT>();
        default: return cudaErrorInvalidValue;
    }
}

template <class ImgT>
cudaError_t launch_update(const TiledGroup &g, int parity, Profiler *prof, cudaStream_t s) {
    switch (g.force ? 0 : g.taps.R) {
        case 0: return launch_update_r<0, ImgT>(g, parity, prof, s);
        case 2: return launch_update_r<2, ImgT>(g, parity, prof, s);
        case 3: return launch_update_r<3, ImgT>(g, parity, prof, s);
        case 4: return launch_update_r<4, ImgT>(g, parity, prof, s);
        case 5: return launch_update_r<5, ImgT>(g, parity, prof, s);
        case 6: return launch_update_r<6, ImgT>(g, parity, prof, s);
        case 8: return launch_update_r<8, ImgT>(g, parity, prof, s);
        case 10: return launch_update_r<10, ImgT>(g, parity, prof, s);
        case 12: return launch_update_r<12, ImgT>(g, parity, prof, s);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace tiled
}  // namespace rsf
