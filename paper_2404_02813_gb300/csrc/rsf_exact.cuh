// rsf_exact.cuh -- the tiled iteration in the exact arithmetic: IEEE divisions and square
// roots, atanf, both sides of Eq. (10) convolved directly, Li's data terms, on the centred
// FP32 image.  Every radius 1 to 16 (the fast arithmetic of rsf_tiled_*.cu has 2-6, 8, 10,
// 12).  The same four kernels as the other forms (rsf_tiled.cuh) with EX / AB set; results
// equal the six separable passes (rsf_passes.cu) bit for bit, which keep radius 0, volumes of
// 2^32 pitched voxels or more, what does not fit rsf_evolve_noalloc's static memory, and
// RSF_PATH_PASSES.
// 224 x 208 x 192 uint8, radius 7, per iteration: 1.53 ms in the passes (a normal's six
// neighbours from global memory at each of seven places, 0.84 ms alone), 0.33 ms here: x/y
// 0.087, z 0.043, x/y 0.038, update 0.158.
#pragma once

#include "rsf_tiled.cuh"

namespace rsf {
namespace tiled {

template <int R>
constexpr size_t exact_taxy_smem() { return XYSmem<R, SrcH<R, float, 2, true>>::bytes; }

template <int R>
int &exact_persist() {
    static int n = 152;
    return n;
}

template <int R>
cudaError_t prepare_exact_r() {
    cudaError_t e;
    if ((e = prepare_kernel(k_ta_xy<R, float, 2, true>, exact_taxy_smem<R>())) != cudaSuccess) return e;
    if ((e = prepare_kernel(k_ta_z4<R, true>, az4_smem<R>())) != cudaSuccess) return e;
    if ((e = prepare_kernel(k_tb_xy<R, float>, tbxy_smem<R, float>())) != cudaSuccess) return e;
    if ((e = prepare_kernel(k_tb_z<R, float, false, true>, TBZ<R, true>::bytes)) != cudaSuccess) return e;
    if ((e = prepare_kernel(k_tb_z<R, float, true, true>, TBZ<R, true>::bytes)) != cudaSuccess) return e;
    int dev = 0, sms = 0, occ = 0;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
    if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
    if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_ta_z4<R, true>, kAZThreads, az4_smem<R>())) !=
        cudaSuccess) return e;
    exact_persist<R>() = sms * (occ > 0 ? occ : 1);
    return cudaSuccess;
}

template <int R>
cudaError_t launch_exact_r(const TiledGroup &g, int parity, Profiler *prof, cudaStream_t s) {
    GroupArgs G{g.bricks, nullptr, g.nb, parity, g.err, g.fault_tx};
    const TapPairs tp = tap_pairs(g.taps);
    {
        ProfScope ps(prof, KID_TA_XY);
        G.starts = g.starts[0];
        launch_next(g.overlap, k_ta_xy<R, float, 2, true>, g.ncta[0], kXYThreads, exact_taxy_smem<R>(), s, G, tp);
    }
    {
        ProfScope ps(prof, KID_TA_Z);
        G.starts = g.starts[1];
        const unsigned grid = g.ncta[1] < (unsigned)exact_persist<R>() ? g.ncta[1] : (unsigned)exact_persist<R>();
        launch_next(g.overlap, k_ta_z4<R, true>, grid, kAZThreads, az4_smem<R>(), s, G, tp);
    }
    {
        ProfScope ps(prof, KID_TB_XY);
        G.starts = g.starts[2];
        launch_next(g.overlap, k_tb_xy<R, float>, g.ncta[2], kXYThreads, tbxy_smem<R, float>(), s, G, tp);
    }
    {
        ProfScope ps(prof, KID_TB_Z);
        G.starts = g.starts[3];
        if (g.dump)
            launch_next(g.overlap, k_tb_z<R, float, true, true>, g.ncta[3], TBZ<R, true>::THREADS, TBZ<R, true>::bytes, s, G, tp);
        else
            launch_next(g.overlap, k_tb_z<R, float, false, true>, g.ncta[3], TBZ<R, true>::THREADS, TBZ<R, true>::bytes, s, G, tp);
    }
    return cudaGetLastError();
}

}  // namespace tiled
}  // namespace rsf
