// rsf_tiled_f32.cu -- instantiates the tiled iteration with FP32 storage (see
// rsf_tiled.cuh), the set-up kernels and the host-side launch dispatch.
#include <cudaTypedefs.h>  // PFN_cuTensorMapEncodeTiled

#include <cmath>

#include "rsf_tiled.cuh"

namespace rsf {
namespace tiled {

namespace {
// The start of one brick by gridDim.x blocks: phi0 to phi, q of it at a pitch of qp, the image
// to img_t at a pitch of ip where that differs.  A warp per row, four values per lane and load
// where rows are dense multiples of 4 (then the brick is one long row).  Ragged rows and copied
// images: a lane has kRowLoads loads in flight (with one, load latency held them at a third of
// the copy rate): 500^3 uint8 with its image copied in words 0.387 -> 0.191 ms, 112 M voxels of
// uint16 bricks 0.442 -> 0.323 ms, 253 x 189 x 147 float 49 -> 19 us.
constexpr int kRowLoads = 4;
template <class T>
__device__ __forceinline__ void copy_rows(const T *__restrict__ src, T *__restrict__ dst, long long rows, int nx, int ip,
                                          long long first, long long step) {
    const int lane = threadIdx.x & 31;
    for (long long r = first; r < rows; r += step) {
        const T *const in = src + r * nx;
        T *const out = dst + r * ip;
        for (int x = lane; x < nx; x += 32 * kRowLoads) {
            T v[kRowLoads];
#pragma unroll
            for (int k = 0; k < kRowLoads; ++k)
                if (x + 32 * k < nx) v[k] = __ldg(in + x + 32 * k);
#pragma unroll
            for (int k = 0; k < kRowLoads; ++k)
                if (x + 32 * k < nx) out[x + 32 * k] = v[k];
        }
    }
}
// the image's rows in words of four bytes where they start and end on one (dst and its pitch do)
template <class T>
__device__ __forceinline__ void copy_image(const SetupBrick &b, long long first, long long step) {
    const int bytes = b.nx * (int)sizeof(T);
    if (sizeof(T) < 4 && bytes % 4 == 0 && reinterpret_cast<uintptr_t>(b.img) % 4 == 0)
        copy_rows(static_cast<const unsigned *>(b.img), static_cast<unsigned *>(b.img_t), b.rows, bytes / 4,
                  b.ip * (int)sizeof(T) / 4, first, step);
    else
        copy_rows(static_cast<const T *>(b.img), static_cast<T *>(b.img_t), b.rows, b.nx, b.ip, first, step);
}
template <bool EX>
__device__ __forceinline__ void start_brick(const SetupBrick &b) {
    const auto q_of = [&](float u) { return EX ? heaviside_q_exact(u, b.eps) : heaviside_q_fast(u, b.eps); };
    const int lane = threadIdx.x & 31;
    const long long first = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5, step = ((long long)gridDim.x * blockDim.x) >> 5;
    const bool copy = b.src != b.phi;
    const uintptr_t at = reinterpret_cast<uintptr_t>(b.src) | reinterpret_cast<uintptr_t>(b.phi);
    if (b.qp == b.nx && at % 16 == 0) {
        const long long n4 = b.rows * b.nx / 4;
        for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n4; i += (long long)gridDim.x * blockDim.x) {
            const float4 u = __ldg(reinterpret_cast<const float4 *>(b.src) + i);
            if (copy) reinterpret_cast<float4 *>(b.phi)[i] = u;
            reinterpret_cast<float4 *>(b.q)[i] = make_float4(q_of(u.x), q_of(u.y), q_of(u.z), q_of(u.w));
        }
    } else {
        for (long long r = first; r < b.rows; r += step) {
            const float *const in = b.src + r * b.nx;
            float *const out = b.phi + r * b.nx, *const q = b.q + r * b.qp;
            for (int x = lane; x < b.nx; x += 32 * kRowLoads) {
                float u[kRowLoads];
#pragma unroll
                for (int k = 0; k < kRowLoads; ++k)
                    if (x + 32 * k < b.nx) u[k] = __ldg(in + x + 32 * k);
#pragma unroll
                for (int k = 0; k < kRowLoads; ++k)
                    if (x + 32 * k < b.nx) {
                        if (copy) out[x + 32 * k] = u[k];
                        q[x + 32 * k] = q_of(u[k]);
                    }
            }
        }
    }
    if (b.img_t != b.img) {
        switch (b.imgtype) {
            case 0: copy_image<uint8_t>(b, first, step); break;
            case 1: copy_image<uint16_t>(b, first, step); break;
            default: copy_image<float>(b, first, step);
        }
    }
}
template <bool EX>
__global__ void __launch_bounds__(256) k_start(SetupBrick b) { start_brick<EX>(b); }
__global__ void __launch_bounds__(256) k_start_many(const SetupBrick *__restrict__ d) { start_brick<false>(d[blockIdx.y]); }
// the centred image (I - m) / s, rows of nx values at a pitch of ip
template <class T>
__global__ void k_center_rows(const T *__restrict__ vol, const float *__restrict__ cs, float *__restrict__ dst,
                              long long rows, int nx, int ip) {
    const float m = cs[0], inv_s = cs[1];
    const int lane = threadIdx.x & 31;
    for (long long r = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5; r < rows;
         r += ((long long)gridDim.x * blockDim.x) >> 5)
        for (int x = lane; x < nx; x += 32) dst[r * ip + x] = ((float)vol[r * nx + x] - m) * inv_s;
}
}  // namespace

// the update kernel per image type (rsf_tiled_update_*.cu)
cudaError_t prepare_update_u8(int R);
cudaError_t prepare_update_u16(int R);
cudaError_t prepare_update_img32(int R);
cudaError_t launch_update_u8(const TiledGroup &g, int parity, Profiler *prof, cudaStream_t s);
cudaError_t launch_update_u16(const TiledGroup &g, int parity, Profiler *prof, cudaStream_t s);
cudaError_t launch_update_img32(const TiledGroup &g, int parity, Profiler *prof, cudaStream_t s);

cudaError_t prepare_tb_z(int R) {
    cudaError_t e = prepare_update_u8(R);
    if (e == cudaSuccess) e = prepare_update_u16(R);
    return e != cudaSuccess ? e : prepare_update_img32(R);
}

cudaError_t launch_tb_z(const TiledGroup &g, int parity, Profiler *prof, cudaStream_t s) {
    switch (g.imgtype) {
        case 0: return launch_update_u8(g, parity, prof, s);
        case 1: return launch_update_u16(g, parity, prof, s);
        default: return launch_update_img32(g, parity, prof, s);
    }
}

}  // namespace tiled

bool tiled_supports(int R) {
    switch (R) {
        case 2: case 3: case 4: case 5: case 6: case 8: case 10: case 12: return true;
        default: return false;
    }
}

int tiled_pitch(int nx) { return (nx + tiled::kZX - 1) / tiled::kZX * tiled::kZX; }

bool tiled_fits(long long nx, long long ny, long long nz) {
    return (long long)tiled_pitch((int)nx) * ny * nz < (1LL << 32);
}

namespace {
// cuTensorMapEncodeTiled, reached through the runtime's driver entry point (no
// link against the driver library); null if the driver does not provide it.
PFN_cuTensorMapEncodeTiled_v12000 tensor_map_encoder() {
    static const PFN_cuTensorMapEncodeTiled_v12000 fn = [] {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q = cudaDriverEntryPointSymbolNotFound;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) !=
                cudaSuccess ||
            q != cudaDriverEntryPointSuccess)
            p = nullptr;
        return reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
    }();
    return fn;
}

// The unit's rules for a 3-D tiled map: base 16-byte aligned, row and plane
// strides multiples of 16 bytes, boxes of 1..256 elements per dimension whose
// rows are a multiple of 16 bytes.
bool map_ok(const void *base, unsigned long long row_bytes, int bx, int by, int bz, int esize) {
    return base && reinterpret_cast<uintptr_t>(base) % 16 == 0 && row_bytes % 16 == 0 &&
           ((unsigned long long)bx * esize) % 16 == 0 && bx >= 1 && bx <= 256 && by >= 1 && by <= 256 && bz >= 1 &&
           bz <= 256;
}

// View [nz][ny][c nx] of a field of `type` elements (esize bytes) with c elements per
// voxel and a row pitch of c rx elements, read in boxes of bx x by x bz elements.
// Elements outside the view (columns < 0 or >= c nx, rows and planes likewise)
// arrive as zeros.
cudaError_t encode_typed(CUtensorMap *m, CUtensorMapDataType type, int esize, const void *base, int c, int rx,
                         const BrickDev &b, int bx, int by, int bz) {
    const PFN_cuTensorMapEncodeTiled_v12000 enc = tensor_map_encoder();
    if (!enc) return cudaErrorNotSupported;
    const unsigned long long row = (unsigned long long)esize * c * rx;
    if (!map_ok(base, row, bx, by, bz, esize)) return cudaErrorInvalidValue;
    const cuuint64_t dims[3] = {(cuuint64_t)c * b.nx, (cuuint64_t)b.ny, (cuuint64_t)b.nz};
    const cuuint64_t strides[2] = {(cuuint64_t)row, (cuuint64_t)row * b.ny};
    const cuuint32_t box[3] = {(cuuint32_t)bx, (cuuint32_t)by, (cuuint32_t)bz};
    const cuuint32_t elem[3] = {1u, 1u, 1u};
    const CUresult r = enc(m, type, 3, const_cast<void *>(base), dims, strides, box, elem,
                           CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                           CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

// FP32 view [nz][ny][c nx] of a pitched field (row pitch c px floats).
cudaError_t encode_map(CUtensorMap *m, const void *base, int c, const BrickDev &b, int bx, int by, int bz) {
    return encode_typed(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, base, c, b.px, b, bx, by, bz);
}

// Box widths (values) and rows of the x/y kernels' staged planes.
struct XYBoxes { int rows, q, img, ab32, ab16; };
template <int R>
XYBoxes xy_boxes_r(int imgtype, int ny) {
    using namespace tiled;
    const int img = imgtype == 0 ? SrcH<R, uint8_t, 1, false>::FI::W : (imgtype == 1 ? SrcH<R, uint16_t, 1, false>::FI::W : SrcH<R, float, 1, false>::FI::W);
    return XYBoxes{xy_box_rows<R>(ny), SrcH<R, float, 1, false>::FQ::W, img, SrcAB<R, float>::FA::W, SrcAB<R, __half>::FA::W};
}
XYBoxes xy_boxes(int R, int imgtype, int ny) {
    switch (R) {
        case 1: return xy_boxes_r<1>(imgtype, ny);
        case 2: return xy_boxes_r<2>(imgtype, ny);
        case 3: return xy_boxes_r<3>(imgtype, ny);
        case 4: return xy_boxes_r<4>(imgtype, ny);
        case 5: return xy_boxes_r<5>(imgtype, ny);
        case 6: return xy_boxes_r<6>(imgtype, ny);
        case 7: return xy_boxes_r<7>(imgtype, ny);
        case 8: return xy_boxes_r<8>(imgtype, ny);
        case 9: return xy_boxes_r<9>(imgtype, ny);
        case 10: return xy_boxes_r<10>(imgtype, ny);
        case 11: return xy_boxes_r<11>(imgtype, ny);
        case 12: return xy_boxes_r<12>(imgtype, ny);
        case 13: return xy_boxes_r<13>(imgtype, ny);
        case 14: return xy_boxes_r<14>(imgtype, ny);
        case 15: return xy_boxes_r<15>(imgtype, ny);
        default: return xy_boxes_r<16>(imgtype, ny);
    }
}
}  // namespace

cudaError_t tiled_encode_maps(BrickDev &b, int force, int storage, int imgtype, int R) {
    const int zrows = tiled::kAZT + 2 * R;
    const XYBoxes box = xy_boxes(R, imgtype, b.ny);
    b.tm_k = b.tm_ab = CUtensorMap{};
    cudaError_t e = encode_typed(&b.tm_q, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, b.q, 1, b.qp, b, box.q, box.rows, 1);
    if (e != cudaSuccess) return e;
    switch (imgtype) {
        case 0: e = encode_typed(&b.tm_img, CU_TENSOR_MAP_DATA_TYPE_UINT8, 1, b.img_t, 1, b.ip, b, box.img, box.rows, 1); break;
        case 1: e = encode_typed(&b.tm_img, CU_TENSOR_MAP_DATA_TYPE_UINT16, 2, b.img_t, 1, b.ip, b, box.img, box.rows, 1); break;
        default: e = encode_typed(&b.tm_img, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, b.img_t, 1, b.ip, b, box.img, box.rows, 1);
    }
    if (e != cudaSuccess) return e;
    if (force != 0) {  // four fields per voxel, no K*I~; the Eq. (15) form: no group B
        e = encode_typed(&b.tm_u, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, b.u2, 4, b.up, b, 128, 1, zrows);
        if (e != cudaSuccess || force == 1) return e;
        return encode_map(&b.tm_ab, b.ab, 2, b, 2 * box.ab32, box.rows, 1);
    }
    e = encode_map(&b.tm_u, b.u2, 2, b, 64, 1, zrows);
    if (e == cudaSuccess) e = encode_map(&b.tm_k, b.ki, 1, b, 32, 1, tiled::kAZT);
    if (e != cudaSuccess) return e;
    if (storage == 0) return encode_map(&b.tm_ab, b.ab, 2, b, 2 * box.ab32, box.rows, 1);
    // a 16-bit pair is one 32-bit value of the map
    return encode_typed(&b.tm_ab, CU_TENSOR_MAP_DATA_TYPE_UINT32, 4, b.ab, 1, b.px, b, box.ab16, box.rows, 1);
}

SetupBrick setup_of(const BrickDev &b, int imgtype, const float *phi0, float *partials, float *cs) {
    return SetupBrick{b.img, imgtype, b.nx, b.qp, b.ip, (long long)b.ny * b.nz, phi0, b.phi[0], b.q,
                      const_cast<void *>(b.img_t), partials, cs, b.eps};
}

namespace {
unsigned start_blocks(long long n) { return (unsigned)(n < 2048LL * 1216 ? (n + 2047) / 2048 : 1216); }
}  // namespace

cudaError_t setup_start(const SetupBrick *d, int n, cudaStream_t s) {
    for (int o = 0; o < n; o += 32768)
        tiled::k_start_many<<<dim3(n >= 8 ? 152 : 1216 / n, n - o < 32768 ? n - o : 32768), 256, 0, s>>>(d + o);
    return cudaGetLastError();
}

cudaError_t tiled_start(const BrickDev &b, int imgtype, const float *phi0, cudaStream_t s) {
    const SetupBrick d = setup_of(b, imgtype, phi0, nullptr, nullptr);
    tiled::k_start<false><<<start_blocks(d.rows * d.nx), 256, 0, s>>>(d);
    return cudaGetLastError();
}

cudaError_t exact_start(const BrickDev &b, const void *vol, int vt, cudaStream_t s) {
    const long long rows = (long long)b.ny * b.nz;
    float *d = static_cast<float *>(const_cast<void *>(b.img));
    const unsigned grid = (unsigned)(rows < 8 * 1216 ? (rows + 7) / 8 : 1216);
    switch (vt) {
        case 0: tiled::k_center_rows<<<grid, 256, 0, s>>>((const uint8_t *)vol, b.cs, d, rows, b.nx, b.ip); break;
        case 1: tiled::k_center_rows<<<grid, 256, 0, s>>>((const uint16_t *)vol, b.cs, d, rows, b.nx, b.ip); break;
        default: tiled::k_center_rows<<<grid, 256, 0, s>>>((const float *)vol, b.cs, d, rows, b.nx, b.ip);
    }
    SetupBrick st = setup_of(b, 2, b.phi[0], nullptr, nullptr);
    st.img_t = const_cast<void *>(st.img);
    tiled::k_start<true><<<start_blocks(rows * b.nx), 256, 0, s>>>(st);
    return cudaGetLastError();
}

cudaError_t tiled_launch_f16(const TiledGroup &g, int parity, Profiler *prof, cudaStream_t s);
cudaError_t tiled_launch_bf16(const TiledGroup &g, int parity, Profiler *prof, cudaStream_t s);
cudaError_t tiled_prepare_f16(int R);
cudaError_t tiled_prepare_bf16(int R);

cudaError_t tiled_prepare_eq15(int R);
namespace tiled {  // the exact arithmetic, four radii per translation unit (rsf_exact_r*.cu)
cudaError_t prepare_exact_r1(int R);
cudaError_t prepare_exact_r5(int R);
cudaError_t prepare_exact_r9(int R);
cudaError_t prepare_exact_r13(int R);
cudaError_t launch_exact_r1(const TiledGroup &g, int parity, Profiler *prof, cudaStream_t s);
cudaError_t launch_exact_r5(const TiledGroup &g, int parity, Profiler *prof, cudaStream_t s);
cudaError_t launch_exact_r9(const TiledGroup &g, int parity, Profiler *prof, cudaStream_t s);
cudaError_t launch_exact_r13(const TiledGroup &g, int parity, Profiler *prof, cudaStream_t s);
}  // namespace tiled
cudaError_t tiled_launch_eq15(const TiledGroup &g, int parity, Profiler *prof, cudaStream_t s);

cudaError_t tiled_prepare(int storage, int R, int force) {
    if (force == kForceExact)
        return R <= 4 ? tiled::prepare_exact_r1(R) : (R <= 8 ? tiled::prepare_exact_r5(R) : (R <= 12 ? tiled::prepare_exact_r9(R) : tiled::prepare_exact_r13(R)));
    const cudaError_t e = tiled::prepare_tb_z(force ? 0 : R);
    if (e != cudaSuccess) return e;
    if (force) return tiled_prepare_eq15(R);  // FP32 intermediates whatever the storage option
    switch (storage) {
        case 0: return tiled::prepare_group_s<float>(R);
        case 1: return tiled_prepare_bf16(R);
        case 2: return tiled_prepare_f16(R);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t load_exact() {
    cudaError_t e = load_kernels(tiled::k_start<true>, tiled::k_center_rows<uint8_t>, tiled::k_center_rows<uint16_t>,
                                 tiled::k_center_rows<float>);
    for (int R = 1; R <= RMAX && e == cudaSuccess; ++R) e = tiled_prepare(0, R, kForceExact);
    return e;
}

cudaError_t tiled_iterate(const TiledGroup &g, int parity, Profiler *prof, cudaStream_t s) {
    const int R = g.taps.R;
    if (g.force == kForceExact)
        return R <= 4 ? tiled::launch_exact_r1(g, parity, prof, s) : (R <= 8 ? tiled::launch_exact_r5(g, parity, prof, s) : (R <= 12 ? tiled::launch_exact_r9(g, parity, prof, s) : tiled::launch_exact_r13(g, parity, prof, s)));
    if (g.force) return tiled_launch_eq15(g, parity, prof, s);
    switch (g.storage) {
        case 0: return tiled::launch_group_s<float>(g, parity, prof, s);
        case 1: return tiled_launch_bf16(g, parity, prof, s);
        case 2: return tiled_launch_f16(g, parity, prof, s);
        default: return cudaErrorInvalidValue;
    }
}

namespace {
// Tile rows and (a, b) ring planes of the update kernel for radius R (0: the Eq. (15) form).
struct UpdateTile { int rows, planes; };
template <int R>
UpdateTile update_tile_r(bool exact) {
    return exact ? UpdateTile{tiled::TBZ<R, true>::TY, tiled::TBZ<R, true>::M} : UpdateTile{tiled::TBZ<R>::TY, tiled::TBZ<R>::M};
}
UpdateTile update_tile(int force, int R) {
    const bool exact = force == kForceExact;
    switch (force == 1 ? 0 : R) {
        case 0: return update_tile_r<0>(exact);
        case 1: return update_tile_r<1>(exact);
        case 2: return update_tile_r<2>(exact);
        case 3: return update_tile_r<3>(exact);
        case 4: return update_tile_r<4>(exact);
        case 5: return update_tile_r<5>(exact);
        case 6: return update_tile_r<6>(exact);
        case 7: return update_tile_r<7>(exact);
        case 8: return update_tile_r<8>(exact);
        case 9: return update_tile_r<9>(exact);
        case 10: return update_tile_r<10>(exact);
        case 11: return update_tile_r<11>(exact);
        case 12: return update_tile_r<12>(exact);
        case 13: return update_tile_r<13>(exact);
        case 14: return update_tile_r<14>(exact);
        case 15: return update_tile_r<15>(exact);
        default: return update_tile_r<16>(exact);
    }
}
// Output rows of the x/y kernels' tiles.
int xy_rows(int R) { return R <= 8 ? tiled::XYG<8>::TH : (R <= 12 ? tiled::XYG<12>::TH : tiled::XYG<16>::TH); }
}  // namespace

void tiled_cta_counts(const BrickDev &b, int force, int R, unsigned counts[4]) {
    const unsigned th = xy_rows(R);
    const unsigned ntx = (b.nx + tiled::kXYT - 1) / tiled::kXYT, nty = (b.ny + th - 1) / th;
    const unsigned nzp = (b.nz + b.xyp - 1) / b.xyp;
    const int rows = update_tile(force, R).rows;
    counts[0] = ntx * nty * nzp;
    counts[1] = (unsigned)((b.nz + tiled::kAZT - 1) / tiled::kAZT) * ((b.nx + 31) / 32) * b.ny;
    counts[2] = counts[0];
    counts[3] = (unsigned)((b.nx + tiled::kZX - 1) / tiled::kZX) * ((b.ny + rows - 1) / rows) *
                ((b.nz + b.zc - 1) / b.zc) * ((b.zc + b.zs - 1) / b.zs);
}

// Overlapping consecutive kernels hides a launch's latency and start-up, which counts where the
// kernels are short (64^3: 1.74 -> 1.25 ms for 50 iterations; 253 x 189 x 147: 2.05 -> 1.90 ms
// for 12), and costs long ones more than that: an SM whose shared-memory carve-out an earlier
// kernel set lower keeps it until it drains, and with the largest carve-out everywhere the L1
// is too small (five iterations of 512^3: 11.3 ms without overlap, 12.2 with it, 11.6 with the
// carve-out too; 160^3 sub-volumes, 2400 CTAs, 9.65, 10.0, 9.80 ms).  The line: eight CTAs per SM
// in group A's x/y kernel, two waves of Li's form (four share an SM), 2.7 of the others (three).
bool tiled_overlap(const TiledGroup &g, int sms) { return g.ncta[0] <= 8u * (unsigned)sms; }

// A CTA of the x/y kernels costs its planes plus about one plane time (set-up and the first
// copies; 64^3: 1 plane per CTA 8.1 us, 16 planes 37 us; 512^3: 16 planes 0.463 ms, 32 planes
// 0.480 ms, so 16 is the most); three or four share an SM.  Few CTAs run in whole waves; many even out but for
// about half a CTA at the end.
int tiled_xy_planes(const BrickDev *bricks, int nb, int force, int R, int sms) {
    const int th = xy_rows(R);
    const double slots = (force ? 3.0 : 4.0) * sms;
    int best = 1;
    double best_cost = 0.0;
    for (int p : {1, 2, 3, 4, 6, 8, 12, 16}) {
        double ctas = 0.0;
        for (const BrickDev *b = bricks; b != bricks + nb; ++b)
            ctas += (double)((b->nx + tiled::kXYT - 1) / tiled::kXYT) * ((b->ny + th - 1) / th) * ((b->nz + p - 1) / p);
        const double waves = ctas / slots;
        const double cost = (waves < 4.0 ? std::ceil(waves) : waves + 0.5) * (p + 1.0);
        if (p == 1 || cost < best_cost) {
            best_cost = cost;
            best = p;
        }
    }
    return best;
}

// A CTA of the update kernel costs its zs output planes plus about 4 + 0.4 M plane times to
// fill its rings (M (a, b) planes at 8 of the 22 bytes a voxel moves, and the latency of the
// first copies).  Two CTAs share an SM.  Few CTAs run in whole waves; many even out but for
// about half a CTA at the end.
int tiled_update_planes(const BrickDev *bricks, int nb, int force, int R, int zc, int sms) {
    const UpdateTile tile = update_tile(force, R);
    const double fill = 4.0 + 0.4 * tile.planes, slots = 2.0 * sms;
    int best = zc, last = 0;
    double best_cost = 0.0;
    for (int parts = 1; parts <= zc; ++parts) {
        int zs = (zc + parts - 1) / parts;
        if (parts > 1) zs = (zs + 3) / 4 * 4;
        if (zs == last) {
            if (zs <= 4) break;
            continue;
        }
        last = zs;
        double ctas = 0.0;
        for (const BrickDev *b = bricks; b != bricks + nb; ++b) {
            const int chunks = b->nz / zc, rest = b->nz % zc;
            ctas += (double)((b->nx + tiled::kZX - 1) / tiled::kZX) * ((b->ny + tile.rows - 1) / tile.rows) *
                    (chunks * ((zc + zs - 1) / zs) + (rest + zs - 1) / zs);
        }
        const double waves = ctas / slots;
        const double cost = (waves < 4.0 ? std::ceil(waves) : waves + 0.5) * (zs + fill);
        if (parts == 1 || cost < best_cost) {
            best_cost = cost;
            best = zs;
        }
    }
    return best;
}

// Per pitched voxel, Li's form: (H I~, H) and, after it in the same memory, the x/y-convolved
// (a, b): 8 bytes; (a, b) 2 elements of the storage type; K*I~ 4 bytes; 8 bytes left.  The
// Eq. (15) form: the two x/y-convolved pairs 16 bytes, the fits (f1, f2) 8 bytes; 4 bytes left
// with FP32 storage, none with 16-bit.  What is left, or what q leaves of its block, holds the
// copied image of a brick whose rows are not 16-byte aligned (at most 4 bytes per pitched voxel).
size_t tiled_stage_bytes(int storage, long long np) { return (size_t)(storage == 0 ? 28 : 24) * (size_t)np; }

namespace {
int image_size(int imgtype) { return imgtype == 0 ? 1 : (imgtype == 1 ? 2 : 4); }
int image_pitch(int nx, int imgtype) {
    const int per = 16 / image_size(imgtype);
    return (nx + per - 1) / per * per;
}
bool copied_image(const void *img, int nx, int imgtype) {
    return image_pitch(nx, imgtype) != nx || reinterpret_cast<uintptr_t>(img) % 16 != 0;
}
size_t field_bytes(int storage, int force, long long np) { return (size_t)(force ? 24 : (storage == 0 ? 20 : 16)) * np; }
int q_pitch(int nx) { return (nx + 3) / 4 * 4; }
}  // namespace

size_t tiled_q_bytes(int nx, long long rows) { return 2 * ((sizeof(float) * nx * rows + 255) / 256 * 256); }

// Per pitched voxel: both x/y-convolved pairs 16 bytes (then, in the same memory, the
// x/y-convolved (a, b)), (a, b) 8, the centred image at most 4.
void exact_place_fields(BrickDev &b, void *stage, float *q) {
    b.px = b.up = tiled_pitch(b.nx);
    const long long np = (long long)b.px * b.ny * b.nz;
    char *p = static_cast<char *>(stage);
    b.u2 = b.abxy = reinterpret_cast<float2 *>(p);
    b.ab = p + 16 * np;
    b.ki = nullptr;
    b.img = b.img_t = p + 24 * np;
    b.q = q;
    b.qp = b.ip = q_pitch(b.nx);
}
size_t exact_stage_bytes(int nx, int ny, int nz) {
    return (24ull * tiled_pitch(nx) + 4ull * q_pitch(nx)) * ny * nz;
}
size_t exact_q_bytes(int nx, int ny, int nz) { return 4ull * q_pitch(nx) * ny * nz; }
bool exact_supports(int R) { return R >= 1 && R <= RMAX; }

void tiled_place_fields(BrickDev &b, int storage, int force, int imgtype, void *stage, size_t stage_bytes, void *q) {
    const long long rows = (long long)b.ny * b.nz;
    b.px = b.up = tiled_pitch(b.nx);
    const long long np = b.px * rows;
    char *p = static_cast<char *>(stage);
    b.u2 = reinterpret_cast<float2 *>(p);
    if (force) {
        b.ab = nullptr;
        b.abxy = reinterpret_cast<float2 *>(p + 16 * np);
        b.ki = nullptr;
    } else {
        b.abxy = b.u2;
        b.ab = p + 8 * np;
        b.ki = reinterpret_cast<float *>(p + (storage == 0 ? 16 : 12) * np);
    }
    b.q = static_cast<float *>(q);
    b.qp = q_pitch(b.nx);
    b.img_t = b.img;
    b.ip = b.nx;
    if (copied_image(b.img, b.nx, imgtype)) {
        b.ip = image_pitch(b.nx, imgtype);
        const size_t need = (size_t)image_size(imgtype) * b.ip * rows, used = field_bytes(storage, force, np);
        const size_t qb = 4ull * b.qp * rows;  // a multiple of 16
        if (used + need <= stage_bytes) {
            b.img_t = p + used;
        } else {
            b.img_t = static_cast<char *>(q) + qb;
            if (qb + need > tiled_q_bytes(b.nx, rows)) {
                // Eq. (15) form, 24 bytes per voxel of stage, FP32 rows of 4 k + 1 .. 3 values (or
                // short rows): the image runs on into the stage block behind the q block, by at
                // most 8 (qp - nx) bytes a row, and the pair field, without padded columns, ends
                // 16 (px - nx) bytes a row earlier
                const size_t spill = qb + need - tiled_q_bytes(b.nx, rows);
                b.up = b.nx;
                b.u2 = reinterpret_cast<float2 *>(p + spill);
                b.abxy = reinterpret_cast<float2 *>(p + spill + 16ull * b.nx * rows);
            }
        }
    }
}

namespace {
template <int R, class ImgT>
cudaError_t ki_init_r(const TiledGroup &g, cudaStream_t s) {
    constexpr size_t sm = tiled::XYSmem<R, tiled::SrcI<R, ImgT>>::bytes;
    static_assert(sm <= 48 * 1024 && tiled::ki_smem<R>() <= 48 * 1024, "no shared-memory opt-in");
    const tiled::TapPairs tp = tiled::tap_pairs(g.taps);
    tiled::GroupArgs G{g.bricks, g.starts[0], g.nb, 0, g.err, 0u};
    tiled::k_ki_xy<R, ImgT><<<g.ncta[0], tiled::kXYThreads, sm, s>>>(G, tp);
    G.starts = g.starts[1];
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    const unsigned most = (unsigned)(tiled::kAZCtas * sms);
    tiled::k_ki_z<R><<<g.ncta[1] < most ? g.ncta[1] : most, tiled::kAZThreads, tiled::ki_smem<R>(), s>>>(G, tp);
    return cudaGetLastError();
}
template <int R>
cudaError_t ki_init_i(const TiledGroup &g, cudaStream_t s) {
    switch (g.imgtype) {
        case 0: return ki_init_r<R, uint8_t>(g, s);
        case 1: return ki_init_r<R, uint16_t>(g, s);
        default: return ki_init_r<R, float>(g, s);
    }
}
}  // namespace

cudaError_t tiled_ki_init(const TiledGroup &g, cudaStream_t s) {
    if (g.force != 0) return cudaSuccess;  // the other forms convolve the complement directly
    switch (g.taps.R) {
        case 2: return ki_init_i<2>(g, s);
        case 3: return ki_init_i<3>(g, s);
        case 4: return ki_init_i<4>(g, s);
        case 5: return ki_init_i<5>(g, s);
        case 6: return ki_init_i<6>(g, s);
        case 8: return ki_init_i<8>(g, s);
        case 10: return ki_init_i<10>(g, s);
        case 12: return ki_init_i<12>(g, s);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace rsf
