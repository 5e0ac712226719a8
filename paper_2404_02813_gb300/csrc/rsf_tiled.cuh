// rsf_tiled.cuh -- the tiled four-kernel RSF iteration (arXiv 2404.02813,
// Sec. 3 and 4.2) over a table of bricks.
//
// A launch covers every brick of one group (same kernel radius R and image
// type); a plain volume is a group of one brick.  Each brick is an independent
// volume with its own boundaries, fields and scalars (the sub-volumes of the
// paper's volume-level parallelism, Sec. 4.1).  A CTA finds its brick by a
// binary search over the per-kernel CTA offsets of the group.
//
//   rsf_ta_xy  per z-plane and 32-column tile, q = +-atan(eps/|phi|)/pi and the
//              image by TMA; forms H I~ and H (Eqs. 6, 8-10; the image centred)
//              as it reads them, convolves the pair along x then y (packed f32x2
//              FMAs) and stores it (FP32).
//   rsf_ta_z   x-z slabs (32 columns x 64 output planes) brought to shared
//              memory by TMA, two slabs in flight; z convolution streamed into
//              eight accumulators per column; the local fits f1 = K*(H I~)/K*H and
//              f2 = K*((1-H) I~)/K*(1-H), the latter from the linearity of the
//              convolution as (K*I~ - K*(H I~)) / (K*1 - K*H) with K*I~ fixed
//              for the solve (rsf_ki_xy / rsf_ki_z, once) and K*1 the product of
//              the three 1-D zero-padding profiles; a = l1 f1 - l2 f2,
//              b = l1 f1^2 - l2 f2^2 (stored FP32, FP16 or BF16).
//   rsf_tb_xy  the x/y kernel on (a, b); its output stays FP32 (the data term
//              below is a difference of terms much larger than itself).
//   rsf_tb_z   a z march over a 32 x 14 column tile (12 or 10 rows at larger
//              radii), two columns per thread: (a, b) and phi rings in shared
//              memory filled by cp.async, the unit normal computed once per
//              column and plane;
//              g = s^2 [ (l1 - l2) K1 I~^2 - 2 I~ K*a + K*b ]  (Eqs. 11-12),
//              kappa and the Laplacian (Eqs. 3-4), the update of Eqs. (1),
//              (13), (14), and q of the new phi for the next rsf_ta_xy.
//
// Convolutions use zero padding, taps summed k = -R..R, FP32 accumulation;
// finite differences use reflect-101 for phi and for the normal.  The
// intermediate fields are stored with an x pitch rounded up to 32 columns.
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <cstdint>
#include <type_traits>
#include <utility>

#include "rsf_internal.h"

namespace rsf {
namespace tiled {

constexpr int kXYT = 32;          // x/y kernel: output columns of a tile (its rows: XYG)
constexpr int kXYThreads = 256;   // 8 warps
constexpr int kZX = 32;           // z march: columns (x) per CTA
constexpr int kAZT = 64;          // x-z slab: output planes per CTA
constexpr int kAZThreads = 256;
constexpr int kAZO = kAZT / (kAZThreads / 32);
constexpr int kAZCtas = 3;        // per SM

__device__ __forceinline__ float2 f2fma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }

// The taps of Eq. (7) duplicated into (g_k, g_k) pairs, passed by value: the
// first operand of a packed f32x2 FMA over a field pair, read from the
// kernel's parameter space.
struct TapPairs {
    float2 g[2 * RMAX + 1];
};
inline TapPairs tap_pairs(const Taps &t) {
    TapPairs p{};
    for (int k = 0; k <= 2 * t.R; ++k) p.g[k] = make_float2(t.g[k], t.g[k]);
    return p;
}
__device__ __forceinline__ int clampi(int v, int lo, int hi) { return v < lo ? lo : (v > hi ? hi : v); }

// ------------------------------------------------------------- storage

template <class S> struct Store;
template <> struct Store<float> {
    using V2 = float2;
    __device__ __forceinline__ static V2 pack2(float2 v) { return v; }
    __device__ __forceinline__ static float2 unpack2(V2 v) { return v; }
};
template <> struct Store<__half> {
    using V2 = uint32_t;
    __device__ __forceinline__ static uint32_t p(float a, float b) {
        __half2 h = __floats2half2_rn(a, b);
        return *reinterpret_cast<uint32_t *>(&h);
    }
    __device__ __forceinline__ static float2 u(uint32_t w) { return __half22float2(*reinterpret_cast<__half2 *>(&w)); }
    __device__ __forceinline__ static V2 pack2(float2 v) { return p(v.x, v.y); }
    __device__ __forceinline__ static float2 unpack2(V2 v) { return u(v); }
};
template <> struct Store<__nv_bfloat16> {
    using V2 = uint32_t;
    __device__ __forceinline__ static uint32_t p(float a, float b) {
        __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
        return *reinterpret_cast<uint32_t *>(&h);
    }
    __device__ __forceinline__ static float2 u(uint32_t w) {
        return __bfloat1622float2(*reinterpret_cast<__nv_bfloat162 *>(&w));
    }
    __device__ __forceinline__ static V2 pack2(float2 v) { return p(v.x, v.y); }
    __device__ __forceinline__ static float2 unpack2(V2 v) { return u(v); }
};

// ------------------------------------------------------------ brick table

__device__ __forceinline__ int find_brick(const int *__restrict__ starts, int nb, int cta) {
    int lo = 0, hi = nb;  // starts[lo] <= cta < starts[hi]
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (__ldg(starts + mid) <= cta) lo = mid; else hi = mid;
    }
    return lo;
}

struct GroupArgs {
    const BrickDev *bricks;
    const int *starts;  // nb + 1 CTA offsets of this kernel within the launch
    int nb;
    int parity;         // launch parity: a brick reads phi[p] with p = parity ^ flip, writes the other
    int *err;           // the group's error word (bounded waits), may be null
    unsigned fault_tx;  // extra bytes the TMA barriers expect (0; > 0 only in a fault test)
};

// ---- TMA tile copies completing on shared-memory mbarriers (PTX ISA: mbarrier,
// cp.async.bulk.tensor).  One thread arms a barrier with the bytes it expects and
// issues the copies; every thread waits for the phase to complete, for at most
// kWaitNs (then the kernel reports through the group's error word).
constexpr unsigned long long kWaitNs = 1000000000ull;  // 1 s

__device__ __forceinline__ unsigned smem_addr(const void *p) { return (unsigned)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mbar_init(uint64_t *bar, unsigned count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(smem_addr(bar)), "r"(count) : "memory");
}
// makes initialised barriers visible to the other threads and to the copy unit
__device__ __forceinline__ void mbar_init_fence() {
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
}
__device__ __forceinline__ void mbar_inval(uint64_t *bar) {
    asm volatile("mbarrier.inval.shared::cta.b64 [%0];\n" ::"r"(smem_addr(bar)) : "memory");
}
// one arrival that also raises the phase's expected transaction count by `bytes`
__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t *bar, unsigned bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(smem_addr(bar)), "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, unsigned parity) {
    unsigned done;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(done)
        : "r"(smem_addr(bar)), "r"(parity)
        : "memory");
    return done != 0;
}
__device__ __forceinline__ unsigned long long globaltimer_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;\n" : "=l"(t));
    return t;
}
// waits for the completion of the barrier's phase of the given parity until the
// global timer passes `deadline`; false if it did not complete by then
__device__ __forceinline__ bool mbar_wait_until(uint64_t *bar, unsigned parity, unsigned long long deadline) {
    while (!mbar_try_wait(bar, parity))
        if (globaltimer_ns() > deadline) return false;
    return true;
}
// the same for at most kWaitNs from the first failed try (the timer is read only then)
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, unsigned parity) {
    return mbar_try_wait(bar, parity) || mbar_wait_until(bar, parity, globaltimer_ns() + kWaitNs);
}
// orders this thread's earlier generic-proxy accesses to shared memory before
// later copies of the async proxy (the copy unit) into it
__device__ __forceinline__ void fence_proxy_async_smem() {
    asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
}
// The tensor map at `map` in global memory as it is now (the host rewrites the
// descriptor array between launches, perhaps over maps the copy unit has seen).
__device__ __forceinline__ void fence_tensormap(const CUtensorMap *map) {
    asm volatile("fence.proxy.tensormap::generic.acquire.gpu [%0], 128;\n" ::"l"(reinterpret_cast<uint64_t>(map))
                 : "memory");
}
// 3-D tile load of the box at element coordinates (x, y, z) of `map` into `dst`
// (128-byte aligned), completing `bytes of the box` on `bar`.  x times the
// element size must be a multiple of 16 bytes; y and z may lie outside the
// tensor (those elements arrive as zeros).
__device__ __forceinline__ void tma_load_3d(void *dst, const CUtensorMap *map, int x, int y, int z, uint64_t *bar) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], "
        "[%5];\n" ::"r"(smem_addr(dst)),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(z), "r"(smem_addr(bar))
        : "memory");
}
// Programmatic dependent launch: every kernel of an iteration lets the next one start as
// soon as all of its CTAs have (dependents_may_start, first thing), and waits for the
// completion of the one before, its writes included, before it reads or writes a field
// (wait_for_previous, every thread).  What comes before that -- finding the brick, offsets,
// barriers -- overlaps the previous kernel's end; only descriptors and constants written
// before the first iteration are read there.
__device__ __forceinline__ void dependents_may_start() { asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory"); }
__device__ __forceinline__ void wait_for_previous() { asm volatile("griddepcontrol.wait;\n" ::: "memory"); }
template <class K>
cudaError_t prepare_kernel(K *kernel, size_t smem) {
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
}
template <class... P, class... A>
void launch_next(bool overlap, void (*kernel)(P...), unsigned grid, unsigned threads, size_t smem, cudaStream_t s,
                 A... args) {
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = overlap ? 1 : 0;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, kernel, P(args)...);  // an error stays for cudaGetLastError
}
// records an error in the group's error word (mapped host memory), once per CTA
__device__ __forceinline__ void report_error(int *err, int code) {
    if (err && threadIdx.x == 0) {
        *reinterpret_cast<volatile int *>(err) = code;
        __threadfence_system();
    }
}

// ---------------------------------------------------------------- x / y

// The x/y kernels: per z-plane and tile of 32 columns x XYG::TH rows, the x then the y
// convolution (zero padding) of one or two FP32 pairs per voxel.
//
// What bounds them: the shared-memory pipe (an earlier form, with 32 x 32 tiles, a pass
// that wrote the products into a tile of their own and four outputs per thread in both
// phases, moved 1.02 wavefronts per voxel at radius 6 and kept that pipe 85 % busy).  So
//  - the TMA box of a plane (q and image, or (a, b)) is the x phase's own input: the
//    products H I~, H are formed in registers as the window is read;
//  - a warp's x phase is one item of 8 rows x 32 columns, eight outputs per lane, so that
//    a window of 8 + 2R inputs serves eight outputs; rows of all items are at most 64,
//    one item per warp;
//  - the y phase gives each lane TH / 8 rows of one column.
// Reads and writes are 16 bytes wherever the row pitch allows; an 8-lane phase covers
// 8 rows, whose pitch is an odd number of 16-byte units: no bank conflicts.
// A staging buffer is refilled as soon as the x phase has read it.  (H I~, H): one buffer,
// four CTAs per SM (two buffers: the same time; three CTAs: 4 % slower).  (a, b), whose
// boxes are larger and whose phases shorter: two buffers, three CTAs per SM (0.342 against
// 0.370 ms at 512^3 with one buffer and four CTAs).
//
// Per launch, before and now: 512^3 uint16 radius 6, (H I~, H) 0.541 -> 0.459 ms (issue and
// FMA pipe 60 and 50 % busy), (a, b) 0.393 -> 0.342 ms (0.92 of the HBM rate); 512 x 448 x
// 320 radius 10 0.519 -> 0.400 and 0.327 -> 0.282 ms; both pairs, 500^3 uint8 radius 10,
// 1.741 -> 1.12 ms (FMA pipe 65 %: 105 packed FMAs per voxel); (a, b) in BF16, 768^3, 1.764
// -> 1.083 ms; 64^3 uint8 21.6 -> 8.1 and 15.7 -> 6.3 us (fewer planes per CTA).
template <int R>
struct XYG {
    static constexpr int TH = R <= 8 ? 48 : (R <= 12 ? 40 : 32);  // output rows
    static constexpr int H = TH + 2 * R;         // staged rows: at most 64 (one item of 8 rows per warp)
    static constexpr int YT = TH / (kXYThreads / 32);
    static constexpr int NI = 8 + 2 * R;         // inputs of an x-phase window
    static constexpr int T = 2 * R + 1;
    static_assert(H <= 64 && TH % 8 == 0, "x/y tile rows");
};
// Rows of a plane's boxes: a brick thinner than a tile stages its own rows and their halo only
// (1024 x 4 x 1024 at radius 2: (H I~, H) 116 -> 80 us, (a, b) 78 -> 47; with whole boxes
// a volume of 4 to 8 rows was up to 17 % slower per iteration than with tiles of 32 rows).
template <int R>
__host__ __device__ constexpr int xy_box_rows(int ny) { return ny + 2 * R < XYG<R>::H ? ny + 2 * R : XYG<R>::H; }
constexpr int round_up(int v, int m) { return (v + m - 1) / m * m; }
// the smallest multiple of `unit` >= need that is an odd number of units
constexpr int odd_pitch(int need, int unit) { return (round_up(need, unit) / unit) % 2 ? round_up(need, unit) : round_up(need, unit) + unit; }
// Staging geometry of one field with E values per 16 bytes, read by windows of V values
// (V values are 8 or 16 bytes): the box starts RA >= R columns left of the tile (16-byte
// aligned), a window's first aligned read at column xo + B, its first input O values in.
template <int R, int E, int V>
struct XYField {
    static constexpr int RA = round_up(R, E);
    static constexpr int O = (RA - R) % V, B = RA - R - O;
    static constexpr int N = (O + XYG<R>::NI + V - 1) / V;  // reads per window
    static constexpr int need = 24 + B + N * V > 32 + RA + R ? 24 + B + N * V : 32 + RA + R;
    static constexpr int W = odd_pitch(need, E);            // box width and row pitch (values)
    static_assert(W <= 256, "box width");
};

template <class T> struct ImgVec;  // eight bytes of uint8, sixteen of the others
template <> struct ImgVec<uint8_t> {
    static constexpr int V = 8;
    uint2 w;
    __device__ __forceinline__ void load(const uint8_t *p) { w = *reinterpret_cast<const uint2 *>(p); }
    __device__ __forceinline__ float get(int i) const { return (float)(((i < 4 ? w.x : w.y) >> (8 * (i & 3))) & 255u); }
};
template <> struct ImgVec<uint16_t> {
    static constexpr int V = 8;
    uint4 w;
    __device__ __forceinline__ void load(const uint16_t *p) { w = *reinterpret_cast<const uint4 *>(p); }
    __device__ __forceinline__ float get(int i) const {
        const uint32_t u = i < 2 ? w.x : (i < 4 ? w.y : (i < 6 ? w.z : w.w));
        return (float)((u >> (16 * (i & 1))) & 0xffffu);
    }
};
template <> struct ImgVec<float> {
    static constexpr int V = 4;
    float4 w;
    __device__ __forceinline__ void load(const float *p) { w = *reinterpret_cast<const float4 *>(p); }
    __device__ __forceinline__ float get(int i) const { return i == 0 ? w.x : (i == 1 ? w.y : (i == 2 ? w.z : w.w)); }
};

// A source of the x phase: CTAs per SM and staging buffers its kernel is built for, geometry of
// its staging buffer, issue() of one plane's boxes
// (one thread), fix() of what the copies' zero fill gets wrong outside the brick (all
// threads; FIX: it is needed), and window(): f(j, pairs) for the NI inputs of a window.
// EX: q from the exact arithmetic, whose zero keeps its sign (q = -0: H = 0)
template <int R, class ImgT, int NP_, bool EX>
struct SrcH {  // NP = 1: (H I~, H); NP = 2: also ((1-H) I~, 1-H), the other side of Eq. (10)
    using V = float2;
    static constexpr int NP = NP_, CTAS = NP == 1 ? 4 : 3, NS = 1;
    static constexpr bool FIX = true;
    using G = XYG<R>;
    using FQ = XYField<R, 4, 4>;
    using FI = XYField<R, 16 / (int)sizeof(ImgT), ImgVec<ImgT>::V>;
    static constexpr int QB = FQ::W * G::H * 4, IB = FI::W * G::H * (int)sizeof(ImgT);
    static constexpr int IOFF = round_up(QB, 128), BYTES = IOFF + round_up(IB, 128);
    const CUtensorMap *mq, *mi;
    float inv_s, nms;
    __device__ __forceinline__ void fence() const {
        fence_tensormap(mq);
        fence_tensormap(mi);
    }
    __device__ __forceinline__ void issue(unsigned char *st, int x0, int y0, int z, int rows, uint64_t *bar,
                                          unsigned more) const {
        mbar_arrive_expect_tx(bar, (unsigned)(rows * (FQ::W * 4 + FI::W * (int)sizeof(ImgT))) + more);
        tma_load_3d(st, mq, x0 - FQ::RA, y0 - R, z, bar);
        tma_load_3d(st + IOFF, mi, x0 - FI::RA, y0 - R, z, bar);
    }
    // q is the small side of Eq. (10), atan(eps/|phi|)/pi with the sign of phi: H = -q where it is
    // negative, else 1 - q.  q = 1 outside the brick: H = 0, so both products vanish there (q
    // itself is at most 1/2 in magnitude; zero-filled q would read as H = 1)
    __device__ __forceinline__ void fix(unsigned char *st, int x0, int y0, int nx, int ny, int rows) const {
        float *q = reinterpret_cast<float *>(st);
        const int lane = threadIdx.x & 31;
        for (int row = threadIdx.x >> 5; row < rows; row += kXYThreads / 32) {
            const bool out = (unsigned)(y0 - R + row) >= (unsigned)ny;
            for (int c = lane; c < FQ::W; c += 32)
                if (out || (unsigned)(x0 - FQ::RA + c) >= (unsigned)nx) q[row * FQ::W + c] = 1.f;
        }
    }
    template <class F>
    __device__ __forceinline__ void window(const unsigned char *st, int row, int xo, const F &f) const {
        const float *q = reinterpret_cast<const float *>(st) + row * FQ::W + xo + FQ::B;
        const ImgT *im = reinterpret_cast<const ImgT *>(st + IOFF) + row * FI::W + xo + FI::B;
        float4 q4 = make_float4(0.f, 0.f, 0.f, 0.f);
        ImgVec<ImgT> iv;
#pragma unroll
        for (int j = 0; j < G::NI; ++j) {
            const int jq = j + FQ::O, ji = j + FI::O;
            if (j == 0 || jq % 4 == 0) q4 = *reinterpret_cast<const float4 *>(q + jq / 4 * 4);
            if (j == 0 || ji % ImgVec<ImgT>::V == 0) iv.load(im + ji / ImgVec<ImgT>::V * ImgVec<ImgT>::V);
            const float qj = jq % 4 == 0 ? q4.x : (jq % 4 == 1 ? q4.y : (jq % 4 == 2 ? q4.z : q4.w));
            const float v = fmaf(iv.get(ji % ImgVec<ImgT>::V), inv_s, nms);
            const bool neg = EX ? __float_as_int(qj) < 0 : qj < 0.f;
            const float h = neg ? -qj : 1.f - qj;
            float2 p[NP];
            p[0] = make_float2(__fmul_rn(h, v), h);
            if constexpr (NP == 2) {
                const float hc = qj >= 0.75f ? 0.f : (neg ? 1.f + qj : qj);  // the mark of fix()
                p[1] = make_float2(__fmul_rn(hc, v), hc);
            }
            f(j, p);
        }
    }
};

template <int R, class ImgT>
struct SrcI {  // the centred image alone, one float per voxel, for K*I~
    using V = float;
    static constexpr int NP = 1, CTAS = 4, NS = 1;
    static constexpr bool FIX = false;
    using G = XYG<R>;
    using FI = XYField<R, 16 / (int)sizeof(ImgT), ImgVec<ImgT>::V>;
    static constexpr int IB = FI::W * G::H * (int)sizeof(ImgT), BYTES = round_up(IB, 128);
    const CUtensorMap *mi;
    float inv_s, nms;
    int x0, y0, nx, ny;
    __device__ __forceinline__ void fence() const { fence_tensormap(mi); }
    __device__ __forceinline__ void issue(unsigned char *st, int, int, int z, int rows, uint64_t *bar,
                                          unsigned more) const {
        mbar_arrive_expect_tx(bar, (unsigned)(rows * FI::W * (int)sizeof(ImgT)) + more);
        tma_load_3d(st, mi, x0 - FI::RA, y0 - R, z, bar);
    }
    __device__ __forceinline__ void fix(unsigned char *, int, int, int, int, int) const {}
    template <class F>
    __device__ __forceinline__ void window(const unsigned char *st, int row, int xo, const F &f) const {
        const ImgT *im = reinterpret_cast<const ImgT *>(st) + row * FI::W + xo + FI::B;
        const bool in_y = (unsigned)(y0 - R + row) < (unsigned)ny;
        const int gx = x0 - R + xo;
        ImgVec<ImgT> iv;
#pragma unroll
        for (int j = 0; j < G::NI; ++j) {
            const int ji = j + FI::O;
            if (j == 0 || ji % ImgVec<ImgT>::V == 0) iv.load(im + ji / ImgVec<ImgT>::V * ImgVec<ImgT>::V);
            const bool in = in_y && (unsigned)(gx + j) < (unsigned)nx;
            const float p[1] = {in ? fmaf(iv.get(ji % ImgVec<ImgT>::V), inv_s, nms) : 0.f};
            f(j, p);
        }
    }
};

// (a, b) as stored by rsf_ta_z: FP32 pairs, or 16-bit pairs widened as the window is read
template <int R, class S>
struct SrcAB {
    using V = float2;
    static constexpr int NP = 1, CTAS = 3, NS = 2;
    static constexpr bool FIX = false;  // the zero fill is the convolution's padding
    using G = XYG<R>;
    using V2 = typename Store<S>::V2;
    static constexpr int E = 16 / (int)sizeof(V2);  // pairs per 16 bytes
    using FA = XYField<R, E, E>;
    static constexpr int AB = FA::W * G::H * (int)sizeof(V2), BYTES = round_up(AB, 128);
    const CUtensorMap *ma;
    __device__ __forceinline__ void fence() const { fence_tensormap(ma); }
    __device__ __forceinline__ void issue(unsigned char *st, int x0, int y0, int z, int rows, uint64_t *bar,
                                          unsigned more) const {
        mbar_arrive_expect_tx(bar, (unsigned)(rows * FA::W * (int)sizeof(V2)) + more);
        tma_load_3d(st, ma, (x0 - FA::RA) * (int)(sizeof(V2) / 4), y0 - R, z, bar);
    }
    __device__ __forceinline__ void fix(unsigned char *, int, int, int, int, int) const {}
    template <class F>
    __device__ __forceinline__ void window(const unsigned char *st, int row, int xo, const F &f) const {
        const V2 *a = reinterpret_cast<const V2 *>(st) + row * FA::W + xo + FA::B;
        float2 v[E];
#pragma unroll
        for (int j = 0; j < G::NI; ++j) {
            const int ja = j + FA::O;
            if (j == 0 || ja % E == 0) {
                const uint4 w = *reinterpret_cast<const uint4 *>(a + ja / E * E);
                const V2 *u = reinterpret_cast<const V2 *>(&w);
#pragma unroll
                for (int e = 0; e < E; ++e) v[e] = Store<S>::unpack2(u[e]);
            }
            const float2 p[1] = {v[ja % E]};
            f(j, p);
        }
    }
};

// Where the x/y-convolved fields go: pitched, FP32, a voxel's values side by side.
struct OutXY {
    float *u;
    int px;
    long long pplane;
};

// Shared memory: NS staging buffers, the x-convolved rows, an mbarrier per buffer.  Row pitch
// of the x-convolved rows: an odd number of 16-byte units (36 floats, 34 float2 or 33 float4).
template <int R, class Src>
struct XYSmem {
    using V = typename Src::V;
    static constexpr int XS = Src::NP == 2 ? 33 : (sizeof(V) == 8 ? 34 : 36);
    static constexpr int XC = Src::NP * (int)sizeof(V) * XYG<R>::H * XS;
    static constexpr int NS = Src::NS;
    static constexpr size_t bytes = NS * Src::BYTES + XC + NS * sizeof(uint64_t);
};

__device__ __forceinline__ float2 tap_fma(float2 g, float2 v, float2 a) { return f2fma(g, v, a); }
__device__ __forceinline__ float tap_fma(float2 g, float v, float a) { return fmaf(g.x, v, a); }

// Planes [za, za + np) of tile (x0, y0).  Waits are bounded (expiry reported in the group's
// error word).
template <int R, class Src>
__device__ __forceinline__ void xy_tile(const GroupArgs &G, const Src &src, const OutXY &out, int nx, int ny, int nz,
                                        int x0, int y0, int za, int np, const TapPairs &t, unsigned char *sm) {
    using X = XYG<R>;
    constexpr int NP = Src::NP, T = X::T, YT = X::YT;
    constexpr int XS = XYSmem<R, Src>::XS, NS = XYSmem<R, Src>::NS;
    using V = typename Src::V;
    V *xc = reinterpret_cast<V *>(sm + NS * Src::BYTES);
    uint64_t *bar = reinterpret_cast<uint64_t *>(sm + NS * Src::BYTES + XYSmem<R, Src>::XC);
    if (smem_addr(sm) % 128u != 0u) {
        report_error(G.err, kErrSmemAlign);
        return;
    }
    const int zb_end = min(za + np, nz);
    if (za >= zb_end) return;
    if (threadIdx.x == 0) {
        for (int i = 0; i < NS; ++i) mbar_init(bar + i, 1);
        mbar_init_fence();
    }
    __syncthreads();
    wait_for_previous();
    if (threadIdx.x == 0) {
        src.fence();
        for (int i = 0; i < NS && za + i < zb_end; ++i)
            src.issue(sm + i * Src::BYTES, x0, y0, za + i, xy_box_rows<R>(ny), bar + i, G.fault_tx);
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int row = warp * 8 + (lane & 7), xo = (lane >> 3) * 8;  // x phase: eight outputs of one row
    const int rows = min(X::TH, ny - y0);                        // output rows inside the brick
    const bool xrow = row < rows + 2 * R;
    const bool fix = Src::FIX && (x0 < R || y0 < R || x0 + 32 + R > nx || y0 + X::TH + R > ny);
    const int yr = warp * YT;                                    // y phase: YT rows of one column
    const bool yrow = yr < rows, col = x0 + lane < nx;
    V *o = reinterpret_cast<V *>(out.u) + ((long long)za * out.pplane + (long long)(y0 + yr) * out.px + x0 + lane) * NP;
    for (int z = za; z < zb_end; ++z) {
        const int i = (z - za) % NS;
        const unsigned phase = (unsigned)((z - za) / NS) & 1u;
        unsigned char *const st = sm + i * Src::BYTES;
        if (!mbar_wait(bar + i, phase)) {  // then the same time again for the copies to land
            report_error(G.err, kErrWaitExpired);
            const unsigned long long deadline = globaltimer_ns() + kWaitNs;
            mbar_wait_until(bar + i, phase, deadline);
            if (NS == 2 && z + 1 < zb_end) mbar_wait_until(bar + (i ^ 1), (unsigned)((z + 1 - za) / NS) & 1u, deadline);
            return;
        }
        if (fix) {
            src.fix(st, x0, y0, nx, ny, rows + 2 * R);
            __syncthreads();
        }
        if (xrow) {
            V acc[NP][8];
#pragma unroll
            for (int p = 0; p < NP; ++p)
#pragma unroll
                for (int i = 0; i < 8; ++i) acc[p][i] = V{};
            // each input feeds the outputs it contributes to: output i takes taps 0 .. T-1 in order
            src.window(st, row, xo, [&](int j, const V *v) {
#pragma unroll
                for (int i = 0; i < 8; ++i)
                    if (j - i >= 0 && j - i < T)
#pragma unroll
                        for (int p = 0; p < NP; ++p) acc[p][i] = tap_fma(t.g[j - i], v[p], acc[p][i]);
            });
            if constexpr (sizeof(V) == 4) {
                float4 *dst = reinterpret_cast<float4 *>(xc + row * XS + xo);
                dst[0] = make_float4(acc[0][0], acc[0][1], acc[0][2], acc[0][3]);
                dst[1] = make_float4(acc[0][4], acc[0][5], acc[0][6], acc[0][7]);
            } else if constexpr (NP == 1) {
                float4 *dst = reinterpret_cast<float4 *>(xc + row * XS + xo);
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    dst[i] = make_float4(acc[0][2 * i].x, acc[0][2 * i].y, acc[0][2 * i + 1].x, acc[0][2 * i + 1].y);
            } else {
                float4 *dst = reinterpret_cast<float4 *>(xc) + row * XS + xo;
#pragma unroll
                for (int i = 0; i < 8; ++i)
                    dst[i] = make_float4(acc[0][i].x, acc[0][i].y, acc[NP - 1][i].x, acc[NP - 1][i].y);
            }
        }
        __syncthreads();  // the staging buffer is read, the rows complete
        if (threadIdx.x == 0 && z + NS < zb_end) {
            fence_proxy_async_smem();
            src.issue(st, x0, y0, z + NS, xy_box_rows<R>(ny), bar + i, G.fault_tx);
        }
        if (yrow) {
            V res[YT][NP];
#pragma unroll
            for (int i = 0; i < YT; ++i)
#pragma unroll
                for (int p = 0; p < NP; ++p) res[i][p] = V{};
#pragma unroll
            for (int j = 0; j < YT + 2 * R; ++j) {
                V v[NP];
                if constexpr (NP == 1) {
                    v[0] = xc[(yr + j) * XS + lane];
                } else {
                    const float4 w = reinterpret_cast<const float4 *>(xc)[(yr + j) * XS + lane];
                    v[0] = make_float2(w.x, w.y);
                    v[NP - 1] = make_float2(w.z, w.w);
                }
#pragma unroll
                for (int i = 0; i < YT; ++i)
                    if (j - i >= 0 && j - i < T)
#pragma unroll
                        for (int p = 0; p < NP; ++p) res[i][p] = tap_fma(t.g[j - i], v[p], res[i][p]);
            }
            if (col) {
#pragma unroll
                for (int i = 0; i < YT; ++i) {
                    if (yr + i < rows) {
                        V *d = o + (long long)(i * out.px) * NP;
                        if constexpr (NP == 1)
                            *d = res[i][0];
                        else
                            *reinterpret_cast<float4 *>(d) =
                                make_float4(res[i][0].x, res[i][0].y, res[i][NP - 1].x, res[i][NP - 1].y);
                    }
                }
            }
        }
        o += out.pplane * NP;
        __syncthreads();  // the next plane's x phase rewrites the rows
    }
    if (threadIdx.x == 0)
        for (int i = 0; i < NS; ++i) mbar_inval(bar + i);
}

// CTA -> (brick, tile) for the x/y kernels: tiles (tx, ty, tz) of 32 x TH x B.xyp.
struct XYTile {
    int x0, y0, za;
};
template <int R>
__device__ __forceinline__ XYTile xy_tile_of(int local, const BrickDev &B) {
    const int ntx = (B.nx + kXYT - 1) / kXYT, nty = (B.ny + XYG<R>::TH - 1) / XYG<R>::TH;
    const int tx = local % ntx, r = local / ntx;
    return XYTile{tx * kXYT, (r % nty) * XYG<R>::TH, (r / nty) * B.xyp};
}

// Group A's x/y kernel: (H I~, H) into B.u2 (Li's form, NP = 1), or both sides of Eq. (10),
// ((H I~, H), ((1-H) I~, 1-H)) interleaved per voxel (the Eq. (15) form, NP = 2).
template <int R, class ImgT, int NP, bool EX = false>
__global__ void __launch_bounds__(kXYThreads, (SrcH<R, ImgT, NP, EX>::CTAS)) k_ta_xy(GroupArgs G, TapPairs t) {
    extern __shared__ __align__(128) unsigned char xsm[];
    dependents_may_start();
    const int b = find_brick(G.starts, G.nb, blockIdx.x);
    const BrickDev &B = G.bricks[b];
    const XYTile tl = xy_tile_of<R>(blockIdx.x - __ldg(G.starts + b), B);
    const SrcH<R, ImgT, NP, EX> src{&B.tm_q, &B.tm_img, EX ? 1.f : B.cs[1], EX ? 0.f : -B.cs[0] * B.cs[1]};
    const OutXY out{reinterpret_cast<float *>(B.u2), B.up, (long long)B.up * B.ny};
    xy_tile<R>(G, src, out, B.nx, B.ny, B.nz, tl.x0, tl.y0, tl.za, B.xyp, t, xsm);
}

// Group B's x/y kernel: (a, b) into B.abxy.
template <int R, class S>
__global__ void __launch_bounds__(kXYThreads, (SrcAB<R, S>::CTAS)) k_tb_xy(GroupArgs G, TapPairs t) {
    extern __shared__ __align__(128) unsigned char xsm[];
    dependents_may_start();
    const int b = find_brick(G.starts, G.nb, blockIdx.x);
    const BrickDev &B = G.bricks[b];
    const XYTile tl = xy_tile_of<R>(blockIdx.x - __ldg(G.starts + b), B);
    const SrcAB<R, S> src{&B.tm_ab};
    const OutXY out{reinterpret_cast<float *>(B.abxy), B.px, (long long)B.px * B.ny};
    xy_tile<R>(G, src, out, B.nx, B.ny, B.nz, tl.x0, tl.y0, tl.za, B.xyp, t, xsm);
}

// ------------------------------------------------------------------ A: z

// x-z slabs: 32 columns of one y row and kAZT output planes (plus the R-plane
// halos) of the x/y-convolved pair (H I~, H), and the kAZT planes of K*I~ the
// slab's outputs use.  A persistent CTA walks the slabs of the launch
// (consecutive slabs are consecutive z ranges of one row, so shared halos hit
// L2) with a two-stage shared-memory buffer: the TMA boxes of the next slab
// are in flight while the current one is convolved.  Planes outside the brick
// and columns past nx arrive as zeros.
template <int R>
constexpr int az_stage() { return (kAZT + 2 * R) * 32 + kAZT * 16; }  // float2 units per stage
template <int R>
constexpr size_t az_smem() { return 2 * sizeof(float2) * az_stage<R>() + 2 * sizeof(uint64_t); }  // + barriers

__device__ __forceinline__ void cp_async8(void *dst, const void *src, bool valid) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;\n" ::"r"(d), "l"(src), "r"(valid ? 8 : 0) : "memory");
}
__device__ __forceinline__ void cp_async4(void *dst, const void *src, bool valid) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;\n" ::"r"(d), "l"(src), "r"(valid ? 4 : 0) : "memory");
}
__device__ __forceinline__ void cp_async16(void *dst, const void *src, bool valid) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(d), "l"(src), "r"(valid ? 16 : 0) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait1() { asm volatile("cp.async.wait_group 1;\n" ::: "memory"); }


struct AZSlabId {
    int b, x0, y, z0;
};
// n / d and n % d for n >= 0, d > 0.  Below 2^24 a float quotient, off by at
// most one, corrected once; larger n (very thin bricks only) divide exactly.
__device__ __forceinline__ int divmod24(int n, int d, float inv_d, int &rem) {
    if (n >= (1 << 24)) {
        const int q = n / d;
        rem = n - q * d;
        return q;
    }
    int q = __float2int_rz((float)n * inv_d);
    int r = n - q * d;
    if (r < 0) { --q; r += d; } else if (r >= d) { ++q; r -= d; }
    rem = r;
    return q;
}
__device__ __forceinline__ AZSlabId az_slab_of(const GroupArgs &G, int slab) {
    const int b = find_brick(G.starts, G.nb, slab);
    const BrickDev &B = G.bricks[b];
    const int local = slab - __ldg(G.starts + b);
    const int nzt = (B.nz + kAZT - 1) / kAZT, nxt = (B.nx + 31) / 32;
    int zt, xt;
    const int rest = divmod24(local, nzt, __frcp_rn((float)nzt), zt);
    const int y = divmod24(rest, nxt, __frcp_rn((float)nxt), xt);
    return AZSlabId{b, xt * 32, y, zt * kAZT};
}

// The persistent slab walk of group A's z kernels: each CTA takes the slabs
// blockIdx.x, blockIdx.x + gridDim.x, ... of the launch through two stage
// buffers of STAGE_BYTES in dynamic shared memory, followed by one mbarrier per
// stage.  Thread 0 issues a slab's TMA copies (issue(id, buf, bar)) one slab
// ahead, into the stage the previous slab left; every thread waits for its
// stage's barrier, then body(id, buf) convolves the slab.  The last argument of
// issue asks it to fence the brick's tensor maps (first slab of each brick).  A wait that runs out
// (kWaitNs) is reported in the group's error word; the CTA then gives the copies
// still in flight the same time to land and returns.
template <int STAGE_BYTES, class Issue, class Body>
__device__ __forceinline__ void az_walk(const GroupArgs &G, unsigned char *smem, const Issue &issue,
                                        const Body &body) {
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem + 2 * STAGE_BYTES);
    if (smem_addr(smem) % 128u != 0u) {  // the copies' destinations must be 128-byte aligned
        report_error(G.err, kErrSmemAlign);
        return;
    }
    dependents_may_start();
    const int total = __ldg(G.starts + G.nb);
    if (threadIdx.x == 0) {
        mbar_init(bars, 1);
        mbar_init(bars + 1, 1);
        mbar_init_fence();
    }
    __syncthreads();
    wait_for_previous();
    unsigned phase = 0u, pending = 0u;  // bit s: parity of stage s's next phase; stage s awaits copies
    AZSlabId next{};
    int last_b = -1;  // thread 0: the brick whose maps it fenced last
    if ((int)blockIdx.x < total) {
        next = az_slab_of(G, blockIdx.x);
        if (threadIdx.x == 0) {
            issue(next, smem, bars, true);
            last_b = next.b;
        }
        pending = 1u;
    }
    int stage = 0;
    bool ok = true;
    for (int sl = blockIdx.x; sl < total; sl += gridDim.x) {
        const AZSlabId id = next;
        if (sl + (int)gridDim.x < total) {
            next = az_slab_of(G, sl + gridDim.x);
            if (threadIdx.x == 0) {
                fence_proxy_async_smem();  // the reads of that stage (before the last barrier) come first
                issue(next, smem + (stage ^ 1) * STAGE_BYTES, bars + (stage ^ 1), next.b != last_b);
                last_b = next.b;
            }
            pending |= 1u << (stage ^ 1);
        }
        if (!mbar_wait(bars + stage, (phase >> stage) & 1u)) {
            ok = false;
            break;
        }
        phase ^= 1u << stage;
        pending &= ~(1u << stage);
        body(id, smem + stage * STAGE_BYTES);
        __syncthreads();  // this stage is refilled by the next iteration's copies
        stage ^= 1;
    }
    if (!ok) {
        report_error(G.err, kErrWaitExpired);
        const unsigned long long deadline = globaltimer_ns() + kWaitNs;
        for (int s = 0; s < 2; ++s)
            if ((pending >> s) & 1u) mbar_wait_until(bars + s, (phase >> s) & 1u, deadline);
        return;
    }
    if (threadIdx.x == 0) {
        mbar_inval(bars);
        mbar_inval(bars + 1);
    }
}

template <int R, class S>
__global__ void __launch_bounds__(kAZThreads, kAZCtas) k_ta_z(GroupArgs G, TapPairs t) {
    constexpr int T = 2 * R + 1;
    constexpr int ROWS = kAZT + 2 * R;
    constexpr int WIN = kAZO + 2 * R;
    constexpr int STAGE_BYTES = (int)sizeof(float2) * az_stage<R>();
    using V2 = typename Store<S>::V2;
    // [2 stages]{[ROWS][32] pairs, [kAZT][32] K*I~}, then the two barriers
    extern __shared__ __align__(128) unsigned char az_sm[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // the slab's boxes: ROWS planes of the pair field from plane z0 - R, kAZT planes of K*I~
    // from z0 (planes outside the brick and columns past nx arrive as zeros)
    const auto issue = [&](const AZSlabId &id, unsigned char *buf, uint64_t *bar, bool fence) {
        const BrickDev &B = G.bricks[id.b];
        if (fence) {
            fence_tensormap(&B.tm_u);
            fence_tensormap(&B.tm_k);
        }
        mbar_arrive_expect_tx(bar, (unsigned)STAGE_BYTES + G.fault_tx);
        tma_load_3d(buf, &B.tm_u, 2 * id.x0, id.y, id.z0 - R, bar);
        tma_load_3d(buf + ROWS * 32 * sizeof(float2), &B.tm_k, id.x0, id.y, id.z0, bar);
    };
    const auto body = [&](const AZSlabId &id, const unsigned char *sbuf) {
        const float2 *buf = reinterpret_cast<const float2 *>(sbuf);
        const BrickDev &B = G.bricks[id.b];
        const int x = id.x0 + lane;
        const int zb = warp * kAZO;
        const int bnx = B.nx, bny = B.ny, bnz = B.nz;  // read once: the stores below might alias B
        if (x >= bnx) return;
        const float l1 = B.lambda1, l2 = B.lambda2;
        // each plane read feeds the outputs it contributes to (output o takes taps 0 .. T-1 in
        // order): eight accumulators instead of a window of 8 + 2R planes in registers, so that
        // three CTAs share an SM at every radius (two above radius 6 with the window: 512 x 448
        // x 320 at radius 10 0.291 -> 0.259 ms, 112 M voxels of bricks at radius 8 0.555 -> 0.497;
        // 512^3 at radius 6 0.446 -> 0.435 ms, 0.91 of the HBM rate; with four CTAs 0.462)
        float2 sum[kAZO];  // (K*(H I~), K*H)
#pragma unroll
        for (int o = 0; o < kAZO; ++o) sum[o] = make_float2(0.f, 0.f);
#pragma unroll
        for (int j = 0; j < WIN; ++j) {
            const float2 w = buf[(zb + j) * 32 + lane];
#pragma unroll
            for (int o = 0; o < kAZO; ++o)
                if (j - o >= 0 && j - o < T) sum[o] = f2fma(t.g[j - o], w, sum[o]);
        }
        const long long pplane = (long long)B.px * bny;
        const long long off = (long long)(id.z0 + zb) * pplane + (long long)id.y * B.px + x;
        V2 *ab = reinterpret_cast<V2 *>(B.ab) + off;
        const float *ki = reinterpret_cast<const float *>(buf + ROWS * 32) + zb * 32 + lane;
        const float kxy = __ldg(B.prof + x) * __ldg(B.prof + bnx + id.y);
        float2 res = make_float2(0.f, 0.f);  // rounding residual carried along z (16-bit storage)
        const float *pz = B.prof + bnx + bny + id.z0 + zb;
        float *const dump = B.dump;
#pragma unroll
        for (int o = 0; o < kAZO; ++o) {
            const int zo = id.z0 + zb + o;
            if (zo < bnz) {
                const float2 acc = sum[o];
                const float f1 = __fdividef(acc.x, acc.y);
                // K*(1-H) = K*1 - K*H keeps few significant bits once 1-H < ~1e-6 over the
                // whole window (phi > ~3e5 there, delta < 4e-12); the fit is then taken as
                // f1, the window mean in that limit, so that it stays finite
                const float k1 = kxy * __ldg(pz + o), den = k1 - acc.y;
                const float f2 = den > 0x1p-20f * k1 ? __fdividef(ki[o * 32] - acc.x, den) : f1;
                const float2 v = make_float2(l1 * f1 - l2 * f2, l1 * (f1 * f1) - l2 * (f2 * f2));
                if constexpr (std::is_same<S, float>::value) {
                    *ab = v;
                } else {
                    // 16-bit storage: the rounding residual of each plane is carried into the
                    // next plane of the column before it is rounded (first-order noise
                    // shaping along z), so that the stored field's rounding error is a
                    // difference of neighbours, which the Gaussian of group B averages out
                    const float2 want = make_float2(v.x + res.x, v.y + res.y);
                    const V2 st = Store<S>::pack2(want);
                    const float2 got = Store<S>::unpack2(st);
                    res = make_float2(want.x - got.x, want.y - got.y);
                    *ab = st;
                }
                ab += pplane;
                if (dump) {
                    const long long q = (long long)zo * B.nx * B.ny + (long long)id.y * B.nx + x;
                    const long long n = (long long)B.nx * B.ny * B.nz;
                    dump[q] = f1 * B.cs[3] + B.cs[0];
                    dump[n + q] = f2 * B.cs[3] + B.cs[0];
                }
            }
        }
    };
    az_walk<STAGE_BYTES>(G, az_sm, issue, body);
}

// The z pass of the Eq. (15) form: the same x-z slabs and persistent walk,
// over the four x/y-convolved fields ((H I~, H), ((1-H) I~, 1-H)) staged as
// one float4 per row and column; writes the fits f1 = K*(H I~)/K*H and
// f2 = K*((1-H) I~)/K*(1-H) (Eq. 6, both sides convolved directly) in FP32
// to B.abxy, where the update kernel forms (I~ - f_i)^2 (Eq. 15, sigma_2 = 0).
template <int R>
constexpr int az4_stage() { return (kAZT + 2 * R) * 32; }  // float4 units per stage
template <int R>
constexpr size_t az4_smem() { return 2 * sizeof(float4) * az4_stage<R>() + 2 * sizeof(uint64_t); }  // + barriers

// AB: the exact arithmetic of Li's form, IEEE divisions and a = l1 f1 - l2 f2,
// b = l1 f1^2 - l2 f2^2 to B.ab instead of the fits.
template <int R, bool AB = false>
__global__ void __launch_bounds__(kAZThreads, 2) k_ta_z4(GroupArgs G, TapPairs t) {
    constexpr int T = 2 * R + 1;
    constexpr int WIN = kAZO + 2 * R;
    constexpr int STAGE_BYTES = (int)sizeof(float4) * az4_stage<R>();
    extern __shared__ __align__(128) unsigned char az_sm[];  // [2 stages][ROWS][32] float4, then the barriers
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // the slab's box: ROWS planes of the four fields from plane z0 - R (planes outside the
    // brick and columns past nx arrive as zeros)
    const auto issue = [&](const AZSlabId &id, unsigned char *buf, uint64_t *bar, bool fence) {
        const CUtensorMap *map = &G.bricks[id.b].tm_u;
        if (fence) fence_tensormap(map);
        mbar_arrive_expect_tx(bar, (unsigned)STAGE_BYTES + G.fault_tx);
        tma_load_3d(buf, map, 4 * id.x0, id.y, id.z0 - R, bar);
    };
    const auto body = [&](const AZSlabId &id, const unsigned char *sbuf) {
        const float4 *buf = reinterpret_cast<const float4 *>(sbuf);
        const BrickDev &B = G.bricks[id.b];
        const int x = id.x0 + lane;
        const int zb = warp * kAZO;
        if (x >= B.nx) return;
        float2 acc[2][kAZO];  // (K*(H I~), K*H), (K*((1-H) I~), K*(1-H))
#pragma unroll
        for (int o = 0; o < kAZO; ++o) acc[0][o] = acc[1][o] = make_float2(0.f, 0.f);
#pragma unroll
        for (int j = 0; j < WIN; ++j) {  // as in k_ta_z, both pairs in one 16-byte read
            const float4 w = buf[(zb + j) * 32 + lane];
#pragma unroll
            for (int o = 0; o < kAZO; ++o)
                if (j - o >= 0 && j - o < T) {
                    acc[0][o] = f2fma(t.g[j - o], make_float2(w.x, w.y), acc[0][o]);
                    acc[1][o] = f2fma(t.g[j - o], make_float2(w.z, w.w), acc[1][o]);
                }
        }
        const long long pplane = (long long)B.px * B.ny;
        const long long off = (long long)(id.z0 + zb) * pplane + (long long)id.y * B.px + x;
        float2 *fits = (AB ? reinterpret_cast<float2 *>(B.ab) : B.abxy) + off;
        const float l1 = B.lambda1, l2 = B.lambda2;
        const int bnz = B.nz;
        float *const dump = B.dump;
#pragma unroll
        for (int o = 0; o < kAZO; ++o) {
            const int zo = id.z0 + zb + o;
            if (zo < bnz) {
                float f1, f2;
                if constexpr (AB) {
                    f1 = acc[0][o].x / acc[0][o].y;
                    f2 = acc[1][o].x / acc[1][o].y;
                    *fits = make_float2(l1 * f1 - l2 * f2, l1 * (f1 * f1) - l2 * (f2 * f2));
                } else {
                    f1 = __fdividef(acc[0][o].x, acc[0][o].y);
                    f2 = __fdividef(acc[1][o].x, acc[1][o].y);
                    *fits = make_float2(f1, f2);
                }
                fits += pplane;
                if (dump) {
                    const long long q = (long long)zo * B.nx * B.ny + (long long)id.y * B.nx + x;
                    const long long n = (long long)B.nx * B.ny * B.nz;
                    dump[q] = f1 * B.cs[3] + B.cs[0];
                    dump[n + q] = f2 * B.cs[3] + B.cs[0];
                }
            }
        }
    };
    az_walk<STAGE_BYTES>(G, az_sm, issue, body);
}

// ------------------------------------------------------- set-up: K*I~

// K*I~ of a group's bricks, once per solve: the x/y kernel on I~ into b.abxy, one float per
// voxel in rows of 2 px (the first px used), then the z convolution into b.ki by the slab walk
// of group A: the pair field's map and boxes, read as two adjacent columns per lane (slabs of 64
// columns: those of odd x tiles are empty).  The Li form alone runs it: the others' maps have
// other boxes.  z pass, from global memory with a window in registers before: 512^3 radius 6
// 0.32 -> 0.211 ms, 0.8 of the measured copy rate.
template <int R, class ImgT>
__global__ void __launch_bounds__(kXYThreads, 4) k_ki_xy(GroupArgs G, TapPairs t) {
    extern __shared__ __align__(128) unsigned char xsm[];
    const int b = find_brick(G.starts, G.nb, blockIdx.x);
    const BrickDev &B = G.bricks[b];
    const XYTile tl = xy_tile_of<R>(blockIdx.x - __ldg(G.starts + b), B);
    const SrcI<R, ImgT> src{&B.tm_img, B.cs[1], -B.cs[0] * B.cs[1], tl.x0, tl.y0, B.nx, B.ny};
    const OutXY out{reinterpret_cast<float *>(B.abxy), 2 * B.px, 2LL * B.px * B.ny};
    xy_tile<R>(G, src, out, B.nx, B.ny, B.nz, tl.x0, tl.y0, tl.za, B.xyp, t, xsm);
}

template <int R>
constexpr size_t ki_smem() { return 2 * sizeof(float2) * (kAZT + 2 * R) * 32 + 2 * sizeof(uint64_t); }
template <int R>
__global__ void __launch_bounds__(kAZThreads, kAZCtas) k_ki_z(GroupArgs G, TapPairs t) {
    constexpr int T = 2 * R + 1;
    constexpr int STAGE_BYTES = (int)sizeof(float2) * (kAZT + 2 * R) * 32;
    extern __shared__ __align__(128) unsigned char az_sm[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const auto issue = [&](const AZSlabId &id, unsigned char *buf, uint64_t *bar, bool fence) {
        const CUtensorMap *map = &G.bricks[id.b].tm_u;
        if (fence) fence_tensormap(map);
        const bool some = id.x0 % 64 == 0;
        mbar_arrive_expect_tx(bar, (some ? (unsigned)STAGE_BYTES : 0u) + G.fault_tx);
        if (some) tma_load_3d(buf, map, id.x0, id.y, id.z0 - R, bar);
    };
    const auto body = [&](const AZSlabId &id, const unsigned char *sbuf) {
        const float2 *buf = reinterpret_cast<const float2 *>(sbuf);
        const BrickDev &B = G.bricks[id.b];
        const int x = id.x0 + 2 * lane, zb = warp * kAZO, nx = B.nx, nz = B.nz;
        if (id.x0 % 64 != 0 || x >= nx) return;
        float2 sum[kAZO];
#pragma unroll
        for (int o = 0; o < kAZO; ++o) sum[o] = make_float2(0.f, 0.f);
#pragma unroll
        for (int j = 0; j < kAZO + 2 * R; ++j) {
            const float2 w = buf[(zb + j) * 32 + lane];
#pragma unroll
            for (int o = 0; o < kAZO; ++o)
                if (j - o >= 0 && j - o < T) sum[o] = f2fma(t.g[j - o], w, sum[o]);
        }
        const long long pplane = (long long)B.px * B.ny;
        float *ki = B.ki + (long long)(id.z0 + zb) * pplane + (long long)id.y * B.px + x;
#pragma unroll
        for (int o = 0; o < kAZO; ++o) {
            if (id.z0 + zb + o < nz) {
                if (x + 1 < nx)
                    *reinterpret_cast<float2 *>(ki) = sum[o];
                else
                    *ki = sum[o].x;
            }
            ki += pplane;
        }
    };
    az_walk<STAGE_BYTES>(G, az_sm, issue, body);
}

// ------------------------------------------------------------------ B: z

// q = +-atan(eps/|u|)/pi (the small side of H, sign of u) with the atan
// argument kept in [0, 1]: atan(m/M) for m = min(|u|, eps), M = max(|u|, eps),
// and for |u| < eps, atan(eps/|u|) = pi/2 - atan(|u|/eps).  atan(x)/pi on
// [0, 1] is x P(x^2), P the degree-8 minimax polynomial of relative error
// (coefficients by Lawson's algorithm, atan_poly.py), 1.5e-7 relative in FP32.
// P's coefficients, highest power first (Horner order).
__device__ constexpr float kAtanPi[9] = {9.071480017e-04f, -5.114803091e-03f, 1.358913258e-02f, -2.388691157e-02f,
                              3.387114406e-02f, -4.521160573e-02f, 6.363848597e-02f, -1.061024666e-01f,
                              3.183098733e-01f};
__device__ __forceinline__ float atan01_pi(float x) {
    const float t = x * x;
    float p = kAtanPi[0];
#pragma unroll
    for (int k = 1; k < 9; ++k) p = fmaf(p, t, kAtanPi[k]);
    return x * p;
}
__device__ __forceinline__ float heaviside_q_fast(float u, float eps) {
    const float a = fabsf(u);
    const float at = atan01_pi(fminf(a, eps) * rcp_approx(fmaxf(a, eps)));
    return copysignf(a >= eps ? at : 0.5f - at, u);
}

// Packed f32x2 arithmetic (IEEE round-to-nearest per lane) for two planes at once.
__device__ __forceinline__ float2 f2v(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 f2add(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 f2mul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 f2sub(float2 a, float2 b) { return __ffma2_rn(b, make_float2(-1.f, -1.f), a); }

// heaviside_q_fast of two values with packed arithmetic: per lane the same
// operations in the same order (the ratio, the polynomial, 1/2 - at), so each
// lane equals the scalar function bit for bit.
__device__ __forceinline__ float2 heaviside_q_fast2(float2 u, float eps) {
    const float ax = fabsf(u.x), ay = fabsf(u.y);
    const float2 x = f2mul(make_float2(fminf(ax, eps), fminf(ay, eps)),
                           make_float2(rcp_approx(fmaxf(ax, eps)), rcp_approx(fmaxf(ay, eps))));
    const float2 t = f2mul(x, x);
    float2 p = f2v(kAtanPi[0]);
#pragma unroll
    for (int k = 1; k < 9; ++k) p = __ffma2_rn(p, t, f2v(kAtanPi[k]));
    const float2 at = f2mul(x, p);
    const float2 lo = f2sub(f2v(0.5f), at);
    return make_float2(copysignf(ax >= eps ? at.x : lo.x, u.x), copysignf(ay >= eps ? at.y : lo.y, u.y));
}

// z march over a column tile of one brick: 32 columns x tbz_rows(R) rows, z chunk
// [z0, z0 + zc), two output planes per step.  Planes are numbered relative to the
// chunk start (r = z - z0).
//
// What bounds it: instruction issue first (an earlier form, one column per thread with
// the three normal components of the whole tile in shared memory, issued 204 thread
// instructions per voxel and ran at 0.42 of the HBM rate), the shared-memory pipe next.
// So a thread owns two adjacent columns (x, x + 1): loads, stores and shared-memory
// accesses are 8 or 16 bytes, the pair is one packed f32x2 operand, and what only its
// own columns need stays in registers: phi along z, the z component of the unit
// normal, the in-plane part of the Laplacian (formed from the neighbours the gradient
// has loaded anyway) and of the curvature.  Shared memory passes to the neighbours only
// phi, n_x and n_y.  A warp covers two rows of 16 pairs; one more warp marches the
// rows above and below the tile (for their n_y), the columns left and right of it (for
// their n_x) and loads phi's halo.
//
// Step k, outputs r0 = 2k and r0 + 1:
//   unit normals of planes r0 + 1, r0 + 2 from phi planes r0 .. r0 + 3; n_x and n_y into
//   one of two buffers; wait for the copies issued two steps ago; barrier; issue phi
//   planes r0 + 9, r0 + 10 (cp.async) into the ring slots of r0 + 1, r0 + 2; the
//   neighbours' n_x, n_y; outputs.
// The step k = -1 only brings the march up (normals of planes -1 and 0).
// Every second step convolves (a, b) along z for four planes at once: the thread's own
// 2R + 4 planes are in a shared-memory ring that no other thread reads (16 bytes per
// plane: both columns' pair; cp.async, no barrier), so each 16-byte read serves four
// planes and no radius needs its planes in registers.  The four planes it frees are
// refilled at once, two steps before their use.  The ring's slots are compile-time
// constants in M / 4 copies of the convolution alone (a uniform branch picks the copy);
// the rest of a step is one piece of code.
//
// Tile rows: two CTAs' rings fit an SM's shared memory; 14 rows make eight warps, two on
// each of the SM's quarters, at 128 registers (nine warps are held to 96, and spilled).  The
// exact arithmetic takes 10 rows, six warps at up to 168 registers: nothing spills, so that
// rsf_evolve_noalloc's launches need no local memory.
//
// Finite differences use reflect-101 for phi (the copies read the mirrored voxel) and
// for the normal (the reads of n_x, n_y at the first and last column or row take the
// neighbour on the other side, n_z likewise along z).
//
// 512^3, uint16, per launch: radius 6 1.034 -> 0.726 ms, 448 x 512 x 320 radius 10 0.663 -> 0.467 ms;
// 500^3 uint8, Eq. (15) form 0.906 -> 0.575 ms; 64^3 uint8 21.7 -> 9.1 us (its chunks split).
// At radius 6 it issues 117 thread instructions per voxel and reaches 0.60 of the HBM rate.
template <int R, bool EX>
constexpr int tbz_rows() { return R > 12 ? 8 : (R > 10 || EX ? 10 : (R > 8 ? 12 : 14)); }

template <int R, bool EX = false>
struct TBZ {
    static constexpr int TY = tbz_rows<R, EX>();
    static constexpr int NWC = TY / 2;                  // warps with outputs
    static constexpr int THREADS = (NWC + 1) * 32;
    static constexpr int M = (2 * R + 4 + 3) / 4 * 4;   // (a, b) planes in the ring
    static constexpr int PW = kZX + 4, PH = TY + 4;     // phi plane, halo 2: tile column c at c + 2
    static constexpr int PPL = PW * PH, NPHI = 8;
    static constexpr int NXP = kZX + 4, NYP = kZX, NH = TY + 2;  // n_x, n_y planes: rows -1 .. TY
    static constexpr int NPL = NH * (NXP + NYP);
    static constexpr int ABPL = NWC * 32;               // float4 per (a, b) plane
    static constexpr size_t bytes = sizeof(float4) * M * ABPL + sizeof(float) * (NPHI * PPL + 4 * NPL);
    static_assert(2 * TY <= 32, "one lane per column-halo site");
};
// f(0), f(1), ... with compile-time arguments
template <int... D, class F>
__device__ __forceinline__ void unroll(std::integer_sequence<int, D...>, const F &f) {
    (f(std::integral_constant<int, D>{}), ...);
}

__device__ __forceinline__ void cp_async_wait0() { asm volatile("cp.async.wait_group 0;\n" ::: "memory"); }
__device__ __forceinline__ float sqrt_approx_ftz(float x) {
    float y;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float2 ld2(const float *p) { return *reinterpret_cast<const float2 *>(p); }
// Read-only loads that stay where they are written (a plain load may be moved down to its
// use behind the barrier, where its latency shows), kept as loaded until that use: unpacking
// two 8- or 16-bit values beside the load would wait for it there.
__device__ __forceinline__ float ldg_now(const float *p) {
    float v;
    asm volatile("ld.global.nc.f32 %0, [%1];" : "=f"(v) : "l"(p));
    return v;
}
template <class ImgT> struct ImgPair;  // two columns' image values: both at once (even nx) or one by one
template <> struct ImgPair<float> {
    float a, b;
    __device__ __forceinline__ void load2(const float *p) {
        asm volatile("ld.global.nc.v2.f32 {%0, %1}, [%2];" : "=f"(a), "=f"(b) : "l"(p));
    }
    __device__ __forceinline__ void load_a(const float *p) { a = ldg_now(p); }
    __device__ __forceinline__ void load_b(const float *p) { b = ldg_now(p); }
    template <bool VEC> __device__ __forceinline__ float2 get() const { return make_float2(a, b); }
};
template <> struct ImgPair<uint8_t> {
    uint32_t a, b;
    __device__ __forceinline__ void load2(const uint8_t *p) {
        asm volatile("ld.global.nc.u16 %0, [%1];" : "=r"(a) : "l"(p));
    }
    __device__ __forceinline__ void load_a(const uint8_t *p) {
        asm volatile("ld.global.nc.u8 %0, [%1];" : "=r"(a) : "l"(p));
    }
    __device__ __forceinline__ void load_b(const uint8_t *p) {
        asm volatile("ld.global.nc.u8 %0, [%1];" : "=r"(b) : "l"(p));
    }
    template <bool VEC> __device__ __forceinline__ float2 get() const {
        return VEC ? make_float2((float)(a & 255u), (float)(a >> 8)) : make_float2((float)a, (float)b);
    }
};
template <> struct ImgPair<uint16_t> {
    uint32_t a, b;
    __device__ __forceinline__ void load2(const uint16_t *p) {
        asm volatile("ld.global.nc.u32 %0, [%1];" : "=r"(a) : "l"(p));
    }
    __device__ __forceinline__ void load_a(const uint16_t *p) {
        asm volatile("ld.global.nc.u16 %0, [%1];" : "=r"(a) : "l"(p));
    }
    __device__ __forceinline__ void load_b(const uint16_t *p) {
        asm volatile("ld.global.nc.u16 %0, [%1];" : "=r"(b) : "l"(p));
    }
    template <bool VEC> __device__ __forceinline__ float2 get() const {
        return VEC ? make_float2((float)(a & 0xffffu), (float)(a >> 16)) : make_float2((float)a, (float)b);
    }
};

// Unit normal of two columns from their differences; the central differences' factor
// 1/2 cancels: d / (|d| + 2e-10) = (d/2) / (|d/2| + 1e-10).  (Where |d|^2 is denormal,
// 2e-10 + |d| rounds to 2e-10 whether or not the square root flushes it.)  `first_x`
// takes the sum of squares as z + (x + [y]) instead of z + (y + [x]), [.] rounded alone.
__device__ __forceinline__ void unit_normal2(float2 gx, float2 gy, float2 gz, bool first_x, float2 &nx, float2 &ny,
                                             float2 &nz) {
    float2 ss = __ffma2_rn(gy, gy, f2mul(gx, gx));
    if (first_x) ss = __ffma2_rn(gx, gx, f2mul(gy, gy));
    ss = __ffma2_rn(gz, gz, ss);
    const float2 r = f2add(make_float2(sqrt_approx_ftz(ss.x), sqrt_approx_ftz(ss.y)), f2v(2e-10f));
    const float2 inv = make_float2(rcp_approx(r.x), rcp_approx(r.y));
    nx = f2mul(gx, inv);
    ny = f2mul(gy, inv);
    nz = f2mul(gz, inv);
}

// The same by IEEE operations (the exact arithmetic).
__device__ __forceinline__ float unit_normal_exact(float gx, float gy, float gz, float &hx, float &hy, float &hz) {
    hx = gx * 0.5f;
    hy = gy * 0.5f;
    hz = gz * 0.5f;
    return sqrtf(hx * hx + hy * hy + hz * hz) + 1e-10f;
}
template <bool EX>
__device__ __forceinline__ void normal2(float2 gx, float2 gy, float2 gz, bool first_x, float2 &nx, float2 &ny,
                                        float2 &nz) {
    if constexpr (EX) {
        float2 hx, hy, hz;
        const float m0 = unit_normal_exact(gx.x, gy.x, gz.x, hx.x, hy.x, hz.x);
        const float m1 = unit_normal_exact(gx.y, gy.y, gz.y, hx.y, hy.y, hz.y);
        nx = make_float2(hx.x / m0, hx.y / m1);
        ny = make_float2(hy.x / m0, hy.y / m1);
        nz = make_float2(hz.x / m0, hz.y / m1);
    } else {
        unit_normal2(gx, gy, gz, first_x, nx, ny, nz);
    }
}
// Data term and update of one column in the exact arithmetic, rounded as the compiler
// contracts UpdateEpi of rsf_passes.cu.
__device__ __forceinline__ float update_exact(float ph, float lap, float kap, float im, float K1, float Ka, float Kb,
                                              float s2, const Coeffs &c, float &g) {
    const float X = (c.lambda1 - c.lambda2) * K1, im2 = __fmul_rn(im, im);
    g = s2 * (fmaf(X, im2, -__fmul_rn(2.f * im, Ka)) + Kb);
    const float del = __fmul_rn(c.eps, INV_PI) / fmaf(ph, ph, __fmul_rn(c.eps, c.eps));
    const float f = fmaf(c.nu, kap, -g);
    return fmaf(c.dt, fmaf(c.mu, lap - kap, __fmul_rn(del, f)), ph);
}
// The small side of H with the sign of u (its zero too), by atanf and an IEEE division.
__device__ __forceinline__ float heaviside_q_exact(float u, float eps) {
    return copysignf(atanf(eps / fabsf(u)) * INV_PI, u);
}

// VEC: nx even and the image base aligned for two values, so that a thread's two
// columns are both inside or both outside the brick and are read and written together.
// DUMP: also write g, kappa and L of every output to B.dump (rsf_step_stages); a
// separate instantiation keeps the iteration's kernel free of it.
// EX: the exact arithmetic (IEEE divisions and square roots, atanf) on the centred FP32 image,
// whose rows have q's pitch.
template <int R, class ImgT, bool VEC, bool DUMP, bool EX>
__device__ __forceinline__ void tb_z_march(const GroupArgs &G, const BrickDev &B, int bi, const TapPairs &t) {
    using Z = TBZ<R, EX>;
    constexpr int TY = Z::TY, M = Z::M, PW = Z::PW, PPL = Z::PPL, NXP = Z::NXP, NYP = Z::NYP, NPL = Z::NPL;
    constexpr int T = 2 * R + 1;
    using Img2 = ImgPair<ImgT>;
    extern __shared__ __align__(16) float zsm[];
    float4 *const sab = reinterpret_cast<float4 *>(zsm);  // [M][ABPL]
    float *const sphi = zsm + 4 * M * Z::ABPL;            // [NPHI][PPL]
    float *const snx = sphi + Z::NPHI * PPL;              // [2 buffers][2 planes]{n_x [NH][NXP], n_y [NH][NYP]}

    const int local = blockIdx.x - __ldg(G.starts + bi);
    const int nx = B.nx, ny = B.ny, nz = B.nz;
    const int nbx = (nx + kZX - 1) / kZX, nby = (ny + TY - 1) / TY;
    const int bx = local % nbx, rr = local / nbx;
    const int x0 = bx * kZX, y0 = (rr % nby) * TY;
    const int zpart = rr / nby, parts = (B.zc + B.zs - 1) / B.zs;
    const int zch = zpart / parts * B.zc;                    // the z chunk of this CTA's planes
    const int z0 = zch + zpart % parts * B.zs;
    const int nout = min(min(z0 + B.zs, zch + B.zc), nz) - z0;
    if (nout <= 0) return;
    const unsigned plane = (unsigned)nx * (unsigned)ny;      // offsets within a field are 32-bit
    const int par = G.parity ^ B.flip;
    const float *phi = par ? B.phi[1] : B.phi[0];

    // this thread's pair of columns: rows 2 warp, 2 warp + 1 of the tile, or (halo warp) rows -1, TY
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const bool comp = warp < Z::NWC;
    const int hl = lane >> 4, c = 2 * (lane & 15);
    const int row = comp ? 2 * warp + hl : (hl ? TY : -1);
    const int x = x0 + c, y = y0 + row;
    const bool act0 = comp && x < nx && y < ny, act1 = comp && x + 1 < nx && y < ny;
    const auto refl_y = [&](int v) { return refl101(clampi(v, -2, ny + 1), ny); };
    const auto refl_x = [&](int v) { return refl101(clampi(v, -2, nx + 1), nx); };
    // offsets within a plane of the values copied for a pair: two adjacent ones (VEC: a pair
    // right of the last column is read from nx - 2, whose first value is the mirror of nx)
    struct PairOff { unsigned a, b; };
    const auto pair_off = [&](int yy) -> PairOff {
        const unsigned base = (unsigned)refl_y(yy) * (unsigned)nx;
        if constexpr (VEC) {
            const int xs = x < nx ? x : nx - 2;
            return PairOff{base + xs, base + xs + 1};
        } else {
            return PairOff{base + refl_x(x), base + refl_x(x + 1)};
        }
    };
    const auto copy_pair = [&](float *dst, unsigned zoff, const PairOff &o) {
        if constexpr (VEC) {
            cp_async8(dst, phi + (zoff + o.a), true);
        } else {
            cp_async4(dst, phi + (zoff + o.a), true);
            cp_async4(dst + 1, phi + (zoff + o.b), true);
        }
    };
    const PairOff own = pair_off(y);
    const int si = (row + 2) * PW + c + 2;  // own pair in a phi plane
    // halo warp: the rows -2 and TY + 1; one column site per lane (column -1 or 32) with
    // the column beyond it (-2 or 33); the four corners beside the rows -1 and TY
    const int row2 = hl ? TY + 1 : -2;
    const PairOff far_row = pair_off(y0 + row2);
    const int si2 = (row2 + 2) * PW + c + 2;
    const bool site = !comp && lane < 2 * TY;
    const int side = lane >= TY ? 1 : 0, srow = min(lane - side * TY, TY - 1);
    const int ss = (srow + 2) * PW + (side ? kZX + 2 : 1);       // the site in a phi plane
    const int sf = ss + (side ? 1 : -1);                         // the column beyond it
    const unsigned so = (unsigned)refl_y(y0 + srow) * (unsigned)nx;
    const unsigned site_off = so + refl_x(side ? x0 + kZX : x0 - 1), far_off = so + refl_x(side ? x0 + kZX + 1 : x0 - 2);
    const int crow = (lane & 2) ? TY : -1, ccol = (lane & 1) ? kZX : -1;
    const int sc = (crow + 2) * PW + ccol + 2;
    const unsigned corner_off = (unsigned)refl_y(y0 + crow) * (unsigned)nx + refl_x(x0 + ccol);

    // the phi plane at offset zoff of the field into a ring slot
    const auto copy_phi = [&](float *dst, unsigned zoff) {
        copy_pair(dst + si, zoff, own);
        if (!comp) {
            copy_pair(dst + si2, zoff, far_row);
            if (site) {
                cp_async4(dst + ss, phi + (zoff + site_off), true);
                cp_async4(dst + sf, phi + (zoff + far_off), true);
            }
            if (lane < 4) cp_async4(dst + sc, phi + (zoff + corner_off), true);
        }
    };
    // phi plane r (relative) into its ring slot (r - 1) mod 8; planes outside the brick are
    // the mirrored ones, planes past nout + 1 are never read
    const auto issue_phi = [&](int r) {
        if (r <= nout + 1)
            copy_phi(sphi + ((r + 7) & 7) * PPL, (unsigned)refl101(clampi(z0 + r, -2, nz + 1), nz) * plane);
    };
    // (a, b) planes r .. r + 3 of this thread's columns into its ring slots from `slot`; zero
    // outside the brick (the convolution's padding) and past the chunk.  IN: all inside
    const unsigned px = (unsigned)B.px, pplane = px * (unsigned)ny;
    const float2 *const abxy = B.abxy;
    const unsigned ab0 = (unsigned)min(y, ny - 1) * px + (unsigned)min(x, (int)px - 2);
    float4 *const myab = sab + threadIdx.x;
    const auto issue_ab = [&](auto in, int r, int slot) {
        constexpr bool IN = decltype(in)::value;
        if (!comp) return;
        unsigned off = ab0 + (unsigned)(z0 + r) * pplane;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const bool ok = act0 && (IN || ((unsigned)(z0 + r + j) < (unsigned)nz && r + j < nout + R));
            cp_async16(myab + (slot + j) * Z::ABPL, abxy + (IN || ok ? off : ab0), ok);
            off += pplane;
        }
    };

    // K*1 = p_x p_y p_z; with R = 0 (the Eq. (15) form, sigma_2 = 0) the data terms
    // take no convolution and K*1 is 1
    float2 pxy = make_float2(0.f, 0.f);
    if (R == 0) {
        pxy = f2v(1.f);
    } else if (comp && y < ny) {
        const float py = __ldg(B.prof + nx + y);
        if (act0) pxy.x = __ldg(B.prof + x) * py;
        if (act1) pxy.y = __ldg(B.prof + x + 1) * py;
    }
    const float *profz = B.prof + nx + ny + z0;
    const float l1 = B.lambda1, l2 = B.lambda2, s2 = B.cs[2];
    // the data term's constants folded: s^2 (l1 - l2) p_x p_y (times p_z per plane), -2 s^2, and
    // for the Eq. (15) form s^2 l1, s^2 l2
    const float2 cK = f2mul(f2v(s2 * (l1 - l2)), pxy);
    const float m2s2 = -2.f * s2, s2l1 = s2 * l1, s2l2 = s2 * l2;
    const float inv_s = B.cs[1], nms = -B.cs[0] * B.cs[1];
    const float eps = B.eps, eps2 = eps * eps;
    const float nu = B.nu, dt_mu = B.dt * B.mu, dt_eps_pi = B.dt * (eps * INV_PI);
    const Coeffs co{eps, l1, l2, nu, B.mu, B.dt};
    float *const dump = DUMP ? B.dump : nullptr;
    const long long n = (long long)plane * nz;
    const ImgT *const img = reinterpret_cast<const ImgT *>(B.img);
    float *const phi_out = par ? B.phi[0] : B.phi[1];
    float *const q_out = B.q;
    const unsigned qplane = (unsigned)B.qp * (unsigned)ny;  // q rows have a pitch of their own
    const unsigned out0 = (unsigned)z0 * plane + (unsigned)min(y, ny - 1) * (unsigned)nx + (unsigned)min(x, nx - 1);
    // the image of output plane r at this thread's columns (not read past the chunk)
    const auto img_at = [&](auto in, int r, unsigned off) -> Img2 {
        Img2 v{};
        if (decltype(in)::value || r < nout) {
            if constexpr (VEC) {
                if (act0) v.load2(img + off);
            } else {
                if (act0) v.load_a(img + off);
                if (act1) v.load_b(img + off + 1);
            }
        }
        return v;
    };
    const auto pz_at = [&](auto in, int r) -> float {
        return (R == 0 || (!decltype(in)::value && r >= nout)) ? 1.f : ldg_now(profz + r);
    };

    // reads of the neighbours' n_x, n_y: the mirrored one at the brick's faces
    const int nxi = (row + 1) * NXP + c + 2, nyi = (row + 1) * NYP + c;
    const int nxl = x == 0 ? nxi + 1 : nxi - 1;               // left of the first column
    const int nxr = x + 1 == nx - 1 ? nxi : nxi + 2;          // right of the second
    const bool lone = x == nx - 1;                            // the second column lies outside
    const int nyu = y == 0 ? nyi + NYP : nyi - NYP, nyd = y == ny - 1 ? nyi - NYP : nyi + NYP;
    const int sni = (srow + 1) * NXP + (side ? kZX + 2 : 1);  // the column site's n_x

    wait_for_previous();
    // prologue: phi planes -2 .. 5; (a, b) planes -R .. M - R - 1
    using Edge = std::integral_constant<bool, false>;
    using Inner = std::integral_constant<bool, true>;
#pragma unroll 1
    for (int r = -2; r <= 5; ++r) issue_phi(r);
    cp_async_commit();
#pragma unroll 1
    for (int j = 0; j < M; j += 4) issue_ab(Edge{}, j - R, j);
    cp_async_commit();
    cp_async_wait1();
    __syncthreads();

    float2 phm = f2v(0.f), ph0 = ld2(sphi + 5 * PPL + si), ph1 = ld2(sphi + 6 * PPL + si);
    float st0 = sphi[5 * PPL + ss], st1 = sphi[6 * PPL + ss];  // the column site's phi planes r0, r0 + 1
    float2 lxy0 = f2v(0.f), kxy0 = f2v(0.f), nzm = f2v(0.f), nz0 = f2v(0.f);
    float2 acc[4][2];         // (K*a, K*b) of four planes and both columns,
    Img2 raw[4];              // their image values
    float pzq[4];             // and p_z (two planes at each step instead: 7 % slower)
    unsigned out = out0;      // offset of the step's first output plane at this thread's columns,
    unsigned qout = (unsigned)z0 * qplane + (unsigned)min(y, ny - 1) * (unsigned)B.qp + (unsigned)min(x, nx - 1);  // and in q

    // taps k = -R .. R in order, as each plane of the ring is read once
    const auto convolve = [&](auto dc) {
        constexpr int SLOT = 4 * decltype(dc)::value;
#pragma unroll
        for (int p = 0; p < 4; ++p) acc[p][0] = acc[p][1] = f2v(0.f);
#pragma unroll
        for (int j = 0; j < 2 * R + 4; ++j) {
            const float4 v = myab[(SLOT + j) % M * Z::ABPL];
#pragma unroll
            for (int p = 0; p < 4; ++p)
                if (j - p >= 0 && j - p < T) {
                    acc[p][0] = f2fma(t.g[j - p], make_float2(v.x, v.y), acc[p][0]);
                    acc[p][1] = f2fma(t.g[j - p], make_float2(v.z, v.w), acc[p][1]);
                }
        }
    };
    // Which planes take the other association of the normal's sum of squares: the first four
    // of a z chunk (offsets -1 .. 2) and the brick's last plane at an odd offset.  Results
    // stay bit for bit what they were when these planes had code of their own, so that a
    // suspended run resumes to the same phi.
    const auto first_x = [&](int r) {
        const int o = z0 + r - zch;
        return o <= 2 || (z0 + r == nz - 1 && (o & 1));
    };

    // one step; OUT: -1 none, 0 / 1 outputs from acc planes 2 OUT, 2 OUT + 1; IN: the planes it
    // reads and brings in lie inside the chunk (no mirroring, no checks)
    const auto step = [&](const int k, auto out_c, auto in_c) {
        constexpr int OUT = decltype(out_c)::value;
        constexpr bool IN = decltype(in_c)::value;
        const int r0 = 2 * k;
        float *const pA = sphi + 2 * (k & 3) * PPL, *const pB = pA + PPL;  // planes r0 + 1, r0 + 2 (later r0 + 9, r0 + 10)
        const float *const pC = sphi + 2 * ((k + 1) & 3) * PPL;            // plane r0 + 3
        float *const nA = snx + (OUT == 0 ? 0 : 2) * NPL, *const nB = nA + NPL;
        if constexpr (OUT == 0) {  // used after the barrier
#pragma unroll
            for (int s = 0; s < 4; ++s) {
                raw[s] = img_at(in_c, r0 + s, EX ? qout + s * qplane : out + s * plane);
                pzq[s] = pz_at(in_c, r0 + s);
            }
        }
        const float2 ph2 = ld2(pB + si), ph3 = ld2(pC + si);
        float2 nx1, ny1, nz1, nx2, ny2, nz2, lxy1, lxy2;
        {
            const float2 xp = make_float2(ph1.y, pA[si + 2]), xm = make_float2(pA[si - 1], ph1.x);
            const float2 yp = ld2(pA + si + PW), ym = ld2(pA + si - PW);
            normal2<EX>(f2sub(xp, xm), f2sub(yp, ym), f2sub(ph2, ph0), !IN && first_x(r0 + 1), nx1, ny1, nz1);
            const float2 m2 = f2mul(f2v(-2.f), ph1);
            lxy1 = f2add(f2add(f2add(xp, xm), m2), f2add(f2add(yp, ym), m2));
        }
        {
            const float2 xp = make_float2(ph2.y, pB[si + 2]), xm = make_float2(pB[si - 1], ph2.x);
            const float2 yp = ld2(pB + si + PW), ym = ld2(pB + si - PW);
            normal2<EX>(f2sub(xp, xm), f2sub(yp, ym), f2sub(ph3, ph1), !IN && first_x(r0 + 2), nx2, ny2, nz2);
            const float2 m2 = f2mul(f2v(-2.f), ph2);
            lxy2 = f2add(f2add(f2add(xp, xm), m2), f2add(f2add(yp, ym), m2));
        }
        *reinterpret_cast<float2 *>(nA + nxi) = nx1;
        *reinterpret_cast<float2 *>(nA + Z::NH * NXP + nyi) = ny1;
        *reinterpret_cast<float2 *>(nB + nxi) = nx2;
        *reinterpret_cast<float2 *>(nB + Z::NH * NXP + nyi) = ny2;
        if (!comp) {  // the column sites: planes r0 + 1 and r0 + 2 as the two packed lanes
            const float st2 = pB[ss], st3 = pC[ss];
            if (site) {
                const float2 gx = f2sub(make_float2(pA[ss + 1], pB[ss + 1]), make_float2(pA[ss - 1], pB[ss - 1]));
                const float2 gy = f2sub(make_float2(pA[ss + PW], pB[ss + PW]), make_float2(pA[ss - PW], pB[ss - PW]));
                const float2 gz = f2sub(make_float2(st2, st3), make_float2(st0, st1));
                float2 a, b, d;
                normal2<EX>(gx, gy, gz, !IN && first_x(r0 + 1), a, b, d);
                nA[sni] = a.x;
                if (!IN && !EX) unit_normal2(gx, gy, gz, first_x(r0 + 2), a, b, d);
                nB[sni] = a.y;
            }
            st0 = st2;
            st1 = st3;
        }
        cp_async_wait1();  // the copies issued two steps ago have landed
        __syncthreads();   // for every thread; the normals are complete, phi planes r0 + 1, r0 + 2 free
        if constexpr (IN) {
            const unsigned zoff = (unsigned)(z0 + r0 + 9) * plane;
            copy_phi(pA, zoff);
            copy_phi(pB, zoff + plane);
        } else {
            if constexpr (OUT < 0) issue_phi(6);  // into the slot of plane -2
            issue_phi(r0 + 9);
            issue_phi(r0 + 10);
        }
        if (comp) {
            float2 kxy1, kxy2;
            {
                const float2 l = make_float2(nA[nxl], nx1.x);
                float2 p = make_float2(nx1.y, nA[nxr]);
                if (!VEC && lone) p.x = l.x;
                kxy1 = f2add(f2sub(p, l), f2sub(ld2(nA + Z::NH * NXP + nyd), ld2(nA + Z::NH * NXP + nyu)));
            }
            {
                const float2 l = make_float2(nB[nxl], nx2.x);
                float2 p = make_float2(nx2.y, nB[nxr]);
                if (!VEC && lone) p.x = l.x;
                kxy2 = f2add(f2sub(p, l), f2sub(ld2(nB + Z::NH * NXP + nyd), ld2(nB + Z::NH * NXP + nyu)));
            }
            if constexpr (OUT == 0) {  // K*a, K*b of planes r0 .. r0 + 3
                const int d = (k >> 1) % (M / 4);  // the ring slot of plane r0 - R is 4 d
                unroll(std::make_integer_sequence<int, M / 4>{}, [&](auto dc) {
                    if (d == dc.value) convolve(dc);
                });
                issue_ab(in_c, r0 - R + M, 4 * d);
            }
            if constexpr (OUT >= 0) {
                // the normal beyond the brick's first and last plane is the mirrored one
                const float2 nzb = !IN && z0 + r0 == 0 ? nz1 : nzm;
                const float2 nza = !IN && z0 + r0 == nz - 1 ? nzm : nz1;
                const float2 nzc = !IN && z0 + r0 + 1 == nz - 1 ? nz0 : nz2;
                const float2 kap[2] = {f2mul(f2add(kxy0, f2sub(nza, nzb)), f2v(0.5f)),
                                       f2mul(f2add(kxy1, f2sub(nzc, nz0)), f2v(0.5f))};
                const float2 ph[2] = {ph0, ph1};
                const float2 lap[2] = {f2add(lxy0, f2add(f2add(ph1, phm), f2mul(f2v(-2.f), ph0))),
                                       f2add(lxy1, f2add(f2add(ph2, ph0), f2mul(f2v(-2.f), ph1)))};
                const unsigned o0 = out, o1 = out + plane;
                const unsigned q0 = qout, q1 = qout + qplane;
                out = o1 + plane;
                qout = q1 + qplane;
#pragma unroll
                for (int s = 0; s < 2; ++s) {
                    if (!IN && s == 1 && r0 + 1 >= nout) break;
                    const float2 a0 = acc[2 * OUT + s][0], a1 = acc[2 * OUT + s][1];
                    float2 g, pn, qn;
                    if constexpr (EX) {
                        const float2 im = raw[2 * OUT + s].template get<VEC>();
                        const float pz = pzq[2 * OUT + s];
                        pn.x = update_exact(ph[s].x, lap[s].x, kap[s].x, im.x, pxy.x * pz, a0.x, a0.y, s2, co, g.x);
                        pn.y = update_exact(ph[s].y, lap[s].y, kap[s].y, im.y, pxy.y * pz, a1.x, a1.y, s2, co, g.y);
                        qn = make_float2(heaviside_q_exact(pn.x, eps), heaviside_q_exact(pn.y, eps));
                    } else {
                        const float2 im = f2fma(raw[2 * OUT + s].template get<VEC>(), f2v(inv_s), f2v(nms));
                        if constexpr (R == 0) {  // Eq. (15), sigma_2 = 0: (a, b) are the fits (f1, f2)
                            const float2 d1 = f2sub(im, make_float2(a0.x, a1.x)), d2 = f2sub(im, make_float2(a0.y, a1.y));
                            g = f2fma(f2v(s2l1), f2mul(d1, d1), f2mul(f2v(-s2l2), f2mul(d2, d2)));
                        } else {  // Li's data terms from K*a, K*b: s^2 [(l1 - l2) K1 I~^2 - 2 I~ K*a + K*b]
                            const float2 t1 = f2mul(f2mul(cK, f2v(pzq[2 * OUT + s])), f2mul(im, im));
                            const float2 t2 = f2fma(f2mul(f2v(m2s2), im), make_float2(a0.x, a1.x), t1);
                            g = f2fma(f2v(s2), make_float2(a0.y, a1.y), t2);
                        }
                        const float2 den = f2fma(ph[s], ph[s], f2v(eps2));
                        // dt delta (Eq. 14), then phi + dt mu (L - kappa) + dt delta (nu kappa - g) (Eqs. 1, 13)
                        const float2 dtdel = f2mul(f2v(dt_eps_pi), make_float2(rcp_approx(den.x), rcp_approx(den.y)));
                        pn =
                            f2fma(f2v(dt_mu), f2sub(lap[s], kap[s]),
                                  f2fma(dtdel, f2fma(f2v(nu), kap[s], make_float2(-g.x, -g.y)), ph[s]));
                        qn = heaviside_q_fast2(pn, eps);
                    }
                    const unsigned o = s ? o1 : o0, oq = s ? q1 : q0;
                    if constexpr (VEC) {
                        if (act0) {
                            *reinterpret_cast<float2 *>(phi_out + o) = pn;
                            *reinterpret_cast<float2 *>(q_out + oq) = qn;
                        }
                    } else {
                        if (act0) {
                            phi_out[o] = pn.x;
                            q_out[oq] = qn.x;
                        }
                        if (act1) {
                            phi_out[o + 1] = pn.y;
                            q_out[oq + 1] = qn.y;
                        }
                    }
                    if constexpr (DUMP) {
                        float *const d = dump + o;
                        if (act0) {
                            d[2 * n] = g.x;
                            d[3 * n] = kap[s].x;
                            d[4 * n] = lap[s].x;
                        }
                        if (act1) {
                            d[2 * n + 1] = g.y;
                            d[3 * n + 1] = kap[s].y;
                            d[4 * n + 1] = lap[s].y;
                        }
                    }
                }
            }
            kxy0 = kxy2;
        }
        cp_async_commit();
        phm = ph1;
        ph0 = ph2;
        ph1 = ph3;
        lxy0 = lxy2;
        nzm = nz1;
        nz0 = nz2;
    };
    using Out0 = std::integral_constant<int, 0>;
    using Out1 = std::integral_constant<int, 1>;
    step(-1, std::integral_constant<int, -1>{}, Edge{});
    // two steps at a time; both inner when neither the first planes nor the last the second
    // step brings in (phi r0 + 12, (a, b) r0 - R + M + 3) are near the chunk's ends
    constexpr int AHEAD = M - R + 3 > 12 ? M - R + 3 : 12;
#pragma unroll 1
    for (int k = 0; 2 * k < nout; k += 2) {
        if (k > 0 && 2 * k + AHEAD < nout) {
            step(k, Out0{}, Inner{});
            step(k + 1, Out1{}, Inner{});
        } else {
            step(k, Out0{}, Edge{});
            if (2 * k + 2 < nout) step(k + 1, Out1{}, Edge{});
        }
    }
    cp_async_wait0();  // no copy into this CTA's shared memory outlives it
}

template <int R, class ImgT, bool DUMP = false, bool EX = false>
__global__ void __launch_bounds__((TBZ<R, EX>::THREADS), 2) k_tb_z(GroupArgs G, TapPairs t) {
    dependents_may_start();
    const int bi = find_brick(G.starts, G.nb, blockIdx.x);
    const BrickDev &B = G.bricks[bi];
    const uintptr_t at = reinterpret_cast<uintptr_t>(B.phi[0]) | reinterpret_cast<uintptr_t>(B.phi[1]);
    if (B.nx % 2 == 0 && at % 8 == 0 && reinterpret_cast<uintptr_t>(B.img) % (2 * sizeof(ImgT)) == 0)
        tb_z_march<R, ImgT, true, DUMP, EX>(G, B, bi, t);
    else
        tb_z_march<R, ImgT, false, DUMP, EX>(G, B, bi, t);
}

// ------------------------------------------------------------ launchers

// The update kernel (storage independent; dispatched in rsf_tiled_f32.cu).
cudaError_t launch_tb_z(const TiledGroup &g, int parity, Profiler *prof, cudaStream_t s);
cudaError_t prepare_tb_z(int R);

// Resident CTAs of the persistent z kernel of group A (set by prepare_storage).
template <int R, class S>
int &az_persist() {
    static int n = 152;
    return n;
}

template <int R, class ImgT, int NP>
constexpr size_t taxy_smem() { return XYSmem<R, SrcH<R, ImgT, NP, false>>::bytes; }
template <int R, class S>
constexpr size_t tbxy_smem() { return XYSmem<R, SrcAB<R, S>>::bytes; }

// Dynamic shared memory of group A's x/y kernel for each image type.
template <int R, int NP>
cudaError_t prepare_ta_xy() {
    cudaError_t e;
    if ((e = prepare_kernel(k_ta_xy<R, uint8_t, NP>, taxy_smem<R, uint8_t, NP>())) != cudaSuccess) return e;
    if ((e = prepare_kernel(k_ta_xy<R, uint16_t, NP>, taxy_smem<R, uint16_t, NP>())) != cudaSuccess) return e;
    return prepare_kernel(k_ta_xy<R, float, NP>, taxy_smem<R, float, NP>());
}
template <int R, int NP>
void launch_ta_xy(const TiledGroup &g, const GroupArgs &G, const TapPairs &tp, cudaStream_t s) {
    switch (g.imgtype) {
        case 0: launch_next(g.overlap, k_ta_xy<R, uint8_t, NP>, g.ncta[0], kXYThreads, taxy_smem<R, uint8_t, NP>(), s, G, tp); break;
        case 1: launch_next(g.overlap, k_ta_xy<R, uint16_t, NP>, g.ncta[0], kXYThreads, taxy_smem<R, uint16_t, NP>(), s, G, tp); break;
        default: launch_next(g.overlap, k_ta_xy<R, float, NP>, g.ncta[0], kXYThreads, taxy_smem<R, float, NP>(), s, G, tp);
    }
}

template <int R, class S>
cudaError_t prepare_storage() {
    cudaError_t e;
    if ((e = prepare_ta_xy<R, 1>()) != cudaSuccess) return e;
    if ((e = prepare_kernel(k_ta_z<R, S>, az_smem<R>())) != cudaSuccess) return e;
    {
        int dev = 0, sms = 0, occ = 0;
        if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
        if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
        if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_ta_z<R, S>, kAZThreads, az_smem<R>())) !=
            cudaSuccess) return e;
        if (occ > kAZCtas) occ = kAZCtas;
        az_persist<R, S>() = sms * (occ > 0 ? occ : 1);
    }
    return prepare_kernel(k_tb_xy<R, S>, tbxy_smem<R, S>());
}

// One iteration of Li's form (group A, group B, update) for radius R and storage S.
template <int R, class S>
cudaError_t launch_storage(const TiledGroup &g, int parity, Profiler *prof, cudaStream_t s) {
    GroupArgs G{g.bricks, nullptr, g.nb, parity, g.err, g.fault_tx};
    const TapPairs tp = tap_pairs(g.taps);
    {
        ProfScope ps(prof, KID_TA_XY);
        G.starts = g.starts[0];
        launch_ta_xy<R, 1>(g, G, tp, s);
    }
    {
        ProfScope ps(prof, KID_TA_Z);
        G.starts = g.starts[1];
        const unsigned grid = g.ncta[1] < (unsigned)az_persist<R, S>() ? g.ncta[1] : (unsigned)az_persist<R, S>();
        launch_next(g.overlap, k_ta_z<R, S>, grid, kAZThreads, az_smem<R>(), s, G, tp);
    }
    {
        ProfScope ps(prof, KID_TB_XY);
        G.starts = g.starts[2];
        launch_next(g.overlap, k_tb_xy<R, S>, g.ncta[2], kXYThreads, tbxy_smem<R, S>(), s, G, tp);
    }
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    return launch_tb_z(g, parity, prof, s);
}

template <class S>
cudaError_t prepare_group_s(int R) {
    switch (R) {
        case 2: return prepare_storage<2, S>();
        case 3: return prepare_storage<3, S>();
        case 4: return prepare_storage<4, S>();
        case 5: return prepare_storage<5, S>();
        case 6: return prepare_storage<6, S>();
        case 8: return prepare_storage<8, S>();
        case 10: return prepare_storage<10, S>();
        case 12: return prepare_storage<12, S>();
        default: return cudaErrorInvalidValue;
    }
}

template <class S>
cudaError_t launch_group_s(const TiledGroup &g, int parity, Profiler *prof, cudaStream_t s) {
    switch (g.taps.R) {
        case 2: return launch_storage<2, S>(g, parity, prof, s);
        case 3: return launch_storage<3, S>(g, parity, prof, s);
        case 4: return launch_storage<4, S>(g, parity, prof, s);
        case 5: return launch_storage<5, S>(g, parity, prof, s);
        case 6: return launch_storage<6, S>(g, parity, prof, s);
        case 8: return launch_storage<8, S>(g, parity, prof, s);
        case 10: return launch_storage<10, S>(g, parity, prof, s);
        case 12: return launch_storage<12, S>(g, parity, prof, s);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace tiled
}  // namespace rsf
