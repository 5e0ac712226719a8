// rsf_internal.h -- host-side interfaces between the C ABI layer and the
// kernel translation units of librsf.so.  Not installed; not part of the ABI.
#pragma once

#include <cuda.h>  // CUtensorMap (the encoder is reached through the runtime's driver entry point)
#include <cuda_runtime.h>

#include <cstddef>
#include <cstdint>
#include <vector>

#include "rsf_device.cuh"

namespace rsf {

// Kernel identifiers for the per-launch timing of rsf_prof_*.
enum KernelId {
    KID_AX = 0,    // group A, x pass: H products + x convolution
    KID_AY,        // group A, y pass
    KID_AZ,        // group A, z pass + local fits epilogue
    KID_BX,        // group B, x pass
    KID_BY,        // group B, y pass
    KID_BZ,        // group B, z pass + data term, curvature and update epilogue
    KID_TA_XY,     // tiled: group A, H products + x and y convolution
    KID_TA_Z,      // tiled: group A, z convolution + local fits
    KID_TB_XY,     // tiled: group B, x and y convolution
    KID_TB_Z,      // tiled: group B, z convolution + data term, curvature, update
    KID_COUNT
};
const char *kernel_name(int id);

// Records CUDA event pairs around launches while enabled.
struct Profiler {
    bool on = false;
    cudaStream_t stream = nullptr;
    struct Rec { int id; cudaEvent_t a, b; };
    std::vector<Rec> recs;
    std::vector<cudaEvent_t> pool;
    size_t used = 0;
    int open_id = -1;
    cudaEvent_t open_a = nullptr;

    cudaEvent_t take();
    void begin(int id);
    void end();
    void reset();
    void release();
};

// RAII bracket around one launch.
struct ProfScope {
    Profiler *p;
    ProfScope(Profiler *prof, int id) : p(prof && prof->on ? prof : nullptr) { if (p) p->begin(id); }
    ~ProfScope() { if (p) p->end(); }
};

// Device fields of one volume (all FP32, n elements unless noted).
struct Fields {
    Dims d{};
    float *I = nullptr;       // centred, scaled image  (I - m) / s
    float *prof = nullptr;    // zero-padding profiles p_x[nx], p_y[ny], p_z[nz]; K*1 = p_x p_y p_z
    float *cs = nullptr;      // [0] m, [1] 1/s, [2] s^2, [3] s   (centring constants)
    float *partials = nullptr;// reduction scratch, 3 * kStatBlocks floats
    float *phi[2] = {nullptr, nullptr};
    float *q = nullptr;       // tiled path: 2 n floats, +-atan(eps/|phi|)/pi of the current phi, pitched
    float *t[8] = {};         // stage buffers: one block of 8 * capacity floats, t[i] = t[0] + i * capacity,
                              // capacity >= px * ny * nz (the tiled path's fields: tiled_place_fields)
    int px = 0;               // x pitch of the tiled path's intermediate fields (multiple of 32)
};

constexpr int kStatBlocks = 1024;

// Centring constants (f.cs) from the statistics of `vol`, a device pointer of dtype vt (0 u8,
// 1 u16, 2 f32); enqueues on `s` and never synchronises.
cudaError_t image_stats(const void *vol, int vt, Fields &f, cudaStream_t s);
// Zero-padding profiles p_a(i) = sum of the in-volume taps (double sums rounded
// once), nx + ny + nz floats: K*1 = p_x p_y p_z.
void zero_padding_profiles(const Taps &taps, int nx, int ny, int nz, float *out);

// The same and the centred image f.I.
cudaError_t centre_image(const void *vol, int vt, Fields &f, cudaStream_t s);

// Sets the calling thread's rsf_last_error() text.
void set_last_error(const char *msg);

// One brick of the tiled path: an independent volume with its own fields and
// scalars.  Device copies of these descriptors drive the batched launches.
struct BrickDev {
    int nx, ny, nz, px;     // dimensions; x pitch of the intermediate fields
    int up;                 // x pitch of u2: px, or nx where a copied image needs the room (tiled_place_fields)
    const void *img;        // image, nx*ny*nz values of the group's image type
    const void *img_t;      // the image as the TMA boxes read it: img, or a copy with 16-byte rows
    int ip;                 // row pitch of img_t (values)
    int qp;                 // row pitch of q (nx rounded up to 4)
    const float *cs;        // centring constants [m, 1/s, s^2, s]
    const float *prof;      // K*1 profiles p_x[nx], p_y[ny], p_z[nz]
    float *phi[2];          // ping-pong level set
    float *q;               // q = +-atan(eps/|phi|)/pi of the current phi: read by group A's x/y kernel,
                            // rewritten by the update at the end of the iteration
    float2 *u2;             // pitched x/y-convolved (H I~, H), FP32 (Eq. (15) form: one float4 per voxel,
                            // ((H I~, H), ((1-H) I~, 1-H)))
    void *ab;               // pitched (a, b), storage type
    float2 *abxy;           // pitched x/y-convolved (a, b), FP32 (also the set-up's scratch for ki); the memory
                            // of u2, which is read before this is written (Eq. (15) form: the fits (f1, f2),
                            // memory of their own)
    float *ki;              // pitched K*I~ (the centred image convolved), FP32, set once per solve
    float eps, lambda1, lambda2, nu, mu, dt;
    int zc;                 // z chunk of the update kernel (the normals' rounding follows it)
    int zs;                 // planes per CTA of the update kernel: a z chunk is split into parts of zs
    int xyp;                // z planes per CTA of the x/y kernels
    int flip;               // this brick's buffer parity is the launch parity xor flip
    float *dump;            // optional 5 * n stage fields (f1, f2, g, kappa, L)
    // TMA descriptors (tiled_encode_maps).  Group A's z pass: u2 as FP32 [nz][ny][c nx]
    // (row pitch c px; c = 2, or 4 in the Eq. (15) form) in boxes of 32 c floats x 1 row x
    // (64 + 2R) planes, and ki as FP32 [nz][ny][nx] in boxes of 32 x 1 x 64.  The x/y kernels:
    // one staged plane of a tile (XYField in rsf_tiled.cuh) of q, the image and (Li's form) ab.
    CUtensorMap tm_u, tm_k, tm_ab, tm_q, tm_img;
};

// A set of bricks launched together: same radius, image type and storage.
struct TiledGroup {
    int storage;            // 0 FP32, 1 BF16, 2 FP16 (rsf_storage)
    int force;              // 0 Li's data terms (group B convolutions), 1 Eq. (15) with sigma_2 = 0,
                            // kForceExact Li's in the exact arithmetic
    int imgtype;            // 0 uint8, 1 uint16, 2 float
    Taps taps;
    const BrickDev *bricks; // device array of nb descriptors
    int nb;
    const int *starts[4];   // device: per kernel, nb + 1 CTA offsets
    unsigned ncta[4];       // CTAs per kernel launch
    int dump;               // 1: some brick has a stage dump (its update kernel writes g, kappa, L)
    bool overlap;           // its kernels may start before the one before has ended (tiled_overlap)
    int *err;               // device-visible error word of the kernels' bounded waits (nonzero: expired)
    unsigned fault_tx;      // bytes the TMA barriers expect beyond their copies (0; > 0 in a fault test)
};

constexpr int kForceExact = 2;

// Device error word values (TiledGroup::err).
constexpr int kErrWaitExpired = 1;  // a bounded wait for a TMA copy ran out (1 s)
constexpr int kErrSmemAlign = 2;    // a TMA destination in shared memory was not 128-byte aligned

// Tiled four-kernel path (rsf_tiled*.cu) for the radii it is instantiated for.
bool tiled_supports(int R);
// The tiled kernels address a brick's pitched fields with 32-bit offsets: they take
// bricks of fewer than 2^32 pitched voxels.
bool tiled_fits(long long nx, long long ny, long long nz);
int tiled_pitch(int nx);
// Encodes b's tensor maps from its dimensions, pitches and field views for its
// group's form (force), storage, image type and radius R; those not used are zeroed.
cudaError_t tiled_encode_maps(BrickDev &b, int force, int storage, int imgtype, int R);
cudaError_t tiled_prepare(int storage, int R, int force);
cudaError_t tiled_iterate(const TiledGroup &g, int parity, Profiler *prof, cudaStream_t s);
// Whether a group's consecutive kernels overlap at their boundary (programmatic dependent launch).
bool tiled_overlap(const TiledGroup &g, int sms);
// CTAs of the four kernels for one brick of a group of the given form and radius.
void tiled_cta_counts(const BrickDev &b, int force, int R, unsigned counts[4]);
// Planes per CTA of the x/y kernels for bricks launched together (results do not depend on it).
int tiled_xy_planes(const BrickDev *bricks, int nb, int force, int R, int sms);
// Planes per CTA of the update kernel (at most zc) for bricks launched together with z chunk zc.
int tiled_update_planes(const BrickDev *bricks, int nb, int force, int R, int zc, int sms);
// A brick's working memory beside its phi buffers: a stage block of
// tiled_stage_bytes(storage, px ny nz) bytes, and directly in front of it a q block of
// tiled_q_bytes(nx, ny nz) bytes (anywhere for a stage block of 28 px ny nz bytes or more).
size_t tiled_stage_bytes(int storage, long long np);
size_t tiled_q_bytes(int nx, long long rows);
// Sets b's pitches and field pointers from its dimensions and image (b.nx, ny, nz, img) in
// those two blocks (256-byte aligned; stage may be larger than the minimum).
void tiled_place_fields(BrickDev &b, int storage, int force, int imgtype, void *stage, size_t stage_bytes, void *q);
// One brick's work before the first iteration, for kernels that take many bricks at once
// (blockIdx.y): image statistics, phi0 to phi (or nothing where they are the same), q of it,
// the image copied to img_t where that differs.
struct SetupBrick {
    const void *img;
    int imgtype;
    int nx, qp, ip;
    long long rows;         // ny * nz
    const float *src;       // phi0
    float *phi, *q;
    void *img_t;
    float *partials, *cs;   // 3 * kStatBlocks floats of scratch; the centring constants
    float eps;
};
SetupBrick setup_of(const BrickDev &b, int imgtype, const float *phi0, float *partials, float *cs);
// Statistics (partials, cs) and start (phi, q, img_t) of n bricks described in device memory.
cudaError_t setup_stats(const SetupBrick *d, int n, cudaStream_t s);
cudaError_t setup_start(const SetupBrick *d, int n, cudaStream_t s);
// The start of one brick, described by value.
cudaError_t tiled_start(const BrickDev &b, int imgtype, const float *phi0, cudaStream_t s);
// K*I~ of a group's bricks (b.ki) before its first iteration (after the start; uses b.abxy as
// scratch); nothing in the Eq. (15) form.
cudaError_t tiled_ki_init(const TiledGroup &g, cudaStream_t s);

// The exact arithmetic (rsf_exact.cuh): radii 1 to 16.  Fields in a stage block of
// exact_stage_bytes and a q block of exact_q_bytes (at most the 8 nx ny nz above); before the
// first iteration the centred image (b.img, FP32, pitched; from the caller's vol and b.cs)
// and q.
bool exact_supports(int R);
size_t exact_stage_bytes(int nx, int ny, int nz);
size_t exact_q_bytes(int nx, int ny, int nz);
void exact_place_fields(BrickDev &b, void *stage, float *q);
cudaError_t exact_start(const BrickDev &b, const void *vol, int vt, cudaStream_t s);

// Loads kernels on the current device (by default a kernel's code is loaded, and takes device
// memory, at its first launch).
template <class... K>
cudaError_t load_kernels(K *...kernels) {
    cudaError_t e = cudaSuccess;
    cudaFuncAttributes a;
    for (const void *k : {reinterpret_cast<const void *>(kernels)...})
        if (e == cudaSuccess) e = cudaFuncGetAttributes(&a, k);
    return e;
}
cudaError_t load_exact();   // the exact arithmetic at every radius, its set-up included
cudaError_t load_passes();  // the six passes, statistics and centring
// One iteration of the separable pass path: phi_in -> phi_out.
// `stages`, when not null, receives RSF_NSTAGES fields (f1, f2, g, kappa, L).
cudaError_t iterate_passes(const Taps &taps, const Coeffs &c, Fields &f, const float *phi_in, float *phi_out,
                           float *stages, Profiler *prof, cudaStream_t s);

}  // namespace rsf
