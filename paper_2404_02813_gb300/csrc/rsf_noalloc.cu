// rsf_noalloc.cu -- rsf_evolve_noalloc: the level-set evolution of rsf_evolve
// for small volumes, with every working field held in one file-scope device
// array instead of memory the library allocates.
//
// Who needs it: code that may not allocate GPU memory while it runs -- a
// plug-in whose host application owns all device memory through its own pool,
// a real-time or streaming thread that cannot accept the device-wide
// synchronisation a cudaMalloc / cudaFree can imply, or a service whose
// memory was sized once at start-up.  Those callers bring their own input and
// output buffers and a stream; this entry point touches only them and the
// static array below.
//
// The static array is part of the library image: every GPU that loads
// librsf.so holds it (about 10.5 MB) until the process exits.  All calls on a
// device share it and it keeps the contents of the last call; calls whose
// work overlaps on the GPU (several streams, several host threads) race on it
// and must be serialised by the caller.  No part of it needs to start at zero:
// every field is written in full before it is read.
#include <cuda_runtime.h>

#include <cmath>
#include <cstddef>
#include <cstdio>
#include <cstring>
#include <mutex>

#include "rsf.h"
#include "rsf_ctx.h"
#include "rsf_internal.h"
#include "rsf_tiled.cuh"

namespace {

constexpr long long kMaxVoxels = 1LL << 18;              // 262,144 voxels (for example 64^3)
constexpr long long kMaxProfile = kMaxVoxels / 16 + 8;   // nx+ny+nz when every side is >= 4
constexpr long long kOffPhi = 0;                         // one phi buffer (phi_out is the other)
constexpr long long kOffI = kOffPhi + kMaxVoxels;        // centred image
constexpr long long kOffT = kOffI + kMaxVoxels;          // eight stage buffers
constexpr long long kOffProf = kOffT + 8 * kMaxVoxels;   // K*1 profiles
constexpr long long kOffCs = kOffProf + ((kMaxProfile + 63) / 64) * 64;
constexpr long long kOffPart = kOffCs + 64;              // reduction partials
constexpr long long kScratchFloats = kOffPart + 3 * rsf::kStatBlocks;
constexpr int kMaxDevices = 64;
// The tiled kernels' fields take the same memory from kOffI on: launch descriptor (with the
// CTA offsets and the error word after it), q and stage blocks, where the x pitch (a multiple of 32) leaves room
// for them: 24 bytes per voxel of a row rounded up to 32 and 8 of one rounded up to 4, where the
// voxel limit has 36 per voxel -- always when nx is a multiple of 32, and up to 0.65 of the limit at
// nx = 33, 0.78 at 40, 0.98 at 54, 0.82 at 65, 0.64 at 16, 0.18 at 4.
constexpr size_t kDescBytes = (sizeof(rsf::BrickDev) + 64 + 255) / 256 * 256;
constexpr size_t kFieldBytes = sizeof(float) * 9 * (size_t)kMaxVoxels;

}  // namespace

static __device__ __align__(256) float g_noalloc_scratch[kScratchFloats];

namespace {

std::mutex g_mu;
float *g_scratch_dev[kMaxDevices] = {};

rsf_status err(rsf_status st, const char *msg) {
    rsf::set_last_error(msg);
    return st;
}

// Values written into the static array through kernel parameters, so that no
// host staging buffer and no allocation is involved (24 KB per launch).
constexpr int kParamChunk = 6144;
struct ParamChunk {
    int offset, count;
    float v[kParamChunk];
};

__global__ void k_noalloc_put(ParamChunk c, float *__restrict__ dst);
__global__ void k_noalloc_finish(const int *err, const float *phi, float *phi_out, int n);

// Device address of the static array on the current device, looked up once per
// device (with that device current).  The name g_noalloc_scratch is only a
// host-side stand-in; kernels must be given this address.  The same first call
// loads every kernel of this entry, so that no later one loads code (6 MB of
// device memory over the kernel widths) in the middle of its caller's run.
rsf_status scratch_on_current_device(float **out) {
    int dev = -1;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return err(RSF_E_CUDA, cudaGetErrorString(e));
    if (dev < 0 || dev >= kMaxDevices) return err(RSF_E_CUDA, "device index out of range for rsf_evolve_noalloc");
    std::lock_guard<std::mutex> lk(g_mu);
    if (!g_scratch_dev[dev]) {
        void *p = nullptr;
        e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
        if (e != cudaSuccess) {
            char buf[256];
            snprintf(buf, sizeof buf, "cudaGetSymbolAddress of the static scratch failed: %s", cudaGetErrorString(e));
            return err(RSF_E_CUDA, buf);
        }
        if ((e = rsf::load_kernels(k_noalloc_put, k_noalloc_finish)) == cudaSuccess) e = rsf::load_passes();
        if (e == cudaSuccess) e = rsf::load_exact();
        if (e != cudaSuccess) return err(RSF_E_CUDA, cudaGetErrorString(e));
        g_scratch_dev[dev] = (float *)p;
    }
    *out = g_scratch_dev[dev];
    return RSF_OK;
}

__global__ void k_noalloc_put(ParamChunk c, float *__restrict__ dst) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < c.count; i += gridDim.x * blockDim.x)
        dst[c.offset + i] = c.v[i];
}

// phi, where the last iteration left it, to phi_out.  After a solve in which a kernel's bounded wait
// ran out (it then left tiles unwritten) phi_out is NaN throughout: this entry has no other way to
// tell, as it returns before the kernels run.
__global__ void __launch_bounds__(256) k_noalloc_finish(const int *err, const float *phi, float *phi_out, int n) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    rsf::tiled::wait_for_previous();
    const float v = phi[i];
    const bool bad = *err != 0;
    if (bad || phi != phi_out) phi_out[i] = bad ? NAN : v;
}

void put_floats(const float *v, int n, float *dst, cudaStream_t s) {
    for (int o = 0; o < n; o += kParamChunk) {
        ParamChunk c;
        c.offset = o;
        c.count = n - o < kParamChunk ? n - o : kParamChunk;
        memcpy(c.v, v + o, sizeof(float) * c.count);
        k_noalloc_put<<<(c.count + 255) / 256, 256, 0, s>>>(c, dst);
    }
}

// The iterations in the tiled schedule (rsf_exact.cuh), all fields in `mem`; phi[0] holds phi0,
// phi[1] is phi_out and gets the result.
// fault_tx: as in TiledGroup.
cudaError_t evolve_tiled(rsf::BrickDev b, const void *vol, int vt, const rsf::Taps &taps, int iters, char *mem, int dev,
                         unsigned fault_tx, cudaStream_t s) {
    char *const q = mem + kDescBytes;
    rsf::exact_place_fields(b, q + (rsf::exact_q_bytes(b.nx, b.ny, b.nz) + 255) / 256 * 256, reinterpret_cast<float *>(q));
    int sms = 0;
    cudaError_t e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    if ((e = rsf::tiled_prepare(0, taps.R, rsf::kForceExact)) != cudaSuccess) return e;
    b.xyp = rsf::tiled_xy_planes(&b, 1, rsf::kForceExact, taps.R, sms);
    b.zc = b.nz;
    b.zs = rsf::tiled_update_planes(&b, 1, rsf::kForceExact, taps.R, b.zc, sms);
    if ((e = rsf::tiled_encode_maps(b, rsf::kForceExact, 0, 2, taps.R)) != cudaSuccess) return e;
    rsf::TiledGroup g{};
    g.force = rsf::kForceExact;
    g.imgtype = 2;
    g.taps = taps;
    g.nb = 1;
    rsf::tiled_cta_counts(b, g.force, taps.R, g.ncta);
    g.overlap = rsf::tiled_overlap(g, sms);
    struct {
        rsf::BrickDev b;
        int starts[8];
        int err;  // the bounded waits' error word, cleared with the descriptor's upload
    } d{};
    d.b = b;
    for (int k = 0; k < 4; ++k) d.starts[2 * k + 1] = (int)g.ncta[k];
    static_assert(sizeof(d) <= kDescBytes && sizeof(d) % sizeof(float) == 0, "descriptor");
    const rsf::BrickDev *db = reinterpret_cast<const rsf::BrickDev *>(mem);
    g.bricks = db;
    for (int k = 0; k < 4; ++k) g.starts[k] = reinterpret_cast<const int *>(mem + offsetof(decltype(d), starts)) + 2 * k;
    g.err = reinterpret_cast<int *>(mem + offsetof(decltype(d), err));
    g.fault_tx = fault_tx;
    put_floats(reinterpret_cast<const float *>(&d), (int)(sizeof(d) / sizeof(float)), reinterpret_cast<float *>(mem), s);
    if ((e = rsf::exact_start(b, vol, vt, s)) != cudaSuccess) return e;
    for (int it = 0; it < iters; ++it)
        if ((e = rsf::tiled_iterate(g, it & 1, nullptr, s)) != cudaSuccess) return e;
    const int n = b.nx * b.ny * b.nz;
    rsf::tiled::launch_next(g.overlap, k_noalloc_finish, (n + 255) / 256, 256, 0, s, g.err, b.phi[iters & 1], b.phi[1], n);
    return cudaGetLastError();
}

rsf_status evolve(const void *volume, rsf_dtype vt, int64_t nx, int64_t ny, int64_t nz, const float *phi0,
                  float *phi_out, float sigma, float eps, float lambda1, float lambda2, float nu, float mu, float dt,
                  int32_t iters, void *stream, unsigned fault_tx) {
    if (!volume || !phi0 || !phi_out) return err(RSF_E_INVAL, "null volume, phi0 or phi_out pointer");
    if (vt != RSF_U8 && vt != RSF_U16 && vt != RSF_F32) return err(RSF_E_INVAL, "unknown volume dtype");
    if (nx < 4 || ny < 4 || nz < 4) return err(RSF_E_INVAL, "each dimension must be >= 4");
    if ((double)nx * (double)ny * (double)nz > (double)kMaxVoxels) {
        char buf[200];
        snprintf(buf, sizeof buf, "rsf_evolve_noalloc: %lld voxels exceed its static limit of %lld voxels",
                 (long long)nx * ny * nz, kMaxVoxels);
        return err(RSF_E_INVAL, buf);
    }
    if (!(sigma > 0.f) || !std::isfinite(sigma)) return err(RSF_E_INVAL, "sigma must be positive and finite");
    const int R = (int)std::floor(2.0 * (double)sigma + 0.5);
    if (R > rsf::RMAX) return err(RSF_E_INVAL, "kernel radius round(2 sigma) exceeds 16");
    if (!(eps > 0.f) || !std::isfinite(eps)) return err(RSF_E_INVAL, "eps must be positive and finite");
    if (!(dt > 0.f) || !std::isfinite(dt)) return err(RSF_E_INVAL, "dt must be positive and finite");
    if (iters < 0) return err(RSF_E_INVAL, "iters must be >= 0");
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return err(RSF_E_CUDA, cudaGetErrorString(e));
    // (device memory of another GPU is refused too: without peer access a kernel here would fault on it)
    if (!in_place(volume, dev, 1) || !in_place(phi0, dev, 1) || !in_place(phi_out, dev, 1))
        return err(RSF_E_INVAL, "rsf_evolve_noalloc takes device pointers of the current device only");

    float *base = nullptr;
    rsf_status st = scratch_on_current_device(&base);
    if (st) return st;
    cudaStream_t s = (cudaStream_t)stream;

    rsf::Fields f;
    f.d = rsf::Dims{(int)nx, (int)ny, (int)nz, (long long)nx * ny, (long long)nx * ny * nz};
    f.I = base + kOffI;
    for (int i = 0; i < 8; ++i) f.t[i] = base + kOffT + i * kMaxVoxels;
    f.prof = base + kOffProf;
    f.cs = base + kOffCs;
    f.partials = base + kOffPart;
    float *scratch_phi = base + kOffPhi;
    const long long n = f.d.n;

    const rsf::Taps taps = make_taps(sigma);
    const rsf::Coeffs co{eps, lambda1, lambda2, nu, mu, dt};

    if (iters == 0) {
        if (phi_out != phi0) e = cudaMemcpyAsync(phi_out, phi0, sizeof(float) * n, cudaMemcpyDeviceToDevice, s);
        else e = cudaSuccess;
        return e == cudaSuccess ? RSF_OK : err(RSF_E_CUDA, cudaGetErrorString(e));
    }
    const bool tiled = rsf::exact_supports(R) &&
                       kDescBytes + (rsf::exact_q_bytes((int)nx, (int)ny, (int)nz) + 255) / 256 * 256 +
                               rsf::exact_stage_bytes((int)nx, (int)ny, (int)nz) <= kFieldBytes;
    e = tiled ? rsf::image_stats(volume, (int)vt, f, s) : rsf::centre_image(volume, (int)vt, f, s);
    if (e != cudaSuccess) return err(RSF_E_CUDA, cudaGetErrorString(e));
    // zero-padding profiles (K*1 = p_x p_y p_z), by the same host routine as rsf_evolve's;
    // nx + ny + nz <= kMaxProfile within the voxel limit
    float prof[kMaxProfile];
    rsf::zero_padding_profiles(taps, (int)nx, (int)ny, (int)nz, prof);
    put_floats(prof, (int)(nx + ny + nz), f.prof, s);
    // phi0 is copied first so that phi_out may alias it; the iterations then
    // alternate between the static buffer and phi_out
    if ((e = cudaMemcpyAsync(scratch_phi, phi0, sizeof(float) * n, cudaMemcpyDeviceToDevice, s)) != cudaSuccess)
        return err(RSF_E_CUDA, cudaGetErrorString(e));
    const float *in = scratch_phi;
    if (tiled) {
        rsf::BrickDev b{};
        b.nx = (int)nx;
        b.ny = (int)ny;
        b.nz = (int)nz;
        b.cs = f.cs;
        b.prof = f.prof;
        b.phi[0] = scratch_phi;
        b.phi[1] = phi_out;
        b.eps = eps;
        b.lambda1 = lambda1;
        b.lambda2 = lambda2;
        b.nu = nu;
        b.mu = mu;
        b.dt = dt;
        if ((e = evolve_tiled(b, volume, (int)vt, taps, iters, reinterpret_cast<char *>(base + kOffI), dev, fault_tx,
                              s)) != cudaSuccess)
            return err(RSF_E_CUDA, cudaGetErrorString(e));
        in = phi_out;
    } else {
        float *out = phi_out;
        for (int it = 0; it < iters; ++it) {
            if ((e = rsf::iterate_passes(taps, co, f, in, out, nullptr, nullptr, s)) != cudaSuccess)
                return err(RSF_E_CUDA, cudaGetErrorString(e));
            float *nxt = (out == phi_out) ? scratch_phi : phi_out;
            in = out;
            out = nxt;
        }
    }
    if (in != phi_out) {
        if ((e = cudaMemcpyAsync(phi_out, in, sizeof(float) * n, cudaMemcpyDeviceToDevice, s)) != cudaSuccess)
            return err(RSF_E_CUDA, cudaGetErrorString(e));
    }
    e = cudaGetLastError();
    return e == cudaSuccess ? RSF_OK : err(RSF_E_CUDA, cudaGetErrorString(e));
}

}  // namespace

extern "C" rsf_status rsf_evolve_noalloc(const void *volume, rsf_dtype vt, int64_t nx, int64_t ny, int64_t nz,
                                         const float *phi0, float *phi_out, float sigma, float eps, float lambda1,
                                         float lambda2, float nu, float mu, float dt, int32_t iters, void *stream) {
    return evolve(volume, vt, nx, ny, nz, phi0, phi_out, sigma, eps, lambda1, lambda2, nu, mu, dt, iters, stream, 0u);
}

// Not part of the ABI, for tests: the same with copy barriers armed for 16 bytes more than the
// copies bring (as RSF_OPT_FAULT_WAIT does on a context), so that every bounded wait runs out.
extern "C" rsf_status rsf_test_noalloc_expired_waits(const void *volume, rsf_dtype vt, int64_t nx, int64_t ny, int64_t nz,
                                                     const float *phi0, float *phi_out, float sigma, float eps,
                                                     float lambda1, float lambda2, float nu, float mu, float dt,
                                                     int32_t iters, void *stream) {
    return evolve(volume, vt, nx, ny, nz, phi0, phi_out, sigma, eps, lambda1, lambda2, nu, mu, dt, iters, stream, 16u);
}
