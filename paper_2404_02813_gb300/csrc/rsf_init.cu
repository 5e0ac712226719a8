// rsf_init.cu -- rsf_init_phi0: the seed initialisation of arXiv 2404.02813,
// Sec. 4.3.  Blob seeds come from the determinant of the Hessian in every z
// slice; phi0 is r0 minus the Euclidean distance to the nearest seed (the
// distance the paper's fast sweeping approximates, here exact).
//
//   taps       g_k = exp(-k^2/2s^2)/sum, g'_k = -(k/s^2) g_k,
//              g''_k = (k^2/s^4 - 1/s^2) g_k, k = -R..R, R = round(3 s)
//   filters    in-slice correlation with zero padding: I_xx = (g'' in x, g in y),
//              I_yy = (g in x, g'' in y), I_xy = (g' in x, g' in y)
//   response   D = s^4 (I_xx I_yy - I_xy^2) where I_xx + I_yy < 0, else -inf
//   seeds      D > t * (maximum of D over the slice), that maximum > 0, and D
//              above D at each existing in-slice neighbour (3 x 3)
//   phi0       r0 - sqrt(min over seeds of the squared distance); the squared
//              distances are integers below 2^24, exact in FP32, built by one
//              pass per axis: d_a(i) = min_j (d_{a-1}(j) + (i - j)^2) along the line.
//
// Kernels.  The response is one pass (k_hessian): a tile's image and its three x-filtered
// fields stay in shared memory, the y filters, D and the slice maximum follow.  Distances:
// along x from the seed bits of a row; along y and z each line (32 columns at a time) lies
// in shared memory with the minimum of every 8 of its values, and a voxel searches outwards
// from its own place, skipping groups that cannot improve on what it has and stopping where
// the offset alone exceeds it -- the same minimum as over the whole line, at a cost set by
// the distance to the nearest seed instead of the line's length.  The z pass writes phi0.
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <mutex>
#include <utility>

#include "rsf.h"
#include "rsf_ctx.h"

namespace {

constexpr int kMaxR = 16;

struct DerivTaps {
    int R;
    float g[2 * kMaxR + 1], g1[2 * kMaxR + 1], g2[2 * kMaxR + 1];
};

DerivTaps make_deriv_taps(float s) {
    DerivTaps t{};
    t.R = (int)std::floor(3.0 * s + 0.5);
    double w[2 * kMaxR + 1], sum = 0.0;
    for (int k = -t.R; k <= t.R; ++k) sum += (w[k + t.R] = std::exp(-(double)k * k / (2.0 * s * s)));
    for (int k = -t.R; k <= t.R; ++k) {
        const double g = w[k + t.R] / sum;
        t.g[k + t.R] = (float)g;
        t.g1[k + t.R] = (float)(-(k / ((double)s * s)) * g);
        t.g2[k + t.R] = (float)(((double)k * k / std::pow((double)s, 4) - 1.0 / ((double)s * s)) * g);
    }
    return t;
}

constexpr int kHT = 32;                  // response tile edge
constexpr int kHThreads = 256;
constexpr int kMaxLine = 4096;           // longest line: squared distances stay below 2^24
constexpr int kGroup = 8;                // values per minimum of a line

// Order-preserving signed key of a float (not NaN), for atomicMax; its own inverse.
__device__ __forceinline__ int max_key(float v) {
    const int i = __float_as_int(v);
    return i ^ ((i >> 31) & 0x7fffffff);
}
__device__ __forceinline__ float key_value(int k) { return __int_as_float(k ^ ((k >> 31) & 0x7fffffff)); }

// Determinant-of-Hessian response D of one 32 x 32 tile of a slice and the slice maximum.
// The radius R = round(3 s) is a template argument, each of 0 to 16 an instantiation, so that a
// lane filters a register window -- four outputs of a row from aligned 16-byte reads, then four
// outputs of a column -- with its taps as constant operands (384^3 uint16 at radius 5: 0.368 ms;
// 0.677 ms with a loop over taps, 1.53 ms in two passes with the x-filtered fields in global
// memory).  Bound by instruction issue.
// Shared memory: image [H][P], x-filtered fields [3][H][36], H = 32 + 2R, P = H rounded up
// to an odd number of 16-byte units.
constexpr int kHX = 36;  // row pitch of the x-filtered fields: 9 units of 16 bytes
__host__ __device__ constexpr int hessian_pitch(int R) { return ((kHT + 2 * R + 3) / 4 | 1) * 4; }
template <class T, int R>
__global__ void __launch_bounds__(kHThreads) k_hessian(const T *__restrict__ img, float *__restrict__ D,
                                                       int *__restrict__ smax, int nx, int ny, DerivTaps tp, float s4) {
    extern __shared__ __align__(16) float hsm[];
    __shared__ float red[kHThreads / 32];
    constexpr int W = kHT + 2 * R, P = hessian_pitch(R), FS = W * kHX;  // FS: one x-filtered field
    float *const in = hsm, *const xf = hsm + W * P;
    const int x0 = blockIdx.x * kHT, y0 = blockIdx.y * kHT;
    const long long plane = (long long)nx * ny, slice = blockIdx.z * plane;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int rows = min(W, ny - y0 + 2 * R);  // rows the outputs inside the slice take taps from
    for (int r = warp; r < rows; r += kHThreads / 32) {
        const int gy = y0 - R + r;
        for (int c = lane; c < W; c += 32) {
            const int gx = x0 - R + c;
            in[r * P + c] = (unsigned)gx < (unsigned)nx && (unsigned)gy < (unsigned)ny
                                ? (float)img[slice + (long long)gy * nx + gx] : 0.f;
        }
    }
    __syncthreads();
    const int c4 = (lane & 7) * 4;  // four rows of eight groups of four columns
    for (int r = warp * 4 + (lane >> 3); r < rows; r += kHThreads / 8) {
        float v[(4 + 2 * R + 3) / 4 * 4];
#pragma unroll
        for (int j = 0; j < (4 + 2 * R + 3) / 4; ++j) {
            const float4 q = *reinterpret_cast<const float4 *>(in + r * P + c4 + 4 * j);
            v[4 * j] = q.x;
            v[4 * j + 1] = q.y;
            v[4 * j + 2] = q.z;
            v[4 * j + 3] = q.w;
        }
        float a[4], b[4], c[4];
#pragma unroll
        for (int o = 0; o < 4; ++o) {
            a[o] = b[o] = c[o] = 0.f;
#pragma unroll
            for (int k = 0; k <= 2 * R; ++k) {
                a[o] = fmaf(tp.g[k], v[o + k], a[o]);
                b[o] = fmaf(tp.g1[k], v[o + k], b[o]);
                c[o] = fmaf(tp.g2[k], v[o + k], c[o]);
            }
        }
        float *const o = xf + r * kHX + c4;
        *reinterpret_cast<float4 *>(o) = make_float4(a[0], a[1], a[2], a[3]);
        *reinterpret_cast<float4 *>(o + FS) = make_float4(b[0], b[1], b[2], b[3]);
        *reinterpret_cast<float4 *>(o + 2 * FS) = make_float4(c[0], c[1], c[2], c[3]);
    }
    __syncthreads();
    float best = -INFINITY;
    const int r0 = warp * 4;  // four rows of one column
    if (y0 + r0 < ny) {
        float ixx[4], iyy[4], ixy[4];
#pragma unroll
        for (int o = 0; o < 4; ++o) ixx[o] = iyy[o] = ixy[o] = 0.f;
        const float *const f = xf + r0 * kHX + lane;
#pragma unroll
        for (int j = 0; j < 4 + 2 * R; ++j) {
            const float v0 = f[j * kHX], v1 = f[FS + j * kHX], v2 = f[2 * FS + j * kHX];
#pragma unroll
            for (int o = 0; o < 4; ++o)
                if (j - o >= 0 && j - o <= 2 * R) {
                    ixx[o] = fmaf(tp.g[j - o], v2, ixx[o]);
                    iyy[o] = fmaf(tp.g2[j - o], v0, iyy[o]);
                    ixy[o] = fmaf(tp.g1[j - o], v1, ixy[o]);
                }
        }
        if (x0 + lane < nx) {
#pragma unroll
            for (int o = 0; o < 4; ++o) {
                if (y0 + r0 + o < ny) {
                    const float d = ixx[o] + iyy[o] < 0.f ? s4 * (ixx[o] * iyy[o] - ixy[o] * ixy[o]) : -INFINITY;
                    D[slice + (long long)(y0 + r0 + o) * nx + x0 + lane] = d;
                    best = fmaxf(best, d);
                }
            }
        }
    }
    for (int o = 16; o > 0; o >>= 1) best = fmaxf(best, __shfl_xor_sync(0xffffffffu, best, o));
    if (lane == 0) red[warp] = best;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < kHThreads / 32; ++w) best = fmaxf(best, red[w]);
        atomicMax(smax + blockIdx.z, max_key(best));
    }
}

template <class T, int... R>
void launch_hessian_r(std::integer_sequence<int, R...>, dim3 grid, size_t sm, const T *img, float *D, int *smax, int nx,
                      int ny, const DerivTaps &tp, float s4, cudaStream_t s) {
    using Kernel = void (*)(const T *, float *, int *, int, int, DerivTaps, float);
    constexpr Kernel kernels[] = {k_hessian<T, R>...};
    kernels[tp.R]<<<grid, kHThreads, sm, s>>>(img, D, smax, nx, ny, tp, s4);
}
template <class T>
void launch_hessian(const void *img, float *D, int *smax, int nx, int ny, int nz, const DerivTaps &tp, float s4,
                    cudaStream_t s) {
    const dim3 grid((unsigned)((nx + kHT - 1) / kHT), (unsigned)((ny + kHT - 1) / kHT), (unsigned)nz);
    const size_t sm = sizeof(float) * (size_t)(kHT + 2 * tp.R) * (hessian_pitch(tp.R) + 3 * kHX);  // at most 45 KB
    launch_hessian_r(std::make_integer_sequence<int, kMaxR + 1>{}, grid, sm, static_cast<const T *>(img), D, smax, nx, ny,
                     tp, s4, s);
}

// Seeds of 32 columns x kSeedRows rows of a slice: above t times the slice maximum and above
// each neighbour.
constexpr int kSeedRows = 64;
__global__ void __launch_bounds__(256) k_seeds(const float *__restrict__ D, const int *__restrict__ smax,
                                               uint8_t *__restrict__ mask, unsigned long long *__restrict__ count,
                                               int nx, int ny, float t) {
    const int x = blockIdx.x * 32 + (threadIdx.x & 31);
    const int y1 = min(ny, (int)(blockIdx.y + 1) * kSeedRows);
    const float m = key_value(smax[blockIdx.z]), tm = t * m;
    unsigned found = 0;
    if (x < nx) {
#pragma unroll 4
        for (int y = blockIdx.y * kSeedRows + (threadIdx.x >> 5); y < y1; y += 8) {
            const long long i = ((long long)blockIdx.z * ny + y) * nx + x;
            const float v = D[i];
            bool seed = m > 0.f && v > tm;
            if (seed) {
                for (int dy = -1; dy <= 1; ++dy)
                    for (int dx = -1; dx <= 1; ++dx) {
                        if (dx == 0 && dy == 0) continue;
                        const int xx = x + dx, yy = y + dy;
                        if (xx < 0 || xx >= nx || yy < 0 || yy >= ny) continue;
                        if (!(v > D[i + (long long)dy * nx + dx])) seed = false;
                    }
            }
            mask[i] = seed ? 1 : 0;
            found += seed;
        }
    }
    found = __reduce_add_sync(0xffffffffu, found);
    if (found && (threadIdx.x & 31) == 0) atomicAdd(count, (unsigned long long)found);
}

constexpr unsigned kNoSeed = 0xffffu;  // no seed in the row (distances are at most 4095)

// Distance to the nearest seed of the row: one warp per row, its seeds as bits in shared memory.
__global__ void __launch_bounds__(256) k_dist_x(const uint8_t *__restrict__ mask, uint16_t *__restrict__ out, int nx,
                                                long long nrows) {
    __shared__ unsigned bits[8][kMaxLine / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned *const w = bits[warp];
    const int nw = (nx + 31) / 32;
    for (long long r = blockIdx.x * 8LL + warp; r < nrows; r += gridDim.x * 8LL) {
        const uint8_t *const m = mask + r * nx;
        unsigned any = 0;
        for (int k = 0; k < nw; ++k) {
            const int x = k * 32 + lane;
            const unsigned b = __ballot_sync(0xffffffffu, x < nx && m[x] != 0);
            if (lane == 0) w[k] = b;
            any |= b;
        }
        __syncwarp();
        for (int k = 0; k < nw; ++k) {
            const int x = k * 32 + lane;
            unsigned best = kNoSeed;
            if (any) {
                const unsigned lo = w[k] << (31 - lane), hi = w[k] >> lane;  // bits at and left of, at and right of x
                if (lo) best = min(best, (unsigned)__clz(lo));
                if (hi) best = min(best, (unsigned)(__ffs(hi) - 1));
                for (int j = k - 1; j >= 0; --j)  // the nearest earlier and later words with a seed
                    if (w[j]) {
                        best = min(best, (unsigned)(x - (j * 32 + 31 - __clz(w[j]))));
                        break;
                    }
                for (int j = k + 1; j < nw; ++j)
                    if (w[j]) {
                        best = min(best, (unsigned)(j * 32 + __ffs(w[j]) - 1 - x));
                        break;
                    }
            }
            if (x < nx) out[r * nx + x] = (uint16_t)best;
        }
        __syncwarp();
    }
}

// One axis of the squared distance transform: min over j of in(j) + (i - j)^2 along lines of
// `len` values `stride` apart, WC adjacent columns (x) per block; blockIdx.y: the line's other
// coordinate, `other` apart.  FIRST: the input is k_dist_x's distances (squared here);
// LAST: the output is r0 - sqrt(minimum), written only where there is a seed at all.
// Squared distances are integers below 2^24: every sum is exact.  384^3, light-sheet seeds:
// 0.63 ms along y and 0.54 ms along z, phi0 included (6.1 ms each over whole lines); bound by
// instruction issue in the searches.
template <bool FIRST, bool LAST, int WC>
__global__ void __launch_bounds__(512) k_dist_line(const void *__restrict__ in, float *__restrict__ out, int nx,
                                                   int len, long long stride, long long other, float r0,
                                                   const unsigned long long *__restrict__ count) {
    extern __shared__ float line[];  // [groups * kGroup][WC], then the group minima [groups][WC]
    if (LAST && *count == 0) return;
    const int c = threadIdx.x % WC, t0 = threadIdx.x / WC;
    constexpr int ROWS = 512 / WC;
    const int x = blockIdx.x * WC + c;
    const long long base = blockIdx.y * other + x;
    const int ng = (len + kGroup - 1) / kGroup;
    float *const gmin = line + ng * kGroup * WC;
    if (x < nx) {
        for (int j = t0; j < ng * kGroup; j += ROWS) {
            float v = INFINITY;  // past the end
            if (j >= len) {
            } else if (FIRST) {
                const unsigned d = static_cast<const uint16_t *>(in)[base + j * stride];
                v = d == kNoSeed ? INFINITY : (float)(d * d);
            } else {
                v = static_cast<const float *>(in)[base + j * stride];
            }
            line[j * WC + c] = v;
        }
    }
    __syncthreads();
    if (x < nx) {
        for (int g = t0; g < ng; g += ROWS) {
            float m = INFINITY;
#pragma unroll
            for (int k = 0; k < kGroup; ++k) m = fminf(m, line[(g * kGroup + k) * WC + c]);
            gmin[g * WC + c] = m;
        }
    }
    __syncthreads();
    if (x >= nx) return;
    for (int i = t0; i < len; i += ROWS) {
        const int g0 = i / kGroup;
        float best = INFINITY;
        const auto scan = [&](int g, float d0) {  // d0 = i minus the group's first place
            const float *const l = line + g * kGroup * WC + c;
#pragma unroll
            for (int k = 0; k < kGroup; ++k) {
                const float d = d0 - (float)k;
                best = fminf(best, fmaf(d, d, l[k * WC]));
            }
        };
        const float d0 = (float)(i - g0 * kGroup);
        scan(g0, d0);
        float dl = d0 + 1.f, dr = (float)kGroup - d0;  // to the nearest place of the groups on both sides
        for (int s = 1;; ++s, dl += (float)kGroup, dr += (float)kGroup) {
            const int gl = g0 - s, gr = g0 + s;
            const bool left = gl >= 0 && dl * dl < best, right = gr < ng && dr * dr < best;
            if (!left && !right) break;
            if (left && fmaf(dl, dl, gmin[gl * WC + c]) < best) scan(gl, dl + (float)(kGroup - 1));
            if (right && fmaf(dr, dr, gmin[gr * WC + c]) < best) scan(gr, -dr);
        }
        out[base + i * stride] = LAST ? r0 - sqrtf(best) : best;
    }
}

// Launches one axis: 32 columns per block where a line of 32 columns fits shared memory,
// else 8 (4096 values: 147 KB).
template <bool FIRST, bool LAST>
cudaError_t dist_line(const void *in, float *out, int nx, int len, long long stride, int nother, long long other,
                      float r0, const unsigned long long *count, cudaStream_t s) {
    const int groups = (len + kGroup - 1) / kGroup;
    const size_t per = sizeof(float) * (size_t)(groups * kGroup + groups);
    cudaError_t e;
    if (per * 32 <= 200 * 1024) {
        e = cudaFuncSetAttribute(k_dist_line<FIRST, LAST, 32>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
        if (e != cudaSuccess) return e;
        k_dist_line<FIRST, LAST, 32><<<dim3((nx + 31) / 32, nother), 512, per * 32, s>>>(in, out, nx, len, stride, other, r0, count);
    } else {
        e = cudaFuncSetAttribute(k_dist_line<FIRST, LAST, 8>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
        if (e != cudaSuccess) return e;
        k_dist_line<FIRST, LAST, 8><<<dim3((nx + 7) / 8, nother), 512, per * 8, s>>>(in, out, nx, len, stride, other, r0, count);
    }
    return cudaGetLastError();
}

}  // namespace

extern "C" rsf_status rsf_init_phi0(rsf_ctx *c, const void *volume, rsf_dtype vt, int64_t nx, int64_t ny, int64_t nz,
                                    float blob_sigma, float rel_threshold, float r0, float *phi0_out,
                                    int64_t *nseeds, uint8_t *seeds_out, float *response_out) {
    if (!c) return fail(RSF_E_INVAL, "null context");
    if (!volume || !phi0_out || !nseeds) return fail(RSF_E_INVAL, "null volume, phi0_out or nseeds pointer");
    if (vt != RSF_U8 && vt != RSF_U16 && vt != RSF_F32) return fail(RSF_E_INVAL, "unknown volume dtype %d", (int)vt);
    if (nx < 4 || ny < 4 || nz < 1 || nx > (1 << 20) || ny > (1 << 20) || nz > (1 << 20))
        return fail(RSF_E_INVAL, "dimensions must lie in [4, 2^20] (x, y) and [1, 2^20] (z)");
    if ((double)nx * ny * nz > 17179869184.0) return fail(RSF_E_INVAL, "nx*ny*nz exceeds 2^34");
    if ((double)(nx - 1) * (nx - 1) + (double)(ny - 1) * (ny - 1) + (double)(nz - 1) * (nz - 1) >= 16777216.0)
        return fail(RSF_E_INVAL, "squared distances would exceed 2^24 (exact FP32 range)");
    if (!(blob_sigma > 0.f) || std::floor(3.0 * blob_sigma + 0.5) > kMaxR)
        return fail(RSF_E_INVAL, "blob sigma must be positive with round(3 sigma) <= %d", kMaxR);
    if (!(rel_threshold >= 0.f && rel_threshold < 1.f)) return fail(RSF_E_INVAL, "relative threshold must lie in [0, 1)");
    if (!(r0 > 0.f) || !std::isfinite(r0)) return fail(RSF_E_INVAL, "r0 must be positive and finite");

    const long long n = nx * ny * nz, plane = nx * ny;
    const size_t es = dtype_size(vt);
    auto align = [](size_t b) { return (b + 255) & ~size_t(255); };
    const bool host_vol = !on_device(volume), host_phi = !in_place(phi0_out, c->device);
    // destinations that this device's kernels may write are written in place, unless they share
    // memory with something still read
    const size_t fb = sizeof(float) * (size_t)n;
    const bool shared = share_bytes(response_out, fb, seeds_out, n);
    const bool own_D = !response_out || !in_place(response_out, c->device) || shared || share_bytes(response_out, fb, volume, es * n);
    const bool own_mask = !seeds_out || !in_place(seeds_out, c->device, 1) || shared || share_bytes(seeds_out, n, volume, es * n);
    size_t bytes = align(sizeof(uint16_t) * n) + align(sizeof(float) * n) + align(sizeof(int) * nz) + 256;
    if (own_D) bytes += align(sizeof(float) * n);
    if (own_mask) bytes += align(n);
    if (host_phi) bytes += align(sizeof(float) * n);
    if (host_vol) bytes += align(es * n);
    void *mem = nullptr;
    rsf_status st = dev_alloc(c, &mem, bytes);
    if (st) return st;
    struct Release {
        rsf_ctx *c;
        void *p;
        size_t b;
        ~Release() { dev_free(c, p, b); }
    } release{c, mem, bytes};
    char *p = static_cast<char *>(mem);
    auto take = [&](size_t b) {
        char *q = p;
        p += align(b);
        return q;
    };
    uint16_t *dx = reinterpret_cast<uint16_t *>(take(sizeof(uint16_t) * n));  // distance along x
    float *dxy = reinterpret_cast<float *>(take(sizeof(float) * n));          // squared, within the slice
    int *smax = reinterpret_cast<int *>(take(sizeof(int) * nz));
    unsigned long long *count = reinterpret_cast<unsigned long long *>(take(sizeof(unsigned long long)));
    float *D = own_D ? reinterpret_cast<float *>(take(sizeof(float) * n)) : response_out;
    uint8_t *mask = own_mask ? reinterpret_cast<uint8_t *>(take(n)) : seeds_out;
    float *phi = host_phi ? reinterpret_cast<float *>(take(sizeof(float) * n)) : phi0_out;

    std::lock_guard<std::mutex> lk(c->mu);
    RSF_CUDA(cudaSetDevice(c->device));
    cudaStream_t s = c->stream;
    const void *img = volume;
    if (host_vol) {
        void *d = take(es * n);
        RSF_CUDA(xfer(d, volume, es * n, s));
        img = d;
    }
    const DerivTaps tp = make_deriv_taps(blob_sigma);
    const float s2 = blob_sigma * blob_sigma;
    RSF_CUDA(cudaMemsetAsync(smax, 0x80, sizeof(int) * nz, s));  // a key below those of all values but -inf
    RSF_CUDA(cudaMemsetAsync(count, 0, sizeof(unsigned long long), s));
    switch (vt) {
        case RSF_U8: launch_hessian<uint8_t>(img, D, smax, (int)nx, (int)ny, (int)nz, tp, s2 * s2, s); break;
        case RSF_U16: launch_hessian<uint16_t>(img, D, smax, (int)nx, (int)ny, (int)nz, tp, s2 * s2, s); break;
        default: launch_hessian<float>(img, D, smax, (int)nx, (int)ny, (int)nz, tp, s2 * s2, s);
    }
    k_seeds<<<dim3((unsigned)((nx + 31) / 32), (unsigned)((ny + kSeedRows - 1) / kSeedRows), (unsigned)nz), 256, 0, s>>>(D, smax, mask, count, (int)nx, (int)ny, rel_threshold);
    k_dist_x<<<(unsigned)std::min<long long>(4864, (ny * nz + 7) / 8), 256, 0, s>>>(mask, dx, (int)nx, ny * nz);
    RSF_CUDA(cudaGetLastError());
    // outputs that share memory are written in the order response, mask, phi0
    if (response_out && own_D) RSF_CUDA(xfer(response_out, D, fb, s));
    if (seeds_out && own_mask) RSF_CUDA(xfer(seeds_out, mask, n, s));
    RSF_CUDA((dist_line<true, false>(dx, dxy, (int)nx, (int)ny, nx, (int)nz, plane, r0, count, s)));
    RSF_CUDA((dist_line<false, true>(dxy, phi, (int)nx, (int)nz, plane, (int)ny, nx, r0, count, s)));
    unsigned long long found = 0;
    RSF_CUDA(cudaMemcpyAsync(&found, count, sizeof(found), cudaMemcpyDeviceToHost, s));
    RSF_CUDA(cudaStreamSynchronize(s));
    *nseeds = (int64_t)found;
    if (found && host_phi) RSF_CUDA(xfer(phi0_out, phi, sizeof(float) * n, s));
    RSF_CUDA(cudaStreamSynchronize(s));
    if (found == 0) return fail(RSF_E_INVAL, "no seed found (relative threshold %g)", (double)rel_threshold);
    return RSF_OK;
}

// ------------------------------------------------------------ validation

namespace {

// Counts |phi > 0|, |truth != 0| and their intersection (warp sums, one atomic
// per warp per count).
__global__ void k_overlap(const float *__restrict__ phi, const uint8_t *__restrict__ truth, long long n,
                          unsigned long long *__restrict__ out) {
    unsigned long long a = 0, b = 0, c = 0;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const bool s = phi[i] > 0.f, t = truth[i] != 0;
        a += s;
        b += t;
        c += s && t;
    }
    for (int o = 16; o > 0; o >>= 1) {
        a += __shfl_down_sync(0xffffffffu, a, o);
        b += __shfl_down_sync(0xffffffffu, b, o);
        c += __shfl_down_sync(0xffffffffu, c, o);
    }
    if ((threadIdx.x & 31) == 0) {
        atomicAdd(out + 0, a);
        atomicAdd(out + 1, b);
        atomicAdd(out + 2, c);
    }
}

}  // namespace

extern "C" rsf_status rsf_overlap(rsf_ctx *c, const float *phi, const uint8_t *truth, int64_t n, int64_t counts[3]) {
    if (!c) return fail(RSF_E_INVAL, "null context");
    if (!phi || !truth || !counts) return fail(RSF_E_INVAL, "null phi, truth or counts pointer");
    if (n < 0 || n > (int64_t)1 << 34) return fail(RSF_E_INVAL, "n must lie in [0, 2^34]");
    auto align = [](size_t b) { return (b + 255) & ~size_t(255); };
    const bool host_phi = !on_device(phi), host_truth = !on_device(truth);
    size_t bytes = 256 + (host_phi ? align(sizeof(float) * n) : 0) + (host_truth ? align(n) : 0);
    void *mem = nullptr;
    rsf_status st = dev_alloc(c, &mem, bytes);
    if (st) return st;
    struct Release {
        rsf_ctx *c;
        void *p;
        size_t b;
        ~Release() { dev_free(c, p, b); }
    } release{c, mem, bytes};
    char *p = static_cast<char *>(mem);
    unsigned long long *out = reinterpret_cast<unsigned long long *>(p);
    p += 256;
    std::lock_guard<std::mutex> lk(c->mu);
    RSF_CUDA(cudaSetDevice(c->device));
    cudaStream_t s = c->stream;
    if (host_phi) {
        RSF_CUDA(xfer(p, phi, sizeof(float) * n, s));
        phi = reinterpret_cast<const float *>(p);
        p += align(sizeof(float) * n);
    }
    if (host_truth) {
        RSF_CUDA(xfer(p, truth, n, s));
        truth = reinterpret_cast<const uint8_t *>(p);
    }
    RSF_CUDA(cudaMemsetAsync(out, 0, 3 * sizeof(unsigned long long), s));
    if (n > 0) {
        k_overlap<<<(int)std::min<long long>(1216, (n + 255) / 256), 256, 0, s>>>(phi, truth, n, out);
        RSF_CUDA(cudaGetLastError());
    }
    unsigned long long h[3];
    RSF_CUDA(cudaMemcpyAsync(h, out, sizeof(h), cudaMemcpyDeviceToHost, s));
    RSF_CUDA(cudaStreamSynchronize(s));
    for (int k = 0; k < 3; ++k) counts[k] = (int64_t)h[k];
    return RSF_OK;
}
