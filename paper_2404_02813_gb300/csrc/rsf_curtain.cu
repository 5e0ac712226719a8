// rsf_curtain.cu -- rsf_evolve_curtain: the volume-level parallelism of
// arXiv 2404.02813, Sec. 4.1.  The volume is divided into overlapping
// sub-volumes, every sub-volume is evolved as a volume of its own (all of them
// together, through rsf_evolve_batch), and neighbouring results are merged by
// linear interpolation across the overlap (the curtain).
//
// Layout along each axis of length n: sub-volumes of `edge` voxels start at
// multiples of edge - curtain and the last one is moved to end at n (a single
// sub-volume when edge >= n).  Sub-volume b carries the weight
// w_b(x) = prod over axes of h_b(x_a), with h = 1 inside, rising linearly
// over the `curtain` voxels next to each face interior to the volume:
// h = min(1, (x - s + 1/2) / curtain) after a start face s > 0 and
// min(1, (e - x - 1/2) / curtain) before an end face e < n.  The merged phi is
// sum_b w_b phi_b / sum_b w_b; across an overlap of exactly `curtain` voxels
// this is the linear interpolation between the two neighbours.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <mutex>
#include <vector>

#include "rsf.h"
#include "rsf_ctx.h"

namespace {

constexpr int kMaxCover = 4;  // sub-volumes covering one coordinate of an axis (at most 3 when curtain <= edge/2)

std::vector<int> starts_of(int n, int edge, int curtain) {
    std::vector<int> s;
    if (edge >= n) {
        s.push_back(0);
        return s;
    }
    for (int a = 0; a < n - edge; a += edge - curtain) s.push_back(a);
    s.push_back(n - edge);
    return s;
}

// Per coordinate of one axis: the covering sub-volumes, the coordinate local to
// each and the axis factor h of its weight.
struct AxisTable {
    std::vector<int> count, box, local;
    std::vector<float> weight;
};

bool axis_table(int n, int edge, int curtain, const std::vector<int> &starts, AxisTable *t) {
    t->count.assign(n, 0);
    t->box.assign((size_t)n * kMaxCover, 0);
    t->local.assign((size_t)n * kMaxCover, 0);
    t->weight.assign((size_t)n * kMaxCover, 0.f);
    for (int k = 0; k < (int)starts.size(); ++k) {
        const int s = starts[k], e = std::min(s + edge, n);
        for (int x = s; x < e; ++x) {
            double h = 1.0;
            if (s > 0) h = std::min(h, (x - s + 0.5) / curtain);
            if (e < n) h = std::min(h, (e - x - 0.5) / curtain);
            const int c = t->count[x]++;
            if (c >= kMaxCover) return false;
            t->box[(size_t)x * kMaxCover + c] = k;
            t->local[(size_t)x * kMaxCover + c] = x - s;
            t->weight[(size_t)x * kMaxCover + c] = (float)std::max(h, 0.0);
        }
    }
    return true;
}

// Every sub-volume's image and phi0 in one launch: blockIdx.y is the sub-volume, a warp copies
// rows (one element per thread with 64-bit divisions: 22 us per array of 160^3; 12 images and level
// sets here: 90 us, the copy rate).
struct GatherArgs {
    int step;                 // sub-volume k of an axis starts at min(k step, n - ext) (starts_of)
    int nb[3], ext[3], n[3];  // sub-volumes, their extents and the volume's, per axis (x, y, z)
    int first;                // blockIdx.y = 0's sub-volume (a launch takes at most 32768)
    char *box0;               // sub-volume id's image and phi at box0 + id * stride
    size_t stride, phi_at;
};
template <class T>
__global__ void __launch_bounds__(256) k_gather(const T *__restrict__ vol, const float *__restrict__ phi0, GatherArgs a) {
    const int id = a.first + blockIdx.y, kx = id % a.nb[0], ky = id / a.nb[0] % a.nb[1], kz = id / a.nb[0] / a.nb[1];
    const int bx = a.ext[0], by = a.ext[1];
    const int x0 = min(kx * a.step, a.n[0] - bx), y0 = min(ky * a.step, a.n[1] - by);
    const int z0 = min(kz * a.step, a.n[2] - a.ext[2]);
    const long long rows = (long long)by * a.ext[2];
    T *const img = reinterpret_cast<T *>(a.box0 + id * a.stride);
    float *const phi = reinterpret_cast<float *>(a.box0 + id * a.stride + a.phi_at);
    const int lane = threadIdx.x & 31;
    for (long long r = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5; r < rows;
         r += ((long long)gridDim.x * blockDim.x) >> 5) {
        const int y = (int)(r % by), z = (int)(r / by);
        const long long src = ((long long)(z0 + z) * a.n[1] + y0 + y) * a.n[0] + x0;
        for (int x = lane; x < bx; x += 32) {
            img[r * bx + x] = vol[src + x];
            phi[r * bx + x] = phi0[src + x];
        }
    }
}

struct MergeArgs {
    const float *const *phi;  // per sub-volume (bz, by, bx) in z-major order, its evolved phi
    const int *ext[3];        // sub-volume extent per axis index (x, y, z)
    const int *count[3], *box[3], *local[3];
    const float *weight[3];
    int n[3], nb[3];
};

// A warp per output row: the y and z tables are read once per row.  A voxel's sum is a chain of
// table, pointer and value loads (0.12 of the copy rate with one voxel at a time per lane), so a
// lane sums four columns side by side, the x tables of their first sub-volume read up front (most
// columns have no other).  320 x 288 x 256 from 12
// sub-volumes of 160^3: 0.237 -> 0.175 ms, still the chain per row and sub-volume.
constexpr int kMergeCols = 4;
__global__ void __launch_bounds__(256) k_merge(MergeArgs a, float *__restrict__ out) {
    const int nx = a.n[0], lane = threadIdx.x & 31;
    const long long rows = (long long)a.n[1] * a.n[2];
    for (long long r = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5; r < rows;
         r += ((long long)gridDim.x * blockDim.x) >> 5) {
        const int y = (int)(r % a.n[1]), z = (int)(r / a.n[1]);
        const int cz = __ldg(a.count[2] + z), cy = __ldg(a.count[1] + y);
        for (int x0 = lane; x0 < nx; x0 += 32 * kMergeCols) {
            float num[kMergeCols], den[kMergeCols], w0[kMergeCols];
            int cx[kMergeCols], k0[kMergeCols], l0[kMergeCols], e0[kMergeCols];
            int most = 0;
#pragma unroll
            for (int c = 0; c < kMergeCols; ++c) {
                const int x = min(x0 + 32 * c, nx - 1);  // a column past the row repeats the last one
                cx[c] = __ldg(a.count[0] + x);
                k0[c] = __ldg(a.box[0] + x * kMaxCover);
                l0[c] = __ldg(a.local[0] + x * kMaxCover);
                w0[c] = __ldg(a.weight[0] + x * kMaxCover);
                num[c] = den[c] = 0.f;
            }
#pragma unroll
            for (int c = 0; c < kMergeCols; ++c) {
                e0[c] = __ldg(a.ext[0] + k0[c]);
                most = max(most, cx[c]);
            }
            for (int iz = 0; iz < cz; ++iz) {
                const int kz = __ldg(a.box[2] + z * kMaxCover + iz), lz = __ldg(a.local[2] + z * kMaxCover + iz);
                const float wz = __ldg(a.weight[2] + z * kMaxCover + iz);
                for (int iy = 0; iy < cy; ++iy) {
                    const int ky = __ldg(a.box[1] + y * kMaxCover + iy), ly = __ldg(a.local[1] + y * kMaxCover + iy);
                    const float wzy = wz * __ldg(a.weight[1] + y * kMaxCover + iy);
                    const long long row = (long long)lz * __ldg(a.ext[1] + ky) + ly;
                    const float *const *const phi = a.phi + ((long long)kz * a.nb[1] + ky) * a.nb[0];
                    const float *p[kMergeCols];
                    float v[kMergeCols];
#pragma unroll
                    for (int c = 0; c < kMergeCols; ++c) p[c] = phi[k0[c]];
#pragma unroll
                    for (int c = 0; c < kMergeCols; ++c) v[c] = __ldg(p[c] + row * e0[c] + l0[c]);
#pragma unroll
                    for (int c = 0; c < kMergeCols; ++c) {
                        const float w = wzy * w0[c];
                        num[c] = fmaf(w, v[c], num[c]);
                        den[c] += w;
                    }
                    for (int ix = 1; ix < most; ++ix)
#pragma unroll
                        for (int c = 0; c < kMergeCols; ++c)
                            if (ix < cx[c]) {
                                const int i = min(x0 + 32 * c, nx - 1) * kMaxCover + ix, kx = __ldg(a.box[0] + i);
                                const float w = wzy * __ldg(a.weight[0] + i);
                                num[c] = fmaf(w, __ldg(phi[kx] + row * __ldg(a.ext[0] + kx) + __ldg(a.local[0] + i)), num[c]);
                                den[c] += w;
                            }
                }
            }
#pragma unroll
            for (int c = 0; c < kMergeCols; ++c)
                if (x0 + 32 * c < nx) out[r * nx + x0 + 32 * c] = num[c] / den[c];
        }
    }
}

}  // namespace

extern "C" rsf_status rsf_evolve_curtain(rsf_ctx *c, const void *volume, rsf_dtype vt, int64_t nx, int64_t ny,
                                         int64_t nz, const float *phi0, float *phi_out, float sigma, float eps,
                                         float lambda1, float lambda2, float nu, float mu, float dt, int32_t iters,
                                         int32_t edge, int32_t curtain) {
    if (!c) return fail(RSF_E_INVAL, "null context");
    rsf_status st = check_args(volume, vt, nx, ny, nz, phi0, phi_out, sigma, eps, dt, iters);
    if (st) return st;
    if (edge < 4) return fail(RSF_E_INVAL, "sub-volume edge %d is below 4", (int)edge);
    if (curtain < 1 || 2 * curtain > edge)
        return fail(RSF_E_INVAL, "curtain %d must lie in [1, edge/2] (edge %d)", (int)curtain, (int)edge);
    const int n[3] = {(int)nx, (int)ny, (int)nz};
    std::vector<int> starts[3];
    AxisTable tab[3];
    for (int a = 0; a < 3; ++a) {
        starts[a] = starts_of(n[a], edge, curtain);
        if (!axis_table(n[a], edge, curtain, starts[a], &tab[a]))
            return fail(RSF_E_INVAL, "more than %d sub-volumes cover one coordinate", kMaxCover);
    }
    const int nb[3] = {(int)starts[0].size(), (int)starts[1].size(), (int)starts[2].size()};
    const long long nbox = (long long)nb[0] * nb[1] * nb[2];
    const size_t es = dtype_size(vt);
    const long long nvox = (long long)nx * ny * nz;

    // device memory: sub-volume images and phi, staging of host inputs and output, tables
    size_t bytes = 0;
    auto align = [](size_t b) { return (b + 255) & ~size_t(255); };
    const int ext[3] = {std::min(edge, n[0]), std::min(edge, n[1]), std::min(edge, n[2])};
    const long long bvox = (long long)ext[0] * ext[1] * ext[2];  // every sub-volume has these extents
    const size_t stride = align(es * bvox) + align(sizeof(float) * bvox);
    bytes += stride * nbox;
    const bool host_vol = !on_device(volume), host_phi = !on_device(phi0), host_out = !on_device(phi_out);
    if (host_vol) bytes += align(es * nvox);
    if (host_phi) bytes += align(sizeof(float) * nvox);
    if (host_out) bytes += align(sizeof(float) * nvox);
    size_t tab_bytes = sizeof(float *) * nbox;
    for (int a = 0; a < 3; ++a)
        tab_bytes += sizeof(int) * (nb[a] + n[a] * (1 + 2 * kMaxCover)) + sizeof(float) * n[a] * kMaxCover;
    bytes += align(tab_bytes) + 1024;
    void *mem = nullptr;
    if ((st = dev_alloc(c, &mem, bytes))) return st;
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

    std::vector<rsf_brick> bricks(nbox);
    std::vector<const float *> phis(nbox);
    MergeArgs m{};
    HostCopies copies(c->stream);
    {
        std::lock_guard<std::mutex> lk(c->mu);
        RSF_CUDA(cudaSetDevice(c->device));
        const void *vol = volume;
        const float *ph0 = phi0;
        if (host_vol) {
            void *d = take(es * nvox);
            RSF_CUDA(xfer(d, volume, es * nvox, c->stream));
            vol = d;
        }
        if (host_phi) {
            float *d = reinterpret_cast<float *>(take(sizeof(float) * nvox));
            RSF_CUDA(xfer(d, phi0, sizeof(float) * nvox, c->stream));
            ph0 = d;
        }
        GatherArgs ga{};
        ga.box0 = take(stride * nbox);
        ga.stride = stride;
        ga.step = edge - curtain;
        ga.phi_at = align(es * bvox);
        for (long long id = 0; id < nbox; ++id) {
            char *const box = ga.box0 + id * stride;
            float *const ph = reinterpret_cast<float *>(box + ga.phi_at);
            bricks[id] = rsf_brick{box, vt, ext[0], ext[1], ext[2], ph, ph, sigma, eps, lambda1, lambda2, nu, mu, dt, iters};
            phis[id] = ph;
        }
        char *tb = take(tab_bytes);
        std::vector<char> host_tab(tab_bytes);
        size_t off = 0;
        auto put = [&](const void *src, size_t b) {
            memcpy(host_tab.data() + off, src, b);
            const char *d = tb + off;
            off += b;
            return d;
        };
        m.phi = reinterpret_cast<const float *const *>(put(phis.data(), sizeof(float *) * nbox));
        for (int a = 0; a < 3; ++a) {
            std::vector<int> exts(nb[a], ext[a]);
            m.ext[a] = reinterpret_cast<const int *>(put(exts.data(), sizeof(int) * nb[a]));
            m.count[a] = reinterpret_cast<const int *>(put(tab[a].count.data(), sizeof(int) * n[a]));
            m.box[a] = reinterpret_cast<const int *>(put(tab[a].box.data(), sizeof(int) * n[a] * kMaxCover));
            m.local[a] = reinterpret_cast<const int *>(put(tab[a].local.data(), sizeof(int) * n[a] * kMaxCover));
            m.weight[a] = reinterpret_cast<const float *>(put(tab[a].weight.data(), sizeof(float) * n[a] * kMaxCover));
            ga.nb[a] = nb[a];
            ga.ext[a] = ext[a];
            ga.n[a] = n[a];
            m.n[a] = n[a];
            m.nb[a] = nb[a];
        }
        host_tab.resize(off);
        RSF_CUDA(copies.put(tb, std::move(host_tab)));
        for (long long first = 0; first < nbox; first += 32768) {
            ga.first = (int)first;
            const dim3 grid((unsigned)std::min<long long>(((long long)ext[1] * ext[2] + 7) / 8, nbox >= 16 ? 152 : 1216),
                            (unsigned)std::min<long long>(32768, nbox - first));
            switch (vt) {
                case RSF_U8: k_gather<<<grid, 256, 0, c->stream>>>(static_cast<const uint8_t *>(vol), ph0, ga); break;
                case RSF_U16: k_gather<<<grid, 256, 0, c->stream>>>(static_cast<const uint16_t *>(vol), ph0, ga); break;
                default: k_gather<<<grid, 256, 0, c->stream>>>(static_cast<const float *>(vol), ph0, ga);
            }
        }
        RSF_CUDA(cudaGetLastError());
    }
    // every sub-volume evolved as its own volume, all together (same stream, so
    // the gathers above are ordered before the batch's first launch)
    if ((st = rsf_evolve_batch(c, bricks.data(), (int32_t)nbox))) return st;

    std::lock_guard<std::mutex> lk(c->mu);
    float *out = host_out ? reinterpret_cast<float *>(take(sizeof(float) * nvox)) : phi_out;
    k_merge<<<(unsigned)std::min<long long>(4864, ((long long)ny * nz + 7) / 8), 256, 0, c->stream>>>(m, out);
    RSF_CUDA(cudaGetLastError());
    if (host_out) RSF_CUDA(xfer(phi_out, out, sizeof(float) * nvox, c->stream));
    RSF_CUDA(cudaStreamSynchronize(c->stream));
    copies.done();
    return RSF_OK;
}
