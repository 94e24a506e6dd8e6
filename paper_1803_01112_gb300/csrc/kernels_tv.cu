// TV kernels: gradient of phi_eps with its FP64 norm, phi in FP64, and the perturbation
// x <- x + beta v, v = -g/||g|| (arXiv 1803.01112, Appendix A/C; phi = TV as the sum of
// local variations, introduced in Sec. II).  Forward differences on index spacing, zero past the last
// index.  The image is tiny next to the system matrix (V floats), so these kernels live
// in L2; every reduction is FP64 with a fixed reduction order (deterministic).
#include <algorithm>

#include "common.cuh"
#include "voxel_coords.cuh"

namespace ntvs {

int red_grid(int64_t n, int sm_count) {
    int64_t need = (n + kRedThreads - 1) / kRedThreads;
    int64_t cap = (int64_t)sm_count * 8;
    if (need < 1) need = 1;
    return (int)(need < cap ? need : cap);
}

// n / D for several n and D = sqrt(s): every product n (1/D) corrected by its residual
// (Markstein 1990), 3 FP64 operations a quotient instead of a division.  D outside the range
// where the residual is exact divides.
struct Quotients {
    double D, r;
    bool safe;
    __device__ __forceinline__ explicit Quotients(double s) {
        D = sqrt_and_inverse(s, &r);
        const int e = __double2hiint(D);   // 2^-400 < D < 2^400
        safe = e > 0x26f00000 && e < 0x58f00000;
    }
    __device__ __forceinline__ double operator()(double n) const {
        if (!safe) return D > 0.0 ? n / D : 0.0;
        const double q = n * r;
        return fma(fma(-q, D, n), r, q);
    }
};

// FP64 path, images that fill them: grad phi_eps on tiles of 31 x (TY - 1) voxels, marching along z:
//   g_q = -sum_a d_a(q) / D_q + sum_{a: q-e_a inside} d_a(q-e_a) / D_{q-e_a}
// with d_a(c) = x_{c+e_a} - x_c (0 past the last index) and D_c = sqrt(eps + |d(c)|^2).
// Every voxel of the tile and of its low halo forms its three quotients d_a / D once; the x and
// y ones go to the next voxels through shared memory, the z one stays in the thread for the
// next slice.
// One thread per voxel forming all four D's of its stencil itself spent 4 square roots and 6
// divisions a voxel on a pipe of 2 lanes per clock and SM: 145 us on 200x200x16, 67 us here.
// The FP32 path is bound by the latency of its loads instead and keeps one thread per voxel
// (tiles: 7.5 against 5.5 us on 41x37x5, 58 against 59 us on 256x256x64).
// PHI: also phi_0(x).
//
// TY: threads of a tile in y.  16 where the tiles fill the SMs; an image of few tiles takes 4 (a
// quarter of the FP64 work on each of four times as many SMs, for a halo of a row in 3): 10.2 us
// with 16 and 5.5 us with 4 on 32x32x1.
constexpr int kGradTx = 32;   // threads of a tile in x: its voxels and one low halo column

template <bool PHI, int kGradTy>
__global__ void __launch_bounds__(kGradTx * kGradTy)
tv_grad_tile_kernel(const double* __restrict__ x, double* __restrict__ g, int nx, int ny, int nz, double eps, int zc,
                    int tiles_x, int tiles, int work, double* partials, unsigned* ticket, double* gnorm2,
                    double* phi) {
    __shared__ double qxs[2][kGradTy][kGradTx], qys[2][kGradTy][kGradTx];
    const int tx = threadIdx.x % kGradTx, ty = threadIdx.x / kGradTx;
    const uint32_t sxy = (uint32_t)nx * (uint32_t)ny;   // images hold fewer than 2^31 voxels
    double acc[PHI ? 2 : 1] = {};
    for (int w = blockIdx.x; w < work; w += gridDim.x) {
        const int zi = w / tiles, tile = w - zi * tiles, by = tile / tiles_x, bx = tile - by * tiles_x;
        const int ix = bx * (kGradTx - 1) + tx - 1, iy = by * (kGradTy - 1) + ty - 1;
        const bool in = ix >= 0 && ix < nx && iy >= 0 && iy < ny, own = in && tx > 0 && ty > 0;
        const int z0 = zi * zc, z1 = min(nz, z0 + zc), zs = z0 > 0 ? z0 - 1 : 0;
        const bool hx = ix + 1 < nx, hy = iy + 1 < ny;
        double zprev = 0.0;
        uint32_t p = ((uint32_t)zs * (uint32_t)ny + (uint32_t)iy) * (uint32_t)nx + (uint32_t)ix;
        double xc = in ? __ldg(x + p) : 0.0;
        for (int z = zs; z < z1; ++z, p += sxy) {
            double dx = 0.0, dy = 0.0, dz = 0.0;
            if (in) {
                if (hx) dx = __ldg(x + p + 1) - xc;
                if (hy) dy = __ldg(x + p + nx) - xc;
                if (z + 1 < nz) {
                    const double xn = __ldg(x + p + sxy);
                    dz = xn - xc;
                    xc = xn;
                }
            }
            const double d2 = dx * dx + dy * dy + dz * dz;
            const Quotients over(eps + d2);
            const int buf = z & 1;
            qxs[buf][ty][tx] = over(dx);
            qys[buf][ty][tx] = over(dy);
            const double qz = over(dz);
            __syncthreads();   // one a slice: the buffers alternate
            if (own && z >= z0) {
                double gq = over(-(dx + dy + dz));
                if (ix > 0) gq += qxs[buf][ty][tx - 1];
                if (iy > 0) gq += qys[buf][ty - 1][tx];
                if (z > 0) gq += zprev;
                g[p] = gq;
                acc[0] += gq * gq;
                if constexpr (PHI) acc[1] += sqrt(d2);
            }
            zprev = qz;
        }
        __syncthreads();   // before the next tile writes the buffers
    }
    if constexpr (PHI) {
        double* const outs[2] = {gnorm2, phi};
        grid_reduce<2>(acc, partials, ticket, outs);
    } else {
        double* const outs[1] = {gnorm2};
        grid_reduce<1>(acc, partials, ticket, outs);
    }
}

// One thread per voxel (the FP32 path, and FP64 images too thin for tiles).  SPLIT (FP32): neighbour
// differences are (xh_a - xh_b) + (xl_a - xl_b) from the split copies of the master image, so the
// stencil runs without FP64 arithmetic (only ||g||^2 is accumulated in FP64).  Otherwise they are
// formed in FP64 from the master image and rounded once to T, the stencil's type; with PHI also
// phi_0(x), from the same differences (FP32 on 128x128x16: 31.8 us so and 28.6 with the split ones,
// which lose what xl has no bits for, 2^-49 of the voxel).
template <typename T, bool SPLIT, bool PHI>
__global__ void __launch_bounds__(kRedThreads)
tv_grad_voxel_kernel(const double* __restrict__ x, const float* __restrict__ xh, const float* __restrict__ xl,
                     T* __restrict__ g, int nx, int ny, int nz, T eps, double* partials, unsigned* ticket,
                     double* gnorm2, double* phi) {
    static_assert(!(SPLIT && PHI), "phi takes the differences of the master image");
    const int64_t sxy = (int64_t)nx * ny, V = sxy * nz;
    auto dif = [&](int64_t a, int64_t b) -> T {
        if constexpr (SPLIT) return (__ldg(xh + a) - __ldg(xh + b)) + (__ldg(xl + a) - __ldg(xl + b));
        else return (T)(__ldg(x + a) - __ldg(x + b));
    };
    double acc[PHI ? 2 : 1] = {};
    for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < V; p += (int64_t)gridDim.x * blockDim.x) {
        int ix, iy, iz;
        voxel_coords(p, nx, ny, ix, iy, iz);
        const bool hx = ix + 1 < nx, hy = iy + 1 < ny, hz = iz + 1 < nz;
        double ex = 0.0, ey = 0.0, ez = 0.0;
        T dx, dy, dz;
        if constexpr (PHI) {
            const double xc = __ldg(x + p);
            ex = hx ? __ldg(x + p + 1) - xc : 0.0;
            ey = hy ? __ldg(x + p + nx) - xc : 0.0;
            ez = hz ? __ldg(x + p + sxy) - xc : 0.0;
            dx = (T)ex, dy = (T)ey, dz = (T)ez;
        } else {
            dx = hx ? dif(p + 1, p) : (T)0, dy = hy ? dif(p + nx, p) : (T)0, dz = hz ? dif(p + sxy, p) : (T)0;
        }
        const T D = sqrt(eps + (dx * dx + dy * dy + dz * dz));
        T gq = (D > (T)0) ? -(dx + dy + dz) / D : (T)0;
        if (ix > 0) {
            const int64_t q = p - 1;
            const T a = dif(p, q), b = hy ? dif(q + nx, q) : (T)0, c = hz ? dif(q + sxy, q) : (T)0;
            const T Dm = sqrt(eps + (a * a + b * b + c * c));
            if (Dm > (T)0) gq += a / Dm;
        }
        if (iy > 0) {
            const int64_t q = p - nx;
            const T a = dif(p, q), b = hx ? dif(q + 1, q) : (T)0, c = hz ? dif(q + sxy, q) : (T)0;
            const T Dm = sqrt(eps + (a * a + b * b + c * c));
            if (Dm > (T)0) gq += a / Dm;
        }
        if (iz > 0) {
            const int64_t q = p - sxy;
            const T a = dif(p, q), b = hx ? dif(q + 1, q) : (T)0, c = hy ? dif(q + nx, q) : (T)0;
            const T Dm = sqrt(eps + (a * a + b * b + c * c));
            if (Dm > (T)0) gq += a / Dm;
        }
        g[p] = gq;
        acc[0] += (double)gq * (double)gq;
        if constexpr (PHI) acc[1] += sqrt(ex * ex + ey * ey + ez * ez);
    }
    if constexpr (PHI) {
        double* const outs[2] = {gnorm2, phi};
        grid_reduce<2>(acc, partials, ticket, outs);
    } else {
        double* const outs[1] = {gnorm2};
        grid_reduce<1>(acc, partials, ticket, outs);
    }
}

// phi_0(z), z = x - sc*g (z = x if g is null), FP64 from the master image.
template <typename T>
__global__ void __launch_bounds__(kRedThreads)
tv_value_kernel(const double* __restrict__ x, const T* __restrict__ g, const double* gnorm2, double beta, int nx,
                int ny, int nz, double* partials, unsigned* ticket, double* phi, const double* phi_ref, int* accept) {
    const int64_t sxy = (int64_t)nx * ny, V = sxy * nz;
    __shared__ double scale;
    if (g && threadIdx.x == 0) scale = step_scale(beta, gnorm2);
    __syncthreads();
    const double sc = g ? scale : 0.0;
    double acc[1] = {0.0};
    for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < V; p += (int64_t)gridDim.x * blockDim.x) {
        int ix, iy, iz;
        voxel_coords(p, nx, ny, ix, iy, iz);
        auto zat = [&](int64_t q) -> double {
            return g ? perturbed(__ldg(x + q), sc, (double)__ldg(g + q)) : __ldg(x + q);
        };
        const double zc = zat(p);
        const double ex = (ix + 1 < nx) ? zat(p + 1) - zc : 0.0;
        const double ey = (iy + 1 < ny) ? zat(p + nx) - zc : 0.0;
        const double ez = (iz + 1 < nz) ? zat(p + sxy) - zc : 0.0;
        acc[0] += sqrt(ex * ex + ey * ey + ez * ez);
    }
    double* const outs[1] = {phi};
    if (grid_reduce<1>(acc, partials, ticket, outs)) {
        if (threadIdx.x == 0 && phi_ref && accept) {
            __threadfence();
            *accept = (__ldcg(phi) <= *phi_ref) ? 1 : 0;
        }
    }
}

// x <- x - sc*g on the master image (and its FP32 copies when present).  The step's scale, an
// FP64 square root and division, is formed once per CTA: formed by every thread it took more of
// the FP64 pipe than the voxels' own arithmetic.
template <typename T, int U>
__global__ void __launch_bounds__(kRedThreads)
tv_apply_kernel(double* __restrict__ x, ImgCopies c, const T* __restrict__ g, const double* gnorm2, double beta,
                const int* accept, int64_t V) {
    if (accept && *accept == 0) return;
    __shared__ double scale;
    if (threadIdx.x == 0) scale = step_scale(beta, gnorm2);
    __syncthreads();
    const double sc = scale;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t j0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j0 < V; j0 += U * stride) {
        double xv[U];
        T gv[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int64_t j = min(j0 + u * stride, V - 1);   // clamped: the loads issue together
            xv[u] = x[j];
            gv[u] = g[j];
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int64_t j = j0 + u * stride;
            if (j < V) {
                const double z = perturbed(xv[u], sc, (double)gv[u]);
                x[j] = z;
                store_copies(c, j, z);
            }
        }
    }
}

template <int U>
__global__ void __launch_bounds__(kRedThreads) x32_from_x64_kernel(const double* __restrict__ x, ImgCopies c) {
    const int64_t V = (int64_t)c.m.nx * c.m.ny * c.m.nz, stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t j0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j0 < V; j0 += U * stride) {
        double xv[U];
#pragma unroll
        for (int u = 0; u < U; ++u) xv[u] = x[min(j0 + u * stride, V - 1)];
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (j0 + u * stride < V) store_copies(c, j0 + u * stride, xv[u]);
    }
}

// the gather image of canonical image src: out[internal(j)] = (float)src[j]
template <typename S>
__global__ void gather_image_kernel(const S* __restrict__ src, float* __restrict__ out, VoxMap m, int64_t V) {
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < V; j += (int64_t)gridDim.x * blockDim.x)
        out[vox_internal(m, j)] = (float)src[j];
}

static int g_sm_count = 0;
static int sm_count() {
    if (!g_sm_count) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&g_sm_count, cudaDevAttrMultiProcessorCount, dev);
        if (g_sm_count <= 0) g_sm_count = 1;
    }
    return g_sm_count;
}

static int64_t grad_tiles(int nx, int ny, int ty) {
    return (int64_t)((nx + kGradTx - 2) / (kGradTx - 1)) * ((ny + ty - 2) / (ty - 1));
}

template <bool PHI, int kGradTy>
static cudaError_t launch_grad_tile(const double* x, double* g, int nx, int ny, int nz, double eps, RedScratch r,
                                    double* gnorm2, double* phi, cudaStream_t s) {
    const int tiles_x = (nx + kGradTx - 2) / (kGradTx - 1);
    const int64_t tiles = grad_tiles(nx, ny, kGradTy);
    const int sms = sm_count();
    // slices per CTA: the fewest slice steps (a slice of halo each) on the busiest SM
    int zc = 1;
    int64_t best = INT64_MAX;
    for (int c = 1; c <= nz && c <= 32; ++c) {
        const int64_t ctas = tiles * ((nz + c - 1) / c), cost = (ctas + sms - 1) / sms * (c + (c < nz ? 1 : 0));
        if (cost < best) {
            best = cost;
            zc = c;
        }
    }
    const int64_t work = tiles * ((nz + zc - 1) / zc);   // below the voxel count's 2^31
    const int grid = (int)(work < (int64_t)sms * 4 ? work : (int64_t)sms * 4);
    tv_grad_tile_kernel<PHI, kGradTy><<<grid, kGradTx * kGradTy, 0, s>>>(x, g, nx, ny, nz, eps, zc, tiles_x, (int)tiles,
                                                               (int)work, r.partials, r.ticket, gnorm2, phi);
    return cudaGetLastError();
}

cudaError_t k_tv_grad(int cdt, const double* x, const float* xh, const float* xl, void* g, int nx, int ny, int nz,
                      double eps, RedScratch r, double* gnorm2, double* phi, cudaStream_t s) {
    if (cdt == F64) {
        const int64_t V = (int64_t)nx * ny * nz, slice = (int64_t)sm_count() * kGradTx * 16;   // a tile slice an SM
        const bool few = V < slice;
        // In tiles every thread does a voxel's work, inside the image or not; by itself a voxel costs more
        // than twice as much.  So tiles as long as they have at most three threads a voxel, or all run at
        // once.  us a step in tiles / without, by threads a voxel: 63x33x64 (2.2) 35 / 41, 33x33x200 (2.8)
        // 56 / 59, 31x5x3000 (3.3) 90 / 103, 34x18x128 (3.3) 33 / 31, 16x16x400 (4.0) 43 / 33, 400x2x200 (5)
        // 82 / 47, 1x2000x50 (17) 256 / 29.
        const int64_t threads = grad_tiles(nx, ny, few ? 4 : 16) * nz * kGradTx * (few ? 4 : 16);
        if (threads > std::max(3 * V, slice)) {
            const auto kern = phi ? tv_grad_voxel_kernel<double, false, true> : tv_grad_voxel_kernel<double, false, false>;
            kern<<<r.grid, kRedThreads, 0, s>>>(x, xh, xl, (double*)g, nx, ny, nz, eps, r.partials, r.ticket, gnorm2, phi);
            return cudaGetLastError();
        }
        const auto run = few ? (phi ? launch_grad_tile<true, 4> : launch_grad_tile<false, 4>)
                             : (phi ? launch_grad_tile<true, 16> : launch_grad_tile<false, 16>);
        return run(x, (double*)g, nx, ny, nz, eps, r, gnorm2, phi, s);
    }
    if (!phi && (!xh || !xl)) return cudaErrorInvalidValue;   // the FP32 path keeps the split copies
    const auto kern = phi ? tv_grad_voxel_kernel<float, false, true> : tv_grad_voxel_kernel<float, true, false>;
    kern<<<r.grid, kRedThreads, 0, s>>>(x, xh, xl, (float*)g, nx, ny, nz, (float)eps, r.partials, r.ticket, gnorm2, phi);
    return cudaGetLastError();
}

cudaError_t k_tv_value(int cdt, const double* x, const void* g, const double* gnorm2, double beta, int nx, int ny,
                       int nz, RedScratch r, double* phi, const double* phi_ref, int* accept, cudaStream_t s) {
    if (cdt == F64)
        tv_value_kernel<double><<<r.grid, kRedThreads, 0, s>>>(x, (const double*)g, gnorm2, beta, nx, ny, nz,
                                                               r.partials, r.ticket, phi, phi_ref, accept);
    else
        tv_value_kernel<float><<<r.grid, kRedThreads, 0, s>>>(x, (const float*)g, gnorm2, beta, nx, ny, nz,
                                                              r.partials, r.ticket, phi, phi_ref, accept);
    return cudaGetLastError();
}

cudaError_t k_tv_apply(int cdt, double* x, ImgCopies c, const void* g, const double* gnorm2, double beta,
                       const int* accept, int64_t V, cudaStream_t s) {
    const int grid = red_grid(V, sm_count());
    const bool many = vox_unrolled(V, grid);
    if (cdt == F64)
        (many ? tv_apply_kernel<double, kVoxUnroll> : tv_apply_kernel<double, 1>)<<<grid, kRedThreads, 0, s>>>(
            x, c, (const double*)g, gnorm2, beta, accept, V);
    else
        (many ? tv_apply_kernel<float, kVoxUnroll> : tv_apply_kernel<float, 1>)<<<grid, kRedThreads, 0, s>>>(
            x, c, (const float*)g, gnorm2, beta, accept, V);
    return cudaGetLastError();
}

cudaError_t k_x32_from_x64(const double* x, ImgCopies c, cudaStream_t s) {
    const int64_t V = (int64_t)c.m.nx * c.m.ny * c.m.nz;
    const int grid = red_grid(V, sm_count());
    (vox_unrolled(V, grid) ? x32_from_x64_kernel<kVoxUnroll> : x32_from_x64_kernel<1>)<<<grid, kRedThreads, 0, s>>>(x, c);
    return cudaGetLastError();
}

cudaError_t k_gather_image(const void* src, int sdt, float* out, const VoxMap& m, cudaStream_t s) {
    const int64_t V = (int64_t)m.nx * m.ny * m.nz;
    const int grid = red_grid(V, sm_count());
    if (sdt == F64) gather_image_kernel<double><<<grid, 256, 0, s>>>((const double*)src, out, m, V);
    else gather_image_kernel<float><<<grid, 256, 0, s>>>((const float*)src, out, m, V);
    return cudaGetLastError();
}

// ------------------------------------------------------------------ conversions
template <typename S, typename D>
__global__ void convert_kernel(const S* __restrict__ src, D* __restrict__ dst, int64_t n) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        dst[i] = (D)src[i];
}

cudaError_t k_convert(const void* src, int sdt, void* dst, int ddt, int64_t n, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    const int grid = red_grid(n, sm_count());
    if (sdt == F64 && ddt == F32) convert_kernel<double, float><<<grid, 256, 0, s>>>((const double*)src, (float*)dst, n);
    else if (sdt == F32 && ddt == F64) convert_kernel<float, double><<<grid, 256, 0, s>>>((const float*)src, (double*)dst, n);
    else if (sdt == ddt) return cudaMemcpyAsync(dst, src, (size_t)n * dt_size(sdt), cudaMemcpyDeviceToDevice, s);
    else return cudaErrorInvalidValue;
    return cudaGetLastError();
}

}  // namespace ntvs
