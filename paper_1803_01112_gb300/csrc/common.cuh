// Device helpers shared by the kernel translation units.
#pragma once
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "ntvs_internal.h"

namespace ntvs {

template <typename T> struct StorageOf;
__device__ __forceinline__ float to_compute(float v) { return v; }
__device__ __forceinline__ double to_compute(double v) { return v; }
__device__ __forceinline__ float to_compute(__half v) { return __half2float(v); }
__device__ __forceinline__ float to_compute(__nv_bfloat16 v) { return __bfloat162float(v); }

// the 16-bit value in the high half of a DELTA16 word: BF16 bits are the FP32 value's high half
template <typename V>
__device__ __forceinline__ float word_value(uint32_t e) {
    if constexpr (std::is_same<V, __nv_bfloat16>::value) return __uint_as_float(e & 0xffff0000u);
    else return __half2float(__ushort_as_half((unsigned short)(e >> 16)));
}

// fused x - s*g on the FP64 master image, spelled out so every kernel that forms a
// perturbed voxel rounds alike
__device__ __forceinline__ double perturbed(double x, double s, double g) { return __fma_rn(-s, g, x); }

// Voxels a thread of the kernels over all voxels takes at once (a grid stride apart) on large
// images, their loads issued together: with the loads of one voxel in flight per thread the
// image copies of 256x256x64 voxels ran at 2.5 TB/s (latency).  Block apply there 37.6 ->
// 31.3 us, TV step 59.6 -> 50.7 us.  An image of at most two voxels a thread (200x200x16
// and smaller) has all its loads in flight anyway and keeps one at a time (with four, the FP64
// apply took 7.1 instead of 4.5 us).
constexpr int kVoxUnroll = 4;
inline bool vox_unrolled(int64_t V, int grid) { return V > (int64_t)grid * 256 * 3; }

// sqrt(s), and *r close to 1 / sqrt(s) (relative error below 2^-42), in FP64 by one Goldschmidt
// step (1964) from the FP32 reciprocal square root and a Markstein correction of the root by its
// residual (1990): the seed is within 2^-21.9, the step squares that, and the correction leaves
// the rounding of its last FMA.  In 1.8e8 samples over 2^-120..2^120, seeds two ulp off
// included, the result was the correctly rounded root.  It pays where both are wanted (the FP64
// gradient, 74 -> 67 us at 200x200x16); for a root alone sqrt() is as fast (phi of 256x256x64
// voxels 186 us with it, 194 with this).  Outside the FP32 range, zeros, infinities and NaN:
// sqrt() and a division.
__device__ __forceinline__ double sqrt_and_inverse(double s, double* r) {
    const float f = (float)s;
    if (!(f > 1e-36f && f < 1e36f)) {
        const double d = sqrt(s);
        *r = d > 0.0 ? 1.0 / d : 0.0;
        return d;
    }
    const double y = (double)rsqrtf(f);
    double g = s * y, h = 0.5 * y;
    const double e = fma(-g, h, 0.5);
    g = fma(g, e, g);
    h = fma(h, e, h);
    *r = h + h;
    return fma(fma(-g, g, s), h, g);
}
// s = beta / ||g|| (0 when g = 0, i.e. v = 0)
__device__ __forceinline__ double step_scale(double beta, const double* gnorm2) {
    const double n2 = *gnorm2;
    return (n2 > 0.0) ? beta / sqrt(n2) : 0.0;
}

__device__ __forceinline__ uint32_t fast_div(uint32_t u, const FastDiv& f) { return f.m ? __umulhi(u, f.m) >> f.s : u; }

// internal index of canonical voxel j (see VoxMap); 32-bit arithmetic, as every index
// of either order is below 2^31
__device__ __forceinline__ int64_t vox_internal(const VoxMap& m, int64_t j) {
    if (m.tx == 1 && m.ty == 1 && !m.sw) return j;
    const uint32_t u = (uint32_t)j, nx = (uint32_t)m.nx, ny = (uint32_t)m.ny;
    const uint32_t t = fast_div(u, m.dnx), ix = u - t * nx;
    const uint32_t iz = fast_div(t, m.dny), iy = t - iz * ny;
    const uint32_t ntx = (uint32_t)m.nxp >> m.ltx;
    const uint32_t tile = (iy >> m.lty) * ntx + (ix >> m.ltx);
    uint32_t p = (tile << (m.ltx + m.lty)) + ((iy & (uint32_t)(m.ty - 1)) << m.ltx) + (ix & (uint32_t)(m.tx - 1));
    if (m.sw) p ^= (p >> 5) & 31u;
    return (int64_t)(iz * (uint32_t)m.slice_p + p);
}

// the FP32 copies of master value v of the voxel with canonical index j and internal index p
__device__ __forceinline__ void store_copies(const ImgCopies& c, int64_t j, uint32_t p, double v) {
    const float h = (float)v;
    if (c.x32) c.x32[p] = h;
    if (c.xh) {
        c.xh[j] = h;
        c.xl[j] = (float)(v - (double)h);
    }
}
__device__ __forceinline__ void store_copies(const ImgCopies& c, int64_t j, double v) {
    store_copies(c, j, c.x32 ? (uint32_t)vox_internal(c.m, j) : 0u, v);
}

// Scale of an FP32 scatter window that accumulates in int32 (kept in shared memory, uniform over
// the CTA, so that the row loop's registers hold the matrix entries): quantum Q = 1 / invQ; rows
// with |r_i / lambda| above `bound` scatter globally (invQ = 0 sends every row there), which
// keeps every window slot below 2^30 Q and every converted term below 2^22 in magnitude.
struct WinScale {
    float invQ, bound, Q;
};

// The scale for a block whose rows have the statistics st (WinStat), rms being the root mean
// square residual of the block swept before it (win_rms).  The bound on a row of mean ||a||^2 is
// 10 rms, or 4 once the residuals are of the size of b itself (they are then mostly of one sign, not
// noise), between 1/16 and 64 of the block's mean |b|; without an rms 1/4 of it (NaN: the image was
// set since) or 4 (below 0: the zero image of a load, whose residual is b).  So the quantum follows
// the residuals of the image being swept, and rows of very short chords, whose |r / lambda| is far
// above the others', scatter globally instead of coarsening them.  At 10 rms the error of a sweep
// against 64 bits is that of FP32 reductions (2.773e-8 of the image at 200x200x16, 2M rows in
// detected order, both ways).
// A scale taken inside the launch, from its own first rows, was exact about the image but cost 6
// of 62 us a block of 100k rows (the other warps wait for it, or scatter globally until it stands).
__device__ __forceinline__ WinScale win_scale(float lambda, const WinStat& st, float rms) {
    float bound = rms >= 0.f  ? fminf(10.f * rms, 4.f * fmaxf(rms, st.mean_b))
                  : rms < 0.f ? 4.f * st.mean_b
                              : 0.25f * st.mean_b;
    if (st.mean_b > 0.f) bound = fminf(fmaxf(bound, 0.0625f * st.mean_b), 64.f * st.mean_b);
    bound *= st.inv_norm2;
    const float lam = fabsf(lambda), Q = lam * bound * st.lmax * 0x1p-30f, iq = 1.f / Q;
    if (!(st.amax > 0.f && Q > 0.f && isfinite(Q) && isfinite(iq))) return WinScale{0.f, 0.f, 0.f};
    return WinScale{iq, fminf(bound, 0x1p22f * Q / (lam * st.amax)), Q};
}
// The rms residual of a swept block of `rows` rows from the sums over its runs of rows (a CTA's each,
// of about equal length): {sum of log2(residual sum of squares), runs with any}.  Their geometric
// mean, which a few rows of corrupt data in a few runs hardly move.
__device__ __forceinline__ float win_rms(float2 sums, float rows) {
    return sums.y > 0.f ? exp2f(0.5f * (sums.x / sums.y - __log2f(rows / sums.y))) : 0.f;
}

// %globaltimer in nanoseconds (the clock of every bounded device-side wait)
__device__ __forceinline__ uint64_t globaltimer_ns() {
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Sum of v over the CTA (blockDim.x multiple of 32, <= 1024); result valid in thread 0.
__device__ __forceinline__ double block_sum(double v, double* sh /* >= 32 */) {
    v = warp_sum(v);
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    __syncthreads();
    if (l == 0) sh[w] = v;
    __syncthreads();
    double r = 0.0;
    if (w == 0) {
        r = (l < (int)(blockDim.x >> 5)) ? sh[l] : 0.0;
        r = warp_sum(r);
    }
    return r;
}

// Deterministic grid reduction of NV values per CTA: CTA b writes partials[q*grid + b];
// the last CTA to finish sums each q in a fixed order into out[q] and resets the ticket.
// Returns true in the last CTA (all threads), after out[] is written.
template <int NV>
__device__ __forceinline__ bool grid_reduce(const double (&v)[NV], double* partials, unsigned* ticket,
                                            double* const (&out)[NV]) {
    __shared__ double sh[32];
    __shared__ bool last;
    double tot[NV];
#pragma unroll
    for (int q = 0; q < NV; ++q) tot[q] = block_sum(v[q], sh);
    if (threadIdx.x == 0) {
#pragma unroll
        for (int q = 0; q < NV; ++q) partials[q * gridDim.x + blockIdx.x] = tot[q];
        __threadfence();
        unsigned t = atomicAdd(ticket, 1u);
        last = (t == gridDim.x - 1);
    }
    __syncthreads();
    if (!last) return false;
    __threadfence();
#pragma unroll
    for (int q = 0; q < NV; ++q) {
        double a = 0.0;
        for (int i = threadIdx.x; i < (int)gridDim.x; i += blockDim.x) a += __ldcg(&partials[q * gridDim.x + i]);
        a = block_sum(a, sh);
        if (threadIdx.x == 0 && out[q]) *out[q] = a;
    }
    if (threadIdx.x == 0) *ticket = 0u;
    return true;
}

}  // namespace ntvs
