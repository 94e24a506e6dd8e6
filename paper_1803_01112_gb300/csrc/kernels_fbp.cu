// Initial iterate x-bar (arXiv 1803.01112: x-bar of Appendix A, FBP of Sec. II, median
// filter of radius 2 on the initial iterate in Sec. V-A): chord binning, Ram-Lak filter,
// back-projection, median filter and threshold hull, all in FP64.  The steps follow the
// specification in include/ntvs_fbp.h.
//
// Kernels and their bounds (CTP404 scale: 10M histories, 16 x 180 x 200 bins, 200x200x16
// voxels):
//   fbp_bin_kernel       one thread per history; 24 B read per history; bins decided in FP32
//                        wherever that is certain, else in FP64; bin sums by one FP64 atomic
//                        per run of equal bins in a warp (segmented suffix sum; acquisition
//                        order gives runs).
//   fbp_filter_kernel    one CTA per (slice, angle) row; the row and the odd-lag kernel in
//                        shared memory; n_t^2/2 FMAs per row.
//   fbp_backproject_tile_kernel 32 x 16 voxel tiles; fixed-point positions, the row's
//                        interpolation pairs in shared memory, 3 FP64-pipe operations per
//                        (voxel, angle): FP64-pipe bound on GB300.
//   fbp_backproject_kernel  geometries outside the tile kernel's limits: one thread per 4
//                        voxels of a row, 7 FP64-pipe operations per (voxel, angle).
//   median_kernel        one thread per voxel; the window as monotone 64-bit integer keys
//                        in registers, the element floor(n/2) by rank counting (W^2
//                        integer compares, no FP64 pipe); the hull fused into the store.
#include <math.h>

#include <string>

#include "common.cuh"
#include "ntvs_fbp.h"

namespace ntvs {

namespace {

constexpr int kMaxNt = 8192;
constexpr int kMaxNtheta = 4096;
constexpr int kMaxMedianRadius = 3;
constexpr double kPi = 3.14159265358979323846;

int fbp_fail(int code, const std::string& msg) {
    set_last_error(msg);   // read back with ntvs_last_error()
    return code;
}

int launch_status(const char* where) {
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return fbp_fail(NTVS_ERR_CUDA, std::string(where) + ": " + cudaGetErrorString(e));
    return NTVS_OK;
}

bool finite_pos(double v) { return std::isfinite(v) && v > 0.0; }

int check_geom(const ntvs_fbp_geom* g, const char* where) {
    if (!g) return fbp_fail(NTVS_ERR_ARG, std::string(where) + ": null geometry");
    if (g->nx < 1 || g->ny < 1 || g->nz < 1 || g->n_theta < 1 || g->n_t < 1)
        return fbp_fail(NTVS_ERR_ARG, std::string(where) + ": grid and bin counts must be >= 1");
    if (g->reserved != 0) return fbp_fail(NTVS_ERR_ARG, std::string(where) + ": reserved must be 0");
    if (g->n_t > kMaxNt) return fbp_fail(NTVS_ERR_ARG, std::string(where) + ": n_t > 8192");
    if (g->n_theta > kMaxNtheta) return fbp_fail(NTVS_ERR_ARG, std::string(where) + ": n_theta > 4096");
    if (g->nz > 65535) return fbp_fail(NTVS_ERR_ARG, std::string(where) + ": nz > 65535");
    if (!finite_pos(g->dx) || !finite_pos(g->dy) || !finite_pos(g->dz) || !finite_pos(g->dt))
        return fbp_fail(NTVS_ERR_ARG, std::string(where) + ": dx, dy, dz and dt must be finite and > 0");
    if (!std::isfinite(g->theta0) || fabs(g->theta0) > 16.0 * kPi)
        return fbp_fail(NTVS_ERR_ARG, std::string(where) + ": theta0 must be finite with |theta0| <= 16 pi");
    const int64_t V = (int64_t)g->nx * g->ny * g->nz;
    const int64_t S = (int64_t)g->nz * g->n_theta * g->n_t;
    if (V > INT32_MAX || S > INT32_MAX)
        return fbp_fail(NTVS_ERR_ARG, std::string(where) + ": more than 2^31 - 1 voxels or bins");
    return NTVS_OK;
}

// ---------------------------------------------------------------- 1. binning

// (phi, t) of a line whose normal is at angle theta (any value in [-pi, 2 pi)) with
// lateral offset t: the fold into [0, pi) and the rebase to theta0 of step 1.
__device__ __forceinline__ double fold_rebase(double theta, double& t, double theta0) {
    if (theta < 0.0) theta += 2.0 * kPi;
    if (theta >= kPi) {
        theta -= kPi;
        t = -t;
    }
    double phi = theta - theta0;   // |theta0| <= 16 pi is checked by the host: at most 18 steps
    for (int i = 0; i < 64 && phi < 0.0; ++i) {
        phi += kPi;
        t = -t;
    }
    for (int i = 0; i < 64 && phi >= kPi; ++i) {
        phi -= kPi;
        t = -t;
    }
    return phi;
}

// Flat bin of one chord record, or -1 when it falls outside the bins (step 1), decided in
// FP64.  The normal's angle is first taken from the FP32 atan2 of the chord direction
// (error below 1e-6 rad, the FP32 rounding of the direction included): when the rebased
// angle lies more than 1e-5 rad from every angle-bin edge (the fold at theta = pi is
// continuous in the bin it gives, except where it is itself an edge), the FP64 angle gives
// the same bin; otherwise the angle is recomputed with the FP64 atan2.  t is the FP64
// projection of P_in on the unit normal.
__device__ __forceinline__ int64_t bin_of(const float* __restrict__ rec, const ntvs_fbp_geom& g) {
    const double px = __ldg(rec + 0), py = __ldg(rec + 1), pz = __ldg(rec + 2);
    const double qx = __ldg(rec + 3), qy = __ldg(rec + 4), qz = __ldg(rec + 5);
    const double ddx = qx - px, ddy = qy - py;
    const double len = sqrt(__dadd_rn(__dmul_rn(ddx, ddx), __dmul_rn(ddy, ddy)));
    if (!(len > 0.0)) return -1;
    const double t0 = __dadd_rn(__dmul_rn(px, -ddy), __dmul_rn(py, ddx)) / len;   // normal (-ddy, ddx)/len
    const double w = kPi / g.n_theta;
    double t = t0;
    double phi = fold_rebase((double)atan2f((float)ddx, (float)-ddy), t, g.theta0);
    const double f = phi / w - floor(phi / w);
    if (fmin(f, 1.0 - f) * w < 1e-5 || len < 1e-30) {   // near an edge, or FP32 would underflow
        t = t0;
        phi = fold_rebase(atan2(ddx, -ddy), t, g.theta0);
    }
    if (!(phi >= 0.0 && phi < kPi)) return -1;   // unreachable for |theta0| <= 16 pi
    int64_t a = (int64_t)floor(phi / w);
    a = a < 0 ? 0 : (a > g.n_theta - 1 ? g.n_theta - 1 : a);
    const double u = __dadd_rn(t / g.dt, 0.5 * g.n_t);
    if (!(u >= 0.0 && u < (double)g.n_t)) return -1;
    const double v = __dmul_rn(0.5, pz + qz) / g.dz;
    if (!(v >= 0.0 && v < (double)g.nz)) return -1;
    int64_t k = (int64_t)floor(u), iz = (int64_t)floor(v);
    if (k > g.n_t - 1) k = g.n_t - 1;
    if (iz > g.nz - 1) iz = g.nz - 1;
    return (iz * g.n_theta + a) * g.n_t + k;
}

// FP32 constants of the binning prefilter (host-made); usable = 0 sends every history to
// the FP64 decision.
struct BinFast {
    float inv_w, w, theta0, inv_dt, half_nt, inv_dz;
    int usable;
};

// The bin of one chord record, decided in FP32 where FP32 decides it for certain: the angle,
// the lateral position and the height are formed in FP32 with a bound on their distance from
// the FP64 values, and a history closer than that to any bin edge (or with a degenerate or
// non-finite chord) returns -2 and is decided by bin_of.  Bounds, with e = 2^-24: each FP32
// operation is within e of its exact result, so t (four products and a quotient of values up
// to |P|) is within 16 e |P| and u = t / dt + n_t / 2 within that over dt plus 4 e (|u| + n_t);
// theta is within 1e-6 rad (atan2f) plus 4 e per fold by pi; z within 8 e.  FP64 arithmetic
// here is the whole cost of a history (FP64 divisions and a square root run at 1/64 of the
// FP32 rate): the FP64 decision for every history took 1825 us on 10M histories, against
// 150 us with the prefilter.
__device__ __forceinline__ int bin_fast(const float* __restrict__ rec, const ntvs_fbp_geom& g, const BinFast& f) {
    const float px = __ldg(rec + 0), py = __ldg(rec + 1), pz = __ldg(rec + 2);
    const float qx = __ldg(rec + 3), qy = __ldg(rec + 4), qz = __ldg(rec + 5);
    const float ddx = qx - px, ddy = qy - py;
    const float len = sqrtf(ddx * ddx + ddy * ddy);
    if (!(f.usable && len > 1e-12f && len < 1e12f)) return -2;
    float t = (py * ddx - px * ddy) / len;
    const float mag = fabsf(px) + fabsf(py);
    float phi = atan2f(ddx, -ddy) - f.theta0;   // |phi| < 2 pi + |theta0| <= 4 pi
    const float pi = 3.14159265f;
    for (int i = 0; i < 5 && phi < 0.f; ++i) {
        phi += pi;
        t = -t;
    }
    for (int i = 0; i < 5 && phi >= pi; ++i) {
        phi -= pi;
        t = -t;
    }
    const float fa = phi * f.inv_w, fl = floorf(fa), fr = fa - fl;
    const float u = fmaf(t, f.inv_dt, f.half_nt), ul = floorf(u), ur = u - ul;
    const float eu = 1e-6f * mag * f.inv_dt + 2.4e-7f * (fabsf(u) + 2.f * f.half_nt);
    const float v = 0.5f * (pz + qz) * f.inv_dz, vl = floorf(v), vr = v - vl;
    const float ev = 5e-7f * (fabsf(pz) + fabsf(qz)) * f.inv_dz;
    const bool sure = fminf(fr, 1.f - fr) * f.w > 2e-5f && fminf(ur, 1.f - ur) > eu && fminf(vr, 1.f - vr) > ev &&
                      fl >= 0.f && fl < (float)g.n_theta;
    if (!sure) return -2;   // NaNs too: every comparison above is false for them
    if (!(ul >= 0.f && ul < (float)g.n_t && vl >= 0.f && vl < (float)g.nz)) return -1;
    return ((int)vl * g.n_theta + (int)fl) * g.n_t + (int)ul;
}

// Bin sums and counts.  Every lane of a warp takes one history.  Lanes with equal bins
// next to each other form a run (histories in acquisition order give runs of one bin);
// a segmented suffix sum over each run (as many shuffle steps as the longest run needs)
// leaves the run's sum in its first lane, which adds it and the run length with one atomic
// each.  Equal bins that are not adjacent make separate runs, which is still correct.  The
// loop bound is warp-uniform so that every shuffle has all 32 lanes.
__global__ void __launch_bounds__(256) fbp_bin_kernel(ntvs_fbp_geom g, BinFast f, const float* __restrict__ paths,
                                                      const double* __restrict__ wepl, int64_t M,
                                                      double* __restrict__ sum, int32_t* __restrict__ count) {
    const int lane = threadIdx.x & 31;
    const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t base = warp * 32; base < M; base += nwarps * 32) {
        const int64_t h = base + lane;
        int key = -1;   // bins are counted below 2^31
        double w = 0.0;
        if (h < M) {
            w = __ldg(wepl + h);
            key = bin_fast(paths + 10 * h, g, f);
            if (key == -2) key = (int)bin_of(paths + 10 * h, g);
        }
        const int next = __shfl_down_sync(0xffffffffu, key, 1);
        const unsigned last = __ballot_sync(0xffffffffu, lane == 31 || next != key);   // bit l: run ends at l
        const int end = __ffs(last & (0xffffffffu << lane)) - 1;                     // this lane's run end
        const int longest = __reduce_max_sync(0xffffffffu, end - lane);
        double s = w;
        for (int o = 1; o <= longest; o <<= 1) {
            const double v = __shfl_down_sync(0xffffffffu, s, o);
            if (lane + o <= end) s += v;
        }
        const bool head = lane == 0 || ((last >> (lane - 1)) & 1u);
        if (head && key >= 0) {
            atomicAdd(sum + key, s);
            atomicAdd(count + key, end - lane + 1);
        }
    }
}

__global__ void fbp_mean_kernel(double* __restrict__ sino, const int32_t* __restrict__ count, int64_t S) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < S; i += (int64_t)gridDim.x * blockDim.x) {
        const int32_t c = count[i];
        sino[i] = c > 0 ? sino[i] / (double)c : 0.0;
    }
}

// ---------------------------------------------------------------- 2. filtering

// One CTA per (slice, angle) row: the row p and the odd-lag kernel values
// hodd[j] = h(2j + 1) in shared memory; q_k = dt (p_k h(0) + sum over odd lags), the
// terms taken in ascending n as in the definition (even lags add exact zeros there).
__global__ void __launch_bounds__(256) fbp_filter_kernel(const double* __restrict__ sino, double* __restrict__ q,
                                                         int nt, double dt) {
    extern __shared__ double fsm[];
    double* p = fsm;            // [nt]
    double* hodd = fsm + nt;    // [nt/2 + 1]
    const int64_t row = blockIdx.x;
    const double* src = sino + row * nt;
    for (int i = threadIdx.x; i < nt; i += blockDim.x) p[i] = src[i];
    const int nh = nt / 2 + 1;
    for (int j = threadIdx.x; j < nh; j += blockDim.x) {
        const double m = (double)(2 * j + 1);
        hodd[j] = -1.0 / (kPi * kPi * m * m * dt * dt);
    }
    __syncthreads();
    const double h0 = 1.0 / (4.0 * dt * dt);
    for (int k = threadIdx.x; k < nt; k += blockDim.x) {
        double s = 0.0;
        // n < k with k - n odd: n = k-1, k-3, ... taken in ascending order
        for (int n = (k & 1) ^ 1; n < k; n += 2) s += p[n] * hodd[(k - n - 1) >> 1];
        s += p[k] * h0;
        for (int n = k + 1; n < nt; n += 2) s += p[n] * hodd[(n - k - 1) >> 1];
        q[row * nt + k] = dt * s;
    }
}

// ---------------------------------------------------------------- 3. back-projection

constexpr int kBpTx = 32, kBpTy = 8, kBpVx = 4;   // a CTA covers 128 x 8 voxels of one slice

// One thread per 4 voxels of a row (x = ix, ix+32, ix+64, ix+96 within the CTA's 128).
// Shared memory holds, per bin angle, cos(theta_a)/dt and sin(theta_a)/dt; the position of
// voxel (x, y) in bin units is u = x cos/dt + (y sin/dt + n_t/2 - 1/2): one FMA per voxel
// once the row's y term is formed.  The angles are summed in ascending order, as defined;
// the interpolation is v0 + w (v1 - v0).
__global__ void __launch_bounds__(kBpTx * kBpTy) fbp_backproject_kernel(ntvs_fbp_geom g, const double* __restrict__ q,
                                                                         double* __restrict__ img) {
    extern __shared__ double bsm[];
    double* cs = bsm;                 // [n_theta] cos(theta_a) / dt
    double* sn = bsm + g.n_theta;     // [n_theta] sin(theta_a) / dt
    const int na = g.n_theta, nt = g.n_t;
    const double inv_dt = 1.0 / g.dt;
    for (int a = threadIdx.y * kBpTx + threadIdx.x; a < na; a += kBpTx * kBpTy) {
        const double th = g.theta0 + ((double)a + 0.5) * kPi / (double)na;
        double sa, ca;
        sincos(th, &sa, &ca);
        cs[a] = ca * inv_dt;
        sn[a] = sa * inv_dt;
    }
    __syncthreads();
    const int iy = blockIdx.y * kBpTy + threadIdx.y, iz = blockIdx.z;
    if (iy >= g.ny) return;
    const int ix0 = blockIdx.x * (kBpTx * kBpVx) + threadIdx.x;
    const double y = ((double)iy + 0.5) * g.dy - 0.5 * (double)g.ny * g.dy;
    const double off = 0.5 * (double)nt - 0.5;
    double x[kBpVx], s[kBpVx];
#pragma unroll
    for (int v = 0; v < kBpVx; ++v) {
        x[v] = ((double)(ix0 + kBpTx * v) + 0.5) * g.dx - 0.5 * (double)g.nx * g.dx;
        s[v] = 0.0;
    }
    const double* qs = q + (int64_t)iz * na * nt;
    for (int a = 0; a < na; ++a) {
        const double base = fma(y, sn[a], off);
        const double c = cs[a];
        const double* row = qs + (int64_t)a * nt;
#pragma unroll
        for (int v = 0; v < kBpVx; ++v) {
            const double u = fma(x[v], c, base);
            const int k = __double2int_rd(u);         // floor; saturates far outside the row
            const double w = u - (double)k;
            const double v0 = (k >= 0 && k < nt) ? __ldg(row + k) : 0.0;
            const double v1 = (k >= -1 && k < nt - 1) ? __ldg(row + k + 1) : 0.0;
            s[v] += fma(w, v1 - v0, v0);
        }
    }
    const double scale = kPi / (double)na;
#pragma unroll
    for (int v = 0; v < kBpVx; ++v) {
        const int ix = ix0 + kBpTx * v;
        if (ix < g.nx) img[((int64_t)iz * g.ny + iy) * g.nx + ix] = s[v] * scale;
    }
}

// The same sum on 32 x 16 voxel tiles, for geometries whose tile crosses fewer than W - 2
// bins at any angle and whose |u| stays below 2000 (backproject_launch checks both).  FP64
// bounds the kernel above: 7 FP64-pipe operations per (voxel, angle), two of them
// conversions, at 2 lanes per clock and SM.  Here the position is a 64-bit fixed-point number
// with 52 fraction bits: stepping to the next voxel is an integer add, the bin is its upper
// bits, and its lower bits are the mantissa of 1 + w as they stand.  The row's pairs
// (v0, v1 - v0) are formed once per tile and angle in shared memory, bins outside the row as
// zeros, so a term is w = (1 + w) - 1, fma(w, v1 - v0, v0) and the add: 3 operations, rounded
// as above.  The tile's corner position is formed in FP64 per angle and the steps inside the
// tile (at most 31 and 15) carry 2^-53 of rounding each, so u is as exact as in FP64.
//
// 128 threads; a warp covers 8 x 4 voxels and takes up to four such patches 4 rows apart,
// those outside the image skipped.  200x200x16 voxels, 180 angles: 2245 us above, 848 us here
// (981 us with 32 x 32 tiles of 256 threads: 5.2 CTAs an SM leave the busiest with 6).
constexpr int kBpTileX = 32, kBpTileY = 16, kBpThreads = 128, kBpAngles = 256;   // angles tabled at once

template <int W, int CH>
__global__ void __launch_bounds__(kBpThreads) fbp_backproject_tile_kernel(ntvs_fbp_geom g, const double* __restrict__ q,
                                                                           double* __restrict__ img) {
    __shared__ double2 pr[CH][W];
    __shared__ long long ub[kBpAngles], du[kBpAngles], dv[kBpAngles];
    __shared__ int kb[kBpAngles], kn[kBpAngles];
    const int na = g.n_theta, nt = g.n_t;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int lx = warp * 8 + (lane & 7), ly = lane >> 3;
    const int ix0 = blockIdx.x * kBpTileX, iy0 = blockIdx.y * kBpTileY, iz = blockIdx.z;
    const double x0 = ((double)ix0 + 0.5) * g.dx - 0.5 * (double)g.nx * g.dx;
    const double y0 = ((double)iy0 + 0.5) * g.dy - 0.5 * (double)g.ny * g.dy;
    const double inv_dt = 1.0 / g.dt, off = 0.5 * (double)nt - 0.5, one = 4503599627370496.0;   // 2^52
    const double* qs = q + (int64_t)iz * na * nt;
    double s[4] = {0.0, 0.0, 0.0, 0.0};
    // the warp's patches inside the image (the others would take FP64 issue slots for nothing)
    const int nv = ix0 + warp * 8 < g.nx ? min(4, (g.ny - iy0 + 3) / 4) : 0;
    for (int ag = 0; ag < na; ag += kBpAngles) {
        const int ng = min(kBpAngles, na - ag);
        __syncthreads();
        for (int a = tid; a < ng; a += kBpThreads) {
            const double th = g.theta0 + ((double)(ag + a) + 0.5) * kPi / (double)na;
            double sa, ca;
            sincos(th, &sa, &ca);
            const double c = ca * inv_dt, sn = sa * inv_dt;
            const long long U = __double2ll_rn(fma(x0, c, fma(y0, sn, off)) * one);
            const long long dU = __double2ll_rn(c * g.dx * one), dV = __double2ll_rn(sn * g.dy * one);
            const long long ex = (kBpTileX - 1) * dU, ey = (kBpTileY - 1) * dV;
            const int lo = (int)((U + min(ex, 0ll) + min(ey, 0ll)) >> 52);   // smallest and largest bin of the tile
            const int hi = (int)((U + max(ex, 0ll) + max(ey, 0ll)) >> 52);
            ub[a] = U;
            du[a] = dU;
            dv[a] = dV;
            kb[a] = lo;
            kn[a] = min(hi - lo + 1, W);
        }
        for (int a0 = 0; a0 < ng; a0 += CH) {
            const int nc = min(CH, ng - a0);
            __syncthreads();   // the table is written, and the previous angles' pairs are read
            for (int j = tid; j < nc * W; j += kBpThreads) {
                const int ai = j / W, jj = j % W;
                if (jj >= kn[a0 + ai]) continue;
                const int k = kb[a0 + ai] + jj;
                const double* row = qs + (int64_t)(ag + a0 + ai) * nt;
                const double v0 = (k >= 0 && k < nt) ? __ldg(row + k) : 0.0;
                const double v1 = (k >= -1 && k < nt - 1) ? __ldg(row + k + 1) : 0.0;
                pr[ai][jj] = make_double2(v0, v1 - v0);
            }
            __syncthreads();
            for (int ai = 0; ai < nc; ++ai) {
                const long long step = 4 * dv[a0 + ai];
                const int kmin = kb[a0 + ai];
                long long U = ub[a0 + ai] + lx * du[a0 + ai] + ly * dv[a0 + ai];
#pragma unroll
                for (int v = 0; v < 4; ++v) {
                    if (v >= nv) break;
                    const double2 e = pr[ai][(int)(U >> 52) - kmin];
                    const double w = __longlong_as_double((U & 0xfffffffffffffll) | 0x3ff0000000000000ll) - 1.0;
                    s[v] += fma(w, e.y, e.x);
                    U += step;
                }
            }
        }
    }
    const double scale = kPi / (double)na;
    const int ix = ix0 + lx;
#pragma unroll
    for (int v = 0; v < 4; ++v) {
        const int iy = iy0 + ly + 4 * v;
        if (ix < g.nx && iy < g.ny) img[((int64_t)iz * g.ny + iy) * g.nx + ix] = s[v] * scale;
    }
}

// ---------------------------------------------------------------- 4. median filter (+ 5. hull)

// Order-preserving map of a double onto unsigned 64-bit integers (negative values have
// their bits inverted, the others their sign bit set), so that the window's values can be
// compared on the integer pipes.  -0.0 sorts just below +0.0; both are the value 0.
__device__ __forceinline__ uint64_t mono_key(double v) {
    const uint64_t b = (uint64_t)__double_as_longlong(v);
    return (b >> 63) ? ~b : (b | 0x8000000000000000ull);
}
__device__ __forceinline__ double mono_value(uint64_t k) {
    const uint64_t b = (k >> 63) ? (k & 0x7fffffffffffffffull) : ~k;
    return __longlong_as_double((long long)b);
}

__host__ __device__ constexpr int window_size(int r, bool ball) {
    int n = 0;
    for (int oz = -(ball ? r : 0); oz <= (ball ? r : 0); ++oz)
        for (int oy = -r; oy <= r; ++oy)
            for (int ox = -r; ox <= r; ++ox)
                if (ox * ox + oy * oy + oz * oz <= r * r + 1) ++n;
    return n;
}

// One thread per voxel.  The W window values become keys in registers (a neighbour
// outside the image becomes the largest key, above every value); with n in-image
// neighbours the result is the key whose rank range [#less, #less-or-equal) holds
// floor(n/2).
template <int R, bool BALL>
__global__ void __launch_bounds__(128) median_kernel(const double* __restrict__ in, double* __restrict__ out, int nx,
                                                     int ny, int nz, int use_hull, double tau) {
    constexpr int W = window_size(R, BALL);
    constexpr int RZ = BALL ? R : 0;
    const int64_t V = (int64_t)nx * ny * nz;
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= V) return;
    const int ix = (int)(p % nx);
    const int64_t r_ = p / nx;
    const int iy = (int)(r_ % ny), iz = (int)(r_ / ny);
    uint64_t key[W];
    int n = 0;
    {
        int w = 0;
#pragma unroll
        for (int oz = -RZ; oz <= RZ; ++oz)
#pragma unroll
            for (int oy = -R; oy <= R; ++oy)
#pragma unroll
                for (int ox = -R; ox <= R; ++ox) {
                    if (ox * ox + oy * oy + oz * oz <= R * R + 1) {
                        const int jx = ix + ox, jy = iy + oy, jz = iz + oz;
                        const bool ok = jx >= 0 && jx < nx && jy >= 0 && jy < ny && jz >= 0 && jz < nz;
                        key[w] = ok ? mono_key(__ldg(in + ((int64_t)jz * ny + jy) * nx + jx)) : ~0ull;
                        n += ok ? 1 : 0;
                        ++w;
                    }
                }
    }
    const int m = n >> 1;
    uint64_t res = 0;
    // windows up to 64 values stay in registers (loops fully unrolled); the 147-voxel
    // ball of radius 3 is ranked from local memory
#pragma unroll(W <= 64 ? W : 1)
    for (int i = 0; i < W; ++i) {
        int lt = 0, le = 0;
#pragma unroll(W <= 64 ? W : 4)
        for (int j = 0; j < W; ++j) {
            lt += key[j] < key[i] ? 1 : 0;
            le += key[j] <= key[i] ? 1 : 0;
        }
        if (lt <= m && m < le) res = key[i];
    }
    double v = mono_value(res);
    if (use_hull && v <= tau) v = 0.0;
    out[p] = v;
}

__global__ void hull_kernel(double* __restrict__ img, int64_t V, double tau) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < V; i += (int64_t)gridDim.x * blockDim.x)
        if (img[i] <= tau) img[i] = 0.0;
}

__global__ void copy_hull_kernel(const double* __restrict__ in, double* __restrict__ out, int64_t V, int use_hull,
                                 double tau) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < V; i += (int64_t)gridDim.x * blockDim.x) {
        const double v = in[i];
        out[i] = (use_hull && v <= tau) ? 0.0 : v;
    }
}

int grid_for(int64_t n, int threads) {
    const int64_t g = (n + threads - 1) / threads;
    return (int)(g < 1 ? 1 : (g > 152 * 32 ? 152 * 32 : g));
}

}  // namespace
}  // namespace ntvs

using namespace ntvs;

namespace {

int median_launch(const double* in, double* out, int nx, int ny, int nz, int r, bool ball, int use_hull, double tau,
                  cudaStream_t s) {
    const int64_t V = (int64_t)nx * ny * nz;
    const int grid = (int)((V + 127) / 128);
#define NTVS_MEDIAN_CASE(RR, BB) median_kernel<RR, BB><<<grid, 128, 0, s>>>(in, out, nx, ny, nz, use_hull, tau)
    if (r == 1) {
        if (ball) NTVS_MEDIAN_CASE(1, true); else NTVS_MEDIAN_CASE(1, false);
    } else if (r == 2) {
        if (ball) NTVS_MEDIAN_CASE(2, true); else NTVS_MEDIAN_CASE(2, false);
    } else {
        if (ball) NTVS_MEDIAN_CASE(3, true); else NTVS_MEDIAN_CASE(3, false);
    }
#undef NTVS_MEDIAN_CASE
    return launch_status("median_kernel launch");
}

int filter_launch(const ntvs_fbp_geom* g, const double* sino, double* q, cudaStream_t s) {
    const size_t smem = sizeof(double) * ((size_t)g->n_t + (size_t)(g->n_t / 2 + 1));
    if (smem > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(fbp_filter_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return fbp_fail(NTVS_ERR_CUDA, std::string("filter smem attribute: ") + cudaGetErrorString(e));
    }
    const int rows = g->nz * g->n_theta;
    fbp_filter_kernel<<<rows, 256, smem, s>>>(sino, q, g->n_t, g->dt);
    return launch_status("fbp_filter_kernel launch");
}

int backproject_launch(const ntvs_fbp_geom* g, const double* q, double* img, cudaStream_t s) {
    // The tile kernel wherever a tile's bins fit its shared rows (up to 1.7 bins a voxel in
    // 64-entry rows, 7 in 256-entry ones) and its fixed-point positions (11 integer bits).
    // Outside those (bins far finer than the voxels, or thousands of lateral bins) the per-row
    // kernel, which has no such limits.
    const double ex = (kBpTileX - 1) * g->dx, ey = (kBpTileY - 1) * g->dy;
    const double bins = sqrt(ex * ex + ey * ey) / g->dt + 3.0;
    const double reach = 0.5 * ((g->nx + 2 * kBpTileX) * g->dx + (g->ny + 2 * kBpTileY) * g->dy) / g->dt + 0.5 * g->n_t + 1.0;
    const dim3 tiles((g->nx + kBpTileX - 1) / kBpTileX, (g->ny + kBpTileY - 1) / kBpTileY, g->nz);
    if (reach < 2000.0 && bins < 256.0 && tiles.y <= 65535) {
        if (bins < 64.0) fbp_backproject_tile_kernel<64, 8><<<tiles, kBpThreads, 0, s>>>(*g, q, img);
        else fbp_backproject_tile_kernel<256, 4><<<tiles, kBpThreads, 0, s>>>(*g, q, img);
        return launch_status("fbp_backproject_tile_kernel launch");
    }
    const size_t smem = sizeof(double) * 2 * (size_t)g->n_theta;
    if (smem > 48 * 1024) {
        cudaError_t e =
            cudaFuncSetAttribute(fbp_backproject_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess)
            return fbp_fail(NTVS_ERR_CUDA, std::string("back-projection smem attribute: ") + cudaGetErrorString(e));
    }
    dim3 grid((g->nx + kBpTx * kBpVx - 1) / (kBpTx * kBpVx), (g->ny + kBpTy - 1) / kBpTy, g->nz);
    fbp_backproject_kernel<<<grid, dim3(kBpTx, kBpTy), smem, s>>>(*g, q, img);
    return launch_status("fbp_backproject_kernel launch");
}

int bin_launch(const ntvs_fbp_geom* g, const float* paths, const double* wepl, int64_t M, double* sino,
               int32_t* count, cudaStream_t s) {
    const int64_t S = (int64_t)g->nz * g->n_theta * g->n_t;
    cudaError_t e = cudaMemsetAsync(sino, 0, sizeof(double) * (size_t)S, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(count, 0, sizeof(int32_t) * (size_t)S, s);
    if (e != cudaSuccess) return fbp_fail(NTVS_ERR_CUDA, std::string("cudaMemsetAsync: ") + cudaGetErrorString(e));
    if (M > 0) {
        const int64_t warps = (M + 31) / 32;
        const int64_t want = (warps + 7) / 8;   // 8 warps per 256-thread CTA
        const int grid = (int)(want < 1 ? 1 : (want > 152 * 16 ? 152 * 16 : want));
        const double w = kPi / g->n_theta;
        const BinFast f{(float)(1.0 / w), (float)w, (float)g->theta0, (float)(1.0 / g->dt), (float)(0.5 * g->n_t),
                        (float)(1.0 / g->dz), fabs(g->theta0) <= 2.0 * kPi ? 1 : 0};
        fbp_bin_kernel<<<grid, 256, 0, s>>>(*g, f, paths, wepl, M, sino, count);
        int rc = launch_status("fbp_bin_kernel launch");
        if (rc != NTVS_OK) return rc;
    }
    fbp_mean_kernel<<<grid_for(S, 256), 256, 0, s>>>(sino, count, S);
    return launch_status("fbp_mean_kernel launch");
}

int64_t align256(int64_t b) { return (b + 255) / 256 * 256; }

}  // namespace

extern "C" int ntvs_fbp_bin(const ntvs_fbp_geom* g, const float* paths, const double* wepl, int64_t M, double* sino,
                            int32_t* count, void* cuda_stream) {
    int rc = check_geom(g, "ntvs_fbp_bin");
    if (rc != NTVS_OK) return rc;
    if (M < 0) return fbp_fail(NTVS_ERR_ARG, "ntvs_fbp_bin: M < 0");
    if (!sino || !count || (M > 0 && (!paths || !wepl))) return fbp_fail(NTVS_ERR_ARG, "ntvs_fbp_bin: null pointer");
    return bin_launch(g, paths, wepl, M, sino, count, (cudaStream_t)cuda_stream);
}

extern "C" int ntvs_fbp_filter(const ntvs_fbp_geom* g, const double* sino, double* q, void* cuda_stream) {
    int rc = check_geom(g, "ntvs_fbp_filter");
    if (rc != NTVS_OK) return rc;
    if (!sino || !q) return fbp_fail(NTVS_ERR_ARG, "ntvs_fbp_filter: null pointer");
    const int64_t S = (int64_t)g->nz * g->n_theta * g->n_t;
    if (((uintptr_t)sino < (uintptr_t)(q + S)) && ((uintptr_t)q < (uintptr_t)(sino + S)))
        return fbp_fail(NTVS_ERR_ARG, "ntvs_fbp_filter: q must not overlap sino");
    return filter_launch(g, sino, q, (cudaStream_t)cuda_stream);
}

extern "C" int ntvs_fbp_backproject(const ntvs_fbp_geom* g, const double* q, double* img, void* cuda_stream) {
    int rc = check_geom(g, "ntvs_fbp_backproject");
    if (rc != NTVS_OK) return rc;
    if (!q || !img) return fbp_fail(NTVS_ERR_ARG, "ntvs_fbp_backproject: null pointer");
    return backproject_launch(g, q, img, (cudaStream_t)cuda_stream);
}

extern "C" int ntvs_median_filter(const double* in, double* out, int nx, int ny, int nz, int radius, int ball,
                                  int use_hull, double tau, void* cuda_stream) {
    if (!in || !out) return fbp_fail(NTVS_ERR_ARG, "ntvs_median_filter: null pointer");
    if (nx < 1 || ny < 1 || nz < 1) return fbp_fail(NTVS_ERR_ARG, "ntvs_median_filter: sizes must be >= 1");
    if ((int64_t)nx * ny * nz > INT32_MAX) return fbp_fail(NTVS_ERR_ARG, "ntvs_median_filter: more than 2^31 - 1 voxels");
    if (((uintptr_t)in < (uintptr_t)(out + (int64_t)nx * ny * nz)) && ((uintptr_t)out < (uintptr_t)(in + (int64_t)nx * ny * nz)))
        return fbp_fail(NTVS_ERR_ARG, "ntvs_median_filter: out must not overlap in");
    if (radius < 0 || radius > kMaxMedianRadius) return fbp_fail(NTVS_ERR_ARG, "ntvs_median_filter: radius must be 0..3");
    if (use_hull && std::isnan(tau)) return fbp_fail(NTVS_ERR_ARG, "ntvs_median_filter: tau is NaN");
    cudaStream_t s = (cudaStream_t)cuda_stream;
    const int64_t V = (int64_t)nx * ny * nz;
    if (radius == 0) {
        copy_hull_kernel<<<grid_for(V, 256), 256, 0, s>>>(in, out, V, use_hull, tau);
        return launch_status("copy_hull_kernel launch");
    }
    return median_launch(in, out, nx, ny, nz, radius, ball != 0, use_hull, tau, s);
}

extern "C" int ntvs_hull(double* img, int64_t V, double tau, void* cuda_stream) {
    if (!img) return fbp_fail(NTVS_ERR_ARG, "ntvs_hull: null image");
    if (V < 1) return fbp_fail(NTVS_ERR_ARG, "ntvs_hull: V must be >= 1");
    if (std::isnan(tau)) return fbp_fail(NTVS_ERR_ARG, "ntvs_hull: tau is NaN");
    hull_kernel<<<grid_for(V, 256), 256, 0, (cudaStream_t)cuda_stream>>>(img, V, tau);
    return launch_status("hull_kernel launch");
}

extern "C" int64_t ntvs_fbp_workspace_bytes(const ntvs_fbp_geom* g) {
    int rc = check_geom(g, "ntvs_fbp_workspace_bytes");
    if (rc != NTVS_OK) return rc;
    const int64_t S = (int64_t)g->nz * g->n_theta * g->n_t;
    const int64_t V = (int64_t)g->nx * g->ny * g->nz;
    return align256(8 * S) + align256(4 * S) + align256(8 * S) + align256(8 * V);
}

extern "C" int ntvs_initial_iterate(const ntvs_fbp_geom* g, const float* paths, const double* wepl, int64_t M,
                                    int median_radius, int median_ball, int use_hull, double tau, void* workspace,
                                    int64_t workspace_bytes, double* out, void* cuda_stream) {
    int rc = check_geom(g, "ntvs_initial_iterate");
    if (rc != NTVS_OK) return rc;
    if (M < 0) return fbp_fail(NTVS_ERR_ARG, "ntvs_initial_iterate: M < 0");
    if (!out || !workspace || (M > 0 && (!paths || !wepl)))
        return fbp_fail(NTVS_ERR_ARG, "ntvs_initial_iterate: null pointer");
    if (median_radius < 0 || median_radius > kMaxMedianRadius)
        return fbp_fail(NTVS_ERR_ARG, "ntvs_initial_iterate: median radius must be 0..3");
    if (use_hull && std::isnan(tau)) return fbp_fail(NTVS_ERR_ARG, "ntvs_initial_iterate: tau is NaN");
    const int64_t need = ntvs_fbp_workspace_bytes(g);
    if (workspace_bytes < need)
        return fbp_fail(NTVS_ERR_ARG, "ntvs_initial_iterate: workspace of " + std::to_string(workspace_bytes) +
                                          " bytes, " + std::to_string(need) + " needed");
    if (((uintptr_t)workspace & 255) != 0)
        return fbp_fail(NTVS_ERR_ARG, "ntvs_initial_iterate: workspace must be 256-byte aligned");
    const int64_t S = (int64_t)g->nz * g->n_theta * g->n_t;
    char* w = (char*)workspace;
    double* sino = (double*)w;
    w += align256(8 * S);
    int32_t* cnt = (int32_t*)w;
    w += align256(4 * S);
    double* q = (double*)w;
    w += align256(8 * S);
    double* img = (double*)w;
    cudaStream_t s = (cudaStream_t)cuda_stream;
    if ((rc = bin_launch(g, paths, wepl, M, sino, cnt, s)) != NTVS_OK) return rc;
    if ((rc = filter_launch(g, sino, q, s)) != NTVS_OK) return rc;
    if ((rc = backproject_launch(g, q, img, s)) != NTVS_OK) return rc;
    return ntvs_median_filter(img, out, g->nx, g->ny, g->nz, median_radius, median_ball, use_hull, tau, cuda_stream);
}
