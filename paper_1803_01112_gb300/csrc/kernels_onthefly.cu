// On-the-fly DROP rows (P_T of arXiv 1803.01112 Appendix C with the system never stored):
// row i is the intersection-length vector of history i's path with the voxel grid
// (Sec. I: a row holds the lengths of one tracked proton's path through the voxels).
// A path is a chord P_in -> P_out plus cubic-Hermite offsets A h10(s) + B h11(s) along the
// in-plane normal and along z, split into n_seg straight segments; every sweep traces it
// again, in FP32: each segment is cut at every voxel plane it crosses (three per-axis
// crossing sequences merged in order) and each piece is credited to the voxel holding its
// midpoint.  Pieces shorter than min_len are dropped.  Only 44 bytes per history live in
// HBM (10 path floats + b); the work is ALU (tracing) and L2 atomics (scatter).
//
// Load time: one thread per row traces the whole path in order, merges consecutive pieces
// of one voxel (segment joins), and accumulates ||a_i||^2 (FP64) and the per-block hit
// counts s_j^t.
#include "common.cuh"

namespace ntvs {

namespace {

struct Grid3 {
    float ox, oy, oz, hx, hy, hz;
    float ihx, ihy, ihz;   // 1 / voxel size
    int nx, ny, nz;
    int ltx, lty, ntx;     // internal voxel order: tiles of 2^ltx x 2^lty, ntx tiles per row
    int slice_p;           // voxels per padded slice
};

// internal index (see VoxMap) of voxel (ix, iy, iz)
__device__ __forceinline__ int grid_index(const Grid3& g, int ix, int iy, int iz) {
    const int tile = (iy >> g.lty) * g.ntx + (ix >> g.ltx);
    return iz * g.slice_p + (tile << (g.ltx + g.lty)) + ((iy & ((1 << g.lty) - 1)) << g.ltx) +
           (ix & ((1 << g.ltx) - 1));
}

__device__ __forceinline__ float h10f(float s) { return s * s * s - 2.f * s * s + s; }
__device__ __forceinline__ float h11f(float s) { return s * s * s - s * s; }

// point of the path at parameter s
__device__ __forceinline__ void path_point(const float* pr, float nxv, float nyv, float s, float out[3]) {
    const float ol = pr[6] * h10f(s) + pr[7] * h11f(s), oz = pr[8] * h10f(s) + pr[9] * h11f(s);
    out[0] = pr[0] + s * (pr[3] - pr[0]) + ol * nxv;
    out[1] = pr[1] + s * (pr[4] - pr[1]) + ol * nyv;
    out[2] = pr[2] + s * (pr[5] - pr[2]) + oz;
}

// in-plane unit normal (-u_y, u_x) of the chord
__device__ __forceinline__ void chord_normal(const float* pr, float& nxv, float& nyv) {
    const float ux = pr[3] - pr[0], uy = pr[4] - pr[1];
    const float l = sqrtf(ux * ux + uy * uy);
    if (l > 0.f) { nxv = -uy / l; nyv = ux / l; }
    else { nxv = 1.f; nyv = 0.f; }
}

// The pieces of one straight segment P -> Q inside the grid, in order.  The segment is clipped
// to the grid, and each axis crosses its planes in order, plane k at t = (o + k h - P) / D
// (computed with the reciprocal of D).  Only planes inside the grid are crossings (an axis
// whose crossings are used up has t = 2), and their number is fixed before the walk, so the
// number of pieces is known in advance and the voxel, stepped by one along the axis of every
// crossing, stays inside the grid whatever the rounding of t.  The internal voxel index is a
// sum of three terms: x keeps its term with the bits of the tile's y offset free, so that a
// step is an add whose carry (or borrow) runs over those bits and a mask; y's term is formed
// from its index; z's steps by a slice.
//
// SEQ (the DROP sweep): an axis' later crossings are taken from its first one, t + j h / |D|, a
// counter and one FMA (151 against 172 us per 100k rows on 256x256x64).  They round
// differently from the plane formula by about an ulp of t, so the rows' statistics and stored
// rows, which decide by length which pieces count, keep the formula.
struct Walk {
    float t0, hi, L;
    float t[3], k[3], P[3], inv[3], c[3];   // next crossing, its plane, start, 1 / D, crossings left
                                            // (SEQ: k counts crossings, P the first t, inv their spacing)
    int fx, iy, fy, fz;   // x term, y index and its term, z term
    int sx, sy, sz;       // steps of fx, iy and fz
};

// the axis steps to its next plane
template <bool SEQ>
__device__ __forceinline__ void walk_cross(Walk& w, int a, float o, float h) {
    w.k[a] += SEQ ? 1.f : copysignf(1.f, w.inv[a]);
    w.c[a] -= 1.f;
    const float t = SEQ ? fmaf(w.k[a], w.inv[a], w.P[a]) : (o + w.k[a] * h - w.P[a]) * w.inv[a];
    w.t[a] = w.c[a] > 0.f ? t : 2.f;
}

// pieces of the segment (0: outside the grid); w is left at the first one
template <bool SEQ>
__device__ __forceinline__ int walk_begin(const Grid3& g, const float P[3], const float Q[3], Walk& w) {
    const float D[3] = {Q[0] - P[0], Q[1] - P[1], Q[2] - P[2]};
    w.L = sqrtf(D[0] * D[0] + D[1] * D[1] + D[2] * D[2]);
    if (!(w.L > 0.f)) return 0;
    const float o[3] = {g.ox, g.oy, g.oz}, h[3] = {g.hx, g.hy, g.hz}, ih[3] = {g.ihx, g.ihy, g.ihz};
    const int n[3] = {g.nx, g.ny, g.nz};
    float inv[3];
    float lo = 0.f, hi = 1.f;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const float e0 = o[a], e1 = o[a] + n[a] * h[a];
        inv[a] = D[a] != 0.f ? 1.f / D[a] : 0.f;
        if (D[a] == 0.f) {
            if (P[a] < e0 || P[a] > e1) return 0;
        } else {
            const float s0 = (e0 - P[a]) * inv[a], s1 = (e1 - P[a]) * inv[a];
            lo = fmaxf(lo, fminf(s0, s1));
            hi = fminf(hi, fmaxf(s0, s1));
        }
    }
    if (!(hi > lo)) return 0;
    w.t0 = lo;
    w.hi = hi;
    int idx[3], total = 1;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        w.P[a] = P[a];
        w.inv[a] = inv[a];
        w.k[a] = 0.f;
        float c = 0.f, t = 2.f;
        if (D[a] == 0.f) {
            idx[a] = min(max((int)floorf((P[a] - o[a]) * ih[a]), 0), n[a] - 1);
        } else {
            const float u = (P[a] + lo * D[a] - o[a]) * ih[a];
            const bool up = D[a] > 0.f;
            int k = up ? (int)floorf(u) + 1 : (int)ceilf(u) - 1;
            if ((o[a] + k * h[a] - P[a]) * inv[a] <= lo) k += up ? 1 : -1;   // the start lies on plane k
            k = up ? min(max(k, 1), n[a]) : min(max(k, 0), n[a] - 1);
            w.k[a] = (float)k;
            t = (o[a] + k * h[a] - P[a]) * inv[a];
            // planes k .. n - 1 upwards, k .. 1 downwards; as many of them as lie before hi (one
            // too many at most, which then makes an empty piece at hi)
            if (t < hi) c = fminf((float)(up ? n[a] - k : k), ceilf((hi - t) * fabsf(D[a]) * ih[a] + 1e-4f));
            idx[a] = up ? k - 1 : k;
        }
        if (SEQ) {
            w.k[a] = 0.f;
            w.P[a] = t;
            w.inv[a] = h[a] * fabsf(inv[a]);
        }
        w.c[a] = c;
        w.t[a] = c > 0.f ? t : 2.f;
        total += (int)c;
    }
    w.iy = idx[1];
    w.fx = grid_index(g, idx[0], 0, 0);
    w.fy = grid_index(g, 0, idx[1], 0);
    w.fz = idx[2] * g.slice_p;
    w.sx = D[0] > 0.f ? 1 + (((1 << g.lty) - 1) << g.ltx) : -1;
    w.sy = D[1] > 0.f ? 1 : -1;
    w.sz = D[2] > 0.f ? g.slice_p : -g.slice_p;
    return total;
}

// length of the current piece (0 when it is empty), then the step to the next one; v is the
// piece's voxel
template <bool SEQ>
__device__ __forceinline__ float walk_next(const Grid3& g, Walk& w, int& v) {
    const float m = fminf(fminf(w.t[0], w.t[1]), w.t[2]), t1 = fminf(m, w.hi), dt = t1 - w.t0;
    v = w.fx + w.fy + w.fz;
    w.t0 = t1;
    const bool px = w.t[0] == m, py = !px && w.t[1] == m;   // one axis steps; short enough to be predicated
    if (px) {
        w.fx = (w.fx + w.sx) & ~(((1 << g.lty) - 1) << g.ltx);
        walk_cross<SEQ>(w, 0, g.ox, g.hx);
    }
    if (py) {
        w.iy += w.sy;
        w.fy = (w.iy << g.ltx) + (w.iy >> g.lty) * ((g.ntx - 1) << (g.ltx + g.lty));
        walk_cross<SEQ>(w, 1, g.oy, g.hy);
    }
    if (!px && !py) {
        w.fz += w.sz;
        walk_cross<SEQ>(w, 2, g.oz, g.hz);
    }
    return dt > 1e-7f ? dt * w.L : 0.f;
}

// Calls f(voxel, length) for every piece of segment P -> Q inside the grid.
template <bool SEQ = false, typename F>
__device__ __forceinline__ void trace_segment(const Grid3& g, const float P[3], const float Q[3], F&& f) {
    Walk w;
    const int n = walk_begin<SEQ>(g, P, Q, w);
    for (int q = 0; q < n; ++q) {
        int v;
        const float l = walk_next<SEQ>(g, w, v);
        if (l > 0.f) f(v, l);
    }
}

// ---------------------------------------------------------------- load-time row statistics
__global__ void otf_prep_kernel(const float* __restrict__ paths, int64_t r0, int64_t r1, Grid3 g, int n_seg,
                                float min_len, float* __restrict__ inv_norm2, int32_t* __restrict__ cnt) {
    for (int64_t i = r0 + (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < r1;
         i += (int64_t)gridDim.x * blockDim.x) {
        float pr[10];
#pragma unroll
        for (int q = 0; q < 10; ++q) pr[q] = paths[i * 10 + q];
        float nxv, nyv;
        chord_normal(pr, nxv, nyv);
        double n2 = 0.0;
        int cur = -1;
        float acc = 0.f;
        auto close = [&]() {
            if (cur >= 0 && acc >= min_len) {
                n2 += (double)acc * (double)acc;
                atomicAdd(cnt + cur, 1);
            }
        };
        float A[3], B[3];
        path_point(pr, nxv, nyv, 0.f, A);
        for (int sg = 0; sg < n_seg; ++sg) {
            path_point(pr, nxv, nyv, (float)(sg + 1) / (float)n_seg, B);
            trace_segment(g, A, B, [&](int v, float l) {
                if (v == cur) { acc += l; return; }
                close();
                cur = v;
                acc = l;
            });
            A[0] = B[0]; A[1] = B[1]; A[2] = B[2];
        }
        close();
        inv_norm2[i] = n2 > 0.0 ? (float)(1.0 / n2) : 0.f;
    }
}

// ---------------------------------------------------------------- stored rows from paths
// Row i as the load-time statistics see it: the path traced in order by one thread,
// consecutive pieces of one voxel merged, merged pieces shorter than min_len dropped.
// Pass 1 counts the entries of every row; pass 2 writes them (voxel index in the order of
// g, length) from row_ptr[i].  Both passes run the same code, so they agree entry by entry.
template <bool FILL>
__global__ void otf_rows_kernel(const float* __restrict__ paths, int64_t M, Grid3 g, int n_seg, float min_len,
                                int32_t* __restrict__ nnz_row, const int64_t* __restrict__ row_ptr,
                                int32_t* __restrict__ col, float* __restrict__ val) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < M; i += (int64_t)gridDim.x * blockDim.x) {
        float pr[10];
#pragma unroll
        for (int q = 0; q < 10; ++q) pr[q] = paths[i * 10 + q];
        float nxv, nyv;
        chord_normal(pr, nxv, nyv);
        int64_t pos = FILL ? row_ptr[i] : 0;
        int n = 0;
        int cur = -1;
        float acc = 0.f;
        auto close = [&]() {
            if (cur >= 0 && acc >= min_len) {
                if (FILL) {
                    col[pos] = cur;
                    val[pos] = acc;
                    ++pos;
                }
                ++n;
            }
        };
        float A[3], B[3];
        path_point(pr, nxv, nyv, 0.f, A);
        for (int sg = 0; sg < n_seg; ++sg) {
            path_point(pr, nxv, nyv, (float)(sg + 1) / (float)n_seg, B);
            trace_segment(g, A, B, [&](int v, float l) {
                if (v == cur) { acc += l; return; }
                close();
                cur = v;
                acc = l;
            });
            A[0] = B[0]; A[1] = B[1]; A[2] = B[2];
        }
        close();
        if (!FILL) nnz_row[i] = n;
    }
}

// ---------------------------------------------------------------- the DROP block
// A warp takes two rows, 16 lanes each; lane s traces segments s, s + 16, ...  The pieces of
// both rows are laid out along their paths in the warp's piece buffer in shared memory: a
// segment's number of pieces is known before it is walked (walk_begin), so a prefix sum over
// the lanes gives every lane its place.  The dot product and the scatter then read the buffer
// with neighbouring lanes on neighbouring pieces, as the stored rows do: a gather or a
// reduction of 16 consecutive pieces touches about 6 sectors of the tiled voxel order.  With
// each lane on a segment of its own (the layout before this one) every lane touched a sector
// of its own, and the L2's atomic sectors bounded the kernel: 262 us per 100k rows of the
// 256x256x64 grid, 151 us with the buffer (issue slots 63 %, L2 42 %).
// Pieces that are empty or shorter than min_len keep their place with length 0 and take no
// part.  When a run of 16 segments a row does not fit into what is left of the buffer, it is
// gathered and scattered piece by piece as it is traced (once for each).
constexpr int kOtfThreads = 256;
constexpr int kOtfWarps = kOtfThreads / 32;

// Entries of a warp's buffer, from two rows' pieces on the grid's diagonal (every plane of x and y
// crossed; straight in z) with their segment joins: 54 or 72 KB a CTA and three CTAs an SM, 114 KB
// and two, or 225 KB and one.  Rows off the diagonal have fewer pieces (1.27 n on average on n x n voxels,
// against 2 n), so a size serves grids somewhat past its diagonal; what does not fit is walked twice.
// Where most rows do not, a few entries serve as well, with three CTAs and the L1 for the image: 1536x1536,
// 400k rows 5271 us with one CTA and 3773 so (4766 before the buffer), 1024x1024x2 3053 / 2979, 896x896x4
// 2668 / 2881.  Keeping the segments of such a row that fit, the others walked twice, was slower than
// either (5692 us on 2048x2048; 4516 / 2794) and cost the others 8 %.  Sweeps of 400k rows of 16 segments with three / two / one CTA, us (24 cached
// pieces a lane, before the buffer: last number):
//   256x256x16  669 / 704 / 1099 (1088)     512x512x16  2410 / 1483 / 1878 (2379)
//   320x320x16  913 / 837 / 1295 (1413)     576x576x16  3050 / 1962 / 2064 (2745)
//   448x448x16  1837 / 1142 / 1691 (2059)   640x640x8   2945 / 2352 / 2092 (2833)
//   1024x256x8  1886 / 1554 / 1666 (2019)   1024x1024x4 4566 / 4175 / 3253 (4302)
// Four CTAs, which fit with smaller buffers on small grids, spill: 64x64x8, 100k rows of 16 / 24
// segments, 155 / 205 us with four and 129 / 170 with three (152 / 173 before the buffer).
struct OtfBuffer {
    int entries, ctas;   // per warp; CTAs an SM
};
static OtfBuffer otf_buffer(const OtfArgs& a) {
    const int64_t need = 2 * ((int64_t)a.nx + a.ny + 2 * a.n_seg + 8);
    if (need <= 864) return {864, 3};
    if (need <= 1136) return {1136, 3};
    if (need <= 2500) return {1776, 2};
    if (need <= 4100) return {3520, 1};
    return {64, 3};   // no buffer to speak of
}

template <int MINB>
__global__ void __launch_bounds__(kOtfThreads, MINB) otf_drop_kernel(const float* __restrict__ paths,
                                                                   const float* __restrict__ b,
                                                                   const float* __restrict__ inv_norm2, int64_t r0,
                                                                   int64_t r1, Grid3 g, int n_seg, float min_len,
                                                                   const float* __restrict__ x,
                                                                   float* __restrict__ delta, float lambda,
                                                                   double* resid_ss, int cap) {
    constexpr int LPR = 16;
    extern __shared__ __align__(16) unsigned char otf_smem[];
    const int tid = threadIdx.x;
    const int lane = tid & 31, sub = lane % LPR, half = lane / LPR;
    int2* buf = reinterpret_cast<int2*>(otf_smem) + (size_t)(tid >> 5) * cap;   // {voxel, length bits}
    const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + tid) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    double ss = 0.0;
    for (int64_t base = r0 + warp * 2; base < r1; base += nwarps * 2) {
        const int64_t i = base + half;
        const bool valid = i < r1;
        // the ends of segment sg of the row (the record is read again for every run of segments:
        // kept in registers over the walk it spilled)
        auto ends = [&](int sg, float A[3], float B[3]) {
            float pr[10], nxv, nyv;
#pragma unroll
            for (int q = 0; q < 10; ++q) pr[q] = __ldg(paths + i * 10 + q);
            chord_normal(pr, nxv, nyv);
            path_point(pr, nxv, nyv, (float)sg / (float)n_seg, A);
            path_point(pr, nxv, nyv, (float)(sg + 1) / (float)n_seg, B);
        };
        float acc = 0.f;
        int used = 0;   // the row's pieces in the buffer: the first row's from its start, the second's up to its end
        int sg0 = 0;    // segments [0, sg0) are in the buffer
        bool fits = true;
        for (int s0 = 0; s0 < n_seg; s0 += LPR) {
            const int sg = s0 + sub;
            Walk w;
            int n = 0;
            if (valid && sg < n_seg) {
                float A[3], B[3];
                ends(sg, A, B);
                n = walk_begin<true>(g, A, B, w);
            }
            int at = n;   // inclusive prefix sum over the row's lanes
#pragma unroll
            for (int o = 1; o < LPR; o <<= 1) {
                const int u = __shfl_up_sync(0xffffffffu, at, o, LPR);
                if (sub >= o) at += u;
            }
            const int tot = __shfl_sync(0xffffffffu, at, LPR - 1, LPR);
            const int both = used + tot + __shfl_xor_sync(0xffffffffu, used + tot, LPR);
            fits = fits && both <= cap;   // warp-uniform
            if (fits) {
                at = (half ? cap - used - tot : used) + at - n;
                used += tot;
                sg0 = s0 + LPR;
                for (int q = 0; q < n; ++q) {
                    int v;
                    const float l = walk_next<true>(g, w, v);
                    buf[at + q] = make_int2(v, __float_as_int(l >= min_len ? l : 0.f));
                }
            } else {
                for (int q = 0; q < n; ++q) {
                    int v;
                    const float l = walk_next<true>(g, w, v);
                    if (l > 0.f && l >= min_len) acc += l * __ldg(x + v);
                }
            }
        }
        __syncwarp();
        const int2* mine = buf + (half ? cap - used : 0);
        const int most = max(used, __shfl_xor_sync(0xffffffffu, used, LPR));
        for (int q = sub; q < most; q += 4 * LPR) {   // four gathers in flight
            float xv[4], lv[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int2 e = q + u * LPR < used ? mine[q + u * LPR] : make_int2(0, 0);
                lv[u] = __int_as_float(e.y);
                xv[u] = lv[u] > 0.f ? __ldg(x + e.x) : 0.f;
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) acc += lv[u] * xv[u];
        }
#pragma unroll
        for (int o = LPR / 2; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        const float res = valid ? __ldg(b + i) - acc : 0.f;
        const float r = valid ? lambda * res * __ldg(inv_norm2 + i) : 0.f;
        if (valid && sub == 0) ss += (double)res * (double)res;
        for (int q = sub; q < used; q += LPR) {
            const int2 e = mine[q];
            const float l = __int_as_float(e.y);
            if (l > 0.f) atomicAdd(delta + e.x, r * l);
        }
        for (int sg = sg0 + sub; valid && sg < n_seg; sg += LPR) {   // segments past the buffer
            float A[3], B[3];
            ends(sg, A, B);
            trace_segment<true>(g, A, B, [&](int v, float l) {
                if (l >= min_len) atomicAdd(delta + v, r * l);
            });
        }
        __syncwarp();   // the buffer is read: the next rows may overwrite it
    }
    __shared__ double sh[32];
    const double tot = block_sum(ss, sh);
    if (threadIdx.x == 0 && tot != 0.0) atomicAdd(resid_ss, tot);
}

// ---------------------------------------------------------------- forward projection
// out_i = sum of l * x_v over the accepted pieces (voxel v, length l >= min_len) of history
// i's path, the stored rows' lengths (the DROP sweeps step their crossings and differ by about an
// ulp of t in each); 16 lanes per row, each tracing every 16th segment.
__global__ void __launch_bounds__(256) otf_project_kernel(const float* __restrict__ paths, int64_t M, Grid3 g,
                                                           int n_seg, float min_len, const float* __restrict__ x,
                                                           void* __restrict__ out, int out64) {
    constexpr int LPR = 16;
    const int lane = threadIdx.x & 31, sub = lane % LPR;
    const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t base = warp * 2; base < M; base += nwarps * 2) {
        const int64_t i = base + lane / LPR;
        const bool valid = i < M;
        float acc = 0.f;
        if (valid) {
            float pr[10];
#pragma unroll
            for (int q = 0; q < 10; ++q) pr[q] = __ldg(paths + i * 10 + q);
            float nxv, nyv;
            chord_normal(pr, nxv, nyv);
            for (int sg = sub; sg < n_seg; sg += LPR) {
                float A[3], B[3];
                path_point(pr, nxv, nyv, (float)sg / (float)n_seg, A);
                path_point(pr, nxv, nyv, (float)(sg + 1) / (float)n_seg, B);
                trace_segment(g, A, B, [&](int v, float l) {
                    if (l >= min_len) acc += l * __ldg(x + v);
                });
            }
        }
#pragma unroll
        for (int o = LPR / 2; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        if (valid && sub == 0) {
            if (out64) static_cast<double*>(out)[i] = (double)acc;
            else static_cast<float*>(out)[i] = acc;
        }
    }
}

// History data (P_in, P_out, d_in, d_out) -> path record (P_in, P_out, A_lat, B_lat, A_z, B_z):
// end tangents m = L d / |d| (chord direction for a zero d), deviations m - c projected on
// the chord's in-plane normal and on z.  flags |= 32 on a non-finite history value.
__global__ void hist_to_paths_kernel(const float* __restrict__ hist, int64_t M, float* __restrict__ rec, int* flags) {
    int f = 0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < M; i += (int64_t)gridDim.x * blockDim.x) {
        float h[12];
#pragma unroll
        for (int q = 0; q < 12; ++q) {
            h[q] = hist[i * 12 + q];
            if (!isfinite(h[q])) f |= 32;
        }
        const float c[3] = {h[3] - h[0], h[4] - h[1], h[5] - h[2]};
        const float L = sqrtf(c[0] * c[0] + c[1] * c[1] + c[2] * c[2]);
        float pr[10] = {h[0], h[1], h[2], h[3], h[4], h[5], 0.f, 0.f, 0.f, 0.f};
        float nxv, nyv;
        chord_normal(pr, nxv, nyv);
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const float* d = h + 6 + 3 * e;
            const float dl = sqrtf(d[0] * d[0] + d[1] * d[1] + d[2] * d[2]);
            float m[3];
#pragma unroll
            for (int a = 0; a < 3; ++a) m[a] = dl > 0.f ? L * (d[a] / dl) : c[a];
            const float dev[3] = {m[0] - c[0], m[1] - c[1], m[2] - c[2]};
            pr[6 + e] = dev[0] * nxv + dev[1] * nyv;   // A_lat, B_lat
            pr[8 + e] = dev[2];                         // A_z, B_z
        }
#pragma unroll
        for (int q = 0; q < 10; ++q) rec[i * 10 + q] = pr[q];
    }
    if (f) atomicOr(flags, f);
}

// paths finite, n_seg sane: flags |= 32 on a non-finite path value, 16 on a non-finite b
__global__ void otf_validate_kernel(const float* __restrict__ paths, const float* __restrict__ b, int64_t M,
                                    int* flags) {
    int f = 0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < M; i += (int64_t)gridDim.x * blockDim.x) {
        for (int q = 0; q < 10; ++q)
            if (!isfinite(paths[i * 10 + q])) f |= 32;
        if (!isfinite(b[i])) f |= 16;
    }
    if (f) atomicOr(flags, f);
}

}  // namespace

static Grid3 make_grid(const OtfArgs& a) {
    Grid3 g;
    g.nx = a.nx; g.ny = a.ny; g.nz = a.nz;
    g.hx = (float)a.dx; g.hy = (float)a.dy; g.hz = (float)a.dz;
    g.ihx = 1.f / g.hx; g.ihy = 1.f / g.hy; g.ihz = 1.f / g.hz;
    g.ltx = a.vm.ltx; g.lty = a.vm.lty;
    g.ntx = a.vm.nxp >> a.vm.ltx;
    g.slice_p = (int)a.vm.slice_p;
    g.ox = (float)(-0.5 * a.nx * a.dx); g.oy = (float)(-0.5 * a.ny * a.dy); g.oz = 0.f;
    return g;
}

cudaError_t k_hist_to_paths(const float* hist, int64_t M, float* rec, int* flags, int grid, cudaStream_t s) {
    if (M <= 0) return cudaSuccess;
    hist_to_paths_kernel<<<grid, 256, 0, s>>>(hist, M, rec, flags);
    return cudaGetLastError();
}

cudaError_t k_otf_validate(const OtfArgs& a, int* flags, cudaStream_t s) {
    if (a.M <= 0) return cudaSuccess;
    otf_validate_kernel<<<a.grid, 256, 0, s>>>(a.paths, a.b, a.M, flags);
    return cudaGetLastError();
}

cudaError_t k_otf_prep(const OtfArgs& a, int64_t r0, int64_t r1, float* inv_norm2, int32_t* cnt, cudaStream_t s) {
    if (r1 <= r0) return cudaSuccess;
    otf_prep_kernel<<<a.grid, 128, 0, s>>>(a.paths, r0, r1, make_grid(a), a.n_seg, a.min_len, inv_norm2, cnt);
    return cudaGetLastError();
}

cudaError_t k_otf_drop(const OtfArgs& a, int64_t r0, int64_t r1, const float* inv_norm2, const float* x, float* delta,
                       double lambda, double* resid_ss, cudaStream_t s) {
    if (r1 <= r0) return cudaSuccess;
    const OtfBuffer buf = otf_buffer(a);
    const size_t smem = (size_t)buf.entries * kOtfWarps * sizeof(int2);
    auto kern = buf.ctas == 3 ? otf_drop_kernel<3> : otf_drop_kernel<2>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    const int grid = a.grid / 8 * buf.ctas;   // a.grid: 8 CTAs per SM; one resident wave
    kern<<<grid < 1 ? 1 : grid, kOtfThreads, smem, s>>>(a.paths, a.b, inv_norm2, r0, r1, make_grid(a), a.n_seg, a.min_len, x, delta,
                                           (float)lambda, resid_ss, buf.entries);
    return cudaGetLastError();
}

cudaError_t k_otf_count_rows(const OtfArgs& a, int32_t* nnz_row, cudaStream_t s) {
    if (a.M <= 0) return cudaSuccess;
    otf_rows_kernel<false><<<a.grid, 128, 0, s>>>(a.paths, a.M, make_grid(a), a.n_seg, a.min_len, nnz_row, nullptr,
                                                  nullptr, nullptr);
    return cudaGetLastError();
}

cudaError_t k_otf_fill_rows(const OtfArgs& a, const int64_t* row_ptr, int32_t* col, float* val, cudaStream_t s) {
    if (a.M <= 0) return cudaSuccess;
    otf_rows_kernel<true><<<a.grid, 128, 0, s>>>(a.paths, a.M, make_grid(a), a.n_seg, a.min_len, nullptr, row_ptr,
                                                 col, val);
    return cudaGetLastError();
}

cudaError_t k_otf_project(const OtfArgs& a, const float* x, void* out, int out64, cudaStream_t s) {
    if (a.M <= 0) return cudaSuccess;
    otf_project_kernel<<<a.grid, 256, 0, s>>>(a.paths, a.M, make_grid(a), a.n_seg, a.min_len, x, out, out64);
    return cudaGetLastError();
}

}  // namespace ntvs
