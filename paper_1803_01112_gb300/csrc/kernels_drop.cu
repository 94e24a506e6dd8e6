// Block-DROP kernels (P_T of arXiv 1803.01112 Appendix C; DROP of ref. CEHN08, Sec. III-D).
//
// drop_block: for every row i of block t (all rows see the same x):
//     d_i = <a_i, x>                    (CSR gather, x is L2/L1-resident)
//     r_i = lambda (b_i - d_i) / ||a_i||^2
//     delta_j += r_i a_ij               (scatter-add)
//   A group of LPR lanes owns a row; each lane loads VW consecutive entries per step
//   (16-byte column and value vectors for 4-byte values), and the row's entries stay in
//   registers between the dot product and the scatter, so the matrix streams from HBM
//   exactly once.
//
//   Windowed variant (one 1024-thread CTA per SM): the CTA owns a list of row segments
//   that share a "home" z-slice (assigned at load time), keeps delta for that slice in
//   shared memory and scatters there with shared-memory atomics; entries outside the
//   slice go to global memory.  When the home slice changes, and at the end, the window
//   is flushed into delta with one global reduction per touched voxel.  This replaces
//   ~1 global L2 atomic per matrix entry by ~0.2.
//   Plain variant (any row order): every scatter is a global reduction.
// drop_apply: x_j += delta_j / s_j^t (inverse counts precomputed), delta_j = 0.
#include "kernels_drop.cuh"

namespace ntvs {

template <typename T, int U>
__global__ void __launch_bounds__(256) drop_apply_kernel(double* __restrict__ x, ImgCopies c, T* __restrict__ delta,
                                                         const T* __restrict__ inv_s, int64_t V,
                                                         const float* __restrict__ wlog, int ctas, float rows,
                                                         float* rms) {
    // The last CTA forms the residual that scales the next block's window.  Read by that launch itself,
    // the windowed CTAs' values delayed it by 1.7 us of 7 on a small image; here they cost nothing.
    const int vox_ctas = gridDim.x - (wlog ? 1 : 0);
    if (blockIdx.x == vox_ctas) {
        float2 sums = make_float2(0.f, 0.f);
        for (int c = threadIdx.x; threadIdx.x < 32 && c < ctas; c += 32) {
            const float v = __ldg(wlog + c);
            if (v != INFINITY) sums.x += v, sums.y += 1.f;
        }
        for (int o = 16; o > 0; o >>= 1) {
            sums.x += __shfl_xor_sync(0xffffffffu, sums.x, o);
            sums.y += __shfl_xor_sync(0xffffffffu, sums.y, o);
        }
        if (threadIdx.x == 0) *rms = win_rms(sums, rows);
        return;
    }
    const int64_t stride = (int64_t)vox_ctas * blockDim.x;
    for (int64_t j0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j0 < V; j0 += U * stride) {
        double xv[U];
        T dv[U], sv[U];
        uint32_t p[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int64_t j = min(j0 + u * stride, V - 1);   // clamped: the loads issue together
            p[u] = (uint32_t)vox_internal(c.m, j);
            xv[u] = x[j];
            dv[u] = delta[p[u]];
            sv[u] = __ldg(inv_s + p[u]);
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int64_t j = j0 + u * stride;
            // an untouched voxel keeps its value and its gather copy
            if (j >= V || (dv[u] == (T)0 && !c.xh)) continue;
            const double v = xv[u] + (double)dv[u] * (double)sv[u];
            x[j] = v;
            store_copies(c, j, p[u], v);
            delta[p[u]] = (T)0;
        }
    }
}

// A thread per voxel; the copies' loads go out together, eight at a time.
__global__ void __launch_bounds__(256) drop_apply_copies_kernel(double* __restrict__ x, double* __restrict__ delta,
                                                                int copies, int64_t stride,
                                                                const double* __restrict__ inv_s, int64_t V) {
    const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= V) return;
    double d = 0.0;
    for (int r0 = 0; r0 < copies; r0 += 8) {
        double v[8];
#pragma unroll
        for (int r = 0; r < 8; ++r) v[r] = r0 + r < copies ? delta[(r0 + r) * stride + j] : 0.0;
#pragma unroll
        for (int r = 0; r < 8; ++r) {
            d += v[r];
            if (v[r] != 0.0) delta[(r0 + r) * stride + j] = 0.0;
        }
    }
    if (d != 0.0) x[j] += d * __ldg(inv_s + j);
}

cudaError_t k_drop_apply_copies(double* x, double* delta, int copies, int64_t delta_stride, const double* inv_s,
                                int64_t V, cudaStream_t s) {
    if (V <= 0) return cudaSuccess;
    drop_apply_copies_kernel<<<(unsigned)((V + 255) / 256), 256, 0, s>>>(x, delta, copies, delta_stride, inv_s, V);
    return cudaGetLastError();
}

int64_t k_window_smem_bytes(int64_t slice, int csz, bool d16) {
    return (int64_t)window_smem_bytes(slice, (size_t)csz, d16);
}

cudaError_t k_drop_block(const DropArgs& a, cudaStream_t s) {
    if (a.r1 <= a.r0) return cudaSuccess;
    if (a.use_d16) return k_drop_block_d16(a, s);
    if (a.cdt == F64) {   // FP64 arithmetic on FP64 or FP32 storage
        if (a.vector4) return cudaErrorInvalidValue;
        if (a.vdt == F64) return dispatch<double, double, false>(a, s);
        if (a.vdt == F32) return dispatch<double, float, false>(a, s);
        return cudaErrorInvalidValue;
    }
    switch (a.vdt) {
        case F32: return dispatch<float, float, false>(a, s);
        case F16: return dispatch<float, __half, false>(a, s);
        case BF16: return dispatch<float, __nv_bfloat16, false>(a, s);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t k_drop_apply(int cdt, double* x, ImgCopies c, void* delta, const void* inv_s, int64_t V, int grid,
                         const float* wlog, int ctas, int64_t rows, float* rms, cudaStream_t s) {
    const bool many = vox_unrolled(V, grid);
    if (wlog) ++grid;
    if (cdt == F64)
        (many ? drop_apply_kernel<double, kVoxUnroll> : drop_apply_kernel<double, 1>)<<<grid, 256, 0, s>>>(
            x, c, (double*)delta, (const double*)inv_s, V, wlog, ctas, (float)rows, rms);
    else
        (many ? drop_apply_kernel<float, kVoxUnroll> : drop_apply_kernel<float, 1>)<<<grid, 256, 0, s>>>(
            x, c, (float*)delta, (const float*)inv_s, V, wlog, ctas, (float)rows, rms);
    return cudaGetLastError();
}

// out_i = <a_i, x> for rows [0, M) (x in the gather order of the stored columns), for CSR32
// (packed pairs for FP32 values) or DELTA16 storage (words for 16-bit values); accumulated in
// the compute type T, written as double when out64 is set, else as float.
//
// A warp takes up to 8 consecutive rows: their extents come with one load and their results leave
// with one (row by row, a warp a row, each result was a 4-byte write to a sector of its own), and
// while a row is summed the next one's lines are on their way to L2.  Up to 8 entries a lane
// are loaded before their gathers, summed in the order of the entries.  2M rows of 255 FP32
// pairs: 816 us with one row and one entry at a time, 684 us (0.94 of the measured copy rate).
// Fewer rows than 8 for every warp of the grid go fewer to a warp, so that no warp idles (FEW: the
// number at run time, and the lines of a long row asked of L2 four runs of entries ahead, as its
// warp has no next row to wait behind).  A call on 5000 FP64 rows of 2000 entries took 485 us with 8
// rows a warp and takes 70 so, on 100 rows of 100 000 FP32 pairs 8020 and 476.
constexpr int kProjRows = 8, kProjStep = 8;

template <typename T, typename V, bool D16, bool FEW>
__global__ void __launch_bounds__(256)
project_kernel(const int64_t* __restrict__ row_ptr, const int32_t* __restrict__ col, Delta16 d16,
               const V* __restrict__ val, int64_t M, int few, const T* __restrict__ x, void* __restrict__ out,
               int out64) {
    const int rows = FEW ? few : kProjRows;
    const int lane = threadIdx.x & 31;
    const int64_t w0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t base = w0 * rows; base < M; base += nw * rows) {
        const int n = (int)min((int64_t)rows, M - base);
        const int64_t rp = lane <= n ? __ldg(row_ptr + base + lane) : 0;
        T mine = (T)0;
        for (int r = 0; r < n; ++r) {
            const int64_t p0 = __shfl_sync(0xffffffffu, rp, r), p1 = __shfl_sync(0xffffffffu, rp, r + 1);
            if constexpr (packed_entries<V, D16>()) {
                const int64_t p2 = __shfl_sync(0xffffffffu, rp, min(r + 2, n));
                prefetch_lines_l2(reinterpret_cast<const int2*>(col), p1, p2, lane);
            }
            const int32_t* cbr = D16 ? d16.cbase + (p0 >> 5) + base + r : nullptr;
            T acc = (T)0;
            for (int64_t p = p0 + lane; p < p1; p += 32 * kProjStep) {
                if constexpr (FEW && packed_entries<V, D16>()) {
                    const int64_t q = p - lane + 4 * 32 * kProjStep + 16 * lane;
                    if (lane < 2 * kProjStep && q < p1)
                        asm volatile("prefetch.global.L2 [%0];" ::"l"(reinterpret_cast<const int2*>(col) + q));
                }
                int32_t c[kProjStep];
                T a[kProjStep];
#pragma unroll
                for (int u = 0; u < kProjStep; ++u) {
                    const int64_t q = p + 32 * u;
                    c[u] = -1;
                    a[u] = (T)0;
                    if (q < p1) {
                        if constexpr (packed_entries<V, D16>()) {
                            const int2 e = __ldcs(reinterpret_cast<const int2*>(col) + q);
                            c[u] = e.x;
                            a[u] = (T)__int_as_float(e.y);
                        } else {
                            entry_any<T, V, D16>(col, d16, val, cbr, q, (int)(q - p0), c[u], a[u]);
                        }
                    }
                }
                // FP64: the steps past the row's end are skipped, not predicated off, since a predicated FMA
                // takes its 16 cycles of the FP64 pipe all the same (1M rows of 30 entries: 826 us a call with
                // them, 395 so, 601 with one row and one entry at a time)
                const int64_t left = p1 - (p - lane);
#pragma unroll
                for (int u = 0; u < kProjStep; ++u) {
                    if (sizeof(T) == 8 && 32 * u >= left) break;
                    if (c[u] >= 0) acc += a[u] * __ldg(x + c[u]);
                }
            }
            for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
            if (lane == r) mine = acc;
        }
        if (lane < n) {
            if (out64) static_cast<double*>(out)[base + lane] = (double)mine;
            else static_cast<float*>(out)[base + lane] = (float)mine;
        }
    }
}

template <typename T, typename V>
static cudaError_t launch_project(const DropArgs& a, int64_t M, const void* x, void* out, int out64, cudaStream_t s) {
    const int64_t warps = (int64_t)a.grid * 8;   // 8 a CTA
    const int64_t each = (M + warps - 1) / warps;
    const int rows = (int)(each < kProjRows ? each : kProjRows);
    const int64_t need = (M + 8 * rows - 1) / (8 * rows);
    const int grid = (int)(need < a.grid ? need : a.grid);
    const bool few = rows < kProjRows;
    const auto kern = a.use_d16 ? (few ? project_kernel<T, V, true, true> : project_kernel<T, V, true, false>)
                                : (few ? project_kernel<T, V, false, true> : project_kernel<T, V, false, false>);
    kern<<<grid, 256, 0, s>>>(a.row_ptr, a.col, a.d16, (const V*)a.val, M, rows, (const T*)x, out, out64);
    return cudaGetLastError();
}

// word[p] = off[p] | val[p] << 16 (16-bit value bits) for entries [0, n)
__global__ void pack_words_kernel(const uint16_t* __restrict__ off, const uint16_t* __restrict__ val, int64_t n,
                                  uint32_t* __restrict__ word) {
    for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < n; p += (int64_t)gridDim.x * blockDim.x)
        word[p] = (uint32_t)__ldcs(off + p) | ((uint32_t)__ldcs(val + p) << 16);
}

cudaError_t k_pack_words(const uint16_t* off, const uint16_t* val, int64_t n, uint32_t* word, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    const int64_t need = (n + 255) / 256;
    const int grid = (int)(need < 4096 ? need : 4096);
    pack_words_kernel<<<grid, 256, 0, s>>>(off, val, n, word);
    return cudaGetLastError();
}

cudaError_t k_project(const DropArgs& a, int64_t M, const void* x, void* out, int out64, cudaStream_t s) {
    if (M <= 0) return cudaSuccess;
    if (a.cdt == F64) {
        if (a.vdt == F64) return launch_project<double, double>(a, M, x, out, out64, s);
        if (a.vdt == F32) return launch_project<double, float>(a, M, x, out, out64, s);
        return cudaErrorInvalidValue;
    }
    switch (a.vdt) {
        case F32: return launch_project<float, float>(a, M, x, out, out64, s);
        case F16: return launch_project<float, __half>(a, M, x, out, out64, s);
        case BF16: return launch_project<float, __nv_bfloat16>(a, M, x, out, out64, s);
        default: return cudaErrorInvalidValue;
    }
}

// *out = max(*out, longest row of rows [r0, r1))
__global__ void row_maxlen_kernel(const int64_t* __restrict__ row_ptr, int64_t r0, int64_t r1, unsigned long long* out) {
    unsigned long long m = 0;
    for (int64_t i = r0 + (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < r1; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t l = row_ptr[i + 1] - row_ptr[i];
        m = l > (int64_t)m ? (unsigned long long)l : m;
    }
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long v = __shfl_xor_sync(0xffffffffu, m, o);
        m = v > m ? v : m;
    }
    if ((threadIdx.x & 31) == 0 && m) atomicMax(out, m);
}

cudaError_t k_row_maxlen(const int64_t* row_ptr, int64_t r0, int64_t r1, unsigned long long* out, int grid,
                         cudaStream_t s) {
    if (r1 <= r0) return cudaSuccess;
    row_maxlen_kernel<<<grid, 256, 0, s>>>(row_ptr, r0, r1, out);
    return cudaGetLastError();
}

// home slice of each row: the median of the z-slices of its first, middle and last
// entries (-1 for an empty row); a path that bends out of its slice and back keeps the
// slice it enters and leaves by.  Entry p's column is col[stride * p] (stride 2: the
// packed pairs).
__global__ void row_home_kernel(const int64_t* __restrict__ row_ptr, const int32_t* __restrict__ col, int stride,
                                int64_t M, int64_t slice, int32_t* __restrict__ home) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < M; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t p0 = row_ptr[i], p1 = row_ptr[i + 1];
        if (p1 <= p0) { home[i] = -1; continue; }
        const int32_t a = (int32_t)(col[stride * p0] / slice), m = (int32_t)(col[stride * (p0 + (p1 - p0) / 2)] / slice),
                      c = (int32_t)(col[stride * (p1 - 1)] / slice);
        home[i] = max(min(a, m), min(max(a, m), c));
    }
}

cudaError_t k_row_home(const int64_t* row_ptr, const int32_t* col, int stride, int64_t M, int64_t slice, int32_t* home,
                       int grid, cudaStream_t s) {
    if (M <= 0) return cudaSuccess;
    row_home_kernel<<<grid, 256, 0, s>>>(row_ptr, col, stride, M, slice, home);
    return cudaGetLastError();
}

// A warp per chunk of rows: the chunk's work in issued register steps (k_chunk_cost); a
// chunk of a block without a per-block depth (ch = 0) counts its rows
__global__ void chunk_cost_kernel(const int64_t* __restrict__ row_ptr, const int32_t* __restrict__ order,
                                  const int64_t* __restrict__ cs,
                                  const int8_t* __restrict__ ch, int mid, int64_t nchunks, int64_t* __restrict__ cost) {
    const int lane = threadIdx.x & 31;
    const int64_t w0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t q = w0; q < nchunks; q += nw) {
        const int64_t r0 = cs[q], r1 = cs[q + 1];
        const int64_t d = ch[q];
        long long acc = 0;
        for (int64_t i = r0 + lane; i < r1; i += 32) {
            if (d <= 0) {
                acc += 4;
                continue;
            }
            const int64_t row = order ? order[i] : i;
            const int64_t steps = (row_ptr[row + 1] - row_ptr[row] + 31) / 32;
            const int64_t body = (steps <= kShortBody && d > kShortBody) ? kShortBody
                                 : (mid > 0 && d > mid && steps <= mid) ? mid : d;
            const int64_t live = steps < body ? steps : body;
            acc += 4 + 4 * live + (body - live) + 8 * (steps > d ? steps - d : 0);
        }
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        if (lane == 0) cost[q] = acc;
    }
}

cudaError_t k_chunk_cost(const int64_t* row_ptr, const int32_t* order, const int64_t* cs, const int8_t* ch, int mid,
                         int64_t nchunks, int64_t* cost, int grid, cudaStream_t s) {
    if (nchunks <= 0) return cudaSuccess;
    chunk_cost_kernel<<<grid, 256, 0, s>>>(row_ptr, order, cs, ch, mid, nchunks, cost);
    return cudaGetLastError();
}

// A CTA per block: a stable counting sort of the block's rows by home slice.  Rows go through in
// tiles of 1024 in stored order; a row's place is its home's running count, plus the tile's rows
// of that home in earlier warps, plus those in earlier lanes of its warp.
__global__ void __launch_bounds__(1024) order_rows_kernel(const int32_t* __restrict__ home,
                                                          const int64_t* __restrict__ bp, int homes,
                                                          int32_t* __restrict__ order,
                                                          int32_t* __restrict__ home_sorted) {
    extern __shared__ int order_smem[];
    int* next = order_smem;          // [homes] first free place of each home
    int* cnt = order_smem + homes;   // [32][homes] a tile's rows of each home per warp
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int64_t r0 = bp[blockIdx.x], r1 = bp[blockIdx.x + 1];
    for (int h = tid; h < homes; h += 1024) next[h] = 0;
    __syncthreads();
    for (int64_t i = r0 + tid; i < r1; i += 1024) atomicAdd(next + min(max(home[i], 0), homes - 1), 1);
    __syncthreads();
    if (tid == 0) {
        int sum = 0;
        for (int h = 0; h < homes; ++h) {
            const int n = next[h];
            next[h] = sum;
            sum += n;
        }
    }
    for (int64_t t0 = r0; t0 < r1; t0 += 1024) {
        for (int q = tid; q < 32 * homes; q += 1024) cnt[q] = 0;
        __syncthreads();
        const int64_t i = t0 + tid;
        const int h = i < r1 ? min(max(home[i], 0), homes - 1) : -1;
        const unsigned same = __match_any_sync(0xffffffffu, h);
        const int rank = __popc(same & ((1u << lane) - 1u));
        if (h >= 0 && rank == 0) cnt[warp * homes + h] = __popc(same);
        __syncthreads();
        for (int q = tid; q < homes; q += 1024) {
            int at = next[q];
            for (int w = 0; w < 32; ++w) {
                const int n = cnt[w * homes + q];
                cnt[w * homes + q] = at;
                at += n;
            }
            next[q] = at;
        }
        __syncthreads();
        if (h >= 0) {
            const int64_t q = r0 + cnt[warp * homes + h] + rank;
            order[q] = (int32_t)i;
            home_sorted[q] = h;
        }
        __syncthreads();
    }
}

cudaError_t k_order_rows(const int32_t* home, const int64_t* bp, int B, int homes, int32_t* order,
                         int32_t* home_sorted, cudaStream_t s) {
    if (B <= 0) return cudaSuccess;
    order_rows_kernel<<<B, 1024, sizeof(int) * 33 * (size_t)homes, s>>>(home, bp, homes, order, home_sorted);
    return cudaGetLastError();
}

// A warp per chunk of rows [cs[q], cs[q+1]) (at most 64): the lower median (element n/2
// of the sorted values) of the home slices of its non-empty rows, -1 when all are empty.
// Rows i >= 1 whose home and the previous row's home are both defined and differ are
// counted into *changes.
__global__ void chunk_home_kernel(const int32_t* __restrict__ home, const int64_t* __restrict__ cs, int64_t nchunks,
                                  int32_t* __restrict__ out, unsigned long long* changes) {
    const int lane = threadIdx.x & 31;
    const int64_t w0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    unsigned long long ch = 0;
    for (int64_t q = w0; q < nchunks; q += nw) {
        const int64_t i0 = cs[q], i1 = cs[q + 1];
        const int64_t ia = i0 + lane, ib = i0 + 32 + lane;
        const int32_t ha = ia < i1 ? home[ia] : -1;
        const int32_t hb = ib < i1 ? home[ib] : -1;
        if (ia < i1 && ia > 0) { const int32_t p = home[ia - 1]; ch += (ha >= 0 && p >= 0 && ha != p) ? 1 : 0; }
        if (ib < i1) { const int32_t p = home[ib - 1]; ch += (hb >= 0 && p >= 0 && hb != p) ? 1 : 0; }
        const int nv = __popc(__ballot_sync(0xffffffffu, ha >= 0)) + __popc(__ballot_sync(0xffffffffu, hb >= 0));
        if (nv == 0) {
            if (lane == 0) out[q] = -1;
            continue;
        }
        const int k = nv / 2;
        int la = 0, ea = 0, lb = 0, eb = 0;   // defined values below / at most ha and hb
        for (int src = 0; src < 32; ++src) {
            const int32_t wa = __shfl_sync(0xffffffffu, ha, src), wb = __shfl_sync(0xffffffffu, hb, src);
            if (wa >= 0) { la += wa < ha; ea += wa <= ha; lb += wa < hb; eb += wa <= hb; }
            if (wb >= 0) { la += wb < ha; ea += wb <= ha; lb += wb < hb; eb += wb <= hb; }
        }
        const unsigned ma = __ballot_sync(0xffffffffu, ha >= 0 && la <= k && k < ea);
        const unsigned mb = __ballot_sync(0xffffffffu, hb >= 0 && lb <= k && k < eb);
        const int32_t va = __shfl_sync(0xffffffffu, ha, ma ? __ffs(ma) - 1 : 0);
        const int32_t vb = __shfl_sync(0xffffffffu, hb, mb ? __ffs(mb) - 1 : 0);
        if (lane == 0) out[q] = ma ? va : vb;
    }
    for (int o = 16; o > 0; o >>= 1) ch += __shfl_xor_sync(0xffffffffu, ch, o);
    if (lane == 0 && ch) atomicAdd(changes, ch);
}

cudaError_t k_chunk_home(const int32_t* home, const int64_t* chunk_start, int64_t nchunks, int32_t* out,
                         unsigned long long* changes, int grid, cudaStream_t s) {
    if (nchunks <= 0) return cudaSuccess;
    chunk_home_kernel<<<grid, 256, 0, s>>>(home, chunk_start, nchunks, out, changes);
    return cudaGetLastError();
}

}  // namespace ntvs
