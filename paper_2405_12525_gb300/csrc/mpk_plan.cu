// Planner: the permuted, sliced matrix copy, level groups, row chunks, chunk dependency
// ranges and the unit tables of the level-blocked schedule.
#include "mpk_internal.h"

#include <algorithm>
#include <climits>
#include <cstddef>
#include <memory>

namespace mpk {

static int grid_n(int64_t n) {
    int64_t g = (n + 255) / 256;
    const int64_t cap = (int64_t)device_sms() * 16;
    if (g > cap) g = cap;
    return (int)(g < 1 ? 1 : g);
}

// length of new row r = length of old row perm[r]
__global__ void k_rowlen(int32_t n, const int32_t *rp, const int32_t *perm, int32_t *len) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; r < n; r += stride) {
        const int32_t old = perm ? perm[r] : (int32_t)r;
        len[r] = rp[old + 1] - rp[old];
    }
}

__global__ void k_gather_i32(const int32_t *src, const int32_t *idx, int32_t cnt, int32_t *dst) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < cnt; i += stride) dst[i] = src[idx[i]];
}

__global__ void k_chunk_of_row(const int32_t *chunk_row, int32_t nchunks, int32_t *chunk_of_row) {
    for (int32_t c = blockIdx.x; c < nchunks; c += gridDim.x)
        for (int32_t r = chunk_row[c] + threadIdx.x; r < chunk_row[c + 1]; r += blockDim.x) chunk_of_row[r] = c;
}

// longest row of each 32-row slice; one thread per slice
__global__ void k_slice_width(const int32_t *slice_row, int32_t nslices, const int32_t *rowlen, int32_t *width) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t sl = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; sl < nslices; sl += stride) {
        int32_t w = 0;
        for (int32_t r = slice_row[sl]; r < slice_row[sl + 1]; ++r) w = max(w, rowlen[r]);
        width[sl] = w;
    }
}

// Copies every row of P A P^T into its slice (entry j of lane l at slice_ptr + 32 j + l),
// relabelling columns through iperm, and folds the chunks each row reads into the
// dependency range of its chunk.  When A is not known to be symmetric, a chunk is also
// added to the ranges of the chunks it reads, so that ranges cover both directions.
__device__ __forceinline__ int value_special(double) { return 0; }
__device__ __forceinline__ int value_special(float v) { return binary32_special(__float_as_uint(v)); }
__device__ __forceinline__ int value_special(uint16_t v) { return binary32_special((uint32_t)v << 16); }

template <class T>
__global__ void k_fill(int32_t n, const int32_t *rp, const int32_t *ci, const T *va, const int32_t *perm,
                       const int32_t *iperm, const int32_t *chunk_row, const int32_t *chunk_slice,
                       const int32_t *chunk_of_row, const int64_t *slice_ptr, T *sval, int32_t *scol,
                       int2 *dep, int symmetric, int32_t *special) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; r < n; r += stride) {
        const int32_t c = chunk_of_row[r];
        const int32_t local = (int32_t)r - chunk_row[c];
        const int64_t base = slice_ptr[chunk_slice[c] + (local >> 5)] + (local & 31);
        const int32_t old = perm ? perm[r] : (int32_t)r;
        const int32_t e0 = rp[old], e1 = rp[old + 1];
        int32_t lo = c, hi = c;
        for (int32_t e = e0; e < e1; ++e) {
            const int32_t nc = iperm ? iperm[ci[e]] : ci[e];
            const int64_t dst = base + 32 * (int64_t)(e - e0);
            sval[dst] = va[e];
            if (value_special(va[e])) *special = 1;  // narrow types: subnormal, infinity or NaN
            scol[dst] = nc;
            const int32_t cc = chunk_of_row[nc];
            lo = min(lo, cc);
            hi = max(hi, cc);
            if (!symmetric) {
                if (dep[cc].x > c) atomicMin(&dep[cc].x, c);
                if (dep[cc].y < c) atomicMax(&dep[cc].y, c);
            }
        }
        if (dep[c].x > lo) atomicMin(&dep[c].x, lo);
        if (dep[c].y < hi) atomicMax(&dep[c].y, hi);
    }
}

__global__ void k_dep_init(int2 *dep, int32_t nchunks) {
    for (int32_t c = blockIdx.x * blockDim.x + threadIdx.x; c < nchunks; c += gridDim.x * blockDim.x)
        dep[c] = make_int2(c, c);
}

// Exact dependency sets: bit (cc - hull_lo[c]) of chunk c's bitmap is set when a row of c
// reads a row of chunk cc (and, for patterns not known to be symmetric, when a row of cc
// reads a row of c).  Every chunk depends on itself.
__global__ void k_dep_bits(int32_t n, const int32_t *rowlen, const int32_t *chunk_row, const int32_t *chunk_slice,
                           const int32_t *cor, const int64_t *slice_ptr, const int32_t *scol, const int2 *hull,
                           const int64_t *word_off, uint32_t *bits, int symmetric) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; r < n; r += stride) {
        const int32_t c = cor[r];
        const int32_t local = (int32_t)r - chunk_row[c];
        const int64_t base = slice_ptr[chunk_slice[c] + (local >> 5)] + (local & 31);
        const int32_t lo_c = hull[c].x;
        auto set = [&](int32_t owner, int32_t owner_lo, int32_t target) {
            const int32_t off = target - owner_lo;
            // (most rows of a chunk set the same few bits: look before the atomic; 1.9 M rows, this
            // phase 580 -> 217 us)
            uint32_t *w = &bits[word_off[owner] + (off >> 5)];
            if (!((*w >> (off & 31)) & 1u)) atomicOr(w, 1u << (off & 31));
        };
        set(c, lo_c, c);
        int32_t last = -1;
        for (int32_t j = 0; j < rowlen[r]; ++j) {
            const int32_t cc = cor[scol[base + 32 * (int64_t)j]];
            if (cc == last) continue;
            last = cc;
            set(c, lo_c, cc);
            if (!symmetric) set(cc, hull[cc].x, c);
        }
    }
}

// Compresses each chunk's bitmap into at most kDepRanges ranges of chunk indices: maximal
// runs of set bits, then the runs separated by the smallest gaps are merged.  Chunks with
// more than 64 runs fall back to their hull.  Empty ranges are (0, -1).
__global__ void k_dep_ranges(int32_t nchunks, const int2 *hull, const int64_t *word_off, const uint32_t *bits,
                             int4 *ranges) {
    for (int32_t c = blockIdx.x * blockDim.x + threadIdx.x; c < nchunks; c += gridDim.x * blockDim.x) {
        const int32_t lo = hull[c].x, hi = hull[c].y;
        const int64_t w0 = word_off[c];
        const int32_t nb = hi - lo + 1;
        int32_t rs[64], re[64];
        int nr = 0;
        bool overflow = false;
        int32_t run_start = -1;
        for (int32_t b = 0; b < nb && !overflow; ++b) {
            const bool on = (bits[w0 + (b >> 5)] >> (b & 31)) & 1u;
            if (on && run_start < 0) run_start = b;
            if (!on && run_start >= 0) {
                if (nr == 64) overflow = true;
                else { rs[nr] = lo + run_start; re[nr] = lo + b - 1; ++nr; }
                run_start = -1;
            }
        }
        if (!overflow && run_start >= 0) {
            if (nr == 64) overflow = true;
            else { rs[nr] = lo + run_start; re[nr] = hi; ++nr; }
        }
        if (overflow || nr == 0) {
            nr = 1;
            rs[0] = lo;
            re[0] = hi;
        }
        while (nr > kDepRanges) {  // merge the pair of neighbouring runs with the smallest gap
            int best = 0;
            for (int q = 1; q + 1 < nr; ++q)
                if (rs[q + 1] - re[q] < rs[best + 1] - re[best]) best = q;
            re[best] = re[best + 1];
            for (int q = best + 1; q + 1 < nr; ++q) {
                rs[q] = rs[q + 1];
                re[q] = re[q + 1];
            }
            --nr;
        }
        int32_t out[2 * kDepRanges];
        for (int q = 0; q < kDepRanges; ++q) {
            out[2 * q] = q < nr ? rs[q] : 0;
            out[2 * q + 1] = q < nr ? re[q] : -1;
        }
        ranges[2 * c] = make_int4(out[0], out[1], out[2], out[3]);
        ranges[2 * c + 1] = make_int4(out[4], out[5], out[6], out[7]);
    }
}

// Input-row windows of shape 3: for chunk c and its dependency range q, the smallest and the
// largest column (plan numbering) that a row of c reads from the chunks of range q.  The
// ranges are disjoint and cover every chunk that c reads, so the windows are disjoint and
// hold every column of c.  xw[kXWin * c + q] = (min, max), (INT_MAX, -1) when c reads none.
__global__ void k_xwin(int32_t n, const int32_t *rowlen, const int32_t *chunk_row, const int32_t *chunk_slice,
                       const int32_t *cor, const int64_t *slice_ptr, const int32_t *scol, const int4 *ranges,
                       int2 *xw) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; r < n; r += stride) {
        const int32_t c = cor[r];
        const int32_t local = (int32_t)r - chunk_row[c];
        const int64_t base = slice_ptr[chunk_slice[c] + (local >> 5)] + (local & 31);
        const int4 r0 = ranges[2 * c], r1 = ranges[2 * c + 1];
        const int32_t rlo[kXWin] = {r0.x, r0.z, r1.x, r1.z}, rhi[kXWin] = {r0.y, r0.w, r1.y, r1.w};
        int32_t mn[kXWin], mx[kXWin];
        for (int q = 0; q < kXWin; ++q) {
            mn[q] = INT_MAX;
            mx[q] = -1;
        }
        for (int32_t j = 0; j < rowlen[r]; ++j) {
            const int32_t col = scol[base + 32 * (int64_t)j];
            const int32_t cc = cor[col];
            for (int q = 0; q < kXWin; ++q)
                if (cc >= rlo[q] && cc <= rhi[q]) {
                    mn[q] = min(mn[q], col);
                    mx[q] = max(mx[q], col);
                    break;
                }
        }
        for (int q = 0; q < kXWin; ++q)
            if (mx[q] >= 0) {
                atomicMin(&xw[kXWin * c + q].x, mn[q]);
                atomicMax(&xw[kXWin * c + q].y, mx[q]);
            }
    }
}

// 16-bit position of every entry's column in its chunk's window area: the window q holding
// the column (win[3 kXWin c + 3q ..] = first row, rows, position in rows) gives
// position + column - first row.  Padding keeps 0xffff.
__global__ void k_lcol(int32_t n, const int32_t *rowlen, const int32_t *chunk_row, const int32_t *chunk_slice,
                       const int32_t *cor, const int64_t *slice_ptr, const int32_t *scol, const int32_t *win,
                       uint16_t *lcol) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; r < n; r += stride) {
        const int32_t c = cor[r];
        const int32_t local = (int32_t)r - chunk_row[c];
        const int64_t base = slice_ptr[chunk_slice[c] + (local >> 5)] + (local & 31);
        const int32_t *w = win + 3 * kXWin * (int64_t)c;
        for (int32_t j = 0; j < rowlen[r]; ++j) {
            const int32_t col = scol[base + 32 * (int64_t)j];
            for (int q = 0; q < kXWin; ++q)
                if (w[3 * q + 1] > 0 && col >= w[3 * q] && col < w[3 * q] + w[3 * q + 1]) {
                    lcol[base + 32 * (int64_t)j] = (uint16_t)(w[3 * q + 2] + col - w[3 * q]);
                    break;
                }
        }
    }
}

// One record of kRecInts ints per chunk with everything the kernel's control warp needs:
// [row0, row1, slice0, padded entries, first entry (lo, hi 32 bits), staged, slices,
//  kDepRanges (lo, hi) dependency ranges, slice widths as bytes].  A chunk is staged in
// shared memory when its entries fit a buffer and its widths fit the record.
__global__ void k_chunk_records(int32_t nchunks, const int32_t *chunk_row, const int32_t *chunk_slice,
                                const int64_t *slice_ptr, const int4 *ranges, int32_t stage_entries, const int32_t *win,
                                int32_t max_slices, int32_t *rec) {
    for (int32_t c = blockIdx.x * blockDim.x + threadIdx.x; c < nchunks; c += gridDim.x * blockDim.x) {
        const int32_t sl0 = chunk_slice[c], sl1 = chunk_slice[c + 1], nsl = sl1 - sl0;
        const int64_t e0 = slice_ptr[sl0], e1 = slice_ptr[sl1];
        const int32_t cnt = (int32_t)(e1 - e0);
        const int staged = kStageChunks && cnt > 0 && cnt <= stage_entries && nsl <= max_slices;
        int32_t *o = rec + (int64_t)kRecInts * c;
        o[0] = chunk_row[c];
        o[1] = chunk_row[c + 1];
        o[2] = sl0;
        o[3] = cnt;
        o[4] = (int32_t)(e0 & 0xffffffffLL);
        o[5] = (int32_t)(e0 >> 32);
        o[6] = staged;
        o[7] = nsl;
        const int4 r0 = ranges[2 * c], r1 = ranges[2 * c + 1];
        o[8] = r0.x; o[9] = r0.y; o[10] = r0.z; o[11] = r0.w;
        o[12] = r1.x; o[13] = r1.y; o[14] = r1.z; o[15] = r1.w;
        uint32_t wb[kRecSlicesWide / 4] = {0, 0, 0, 0, 0, 0, 0, 0};
        if (staged)
            for (int32_t q = 0; q < nsl; ++q) {
                const uint32_t w = (uint32_t)((slice_ptr[sl0 + q + 1] - slice_ptr[sl0 + q]) >> 5);
                wb[q >> 2] |= (w & 0xffu) << (8 * (q & 3));
            }
        for (int q = 0; q < 3 * kXWin; ++q) o[kRecWin + q] = win ? win[3 * kXWin * (int64_t)c + q] : 0;
        // widths of slices 0..15, then (shapes without windows) of slices 16..31 over the windows
        for (int q = 0; q < (win ? kRecSlices : kRecSlicesWide) / 4; ++q) o[16 + q] = (int32_t)wb[q];
    }
}

// Unit tables from their Lp-diagram cells: cell i (group g, power k) holds the chunks
// [c0, c0 + nc) of g and starts at slot off[i] of the table; its units are (c << 5) | k in
// chunk order.
__global__ void k_expand_cells(const int64_t *off, const int4 *cell, int32_t ncells, int32_t *units) {
    for (int32_t i = blockIdx.x; i < ncells; i += gridDim.x) {
        const int4 c = cell[i];  // (c0, nc, k, unused)
        const int64_t o = off[i];
        for (int32_t j = threadIdx.x; j < c.y; j += blockDim.x) units[o + j] = ((c.x + j) << 5) | c.z;
    }
}

template <class T> __global__ void k_widen(const T *src, int64_t n, double *dst) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += stride) dst[i] = widen_value(src[i]);
}

void widen_values(int vtype, const void *src, int64_t n, double *dst, cudaStream_t s) {
    if (n <= 0) return;
    if (vtype == MPK_F64)
        k_widen<double><<<grid_n(n), 256, 0, s>>>(static_cast<const double *>(src), n, dst);
    else if (vtype == MPK_F32)
        k_widen<float><<<grid_n(n), 256, 0, s>>>(static_cast<const float *>(src), n, dst);
    else if (vtype == MPK_BF16)
        k_widen<uint16_t><<<grid_n(n), 256, 0, s>>>(static_cast<const uint16_t *>(src), n, dst);
    else
        fail(MPK_ERR_UNSUPPORTED, "value type %d", vtype);
    MPK_LAUNCHED();
}

// sliced copy -> CSR (for inspection and tests), values widened to float64
template <class T>
__global__ void k_export(int32_t n, const int32_t *rowlen, const int32_t *chunk_row, const int32_t *chunk_slice,
                         const int32_t *chunk_of_row, const int64_t *slice_ptr, const T *sval,
                         const int32_t *scol, const int32_t *rp, int32_t *ci, double *va) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; r < n; r += stride) {
        const int32_t c = chunk_of_row[r];
        const int32_t local = (int32_t)r - chunk_row[c];
        const int64_t base = slice_ptr[chunk_slice[c] + (local >> 5)] + (local & 31);
        for (int32_t j = 0; j < rowlen[r]; ++j) {
            ci[rp[r] + j] = scol[base + 32 * (int64_t)j];
            va[rp[r] + j] = widen_value(sval[base + 32 * (int64_t)j]);
        }
    }
}

void export_csr(const Plan &P, int32_t *rp, int32_t *ci, double *va, cudaStream_t s) {
    if (!rp || (P.nnz > 0 && (!ci || !va))) fail(MPK_ERR_INVALID, "NULL output array");
    exclusive_scan(P.rowlen, rp, P.n, s);
    if (P.n == 0) return;
    Tmp<int32_t> cor(P.n, s);
    k_chunk_of_row<<<grid_n(P.num_chunks * 256), 256, 0, s>>>(P.chunk_row, P.num_chunks, cor.p);
    MPK_LAUNCHED();
#define EXPORT(T)                                                                                              \
    k_export<T><<<grid_n(P.n), 256, 0, s>>>(P.n, P.rowlen, P.chunk_row, P.chunk_slice, cor.p, P.slice_ptr, \
                                            static_cast<const T *>(P.val), P.col, rp, ci, va)
    if (P.val_type == MPK_F64)
        EXPORT(double);
    else if (P.val_type == MPK_F32)
        EXPORT(float);
    else
        EXPORT(uint16_t);
#undef EXPORT
    MPK_LAUNCHED();
    MPK_CUDA(cudaStreamSynchronize(s));
}

// ----------------------------------------------------------------------------- wave kernel's tables
// width of every slice (its longest row) and, if map is given, its rows sorted by length: blocks of
// kSortSlices slices, longest first, stable, so that the 32 rows of a slice are about equally long
// (the sorting window of SELL-C-sigma: Kreutzer et al., SIAM J. Sci. Comput. 36(5), 2014)
// (longer blocks pad less but spread a slice's gathers: 2 / 4 / 8 / 32 slices, XXZ L = 24 recurrence 15.1 /
// 15.0 / 15.4 / 15.6 ms, banded graph of 300k rows 271 / 249 / 240 / 238 us)
// (slice s holds the rows [slice_row[s], slice_row[s + 1]) of its block's sorted list).  A block never
// crosses a group: first_slice[b] .. first_slice[b + 1] are its slices.
constexpr int kSortSlices = 8;
__global__ void __launch_bounds__(32 * kSortSlices)
    k_sort_rows(const int32_t *rp, const int32_t *perm, const int32_t *slice_row, const int32_t *block_slice,
                int32_t *width, int32_t *map) {
    constexpr int N = 32 * kSortSlices;
    __shared__ uint32_t key[N];
    const int s0 = block_slice[blockIdx.x], s1 = block_slice[blockIdx.x + 1];
    const int r0 = slice_row[s0], rows = slice_row[s1] - r0, t = threadIdx.x;
    int32_t len = 0;
    if (t < rows) {
        const int32_t old = perm ? perm[r0 + t] : r0 + t;
        len = rp[old + 1] - rp[old];
    }
    // ascending keys: longest first, then by row; lengths beyond 2^21 count as equal
    key[t] = t < rows ? (uint32_t)((1 << 21) - min(len, (1 << 21) - 1)) << 10 | (uint32_t)t : 0xffffffffu;
    for (int size = 2; size <= N; size <<= 1)
        for (int d = size >> 1; d > 0; d >>= 1) {
            __syncthreads();
            const int o = t ^ d;
            if (o > t) {
                const uint32_t x = key[t], y = key[o];
                if ((x > y) == ((t & size) == 0)) {
                    key[t] = y;
                    key[o] = x;
                }
            }
        }
    __syncthreads();
    const int row = t < rows ? r0 + (int)(key[t] & (N - 1)) : -1;
    // (slices of a block are full but for the last, so the sorted position is the slice's lane)
    const int s = s0 + (t >> 5);
    if (s >= s1) return;
    map[32 * (int64_t)s + (t & 31)] = row;
    int32_t w = 0;
    if (row >= 0) {
        const int32_t old = perm ? perm[row] : row;
        w = rp[old + 1] - rp[old];
    }
    w = __reduce_max_sync(0xffffffffu, w);
    if ((t & 31) == 0) width[s] = w;
}

// width of every slice of consecutive rows, one warp per slice
__global__ void k_row_width(const int32_t *rp, const int32_t *perm, const int32_t *slice_row, int32_t nslices,
                            int32_t *width) {
    const int lane = threadIdx.x & 31;
    for (int64_t s = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; s < nslices;
         s += (int64_t)gridDim.x * blockDim.x >> 5) {
        const int32_t r = slice_row[s] + lane;
        int32_t w = 0;
        if (r < slice_row[s + 1]) {
            const int32_t old = perm ? perm[r] : r;
            w = rp[old + 1] - rp[old];
        }
        const int32_t m = __reduce_max_sync(0xffffffffu, w);
        if (lane == 0) width[s] = m;
    }
}

__global__ void k_entries_of_width(const int32_t *width, int32_t nslices, int64_t *entries) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < nslices; s += stride)
        entries[s] = 32 * (int64_t)width[s];
}

// the sliced copy, padding included, one warp per slice (coalesced writes)
template <class T>
__global__ void k_fill_slices(int32_t nslices, const int32_t *rp, const int32_t *ci, const T *va, const int32_t *perm,
                              const int32_t *iperm, const int32_t *slice_row, const int32_t *map, const int64_t *sptr,
                              T *sval, int32_t *scol) {
    const int lane = threadIdx.x & 31;
    for (int64_t s = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; s < nslices;
         s += (int64_t)gridDim.x * blockDim.x >> 5) {
        int32_t row = map ? map[32 * s + lane] : slice_row[s] + lane;
        if (!map && row >= slice_row[s + 1]) row = -1;
        int32_t e0 = 0, len = 0;
        if (row >= 0) {
            const int32_t old = perm ? perm[row] : row;
            e0 = rp[old];
            len = rp[old + 1] - e0;
        }
        const int64_t base = sptr[s] + lane;
        const int32_t w = (int32_t)((sptr[s + 1] - sptr[s]) >> 5);
        for (int32_t j = 0; j < w; ++j) {
            const bool on = j < len;
            const int32_t c = on ? ci[e0 + j] : -1;
            scol[base + 32 * (int64_t)j] = on && iperm ? iperm[c] : c;
            sval[base + 32 * (int64_t)j] = on ? va[e0 + j] : T(0);
        }
    }
}

// the slices' records: (first entry / 32, entries a row, first row or row map entry, rows); packed
// copies (width given): (first unit, width and flag, ...)
__global__ void k_slice_records(const int64_t *sptr, const int32_t *width, const int32_t *slice_row, int32_t nslices,
                                int mapped, int4 *rec) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < nslices; s += stride) {
        const int64_t e0 = sptr[s], e1 = sptr[s + 1];
        rec[s] = make_int4(width ? (int32_t)e0 : (int32_t)(e0 >> 5), width ? width[s] : (int32_t)((e1 - e0) >> 5),
                           mapped ? (int32_t)(32 * s) : slice_row[s], slice_row[s + 1] - slice_row[s]);
    }
}

// How the gathers of x spread, from samples of up to 2048 rows (64 slices; of fewer when they hold over
// 64 K entries): `lines` / `looked`, the 128-byte lines that a gather of one entry of a unit's rows touches,
// per row (looked at for one entry in four: comparing lanes takes most of the kernel's time), and `bytes`,
// those of the different 32-byte sectors that a sample's entries read (counted in a bitmap of hashes, by the
// bits left free), of `rows` gathered rows.
struct GatherSpread {
    unsigned long long lines, looked, rows;
    float bytes;  // of all samples
};

// Different values of a matrix, as bit patterns in an open hash table; given up beyond kDictSize.
constexpr int kDictSlots = 4 * kDictSize;
constexpr unsigned long long kNoValue = 0x7ff8a5c3e1f00d01ULL;  // (a NaN; a matrix holding it is given up)
struct Dict {
    unsigned long long key[kDictSlots];
    int32_t index[kDictSlots];  // number of the slot's value
    double value[kDictSize];
    int32_t count, over;     // (read back together with what follows)
    GatherSpread spread[2];  // of A's numbering and of the plan order
};
__device__ __forceinline__ unsigned long long value_bits(double v) { return (unsigned long long)__double_as_longlong(v); }
__device__ __forceinline__ unsigned long long value_bits(float v) { return __float_as_uint(v); }
__device__ __forceinline__ unsigned long long value_bits(uint16_t v) { return v; }
__device__ __forceinline__ int dict_slot(unsigned long long b) { return (int)((b * 0x9e3779b97f4a7c15ULL) >> 54) & (kDictSlots - 1); }
__global__ void k_dict_init(Dict *d) {
    for (int i = threadIdx.x; i < kDictSlots; i += blockDim.x) d->key[i] = kNoValue;
    for (int i = threadIdx.x; i < kDictSize; i += blockDim.x) d->value[i] = 0.0;
    if (threadIdx.x == 0) d->count = d->over = 0;
    if (threadIdx.x < 2) d->spread[threadIdx.x] = GatherSpread{0, 0, 0, 0.0f};
}
template <class T> __global__ void k_dict(int64_t nnz, const T *va, Dict *d) {
    __shared__ unsigned long long seen[kDictSlots];  // the block's own table: most entries end here
    for (int i = threadIdx.x; i < kDictSlots; i += blockDim.x) seen[i] = kNoValue;
    __syncthreads();
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    unsigned long long last = kNoValue;
    int step = 0;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < nnz; e += stride) {
        const unsigned long long b = value_bits(va[e]);
        if ((step++ & 15) == 0 && *(volatile int32_t *)&d->over) return;
        if (b == kNoValue) d->over = 1;
        if (b == last) continue;
        last = b;
        bool known = false;
        for (int s = dict_slot(b), i = 0; i < kDictSlots; ++i, s = (s + 1) & (kDictSlots - 1)) {
            unsigned long long k = *(volatile unsigned long long *)&seen[s];
            if (k == kNoValue) k = atomicCAS(&seen[s], kNoValue, b);
            known = k == b;
            if (known || k == kNoValue) break;
        }
        if (known) continue;
        for (int s = dict_slot(b), i = 0; i < kDictSlots; ++i, s = (s + 1) & (kDictSlots - 1)) {
            if (*(volatile int32_t *)&d->over) return;
            const unsigned long long k = atomicCAS(&d->key[s], kNoValue, b);
            if (k == kNoValue && atomicAdd(&d->count, 1) >= kDictSize) d->over = 1;
            if (k == b || k == kNoValue) break;
        }
    }
}
// numbers the values found (one block); vt: their stored type
__global__ void k_dict_number(Dict *d, int vt) {
    __shared__ int n;
    if (threadIdx.x == 0) n = 0;
    __syncthreads();
    for (int i = threadIdx.x; i < kDictSlots; i += blockDim.x) {
        const unsigned long long b = d->key[i];
        if (b == kNoValue) continue;
        const int q = atomicAdd(&n, 1);
        if (q >= kDictSize) continue;  // given up
        d->index[i] = q;
        d->value[q] = vt == MPK_F64   ? __longlong_as_double((long long)b)
                      : vt == MPK_F32 ? widen_value(__uint_as_float((uint32_t)b))
                                      : widen_value((uint16_t)b);
    }
}

// Where packed slices come from, one warp per slice: visit() calls f(j, place of the value, column or
// -1) for every entry j a row of the slice.
// A's rows, as k_fill_slices takes them
struct CsrRows {
    const int32_t *rp, *ci, *perm, *iperm, *slice_row, *map, *widths;
    __device__ __forceinline__ int width(int64_t s) const { return widths[s] & (kWideSlice - 1); }
    template <class F> __device__ __forceinline__ void visit(int64_t s, int w, int lane, F f) const {
        int32_t row = map ? map[32 * s + lane] : slice_row[s] + lane;
        if (!map && row >= slice_row[s + 1]) row = -1;
        int32_t e0 = 0, len = 0;
        if (row >= 0) {
            const int32_t old = perm ? perm[row] : row;
            e0 = rp[old];
            len = rp[old + 1] - e0;
        }
        for (int j = 0; j < w; ++j) f(j, (int64_t)(e0 + j), j < len ? (iperm ? iperm[ci[e0 + j]] : ci[e0 + j]) : -1);
    }
};
// the plan's sliced copy: coalesced, where A's rows in plan order are gathered (256^3, plan order: planning
// took 10.2 ms from A, 7.1 ms from the copy)
struct PlanRows {
    const int64_t *sptr;
    const int32_t *col;
    __device__ __forceinline__ int width(int64_t s) const { return (int)((sptr[s + 1] - sptr[s]) >> 5); }
    template <class F> __device__ __forceinline__ void visit(int64_t s, int w, int lane, F f) const {
        const int64_t e0 = sptr[s] + lane;
        for (int j = 0; j < w; ++j) f(j, e0 + 32 * j, col[e0 + 32 * j]);
    }
};
// packed slices: widths, marking those whose columns do not fit 16-bit distances, and sizes in units
template <class R> __global__ void k_pack_size(int32_t nslices, R rows, int32_t *width, int64_t *units) {
    const int lane = threadIdx.x & 31;
    for (int64_t s = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; s < nslices;
         s += (int64_t)gridDim.x * blockDim.x >> 5) {
        const int w = rows.width(s);
        bool wide = false;
        rows.visit(s, w, lane, [&](int, int64_t, int32_t c) {
            const int32_t hi = __reduce_max_sync(0xffffffffu, c);
            const int32_t lo = __reduce_min_sync(0xffffffffu, c < 0 ? INT_MAX : c);
            wide = wide || hi - lo >= kNoCol;  // (an entry that no lane has: -1 - INT_MAX)
        });
        __syncwarp();
        if (lane == 0) {
            width[s] = w | (wide ? kWideSlice : 0);
            units[s] = packed_units(w, wide);
        }
    }
}
template <class R, class T>
__global__ void k_pack_fill(int32_t nslices, R rows, const T *va, const int32_t *width, const int64_t *units,
                            const Dict *d, uint8_t *stream) {
    const int lane = threadIdx.x & 31;
    unsigned long long last = kNoValue;
    int last_q = 0;
    for (int64_t s = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; s < nslices;
         s += (int64_t)gridDim.x * blockDim.x >> 5) {
        const int w = width[s] & (kWideSlice - 1);
        const bool wide = (width[s] & kWideSlice) != 0;
        uint8_t *p = stream + 16 * units[s];
        int32_t *first = reinterpret_cast<int32_t *>(p);
        uint8_t *cols = p + 16 * ((w + 3) / 4), *vals = cols + (wide ? 128 : 64) * (int64_t)w;
        rows.visit(s, w, lane, [&](int j, int64_t e, int32_t c) {
            const int32_t lo = __reduce_min_sync(0xffffffffu, c < 0 ? INT_MAX : c);
            if (lane == 0) first[j] = lo;
            if (wide)
                reinterpret_cast<int32_t *>(cols)[32 * j + lane] = c;
            else
                reinterpret_cast<uint16_t *>(cols)[32 * j + lane] = (uint16_t)(c < 0 ? kNoCol : c - lo);
            int q = 0;
            if (c >= 0) {
                const unsigned long long b = value_bits(va[e]);
                if (b != last) {
                    int t = dict_slot(b);
                    for (int i = 0; i < kDictSlots && d->key[t] != b; ++i) t = (t + 1) & (kDictSlots - 1);
                    last = b;
                    last_q = d->index[t];
                }
                q = last_q;
            }
            vals[32 * (int64_t)j + lane] = (uint8_t)q;
        });
    }
}

constexpr int kSpreadSlices = 64, kSpreadEntries = 1 << 16, kSpreadSamples = 64, kSpreadBits = 1 << 18;
// rows of A (32 consecutive ones a slice)
struct CsrSlices {
    const int32_t *rp, *ci;
    int32_t n;
    // calls f with the number (mod 4) and the columns of the slice's first entries (-1: a row has fewer),
    // four at a time
    template <class F> __device__ __forceinline__ void visit(int64_t s, int most, int lane, F f) const {
        const int64_t r = 32 * s + lane;
        const int32_t e0 = r < n ? rp[r] : 0, len = r < n ? rp[r + 1] - e0 : 0;
        const int w = min(__reduce_max_sync(0xffffffffu, len), most);
        for (int j = 0; j < w; j += 4) {
            int32_t c[4];
#pragma unroll
            for (int t = 0; t < 4; ++t) c[t] = j + t < len ? ci[e0 + j + t] : -1;
#pragma unroll
            for (int t = 0; t < 4; ++t) f(t, c[t]);
        }
    }
};
// slices of the plan's copy
struct PlanSlices {
    const int64_t *sptr;
    const int32_t *col;
    template <class F> __device__ __forceinline__ void visit(int64_t s, int most, int lane, F f) const {
        const int64_t e0 = sptr[s];
        const int w = min((int)((sptr[s + 1] - e0) >> 5), most);
        for (int j = 0; j < w; j += 4) {
            int32_t c[4];
#pragma unroll
            for (int t = 0; t < 4; ++t) c[t] = j + t < w ? col[e0 + 32 * (int64_t)(j + t) + lane] : -1;
#pragma unroll
            for (int t = 0; t < 4; ++t) f(t, c[t]);
        }
    }
};
// Sample `block` of `blocks`, of `per` slices; xbytes: of a row of x (all its columns); seen: the bitmap, in
// shared memory
template <class R>
__device__ __forceinline__ void spread_sample(int64_t nslices, int per, const R &rows, int m, int xbytes, int block, int blocks,
                                              uint32_t *seen, GatherSpread *out) {
    __shared__ int s_lines, s_looked, s_rows, s_set;
    for (int i = threadIdx.x; i < kSpreadBits / 32; i += blockDim.x) seen[i] = 0;
    if (threadIdx.x == 0) s_lines = s_looked = s_rows = s_set = 0;
    __syncthreads();
    const int lane = threadIdx.x & 31, sector = max(32, xbytes), shift = 31 - __clz(sector);  // (a power of two)
    const int64_t s0 = blocks > 1 ? (nslices - per) * block / (blocks - 1) : 0;
    int lines = 0, looked = 0, taken = 0;
    for (int q = threadIdx.x >> 5; q < per && s0 + q < nslices; q += blockDim.x >> 5) {
        rows.visit(s0 + q, kSpreadEntries / 32, lane, [&](int t, int32_t c) {
            const unsigned int on = __ballot_sync(0xffffffffu, c >= 0);
            const bool look = t == ((q ^ (q >> 5)) & 3);  // (every entry of the rows in some slice)
            const unsigned long long at = (unsigned long long)max(c, 0) * xbytes;
            bool first = false;
            if (look && c >= 0)  // (a unit: 32 / m rows)
                first = lane == __ffs(__match_any_sync(on, (uint32_t)(at >> 7) << 5 | (unsigned)(lane * m >> 5))) - 1;
            if (c >= 0) {
                const uint32_t h = ((uint32_t)(at >> shift) * 0x9e3779b1u) >> 14;  // (18 bits: kSpreadBits)
                if (!((*(volatile uint32_t *)&seen[h >> 5] >> (h & 31)) & 1u)) atomicOr(&seen[h >> 5], 1u << (h & 31));
            }
            if (look) {
                lines += __popc(__ballot_sync(0xffffffffu, first));
                looked += __popc(on);
            }
            taken += __popc(on);
        });
    }
    if (lane == 0) {
        atomicAdd(&s_lines, lines);
        atomicAdd(&s_looked, looked);
        atomicAdd(&s_rows, taken);
    }
    __syncthreads();
    int set = 0;
    for (int i = threadIdx.x; i < kSpreadBits / 32; i += blockDim.x) set += __popc(seen[i]);
    set = __reduce_add_sync(0xffffffffu, set);
    if (lane == 0) atomicAdd(&s_set, set);
    __syncthreads();
    if (threadIdx.x == 0) {
        atomicAdd(&out->lines, (unsigned long long)s_lines);
        atomicAdd(&out->looked, (unsigned long long)s_looked);
        atomicAdd(&out->rows, (unsigned long long)s_rows);
        const float clear = fmaxf(1.0f, (float)(kSpreadBits - s_set)) / kSpreadBits;  // linear counting
        atomicAdd(&out->bytes, -logf(clear) * (float)kSpreadBits * (float)sector);
    }
}
// samples in A's numbering into out[0], then of the plan's slices into out[1]
__global__ void __launch_bounds__(1024) k_gather_spread(int nat_samples, int64_t nat_slices, CsrSlices nat, int64_t nslices,
                                                        PlanSlices plan, int per, int m, int xbytes, GatherSpread *out) {
    __shared__ uint32_t seen[kSpreadBits / 32];
    if ((int)blockIdx.x < nat_samples)
        spread_sample(nat_slices, per, nat, m, xbytes, blockIdx.x, nat_samples, seen, out);
    else
        spread_sample(nslices, per, plan, m, xbytes, blockIdx.x - nat_samples, gridDim.x - nat_samples, seen, out + 1);
}

// The spread of an order, per row and sample: lines a row, bytes of a sample, and those as a part of the
// bytes that its entries gather.
struct Spread {
    double lines = 0.0, bytes = 0.0, fresh = 0.0;
    // Whether the wave kernel takes its smaller buffer (its figures beside kWaveBytes): gathers that touch
    // about a line a row, and read more than the L1 beside the large one holds, much of it for the first
    // time.  Measured over grids, stencils, the spin chain and banded graphs, in order, permuted and shuffled
    // in windows, 1 to 4 columns, p = 8, time at 200 KB over that at 96 KB: lines up to 0.6 a row: 0.59 to
    // 1.0 (spin chain 0.25 lines: 0.58 to 0.74); above, up to 47 KB: 0.7 to 0.95 (banded graph of 100k rows, 31
    // KB; a permuted grid of 1400^2, 41 KB: 1.57); above, little of it fresh: 0.8 to 1.04 (the same, 2 columns, 62
    // KB, 0.13; of 300k rows, 60 KB, 0.25: 0.92); the rest 1.0 to 2.9, but for 63^3 in windows of 1000 rows (69 KB,
    // 0.6): 0.92.  binary64 values with 4 columns need the lead more: banded graphs (0.23 to 0.54) 0.96, permuted
    // grids (above) 1.06 to 1.2.
    bool lead = false;
    bool scattered() const {
        return lines > 0.62 && bytes > 47e3 && (lead ? fresh > 0.56 : fresh > 0.3 || (fresh > 0.22 && bytes > 96e3));
    }
};
// A run of groups whose powers are computed together: a whole plan, or an instance of a batch plan
struct WaveRange {
    int32_t g0, g1;  // groups
    int32_t p;       // powers (batch plans; a single plan has a table for every p)
    int64_t bytes;   // matrix and vectors
};

// Tables of the wave kernel over the slices of `srow` (first rows, and the end), whose groups start
// at the slices vs: cells, records of the slices, slices of the groups, counters (zero), in one block of
// device memory.  False, and nothing done, when there are too many cells or they do not fit the
// memory budget.
// A batch plan's instances are taken in bundles that fit L2 together: inside a bundle the lines of all
// instances alternate, so that one instance's cells fill the hand-over of another's powers.
static bool wave_tables(Plan &P, WaveSet &w, const std::vector<int32_t> &vs, const std::vector<WaveRange> &ranges,
                        const int64_t *sptr, const int32_t *d_width, const int32_t *d_srow, int32_t NS,
                        std::vector<int32_t> &host, int64_t extra,
                        cudaStream_t s) {
    const int32_t VG = (int32_t)vs.size() - 1, pmax = P.p_max;
    const bool batch = !P.inst_p.empty();
    if ((int64_t)VG * pmax >= kWaveMaxCells || (int64_t)VG * pmax * (pmax + 1) / 2 > (1 << 22)) return false;
    std::vector<int32_t> vc;  // 4 per cell
    w.cell_off.assign((size_t)pmax + 2, 0);
    for (int32_t p = batch ? pmax : 1; p <= pmax; ++p) {
        w.cell_off[p] = (int32_t)(vc.size() / 4);
        for (size_t i = 0; i < ranges.size();) {
            size_t e = i;
            int64_t bytes = 0;
            int32_t dmax = 0;
            for (; e < ranges.size() && (e == i || bytes + ranges[e].bytes <= device_l2_bytes() / 4 * 3); ++e) {
                bytes += ranges[e].bytes;
                dmax = std::max(dmax, ranges[e].g1 - ranges[e].g0 - 1 + kSlotSkew * (batch ? ranges[e].p : p));
            }
            for (int32_t d = kSlotSkew; d <= dmax; ++d)  // lines g + kSlotSkew * k ascending
                for (size_t r = i; r < e; ++r) {
                    const WaveRange &R = ranges[r];
                    for (int32_t k = 1; k <= (batch ? R.p : p); ++k) {  // k ascending inside a line
                        const int32_t g = R.g0 + d - kSlotSkew * k;
                        if (g < R.g0 || g >= R.g1) continue;
                        vc.push_back(vs[g]);
                        vc.push_back(vs[g + 1] - vs[g]);
                        vc.push_back((g << 5) | k);
                        vc.push_back((int32_t)r << 2 | (g > R.g0 ? 1 : 0) | (g + 1 < R.g1 ? 2 : 0));
                    }
                }
            i = e;
        }
    }
    const int64_t ncell = (int64_t)vc.size() / 4, ncount = (int64_t)(pmax + 1) * VG;
    w.cell_off[pmax + 1] = (int32_t)ncell;
    const int64_t words = 4 * ncell + 4 * (int64_t)NS + VG + ncount;
    if (P.arena.budget > 0 && P.arena.bytes + 4 * words + extra > P.arena.budget) return false;
    w.maxsl = 0;
    for (int32_t g = 0; g < VG; ++g) {
        vc.push_back(vs[g + 1] - vs[g]);
        w.maxsl = std::max(w.maxsl, vs[g + 1] - vs[g]);
    }
    host.swap(vc);  // the caller keeps it until the copies are done
    w.ngroups = VG;
    int32_t *dev = P.arena.alloc_n<int32_t>(words);
    w.cell = reinterpret_cast<int4 *>(dev);
    w.slice = w.cell + ncell;
    w.gsl = dev + 4 * (ncell + NS);
    w.count = w.gsl + VG;
    MPK_CUDA(cudaMemcpyAsync(w.cell, host.data(), sizeof(int4) * (size_t)ncell, cudaMemcpyHostToDevice, s));
    MPK_CUDA(cudaMemcpyAsync(w.gsl, host.data() + 4 * ncell, sizeof(int32_t) * (size_t)VG, cudaMemcpyHostToDevice, s));
    MPK_CUDA(cudaMemsetAsync(w.count, 0, sizeof(int32_t) * (size_t)ncount, s));
    k_slice_records<<<grid_n(NS), 256, 0, s>>>(sptr, d_width, d_srow, NS, w.rowmap != nullptr, w.slice);
    MPK_LAUNCHED();
    return true;
}

// What the choice of copies and buffers rests on, with one wait for the device: the spread of the gathers in
// A's numbering (at[0], if `natural`) and in plan order (at[1]), if `spread`; and, if `values`, the table of
// A's values in d, false if there are more than kDictSize (a matrix of random values is given up after its
// first entries).  The set-up takes as long with packed copies as without: what the table costs, the smaller
// copy saves (131 x 127 x 113: 5.29 against 5.35 ms).
static bool look_over(const Plan &P, const mpk_csr *A, bool spread, bool natural, Spread (&at)[2], bool values, Dict *d,
                      cudaStream_t s) {
    k_dict_init<<<1, 1024, 0, s>>>(d);
    MPK_LAUNCHED();
    const int per = (int)std::max<int64_t>(1, std::min<int64_t>(kSpreadSlices, kSpreadEntries / (32 * (P.nnz / P.n + 1))));
    const int xbytes = (P.accum == MPK_F32 ? 4 : 8) * P.m;
    auto samples = [&](int64_t nslices) { return (int)std::max<int64_t>(1, std::min<int64_t>(kSpreadSamples, nslices / per)); };
    const int64_t ns = ((int64_t)P.n + 31) / 32;
    const int nat = natural ? samples(ns) : 0, plan = samples(P.num_slices);
    if (spread) {
        k_gather_spread<<<nat + plan, 1024, 0, s>>>(nat, ns, CsrSlices{A->row_ptr, A->col, P.n}, P.num_slices,
                                                    PlanSlices{P.slice_ptr, P.col}, per, P.m, xbytes, d->spread);
        MPK_LAUNCHED();
    }
    if (values) {
        if (P.val_type == MPK_F64)
            k_dict<<<grid_n(A->nnz), 256, 0, s>>>(A->nnz, static_cast<const double *>(A->val), d);
        else if (P.val_type == MPK_F32)
            k_dict<<<grid_n(A->nnz), 256, 0, s>>>(A->nnz, static_cast<const float *>(A->val), d);
        else
            k_dict<<<grid_n(A->nnz), 256, 0, s>>>(A->nnz, static_cast<const uint16_t *>(A->val), d);
        MPK_LAUNCHED();
        k_dict_number<<<1, 1024, 0, s>>>(d, P.val_type);
        MPK_LAUNCHED();
    }
    struct {
        int32_t count, over;
        GatherSpread spread[2];
    } h;
    static_assert(sizeof(h) == sizeof(Dict) - offsetof(Dict, count), "the end of the table");
    MPK_CUDA(cudaMemcpyAsync(&h, &d->count, sizeof(h), cudaMemcpyDeviceToHost, s));
    MPK_CUDA(cudaStreamSynchronize(s));
    for (int q = 0; q < 2; ++q) {
        const double rows = (double)std::max<unsigned long long>(h.spread[q].rows, 1);
        at[q].lines = (double)h.spread[q].lines / (double)std::max<unsigned long long>(h.spread[q].looked, 1);
        at[q].bytes = (double)h.spread[q].bytes / std::max(1, q ? plan : nat);
        at[q].fresh = (double)h.spread[q].bytes / (rows * xbytes);
        at[q].lead = P.val_bytes == 8 && P.m == 4;
    }
    return values && !h.over && h.count <= kDictSize;
}

// The packed copy of the slices `rows` (values at `val`); width and units: scratch of a word a slice.
template <class R>
static bool pack_slices(Plan &P, WaveSet &w, const R &rows, const void *val, const std::vector<int32_t> &vs,
                        const std::vector<WaveRange> &ranges, const Dict *dict, const int32_t *d_srow, int32_t NS,
                        Tmp<int32_t> &width, Tmp<int64_t> &units, std::vector<int32_t> &host, cudaStream_t s) {
    const int grid = grid_n(32 * (int64_t)NS);
    k_pack_size<<<grid, 256, 0, s>>>(NS, rows, width.p, units.p);
    MPK_LAUNCHED();
    exclusive_scan(units.p, units.p, NS, s);
    int64_t total = 0;
    MPK_CUDA(cudaMemcpyAsync(&total, units.p + NS, sizeof(total), cudaMemcpyDeviceToHost, s));
    MPK_CUDA(cudaStreamSynchronize(s));
    if (total >= INT32_MAX) return false;
    const int64_t bytes = 16 * total + (int64_t)sizeof(dict->value);
    if (!wave_tables(P, w, vs, ranges, units.p, width.p, d_srow, NS, host, bytes, s)) return false;
    uint8_t *dev = static_cast<uint8_t *>(P.arena.alloc(bytes));  // the table, then the stream
    uint8_t *stream = dev + sizeof(dict->value);
    MPK_CUDA(cudaMemcpyAsync(dev, dict->value, sizeof(dict->value), cudaMemcpyDeviceToDevice, s));
    if (P.val_type == MPK_F64)
        k_pack_fill<<<grid, 256, 0, s>>>(NS, rows, static_cast<const double *>(val), width.p, units.p, dict, stream);
    else if (P.val_type == MPK_F32)
        k_pack_fill<<<grid, 256, 0, s>>>(NS, rows, static_cast<const float *>(val), width.p, units.p, dict, stream);
    else
        k_pack_fill<<<grid, 256, 0, s>>>(NS, rows, static_cast<const uint16_t *>(val), width.p, units.p, dict, stream);
    MPK_LAUNCHED();
    w.val = stream;
    w.dict = reinterpret_cast<const double *>(dev);
    w.ok = true;
    return true;
}

// A sliced copy of its own for the wave kernel: the rows in A's numbering (perm NULL) or in plan
// order, groups of the rows g_row, sorted by length inside blocks of kSortSlices slices when the
// padding of unsorted slices is over 4 % of the entries (sorted anyway, 256^3, p = 8, plan order,
// packed: 1850 -> 2134 us: rows that were neighbours no longer share their loads and stores of
// vectors).  With the table of A's values (dict) the slices are packed.  False when it does not fit.
static bool wave_copy(Plan &P, WaveSet &w, const mpk_csr *A, const int32_t *perm, const int32_t *iperm,
                      const std::vector<int32_t> &g_row, const std::vector<WaveRange> &ranges, const Dict *dict,
                      std::vector<int32_t> &host, cudaStream_t s) {
    const int32_t VG = (int32_t)g_row.size() - 1;
    std::vector<int32_t> vs(1, 0), srow, blocks;
    for (int32_t g = 0; g < VG; ++g) {
        const int32_t s0 = (int32_t)srow.size();
        for (int32_t r = g_row[g]; r < g_row[g + 1]; r += 32) srow.push_back(r);
        for (int32_t b = s0; b < (int32_t)srow.size(); b += kSortSlices) blocks.push_back(b);
        vs.push_back((int32_t)srow.size());
    }
    const int32_t NS = (int32_t)srow.size();
    srow.push_back(g_row[VG]);
    blocks.push_back(NS);
    Tmp<int32_t> d_srow((int64_t)NS + 1, s), d_width(NS, s), d_block((int64_t)blocks.size(), s);
    Tmp<int64_t> d_ent((int64_t)NS + 1, s);
    MPK_CUDA(cudaMemcpyAsync(d_srow.p, srow.data(), sizeof(int32_t) * srow.size(), cudaMemcpyHostToDevice, s));
    int32_t *map = nullptr;
    auto total = [&]() {
        k_entries_of_width<<<grid_n(NS), 256, 0, s>>>(d_width.p, NS, d_ent.p);
        MPK_LAUNCHED();
        exclusive_scan(d_ent.p, d_ent.p, NS, s);
        int64_t h = 0;
        MPK_CUDA(cudaMemcpyAsync(&h, d_ent.p + NS, sizeof(h), cudaMemcpyDeviceToHost, s));
        MPK_CUDA(cudaStreamSynchronize(s));
        return h;
    };
    k_row_width<<<grid_n(32 * (int64_t)NS), 256, 0, s>>>(A->row_ptr, perm, d_srow.p, NS, d_width.p);
    MPK_LAUNCHED();
    int64_t entries = total();
    if (entries > A->nnz + A->nnz / 25) {
        MPK_CUDA(cudaMemcpyAsync(d_block.p, blocks.data(), sizeof(int32_t) * blocks.size(), cudaMemcpyHostToDevice, s));
        const int64_t bytes = 4 * 32 * (int64_t)NS;
        if (P.arena.budget > 0 && P.arena.bytes + bytes > P.arena.budget) return false;
        map = P.arena.alloc_n<int32_t>(32 * (int64_t)NS);
        k_sort_rows<<<(int)blocks.size() - 1, 32 * kSortSlices, 0, s>>>(A->row_ptr, perm, d_srow.p, d_block.p, d_width.p,
                                                                       map);
        MPK_LAUNCHED();
        entries = total();
    }
    if (entries / 32 >= INT32_MAX) return false;
    w.rowmap = map;
    if (dict)
        return pack_slices(P, w, CsrRows{A->row_ptr, A->col, perm, iperm, d_srow.p, map, d_width.p}, A->val, vs, ranges, dict,
                           d_srow.p, NS, d_width, d_ent, host, s);
    const int64_t bytes = (P.val_bytes + 4) * (entries + 32);
    if (!wave_tables(P, w, vs, ranges, d_ent.p, nullptr, d_srow.p, NS, host, bytes, s)) return false;
    int32_t *col = static_cast<int32_t *>(P.arena.alloc((entries + 32) * (4 + P.val_bytes)));  // columns, then values
    void *val = col + (entries + 32);
#define FILL(T)                                                                                                \
    k_fill_slices<T><<<grid_n(32 * (int64_t)NS), 256, 0, s>>>(NS, A->row_ptr, A->col, static_cast<const T *>(A->val), \
                                                              perm, iperm, d_srow.p, map, d_ent.p, static_cast<T *>(val), col)
    if (P.val_type == MPK_F64)
        FILL(double);
    else if (P.val_type == MPK_F32)
        FILL(float);
    else
        FILL(uint16_t);
#undef FILL
    MPK_LAUNCHED();
    w.val = val;
    w.col = col;
    w.ok = true;
    return true;
}

// Runs make(), which builds a set that the plan can do without: when it returns false, or device
// memory runs out, what it allocated is freed and the set stays empty.
template <class F> static bool spare(Plan &P, WaveSet &w, F make) {
    const size_t mark = P.arena.ptrs.size();
    bool made = false;
    try {
        made = make();
    } catch (const Fail &f) {
        if (f.status != MPK_ERR_OOM && f.status != MPK_ERR_BUDGET) throw;
        cudaGetLastError();
    }
    if (!made) {
        while (P.arena.ptrs.size() > mark) P.arena.free(P.arena.ptrs.back());
        w = WaveSet();
    }
    return made;
}

// The wave kernel's sets of a plan.
// Plan order: a matrix within the cache budget beside four of its vectors is one group (each power is
// one cell); others take runs of the plan's groups.  The plan goes without (and runs k_mpk) when a
// chunk reads rows outside its own group and the two beside it, which the kernel's dependency rule
// does not cover (levels of another matrix).  It works on the plan's own sliced copy, or, when that
// has over 4 % of padding and A's numbering is not taken, on one with its rows sorted by length.
// A's own numbering (plans of original order): no gather before and no scatter after the kernel.
// Groups are runs of at least `band` rows (the largest |column - row|), so that a row reads its own
// group and the two beside it.  Taken when the rows of x that a sweep reads around a row fit a
// quarter of L2 (a wider band is better served by the plan's level order), unless its gathers are
// scattered where the levels' are not.
static void plan_wave(Plan &P, const mpk_csr *A, int32_t band, const std::vector<int32_t> &g_row,
                      const std::vector<int32_t> &g_slice, const std::vector<int32_t> &c_slice,
                      const std::vector<int64_t> &sptr, const std::vector<int32_t> &s_row, const std::vector<int2> &hull,
                      const int32_t *d_srow, bool default_budget, std::vector<int32_t> (&host)[2], cudaStream_t s) {
    const int32_t G = P.num_groups, NS = P.num_slices, n = P.n;
    if (P.padded / 32 >= INT32_MAX) return;
    // the kernel's cells pay for a larger budget than k_mpk's, since a block's share of a cell is what
    // hides the cell's hand-over to the next power (256^3, p = 8: 97 / 130 / 160 / 200 MB took 2.18 /
    // 2.09 / 2.09 / 2.14 ms; binary32 sums 100 / 130 / 160 / 200 MB 1.40 / 1.34 / 1.36 / 1.40 ms: one rule for both)
    const int64_t wave_cache = default_budget ? device_l2_bytes() / 4 * 5 : P.cache_bytes;
    const bool batch = !P.inst_p.empty();
    const int64_t row_bytes = 4 + 16 * (int64_t)P.m, vec_bytes = 32 * (int64_t)P.m;
    // the instances: rows, plan groups, the budget of a group, and whether one group holds it all
    struct Inst {
        int32_t r0, r1, g0, g1, p;
        int64_t most, bytes;
        bool one;
    };
    std::vector<Inst> in;
    const size_t ni = batch ? P.inst_p.size() : 1;
    if (ni > kWaveInst) return;
    bool one = true;  // every instance is one group
    for (size_t i = 0; i < ni; ++i) {
        Inst t;
        t.r0 = batch ? P.inst_row[i] : 0;
        t.r1 = batch ? P.inst_row[i + 1] : n;
        t.p = batch ? P.inst_p[i] : P.p_max;
        t.g0 = (int32_t)(std::lower_bound(g_row.begin(), g_row.end() - 1, t.r0) - g_row.begin());
        t.g1 = t.r1 == n ? G : (int32_t)(std::lower_bound(g_row.begin(), g_row.end() - 1, t.r1) - g_row.begin());
        if (t.r1 == t.r0) t.g1 = t.g0;
        const int64_t entries = sptr[g_slice[t.g1]] - sptr[g_slice[t.g0]];
        t.bytes = (P.val_bytes + 4) * entries + vec_bytes * (t.r1 - t.r0);
        t.one = P.identity || t.bytes <= P.cache_bytes;
        t.most = wave_cache / (kSlotSkew * t.p + 1);
        one = one && t.one;
        in.push_back(t);
    }
    // A matrix larger than the cache that has few different values gets packed copies (about 3.2 bytes an
    // entry in place of 12): the copies into shared memory, not HBM, are what they save, so they also help
    // at p = 1.  Measured before the rounding of groups below, us, plain -> packed copies, 256^3 7-point / 150^3 27-point, p = 8:
    //   binary64, A's order:              2215 -> 1966 / 1907 -> 1348;  plan order: 2035 -> 1850 / 1912 -> 1306
    //   binary32, plan order:             1807 -> 1852 / 1477 -> 1306
    //   bfloat16, binary32 sums, A's order: 1470 -> 1524 / 825 -> 715
    //   bfloat16, binary64 sums, A's order: 1974 -> 1968 / 1300 -> 1348
    // and more columns (bfloat16 27-point 100^3, 8 columns: 3054 -> 3277) use an entry too often for
    // its unpacking.
    const bool long_rows = P.nnz / std::max(n, 1) >= 16;
    const bool pack = !batch && !one && P.m == 1 &&
                      (P.val_type == MPK_F64 || (long_rows && (P.val_type == MPK_F32 || P.accum == MPK_F32)));
    bool natural = !P.identity && P.order == MPK_ORDER_ORIGINAL &&
                   std::min<int64_t>(n, 2 * (int64_t)band + 32) * 8 * P.m <= device_l2_bytes() / 4;
    // (not looked at where the large buffer is as good: 8 and 16 columns within 3 %, up to 32768 rows of
    // one column the same)
    const bool look = P.m <= 4 && (int64_t)n * P.m > 32768;
    Spread spread[2];
    std::unique_ptr<Tmp<Dict>> table;
    bool packed = false;
    if (look || pack) try {
            table.reset(new Tmp<Dict>(1, s));
            packed = look_over(P, A, look, natural, spread, pack, table->p, s);
        } catch (const Fail &f) {  // no memory for the table: the plan does without
            if (f.status != MPK_ERR_OOM) throw;
            cudaGetLastError();
        }
    const Dict *dict = packed ? table->p : nullptr;
    // A numbering whose gathers are scattered where the levels' are not is left to the plan order: one
    // column, more rows than the gather and scatter of the vectors make up for.  Time of k_mpk, as it was
    // before this kernel, over A's numbering / plan order (96 KB buffers), apply p = 8 and a recurrence of
    // 32 steps, 7-point grids: 126^3 permuted, bfloat16 1.05 0.89 / 1.01 1.02, shuffled in windows of 10 000
    // rows, binary64 1.01 0.98 / 1.14 1.10, binary32 0.82 0.81 / 1.09 1.02, of 100 000 rows, bfloat16 and binary32
    // sums 0.69 0.75 / 1.01 0.93; 63^3 (0.25 M rows) permuted 1.72 1.38 / 1.48 1.55, kept.  Banded graphs, whose
    // gathers spread alike in both, are better off in A's numbering at every size (1M rows, binary32: 1.00
    // 1.04 / 0.96 1.03), two columns of anything too (126^3 permuted: 1.52 1.15 / 1.29 1.22).
    if (!batch && P.m == 1 && n > 1 << 18 && spread[0].lines > 0.5 && spread[0].bytes > 1.4 * spread[1].bytes) natural = false;
    const double packed_entry = 3.2, entry_bytes = packed ? packed_entry : P.val_bytes + 4;
    if (natural) {
        std::vector<int32_t> nrow;
        std::vector<WaveRange> nranges;
        for (const Inst &t : in) {
            WaveRange r{(int32_t)nrow.size(), 0, t.p, t.bytes};
            int64_t rows = t.r1 - t.r0;
            if (!t.one) {
                // A default budget of 5/4 of L2 where that is a good part of the matrix and its vectors, 3/5 of
                // L2 beyond 3 times L2, where its window no longer stays in L2 (p = 8, us, 5/4 / 3/5 of L2;
                // packed 7-point: 131^3 258 / 269, 200^3 872 / 876, 230^3 1384 / 1318, 256^3 1946 / 1794, 290^3
                // 3007 / 2801; 256^3 bfloat16, binary32 sums: 1457 / 1346; packed 5-point: 2000^2 376 / 382,
                // 4000 x 4100 1513 / 1489)
                const double a_row = entry_bytes * (double)(P.nnz / std::max(n, 1) + 1) + (double)row_bytes;
                const bool large = default_budget && a_row * (double)rows > 3.0 * (double)device_l2_bytes();
                const int64_t most = large ? device_l2_bytes() / 5 * 3 / (kSlotSkew * t.p + 1) : t.most;
                rows = std::max<int64_t>(band, (int64_t)((double)most / a_row));
                // equal shares for the blocks where a group has a few slices for each (27-point stencil on
                // 150^3, p = 8, packed: 1349 -> 1261 us; below, a whole slice more for each would be too much)
                const int64_t even = 32 * (int64_t)device_sms();
                rows = rows >= 2 * even ? (rows + even - 1) / even * even : std::max<int64_t>(32, (rows + 31) / 32 * 32);
            }
            for (int64_t q = t.r0; q < t.r1; q += rows) nrow.push_back((int32_t)q);
            r.g1 = (int32_t)nrow.size();
            nranges.push_back(r);
        }
        nrow.push_back(n);
        natural = spare(P, P.natural, [&]() { return wave_copy(P, P.natural, A, nullptr, nullptr, nrow, nranges, dict, host[1], s); });
        P.natural.scattered = spread[0].scattered();
    }
    // What runs in plan order beside A's numbering (X inside Y, the resumable recurrence, a batch without
    // every output) has the plan's own copy, not one more.
    const Dict *plan_dict = natural ? nullptr : dict;
    const double plan_entry = plan_dict ? packed_entry : P.val_bytes + 4;
    std::vector<int32_t> vs;  // first slice of every group, and the end
    std::vector<WaveRange> ranges;
    for (const Inst &t : in) {
        WaveRange r{(int32_t)vs.size(), 0, t.p, t.bytes};
        int64_t bytes = 0;
        for (int32_t g = t.g0; g < t.g1; ++g) {
            const int64_t b = (int64_t)(plan_entry * (double)(sptr[g_slice[g + 1]] - sptr[g_slice[g]])) +
                              row_bytes * (g_row[g + 1] - g_row[g]);
            if (g == t.g0 || (!t.one && bytes + b > t.most)) {
                vs.push_back(g_slice[g]);
                bytes = 0;
            }
            bytes += b;
        }
        r.g1 = (int32_t)vs.size();
        ranges.push_back(r);  // (an empty instance has no groups)
    }
    vs.push_back(NS);
    const int32_t VG = (int32_t)vs.size() - 1;
    bool near = one || (int32_t)hull.size() == P.num_chunks;
    if (!one && near) {  // (chunk c starts at slice c_slice[c], ascending)
        std::vector<int32_t> vc0((size_t)VG + 1);  // first chunk of every group
        for (int32_t g = 0; g <= VG; ++g)
            vc0[g] = (int32_t)(std::lower_bound(c_slice.begin(), c_slice.end(), vs[g]) - c_slice.begin());
        for (int32_t g = 0; g < VG && near; ++g) {
            const int32_t lo = vc0[std::max(g - 1, 0)], hi = vc0[std::min(g + 2, VG)];
            for (int32_t c = vc0[g]; c < vc0[g + 1]; ++c) near = near && hull[c].x >= lo && hull[c].y < hi;
        }
    }
    if (near) {
        bool own = false;  // a copy of its own
        if (natural) {
            // the plan's
        } else if (P.padded <= P.nnz + P.nnz / 25) {
            if (plan_dict) own = spare(P, P.wave, [&]() {
                    Tmp<int32_t> width(NS, s);
                    Tmp<int64_t> units((int64_t)NS + 1, s);
                    return pack_slices(P, P.wave, PlanRows{P.slice_ptr, P.col}, P.val, vs, ranges, plan_dict, d_srow, NS,
                                       width, units, host[0], s);
                });
        } else {
            std::vector<int32_t> vrow;
            for (int32_t g = 0; g <= VG; ++g) vrow.push_back(s_row[vs[g]]);
            own = spare(P, P.wave, [&]() {
                return wave_copy(P, P.wave, A, P.perm, P.iperm, vrow, ranges, plan_dict, host[0], s);
            });
        }
        if (!own && spare(P, P.wave, [&]() {
                return wave_tables(P, P.wave, vs, ranges, P.slice_ptr, nullptr, d_srow, NS, host[0], 0, s);
            })) {
            P.wave.val = P.val;
            P.wave.col = P.col;
            P.wave.ok = true;
        }
        P.wave.scattered = spread[1].scattered();
    }
}

Plan *build_plan(const mpk_csr *A, const Levels *L, const mpk_plan_opts *o, cudaStream_t s,
                 const std::vector<int32_t> *inst_row, const std::vector<int32_t> *inst_p) {
    if (!o) fail(MPK_ERR_INVALID, "options are NULL");
    int32_t band = 0;
    validate_csr(A, s, &band);
    if (o->p_max < 1 || o->p_max > kMaxP) fail(MPK_ERR_INVALID, "p_max must be in [1, %d]", kMaxP);
    if (!(o->nrhs == 1 || o->nrhs == 2 || o->nrhs == 4 || o->nrhs == 8 || o->nrhs == 16))
        fail(MPK_ERR_UNSUPPORTED, "nrhs must be 1, 2, 4, 8 or 16 (got %d)", o->nrhs);
    // 16 right-hand sides: a row's 16 x values and sums need the registers of the unstaged
    // shape at one block per SM; the staged shapes and the warp engine would spill
    if (o->nrhs == 16 && ((o->shape > 0 && o->shape != 3) || o->engine == MPK_ENGINE_WARP))
        fail(MPK_ERR_UNSUPPORTED, "16 right-hand sides run on the unstaged block shape (plan option shape 0 or 3) "
                                  "of the staged or the sweep engine");
    if (o->order != MPK_ORDER_ORIGINAL && o->order != MPK_ORDER_PLAN) fail(MPK_ERR_INVALID, "bad order");
    int32_t chunk_rows = o->chunk_rows;  // 0: 32 rows per compute warp of the block shape
    if (chunk_rows != 0 && (chunk_rows < 32 || chunk_rows > 8192 || chunk_rows % 32))
        fail(MPK_ERR_INVALID, "chunk_rows must be a multiple of 32 in [32, 8192]");
    if (o->cache_bytes < 0 || o->mem_budget < 0 || o->wait_limit_ns < 0) fail(MPK_ERR_INVALID, "negative option");
    if (L && L->n != A->n) fail(MPK_ERR_INVALID, "levels were built for n = %d, matrix has n = %d", L->n, A->n);

    const int32_t n = A->n, m = o->nrhs, pmax = o->p_max;
    Plan *P = new Plan();
    try {
        P->arena.budget = o->mem_budget;
        P->n = n;
        P->nnz = A->nnz;
        P->m = m;
        P->p_max = pmax;
        P->val_type = A->val_type;
        P->val_bytes = A->val_type == MPK_F64 ? 8 : (A->val_type == MPK_F32 ? 4 : 2);
        // binary32 accumulation: values stored in float32 or bfloat16 (exact in binary32), the
        // staged or sweep engine, single plans
        if (o->accum != MPK_F64 && o->accum != MPK_F32) fail(MPK_ERR_INVALID, "accum must be MPK_F64 or MPK_F32");
        P->accum = o->accum;
        if (P->accum == MPK_F32) {
            if (A->val_type == MPK_F64)
                fail(MPK_ERR_UNSUPPORTED, "binary32 accumulation needs values stored as float32 or bfloat16");
            if (o->engine == MPK_ENGINE_WARP || o->trace || o->level_capped || inst_row != nullptr ||
                o->shape - 1 == kShapeX)
                fail(MPK_ERR_UNSUPPORTED,
                     "binary32 accumulation runs on the staged engine (any shape but the X-staged one) or the "
                     "sweep engine, without trace, level caps or batching");
        }
        P->order = o->order;
        P->identity = (L == nullptr);
        P->chunk_rows = chunk_rows;
        // Units of two slices a warp (block shape 4) are the planner's choice for binary32 sums
        // over 2-byte values, one right-hand side and short rows (decided here from the mean row
        // length, since the budget shapes the groups the slices are cut from); they want larger
        // groups: measured at 256^3, p = 8, 1.575 / 1.486 / 1.459 / 1.468 ms at C = 96 / 128 /
        // 160 / 192 MB.  Every other plan: three quarters of L2.
        const bool two_slices = o->shape == 5 || (o->shape == 0 && o->accum == MPK_F32 && P->val_bytes == 2 &&
                                                  o->nrhs == 1 && A->nnz <= 10 * (int64_t)A->n);
        P->cache_bytes = o->cache_bytes ? o->cache_bytes : device_l2_bytes() / 4 * (two_slices ? 5 : 3);
        P->window = kSlotSkew * pmax + 1;
        P->group_budget = P->cache_bytes / P->window;
        P->wait_ns = o->wait_limit_ns ? o->wait_limit_ns : 2000000000LL;
        P->num_levels = L ? L->num_levels : 0;
        const bool batch = inst_row != nullptr;
        P->level_capped = o->level_capped != 0;
        if (P->level_capped && (!L || batch || o->order != MPK_ORDER_PLAN))
            fail(MPK_ERR_INVALID, "level_capped needs levels, plan order and no batch");
        P->split_levels = o->split_levels != 0;
        if (P->split_levels && (!L || batch || P->level_capped || o->engine == MPK_ENGINE_WARP))
            fail(MPK_ERR_INVALID, "split_levels needs levels and the staged or sweep engine, without level caps or "
                                  "batching");
        if (batch) {
            if (!L || !inst_p || inst_row->size() != inst_p->size() + 1 || inst_row->back() != n)
                fail(MPK_ERR_INVALID, "inconsistent batch description");
            P->inst_row = *inst_row;
            P->inst_p = *inst_p;
        }

        // ---- permutation (plan-owned copies)
        // (arrays that live together share a block: a large cudaMalloc and its cudaFree take 100 us)
        P->rowlen = P->arena.alloc_n<int32_t>((P->identity ? 1 : 3) * (int64_t)std::max(n, 1));
        if (!P->identity && n > 0) {
            P->perm = P->rowlen + n;
            P->iperm = P->perm + n;
            MPK_CUDA(cudaMemcpyAsync(P->perm, L->perm, sizeof(int32_t) * (size_t)n, cudaMemcpyDeviceToDevice, s));
            MPK_CUDA(cudaMemcpyAsync(P->iperm, L->iperm, sizeof(int32_t) * (size_t)n, cudaMemcpyDeviceToDevice, s));
        }
        if (n > 0) {
            k_rowlen<<<grid_n(n), 256, 0, s>>>(n, A->row_ptr, P->perm, P->rowlen);
            MPK_LAUNCHED();
        }

        // ---- groups: greedy rule over levels (host), identical to the written rule
        std::vector<int32_t> g_level, g_row;
        if (P->identity) {
            g_row = {0, n};
        } else if (n > 0) {
            const int32_t NL = L->num_levels;
            Tmp<int32_t> prp((int64_t)n + 1, s);
            exclusive_scan(P->rowlen, prp.p, n, s);
            Tmp<int32_t> lvl_nnz((int64_t)NL + 1, s);
            k_gather_i32<<<grid_n(NL + 1), 256, 0, s>>>(prp.p, L->level_ptr, NL + 1, lvl_nnz.p);
            MPK_LAUNCHED();
            std::vector<int32_t> h_nz((size_t)NL + 1);
            MPK_CUDA(cudaMemcpyAsync(h_nz.data(), lvl_nnz.p, sizeof(int32_t) * ((size_t)NL + 1),
                                     cudaMemcpyDeviceToHost, s));
            MPK_CUDA(cudaStreamSynchronize(s));
            const std::vector<int32_t> &lp = L->h_level_ptr;
            const int64_t B = P->group_budget;
            const int64_t vb = P->val_bytes;  // value bytes of the stored type
            // batch plans: a group never holds levels of two instances (every instance is a
            // union of components, numbered after the previous one, so it starts a level)
            std::vector<char> inst_start((size_t)NL, 0);
            if (batch) {
                for (size_t i = 0; i + 1 < P->inst_row.size(); ++i) {
                    if (P->inst_row[i + 1] == P->inst_row[i]) continue;  // empty instance
                    const auto it = std::lower_bound(lp.begin(), lp.begin() + NL, P->inst_row[i]);
                    if (it == lp.begin() + NL || *it != P->inst_row[i])
                        fail(MPK_ERR_INVALID, "instance %zu does not start a level", i);
                    inst_start[it - lp.begin()] = 1;
                }
            }
            int64_t cur = 0, Bl = B;
            size_t inst = 0;
            g_level.push_back(0);
            for (int32_t l = 0; l < NL; ++l) {
                if (batch) {  // each block's groups share the cache with its own window only
                    while (inst + 1 < P->inst_p.size() && lp[l] >= P->inst_row[inst + 1]) ++inst;
                    Bl = P->cache_bytes / (kSlotSkew * P->inst_p[inst] + 1);
                }
                const int64_t rows = lp[l + 1] - lp[l];
                const int64_t nz = (int64_t)h_nz[l + 1] - h_nz[l];
                const int64_t b = (vb + 4) * nz + 4 * rows + 16 * (int64_t)m * rows;
                // level-capped plans: every level below p_max is a group of its own
                const bool cut = P->level_capped && l <= pmax;
                if (l > 0 && !inst_start[l] && !cut && cur + b <= Bl) {
                    cur += b;
                } else {
                    if (l > 0) g_level.push_back(l);
                    cur = b;
                }
            }
            g_level.push_back(NL);
            if (P->level_capped && NL > 0) P->level0_rows = lp[1];
            for (int32_t gl : g_level) g_row.push_back(lp[gl]);
            if (P->split_levels) {
                // Bulky levels split (the recursion stage of Sec. 6, read as breaking a level too
                // large for the budget into pieces): levels group as above while they fit; a level
                // over the budget closes the current group and is cut into pieces of consecutive
                // rows, each taking rows while its bytes stay <= budget (at least one row), each a
                // group; the next level starts a new group.  A row costs (val_bytes + 4) nnz + 4 +
                // 16 m bytes.  group_level_ptr then holds the level of each group's first row.
                std::vector<int32_t> rl((size_t)n), prow((size_t)n + 1);
                MPK_CUDA(cudaMemcpyAsync(rl.data(), P->rowlen, sizeof(int32_t) * (size_t)n, cudaMemcpyDeviceToHost, s));
                MPK_CUDA(cudaStreamSynchronize(s));
                g_row.assign(1, 0);
                g_level.assign(1, 0);
                int64_t cur2 = 0;
                for (int32_t l = 0; l < NL; ++l) {
                    const int64_t rows = lp[l + 1] - lp[l];
                    const int64_t nz = (int64_t)h_nz[l + 1] - h_nz[l];
                    const int64_t b = (vb + 4) * nz + 4 * rows + 16 * (int64_t)m * rows;
                    if (b > B) {
                        if (l > 0 && g_row.back() != lp[l]) {
                            g_row.push_back(lp[l]);
                            g_level.push_back(l);
                        }
                        int64_t piece = 0;
                        for (int32_t r = lp[l]; r < lp[l + 1]; ++r) {
                            const int64_t rb = (vb + 4) * rl[r] + 4 + 16 * (int64_t)m;
                            if (r > lp[l] && piece + rb > B) {
                                g_row.push_back(r);
                                g_level.push_back(l);
                                piece = 0;
                            }
                            piece += rb;
                        }
                        if (l + 1 < NL) {
                            g_row.push_back(lp[l + 1]);
                            g_level.push_back(l + 1);
                        }
                        cur2 = 0;
                        continue;
                    }
                    if (l > 0 && g_row.back() == lp[l]) {
                        cur2 = b;
                    } else if (l > 0 && cur2 + b <= B) {
                        cur2 += b;
                    } else {
                        if (l > 0) {
                            g_row.push_back(lp[l]);
                            g_level.push_back(l);
                        }
                        cur2 = b;
                    }
                }
                g_row.push_back(lp[NL]);
                g_level.push_back(NL);
            }
        } else {
            g_row = {0, 0};
        }
        const int32_t G = (int32_t)g_row.size() - 1;
        P->num_groups = G;

        // ---- slices: 32-row blocks counted from each group's first row (host)
        std::vector<int32_t> s_row;
        s_row.push_back(0);
        std::vector<int32_t> g_slice;
        for (int32_t g = 0; g < G; ++g) {
            g_slice.push_back((int32_t)s_row.size() - 1);
            for (int32_t r = g_row[g]; r < g_row[g + 1]; r += 32) s_row.push_back(std::min(r + 32, g_row[g + 1]));
        }
        g_slice.push_back((int32_t)s_row.size() - 1);
        const int32_t NS = (int32_t)s_row.size() - 1;
        P->num_slices = NS;
        Tmp<int32_t> d_srow((int64_t)NS + 1, s);
        Tmp<int32_t> d_width(NS, s);
        MPK_CUDA(cudaMemcpyAsync(d_srow.p, s_row.data(), sizeof(int32_t) * ((size_t)NS + 1), cudaMemcpyHostToDevice, s));
        if (NS > 0) {
            k_slice_width<<<grid_n(NS), 256, 0, s>>>(d_srow.p, NS, P->rowlen, d_width.p);
            MPK_LAUNCHED();
        }
        std::vector<int32_t> width((size_t)NS);
        if (NS > 0)
            MPK_CUDA(cudaMemcpyAsync(width.data(), d_width.p, sizeof(int32_t) * (size_t)NS, cudaMemcpyDeviceToHost, s));
        MPK_CUDA(cudaStreamSynchronize(s));
        std::vector<int64_t> sptr((size_t)NS + 1, 0);
        for (int32_t i = 0; i < NS; ++i) sptr[i + 1] = sptr[i] + 32 * (int64_t)width[i];
        P->padded = sptr[NS];

        // ---- block shape: shape 1 when its slot holds at least 6 slices of the mean
        //      width, else unstaged (measured: 27-point stencils run 1.7x
        //      faster unstaged).  Shape 1's fewer, larger units beat shape 0 on the 3-D
        //      Laplacian (2.20 ms against 2.58 ms at 256^3, p = 8), since the per-unit work of
        //      the control warp sets the pace; for the same reason binary32 sums over 2-byte
        //      values take shape 4 (two slices a warp) when its slot holds 24 slices of the
        //      mean width (1.459 against 1.622 ms at their best budgets); shapes 0 and 3 (input
        //      rows staged too) are taken only when the options name them.
        if (o->shape < 0 || o->shape > kNumShapes) fail(MPK_ERR_INVALID, "shape must be in [0, %d]", kNumShapes);
        int fallback_shape = 0;
        bool try_x = false;
        if (o->shape > 0) {
            fallback_shape = o->shape - 1;
            try_x = fallback_shape == kShapeX;
        } else {
            auto fits = [&](int sh, int slices) {
                return (int64_t)slices * P->padded <= (int64_t)kShapes[sh].stage_entries * std::max(NS, 1);
            };
            fallback_shape = (o->nrhs < 16 && fits(1, 6)) ? 1 : 2;  // up to 24 entries a row on average
            if (two_slices && fits(4, 24)) fallback_shape = 4;      // up to 12 entries a row
            try_x = false;
        }
        const bool x_forced = o->shape - 1 == kShapeX;

        // ---- sliced copy and group tables (independent of the chunks)
        P->group_row_ptr = P->arena.alloc_n<int32_t>(G + 1);
        MPK_CUDA(cudaMemcpyAsync(P->group_row_ptr, g_row.data(), sizeof(int32_t) * (G + 1), cudaMemcpyHostToDevice, s));
        if (!P->identity) {
            P->group_level_ptr = P->arena.alloc_n<int32_t>(G + 1);
            MPK_CUDA(cudaMemcpyAsync(P->group_level_ptr, g_level.data(), sizeof(int32_t) * (G + 1),
                                     cudaMemcpyHostToDevice, s));
        }
        P->slice_ptr = P->arena.alloc_n<int64_t>((int64_t)NS + 1);
        MPK_CUDA(cudaMemcpyAsync(P->slice_ptr, sptr.data(), sizeof(int64_t) * ((size_t)NS + 1), cudaMemcpyHostToDevice, s));
        Tmp<int32_t> cor(n, s);
        P->col = static_cast<int32_t *>(P->arena.alloc((P->padded + 32) * (4 + P->val_bytes)));  // columns, then values
        P->val = P->col + (P->padded + 32);
        MPK_CUDA(cudaMemsetAsync(P->val, 0, (size_t)P->val_bytes * (size_t)(P->padded + 32), s));  // +0 in every type
        MPK_CUDA(cudaMemsetAsync(P->col, 0xff, sizeof(int32_t) * (size_t)(P->padded + 32), s));  // padding: col = -1

        std::vector<int32_t> c_row, c_slice, g_chunk;
        std::vector<int2> chunk_hull;  // first and last chunk of each chunk's dependencies
        std::vector<int32_t> h_win;  // shape 3: kXWin (first row, rows, position) per chunk
        int32_t NC = 0, stage_entries = 0;
        for (int attempt = 0;; ++attempt) {
            P->shape = (attempt == 0 && try_x) ? kShapeX : fallback_shape;
            if (attempt > 0 && P->shape == kShapeX) fail(MPK_ERR_UNSUPPORTED, "block shape 3 does not fit this plan");
            stage_entries = kShapes[P->shape].stage_entries;
            const int64_t chunk_entries = stage_entries > 0 ? stage_entries : INT64_MAX;
            chunk_rows = o->chunk_rows ? o->chunk_rows
                                       : 32 * kShapes[P->shape].comp_warps * std::max(1, kShapes[P->shape].slices_per_warp);
            P->chunk_rows = chunk_rows;

            // ---- chunks: consecutive slices of one group, at most chunk_rows rows and at most
            //      stage_entries padded entries (a single wider slice forms its own chunk)
            c_row.assign(1, 0);
            c_slice.assign(1, 0);
            g_chunk.clear();
            for (int32_t g = 0; g < G; ++g) {
                g_chunk.push_back((int32_t)c_row.size() - 1);
                int32_t s0 = g_slice[g];
                while (s0 < g_slice[g + 1]) {
                    int32_t s1 = s0 + 1;
                    while (s1 < g_slice[g + 1] && s_row[s1 + 1] - s_row[s0] <= chunk_rows &&
                           sptr[s1 + 1] - sptr[s0] <= chunk_entries)
                        ++s1;
                    c_row.push_back(s_row[s1]);
                    c_slice.push_back(s1);
                    s0 = s1;
                }
            }
            g_chunk.push_back((int32_t)c_row.size() - 1);
            NC = (int32_t)c_row.size() - 1;
            P->h_chunk_row = c_row;
            if (NC >= (1 << 26)) fail(MPK_ERR_TOO_LARGE, "too many chunks (%d)", NC);
            P->num_chunks = NC;
            P->chunk_row = P->arena.alloc_n<int32_t>(NC + 1);
            P->chunk_slice = P->arena.alloc_n<int32_t>(NC + 1);
            MPK_CUDA(cudaMemcpyAsync(P->chunk_row, c_row.data(), sizeof(int32_t) * (NC + 1), cudaMemcpyHostToDevice, s));
            MPK_CUDA(cudaMemcpyAsync(P->chunk_slice, c_slice.data(), sizeof(int32_t) * (NC + 1), cudaMemcpyHostToDevice,
                                     s));

            // ---- fill the sliced copy; dependency hulls of the chunks
            P->dep = P->arena.alloc_n<int2>(NC > 0 ? NC : 1);
            if (NC > 0) {
                k_dep_init<<<grid_n(NC), 256, 0, s>>>(P->dep, NC);
                MPK_LAUNCHED();
                k_chunk_of_row<<<grid_n((int64_t)NC * 256), 256, 0, s>>>(P->chunk_row, NC, cor.p);
                MPK_LAUNCHED();
#define FILL(T)                                                                                            \
    k_fill<T><<<grid_n(n), 256, 0, s>>>(n, A->row_ptr, A->col, static_cast<const T *>(A->val), P->perm,    \
                                        P->iperm, P->chunk_row, P->chunk_slice, cor.p, P->slice_ptr,         \
                                        static_cast<T *>(P->val), P->col, P->dep, A->is_symmetric ? 1 : 0, special.p)
                Tmp<int32_t> special(1, s);
                MPK_CUDA(cudaMemsetAsync(special.p, 0, sizeof(int32_t), s));
                if (P->val_type == MPK_F64)
                    FILL(double);
                else if (P->val_type == MPK_F32)
                    FILL(float);
                else
                    FILL(uint16_t);
#undef FILL
                MPK_LAUNCHED();
                int32_t has_special = 0;
                MPK_CUDA(cudaMemcpyAsync(&has_special, special.p, sizeof(int32_t), cudaMemcpyDeviceToHost, s));
                MPK_CUDA(cudaStreamSynchronize(s));
                if (has_special)
                    fail(MPK_ERR_UNSUPPORTED,
                         "float32/bfloat16 storage holds zeros and normal numbers only (a value is subnormal, "
                         "infinite or NaN in the narrow type): use MPK_F64 values");
            }
            // ---- dependency ranges: exact chunk sets as bitmaps over each hull, compressed
            P->dep_ranges = P->arena.alloc_n<int4>(2 * (int64_t)(NC > 0 ? NC : 1));
            if (NC > 0) {
                std::vector<int2> &hull = chunk_hull;
                hull.resize((size_t)NC);
                MPK_CUDA(cudaMemcpyAsync(hull.data(), P->dep, sizeof(int2) * (size_t)NC, cudaMemcpyDeviceToHost, s));
                MPK_CUDA(cudaStreamSynchronize(s));
                std::vector<int64_t> woff((size_t)NC + 1, 0);
                for (int32_t c = 0; c < NC; ++c) woff[c + 1] = woff[c] + (hull[c].y - hull[c].x + 32) / 32;
                const int64_t words = woff[NC];
                if (words <= ((int64_t)1 << 27)) {
                    Tmp<int64_t> d_woff((int64_t)NC + 1, s);
                    Tmp<uint32_t> d_bits(words, s);
                    MPK_CUDA(cudaMemcpyAsync(d_woff.p, woff.data(), sizeof(int64_t) * ((size_t)NC + 1),
                                             cudaMemcpyHostToDevice, s));
                    MPK_CUDA(cudaMemsetAsync(d_bits.p, 0, sizeof(uint32_t) * (size_t)words, s));
                    k_dep_bits<<<grid_n(n), 256, 0, s>>>(n, P->rowlen, P->chunk_row, P->chunk_slice, cor.p,
                                                         P->slice_ptr, P->col, P->dep, d_woff.p, d_bits.p,
                                                         A->is_symmetric ? 1 : 0);
                    MPK_LAUNCHED();
                    k_dep_ranges<<<grid_n(NC), 256, 0, s>>>(NC, P->dep, d_woff.p, d_bits.p, P->dep_ranges);
                    MPK_LAUNCHED();
                    MPK_CUDA(cudaStreamSynchronize(s));
                } else {  // bitmaps too large: one range per chunk, the hull
                    std::vector<int4> rr((size_t)2 * NC);
                    for (int32_t c = 0; c < NC; ++c) {
                        rr[2 * c] = make_int4(hull[c].x, hull[c].y, 0, -1);
                        rr[2 * c + 1] = make_int4(0, -1, 0, -1);
                    }
                    MPK_CUDA(cudaMemcpyAsync(P->dep_ranges, rr.data(), sizeof(int4) * rr.size(), cudaMemcpyHostToDevice,
                                             s));
                    MPK_CUDA(cudaStreamSynchronize(s));
                }
            }
            // ---- shape 3: input-row windows per chunk, laid out in the slot's window area
            //      (rows from position 1 on, a gap of 2 / nrhs rows between windows, positions
            //      of the parity of the first row when nrhs = 1; see x_copy in the kernel)
            if (P->shape == kShapeX) {
                bool ok = NC > 0;
                h_win.assign((size_t)3 * kXWin * std::max(NC, 1), 0);
                if (ok) {
                    Tmp<int2> d_xw((int64_t)kXWin * NC, s);
                    std::vector<int2> xw((size_t)kXWin * NC, make_int2(INT_MAX, -1));
                    MPK_CUDA(cudaMemcpyAsync(d_xw.p, xw.data(), sizeof(int2) * xw.size(), cudaMemcpyHostToDevice, s));
                    k_xwin<<<grid_n(n), 256, 0, s>>>(n, P->rowlen, P->chunk_row, P->chunk_slice, cor.p, P->slice_ptr,
                                                     P->col, P->dep_ranges, d_xw.p);
                    MPK_LAUNCHED();
                    MPK_CUDA(cudaMemcpyAsync(xw.data(), d_xw.p, sizeof(int2) * xw.size(), cudaMemcpyDeviceToHost, s));
                    MPK_CUDA(cudaStreamSynchronize(s));
                    const int64_t XW = kShapes[kShapeX].x_words;
                    for (int32_t c = 0; c < NC && ok; ++c) {
                        // every chunk must be staged: its entries fit the slot and its widths the record
                        if (c_slice[c + 1] - c_slice[c] > kRecSlices ||
                            sptr[c_slice[c + 1]] - sptr[c_slice[c]] > stage_entries)
                            ok = false;
                        int64_t pos = 1;
                        for (int q = 0; q < kXWin && ok; ++q) {
                            const int2 w = xw[(size_t)kXWin * c + q];
                            if (w.y < w.x) continue;
                            const int64_t len = (int64_t)w.y - w.x + 1;
                            if (m == 1 && ((pos ^ w.x) & 1)) ++pos;
                            if (m * (pos + len) + 2 > XW) {
                                ok = false;
                                break;
                            }
                            int32_t *hw = &h_win[(size_t)3 * kXWin * c + 3 * q];
                            hw[0] = w.x;
                            hw[1] = (int32_t)len;
                            hw[2] = (int32_t)pos;
                            pos += len + (m == 1 ? 2 : 1);
                        }
                    }
                }
                if (!ok) {
                    if (x_forced)
                        fail(MPK_ERR_UNSUPPORTED,
                             "block shape 3: a chunk's input rows do not fit a staging slot (fewer chunk_rows, or "
                             "another shape)");
                    P->arena.free(P->chunk_row);
                    P->arena.free(P->chunk_slice);
                    P->arena.free(P->dep);
                    P->arena.free(P->dep_ranges);
                    P->chunk_row = P->chunk_slice = nullptr;
                    P->dep = nullptr;
                    P->dep_ranges = nullptr;
                    h_win.clear();
                    continue;
                }
                Tmp<int32_t> d_win((int64_t)h_win.size(), s);
                MPK_CUDA(cudaMemcpyAsync(d_win.p, h_win.data(), sizeof(int32_t) * h_win.size(), cudaMemcpyHostToDevice,
                                         s));
                P->lcol = P->arena.alloc_n<uint16_t>(P->padded + 32);
                MPK_CUDA(cudaMemsetAsync(P->lcol, 0xff, sizeof(uint16_t) * (size_t)(P->padded + 32), s));
                k_lcol<<<grid_n(n), 256, 0, s>>>(n, P->rowlen, P->chunk_row, P->chunk_slice, cor.p, P->slice_ptr,
                                                 P->col, d_win.p, P->lcol);
                MPK_LAUNCHED();
                MPK_CUDA(cudaStreamSynchronize(s));  // d_win goes out of scope
            }
            break;
        }

        P->chunk_rec = reinterpret_cast<int4 *>(P->arena.alloc_n<int32_t>((int64_t)kRecInts * (NC > 0 ? NC : 1)));
        if (NC > 0) {
            Tmp<int32_t> d_win(P->shape == kShapeX ? (int64_t)h_win.size() : 0, s);
            if (P->shape == kShapeX)
                MPK_CUDA(cudaMemcpyAsync(d_win.p, h_win.data(), sizeof(int32_t) * h_win.size(), cudaMemcpyHostToDevice,
                                         s));
            k_chunk_records<<<grid_n(NC), 256, 0, s>>>(NC, P->chunk_row, P->chunk_slice, P->slice_ptr, P->dep_ranges,
                                                      stage_entries, d_win.p,
                                                      // slices a staged chunk may have: what the shape's
                                                      // compute warps read widths for
                                                      kShapes[P->shape].slices_per_warp > 1 ? kRecSlicesWide : kRecSlices,
                                                      reinterpret_cast<int32_t *>(P->chunk_rec));
            MPK_LAUNCHED();
            MPK_CUDA(cudaStreamSynchronize(s));
        }

        // ---- unit tables: Lp-diagram cells (group g, power k) along lines g + kSlotSkew*k
        //      ascending, k ascending inside a line, chunks in row order; unit = chunk << 5 | k
        P->unit_off.assign((size_t)pmax + 2, 0);
        std::vector<int32_t> units;
        if (batch) {
            // one table: every instance's cells up to its own power, instance after instance;
            // blocks claim the next instance's first units while the previous one drains, and
            // about one instance at a time holds the cache.  Each instance keeps its own order,
            // so dependencies keep smaller tickets.
            const int32_t NI = (int32_t)P->inst_p.size();
            std::vector<int32_t> gi0((size_t)NI), gi1((size_t)NI);
            int32_t dmax = 0;
            for (int32_t i = 0; i < NI; ++i) {
                gi0[i] = (int32_t)(std::lower_bound(g_row.begin(), g_row.end() - 1, P->inst_row[i]) - g_row.begin());
                gi1[i] = (int32_t)(std::lower_bound(g_row.begin(), g_row.end() - 1, P->inst_row[i + 1]) - g_row.begin());
                if (P->inst_row[i + 1] == n) gi1[i] = G;
                const int32_t pi = P->inst_p[i];
                if (pi < 1 || pi > pmax) fail(MPK_ERR_INVALID, "instance %d: p = %d outside [1, p_max]", i, pi);
                if (gi1[i] > gi0[i]) dmax = std::max(dmax, gi1[i] - gi0[i] - 1 + kSlotSkew * pi);
            }
            for (int32_t i = 0; i < NI; ++i)
                for (int32_t d = kSlotSkew; d <= dmax; ++d)
                    for (int32_t k = 1; k <= P->inst_p[i]; ++k) {
                        const int32_t g = gi0[i] + d - kSlotSkew * k;
                        if (g < gi0[i] || g >= gi1[i]) continue;
                        for (int32_t c = g_chunk[g]; c < g_chunk[g + 1]; ++c) units.push_back((c << 5) | k);
                    }
            P->unit_off[pmax + 1] = (int64_t)units.size();  // the table of p = p_max is the batch table
        }
        // level-capped plans: group g (a single level below p_max, or levels >= p_max) takes
        // powers up to its first level
        std::vector<int32_t> g_cap((size_t)G, pmax);
        if (P->level_capped)
            for (int32_t g = 0; g < G; ++g) g_cap[g] = std::min(pmax, g_level[g]);
        // race-detection aid: shuffle_seed != 0 permutes the units of every line (all their
        // dependencies lie on earlier lines, so any order inside a line is a valid schedule and
        // must give the same bits); splitmix64 drives a Fisher-Yates shuffle
        uint64_t rng = (uint64_t)o->shuffle_seed;
        auto next_rand = [&rng]() {
            uint64_t z = (rng += 0x9e3779b97f4a7c15ULL);
            z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ULL;
            z = (z ^ (z >> 27)) * 0x94d049bb133111ebULL;
            return z ^ (z >> 31);
        };
        // split plans: the groups of a split level need not read only their neighbours, so the
        // units follow waves computed from the exact chunk dependencies: w(c, 1) = kSlotSkew + g(c),
        // w(c, k) = max{ w(c', k-1) : c' in the dependency ranges of c } + 2, units by increasing
        // (w, k, chunk).  Every dependency has a smaller wave, hence a smaller ticket: the
        // schedule stays deadlock free.  (For unsplit levels this reproduces the lines g + 3k.)
        std::vector<int64_t> wave;  // wave of unit (c, k) at (k - 1) * NC + c
        if (P->split_levels && NC > 0) {
            std::vector<int4> rr((size_t)2 * NC);
            MPK_CUDA(cudaMemcpyAsync(rr.data(), P->dep_ranges, sizeof(int4) * rr.size(), cudaMemcpyDeviceToHost, s));
            MPK_CUDA(cudaStreamSynchronize(s));
            wave.assign((size_t)pmax * NC, 0);
            for (int32_t g = 0; g < G; ++g)
                for (int32_t c = g_chunk[g]; c < g_chunk[g + 1]; ++c) wave[c] = kSlotSkew + g;
            int lg = 1;
            while ((1 << lg) < NC) ++lg;
            std::vector<int64_t> st((size_t)(lg + 1) * NC);  // sparse table of range maxima
            for (int32_t k = 2; k <= pmax; ++k) {
                const int64_t *prev = wave.data() + (size_t)(k - 2) * NC;
                for (int32_t c = 0; c < NC; ++c) st[c] = prev[c];
                for (int j = 1; j <= lg; ++j)
                    for (int32_t c = 0; c + (1 << j) <= NC; ++c)
                        st[(size_t)j * NC + c] =
                            std::max(st[(size_t)(j - 1) * NC + c], st[(size_t)(j - 1) * NC + c + (1 << (j - 1))]);
                auto range_max = [&](int32_t a, int32_t b) {  // inclusive, a <= b
                    int j = 0;
                    while ((2 << j) <= b - a + 1) ++j;
                    return std::max(st[(size_t)j * NC + a], st[(size_t)j * NC + b - (1 << j) + 1]);
                };
                int64_t *cur = wave.data() + (size_t)(k - 1) * NC;
                for (int32_t c = 0; c < NC; ++c) {
                    const int32_t lo4[4] = {rr[2 * c].x, rr[2 * c].z, rr[2 * c + 1].x, rr[2 * c + 1].z};
                    const int32_t hi4[4] = {rr[2 * c].y, rr[2 * c].w, rr[2 * c + 1].y, rr[2 * c + 1].w};
                    int64_t mx = 0;
                    for (int q = 0; q < 4; ++q)
                        if (hi4[q] >= lo4[q]) mx = std::max(mx, range_max(lo4[q], hi4[q]));
                    cur[c] = mx + 2;
                }
            }
        }
        for (int32_t p = 1; p <= pmax && !batch && P->split_levels; ++p) {
            P->unit_off[p] = (int64_t)units.size();
            std::vector<std::pair<int64_t, int32_t>> ord;  // (wave, unit)
            ord.reserve((size_t)p * NC);
            for (int32_t k = 1; k <= p; ++k)
                for (int32_t c = 0; c < NC; ++c) ord.push_back({wave[(size_t)(k - 1) * NC + c], (c << 5) | k});
            std::sort(ord.begin(), ord.end(), [](const std::pair<int64_t, int32_t> &x, const std::pair<int64_t, int32_t> &y) {
                if (x.first != y.first) return x.first < y.first;
                if ((x.second & 31) != (y.second & 31)) return (x.second & 31) < (y.second & 31);
                return x.second < y.second;
            });
            for (size_t j = 0; j < ord.size();) {  // one wave at a time (shuffled on request)
                size_t e = j;
                while (e < ord.size() && ord[e].first == ord[j].first) ++e;
                const size_t line0 = units.size();
                for (size_t q = j; q < e; ++q) units.push_back(ord[q].second);
                if (o->shuffle_seed != 0)
                    for (size_t q = units.size() - 1; q > line0; --q)
                        std::swap(units[q], units[line0 + next_rand() % (q - line0 + 1)]);
                j = e;
            }
        }
        // line order without shuffling: the tables are listed as cells (group, power) here and
        // expanded into units on the device (1.2 M units at 256^3, p_max = 8: a host loop and
        // copy took 2.7 ms); the same order as the host loop below
        const bool cells_on_device = !batch && !P->split_levels && o->shuffle_seed == 0;
        std::vector<int64_t> cell_off;
        std::vector<int4> cell;
        int64_t total_units = 0;
        for (int32_t p = 1; p <= pmax && cells_on_device; ++p) {
            P->unit_off[p] = total_units;
            for (int32_t d = kSlotSkew; d <= G - 1 + kSlotSkew * p; ++d)
                for (int32_t k = 1; k <= p; ++k) {
                    const int32_t g = d - kSlotSkew * k;
                    if (g < 0 || g >= G || k > g_cap[g]) continue;
                    const int32_t nc = g_chunk[g + 1] - g_chunk[g];
                    if (nc <= 0) continue;
                    cell_off.push_back(total_units);
                    cell.push_back(make_int4(g_chunk[g], nc, k, 0));
                    total_units += nc;
                }
        }
        for (int32_t p = 1; p <= pmax && !batch && !P->split_levels && !cells_on_device; ++p) {
            P->unit_off[p] = (int64_t)units.size();
            for (int32_t d = kSlotSkew; d <= G - 1 + kSlotSkew * p; ++d) {
                const size_t line0 = units.size();
                for (int32_t k = 1; k <= p; ++k) {
                    const int32_t g = d - kSlotSkew * k;
                    if (g < 0 || g >= G || k > g_cap[g]) continue;
                    for (int32_t c = g_chunk[g]; c < g_chunk[g + 1]; ++c) units.push_back((c << 5) | k);
                }
                if (o->shuffle_seed != 0)
                    for (size_t j = units.size() - 1; j > line0; --j)
                        std::swap(units[j], units[line0 + next_rand() % (j - line0 + 1)]);
            }
        }
        if (!cells_on_device) total_units = (int64_t)units.size();
        if (!batch) P->unit_off[pmax + 1] = total_units;

        // ---- warp-ticketed engine: the same cells in the same order, split into items of
        //      kWarpSlices slices; counters of finished items per cell
        if (o->engine != MPK_ENGINE_STAGED && o->engine != MPK_ENGINE_WARP && o->engine != MPK_ENGINE_SWEEP)
            fail(MPK_ERR_INVALID, "engine must be MPK_ENGINE_STAGED, MPK_ENGINE_WARP or MPK_ENGINE_SWEEP");
        if (o->engine == MPK_ENGINE_SWEEP) {
            if (batch || P->level_capped) fail(MPK_ERR_INVALID, "batch and level-capped plans need level blocking");
            P->engine = MPK_ENGINE_SWEEP;
        }
        if (o->engine == MPK_ENGINE_WARP) {
            if (batch) fail(MPK_ERR_INVALID, "batch plans run on the staged engine");
            P->engine = MPK_ENGINE_WARP;
            std::vector<int64_t> w_item;
            std::vector<int32_t> w_gk;
            P->w_cell_off.assign((size_t)pmax + 2, 0);
            P->w_items.assign((size_t)pmax + 1, 0);
            for (int32_t p = 1; p <= pmax; ++p) {
                P->w_cell_off[p] = (int64_t)w_item.size();
                int64_t items = 0;
                for (int32_t d = kSlotSkew; d <= G - 1 + kSlotSkew * p; ++d)
                    for (int32_t k = 1; k <= p; ++k) {
                        const int32_t g = d - kSlotSkew * k;
                        if (g < 0 || g >= G || k > g_cap[g]) continue;
                        const int32_t ns = g_slice[g + 1] - g_slice[g];
                        if (ns <= 0) continue;
                        w_item.push_back(items);
                        w_gk.push_back((g << 5) | k);
                        items += (ns + kWarpSlices - 1) / kWarpSlices;
                    }
                P->w_items[p] = items;
                if (items >= ((int64_t)1 << 31) * kWarpQueues) fail(MPK_ERR_TOO_LARGE, "too many items");
            }
            P->w_cell_off[pmax + 1] = (int64_t)w_item.size();
            if (G >= (1 << 26)) fail(MPK_ERR_TOO_LARGE, "too many groups for the warp engine");
            P->g_slice = P->arena.alloc_n<int32_t>((int64_t)G + 1);
            MPK_CUDA(cudaMemcpyAsync(P->g_slice, g_slice.data(), sizeof(int32_t) * ((size_t)G + 1),
                                     cudaMemcpyHostToDevice, s));
            P->w_item = P->arena.alloc_n<int64_t>((int64_t)w_item.size() + 1);
            P->w_gk = P->arena.alloc_n<int32_t>((int64_t)w_gk.size() + 1);
            if (!w_item.empty()) {
                MPK_CUDA(cudaMemcpyAsync(P->w_item, w_item.data(), sizeof(int64_t) * w_item.size(),
                                         cudaMemcpyHostToDevice, s));
                MPK_CUDA(cudaMemcpyAsync(P->w_gk, w_gk.data(), sizeof(int32_t) * w_gk.size(), cudaMemcpyHostToDevice,
                                         s));
            }
            // per chunk: its slices, and in bits 24.. the highest power it computes (a power
            // above it never completes, so a dependency on it is void: level-capped plans)
            std::vector<int32_t> s_chunk((size_t)NS + 1, 0), c_nsl((size_t)NC + 1, 0);
            for (int32_t g = 0; g < G; ++g)
                for (int32_t c = g_chunk[g]; c < g_chunk[g + 1]; ++c) {
                    c_nsl[c] = (c_slice[c + 1] - c_slice[c]) | (g_cap[g] << 24);
                    for (int32_t q = c_slice[c]; q < c_slice[c + 1]; ++q) s_chunk[q] = c;
                }
            P->w_slice_chunk = P->arena.alloc_n<int32_t>((int64_t)NS + 1);
            P->w_chunk_nsl = P->arena.alloc_n<int32_t>((int64_t)NC + 1);
            MPK_CUDA(cudaMemcpyAsync(P->w_slice_chunk, s_chunk.data(), sizeof(int32_t) * ((size_t)NS + 1),
                                     cudaMemcpyHostToDevice, s));
            MPK_CUDA(cudaMemcpyAsync(P->w_chunk_nsl, c_nsl.data(), sizeof(int32_t) * ((size_t)NC + 1),
                                     cudaMemcpyHostToDevice, s));
            P->w_cnt = P->arena.alloc_n<int32_t>((int64_t)(pmax + 1) * std::max(NC, 1) + kWarpQueues);
            MPK_CUDA(cudaStreamSynchronize(s));  // host tables go out of scope
        }
        P->units = P->arena.alloc_n<int32_t>(total_units + 1);
        if (cells_on_device && !cell.empty()) {
            const int32_t ncells = (int32_t)cell.size();
            Tmp<int64_t> d_off(ncells, s);
            Tmp<int4> d_cell(ncells, s);
            MPK_CUDA(cudaMemcpyAsync(d_off.p, cell_off.data(), sizeof(int64_t) * cell_off.size(), cudaMemcpyHostToDevice,
                                     s));
            MPK_CUDA(cudaMemcpyAsync(d_cell.p, cell.data(), sizeof(int4) * cell.size(), cudaMemcpyHostToDevice, s));
            k_expand_cells<<<std::min(ncells, 64 * device_sms()), 128, 0, s>>>(d_off.p, d_cell.p, ncells, P->units);
            MPK_LAUNCHED();
        } else if (!units.empty()) {
            MPK_CUDA(cudaMemcpyAsync(P->units, units.data(), sizeof(int32_t) * units.size(), cudaMemcpyHostToDevice, s));
        }

        // ---- synchronisation state and vector workspace
        P->flags = P->arena.alloc_n<int32_t>((int64_t)(pmax + 1) * (NC > 0 ? NC : 1));
        MPK_CUDA(cudaMemsetAsync(P->flags, 0, sizeof(int32_t) * (size_t)(pmax + 1) * (NC > 0 ? NC : 1), s));
        if (o->trace) {
            P->trace = P->arena.alloc_n<unsigned long long>(MPK_TRACE_COUNTERS);
            MPK_CUDA(cudaMemsetAsync(P->trace, 0, sizeof(unsigned long long) * MPK_TRACE_COUNTERS, s));
        }
        // ticket, exit count, epoch and code of a failed launch, epoch of the last launch
        P->ctl = P->arena.alloc_n<unsigned int>(8);
        MPK_CUDA(cudaMemsetAsync(P->ctl, 0, 8 * sizeof(unsigned int), s));
        P->work_slots = std::max(pmax + 1, 4);  // all powers (original order) or ring of 3 + accumulator
        P->work = P->arena.alloc_n<double>((int64_t)P->work_slots * n * m + 1);
        if (P->accum == MPK_F32) P->shadow = P->arena.alloc_n<float>(2 * (int64_t)n * m + 1);
        std::vector<int32_t> wave_host[2];
        // ---- wave kernel: single plans of the staged engine, at the planner's block shape or the
        //      unstaged one
        if (o->engine == MPK_ENGINE_STAGED && (o->shape == 0 || o->shape == 3) && !P->level_capped && !P->split_levels &&
            !o->trace && o->shuffle_seed == 0 && n > 0)
            plan_wave(*P, A, band, g_row, g_slice, c_slice, sptr, s_row, chunk_hull, d_srow.p, o->cache_bytes == 0,
                      wave_host, s);
        MPK_CUDA(cudaStreamSynchronize(s));  // host vectors above must outlive their copies
    } catch (...) {
        P->arena.release();
        delete P;
        throw;
    }
    return P;
}

}  // namespace mpk
