// Level builder: CSR validation, the pattern of A + A^T, level-synchronous BFS and the
// BFS permutation (Sec. 3, level definition, prose and Fig. 1).
#include "mpk_internal.h"

#include <algorithm>
#include <climits>

namespace mpk {

// err[0]: bad row pointer, err[1]: column out of range, err[2]: largest |column - row|
__global__ void k_validate(int32_t n, int32_t nnz, const int32_t *rp, const int32_t *ci, int32_t *err) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    int32_t band = 0;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += stride) {
        const int32_t a = rp[i], b = rp[i + 1];
        if (a > b || a < 0 || b > nnz || (i == 0 && a != 0) || (i == n - 1 && b != nnz)) {
            atomicExch(&err[0], 1);
            continue;
        }
        for (int32_t e = a; e < b; ++e) {
            const int32_t c = ci[e];
            if (c < 0 || c >= n) {
                atomicExch(&err[1], 1);
                break;
            }
            band = max(band, abs(c - (int32_t)i));
        }
    }
    band = __reduce_max_sync(0xffffffffu, band);
    if ((threadIdx.x & 31) == 0 && band > err[2]) atomicMax(&err[2], band);
}

void validate_csr(const mpk_csr *A, cudaStream_t s, int32_t *bandwidth) {
    if (bandwidth) *bandwidth = 0;
    if (!A) fail(MPK_ERR_INVALID, "matrix is NULL");
    if (A->n < 0 || A->nnz < 0) fail(MPK_ERR_INVALID, "negative n (%d) or nnz (%d)", A->n, A->nnz);
    if (A->val_type != MPK_F64 && A->val_type != MPK_F32 && A->val_type != MPK_BF16)
        fail(MPK_ERR_UNSUPPORTED, "value type %d (MPK_F64, MPK_F32 or MPK_BF16)", A->val_type);
    if (A->n == 0) return;
    if (!A->row_ptr || (A->nnz > 0 && (!A->col || !A->val)))
        fail(MPK_ERR_INVALID, "NULL CSR array");
    Tmp<int32_t> err(3, s);
    MPK_CUDA(cudaMemsetAsync(err.p, 0, 3 * sizeof(int32_t), s));
    int g = (int)((A->n + 255) / 256);
    if (g > device_sms() * 16) g = device_sms() * 16;
    k_validate<<<g, 256, 0, s>>>(A->n, A->nnz, A->row_ptr, A->col, err.p);
    MPK_LAUNCHED();
    int32_t h[3];
    MPK_CUDA(cudaMemcpyAsync(h, err.p, sizeof(h), cudaMemcpyDeviceToHost, s));
    MPK_CUDA(cudaStreamSynchronize(s));
    if (h[0]) fail(MPK_ERR_INVALID, "row_ptr is not a valid CSR row pointer (0 .. nnz, non-decreasing)");
    if (h[1]) fail(MPK_ERR_INVALID, "column index outside [0, n)");
    if (bandwidth) *bandwidth = h[2];
}

// ----------------------------------------------------------------------------- A^T pattern
__global__ void k_tcount(int32_t n, const int32_t *rp, const int32_t *ci, int32_t *cnt) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += stride)
        for (int32_t e = rp[i]; e < rp[i + 1]; ++e)
            if (ci[e] != i) atomicAdd(&cnt[ci[e]], 1);
}
__global__ void k_tfill(int32_t n, const int32_t *rp, const int32_t *ci, int32_t *pos, int32_t *tci) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += stride)
        for (int32_t e = rp[i]; e < rp[i + 1]; ++e)
            if (ci[e] != i) tci[atomicAdd(&pos[ci[e]], 1)] = (int32_t)i;
}

// ----------------------------------------------------------------------------- BFS on the device
// The whole level-synchronous BFS in one cooperative launch (every block resident): per level the
// blocks expand the frontier queue[head, tail) into level lev + 1 (appending behind it) and meet at a
// grid barrier whose word also carries the number of vertices found so far, so every block advances
// head, tail and lev identically.  A level is bound by its chain of dependent round trips: queue
// entry with its row bounds, columns, levels, claims, one addition to the queue's end per warp
// beside the winners' row bounds, and the barrier's two.  Levels of up to kBfsNarrow vertices are
// expanded by one block alone (256 / 512 / 1024 / 2048: 1500x1300 grid, 2799 levels, 13.6 / 12.6 /
// 14.6 / 18.1 ms).  Against a version that appended neighbour by neighbour and read the count after
// the barrier: 256^3 8.99 -> 7.97 ms, 131x127x113 3.14 -> 2.95 ms, banded 300k 2.70 -> 2.03 ms.
// (Claims without a look at the level first, and prefetches of the winners' columns: slower.)
// A graph whose search runs dry before every vertex is reached continues from the smallest
// untouched vertex, which opens the next level: block 0 looks for it beside the narrow levels
// (20000 vertices without edges: 27 ms; by the grid alone 166 to 187), the grid when it is not among
// the next kBfsNear * kBfsBS (a grid-wide minimum, one barrier, and one more to publish it); the
// minima rotate through three slots, so that a slot is reset only
// after its last readers passed the next barrier.  Every barrier wait is bounded; on expiry the
// kernel records the failure and all blocks leave.
constexpr int64_t kBfsWaitNs = 2000000000LL;  // bound of one grid-barrier wait (2 s)
constexpr int kBfsBS = 512;                   // one block an SM: half the arrivals of two blocks of 256
constexpr int kBfsNarrow = 512;               // vertices of a level that one block expands alone
constexpr int kBfsAlone = 1 << 15;            // levels it expands before it meets the others,
constexpr int kBfsNear = 16;                  // blocks of kBfsBS vertices it looks at for a restart
constexpr int kBfsAloneShare = 8;             // within 1/8 of the others' bound (see k_bfs_all)
struct BfsState {
    unsigned long long bar;  // arrivals at grid barriers, all rounds, << 32 | vertices found, all levels
    int4 left[2];      // where block 0 left the narrow levels: head, tail, level, cursor
    int32_t tail;      // end of the queue
    int32_t minv[3];   // smallest untouched vertex per restart (INT_MAX: none)
    int32_t levels;    // number of levels (written at the end)
    int32_t err;       // 1: a barrier wait expired, 2: the search lost track of untouched vertices
};

__device__ __forceinline__ uint64_t bfs_clock() {
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
// all blocks of the grid, barrier number `round` (counted by the caller, the same in every
// block): the arrivals only grow, and barrier r is passed once r * gridDim.x blocks arrived.
// Thread 0 arrives with an acquire-release add (the block's writes, ordered before it by the
// block barrier, are released; the earlier arrivals acquired) and polls with acquire loads.
// `found`: what this block's threads found since the last barrier (in shared memory; cleared).
// Returns the vertices found by all blocks so far, or -1 when the wait expired (recorded in st->err).
__device__ __forceinline__ int64_t bfs_grid_barrier(BfsState *st, unsigned int round, int *found, int64_t limit_ns) {
    __shared__ int64_t s_all;
    __syncthreads();
    if (threadIdx.x == 0) {
        const unsigned int target = round * gridDim.x;
        const unsigned long long add = (1ULL << 32) | (unsigned int)*found;
        unsigned long long v;
        asm volatile("atom.add.acq_rel.gpu.global.u64 %0, [%1], %2;" : "=l"(v) : "l"(&st->bar), "l"(add) : "memory");
        v += add;
        *found = 0;
        bool ok = true;
        if ((unsigned int)(v >> 32) != target) {
            uint64_t t0 = 0;
            for (int spin = 1;; ++spin) {
                asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(&st->bar) : "memory");
                // (the next round's arrivals cannot come before this block passed this one)
                if ((unsigned int)(v >> 32) >= target) break;
                if ((spin & 63) == 0) {
                    const uint64_t t = bfs_clock();
                    if (t0 == 0) t0 = t;
                    if (t - t0 > (uint64_t)limit_ns) {
                        atomicCAS(&st->err, 0, 1);
                        ok = false;
                        break;
                    }
                }
            }
        }
        s_all = ok ? (int64_t)(v & 0xffffffffULL) : -1;
    }
    __syncthreads();
    return s_all;
}

// Neighbours vi[e0 .. e1) of v (none when e0 == e1) join level `next` unless reached (compare-and-swap
// from -1), eight at a time, by a whole warp: the claims of all lanes, then one addition to the
// queue's end for all that the warp won (its entries: the vertex and its row bounds).  Returns the
// warp's wins.
__device__ __forceinline__ int bfs_visit(const int32_t *rp, const int32_t *vi, int32_t e0, int32_t e1,
                                         int32_t v, int32_t *level_of, int32_t next, int4 *queue, int32_t *tail, int lane) {
    int all = 0;
    const int most = __reduce_max_sync(0xffffffffu, e1 - e0);
    for (int j = 0; j < most; j += 8) {
        int32_t u[8];
        int32_t old[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) u[q] = (e0 + j + q < e1) ? vi[e0 + j + q] : v;
#pragma unroll
        for (int q = 0; q < 8; ++q) old[q] = u[q] != v ? *(volatile int32_t *)&level_of[u[q]] : 0;
#pragma unroll
        for (int q = 0; q < 8; ++q)
            if (old[q] == -1) old[q] = atomicCAS(&level_of[u[q]], -1, next);
        // row bounds of the vertices won, for their queue entries: on their way with the addition below
        int32_t b0[8], b1[8];
        int mine = 0;
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            b0[q] = b1[q] = 0;
            if (old[q] == -1) {
                b0[q] = rp[u[q]];
                b1[q] = rp[u[q] + 1];
                ++mine;
            }
        }
        int end = mine;  // inclusive prefix sum over the warp
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int x = __shfl_up_sync(0xffffffffu, end, o);
            if (lane >= o) end += x;
        }
        const int total = __shfl_sync(0xffffffffu, end, 31);
        if (total == 0) continue;
        int base = 0;
        if (lane == 0) base = atomicAdd(tail, total);
        int at = __shfl_sync(0xffffffffu, base, 0) + end - mine;
#pragma unroll
        for (int q = 0; q < 8; ++q)
            if (old[q] == -1) queue[at++] = make_int4(u[q], b0[q], b1[q], 0);
        all += total;
    }
    return all;
}

__global__ void __launch_bounds__(kBfsBS, 1) k_bfs_all(const int32_t *rp, const int32_t *ci, const int32_t *tp,
                                                    const int32_t *tci, int32_t *level_of, int4 *queue, int32_t n,
                                                    int32_t head0, int32_t tail0, BfsState *st, int64_t limit_ns) {
    __shared__ int s_found, s_root;
    __shared__ int2 s_end;  // end of the queue, and whether the narrow levels end here
    const int64_t gtid = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int64_t gstride = (int64_t)gridDim.x * blockDim.x;
    const int lane = threadIdx.x & 31;
    int64_t head = head0, tail = tail0, cursor = 0, found0 = 0;
    int32_t lev = 0;
    int q = 0;               // restart
    unsigned int round = 0;  // grid barriers passed
    if (threadIdx.x == 0) s_found = 0;
    __syncthreads();
    // the vertices queue[t], t = first, first + step, ... below `last` (whole warps), into level `next`
    auto expand = [&](int64_t first, int64_t step, int64_t last, int32_t next, int32_t *end) -> int {
        int wins = 0;
        for (int64_t t = first; t - lane < last; t += step) {
            const bool on = t < last;
            const int4 e = on ? queue[t] : make_int4(0, 0, 0, 0);
            int32_t f0 = 0, f1 = 0;  // (loaded before the first visit, not after it)
            if (tp && on) {
                f0 = tp[e.x];
                f1 = tp[e.x + 1];
            }
            wins += bfs_visit(rp, ci, e.y, e.z, e.x, level_of, next, queue, end, lane);
            if (tp) {
                wins += bfs_visit(rp, tci, f0, f1, e.x, level_of, next, queue, end, lane);
            }
        }
        return wins;
    };
    for (;;) {
        if (tail > head && tail - head <= kBfsNarrow) {
            // narrow levels: block 0 alone, with block barriers and the queue's end in shared memory,
            // while the others wait at one grid barrier.  A level takes a few us, but one with a long
            // row takes as long as the row's walk (a hub of 500 neighbours: 200 us), so the loop ends
            // by time too: no level starts after limit_ns / 8 cycles (1/8 of the bound at 1 GHz), and the
            // others wait for twice the bound, which leaves the last level the whole of it
            if (blockIdx.x == 0) {
                int32_t h = (int32_t)head, t = (int32_t)tail, l = lev;
                int64_t cur = cursor;  // all vertices below are reached
                const long long c0 = clock64();
                bool late = false;
                for (int it = 0; it < kBfsAlone && !late && t - h <= kBfsNarrow; ++it) {
                    if (t == h) {  // ran dry: the smallest untouched vertex, if it is near
                        if (t >= n) break;
                        if (threadIdx.x == 0) s_root = INT_MAX;
                        bool any = false;
                        for (int c = 0; c < kBfsNear && cur < n && !any; ++c, cur += any ? 0 : kBfsBS) {
                            const int64_t i = cur + threadIdx.x;
                            const bool free = i < n && *(volatile int32_t *)&level_of[i] < 0;
                            any = __syncthreads_or(free);
                            if (free) atomicMin(&s_root, (int)i);
                        }
                        if (!any) break;
                        __syncthreads();
                        cur = s_root;
                        ++l;
                        if (threadIdx.x == 0) {
                            level_of[cur] = l;
                            queue[t] = make_int4((int)cur, rp[cur], rp[cur + 1], 0);
                        }
                        ++t;
                    }
                    if (threadIdx.x == 0) s_end.x = t;
                    __syncthreads();
                    expand(h + threadIdx.x, blockDim.x, t, l + 1, &s_end.x);
                    // (by the last thread, whose warp has the least to do)
                    if (threadIdx.x == kBfsBS - 1) s_end.y = clock64() - c0 > limit_ns / kBfsAloneShare;
                    __syncthreads();
                    h = t;
                    const int2 end = s_end;
                    t = end.x;
                    late = end.y != 0;
                    if (t > h) ++l;
                    __syncthreads();
                }
                if (threadIdx.x == 0) {
                    st->tail = t;
                    st->left[(round + 1) & 1] = make_int4(h, t, l, (int32_t)min(cur, (int64_t)n));
                }
            }
            if (bfs_grid_barrier(st, ++round, &s_found, 2 * limit_ns) < 0) return;
            // (two places in turn: block 0 writes this one again only after the next barrier)
            const volatile int4 *left = &st->left[round & 1];
            head = left->x;
            tail = left->y;
            lev = left->z;
            cursor = left->w;
            continue;
        }
        if (tail > head) {  // expand level lev (st->tail == tail)
            const int wins = expand(head + gtid, gstride, tail, lev + 1, &st->tail);
            if (lane == 0 && wins) atomicAdd(&s_found, wins);
            const int64_t all = bfs_grid_barrier(st, ++round, &s_found, limit_ns);
            if (all < 0) return;
            head = tail;
            tail += all - found0;
            if (all > found0) ++lev;
            found0 = all;
            continue;
        }
        if (tail >= n) break;
        // the search ran dry: the smallest untouched vertex (all below cursor are reached)
        int32_t *mn = &st->minv[q % 3];
        for (int64_t i = cursor + gtid; i < n; i += gstride)
            if (level_of[i] < 0) {
                atomicMin(mn, (int32_t)i);
                break;
            }
        if (gtid == 0) st->minv[(q + 1) % 3] = INT_MAX;
        if (bfs_grid_barrier(st, ++round, &s_found, limit_ns) < 0) return;
        const int32_t v = *(volatile int32_t *)mn;
        ++q;
        if (v == INT_MAX) {
            if (gtid == 0) atomicCAS(&st->err, 0, 2);
            return;
        }
        cursor = v;
        ++lev;
        if (gtid == 0) {
            level_of[v] = lev;
            queue[tail] = make_int4(v, rp[v], rp[v + 1], 0);
            st->tail = (int32_t)tail + 1;
        }
        tail += 1;
        if (bfs_grid_barrier(st, ++round, &s_found, limit_ns) < 0) return;  // the new root before its expansion
    }
    if (gtid == 0) st->levels = lev + 1;
}

__global__ void k_set_root(const int32_t *rp, int32_t *level_of, int4 *queue_slot, int32_t v, int32_t level) {
    level_of[v] = level;
    *queue_slot = make_int4(v, rp[v], rp[v + 1], 0);
}

// level 0 = every root (roots distinct)
__global__ void k_set_roots(const int32_t *rp, int32_t *level_of, int4 *queue, const int32_t *roots, int32_t nroots) {
    for (int32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < nroots; i += gridDim.x * blockDim.x) {
        level_of[roots[i]] = 0;
        queue[i] = make_int4(roots[i], rp[roots[i]], rp[roots[i] + 1], 0);
    }
}

__global__ void k_inverse(const uint32_t *perm, int32_t *iperm, int32_t *perm_out, int64_t n) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; r < n; r += stride) {
        const int32_t old = (int32_t)perm[r];
        iperm[old] = (int32_t)r;
        perm_out[r] = old;
    }
}

// level_ptr from the sorted level keys (levels are 0..L-1 without gaps)
__global__ void k_level_bounds(const uint32_t *sorted_levels, int64_t n, int32_t *level_ptr, int32_t L) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; r < n; r += stride) {
        const int32_t l = (int32_t)sorted_levels[r];
        const int32_t prev = r == 0 ? -1 : (int32_t)sorted_levels[r - 1];
        for (int32_t q = prev + 1; q <= l; ++q) level_ptr[q] = (int32_t)r;
        if (r == n - 1) level_ptr[L] = (int32_t)n;
    }
}

static int grid_n(int64_t n) {
    int64_t g = (n + 255) / 256;
    const int64_t cap = (int64_t)device_sms() * 16;
    if (g > cap) g = cap;
    return (int)(g < 1 ? 1 : g);
}

Levels *build_levels(const mpk_csr *A, int32_t root, cudaStream_t s, const std::vector<int32_t> *roots) {
    validate_csr(A, s);
    const int32_t n = A->n;
    if (roots) {  // level 0 is the whole root set: a BFS distance from the set
        if (n > 0 && roots->empty()) fail(MPK_ERR_INVALID, "empty root set");
        for (size_t i = 0; i < roots->size(); ++i)
            if ((*roots)[i] < 0 || (*roots)[i] >= n || (i > 0 && (*roots)[i] <= (*roots)[i - 1]))
                fail(MPK_ERR_INVALID, "roots must be ascending, distinct and in [0, %d)", n);
    } else if (n > 0 && (root < 0 || root >= n)) {
        fail(MPK_ERR_INVALID, "root %d outside [0, %d)", root, n);
    }
    Levels *L = new Levels();
    try {
        L->n = n;
        L->perm = L->arena.alloc_n<int32_t>(4 * (int64_t)n + 1);  // one block (a large cudaMalloc takes 50 us)
        L->iperm = L->perm + n;
        L->level_of = L->iperm + n;
        L->level_ptr = L->level_of + n;
        if (n == 0) {
            MPK_CUDA(cudaMemsetAsync(L->level_ptr, 0, sizeof(int32_t), s));
            MPK_CUDA(cudaStreamSynchronize(s));
            L->h_level_ptr = {0};
            return L;
        }
        // pattern of A^T without the diagonal, only when A is not declared symmetric
        Tmp<int32_t> tp(A->is_symmetric ? 0 : (int64_t)n + 1, s);
        Tmp<int32_t> tci(A->is_symmetric ? 0 : (int64_t)A->nnz, s);
        if (!A->is_symmetric) {
            Tmp<int32_t> cnt((int64_t)n + 1, s);
            MPK_CUDA(cudaMemsetAsync(cnt.p, 0, sizeof(int32_t) * ((size_t)n + 1), s));
            k_tcount<<<grid_n(n), 256, 0, s>>>(n, A->row_ptr, A->col, cnt.p);
            MPK_LAUNCHED();
            exclusive_scan(cnt.p, tp.p, n, s);
            MPK_CUDA(cudaMemcpyAsync(cnt.p, tp.p, sizeof(int32_t) * (size_t)n, cudaMemcpyDeviceToDevice, s));
            k_tfill<<<grid_n(n), 256, 0, s>>>(n, A->row_ptr, A->col, cnt.p, tci.p);
            MPK_LAUNCHED();
            MPK_CUDA(cudaStreamSynchronize(s));
        }
        // level-synchronous BFS; queue holds the levels back to back
        Tmp<int4> queue(n, s);  // (vertex, its row bounds)
        MPK_CUDA(cudaMemsetAsync(L->level_of, 0xff, sizeof(int32_t) * (size_t)n, s));
        int64_t head = 0, tail = 1;
        if (roots) {
            const int32_t nr = (int32_t)roots->size();
            Tmp<int32_t> d_roots(nr, s);
            MPK_CUDA(cudaMemcpyAsync(d_roots.p, roots->data(), sizeof(int32_t) * (size_t)nr, cudaMemcpyHostToDevice, s));
            k_set_roots<<<grid_n(nr), 256, 0, s>>>(A->row_ptr, L->level_of, queue.p, d_roots.p, nr);
            MPK_LAUNCHED();
            MPK_CUDA(cudaStreamSynchronize(s));  // the host root list and d_roots go out of scope
            tail = nr;
        } else {
            k_set_root<<<1, 1, 0, s>>>(A->row_ptr, L->level_of, queue.p, root, 0);
            MPK_LAUNCHED();
        }
        // the levels, in one cooperative launch (every block resident)
        Tmp<BfsState> st(1, s);
        const BfsState st0{0, {}, (int32_t)tail, {INT_MAX, INT_MAX, INT_MAX}, 0, 0};
        MPK_CUDA(cudaMemcpyAsync(st.p, &st0, sizeof(BfsState), cudaMemcpyHostToDevice, s));
        int per_sm = 0;
        MPK_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_bfs_all, kBfsBS, 0));
        if (per_sm < 1) fail(MPK_ERR_CUDA, "the BFS kernel does not fit an SM");
        const int grid = device_sms();
        const int32_t *rpp = A->row_ptr, *cip = A->col;
        const int32_t *tpp = A->is_symmetric ? nullptr : tp.p;
        const int32_t *tcip = tci.p;
        int32_t *lvl = L->level_of;
        int4 *qp = queue.p;
        int32_t nn = n, h0 = (int32_t)head, t0 = (int32_t)tail;
        BfsState *stp = st.p;
        int64_t limit = kBfsWaitNs;
        void *args[] = {(void *)&rpp, (void *)&cip, (void *)&tpp, (void *)&tcip, (void *)&lvl, (void *)&qp,
                        (void *)&nn, (void *)&h0, (void *)&t0, (void *)&stp, (void *)&limit};
        MPK_CUDA(cudaLaunchCooperativeKernel((const void *)k_bfs_all, dim3(grid), dim3(kBfsBS), args, 0, s));
        MPK_LAUNCHED();
        BfsState hs;
        MPK_CUDA(cudaMemcpyAsync(&hs, st.p, sizeof(BfsState), cudaMemcpyDeviceToHost, s));
        MPK_CUDA(cudaStreamSynchronize(s));
        if (hs.err == 1) fail(MPK_ERR_TIMEOUT, "BFS: a grid barrier wait expired");
        if (hs.err != 0) fail(MPK_ERR_CUDA, "BFS lost track of unvisited vertices");
        const int32_t lev = hs.levels - 1;
        const int32_t nl = lev + 1;
        L->num_levels = nl;
        // permutation: stable sort of (level, id) pairs with ids ascending as input order
        Tmp<uint32_t> k0(n, s), v0(n, s), k1(n, s), v1(n, s);
        MPK_CUDA(cudaMemcpyAsync(k0.p, L->level_of, sizeof(int32_t) * (size_t)n, cudaMemcpyDeviceToDevice, s));
        iota_i32(reinterpret_cast<int32_t *>(v0.p), n, s);
        int bits = 0;
        while (bits < 32 && ((int64_t)1 << bits) < nl) ++bits;
        uint32_t *ks = nullptr, *vs = nullptr;
        radix_sort_pairs(k0.p, v0.p, k1.p, v1.p, n, bits, s, &ks, &vs);
        k_inverse<<<grid_n(n), 256, 0, s>>>(vs, L->iperm, L->perm, n);
        MPK_LAUNCHED();
        k_level_bounds<<<grid_n(n), 256, 0, s>>>(ks, n, L->level_ptr, nl);
        MPK_LAUNCHED();
        L->h_level_ptr.resize((size_t)nl + 1);
        MPK_CUDA(cudaMemcpyAsync(L->h_level_ptr.data(), L->level_ptr, sizeof(int32_t) * ((size_t)nl + 1),
                                 cudaMemcpyDeviceToHost, s));
        MPK_CUDA(cudaStreamSynchronize(s));
    } catch (...) {
        L->arena.release();
        delete L;
        throw;
    }
    return L;
}

}  // namespace mpk
