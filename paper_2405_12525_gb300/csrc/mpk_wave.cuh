// The wave kernel: level-blocked powers on a static schedule (device code; instantiated per
// value type in mpk_wave_f64.cu, mpk_wave_f32.cu and mpk_wave_bf16.cu, for packed copies in
// mpk_wave_dict.cu).
#pragma once
#include "mpk_kernel_dev.cuh"

namespace mpk {

// What bounds it.  An FP64 FMA holds an SM quarter's pipe for 67 cycles (0.594 T FMA/s measured on
// all SMs), so 256^3, p = 8 needs 1.58 ms of it; k_mpk's units (claimed through a ticket, handed
// over block-wide, 8 FMA slots for a row of 7 entries) took 2.08 ms.  Here nothing is claimed and
// nothing handed over block-wide, a row takes exactly its slice's width of FMAs, and 28 warps
// work on as many slices: 2.03 ms, and 1.84 ms with packed copies (below); binary32 sums, bound by
// instruction issue and the latency of the gathers: 1.45 -> 1.37 ms.  Blocks of right-hand sides,
// where k_mpk's gathers of one column at a time made L1 the bound: 100^3 27-point stencil, 8
// columns, p = 8: 4.21 -> 2.90 ms.  What is left above the FMAs is the cells' hand-over (blocks
// that wait for the slowest one) and slices that wait for their copies.
//
// Packed copies (VT = ValDict; matrices of at most 256 different values, one right-hand side): a
// slice is one stream of 16-byte units, per entry the smallest column among the 32 rows, then 32
// column distances of 16 bits (32-bit columns in a slice where they do not fit), then 32 value
// numbers of 8 bits, whose values lie in a table in shared memory.  About 3.2 bytes an entry in
// place of 12, so the buffer holds three times the slices, the copies run further ahead, and a cell
// of the same bytes has more rows; the FMAs and their operands are the same.  27-point stencil
// on 150^3, p = 8: 1.91 -> 1.31 ms.
//
// One cooperative launch, one block per SM.  The Lp-diagram cells (group g, power k) are walked
// in line order, as k_mpk does; every cell's 32-row slices are divided evenly over the blocks,
// so nothing is claimed at run time and a slice is the unit of work: a compute warp waits for
// nothing but its own entries and the cell's dependencies.
//
// Warp roles of a block:
//  - warp 0 (dispatcher) lists the block's slices of every cell in schedule order in a ring of
//    descriptors in shared memory, 32 a step;
//  - warp 1 (loader) copies the entries of the listed slices into a circular buffer in shared
//    memory, a tile of up to 32 slices on one mbarrier, with one pair of bulk copies per run of
//    neighbouring slices.  The copies need no dependency and run ahead of the cells by the
//    buffer's size;
//  - warp 2 (poller) reads the completion counters of the cells that the next 32 cells depend on
//    and stores how many cells may run in s_ready;
//  - warp 3 (publisher) sees from the warps' progress words which cells the block has finished,
//    issues one fence at GPU scope for all of them and adds the block's slices to the cells'
//    counters;
//  - the others compute.  A lane owns one (row, right-hand side) pair, so a slice is M units of
//    32 / M rows, and warp w takes the units w, w + W, ...: it waits for the slice's tile and
//    cell, gathers x and runs the row sums.
// A cell (g, k) is ready when the cells (g-1 .. g+1, k-1) are complete: groups are whole levels,
// and a row reads its own level and the two beside it.  The same wait covers what the cell
// overwrites in the rings of the recurrence (three blocks) and of the binary32 copy (two).
//
// With lanes along the right-hand sides a gather reads whole rows of x (8 M consecutive bytes)
// instead of one column of 32 rows, which would touch 32 lines an instruction and make L1 the
// bound from M = 4 on.
//
// Deadlock freedom: every block is resident (cooperative launch); cells are dispatched, polled,
// computed and published in one order, and a cell depends on earlier cells only, so the first
// unfinished cell can always run.  Every wait is bounded by a.wait_ns (globaltimer); on expiry
// the launch's epoch and MPK_ERR_TIMEOUT are recorded in a.err, all blocks leave, and no block
// leaves with a bulk copy of its own in flight.
//
// The counters start at zero: the last block whose poller and publisher are done (nothing is
// polled or published after that) clears them for the next launch, and stores the epoch, while
// the compute warps still finish the last power, whose cells nothing waits for.
constexpr int kWaveAux = 4;     // dispatcher, loader, poller, publisher
constexpr int kWaveWarps = 28;  // compute warps: 16 / 20 / 24 / 28 took 2.34 / 2.15 / 2.03 / 1.99 ms at 256^3, p = 8
constexpr int kWaveBS = 32 * (kWaveWarps + kWaveAux);
constexpr int kDescRing = 512;  // slice descriptors in shared memory
constexpr int kWaveTiles = 32;  // tiles in shared memory or in flight
constexpr int kStagedWidth = 64;  // entries a row of the widest slice that the buffer takes
// The circular buffer: its bytes, and its entries `cap`, of which the widest slice it takes (a wider
// one is read from global memory) and a tile are parts.  A slice that starts near the end of the
// buffer runs on past it, into room for one slice.
//
// 200 KB let the copies run furthest ahead (96 KB: structured binary64 grids the same, others 5 to
// 30 % slower), but leave 28 KB of L1, in whose lines the gathers in flight wait for L2.  Gathers that
// touch a line a row then queue for lines: with 96 KB a grid of 126^3 with its rows shuffled, p = 8, plan
// order, takes 381 in place of 839 us (binary64), 407 in place of 714 us (bfloat16; the ticketed kernel,
// whose blocks stage less: 417).  A set of tables says which of the two its gathers need (WaveSet::scattered).
constexpr int kWaveBytes = 200 * 1024, kWaveBytesScattered = 96 * 1024;
template <class VT> struct WaveBuf {
    static constexpr int ENTRY = (int)sizeof(typename VT::T) + 4;
    static constexpr int SLICE = 32 * kStagedWidth;
    static constexpr int CAP = (kWaveBytes / ENTRY - SLICE) / 256 * 256;
    static constexpr int CAP_SCATTERED = (kWaveBytesScattered / ENTRY - SLICE) / 256 * 256;
    static_assert(CAP_SCATTERED / 3 >= SLICE, "a slice fits a tile");
};

// packed slices: positions and sizes count 16-byte units
struct ValDict {
    using T = uint8_t;
};
template <> struct WaveBuf<ValDict> {
    static constexpr int ENTRY = 16;
    static constexpr int SLICE = (kStagedWidth + 3) / 4 + 10 * kStagedWidth;
    static constexpr int CAP = (kWaveBytes / ENTRY - SLICE) / 16 * 16;
    static constexpr int CAP_SCATTERED = (kWaveBytesScattered / ENTRY - SLICE) / 16 * 16;
    static_assert(CAP_SCATTERED / 3 >= SLICE, "a slice fits a tile");
};

struct __align__(16) WaveDesc {
    int32_t e32;    // first entry of the slice / 32 (packed: its place in the stream, units)
    int32_t width;  // entries a row; top bit: first of a run of neighbouring slices; packed: next bit: wide
    int32_t row0;   // first row, or the slice's first entry of the row map
    uint32_t ckr;   // cell << 11 | power << 6 | rows
};

__device__ __forceinline__ int ld_acquire_cta_shared(const int *p) {
    int v;
    asm volatile("ld.acquire.cta.shared.b32 %0, [%1];" : "=r"(v) : "r"(smem_u32(p)) : "memory");
    return v;
}
__device__ __forceinline__ void st_release_cta_shared(int *p, int v) {
    asm volatile("st.release.cta.shared.b32 [%0], %1;" ::"r"(smem_u32(p)), "r"(v) : "memory");
}

// Bound of a wait, for use in its spin loop only: the first call starts the clock, and the clock
// (slow to read) is looked at every 64 calls.
struct Deadline {
    uint64_t t0 = 0;
    int calls = 0;
    __device__ __forceinline__ bool expired(int64_t limit_ns) {
        if (calls++ & 63) return false;
        const uint64_t t = globaltimer();
        if (t0 == 0) t0 = t;
        return t - t0 > (uint64_t)limit_ns;
    }
};

// the block's share of a cell of nsl slices: [x, y)
__device__ __forceinline__ int2 wave_share(int nsl, int block, int blocks) {
    return make_int2((int)((int64_t)nsl * block / blocks), (int)((int64_t)nsl * (block + 1) / blocks));
}

// The body of the kernel.  BATCH (powers of a batch plan): the vectors of the instances lie apart, at
// the places in `inst`.
template <int M, int MODE, class VT, bool A32, bool BATCH>
__device__ __forceinline__ void wave_body(const KArgs &a, const WaveBatch *inst) {
    using AT = typename std::conditional<A32, float, double>::type;
    using T = typename VT::T;
    constexpr bool PACK = std::is_same<VT, ValDict>::value;
    // a slice's entries a row and its size in the buffer, from the width field of its record
    auto width_of = [](int f) { return PACK ? f & (kWideSlice - 1) : f & 0x7fffffff; };
    auto size_of = [&](int f) { return PACK ? packed_units(width_of(f), (f & kWideSlice) != 0) : 32 * width_of(f); };
    constexpr int G = 32 / M;  // rows of a unit
    using Buf = WaveBuf<VT>;
    const uint32_t cap = (uint32_t)a.v_cap;  // entries of the buffer
    extern __shared__ __align__(128) unsigned char smem[];  // values, then columns
    T *const sval = reinterpret_cast<T *>(smem);
    int32_t *const scol = reinterpret_cast<int32_t *>(smem + (cap + Buf::SLICE) * sizeof(T));  // (packed: unused)
    __shared__ AT s_dict[PACK ? kDictSize : 1];
    if constexpr (PACK)
        for (int i = threadIdx.x; i < kDictSize; i += kWaveBS) s_dict[i] = (AT)a.v_dict[i];  // exact
    __shared__ WaveDesc desc[kDescRing];
    __shared__ uint8_t dinst[BATCH ? kDescRing : 1];  // instance of each descriptor
    __shared__ uint32_t vpos[kDescRing];  // entries of the buffer's slices before this one, all in all
    __shared__ int loc[kDescRing];  // where a slice's entries are: offset / 32, tile << 16, phase << 24; -1: global memory
    __shared__ __align__(8) uint64_t full[kWaveTiles];
    __shared__ int s_ready, s_pushed, s_loaded, s_total, s_abort, s_left;
    __shared__ int s_done;  // descriptors finished, as the loader last saw it: those before it may be overwritten
    __shared__ int s_prog[32];  // units finished by each compute warp
    __shared__ int32_t s_epoch;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int block = blockIdx.x, blocks = gridDim.x;
    if (tid < 32) s_prog[tid] = 0;
    if (tid == 0) {
        s_epoch = (int32_t)ld_relaxed(reinterpret_cast<const int32_t *>(a.epoch_word)) + 1;
        s_ready = 0;
        s_pushed = 0;
        s_loaded = 0;
        s_done = 0;
        s_total = -1;
        s_abort = 0;
        s_left = 0;
        for (int q = 0; q < kWaveTiles; ++q) mbar_init(&full[q], 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    const int32_t epoch = s_epoch;
    const int4 *cells = a.v_cell;  // (first slice, slices, g << 5 | k, instance << 2 | neighbours: 1 before, 2 after)
    const int ncells = a.v_ncells;

    auto give_up = [&]() {  // a wait expired: tell this block and the others
        if (atomicExch(a.err, epoch) != epoch) st_relaxed(a.err + 1, (int)MPK_ERR_TIMEOUT);
        *(volatile int *)&s_abort = 1;
    };
    auto aborted = [&]() -> bool { return *(volatile int *)&s_abort != 0; };
    // smallest descriptor that is not finished (every lane of an auxiliary warp)
    auto frontier = [&]() -> int {
        const int v = lane < kWaveWarps ? ld_acquire_cta_shared(&s_prog[lane]) * kWaveWarps + lane : INT_MAX;
        return __reduce_min_sync(0xffffffffu, v) / M;
    };

    if (warp == 0) {
        // ------------------------------------------------------------------ dispatcher
        int pushed = 0, room = kDescRing;  // descriptors below `room` may be written
        uint32_t vnext = 0;
        bool stop = false;
        for (int c0 = 0; c0 < ncells && !stop; c0 += 32) {
            const int4 ce = c0 + lane < ncells ? __ldg(cells + c0 + lane) : make_int4(0, 0, 0, 0);
            const int2 sh = wave_share(ce.y, block, blocks);
            int end = sh.y - sh.x;  // inclusive prefix sum over the 32 cells
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int v = __shfl_up_sync(0xffffffffu, end, o);
                if (lane >= o) end += v;
            }
            const int total = __shfl_sync(0xffffffffu, end, 31);
            for (int t0 = 0; t0 < total && !stop; t0 += 32) {
                const int t = t0 + lane;
                int q = 0;  // the cell of item t: the number of cells that end at or before it
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) {
                    const int v = __shfl_sync(0xffffffffu, end, q + o - 1);
                    if (v <= t) q += o;
                }
                const int qc = min(q, 31);
                const int first = __shfl_sync(0xffffffffu, ce.x + sh.x, qc);
                const int csize = __shfl_sync(0xffffffffu, sh.y - sh.x, qc);
                const int qend = __shfl_sync(0xffffffffu, end, qc);
                const int gk = __shfl_sync(0xffffffffu, ce.z, qc);
                const int ci = BATCH ? __shfl_sync(0xffffffffu, ce.w, qc) >> 2 : 0;
                WaveDesc d{0, 0, 0, 0};
                if (t < total) {
                    const int4 rec = __ldg(a.v_slice + first + (t - (qend - csize)));
                    d.e32 = rec.x;
                    d.width = rec.y;
                    d.row0 = rec.z;
                    d.ckr = (uint32_t)(c0 + qc) << 11 | (uint32_t)(gk & 31) << 6 | (uint32_t)rec.w;
                }
                const int cnt = min(32, total - t0);
                // where the entries go, and where runs start: at a cell's first slice and after a slice
                // that is not copied (and, for the loader, where the buffer starts over)
                const int size = width_of(d.width) <= kStagedWidth ? size_of(d.width) : 0;
                uint32_t vp = (uint32_t)size;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const uint32_t v = __shfl_up_sync(0xffffffffu, vp, o);
                    if (lane >= o) vp += v;
                }
                const uint32_t vend = vnext + __shfl_sync(0xffffffffu, vp, 31);
                vp += vnext - (uint32_t)size;
                vnext = vend;
                const int psize = __shfl_up_sync(0xffffffffu, size, 1);
                if (lane == 0 || t == qend - csize || psize == 0)
                    d.width |= (int)0x80000000;
                if (pushed + cnt > room) {
                    Deadline w0;
                    for (;;) {
                        room = __shfl_sync(0xffffffffu, ld_acquire_cta_shared(&s_done), 0) + kDescRing;
                        __syncwarp();
                        if (pushed + cnt <= room) break;
                        const bool late = aborted() || w0.expired(2 * a.wait_ns + 100000000LL);
                        if (__any_sync(0xffffffffu, late)) {
                            if (lane == 0) give_up();
                            stop = true;
                            break;
                        }
                        __nanosleep(100);
                    }
                    if (stop) break;
                }
                if (lane < cnt) {
                    desc[(pushed + lane) & (kDescRing - 1)] = d;
                    if constexpr (BATCH) dinst[(pushed + lane) & (kDescRing - 1)] = (uint8_t)ci;
                    vpos[(pushed + lane) & (kDescRing - 1)] = vp;
                }
                pushed += cnt;
                __syncwarp();
                if (lane == 0) st_release_cta_shared(&s_pushed, pushed);
            }
        }
        if (lane == 0) st_release_cta_shared(&s_total, pushed);
    } else if (warp == 1) {
        // ------------------------------------------------------------------ loader
        int next = 0, tile = 0, old = 0;  // next descriptor, next tile, oldest tile in use
        uint32_t tail = 0;                // position of the oldest slice in use
        uint32_t turn = 0;                // position at which the buffer last started over, before `next`
        const uint32_t tile_cap = cap / 3;
        int t_desc = 0;                   // descriptors before the end of the tile with number lane (mod 32)
        Deadline w0;
        bool stop = false;
        while (!stop) {
            // descriptors finished; the dispatcher may overwrite those before (not this one: its
            // position is read below)
            int done = frontier();
            if (lane == 0) st_release_cta_shared(&s_done, done);
            const int total_desc = ld_acquire_cta_shared(&s_total);  // before s_pushed: it is final then
            const int have = __shfl_sync(0xffffffffu, ld_acquire_cta_shared(&s_pushed), 0) - next;
            if (have <= 0) {
                if (__any_sync(0xffffffffu, total_desc >= 0 || aborted())) {
                    if (__any_sync(0xffffffffu, aborted())) break;
                    if (__shfl_sync(0xffffffffu, ld_acquire_cta_shared(&s_pushed), 0) <= next) break;
                    continue;
                }
                if (__any_sync(0xffffffffu, w0.expired(2 * a.wait_ns + 200000000LL))) {
                    if (lane == 0) give_up();
                    break;
                }
                __nanosleep(50);
                continue;
            }
            __syncwarp();
            WaveDesc d{0, 0, 0, 0};
            uint32_t vp = 0;
            if (lane < have) {
                d = desc[(next + lane) & (kDescRing - 1)];
                vp = vpos[(next + lane) & (kDescRing - 1)];
            }
            const bool staged = width_of(d.width) <= kStagedWidth;
            const uint32_t ve = vp + (staged ? (uint32_t)size_of(d.width) : 0u);
            const uint32_t v0 = __shfl_sync(0xffffffffu, vp, 0);
            const unsigned int over = __ballot_sync(0xffffffffu, lane >= have || ve - v0 > tile_cap);
            const int cnt = over ? __ffs(over) - 1 : 32;  // at least 1: a slice fits a tile
            const uint32_t vend = __shfl_sync(0xffffffffu, ve, cnt - 1);
            while (vend - tail > cap || tile - old >= kWaveTiles) {  // room, and a free tile
                done = frontier();
                if (lane == 0) st_release_cta_shared(&s_done, done);
                while (old < tile && __shfl_sync(0xffffffffu, t_desc, old & 31) <= done) ++old;
                tail = done >= next ? v0 : vpos[done & (kDescRing - 1)];
                if (vend - tail <= cap && tile - old < kWaveTiles) break;
                if (__any_sync(0xffffffffu, aborted() || w0.expired(2 * a.wait_ns + 200000000LL))) {
                    if (lane == 0) give_up();
                    stop = true;
                    break;
                }
            }
            if (stop) break;
            const int b = tile & (kWaveTiles - 1);
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // every lane that copies
            if (lane == 0) mbar_expect_tx(&full[b], (vend - v0) * (uint32_t)Buf::ENTRY);
            __syncwarp();
            // (a tile is a third of the buffer at most: it starts over once at most inside it)
            const bool over_end = vp - turn >= cap;
            const bool before = __shfl_up_sync(0xffffffffu, over_end, 1);
            const uint32_t o = vp - turn - (over_end ? cap : 0u);
            if (vend - turn >= cap) turn += cap;
            if (lane < cnt)
                loc[(next + lane) & (kDescRing - 1)] =
                    staged ? (int)(PACK ? o : o >> 5) | b << 16 | ((tile / kWaveTiles) & 1) << 24 : -1;
            // a run of neighbouring slices: one pair of copies, by the run's first lane
            const bool head = lane < cnt && staged && (lane == 0 || d.width < 0 || over_end != before);
            const unsigned int heads = __ballot_sync(0xffffffffu, head || lane >= cnt || !staged);
            const unsigned int after = lane == 31 ? 0u : heads & (0xfffffffeu << lane);
            const uint32_t run = __shfl_sync(0xffffffffu, ve, after ? __ffs(after) - 2 : 31) - vp;
            if (head && run > 0) {
                // the launch's last power is the last use of the entries (see k_mpk)
                const bool last_use = a.stream_last && ((d.ckr >> 6) & 31u) == (uint32_t)a.p_launch;
                if constexpr (PACK) {
                    bulk_g2s(smem + 16 * o, static_cast<const uint8_t *>(a.v_val) + 16 * (int64_t)d.e32, run * 16u, &full[b],
                             last_use);
                } else {
                    bulk_g2s(sval + o, static_cast<const T *>(a.v_val) + 32 * (int64_t)d.e32, run * (uint32_t)sizeof(T),
                             &full[b], last_use);
                    bulk_g2s(scol + o, a.v_col + 32 * (int64_t)d.e32, run * 4u, &full[b], last_use);
                }
            }
            next += cnt;
            if (lane == b) t_desc = next;
            ++tile;
            __syncwarp();
            if (lane == 0) st_release_cta_shared(&s_loaded, next);
            w0 = Deadline();
        }
        // the copies in flight land before the warp leaves, whatever the compute warps do
        for (int q = old; q < tile; ++q) {
            Deadline w1;
            while (!mbar_try_wait(&full[q & (kWaveTiles - 1)], (q / kWaveTiles) & 1))
                if (w1.expired(a.wait_ns)) break;
        }
    } else if (warp < kWaveAux) {
        if (warp == 2) {
            // -------------------------------------------------------------- poller
            const int ng = a.v_ngroups;
            bool stop = false;
            for (int c0 = 0; c0 < ncells && !stop; c0 += 32) {
                const int4 ce = c0 + lane < ncells ? __ldg(cells + c0 + lane) : make_int4(0, 0, 0, 0);
                const int k = ce.z & 31, g = ce.z >> 5;
                const int32_t *cnt = a.v_count + (int64_t)(k - 1) * ng;
                int need[3];
                bool ok = k <= 1;
#pragma unroll
                for (int q = 0; q < 3; ++q) {
                    // the group itself, and its neighbours inside the instance
                    need[q] = !ok && (q == 1 || (ce.w & (q == 0 ? 1 : 2))) ? __ldg(a.v_gsl + g - 1 + q) : 0;
                }
                int known = 0;  // leading cells of the 32 already announced
                Deadline w0;
                while (known < 32) {
                    const int err = ld_relaxed(a.err);
                    if (!ok) {
                        int got[3];
#pragma unroll
                        for (int q = 0; q < 3; ++q) got[q] = need[q] > 0 ? (ng == 1 ? ld_acquire(cnt + g - 1 + q) : ld_relaxed(cnt + g - 1 + q)) : 0;
                        ok = got[0] >= need[0] && got[1] >= need[1] && got[2] >= need[2];
                    }
                    const unsigned int m = __ballot_sync(0xffffffffu, ok);
                    const int run = m == 0xffffffffu ? 32 : __ffs(~m) - 1;
                    if (run > known) {
                        // The counted rows before this block's reads of them.  With one group the loads
                        // above acquire (a fence after them would add 900 cycles to every power; L1
                        // holds nothing worth keeping while the block waits); with many they would
                        // empty L1 at every poll, and one fence serves all that became ready.
                        if (ng > 1) fence_acq_rel_gpu();
                        __syncwarp();
                        if (lane == 0) st_release_cta_shared(&s_ready, c0 + run);
                        known = run;
                        w0 = Deadline();
                        continue;
                    }
                    const bool late = err == epoch || aborted() || w0.expired(a.wait_ns);
                    if (__any_sync(0xffffffffu, late)) {
                        if (lane == 0) give_up();
                        stop = true;
                        break;
                    }
                }
            }
        } else {
            // -------------------------------------------------------------- publisher
            int base = 0;  // descriptors of the cells before the 32 at hand
            bool stop = false;
            for (int c0 = 0; c0 < ncells && !stop; c0 += 32) {
                const int4 ce = c0 + lane < ncells ? __ldg(cells + c0 + lane) : make_int4(0, 0, 0, 0);
                const int2 sh = wave_share(ce.y, block, blocks);
                const int size = sh.y - sh.x, k = ce.z & 31;
                int end = size;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int v = __shfl_up_sync(0xffffffffu, end, o);
                    if (lane >= o) end += v;
                }
                const int total = __shfl_sync(0xffffffffu, end, 31);
                end += base;
                base += total;
                // (nothing waits for the last power)
                bool todo = size > 0 && k < a.p_launch && ce.z != a.v_drop;
                Deadline w0;
                for (;;) {
                    const unsigned int left = __ballot_sync(0xffffffffu, todo);
                    if (left == 0) break;
                    const int done = frontier();
                    const bool now = todo && end <= done;
                    if (__any_sync(0xffffffffu, now)) {
                        __syncwarp();         // every lane's view of the progress words
                        fence_acq_rel_gpu();  // acquires the finished slices' rows, releases them
                        if (now)
                            atomicAdd(a.v_count + (int64_t)k * a.v_ngroups + (ce.z >> 5), size);
                        todo = todo && !now;
                        w0 = Deadline();
                        continue;
                    }
                    const bool late = aborted() || w0.expired(2 * a.wait_ns + 100000000LL);
                    if (__any_sync(0xffffffffu, late)) {
                        if (lane == 0) give_up();
                        stop = true;
                        break;
                    }
                    __nanosleep(32);
                }
            }
        }
        // both done: this block neither polls nor publishes any more
        __syncwarp();
        int last = 0;
        if (lane == 0) {
            __threadfence();
            if (atomicAdd(&s_left, 1) == 1) {
                __threadfence();
                last = atomicAdd(a.exit_count, 1u) == (unsigned int)blocks - 1;
            }
        }
        if (__shfl_sync(0xffffffffu, last, 0)) {
            __threadfence();
            for (int64_t i = lane; i < (int64_t)a.p_launch * a.v_ngroups; i += 32) a.v_count[a.v_ngroups + i] = 0;
            if (lane == 0) {
                *a.exit_count = 0u;
                *a.epoch_word = (unsigned int)epoch;
            }
            __threadfence();
        }
    } else {
        // ------------------------------------------------------------------ compute warps
        const int w = warp - kWaveAux;
        int done = 0, ready = 0, seen = 0;
        for (int unit = w;; unit += kWaveWarps) {
            const int idx = unit / M, q = unit % M;
            if (idx >= seen) {  // wait for the descriptor, or the end
                Deadline w0;
                bool none = false;
                for (;;) {
                    const int total = ld_acquire_cta_shared(&s_total);
                    seen = ld_acquire_cta_shared(&s_loaded);
                    if (idx < seen) break;
                    if ((total >= 0 && idx >= total) || aborted() || w0.expired(2 * a.wait_ns + 300000000LL)) {
                        none = true;
                        break;
                    }
                    __nanosleep(20);
                }
                if (__any_sync(0xffffffffu, none)) break;
                seen = __shfl_sync(0xffffffffu, seen, 0);
                __syncwarp();  // lane 0's acquire, for every lane while `seen` holds
            }
            WaveDesc d = desc[idx & (kDescRing - 1)];
            const bool wide = PACK && (d.width & kWideSlice) != 0;
            d.width = width_of(d.width);
            const int lc = loc[idx & (kDescRing - 1)];
            const int cell = (int)(d.ckr >> 11), k = (int)(d.ckr >> 6) & 31, rows = (int)(d.ckr & 63u);
            if (cell >= ready) {  // the cell's dependencies
                Deadline w0;
                bool none = false;
                for (;;) {
                    ready = ld_acquire_cta_shared(&s_ready);
                    if (cell < ready) break;
                    if (aborted() || w0.expired(2 * a.wait_ns + 100000000LL)) {
                        none = true;
                        break;
                    }
                }
                if (__any_sync(0xffffffffu, none)) break;
                ready = __shfl_sync(0xffffffffu, ready, 0);
                __syncwarp();  // lane 0's acquire, for every lane while `ready` holds
            }
            if (lc >= 0) {  // the slice's tile
                uint64_t *const bar = &full[(lc >> 16) & 31];
                const uint32_t phase = (uint32_t)lc >> 24;
                if (!mbar_try_wait(bar, phase)) {
                    Deadline w0;
                    while (!mbar_try_wait(bar, phase))
                        if (w0.expired(a.wait_ns)) break;
                    if (!__all_sync(0xffffffffu, mbar_try_wait(bar, phase))) {
                        if (lane == 0) give_up();
                        break;
                    }
                }
            }
            if (q * G < rows) {
                const int rl = q * G + lane / M;
                const bool valid = rl < rows;
                // rows in order, or the row map's (slices of rows sorted by length)
                const int64_t row = a.v_rowmap ? (valid ? __ldg(a.v_rowmap + d.row0 + rl) : 0) : d.row0 + rl;
                // calls f(values, columns) with the slice's entries, wherever they are
                auto entries = [&](auto f) {
                    if constexpr (PACK) {
                        auto at = [&](const uint8_t *p) {
                            const int32_t *first = reinterpret_cast<const int32_t *>(p);
                            const uint8_t *c = p + 16 * ((d.width + 3) / 4);
                            const DictVal<AT> v{c + (wide ? 128 : 64) * (int64_t)d.width, s_dict};
                            if (wide)
                                f(v, SCol{reinterpret_cast<const int32_t *>(c)});
                            else
                                f(v, NearCol{reinterpret_cast<const uint16_t *>(c), first});
                        };
                        if (lc >= 0)
                            at(smem + 16 * (lc & 0xffff));
                        else
                            at(static_cast<const uint8_t *>(a.v_val) + 16 * (int64_t)d.e32);
                    } else if (lc >= 0) {
                        const int o = 32 * (lc & 0xffff);
                        f(SVal<VT, AT>{sval + o}, SCol{scol + o});
                    } else {  // a slice wider than the buffer takes: entries from global memory
                        const int64_t e = 32 * (int64_t)d.e32;
                        f(GVal<VT, AT>{static_cast<const T *>(a.v_val) + e}, GCol{a.v_col + e});
                    }
                };
                if constexpr (BATCH) {
                    // the instance's vectors, addressed by rows of the whole batch
                    const WaveInst in = inst->at[dinst[idx & (kDescRing - 1)]];
                    const int64_t at = row * M + lane % M;
                    double *const y = in.y + (k * in.rows - in.row0) * M;
                    const double *const x = (k == 1 ? in.x - in.row0 * M : y - in.rows * M) + lane % M;
                    // where the plan's workspace has the row
                    const int64_t aw = (a.v_iperm && valid ? __ldg(a.v_iperm + row) : row) * M + lane % M;
                    double own = 0.0, acc = 0.0;
                    if (k == 1 && valid) own = in.x[at - in.row0 * M];
                    entries([&](auto sv, auto sc) {
                        sv.lane(rl);
                        sc.lane(rl);
                        acc = unit_sum<M, double>(sv, sc, d.width, x);
                    });
                    if (valid) {
                        y[at] = acc;
                        __stcs(a.ybase + k * a.ystride + aw, acc);
                        if (k == 1) {
                            if (in.y != in.x) in.y[at - in.row0 * M] = own;
                            __stcs(a.ybase + aw, own);
                        }
                    }
                } else {
                    const double *xin = input_block<M>(a, k);
                    const AT *xacc = InputAcc<M, AT>::get(a, k);
                    entries([&](auto sv, auto sc) {
                        unit_row<M, MODE, AT>(a, k, sv, sc, d.width, rl, row, valid, xin, xacc, lane);
                    });
                }
            }
            __syncwarp();
            ++done;
            if (lane == 0) st_release_cta_shared(&s_prog[w], done);
        }
    }
}

template <int M, int MODE, class VT, bool A32>
__global__ void __launch_bounds__(kWaveBS, 1) k_wave(const __grid_constant__ KArgs a) {
    wave_body<M, MODE, VT, A32, false>(a, nullptr);
}
template <int M, class VT>
__global__ void __launch_bounds__(kWaveBS, 1) k_wave_batch(const __grid_constant__ KArgs a,
                                                           const __grid_constant__ WaveBatch inst) {
    wave_body<M, MODE_POWERS, VT, false, true>(a, &inst);
}

template <class VT, int M> static void *wave_fn(int mode, bool a32) {
    if constexpr (!std::is_same<VT, ValDict>::value)  // (batch plans have no packed copies)
        if (mode == kWaveBatchMode) return (void *)k_wave_batch<M, VT>;
    if constexpr (!std::is_same<VT, ValF64>::value)
        if (a32) {
            if (mode == MODE_HOST) {
                if constexpr (M == 1) return (void *)k_wave<1, MODE_HOST, VT, true>;
            }
            return mode == MODE_POWERS ? (void *)k_wave<M, MODE_POWERS, VT, true> : (void *)k_wave<M, MODE_CHEB, VT, true>;
        }
    if (mode == MODE_HOST) {
        if constexpr (M == 1) return (void *)k_wave<1, MODE_HOST, VT, false>;
        fail(MPK_ERR_UNSUPPORTED, "host output needs nrhs 1");
    }
    return mode == MODE_POWERS ? (void *)k_wave<M, MODE_POWERS, VT, false> : (void *)k_wave<M, MODE_CHEB, VT, false>;
}

// entries of the buffer, [scattered], of a slice's room after it, and bytes of one
struct WaveSize {
    int cap[2], slice, entry;
    int smem(bool scattered) const { return (cap[scattered] + slice) * entry; }
    template <class VT> void set() {
        using Buf = WaveBuf<VT>;
        *this = WaveSize{{Buf::CAP, Buf::CAP_SCATTERED}, Buf::SLICE, Buf::ENTRY};
    }
};
template <class VT> void *select_wave_vt(int mode, int m, bool a32, WaveSize *size) {
    size->set<VT>();
    switch (m) {
        case 1: return wave_fn<VT, 1>(mode, a32);
        case 2: return wave_fn<VT, 2>(mode, a32);
        case 4: return wave_fn<VT, 4>(mode, a32);
        case 8: return wave_fn<VT, 8>(mode, a32);
        case 16: return wave_fn<VT, 16>(mode, a32);
    }
    fail(MPK_ERR_UNSUPPORTED, "nrhs %d", m);
}

// defined in mpk_wave_<type>.cu: the kernel for (mode, nrhs, accumulator)
void *select_wave_f64(int mode, int m, bool a32, WaveSize *size);
void *select_wave_f32(int mode, int m, bool a32, WaveSize *size);
void *select_wave_bf16(int mode, int m, bool a32, WaveSize *size);
void *select_wave_dict(int mode, int m, bool a32, WaveSize *size);  // packed copies

}  // namespace mpk
