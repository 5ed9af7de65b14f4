// Blocked iteration path: positions staged in shared memory by tiles, the
// k-hop ids rearranged once so that every CTA streams one contiguous block.
//
// Tiles: tile j holds the positions of ids [j tv, (j+1) tv). Ranges: each
// tile's rows are cut into contiguous ranges on their own, so that the
// blocks (j, r) cost about the same whichever tile holds the most entries
// (on a power-law graph the hubs' tile holds twice the mean). Block (j, r)
// holds, for every row u of range r in order, the entries of u's k-hop row
// that fall in tile j, in an order chosen so that the lanes of one gather
// read distinct shared-memory banks; block starts are 16-byte aligned. An
// entry is stored as a 16-bit id relative to the tile's first id (a tile
// holds at most 65,534 positions), so the id stream, the only compulsory
// DRAM traffic of an iteration, is 2 bytes per entry instead of 4. One
// CTA per block loads tile j and the block's row directory into shared
// memory; each thread takes an equal, 8-aligned share of the block's
// entries (stored so that a warp's 16-byte id loads of one step, eight ids
// per lane, are contiguous), gathers positions from the tile and sums them
// row by row on its own. A row wholly inside a share is stored by its
// thread; the parts of rows cut by share bounds are added by a segmented
// scan across the warp, and rows cut by warp bounds by a second segmented
// scan in warp order, then stored as the row's partial for tile j. A
// second kernel adds each row's tile partials in tile order, adds its
// attraction terms and applies the capped move. (Window mode, for banded
// graphs: one window of positions per range instead of tiles, and the CTA
// finishes its rows itself.) Every partial has a fixed place and a fixed
// order of additions, so results do not depend on scheduling.
#include <algorithm>
#include <atomic>
#include <cmath>
#include <vector>

#include "device_util.cuh"
#include "ff.cuh"
#include "force.cuh"
#include "gila_impl.h"

namespace gila {

namespace {

constexpr int kBThreads = 1024;
constexpr int kBWarps = kBThreads / 32;
static_assert(kBWarps == 32, "the slot flush gives lane w of warp 0 the slots of warp w");
constexpr int kSmemCap = 227 * 1024;
constexpr int kMaxRows = 4096;  // rows per range (directory in shared memory)
constexpr int kMaxRowsTiles = 8192;  // tile mode: the directory may grow to this where the
                                     // 4096-row limit alone would exceed the CTA target
constexpr int kTileBudget = kSmemCap - (kMaxRows + 1) * 4 - 4096;
constexpr int64_t kMaxTile = 65534;  // tile-relative ids and the far slot's id fit 16 bits
constexpr uint32_t kBulkChunk = 32768;      // bytes per bulk copy instruction
constexpr int64_t kBlockedMinNnz = 4000000;  // automatic mode: k-hop entries needed (tiles)
constexpr int kWeightedMinSeg = 8;  // automatic mode with weights: mean entries of a segment
constexpr uint64_t kWaitNs = 1000000000ull;  // bound on a tile wait (1 s, far above any copy)
constexpr uint64_t kTestWaitNs = 1000000ull;   // the bound while the wait test hook is on
// Every (tile j, row) segment is padded to a multiple of 8 entries with the
// relative id tv, whose tile slot (one past the tile) holds a position so far
// away that its term is exactly zero: in FP32 the factor rcp(r^2 + 2^-100)
// of r^2 = 2e38 is below the smallest normal and flushes to 0; in FP64 r^2
// = 1.48e308 flushes rcp to 0 the same way; the generic model cuts terms
// beyond r^2 = 1e38 (FP32) or 1e300 (FP64). 0 * Delta then adds nothing.
// (FarSlot, force.cuh)

constexpr int kPrefetch = 4;  // steps between an L2 prefetch of ids and their ring load (4, 12, 24
                               // measured: 4 best; longer distances crowd L2)

// Set when a CTA gave up waiting for its tile copy (the launch's partials
// are then incomplete); read and cleared by blocked_tile_wait_failed().
__device__ int g_tile_wait_failed = 0;

struct BlockedArgs {
    const uint16_t* tk;        // tile-relative ids, block by block, in share storage order
    const int32_t* toff;       // nt n: start of segment (tile j, row u) within its block
    const int64_t* blk;        // 2 nb: first slot in tk and entry count of block b
    const int4* bdesc;         // nb: first row, end row and tile of block b
    int64_t n;
    int32_t nt, tv;
    int q;
    const void* pos;
    void* part;                // nt n cells of 4 T: (sx, sy, cx, cy) without the factor d^2
    uint64_t wait_ns;          // bound on the tile wait
    int skip_copy;             // test hook: announce the tile but copy nothing
    // window mode (one window of positions per row range, rows finished in
    // the CTA): first id and length of block b's window, the largest window
    // and range, and what the finish needs
    const int64_t* wbase;      // 2 nb
    int32_t wmax, rmax;
    const int64_t* row;
    const int32_t* col;
    ForceConsts c;
    int p;
    void* pos_out;
    void* disp_out;
    int uniform;               // FP32 steps taken warp-uniformly (tuning step_schedule >= 0)
    const void* wt;            // weighted tiles: repulsion weights (T[n])
};

template <class T, bool COMP>
struct Slot {
    int32_t row;
    T v[4];
};

// Cell (tile j, row u) of the partials: the sum as one position-type pair,
// followed by its compensation pair in the compensated mode (8 bytes a cell
// for plain FP32, so that the partials of short-row graphs with many tiles
// do not outweigh their id stream).
template <class T, bool COMP>
__device__ __forceinline__ typename V2<T>::type* cell_ptr(void* part, int64_t n, int j, int64_t u)
{
    using P2 = typename V2<T>::type;
    return reinterpret_cast<P2*>(part) + ((int64_t)j * n + u) * (COMP ? 2 : 1);
}

template <class T, bool COMP>
__device__ __forceinline__ void store_cell(typename V2<T>::type* c, const Acc<T, COMP>& a)
{
    using P2 = typename V2<T>::type;
    P2 s;
    s.x = a.sx;
    s.y = a.sy;
    c[0] = s;
    if (COMP) {
        P2 k;
        k.x = a.cx;
        k.y = a.cy;
        c[1] = k;
    }
}

// Entries per step: one 16-byte load of eight 16-bit ids.
constexpr int kStep = 8;

// Entries of block (j, r) per thread: thread t takes [lane_start(L, t),
// lane_start(L, t + 1)), 8-aligned; in storage every thread has lane_len(L)
// slots (a multiple of 8, at least its share), laid out per warp step-major:
// the k-th group of eight slots of lane l of warp w is at
// (w 32 lane_len + 256 k + 8 l) from the block's start, so that a warp's
// 16-byte loads of one step are one contiguous 512-byte run.
__host__ __device__ __forceinline__ int32_t lane_start(int32_t L, int t)
{
    return (t >= kBThreads) ? L : (int32_t)(((int64_t)L * t / kBThreads) & ~int64_t(kStep - 1));
}
__host__ __device__ __forceinline__ int32_t lane_len(int32_t L)
{
    // a share is at most L / kBThreads + 8 entries (8-aligned cuts)
    return (L == 0) ? 0 : ((L / kBThreads + 2 * kStep - 1) & ~(kStep - 1));
}

// Window mode's finish of the rows [u0, u0 + nrows) of a range, after their
// cells (sum of the unscaled repulsion terms, with compensation) are
// complete in shared memory: F = d^2 cell + attraction, then the capped move.
// Rows with at most kFinishDeg neighbours take one thread each; longer ones
// are taken by the whole warp their row falls to, lanes striding the
// adjacency row. Every row's order of additions is fixed.
template <class T, int MODEL, bool COMP>
__device__ __forceinline__ void window_finish(const struct BlockedArgs& A,
                                              const typename V2<T>::type* tile, int64_t tb,
                                              const typename V2<T>::type* cells, int64_t u0,
                                              int nrows);

// Window mode's finish: rows whose adjacency row is longer than this are
// finished by a whole warp (a few per range), the others by one thread.
constexpr int kFinishDeg = 32;

// Bytes of a weighted tile before its weights: positions, far slot, row
// directory, rounded up to 16 for the bulk copy of the weights.
__host__ __device__ __forceinline__ size_t weights_at(int64_t tv, int64_t rmax, size_t esz)
{
    return ((size_t)(tv + 1) * esz + (size_t)(rmax + 1) * 4 + 15) & ~size_t(15);
}

// W (tile mode): the tile's repulsion weights beside its positions, one more
// shared-memory read and product per entry. (The plain kernel gathers a
// position and a weight per entry through L2, 62% busy: the pruned Chung-Lu
// graph of 100,000 vertices, k = 2, 2.2e7 entries, 104 -> 45 us an iteration.)
template <class T, int MODEL, bool COMP, bool WIN, bool W>
__global__ void __launch_bounds__(kBThreads, 1) blocked_kernel(const BlockedArgs A)
{
    static_assert(!(WIN && W), "weights come with tiles");
    using P2 = typename V2<T>::type;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    // shared memory: the tile (or the range's window) with one more slot for
    // the padding's far position, the row directory, and in window mode the
    // rows' force cells
    const int tcap = WIN ? A.wmax : A.tv;
    P2* tile = reinterpret_cast<P2*>(smem_raw);
    int32_t* D = reinterpret_cast<int32_t*>(smem_raw + (size_t)(tcap + 1) * sizeof(P2));
    P2* cells = reinterpret_cast<P2*>(
        smem_raw + (((size_t)(tcap + 1) * sizeof(P2) + (size_t)(A.rmax + 1) * 4 + 15) & ~size_t(15)));
    __shared__ Slot<T, COMP> head[kBWarps], tail[kBWarps];
    __shared__ __align__(8) uint64_t tile_bar;
    __shared__ int tile_ok;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int4 bd = A.bdesc[blockIdx.x];  // rows [bd.x, bd.y) of tile bd.z (0 in window mode)
    const int j = WIN ? 0 : bd.z;
    const int64_t u0 = bd.x, u1 = bd.y;
    const int nrows = (int)(u1 - u0);
    const int64_t bsp = A.blk[2 * (int64_t)blockIdx.x];  // the block's first slot in tk
    // a block holds at most kMaxRows segments of at most tv entries: < 2^31
    const int32_t L = (int32_t)A.blk[2 * (int64_t)blockIdx.x + 1];
    const P2* pos = reinterpret_cast<const P2*>(A.pos);
    const int64_t tb = WIN ? A.wbase[2 * blockIdx.x] : (int64_t)j * A.tv;
    const int64_t tn = WIN ? A.wbase[2 * blockIdx.x + 1]
                           : ((A.n - tb < A.tv) ? A.n - tb : (int64_t)A.tv);
    // the cell of row i of the range: in shared memory (window mode) or the
    // global partial of (tile j, row u0 + i)
    auto cellp = [&](int64_t i) -> P2* {
        return WIN ? cells + 2 * i : cell_ptr<T, COMP>(A.part, A.n, j, u0 + i);
    };
    // Early start: the descriptors above and the row directory below are read
    // while the iteration before still runs; the placement, and the partials
    // that the kernel before reads, wait for it.
    pdl_trigger();
    if (threadIdx.x == 0) {
        // tile j by the bulk-copy engine (tv is even and the placement is
        // 16-byte aligned, so the source is too); an odd float2 tail by hand
        const uint32_t bytes = (uint32_t)(((size_t)tn * sizeof(P2)) & ~size_t(15));
        mbar_init(&tile_bar, 1);
        pdl_wait();
        // (a weighted tile starts at a multiple of four vertices)
        const uint32_t wbytes = W ? (uint32_t)(((size_t)tn * sizeof(T)) & ~size_t(15)) : 0u;
        mbar_arrive_expect_tx(&tile_bar, bytes + wbytes);
        const unsigned char* src = reinterpret_cast<const unsigned char*>(pos + tb);
        for (uint32_t o = 0; o < bytes && !A.skip_copy; o += kBulkChunk)
            bulk_g2s(smem_raw + o, src + o, (bytes - o < kBulkChunk) ? bytes - o : kBulkChunk,
                     &tile_bar);
        if constexpr (W) {
            const T* wsrc = reinterpret_cast<const T*>(A.wt) + tb;
            unsigned char* wdst = smem_raw + weights_at(A.tv, A.rmax, sizeof(P2));
            for (uint32_t o = 0; o < wbytes && !A.skip_copy; o += kBulkChunk)
                bulk_g2s(wdst + o, reinterpret_cast<const unsigned char*>(wsrc) + o,
                         (wbytes - o < kBulkChunk) ? wbytes - o : kBulkChunk, &tile_bar);
            T* w = reinterpret_cast<T*>(wdst);
            for (int64_t i = wbytes / sizeof(T); i < tn; ++i) w[i] = wsrc[i];
            w[A.tv] = T(0);  // the padding's
        }
        if ((size_t)tn * sizeof(P2) != bytes) tile[tn - 1] = pos[tb + tn - 1];
        P2 far;  // the padding's slot, outside the copied range
        far.x = FarSlot<T>::v;
        far.y = FarSlot<T>::v;
        tile[WIN ? tn : (int64_t)A.tv] = far;
    }
    for (int i = threadIdx.x; i < nrows; i += kBThreads) D[i] = A.toff[(int64_t)j * A.n + u0 + i];
    pdl_wait();
    if (WIN && threadIdx.x == 32) {
        // the finish's adjacency (row offsets, neighbour ids) and the rows'
        // own positions, pulled into L2 while the window loads and the
        // entries stream
        const int64_t ab = A.row[u0], ae = A.row[u1];
        prefetch_l2_range(A.row + u0, sizeof(int64_t) * (size_t)(u1 - u0 + 1));
        prefetch_l2_range(A.col + ab, sizeof(int32_t) * (size_t)(ae - ab));
        prefetch_l2_range(pos + u0, sizeof(P2) * (size_t)(u1 - u0));
    }
    // zero partials for rows with no entries in this tile
    for (int i = threadIdx.x; i < nrows; i += kBThreads) {
        P2* c = cellp(i);
        P2 z;
        z.x = T(0);
        z.y = T(0);
        c[0] = z;
        if (COMP) c[1] = z;
    }
    if (threadIdx.x == 0) D[nrows] = L;
    if (threadIdx.x < kBWarps) {
        head[threadIdx.x].row = -1;
        tail[threadIdx.x].row = -1;
    }
    if (threadIdx.x == 0) {
        bool ok = mbar_wait(&tile_bar, 0, A.wait_ns);
        if (!ok) {
            atomicExch(&g_tile_wait_failed, 1);
            mbar_wait(&tile_bar, 0, A.wait_ns);  // let the copy land before the CTA ends
        }
        tile_ok = ok ? 1 : 0;
    }
    __syncthreads();
    if (!tile_ok) return;  // uniform across the CTA
    mbar_wait(&tile_bar, 0, A.wait_ns);  // completed: acquires the tile for this thread

    if (L > 0) {
        // d^2 is applied when the partials are added, with weights to each
        // term (the plain kernel's form: a weight's product with an unscaled
        // 1 / r^2 overflows earlier)
        Rep<T, MODEL, COMP, kSrcShared, !W, W> f;
        f.src.set_shared(tile, 0u);  // ids are relative to the tile
        if constexpr (W)
            f.wt = reinterpret_cast<const T*>(smem_raw + weights_at(A.tv, A.rmax, sizeof(P2)));
        f.d2 = W ? const_d2<T>(A.c) : T(1);
        f.q = A.q;
        // this thread's entries [a, b) (a < L), their storage, and the row of a
        const int32_t a = lane_start(L, threadIdx.x), b = lane_start(L, threadIdx.x + 1);
        const int32_t m8 = lane_len(L);
        const uint4* ids4 =
            reinterpret_cast<const uint4*>(A.tk + bsp + (int64_t)warp * 32 * m8) + lane;
        int lo = 0, hi = nrows;
        while (lo < hi) {  // the last i with D[i] <= a
            const int mid = (lo + hi + 1) >> 1;
            if (D[mid] <= a) lo = mid; else hi = mid - 1;
        }
        int ri = lo;
        while (D[ri + 1] <= a) ++ri;  // skip empty rows at a (a < L = D[nrows])
        const int ra = ri;  // the first row
        // it continues the previous share's last row (that share holds its
        // earlier entries, or is empty and ends in the row that holds a)
        const bool open_left =
            D[ra] < a || (threadIdx.x > 0 && lane_start(L, threadIdx.x - 1) == a);
        int32_t re = D[ri + 1];
        // the next nonempty row and its own position, fetched one row ahead
        auto next_row = [&](int i) {
            int x = i + 1;
            while (x < nrows && D[x + 1] == D[x]) ++x;
            return x < nrows ? x : i;
        };
        int nx = next_row(ri);
        P2 xr = pos[u0 + ri];
        P2 xn = pos[u0 + nx];
        f.xu = xr.x;
        f.yu = xr.y;
        Acc<T, COMP> acc, first;
        // compensated mode: the terms of the steps since the last merge,
        // summed plainly; added to acc with its error term at the end of
        // each ring of steps and before a row closes. With weights every term
        // goes through a two-sum, as in the plain kernel, which these graphs
        // took before
        Acc<T, false> pend;
        constexpr bool PEND = COMP && !W;
        auto merge_pending = [&]() {
            if (PEND) {
                add_compensated(acc, pend.sx, pend.sy);
                pend = Acc<T, false>();
            }
        };
        bool in_first = true;
        // the current row is complete: the first row's sum is kept for the
        // warp's scan; a later row lies wholly in [a, b) and is stored
        auto close_row = [&]() {
            merge_pending();
            if (in_first) {
                first = acc;
                in_first = false;
            } else {
                store_cell<T, COMP>(cellp(ri), acc);
            }
            acc = Acc<T, COMP>();
            ri = nx;
            re = D[ri + 1];
            xr = xn;
            f.xu = xr.x;
            f.yu = xr.y;
            nx = next_row(ri);
            xn = pos[u0 + nx];
        };
        // 16-byte id loads run kRing steps ahead (four, three with the
        // compensated sums, which need the registers); each unrolled step
        // consumes its own ring register and refills it: no register moves
        constexpr int kRing = COMP ? 3 : 4;
        const int nsteps = m8 / kStep;  // the same for every thread of the block
        uint4 ring[kRing];
#pragma unroll
        for (int st = 0; st < kRing; ++st) ring[st] = ld_ids4(ids4 + 32 * st);
        // the warp's ids kPrefetch steps ahead of the ring are pulled into L2
        // by one lane, kRing steps (kRing x 512 bytes) at a time
        const uint4* warp_ids = ids4 - lane;
        if (lane == 0)
            for (int k = kRing; k < kPrefetch + kRing && k < nsteps; k += kRing)
                bulk_prefetch_l2(warp_ids + 32 * k,
                                 (uint32_t)(512 * ((nsteps - k < kRing) ? nsteps - k : kRing)));
        // segments and shares are multiples of 8 entries: every step lies in
        // one row, and rows change only between steps. A step before the
        // current row's end (and the share's) goes straight to its eight
        // terms; a step where a row begins first closes the rows before it
        int32_t lim = (re < b) ? re : b;
        int32_t p = a;
        auto eight = [&](const uint4 c) {
            if (PEND) {
                // compensated mode: into the plain pending sum
                f(c.x & 0xffffu, pend);
                f(c.x >> 16, pend);
                f(c.y & 0xffffu, pend);
                f(c.y >> 16, pend);
                f(c.z & 0xffffu, pend);
                f(c.z >> 16, pend);
                f(c.w & 0xffffu, pend);
                f(c.w >> 16, pend);
            } else {
                f(c.x & 0xffffu, acc);
                f(c.x >> 16, acc);
                f(c.y & 0xffffu, acc);
                f(c.y >> 16, acc);
                f(c.z & 0xffffu, acc);
                f(c.z >> 16, acc);
                f(c.w & 0xffffu, acc);
                f(c.w >> 16, acc);
            }
        };
        // one step: its eight terms, after closing the rows that end before
        // it; the ring register refilled kRing steps ahead (the id array has
        // kRing steps of slack at its end, so the refill needs no test)
        auto step = [&](uint4& r, int k) {
            const uint4 c = r;
            r = ld_ids4(ids4 + 32 * (k + kRing));
            if (sizeof(T) == 8) {
                // FP64 (costly terms): the warp takes every step together
                // and only the closing of rows diverges, so no term is
                // issued twice (BA k = 3: 5.15 ms; 7.08 ms as for FP32)
                if (p < b) {
                    while (p >= re) close_row();
                    eight(c);
                }
            } else if (A.uniform) {
                // FP32, default: only the closing of rows diverges, the
                // step's terms are issued once for the warp; steps past the
                // share hold the far slot's id and add zeros
                if (p >= lim) {
                    if (p < b) {
                        while (p >= re) close_row();
                        lim = (re < b) ? re : b;
                    } else {
                        lim = INT32_MAX;
                    }
                }
                eight(c);
            } else if (p < lim) {
                // FP32, tuning step_schedule = -1: lanes that close a row
                // in this step issue its terms apart from the others
                eight(c);
            } else if (p < b) {
                while (p >= re) close_row();
                lim = (re < b) ? re : b;
                eight(c);
            }
            p += kStep;
        };
        int k0 = 0;
        for (; k0 + kRing <= nsteps; k0 += kRing) {
            const int kp = k0 + kPrefetch + kRing;
            if (lane == 0 && kp < nsteps)
                bulk_prefetch_l2(warp_ids + 32 * kp,
                                 (uint32_t)(512 * ((nsteps - kp < kRing) ? nsteps - kp : kRing)));
#pragma unroll
            for (int st = 0; st < kRing; ++st) step(ring[st], k0 + st);
            merge_pending();
        }
#pragma unroll
        for (int st = 0; st < kRing - 1; ++st)
            if (k0 + st < nsteps) step(ring[st], k0 + st);
        merge_pending();
        const bool has_b = !in_first;  // the share ends in a later row than it began
        if (in_first) first = acc;
        const int orow = has_b ? ri : ra;  // the row the share ends in
        const bool open_right = re > b;

        // Rows cut by share bounds, in lane order: element A (row ra, sum
        // first) and, with has_b, element B (row ri, sum acc). A segmented
        // scan of the warp's elements (A continues the previous lane's last
        // row, B always starts a run) gives each run's sum where it ends.
        Acc<T, COMP> x = has_b ? acc : first;
        const int prev_orow = __shfl_up_sync(kFull, orow, 1);
        const bool cont = lane > 0 && prev_orow == ra;
        const bool start = has_b || !cont;
        const unsigned starts = __ballot_sync(kFull, start);
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            // the run of lane - o reaches this lane when no run starts in
            // lanes (lane - o, lane]
            const unsigned span = (lane >= o) ? (((1u << o) - 1u) << (lane - o + 1)) : 0u;
            const T sx = __shfl_up_sync(kFull, x.sx, o);
            const T sy = __shfl_up_sync(kFull, x.sy, o);
            const T cx = COMP ? __shfl_up_sync(kFull, x.cx, o) : T(0);
            const T cy = COMP ? __shfl_up_sync(kFull, x.cy, o) : T(0);
            if (lane >= o && (starts & span) == 0) {
                Acc<T, COMP> y;
                y.sx = sx;
                y.sy = sy;
                y.cx = cx;
                y.cy = cy;
                y.merge(x.sx, x.sy, x.cx, x.cy);
                x = y;
            }
        }
        // the sum of the run that reaches into A of a lane with B
        Acc<T, COMP> carry;
        {
            const T sx = __shfl_up_sync(kFull, x.sx, 1);
            const T sy = __shfl_up_sync(kFull, x.sy, 1);
            const T cx = COMP ? __shfl_up_sync(kFull, x.cx, 1) : T(0);
            const T cy = COMP ? __shfl_up_sync(kFull, x.cy, 1) : T(0);
            if (cont) {
                carry.sx = sx;
                carry.sy = sy;
                carry.cx = cx;
                carry.cy = cy;
            }
        }
        // runs that include lane 0's A belong to a row begun before the
        // warp's entries when lane 0's first row is open on the left; such a
        // run, and one running past the warp's last entry, goes to the
        // warp's slots, every other run to its cell
        const bool lane0_open = __shfl_sync(kFull, open_left, 0);
        const bool lane0_has_b = __shfl_sync(kFull, has_b, 0);
        const bool last_open = __shfl_sync(kFull, open_right, 31);
        const unsigned below = starts & ((2u << lane) - 1u) & ~1u;  // starts in lanes 1..lane
        auto put = [&](int row, const Acc<T, COMP>& v, bool from_lane0, bool past_end) {
            if (from_lane0 && lane0_open) {
                Slot<T, COMP>& sl = head[warp];
                sl.row = row;
                sl.v[0] = v.sx;
                sl.v[1] = v.sy;
                sl.v[2] = v.cx;
                sl.v[3] = v.cy;
            } else if (past_end) {
                Slot<T, COMP>& sl = tail[warp];
                sl.row = row;
                sl.v[0] = v.sx;
                sl.v[1] = v.sy;
                sl.v[2] = v.cx;
                sl.v[3] = v.cy;
            } else {
                store_cell<T, COMP>(cellp(row), v);
            }
        };
        if (has_b) {
            // A's run ends here: the carry plus this lane's first row
            carry.merge(first.sx, first.sy, first.cx, first.cy);
            const bool a_from0 =
                (lane == 0) || (cont && !lane0_has_b && (below & ~(1u << lane)) == 0);
            put(ra, carry, a_from0, false);
        }
        const int next_ra = __shfl_down_sync(kFull, ra, 1);
        const bool ends_here = (lane == 31) || next_ra != orow;
        if (ends_here) {
            const bool o_from0 = !has_b && !lane0_has_b && below == 0;
            put(orow, x, o_from0, lane == 31 && last_open);
        }
    }
    __syncthreads();
    if (warp == 0) {
        // rows cut by warp bounds: warp w's slots (a row begun before the
        // warp, a row running past its end) go to lane w of warp 0, and a
        // segmented scan across the lanes adds each row's slots in warp
        // order (a row's slots lie in consecutive warps; a warp without
        // slots lies between no two slots of one row)
        const Slot<T, COMP>& hs = head[lane];
        const Slot<T, COMP>& ts = tail[lane];
        auto acc_of = [](const Slot<T, COMP>& sl) {
            Acc<T, COMP> v;
            v.sx = sl.v[0];
            v.sy = sl.v[1];
            v.cx = sl.v[2];
            v.cy = sl.v[3];
            return v;
        };
        // the lane's elements: A (its first row) and, with has_b, B (a
        // second row); a lane without slots takes a row no lane has
        const bool hh = hs.row >= 0, ht = ts.row >= 0;
        const int ra = hh ? hs.row : (ht ? ts.row : -2 - lane);
        Acc<T, COMP> ea = hh ? acc_of(hs) : (ht ? acc_of(ts) : Acc<T, COMP>());
        bool has_b = false;
        Acc<T, COMP> eb;
        if (hh && ht) {
            if (ts.row == hs.row) {
                ea.merge(ts.v[0], ts.v[1], ts.v[2], ts.v[3]);
            } else {
                has_b = true;
                eb = acc_of(ts);
            }
        }
        const int orow = has_b ? ts.row : ra;
        Acc<T, COMP> x = has_b ? eb : ea;
        const int prev_orow = __shfl_up_sync(kFull, orow, 1);
        const bool cont = lane > 0 && prev_orow == ra;
        const unsigned starts = __ballot_sync(kFull, has_b || !cont);
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned span = (lane >= o) ? (((1u << o) - 1u) << (lane - o + 1)) : 0u;
            const T sx = __shfl_up_sync(kFull, x.sx, o);
            const T sy = __shfl_up_sync(kFull, x.sy, o);
            const T cx = COMP ? __shfl_up_sync(kFull, x.cx, o) : T(0);
            const T cy = COMP ? __shfl_up_sync(kFull, x.cy, o) : T(0);
            if (lane >= o && (starts & span) == 0) {
                Acc<T, COMP> y;
                y.sx = sx;
                y.sy = sy;
                y.cx = cx;
                y.cy = cy;
                y.merge(x.sx, x.sy, x.cx, x.cy);
                x = y;
            }
        }
        const T px = __shfl_up_sync(kFull, x.sx, 1);
        const T py = __shfl_up_sync(kFull, x.sy, 1);
        const T pcx = COMP ? __shfl_up_sync(kFull, x.cx, 1) : T(0);
        const T pcy = COMP ? __shfl_up_sync(kFull, x.cy, 1) : T(0);
        if (has_b) {
            // A's run ends here: the run reaching into A, then A
            Acc<T, COMP> carry;
            if (cont) {
                carry.sx = px;
                carry.sy = py;
                carry.cx = pcx;
                carry.cy = pcy;
            }
            carry.merge(ea.sx, ea.sy, ea.cx, ea.cy);
            store_cell<T, COMP>(cellp(ra), carry);
        }
        const int next_ra = __shfl_down_sync(kFull, ra, 1);
        if (orow >= 0 && (lane == 31 || next_ra != orow)) store_cell<T, COMP>(cellp(orow), x);
    }
    if constexpr (WIN) {
        // every row of the range is complete here: F = d^2 (its cell) + the
        // attraction over its adjacency row (whose neighbours lie in the
        // window, as A is part of N(k)), then the capped move
        __syncthreads();
        window_finish<T, MODEL, COMP>(A, tile, tb, cells, u0, nrows);
    }
}


template <class T, int MODEL, bool COMP>
__device__ __forceinline__ void finish_row(const BlockedArgs& A, const Att<T, MODEL, COMP, kSrcShared>& att0,
                                           const typename V2<T>::type* cells, int64_t u0, int i,
                                           const Acc<T, COMP>& at)
{
    using P2 = typename V2<T>::type;
    const P2 pu = reinterpret_cast<const P2*>(A.pos)[u0 + i];
    const T d2 = const_d2<T>(A.c);
    Acc<T, COMP> rep;
    const P2 c0 = cells[2 * i];
    rep.sx = c0.x * d2;
    rep.sy = c0.y * d2;
    if (COMP) {
        const P2 c1 = cells[2 * i + 1];
        rep.cx = c1.x * d2;
        rep.cy = c1.y * d2;
    }
    rep.merge(at.sx, at.sy, at.cx, at.cy);
    apply_move<T>(const_t<T>(A.c), A.pos_out, A.disp_out, u0 + i, pu.x, pu.y, rep.fx(), rep.fy());
}

template <class T, int MODEL, bool COMP>
__device__ __forceinline__ void window_finish(const BlockedArgs& A,
                                              const typename V2<T>::type* tile, int64_t tb,
                                              const typename V2<T>::type* cells, int64_t u0,
                                              int nrows)
{
    using P2 = typename V2<T>::type;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const P2* pos = reinterpret_cast<const P2*>(A.pos);
    Att<T, MODEL, COMP, kSrcShared> att;
    att.src.set_shared(tile, (uint32_t)tb);
    att.inv_d = const_inv_d<T>(A.c);
    att.p = A.p;
    const uint32_t* col = reinterpret_cast<const uint32_t*>(A.col);
    // warp w takes rows [32 w, 32 w + 32), then 1024 further on: each lane
    // one row; rows with more than kFinishDeg neighbours are then taken by
    // the whole warp, one after the other, lanes striding the adjacency row
    // (no barrier; a row's order of additions depends only on its length)
    for (int base = warp * 32; base < nrows; base += kBThreads) {
        const int i = base + lane;
        const bool live = i < nrows;
        int64_t rb = 0, re = 0;
        if (live) {
            rb = A.row[u0 + i];
            re = A.row[u0 + i + 1];
        }
        const bool hub = live && re - rb > kFinishDeg;
        if (live && !hub) {
            Att<T, MODEL, COMP, kSrcShared> a1 = att;
            const P2 pu = pos[u0 + i];
            a1.xu = pu.x;
            a1.yu = pu.y;
            Acc<T, COMP> at;
            row_sum_rel(col, rb, re, 0, 1, a1, at);
            finish_row<T, MODEL, COMP>(A, att, cells, u0, i, at);
        }
        unsigned hubs = __ballot_sync(kFull, hub);
        while (hubs) {
            const int l = __ffs(hubs) - 1;
            hubs &= hubs - 1;
            const int ih = base + l;
            const int64_t hb = __shfl_sync(kFull, rb, l), he = __shfl_sync(kFull, re, l);
            const P2 pu = pos[u0 + ih];
            Att<T, MODEL, COMP, kSrcShared> a1 = att;
            a1.xu = pu.x;
            a1.yu = pu.y;
            Acc<T, COMP> at;
            row_sum_rel(col, hb, he, lane, 32, a1, at);
            at.group_reduce(32);
            if (lane == 0) finish_row<T, MODEL, COMP>(A, att, cells, u0, ih, at);
        }
    }
}

// Window mode with a row per lane, for graphs whose rows are of about equal
// length (meshes, grids): a slice is 32 consecutive rows, stored step-major
// (four 16-bit ids of every lane, 256 bytes a step), each row padded with the
// far slot's id to the slice's longest. A lane sums its row in registers and
// moves its vertex: no row changes inside a step, no scan over lanes, no
// cells, no second pass over the rows. The first ids of a row are its
// neighbours (A is part of N(k)), whose attraction is formed from the same
// shared-memory positions, so the adjacency is not read at all. A warp takes
// consecutive slices, one stream of steps, four steps ahead in registers.
// Consecutive rows of a mesh read consecutive positions in each step, which
// keeps their gathers free of bank conflicts without any reordering. 512
// threads at 64 registers put two CTAs on an SM, one loading its window
// while the other computes.
// The mesh 1000 x 1000, k = 3, compensated: 63.5 -> 35 us per iteration (30.2
// since, with early launches and fr_entry)
// against the shares of blocked_kernel; 700 x 700, FP32: 35.3 -> 17.6.
//
// Automatic mode takes it where (us per iteration, FP32, before -> this):
// - mean rows reach kRowMeanLen: random ids within a band conflict in this
//   order and long rows amortise the shares' costs (rows of 151 ids 48 -> 37,
//   183: 54 -> 44, 413: 82 -> 94; a mesh at k = 8, 213 ids: 50 -> 35);
// - a window fits two CTAs on an SM, with up to 16 times as many ranges,
//   else one (random 4-regular graphs of 25,000 vertices, whose every window
//   is the whole graph: rows of 479 ids 21 -> 33);
// - the padding stays within kRowPadding (band graphs at 1.8 slots an
//   entry: 39 -> 29, 30 -> 17);
// - the windows' bytes stay within kRowWindowBytes an entry: they come from
//   L2 once an iteration, and the alternative for a mesh is tiles that most
//   rows have nothing in (mesh 2000 x 2000, k = 2: 4478 -> 77; grid
//   1000 x 1000, k = 2: 364 -> 17; the FP64 mesh 1000 x 1000, k = 3:
//   2453 -> 913, bound by its FP64 operations).
constexpr int kRowThreads = 512;
constexpr int kRowWarps = kRowThreads / 32;
constexpr int kRowAhead = 4;       // steps of ids in registers ahead
constexpr int kRowMaxDeg = 64;     // longest adjacency row taken
constexpr size_t kRowWindow = 110 * 1024;  // a window's bytes for two CTAs per SM
constexpr int64_t kRowWindowBytes = 8;     // automatic mode: windows' bytes per k-hop entry
constexpr double kRowMeanLen = 256.0;      // automatic mode: longest mean row
constexpr double kRowPadding = 2.0;  // most slots per k-hop entry

struct RowsArgs {
    const uint16_t* tk;
    const int4* sdesc;
    const uint16_t* deg;
    const int4* bdesc;
    const int64_t* wbase;
    int64_t n;
    int q, p;
    ForceConsts c;
    const void* pos;
    void* pos_out;
    void* disp_out;
    uint64_t wait_ns;
    int skip_copy;
};

template <class T, int MODEL, bool COMP>
__global__ void __launch_bounds__(kRowThreads, sizeof(T) == 4 ? 2 : 1) rows_kernel(const RowsArgs A)
{
    using P2 = typename V2<T>::type;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    P2* tile = reinterpret_cast<P2*>(smem_raw);
    __shared__ __align__(8) uint64_t tile_bar;
    __shared__ int tile_ok;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const P2* pos = reinterpret_cast<const P2*>(A.pos);
    const int64_t tb = A.wbase[2 * blockIdx.x], tn = A.wbase[2 * blockIdx.x + 1];
    pdl_trigger();
    // this warp's slices and the first steps of their stream, read while the
    // iteration before still runs
    const int4 bd = A.bdesc[blockIdx.x];
    const int s0 = bd.x >> 5, ns = ((bd.y + 31) >> 5) - s0;
    const int sa = s0 + ns * warp / kRowWarps, sb = s0 + ns * (warp + 1) / kRowWarps;
    int4 sd = make_int4(0, 0, 0, 0);
    uint2 next[kRowAhead];
    const uint2* ids = reinterpret_cast<const uint2*>(A.tk) + lane;
    if (sa < sb) {
        sd = A.sdesc[sa];
#pragma unroll
        for (int i = 0; i < kRowAhead; ++i)
            if (i < sd.y) next[i] = ld_ids2(ids + 32 * ((int64_t)sd.x + i));
    }
    pdl_wait();
    if (threadIdx.x == 0) {
        // the window by the bulk-copy engine (its first id is even: 16-byte
        // aligned); an odd float2 tail by hand; the far slot after it
        const uint32_t bytes = (uint32_t)(((size_t)tn * sizeof(P2)) & ~size_t(15));
        mbar_init(&tile_bar, 1);
        mbar_arrive_expect_tx(&tile_bar, bytes);
        const unsigned char* src = reinterpret_cast<const unsigned char*>(pos + tb);
        for (uint32_t o = 0; o < bytes && !A.skip_copy; o += kBulkChunk)
            bulk_g2s(smem_raw + o, src + o, (bytes - o < kBulkChunk) ? bytes - o : kBulkChunk,
                     &tile_bar);
        if ((size_t)tn * sizeof(P2) != bytes) tile[tn - 1] = pos[tb + tn - 1];
        P2 far;
        far.x = FarSlot<T>::v;
        far.y = FarSlot<T>::v;
        tile[tn] = far;
    }
    if (threadIdx.x == 0) {
        bool ok = mbar_wait(&tile_bar, 0, A.wait_ns);
        if (!ok) {
            atomicExch(&g_tile_wait_failed, 1);
            mbar_wait(&tile_bar, 0, A.wait_ns);  // let the copy land before the CTA ends
        }
        tile_ok = ok ? 1 : 0;
    }
    __syncthreads();
    if (!tile_ok) return;  // uniform across the CTA
    mbar_wait(&tile_bar, 0, A.wait_ns);  // completed: acquires the window for this thread

    Rep<T, MODEL, COMP, kSrcShared, true> f;
    f.src.set_shared(tile, 0u);
    f.d2 = T(1);
    f.q = A.q;
    Att<T, MODEL, COMP, kSrcShared> att;
    att.src.set_shared(tile, 0u);
    att.inv_d = const_inv_d<T>(A.c);
    att.p = A.p;
    for (int s = sa; s < sb; ++s) {
        const int64_t u = (int64_t)s * 32 + lane;
        const bool live = u < A.n;
        P2 pu;
        pu.x = T(0);
        pu.y = T(0);
        int deg = 0;
        if (live) {
            pu = pos[u];
            deg = A.deg[u];
        }
        f.xu = att.xu = pu.x;
        f.yu = att.yu = pu.y;
        const int dmax = __reduce_max_sync(kFull, deg);
        const int steps = sd.y;
        const int64_t start = sd.x;
        const int4 sn = (s + 1 < sb) ? A.sdesc[s + 1] : make_int4(0, 0, 0, 0);
        Acc<T, COMP> acc, at;
        for (int k0 = 0; k0 < steps || k0 == 0; k0 += kRowAhead) {
            uint2 cur[kRowAhead];
#pragma unroll
            for (int i = 0; i < kRowAhead; ++i) cur[i] = next[i];
            // refill: the next steps of this slice, or the next slice's first
            const bool more = k0 + kRowAhead < steps;
            const int64_t from = more ? start + k0 + kRowAhead : (int64_t)sn.x;
            const int left = more ? steps - k0 - kRowAhead : sn.y;
#pragma unroll
            for (int i = 0; i < kRowAhead; ++i)
                if (i < left) next[i] = ld_ids2(ids + 32 * (from + i));
            Acc<T, false> pend;
#pragma unroll
            for (int i = 0; i < kRowAhead; ++i) {
                if (k0 + i >= steps) break;
                const uint32_t v0 = cur[i].x & 0xffffu, v1 = cur[i].x >> 16;
                const uint32_t v2 = cur[i].y & 0xffffu, v3 = cur[i].y >> 16;
                const int e = 4 * (k0 + i);
                if constexpr (sizeof(T) == 4 && MODEL == kFR) {
                    if (e < dmax) {  // the rows' first ids are their neighbours
                        auto both = [&](auto& to) {
                            fr_entry(tile[v0], pu.x, pu.y, att.inv_d, e < deg, to, at);
                            fr_entry(tile[v1], pu.x, pu.y, att.inv_d, e + 1 < deg, to, at);
                            fr_entry(tile[v2], pu.x, pu.y, att.inv_d, e + 2 < deg, to, at);
                            fr_entry(tile[v3], pu.x, pu.y, att.inv_d, e + 3 < deg, to, at);
                        };
                        if constexpr (COMP) both(pend); else both(acc);
                        continue;
                    }
                }
                if constexpr (COMP) {
                    f(v0, pend);
                    f(v1, pend);
                    f(v2, pend);
                    f(v3, pend);
                } else {
                    f(v0, acc);
                    f(v1, acc);
                    f(v2, acc);
                    f(v3, acc);
                }
                if (e < dmax) {
                    if (e < deg) att(v0, at);
                    if (e + 1 < deg) att(v1, at);
                    if (e + 2 < deg) att(v2, at);
                    if (e + 3 < deg) att(v3, at);
                }
            }
            // compensated mode: up to sixteen terms summed plainly, then
            // added with their error term
            if constexpr (COMP) add_compensated(acc, pend.sx, pend.sy);
        }
        if (live) {
            const T d2 = const_d2<T>(A.c);
            acc.sx *= d2;
            acc.sy *= d2;
            acc.cx *= d2;
            acc.cy *= d2;
            acc.merge(at.sx, at.sy, at.cx, at.cy);
            // (an isolated vertex has padding only: zeros at a finite place)
            apply_move<T>(const_t<T>(A.c), A.pos_out, A.disp_out, u, pu.x, pu.y,
                          deg > 0 ? acc.fx() : T(0), deg > 0 ? acc.fy() : T(0));
        }
        sd = sn;
    }
}

// The slices of rows_kernel from the k-hop lists: a warp per slice, a row per
// lane. The neighbours first, then the other ids (both lists ascending, one
// merge), then the far slot's id (the window's length). A row whose
// neighbours are not all found among its k-hop ids (an unsorted or repeated
// adjacency, a self-loop) sets *bad, and the plan takes another form.
__global__ void __launch_bounds__(128)
rows_fill_kernel(int64_t n, int64_t nslices, const int64_t* __restrict__ row,
                 const int32_t* __restrict__ col, const int64_t* __restrict__ krow,
                 const uint32_t* __restrict__ kcol, const int4* __restrict__ sdesc,
                 uint16_t* __restrict__ tk, uint16_t* __restrict__ deg_out, int* __restrict__ bad)
{
    const int lane = threadIdx.x & 31;
    const int64_t s = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (s >= nslices) return;  // warp-uniform
    const int4 sd = sdesc[s];
    const int64_t u = s * 32 + lane;
    int64_t kb = 0, ke = 0, ab = 0;
    int deg = 0;
    if (u < n) {
        kb = krow[u];
        ke = krow[u + 1];
        ab = row[u];
        deg = (int)(row[u + 1] - ab);
        deg_out[u] = (uint16_t)deg;
    }
    uint64_t* out = reinterpret_cast<uint64_t*>(tk) + (int64_t)sd.x * 32 + lane;
    const int slots = sd.y * 4;
    uint64_t four = 0;
    int w = 0;
    auto put = [&](uint32_t id) {
        if (w >= slots) return;
        four |= (uint64_t)(uint16_t)id << (16 * (w & 3));
        if ((w & 3) == 3) {
            out[32 * (w >> 2)] = four;
            four = 0;
        }
        ++w;
    };
    for (int a = 0; a < deg; ++a) put((uint32_t)col[ab + a] - (uint32_t)sd.z);
    int a = 0, found = 0;
    for (int64_t i = kb; i < ke; ++i) {
        const uint32_t x = kcol[i];
        while (a < deg && (uint32_t)col[ab + a] < x) ++a;
        if (a < deg && (uint32_t)col[ab + a] == x) ++found;
        else put(x - (uint32_t)sd.z);
    }
    if (found != deg) atomicExch(bad, 1);
    while (w < slots) put((uint32_t)sd.w);
}

struct CombineArgs {
    const int64_t* row;
    const int32_t* col;
    int64_t n;
    int32_t nt;
    ForceConsts c;
    int p;
    const void* pos_in;
    const void* part;
    void* pos_out;
    void* disp_out;
    const int32_t* hubs;  // rows with more than kHubDeg neighbours, one block each
    int32_t nhub;         // hub blocks, first in the grid
    int32_t nreg;         // blocks of the regular part of the grid, after the hubs
};

// Regular rows: four lanes per vertex (more vertices in flight; measured
// 1.8% faster per iteration than eight on the Barabasi-Albert workload).
// Hubs (adjacency rows longer than kHubDeg) take a block of kCombineThreads
// each, at the start of the grid, so no vertex walks a long row on a few
// lanes while the rest of the GPU waits and the hubs do not form a tail.
constexpr int kCombineLanes = 4;
constexpr int kCombineThreads = 256;
constexpr int kHubDeg = 64;

template <class T, bool COMP>
__device__ __forceinline__ void add_cell(const void* part, int64_t n, int j, int64_t u,
                                         Acc<T, COMP>& s)
{
    using P2 = typename V2<T>::type;
    const P2* c = cell_ptr<T, COMP>(const_cast<void*>(part), n, j, u);
    const P2 v = c[0];
    if (COMP) {
        const P2 k = c[1];
        s.merge(v.x, v.y, k.x, k.y);
    } else {
        s.merge(v.x, v.y, T(0), T(0));
    }
}

// F = d^2 (sum of the tile partials) + attraction; then the capped move.
template <class T, bool COMP>
__device__ __forceinline__ void finish_vertex(const CombineArgs& A, int64_t u, T xu, T yu,
                                              Acc<T, COMP> rep, const Acc<T, COMP>& att)
{
    const T d2 = const_d2<T>(A.c);
    rep.sx *= d2;
    rep.sy *= d2;
    rep.cx *= d2;
    rep.cy *= d2;
    rep.merge(att.sx, att.sy, att.cx, att.cy);
    apply_move<T>(const_t<T>(A.c), A.pos_out, A.disp_out, u, xu, yu, rep.fx(), rep.fy());
}

template <class T, int MODEL, bool COMP>
__global__ void __launch_bounds__(kCombineThreads) combine_kernel(const CombineArgs A)
{
    using P2 = typename V2<T>::type;
    // (launched after the kernel before has ended: nothing writes this placement)
    const P2* __restrict__ pos_in = reinterpret_cast<const P2*>(A.pos_in);
    Att<T, MODEL, COMP, kSrcConst> att;
    att.src.pos = pos_in;
    att.inv_d = const_inv_d<T>(A.c);
    att.p = A.p;
    Acc<T, COMP> rep, at;
    pdl_trigger();
    if ((int)blockIdx.x < A.nhub) {
        // one hub per block
        __shared__ T sh[kCombineThreads / 32][8];
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
        const int64_t u = A.hubs[blockIdx.x];
        const int64_t rb = A.row[u], re = A.row[u + 1];
        const P2 pu = pos_in[u];
        for (int jj = threadIdx.x; jj < A.nt; jj += kCombineThreads)
            add_cell<T, COMP>(A.part, A.n, jj, u, rep);
        att.xu = pu.x;
        att.yu = pu.y;
        row_sum_batched<4>(reinterpret_cast<const uint32_t*>(A.col), rb, re, (int)threadIdx.x,
                           kCombineThreads, att, at);
        rep.group_reduce(32);
        at.group_reduce(32);
        if (lane == 0) {
            sh[warp][0] = rep.sx;
            sh[warp][1] = rep.sy;
            sh[warp][2] = rep.cx;
            sh[warp][3] = rep.cy;
            sh[warp][4] = at.sx;
            sh[warp][5] = at.sy;
            sh[warp][6] = at.cx;
            sh[warp][7] = at.cy;
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            Acc<T, COMP> r2, a2;
            for (int w = 0; w < kCombineThreads / 32; ++w) {
                r2.merge(sh[w][0], sh[w][1], sh[w][2], sh[w][3]);
                a2.merge(sh[w][4], sh[w][5], sh[w][6], sh[w][7]);
            }
            finish_vertex<T, COMP>(A, u, pu.x, pu.y, r2, a2);
        }
        return;
    }
    const int gl = threadIdx.x & (kCombineLanes - 1);
    const int64_t u = ((int64_t)(blockIdx.x - A.nhub) * kCombineThreads + threadIdx.x) / kCombineLanes;
    bool live = u < A.n;
    int64_t rb = 0, re = 0;
    if (live) {
        rb = A.row[u];
        re = A.row[u + 1];
        live = re - rb <= kHubDeg;  // hubs are done by their own blocks
    }
    // the neighbours' ids of a lane's first two turns are on their way before
    // the cells (BA n = 100,000, k = 2: 33.5 -> 31.8 us an iteration)
    const uint32_t* col = reinterpret_cast<const uint32_t*>(A.col);
    uint32_t ahead[2] = {0u, 0u};
    const int deg = (int)(re - rb);
    if (live) {
        if (gl < deg) ahead[0] = ld_id(col + rb + gl);
        if (gl + kCombineLanes < deg) ahead[1] = ld_id(col + rb + gl + kCombineLanes);
    }
    P2 pu;
    pu.x = T(0);
    pu.y = T(0);
    if (live) {
        // tile partials first (independent loads), lane gl takes tiles gl, gl + 4, ...
        for (int jj = gl; jj < A.nt; jj += kCombineLanes) add_cell<T, COMP>(A.part, A.n, jj, u, rep);
        pu = pos_in[u];
        att.xu = pu.x;
        att.yu = pu.y;
        if (gl < deg) att(ahead[0], at);
        if (gl + kCombineLanes < deg) att(ahead[1], at);
        if (deg > 2 * kCombineLanes)
            row_sum_batched<2>(col, rb + 2 * kCombineLanes, re, gl, kCombineLanes, att, at);
    }
    rep.group_reduce(kCombineLanes);
    at.group_reduce(kCombineLanes);
    if (live && gl == 0) finish_vertex<T, COMP>(A, u, pu.x, pu.y, rep, at);
}

// Bounds of row u's segment in tile j (binary search on the sorted row).
__device__ __forceinline__ void seg_bounds(const int64_t* __restrict__ krow,
                                           const uint32_t* __restrict__ kcol, int64_t u, int j,
                                           int nt, int tv, int64_t* lo, int64_t* hi)
{
    const int64_t kb = krow[u], ke = krow[u + 1];
    auto lower = [&](uint32_t key) {
        int64_t x = kb, y = ke;
        while (x < y) {
            const int64_t mid = (x + y) >> 1;
            if (kcol[mid] < key) x = mid + 1; else y = mid;
        }
        return x;
    };
    *lo = (j == 0) ? kb : lower((uint32_t)j * (uint32_t)tv);
    *hi = (j == nt - 1) ? ke : lower((uint32_t)(j + 1) * (uint32_t)tv);
}

__global__ void seglen_kernel(int64_t n, const int64_t* __restrict__ krow,
                              const uint32_t* __restrict__ kcol, int nt, int tv,
                              int32_t* __restrict__ len, int32_t* __restrict__ start)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n * nt) return;
    int64_t lo, hi;
    seg_bounds(krow, kcol, i % n, (int)(i / n), nt, tv, &lo, &hi);
    len[i] = (int32_t)(hi - lo);
    start[i] = (int32_t)(lo - krow[i % n]);
}

__global__ void rowlen_kernel(int64_t n, const int64_t* __restrict__ krow, int32_t* __restrict__ len,
                              int32_t* __restrict__ start)
{
    const int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (u >= n) return;
    len[u] = (int32_t)(krow[u + 1] - krow[u]);
    start[u] = 0;
}

// ---- the plan's cut of every tile's rows into ranges, on the device: with
// the segment lengths of n nt cells (4.3 million on BA n = 333,334, k = 2)
// copied to the host, summed, searched and their offsets copied back, the
// host took 19 of the 27.2 ms from reset to the first step, the GPU 8.6;
// 8.2 ms with the plan here.

// A segment's entries as stored, and the cost of its row in the block: the
// padded entries and a per-row term where it has entries (directory, row
// change, cell store), else only the zeroed cell.
__host__ __device__ __forceinline__ int64_t seg_padded(int64_t len)
{
    return (len + kStep - 1) & ~int64_t(kStep - 1);
}
__host__ __device__ __forceinline__ int64_t row_cost(int64_t len)
{
    return len > 0 ? 8 + seg_padded(len) : 1;
}

constexpr int kCellThreads = 256;
constexpr int kCellItems = 8;
constexpr int kCellTile = kCellThreads * kCellItems;

// Totals of padded lengths and costs of every kCellTile cells.
__global__ void __launch_bounds__(kCellThreads)
cell_sums_kernel(int64_t cells, const int32_t* __restrict__ len, int64_t* __restrict__ sums)
{
    __shared__ int64_t wt[kCellThreads / 32 + 1];
    const int64_t base = (int64_t)blockIdx.x * kCellTile;
    int64_t pad = 0, cost = 0;
    for (int i = threadIdx.x; i < kCellTile && base + i < cells; i += kCellThreads) {
        const int64_t l = len[base + i];
        pad += seg_padded(l);
        cost += row_cost(l);
    }
    int64_t tp, tc;
    block_inclusive_scan<int64_t, kCellThreads>(pad, wt, &tp);
    block_inclusive_scan<int64_t, kCellThreads>(cost, wt, &tc);
    if (threadIdx.x == 0) {
        sums[2 * blockIdx.x] = tp;
        sums[2 * blockIdx.x + 1] = tc;
    }
}

// Exclusive scan of both totals, in place, by one block.
__global__ void __launch_bounds__(1024) cell_scan_sums_kernel(int64_t* __restrict__ sums, int64_t nb)
{
    __shared__ int64_t wt[1024 / 32 + 1];
    int64_t cp = 0, cc = 0;
    for (int64_t b0 = 0; b0 < nb; b0 += 1024) {
        const int64_t i = b0 + threadIdx.x;
        const int64_t p = i < nb ? sums[2 * i] : 0, c = i < nb ? sums[2 * i + 1] : 0;
        int64_t tp, tc;
        const int64_t ip = block_inclusive_scan<int64_t, 1024>(p, wt, &tp);
        const int64_t ic = block_inclusive_scan<int64_t, 1024>(c, wt, &tc);
        if (i < nb) {
            sums[2 * i] = cp + ip - p;
            sums[2 * i + 1] = cc + ic - c;
        }
        cp += tp;
        cc += tc;
    }
}

// Exclusive prefix sums of the cells (cells + 1 values each).
__global__ void __launch_bounds__(kCellThreads)
cell_prefix_kernel(int64_t cells, const int32_t* __restrict__ len, const int64_t* __restrict__ sums,
                   int64_t* __restrict__ pre_pad, int64_t* __restrict__ pre_cost)
{
    __shared__ int64_t wt[kCellThreads / 32 + 1];
    __shared__ int64_t sp[kCellTile], sc[kCellTile];
    const int64_t base = (int64_t)blockIdx.x * kCellTile;
    const int t0 = threadIdx.x * kCellItems;
    int32_t l[kCellItems];
    int64_t pad = 0, cost = 0;
#pragma unroll
    for (int i = 0; i < kCellItems; ++i) {
        l[i] = base + t0 + i < cells ? len[base + t0 + i] : -1;
        if (l[i] >= 0) {
            pad += seg_padded(l[i]);
            cost += row_cost(l[i]);
        }
    }
    int64_t tp, tc;
    int64_t rp = sums[2 * blockIdx.x] + block_inclusive_scan<int64_t, kCellThreads>(pad, wt, &tp) - pad;
    int64_t rc = sums[2 * blockIdx.x + 1] + block_inclusive_scan<int64_t, kCellThreads>(cost, wt, &tc) - cost;
#pragma unroll
    for (int i = 0; i < kCellItems; ++i) {
        sp[t0 + i] = rp;
        sc[t0 + i] = rc;
        if (l[i] >= 0) {
            rp += seg_padded(l[i]);
            rc += row_cost(l[i]);
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < kCellTile && base + i < cells; i += kCellThreads) {
        pre_pad[base + i] = sp[i];
        pre_cost[base + i] = sc[i];
    }
    if (base + t0 < cells && base + t0 + kCellItems >= cells) {  // the thread of the last cell
        pre_pad[cells] = rp;
        pre_cost[cells] = rc;
    }
}

// Greedy cut of every tile's rows into ranges of cost at most caps[x] (a
// range takes at least one row) and at most max_rows rows, for as many caps
// as the grid is wide: a warp per (cap, tile) walks the tile, finding each
// range's end by a 32-way search of the prefix costs. counts[x] receives the
// ranges of all tiles; with cuts, tile j's bounds go to
// cuts[(x nt + j) stride ...] and their number to tile_counts[x nt + j]. A
// tile stops once it exceeds limit.
__global__ void __launch_bounds__(256)
cut_kernel(int64_t n, int nt, const int64_t* __restrict__ pre, const int64_t* __restrict__ caps,
           int64_t max_rows, int64_t limit, int* __restrict__ counts, int32_t* __restrict__ cuts,
           int64_t stride, int* __restrict__ tile_counts)
{
    const int lane = threadIdx.x & 31;
    const int j = blockIdx.y * 8 + (threadIdx.x >> 5);
    if (j >= nt) return;
    const int64_t cap = caps[blockIdx.x];
    const int64_t* p = pre + (int64_t)j * n;
    int64_t s = 0, count = 0;
    if (cuts) cuts += ((int64_t)blockIdx.x * nt + j) * stride;
    if (cuts && lane == 0) cuts[0] = 0;
    while (s < n && count <= limit) {
        const int64_t most = p[s] + cap;
        int64_t lo = s + 1, hi = s + max_rows < n ? s + max_rows : n;
        while (lo < hi) {  // the last e in [lo, hi] with p[e] <= most, lo if none
            const int64_t step = (hi - lo + 31) >> 5;
            const int64_t x = lo + step * (lane + 1) < hi ? lo + step * (lane + 1) : hi;
            const int c = __popc(__ballot_sync(kFull, p[x] <= most));
            const int64_t l0 = lo;
            if (c > 0) lo = l0 + step * c < hi ? l0 + step * c : hi;
            if (c < 32 && l0 + step * (c + 1) - 1 < hi) hi = l0 + step * (c + 1) - 1;
        }
        s = lo;
        ++count;
        if (cuts && lane == 0 && count < stride) cuts[count] = (int32_t)s;
    }
    if (lane == 0) {
        atomicAdd(&counts[blockIdx.x], (int)(count < INT32_MAX / 2 ? count : INT32_MAX / 2));
        if (tile_counts) tile_counts[(int64_t)blockIdx.x * nt + j] = (int)count;
    }
}

// Padded entries and cost of blocks given as (first row, end row, tile, -).
__global__ void block_sums_kernel(int64_t n, int64_t cells, int64_t nb, const int4* __restrict__ blocks,
                                  const int64_t* __restrict__ pre, int64_t* __restrict__ out)
{
    const int64_t b = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= nb) return;
    const int4 x = blocks[b];
    const int64_t lo = x.z * n + x.x, hi = x.z * n + x.y;
    out[2 * b] = pre[hi] - pre[lo];
    out[2 * b + 1] = pre[cells + 1 + hi] - pre[cells + 1 + lo];
}

// Starts of the segments within their blocks.
__global__ void toff_kernel(int64_t n, const int4* __restrict__ bdesc,
                            const int64_t* __restrict__ pre_pad, int32_t* __restrict__ toff)
{
    const int4 x = bdesc[blockIdx.x];
    const int64_t* p = pre_pad + x.z * n;
    const int64_t first = p[x.x];
    for (int64_t u = x.x + threadIdx.x; u < x.y; u += blockDim.x)
        toff[x.z * n + u] = (int32_t)(p[u] - first);
}

// Vertices of adjacency degree above kHubDeg, in any order.
__global__ void hubs_kernel(int64_t n, const int64_t* __restrict__ row, int32_t* __restrict__ hubs,
                            int* __restrict__ count)
{
    const int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (u < n && row[u + 1] - row[u] > kHubDeg) hubs[atomicAdd(count, 1)] = (int32_t)u;
}

// Copy every (tile, row) segment into its block's share storage as 16-bit
// ids relative to the tile: entry p of the block, held by the share of
// thread t (s = p - lane_start(L, t)), goes to slot
// (t / 32) 32 lane_len(L) + 256 (s / 8) + 8 (t % 32) + s % 8; the entries up
// to the segment's padded length take the block's padding id.
//
// With SPREAD each segment's ids are also ordered for blocked_kernel's
// shared-memory gathers. A warp's gather is served in groups of G lanes
// (G = 128 bytes / position size: 16 for float2, 8 for double2), one
// wavefront per group when the group's tile offsets are distinct modulo G
// (distinct banks), one more per repeat; in ascending id order the residues
// fall at random and a 16-lane group takes about three. In one gather the
// lanes of a group read entry s of their own shares, so entry s of thread t
// aims at residue (t + s) mod G, distinct across the group for every s. A
// row's sum does not depend on the order of its entries (up to rounding)
// and a segment is one row, so its ids are dealt to its entries: each entry
// takes an id of its target residue while one is left, and the entries left
// over take the ids left over.
//
// Blocks come from the grid, so that a warp looks its block up once and then
// takes rows of it: one at a time, or two where most segments are short
// (SHORTS; the storage then holds the padding already). Three forms by length:
// - up to 32 entries (two rows of up to 16 at once): an id and an entry per
//   lane, matched by (residue, rank) through a table in shared memory;
// - longer: by chunks of at most kSpreadChunk entries; the ids grouped by
//   residue with a counter per lane and residue (no atomics, no matching),
//   then dealt 32 entries at a time; the targets of 32 entries of one share
//   are consecutive residues, so that an entry's rank among the entries of
//   its target is its lane / G and every residue gives 32 / G ids.
// A larger chunk leaves fewer entries without their target residue (each such
// entry costs its half-warp one more gather wavefront): 2048 against 1024
// took Chung-Lu n = 250,000, k = 3 from 4.27 to 4.18 ms per launch, 4096 gave
// 4.15 ms at half the occupancy here.
// The layout of Chung-Lu n = 60,000, k = 3 took 7.85 ms with a warp per
// (tile, row), atomics and a matching step per 32 entries, 3.27 now; BA
// n = 333,334, k = 2 (segments of 12 entries) 3.78 -> 1.34 ms.
constexpr int kSpreadWarps = 8;
constexpr int kSpreadChunk = 2048;

// Shared memory of one warp of the layout kernel.
struct SpreadSmem {
    uint16_t in[kSpreadChunk];            // the chunk's relative ids by residue
    union {
        uint32_t off[16][32];             // next place of (residue, lane) while grouping
        struct {                          // short rows:
            uint8_t slot[32 * 32];        // entry of (residue, rank)
            uint8_t rest[32];             // entries left over
            int32_t cnt[2][32];           // ids and entries of each residue
        } s;
    };
    uint32_t left[kSpreadChunk / 32];     // entries without an id of their residue, a bit each
    int32_t ask[32], base[32];            // counts and places by residue
};

// The slots past each thread's share set to the block's padding id (its far
// slot), so that the FP32 kernel takes a thread's last steps like any other
// (their terms are exact zeros). Shares and block starts are multiples of 8
// slots: whole 16-byte stores. The segments' own padding is written by the
// layout kernel, or, with `all`, here with every other slot: on short
// segments, a third of whose slots are padding, that is cheaper (BA
// n = 333,334, k = 2: 27 us here against 190 there), on long ones it writes
// the whole storage once more (Chung-Lu n = 60,000, k = 3: 278 us, 8 now).
__global__ void __launch_bounds__(kBThreads)
pad_shares_kernel(uint16_t* __restrict__ tk, const int64_t* __restrict__ blk,
                  const int64_t* __restrict__ wbase, int tv, int all)
{
    const int64_t b = blockIdx.x;
    const int32_t L = (int32_t)blk[2 * b + 1], m8 = lane_len(L);
    const int t = threadIdx.x;
    const uint32_t pad = wbase ? (uint32_t)wbase[2 * b + 1] : (uint32_t)tv;
    const uint32_t pp = pad | (pad << 16);
    uint4* dst = reinterpret_cast<uint4*>(tk + blk[2 * b] + (int64_t)(t >> 5) * 32 * m8) + (t & 31);
    const int32_t own = (lane_start(L, t + 1) - lane_start(L, t)) / kStep;
    for (int32_t k = all ? 0 : own; k < m8 / kStep; ++k)
        dst[32 * (int64_t)k] = make_uint4(pp, pp, pp, pp);
}

// The share (thread of blocked_kernel) that holds entry p of a block of L
// entries; inv = kBThreads / L.
__device__ __forceinline__ int share_of(int32_t L, int32_t p, float inv)
{
    // the last t with L t / kBThreads below the end of p's group of eight
    int t = (int)((float)((p & ~(kStep - 1)) + kStep) * inv);
    t = t < kBThreads ? t : kBThreads - 1;
    while (t > 0 && lane_start(L, t) > p) --t;
    while (t < kBThreads - 1 && lane_start(L, t + 1) <= p) ++t;
    return t;
}

// Slot of entry number sidx of share t (see above), from the block's start.
__device__ __forceinline__ int64_t share_slot(int t, int32_t sidx, int32_t m8)
{
    return (int64_t)(t >> 5) * 32 * m8 + 256 * (int64_t)(sidx >> 3) + 8 * (t & 31) + (sidx & 7);
}

// One entry and one id per lane (entry p of the block), of one row or, with
// `second` telling their lanes apart, of two: dealt by residue within a row.
// Lanes with `tail` set store the padding of their row's end.
template <int G>
__device__ __forceinline__ void deal_short(SpreadSmem& S, bool act, bool tail, int32_t p, uint32_t id,
                                           uint16_t pad, bool second, int32_t L, int32_t m8,
                                           float inv, uint16_t* tk, int lane)
{
    const int key = second ? 16 : 0;
    int64_t at = 0;
    int want = 0;
    if (act || tail) {
        const int t = share_of(L, p, inv);
        const int32_t sidx = p - lane_start(L, t);
        at = share_slot(t, sidx, m8);
        want = ((t + sidx) & (G - 1)) + key;
        if (tail) tk[at] = pad;
    }
    const unsigned lt = lanemask_lt();
    const int has = (int)(id & (G - 1)) + key;
    const unsigned mw = __match_any_sync(kFull, act ? want : 64 + lane);
    const unsigned mh = __match_any_sync(kFull, act ? has : 64 + lane);
    const int rw = __popc(mw & lt), rh = __popc(mh & lt);
    S.s.cnt[0][lane] = 0;
    S.s.cnt[1][lane] = 0;
    __syncwarp();
    if (act) {
        S.s.slot[want * 32 + rw] = (uint8_t)lane;
        if (rw == 0) S.s.cnt[1][want] = __popc(mw);
        if (rh == 0) S.s.cnt[0][has] = __popc(mh);
    }
    __syncwarp();
    const bool served = act && rw < S.s.cnt[0][want];  // this lane's entry finds its residue
    const bool placed = act && rh < S.s.cnt[1][has];   // this lane's id finds an entry
    // the rest in lane order: a row has as many entries as ids left over, so
    // that the k-th entry left of all the lanes and the k-th id left belong
    // to the same row
    const unsigned er = __ballot_sync(kFull, act && !served), ir = __ballot_sync(kFull, act && !placed);
    if (act && !served) S.s.rest[__popc(er & lt)] = (uint8_t)lane;
    __syncwarp();
    int to = lane;
    if (placed) to = S.s.slot[has * 32 + rh];
    else if (act) to = S.s.rest[__popc(ir & lt)];
    const int64_t dst = __shfl_sync(kFull, at, to);
    if (act) tk[dst] = (uint16_t)id;
    __syncwarp();  // the next rows reuse the tables
}

template <int G, bool SPREAD, bool SHORTS>
__global__ void __launch_bounds__(kSpreadWarps * 32, 4) block_layout_kernel(
    int64_t n, const int64_t* __restrict__ krow, const uint32_t* __restrict__ kcol, int tv,
    const int64_t* __restrict__ wbase, const int32_t* __restrict__ len,
    const int32_t* __restrict__ start, const int32_t* __restrict__ toff,
    const int64_t* __restrict__ blk, const int4* __restrict__ bdesc, uint16_t* __restrict__ tk_all)
{
    extern __shared__ __align__(128) unsigned char smem_raw[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    SpreadSmem& S = reinterpret_cast<SpreadSmem*>(smem_raw)[warp];
    const int64_t b = blockIdx.x;
    const int4 bd = bdesc[b];
    const int j = bd.z;
    const int32_t L = (int32_t)blk[2 * b + 1];
    if (L == 0) return;
    // ids are relative to tile j, or in window mode to block b's window
    const uint32_t tb = wbase ? (uint32_t)wbase[2 * b] : (uint32_t)j * (uint32_t)tv;
    uint16_t* tk = tk_all + blk[2 * b];
    const int32_t m8 = lane_len(L);
    const float inv = (float)kBThreads / (float)L;
    const int32_t* clen = len + (int64_t)j * n;
    const int32_t* cstart = start + (int64_t)j * n;
    const int32_t* coff = toff + (int64_t)j * n;

    const uint16_t pad = wbase ? (uint16_t)wbase[2 * b + 1] : (uint16_t)tv;
    auto put_pad = [&](int32_t p) {
        const int t = share_of(L, p, inv);
        tk[share_slot(t, p - lane_start(L, t), m8)] = pad;
    };

    auto row = [&](int64_t u, int rl) {  // one row of rl entries by the whole warp
        const uint32_t* src = kcol + krow[u] + cstart[u];
        const int32_t S0 = coff[u];
        const int padded = (int)seg_padded(rl);
        if (!SHORTS && (!SPREAD || rl > 32) && rl + lane < padded) put_pad(S0 + rl + lane);
        if (!SPREAD) {
            for (int e = lane; e < rl; e += 32) {
                const int t = share_of(L, S0 + e, inv);
                tk[share_slot(t, S0 + e - lane_start(L, t), m8)] = (uint16_t)(src[e] - tb);
            }
            return;
        }
        if (rl <= 32) {
            const uint32_t id = lane < rl ? src[lane] - tb : 0u;
            deal_short<G>(S, lane < rl, !SHORTS && lane >= rl && lane < padded, S0 + lane, id, pad, false, L, m8,
                          inv, tk, lane);
            return;
        }
        for (int32_t c0 = 0; c0 < rl; c0 += kSpreadChunk) {
            const int cl = rl - c0 < kSpreadChunk ? rl - c0 : kSpreadChunk;
            const uint32_t* cs = src + c0;
            // ids of each residue on this lane
#pragma unroll
            for (int c = 0; c < G; ++c) S.off[c][lane] = 0;
#pragma unroll 1
            for (int e0 = lane; e0 < cl; e0 += 256) {
                uint32_t id[8];
#pragma unroll
                for (int x = 0; x < 8; ++x) id[x] = e0 + 32 * x < cl ? cs[e0 + 32 * x] - tb : 0u;
#pragma unroll
                for (int x = 0; x < 8; ++x)
                    if (e0 + 32 * x < cl) ++S.off[id[x] & (G - 1)][lane];
            }
            // counters to places: exclusive prefix over residues, then lanes
            int cnt = 0, cst = 0;  // lane c: residue c's ids and where they start
            {
                int run = 0;
#pragma unroll
                for (int c = 0; c < G; ++c) {
                    const int mine = (int)S.off[c][lane];
                    const int incl = warp_inclusive_scan(mine, lane);
                    S.off[c][lane] = (uint32_t)(run + incl - mine);
                    const int tot = __shfl_sync(kFull, incl, 31);
                    if (lane == c) {
                        cnt = tot;
                        cst = run;
                    }
                    run += tot;
                }
            }
#pragma unroll 1
            for (int e0 = lane; e0 < cl; e0 += 256) {
                uint32_t id[8];
#pragma unroll
                for (int x = 0; x < 8; ++x) id[x] = e0 + 32 * x < cl ? cs[e0 + 32 * x] - tb : 0u;
#pragma unroll
                for (int x = 0; x < 8; ++x)
                    if (e0 + 32 * x < cl) S.in[S.off[id[x] & (G - 1)][lane]++] = (uint16_t)id[x];
            }
            __syncwarp();
            // deal: lane c < G keeps residue c's next id and the ids left
            constexpr int kPer = 32 / G;  // entries of one target in 32 consecutive ones
            int rem = cnt, next = cst, nleft = 0;
            int t = share_of(L, S0 + c0, inv);
            int32_t sb = lane_start(L, t), se = lane_start(L, t + 1);
            for (int e0 = 0; e0 < cl;) {
                const int32_t p0 = S0 + c0 + e0;
                while (se <= p0 && t < kBThreads - 1) {  // the share that holds the first entry
                    ++t;
                    sb = se;
                    se = lane_start(L, t + 1);
                }
                const int32_t s0 = p0 - sb;  // a multiple of 8, like every bound here
                const int same = (se - p0 < cl - e0 ? se - p0 : cl - e0) >> 5;
                if (same > 0) {
                    // whole groups of 32 entries of one share: a lane's target
                    // is the same in all of them, and group i takes the ids
                    // kPer i .. of every residue
                    const int want = (t + s0 + lane) & (G - 1), rank = lane / G;
                    const int have = __shfl_sync(kFull, rem, want);
                    const uint16_t* from = S.in + __shfl_sync(kFull, next, want) + rank;
                    uint16_t* to = tk + (int64_t)(t >> 5) * 32 * m8 + 8 * (t & 31) +
                                   256 * ((s0 + lane) >> 3) + (lane & 7);
                    if (__all_sync(kFull, rank + kPer * (same - 1) < have)) {
#pragma unroll 4
                        for (int i = 0; i < same; ++i) to[1024 * i] = from[kPer * i];
                        for (int i = lane; i < same; i += 32) S.left[(e0 >> 5) + i] = 0u;
                    } else {
                        for (int i = 0; i < same; ++i) {
                            const bool got = rank + kPer * i < have;
                            if (got) to[1024 * i] = from[kPer * i];
                            const unsigned lm = __ballot_sync(kFull, !got);
                            if (lane == 0) S.left[(e0 >> 5) + i] = lm;
                            nleft += __popc(lm);
                        }
                    }
                    if (lane < G) {
                        const int give = kPer * same < rem ? kPer * same : rem;
                        rem -= give;
                        next += give;
                    }
                    e0 += 32 * same;
                    continue;
                }
                // 32 entries that reach into the next share, or the last ones
                const int e = e0 + lane;
                const bool act = e < cl;
                int32_t sidx = s0 + lane;
                int tl = t;
                if (act && p0 + lane >= se) {
                    tl = share_of(L, p0 + lane, inv);
                    sidx = p0 + lane - lane_start(L, tl);
                }
                const int want = (tl + sidx) & (G - 1);
                const unsigned m = __match_any_sync(kFull, act ? want : G + lane);
                const int rank = __popc(m & lanemask_lt());
                S.ask[lane] = 0;
                __syncwarp();
                if (act && rank == 0) S.ask[want] = __popc(m);
                __syncwarp();
                const int have = __shfl_sync(kFull, rem, want);
                const int from = __shfl_sync(kFull, next, want);
                const bool got = act && rank < have;
                if (got) tk[share_slot(tl, sidx, m8)] = S.in[from + rank];
                const unsigned lm = __ballot_sync(kFull, act && !got);
                if (lane == 0) S.left[e0 >> 5] = lm;
                nleft += __popc(lm);
                if (lane < G) {
                    const int give = S.ask[lane] < rem ? S.ask[lane] : rem;
                    rem -= give;
                    next += give;
                }
                __syncwarp();
                e0 += 32;
            }
            // the entries left over take the ids left over, in order
            if (nleft > 0) {
                if (lane >= G) rem = 0;
                int incl = rem;
#pragma unroll
                for (int o = 1; o < G; o <<= 1) {
                    const int v = __shfl_up_sync(kFull, incl, o);
                    if (lane >= o) incl += v;
                }
                S.ask[lane] = lane < G ? incl : INT32_MAX;        // ids left up to residue c
                S.base[lane] = next - (incl - rem);               // the k-th id left: in[this + k]
                __syncwarp();
                // listed first (the counters' place is free), then one a lane
                uint16_t* list = reinterpret_cast<uint16_t*>(S.off);
                constexpr int kList = (int)(sizeof(S.off) / 2);
                for (int l0 = 0; l0 < nleft; l0 += kList) {
                    int before = -l0;
                    for (int w0 = 0; w0 * 32 < cl; w0 += 32) {  // a word of 32 entries per lane
                        uint32_t m = (w0 + lane) * 32 < cl ? S.left[w0 + lane] : 0u;
                        const int mine = __popc(m);
                        const int upto = warp_inclusive_scan(mine, lane);
                        for (int k = before + upto - mine; m; m &= m - 1, ++k)
                            if (k >= 0 && k < kList)
                                list[k] = (uint16_t)((w0 + lane) * 32 + __ffs(m) - 1);
                        before += __shfl_sync(kFull, upto, 31);
                    }
                    __syncwarp();
                    const int stop = nleft - l0 < kList ? nleft - l0 : kList;
                    for (int x = lane; x < stop; x += 32) {
                        const int k = l0 + x;
                        int c = 0;  // the residue of the k-th id left
#pragma unroll
                        for (int o = G / 2; o > 0; o >>= 1)
                            if (S.ask[c + o - 1] <= k) c += o;
                        const int32_t p = S0 + c0 + list[x];
                        const int ts = share_of(L, p, inv);
                        tk[share_slot(ts, p - lane_start(L, ts), m8)] = S.in[S.base[c] + k];
                    }
                    __syncwarp();
                }
            }
            __syncwarp();  // the next chunk reuses the buffers
        }
    };
    // this CTA's part of the block's rows, taken by its warps one at a time,
    // or in pairs where most rows are short
    constexpr int unit = SHORTS ? 2 : 1;
    __shared__ int s_next;
    if (threadIdx.x == 0) s_next = 0;
    __syncthreads();
    const int64_t rows = bd.y - bd.x;
    const int64_t u0 = bd.x + rows * blockIdx.y / gridDim.y;
    const int64_t u1 = bd.x + rows * (blockIdx.y + 1) / gridDim.y;
    for (;;) {
        int64_t u = 0;
        if (lane == 0) u = u0 + unit * (int64_t)atomicAdd(&s_next, 1);
        u = __shfl_sync(kFull, u, 0);
        if (u >= u1) break;
        const int l0 = clen[u], l1 = unit == 2 && u + 1 < u1 ? clen[u + 1] : 0;
        if (SPREAD && SHORTS && l0 <= 16 && l1 <= 16) {
            if (l0 + l1 == 0) continue;
            const bool second = lane >= 16;
            const int64_t v = second ? u + 1 : u;
            const int e = lane & 15;
            const int lv = second ? l1 : l0;
            const bool act = e < lv;
            const int32_t p = act ? coff[v] + e : 0;
            const uint32_t id = act ? kcol[krow[v] + cstart[v] + e] - tb : 0u;
            deal_short<G>(S, act, false, p, id, pad, second, L, m8, inv, tk, lane);
            continue;
        }
#pragma unroll 1
        for (int h = 0; h < unit; ++h) {
            const int rl = h ? l1 : l0;
            if (rl) row(u + h, rl);
        }
    }
}

template <class T, int MODEL, bool COMP, bool WIN, bool W>
cudaError_t launch_blocked_typed(gila_graph* g, const BlockedArgs& B, const CombineArgs& C,
                                 int grid, size_t smem, cudaStream_t st, int device)
{
    static std::atomic<uint64_t> configured{0};  // one bit per device; callers may race
    const uint64_t bit = 1ull << (device & 63);
    if (!(configured.load() & bit)) {
        cudaError_t e = cudaFuncSetAttribute(blocked_kernel<T, MODEL, COMP, WIN, W>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             kSmemCap - 4096);
        if (e != cudaSuccess) return e;
        configured.fetch_or(bit);
    }
    cudaEvent_t pa = prof_kernel_begin(g);
    cudaError_t e = launch_dependent(true, blocked_kernel<T, MODEL, COMP, WIN, W>, dim3((unsigned)grid),
                                     kBThreads, smem, st, B);
    count_launch();
    prof_kernel_end(g, pa, WIN ? "blocked_kernel (window)" : "blocked_kernel");
    if (e != cudaSuccess || WIN) return e;
    // Launched after blocked_kernel has ended: blocks that came early and
    // waited on SMs that were done cost more than they hid (BA n = 100,000,
    // k = 2: 35.9 us an iteration against 29.2). blocked_kernel itself comes
    // early, while the combine before it ends: 31.8 -> 29.2 us, k = 3 155.3
    // -> 153.3, BA n = 333,334, k = 2 136.5 -> 134.7; rows_kernel on the mesh
    // 1000 x 1000, k = 3: 36.7 -> 34.2.
    combine_kernel<T, MODEL, COMP><<<(unsigned)(C.nreg + C.nhub), kCombineThreads, 0, st>>>(C);
    count_launch();
    return cudaGetLastError();
}

template <class T, int MODEL, bool COMP>
cudaError_t launch_rows(gila_graph* g, const RowsArgs& R, const TilePlan& P)
{
    static std::atomic<uint64_t> configured{0};  // one bit per device; callers may race
    const uint64_t bit = 1ull << (g->device & 63);
    if (!(configured.load() & bit)) {
        cudaError_t e = cudaFuncSetAttribute(rows_kernel<T, MODEL, COMP>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             kSmemCap - 4096);
        if (e != cudaSuccess) return e;
        configured.fetch_or(bit);
    }
    cudaEvent_t pa = prof_kernel_begin(g);
    cudaError_t e = launch_dependent(true, rows_kernel<T, MODEL, COMP>, dim3((unsigned)P.nb),
                                     kRowThreads, ((size_t)P.tv + 1) * 2 * sizeof(T), g->stream, R);
    count_launch();
    prof_kernel_end(g, pa, "blocked_kernel (window, row per lane)");
    return e;
}

template <class T, int MODEL, bool COMP>
cudaError_t launch_pair(gila_graph* g, const BlockedArgs& B, const CombineArgs& C, int grid,
                        size_t smem, cudaStream_t st, int device, bool win)
{
    if constexpr (MODEL == kFR)
        if (B.wt) return launch_blocked_typed<T, MODEL, COMP, false, true>(g, B, C, grid, smem, st, device);
    return win ? launch_blocked_typed<T, MODEL, COMP, true, false>(g, B, C, grid, smem, st, device)
               : launch_blocked_typed<T, MODEL, COMP, false, false>(g, B, C, grid, smem, st, device);
}

// The k-hop term of the quality reductions, sum over unordered k-hop pairs
// {u, v} of d^2 / delta^q, for FP32 placements that have a blocked plan:
// one CTA per (tile or window, row range), positions from the shared-memory
// tile, each pair counted once from its smaller end. Every row is sorted,
// so the entries of row u in the tile are one contiguous run that starts
// after the row's runs in earlier tiles (the plan's segment lengths), and
// only the tile that holds u itself needs a binary search to drop the ids
// up to u. The CTA takes its rows by batches: their runs are numbered by a
// block scan and each warp takes an equal slice of the batch's entries (a
// warp per row left the CTA's warps waiting on the one with a hub's row:
// barrier stalls 5.1 per issue, 38% issue active on Chung-Lu n = 40,000).
// Each term is in double-float arithmetic (ff.cuh), sixteen terms per lane
// summed as a double-float, then added in FP64; the CTA's FP64 partial goes
// to its own slot, and the partials are added in CTA order.
constexpr int kMetThreads = 1024;
constexpr int kMetWarps = kMetThreads / 32;
constexpr int kMetBatch = 512;  // rows per batch (10.5 KB of shared memory beside the tile)
constexpr int kMetSmemMax = kSmemCap - 12 * 1024;  // the tile's share of shared memory

struct MetricArgs {
    const int64_t* krow;
    const int32_t* len;    // tile mode: nt n segment lengths (row u's entries in tile j)
    const int32_t* start;  // ... and their starts within the rows
    const uint32_t* kcol;
    const int4* bdesc;     // nb: first row, end row and tile of block b
    const int64_t* wbase;  // window mode: 2 nb (first id, length), else null
    int64_t n;
    int32_t nt, tv;
    double d2;
    float d2hi, d2lo;      // d2 as a double-float
    int q;
    int unit;              // d = 1 and q = 1
    const float2* pos;
    double* partial;       // one per CTA
    uint64_t wait_ns;
};

__global__ void __launch_bounds__(kMetThreads, 1) khop_metric_kernel(const MetricArgs A)
{
    extern __shared__ __align__(128) unsigned char smem_raw[];
    float2* tile = reinterpret_cast<float2*>(smem_raw);
    __shared__ __align__(8) uint64_t tile_bar;
    __shared__ int tile_ok;
    __shared__ double s_part[kMetWarps];
    __shared__ int s_wsum[kMetWarps];
    __shared__ int s_pre[kMetBatch + 1];
    __shared__ int64_t s_off[kMetBatch];  // entry i of the batch is kcol[s_off[its row] + i]
    __shared__ float2 s_q[kMetBatch];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int4 bd = A.bdesc[blockIdx.x];
    const int j = bd.z;
    const int64_t u0 = bd.x, u1 = bd.y;
    const int64_t tb = A.wbase ? A.wbase[2 * blockIdx.x] : (int64_t)j * A.tv;
    const int64_t tn = A.wbase ? A.wbase[2 * blockIdx.x + 1]
                               : ((A.n - tb < A.tv) ? A.n - tb : (int64_t)A.tv);
    if (threadIdx.x == 0) {
        const uint32_t bytes = (uint32_t)(((size_t)tn * sizeof(float2)) & ~size_t(15));
        mbar_init(&tile_bar, 1);
        mbar_arrive_expect_tx(&tile_bar, bytes);
        const unsigned char* src = reinterpret_cast<const unsigned char*>(A.pos + tb);
        for (uint32_t o = 0; o < bytes; o += kBulkChunk)
            bulk_g2s(smem_raw + o, src + o, (bytes - o < kBulkChunk) ? bytes - o : kBulkChunk,
                     &tile_bar);
        if ((size_t)tn * sizeof(float2) != bytes) tile[tn - 1] = A.pos[tb + tn - 1];
        bool ok = mbar_wait(&tile_bar, 0, A.wait_ns);
        if (!ok) {
            atomicExch(&g_tile_wait_failed, 1);
            mbar_wait(&tile_bar, 0, A.wait_ns);
        }
        tile_ok = ok ? 1 : 0;
    }
    __syncthreads();
    double part = 0.0;
    if (tile_ok) {
        mbar_wait(&tile_bar, 0, A.wait_ns);
        const Ff d2f = {A.d2hi, A.d2lo};
        const bool unit = A.unit != 0;
        Ff s = {0.f, 0.f};
        // one pair {u, v}: d^2 / delta^q in double-float
        auto term = [&](float2 qu, float2 pv) {
            const Ff r2 = ff_dist2(qu.x, qu.y, pv.x, pv.y);
            if (r2.hi >= 1e-30f && r2.hi <= 1e30f) {
                // d = 1, q = 1 (the defaults): the products by 1 are exact
                // and left out
                s = ff_add(s, unit ? ff_rsqrt(r2) : ff_mul(d2f, ff_rsqrt_pow(r2, A.q)));
            } else {
                const double dx = (double)qu.x - (double)pv.x;
                const double dy = (double)qu.y - (double)pv.y;
                const double dl = sqrt(dx * dx + dy * dy);
                if (dl > 0.0) {
                    double w = 1.0;
                    for (int i = 0; i < A.q; ++i) w *= dl;
                    part += A.d2 / w;
                }
            }
        };
        // rows by batches of kMetBatch: thread t finds row r0 + t's run of
        // ids above u in this tile; a block scan numbers the batch's entries;
        // each warp then takes an equal slice of them (whatever the rows'
        // lengths), lanes striding it and following the row boundaries
        for (int64_t r0 = u0; r0 < u1; r0 += kMetBatch) {
            const int64_t u = r0 + threadIdx.x;
            int64_t lo = 0, hi = 0;
            if (threadIdx.x < kMetBatch && u < u1 && tb + tn > u + 1) {
                // the row's entries in this tile: the whole row in window
                // mode, in tile mode its segment
                lo = A.krow[u];
                if (A.wbase) {
                    hi = A.krow[u + 1];
                } else {
                    lo += A.start[(int64_t)j * A.n + u];
                    hi = lo + A.len[(int64_t)j * A.n + u];
                }
                if (tb <= u) {
                    // the tile holds u: keep the ids above it (binary search)
                    int64_t x = lo, y = hi;
                    while (x < y) {
                        const int64_t mid = (x + y) >> 1;
                        if (A.kcol[mid] <= (uint32_t)u) x = mid + 1; else y = mid;
                    }
                    lo = x;
                }
                if (lo > hi) lo = hi;
            }
            const int len = (int)(hi - lo);
            int incl = len;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int x = __shfl_up_sync(kFull, incl, o);
                if (lane >= o) incl += x;
            }
            if (lane == 31) s_wsum[warp] = incl;
            __syncthreads();
            if (warp == 0) {
                const int x0 = s_wsum[lane];
                int x = x0;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int y = __shfl_up_sync(kFull, x, o);
                    if (lane >= o) x += y;
                }
                s_wsum[lane] = x - x0;  // warps before this one
                if (lane == 31) s_pre[kMetBatch] = x;
            }
            __syncthreads();
            if (threadIdx.x < kMetBatch) {
                s_pre[threadIdx.x] = s_wsum[warp] + incl - len;
                s_off[threadIdx.x] = lo - (s_wsum[warp] + incl - len);
                float2 q = make_float2(0.f, 0.f);
                if (u < u1) q = A.pos[u];
                s_q[threadIdx.x] = q;
            }
            __syncthreads();
            const int total = s_pre[kMetBatch];
            const int beg = (int)((int64_t)total * warp / kMetWarps);
            const int end = (int)((int64_t)total * (warp + 1) / kMetWarps);
            if (beg + lane < end) {
                // the row holding entry beg + lane: the last with s_pre <= it
                int r = 0, hr = kMetBatch - 1;
                while (r < hr) {
                    const int mid = (r + hr + 1) >> 1;
                    if (s_pre[mid] <= beg + lane) r = mid; else hr = mid - 1;
                }
                // sixteen terms of a lane summed as a double-float, then
                // added to its FP64 sum: an inner loop of its own (with a
                // counter tested after every term the compiler formed the
                // FP64 sum each time, and the FP64 pipe was 83% busy: BA
                // n = 100,000, k = 3, 1311 us)
                // The row's bound, offset and position stay in registers
                // until it changes, and the ids and positions of four terms
                // are read before the first of them is formed (BA
                // n = 100,000, k = 3: 860 us with the inner loop alone, 497 now)
                int bound = s_pre[r + 1];
                int64_t off = s_off[r];
                float2 q = s_q[r];
                auto follow = [&](int i) {
                    if (bound <= i) {
                        do bound = s_pre[++r + 1]; while (bound <= i);
                        off = s_off[r];
                        q = s_q[r];
                    }
                };
                int i = beg + lane;
                for (; i + 15 * 32 < end;) {
                    s = {0.f, 0.f};
#pragma unroll 1
                    for (int g4 = 0; g4 < 4; ++g4, i += 128) {
                        float2 qu[4], pv[4];
                        uint32_t id[4];
#pragma unroll
                        for (int c = 0; c < 4; ++c) {
                            follow(i + 32 * c);
                            id[c] = A.kcol[off + (i + 32 * c)];
                            qu[c] = q;
                        }
#pragma unroll
                        for (int c = 0; c < 4; ++c) pv[c] = tile[id[c] - tb];
#pragma unroll
                        for (int c = 0; c < 4; ++c) term(qu[c], pv[c]);
                    }
                    part += (double)s.hi + (double)s.lo;
                }
                s = {0.f, 0.f};
                for (; i < end; i += 32) {
                    follow(i);
                    term(q, tile[A.kcol[off + i] - tb]);
                }
                part += (double)s.hi + (double)s.lo;
            }
            __syncthreads();  // the next batch reuses the arrays
        }
    }
    // fixed-order block sum: lanes, then warps in order
    for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(kFull, part, o);
    if (lane == 0) s_part[warp] = part;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < kMetWarps; ++w) t += s_part[w];
        A.partial[blockIdx.x] = t;
    }
}

// The sum of count values in a fixed order: every 256th by one thread, then
// the threads' sums in a tree (one thread over 456 values took 27 us).
__global__ void __launch_bounds__(256)
sum_partials_kernel(const double* __restrict__ v, int count, double* out)
{
    __shared__ double sh[256];
    double t = 0.0;
    for (int i = threadIdx.x; i < count; i += 256) t += v[i];
    sh[threadIdx.x] = t;
    for (int o = 128; o > 0; o >>= 1) {
        __syncthreads();
        if (threadIdx.x < o) sh[threadIdx.x] += sh[threadIdx.x + o];
    }
    if (threadIdx.x == 0) *out = sh[0];
}

}  // namespace

void invalidate_tile_plans(gila_graph* g)
{
    g->tplan[0].ready = false;
    g->tplan[1].ready = false;
}

gila_status blocked_tile_wait_failed(cudaStream_t st)
{
    int h = 0;
    const int zero = 0;
    GILA_CUDA(cudaMemcpyFromSymbolAsync(&h, g_tile_wait_failed, sizeof(int), 0,
                                        cudaMemcpyDeviceToHost, st));
    GILA_CUDA(cudaStreamSynchronize(st));
    if (h) {
        GILA_CUDA(cudaMemcpyToSymbolAsync(g_tile_wait_failed, &zero, sizeof(int), 0,
                                          cudaMemcpyHostToDevice, st));
        GILA_CUDA(cudaStreamSynchronize(st));
        return fail(GILA_ECUDA, "a tile copy of the iteration kernel did not complete in time");
    }
    return GILA_OK;
}

void free_tile_plans(gila_graph* g)
{
    for (TilePlan& P : g->tplan) {
        cudaFree(P.hubs);
        cudaFree(P.wtile);
        cudaFree(P.rowspan);
        cudaFree(P.sdesc);
        cudaFree(P.deg);
        cudaFree(P.bdesc);
        cudaFree(P.blk);
        cudaFree(P.toff);
        cudaFree(P.tk);
        cudaFree(P.part);
        cudaFree(P.len);
        cudaFree(P.pre_buf);
        cudaFree(P.cut);
        P = TilePlan();
    }
}

// First and last id of every k-hop row (rows are sorted); INT32_MAX and -1
// for empty rows. *widest receives the most ids a row spans.
__global__ void rowspan_kernel(int64_t n, const int64_t* __restrict__ krow,
                               const uint32_t* __restrict__ kcol, int32_t* __restrict__ span,
                               int32_t* __restrict__ widest)
{
    const int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    int32_t wide = 0;
    if (u < n) {
        const int64_t b = krow[u], e = krow[u + 1];
        const int32_t first = b < e ? (int32_t)kcol[b] : INT32_MAX;
        const int32_t last = b < e ? (int32_t)kcol[e - 1] : -1;
        span[2 * u] = first;
        span[2 * u + 1] = last;
        if (b < e) wide = last - first + 1;
    }
    wide = __reduce_max_sync(kFull, wide);
    if ((threadIdx.x & 31) == 0 && wide > 0) atomicMax(widest, wide);
}

// Greedy cut of one tile's rows into ranges of cost at most cap (a range
// takes at least one row) and at most max_rows rows; pre holds the prefix
// sums of the rows' costs (n + 1 values). Returns the number of ranges,
// stopping once it exceeds limit; fills cuts (the range bounds) if given.
int64_t cut_rows(const int64_t* pre, int64_t n, int64_t cap, int64_t limit, int64_t max_rows,
                 std::vector<int32_t>* cuts)
{
    int64_t s = 0, count = 0;
    if (cuts) cuts->assign(1, 0);
    while (s < n) {
        // the last e with pre[e] - pre[s] <= cap, at least s + 1
        int64_t e = (int64_t)(std::upper_bound(pre + s + 1, pre + n + 1, pre[s] + cap) - pre) - 1;
        e = std::min<int64_t>(std::max<int64_t>(e, s + 1), s + max_rows);
        if (cuts) cuts->push_back((int32_t)e);
        if (++count > limit) return count;
        s = e;
    }
    return count;
}

// The same on the host, for window mode (its rows, or slices of rows, as one
// tile): the smallest block cost for which the greedy cut gives at most
// `target` ranges (or the fewest the row limit allows). pre: prefix sums of n
// costs (n + 1 values).
std::vector<int32_t> partition_rows(const std::vector<int64_t>& pre, int64_t n, int64_t target,
                                    int64_t max_rows)
{
    auto count = [&](int64_t cap, int64_t limit) {
        return cut_rows(pre.data(), n, cap, limit, max_rows, nullptr);
    };
    int64_t hi = pre[(size_t)n];  // a cap that all rows fit in: the fewest ranges
    target = std::max<int64_t>(target, count(hi, INT64_MAX));
    int64_t lo = 0;  // count(lo) > target unless single rows already fit
    if (count(lo, target) <= target) hi = lo;
    while (hi - lo > 1) {
        const int64_t mid = lo + (hi - lo) / 2;
        if (count(mid, target) <= target) hi = mid; else lo = mid;
    }
    std::vector<int32_t> cuts;
    cut_rows(pre.data(), n, hi, INT64_MAX, max_rows, &cuts);
    return cuts;
}

// CTAs per SM the blocked grid aims at by default (blocks of equal cost,
// costliest first). Tiles: one wave below 10^8 k-hop entries, where loading
// a tile per CTA is a large part of an iteration (BA n = 100,000, k = 2:
// 0.0374 ms per iteration at 1, 0.0419 at 2); 3 up to 2e9 entries (BA
// n = 100,000, k = 3: 0.140, 0.138, 0.148, 0.157 ms per launch at 2, 3, 4,
// 6); 6 beyond, where a CTA streams tens of MB and the end of the grid
// waits on the slowest (Chung-Lu 1.1e10: 4.38, 4.15, 4.19, 4.19, 4.26 ms
// at 4, 6, 8, 12, 16). Windows: 2 (the mesh, k = 3: 0.0698, 0.0680, 0.0742
// ms at 1, 2, 3).
int64_t default_ctas_per_sm(int64_t nnz_khop, bool window)
{
    if (window) return 2;
    return nnz_khop < 100000000LL ? 1 : nnz_khop < 2000000000LL ? 3 : 6;
}

// CTAs (blocks) the grid aims at: about ctas_per_sm per SM.
int64_t blocks_target(const gila_graph* g, bool window)
{
    const int64_t per_sm = g->tune.ctas_per_sm > 0 ? g->tune.ctas_per_sm
                                                   : default_ctas_per_sm(g->nnz_khop, window);
    return std::max<int64_t>(1, per_sm * (int64_t)sm_count(g->device));
}

// The adjacency rows longer than kHubDeg, which the combine kernel gives a
// block each (fewer than nnz / kHubDeg of them); synchronises.
gila_status plan_hubs(gila_graph* g, TilePlan& P)
{
    const int64_t n = g->n, most = g->nnz_adj / kHubDeg + 1;
    gila_status s = ensure((void**)&P.hubs, &P.hubs_cap, sizeof(int32_t) * ((size_t)most + 1));
    if (s != GILA_OK) return s;
    int* count = P.hubs + most;
    GILA_CUDA(cudaMemsetAsync(count, 0, sizeof(int), g->stream));
    hubs_kernel<<<(unsigned)((n + 255) / 256), 256, 0, g->stream>>>(n, g->row, P.hubs, count);
    count_launch();
    GILA_CUDA(cudaGetLastError());
    GILA_CUDA(cudaMemcpyAsync(&P.nhub, count, sizeof(int), cudaMemcpyDeviceToHost, g->stream));
    GILA_CUDA(cudaStreamSynchronize(g->stream));
    return GILA_OK;
}

// Prefix sums of the cells' padded lengths and costs (P.len, on the device)
// into P.pre: cells + 1 values each.
gila_status prefix_cells(gila_graph* g, TilePlan& P, int64_t cells, size_t esz, bool tiles)
{
    const int64_t nb = (cells + kCellTile - 1) / kCellTile;
    gila_status s;
    if ((s = tiles ? ensure(&P.part, &P.part_cap, 2 * esz * (size_t)cells + 16)
                   : ensure(&P.pre_buf, &P.pre_cap, 16 * ((size_t)cells + 1))) != GILA_OK)
        return s;
    P.pre = (int64_t*)(tiles ? P.part : P.pre_buf);
    if ((s = ensure(&P.cut, &P.cut_cap, sizeof(int64_t) * 2 * (size_t)nb)) != GILA_OK)
        return s;
    int64_t* sums = (int64_t*)P.cut;
    cell_sums_kernel<<<(unsigned)nb, kCellThreads, 0, g->stream>>>(cells, P.len, sums);
    count_launch();
    cell_scan_sums_kernel<<<1, 1024, 0, g->stream>>>(sums, nb);
    count_launch();
    cell_prefix_kernel<<<(unsigned)nb, kCellThreads, 0, g->stream>>>(cells, P.len, sums, P.pre,
                                                                    P.pre + cells + 1);
    count_launch();
    GILA_CUDA(cudaGetLastError());
    return GILA_OK;
}

// Row ranges of every tile, all blocks with at most the same cost: about the
// smallest for which the blocks number at most `target` (or the fewest the
// row limit allows). A grid of about target equal CTAs then ends together,
// where equal row ranges for all tiles left the hubs' tile with CTAs twice
// the mean and one more range than the target sent a few CTAs into a second
// wave (Barabasi-Albert n = 100,000, k = 2: 156 CTAs on 152 SMs, the SMs busy
// 54% of the kernel's time). The cap is searched from below, the mean cost of
// a block, 256 caps at once in steps of 1/128 of it (a cap's walk is a chain
// of dependent loads, 0.2 ms for 150 to 1200 blocks, so many caps at once
// cost what one does). The cuts of every cap are written where they fit
// kCutBytes, else those of the chosen one by another launch.
constexpr size_t kCutBytes = (size_t)64 << 20;

gila_status partition_tiles(gila_graph* g, TilePlan& P, int64_t n, int64_t nt, int64_t target,
                            int64_t max_rows, std::vector<std::vector<int32_t>>& rs)
{
    constexpr int kCaps = 256;
    const int64_t cells = n * nt;
    const int64_t* pre = P.pre + cells + 1;
    target = std::max<int64_t>(target, nt * ((n + max_rows - 1) / max_rows));
    const int64_t stride = target + 2;
    const size_t per_cap = sizeof(int32_t) * (size_t)(nt * stride);
    bool every = per_cap * kCaps <= kCutBytes;
    size_t slots = 0, at_cuts = 0;  // caps whose cuts are written
    gila_status s;
    for (;;) {
        slots = every ? kCaps : 1;
        at_cuts = (kCaps * 12 + sizeof(int) * (size_t)nt * slots + 15) & ~size_t(15);
        s = ensure(&P.cut, &P.cut_cap, at_cuts + per_cap * slots);
        if (s == GILA_OK) break;
        if (!every) return s;
        every = false;
    }
    int64_t* d_caps = (int64_t*)P.cut;
    int* d_counts = (int*)(d_caps + kCaps);
    int* d_tiles = d_counts + kCaps;
    int32_t* d_cuts = (int32_t*)((char*)P.cut + at_cuts);
    int64_t total = 0;
    GILA_CUDA(cudaMemcpyAsync(&total, pre + cells, sizeof(int64_t), cudaMemcpyDeviceToHost, g->stream));
    GILA_CUDA(cudaStreamSynchronize(g->stream));
    std::vector<int64_t> caps(kCaps);
    std::vector<int> counts(kCaps);
    auto count = [&](int used, bool write) -> gila_status {
        GILA_CUDA(cudaMemcpyAsync(d_caps, caps.data(), sizeof(int64_t) * (size_t)used,
                                  cudaMemcpyHostToDevice, g->stream));
        GILA_CUDA(cudaMemsetAsync(d_counts, 0, sizeof(int) * kCaps, g->stream));
        cut_kernel<<<dim3((unsigned)used, (unsigned)((nt + 7) / 8)), 256, 0, g->stream>>>(
            n, (int)nt, pre, d_caps, max_rows, target, d_counts, write ? d_cuts : nullptr, stride,
            write ? d_tiles : nullptr);
        count_launch();
        GILA_CUDA(cudaGetLastError());
        GILA_CUDA(cudaMemcpyAsync(counts.data(), d_counts, sizeof(int) * (size_t)used,
                                  cudaMemcpyDeviceToHost, g->stream));
        GILA_CUDA(cudaStreamSynchronize(g->stream));
        return GILA_OK;
    };
    // at total + 1 every cut reaches the target
    int64_t lo = std::max<int64_t>(1, total / target);
    int pick = kCaps;
    for (int64_t width = lo / 128 + 1; pick == kCaps; width *= 16) {
        for (int i = 0; i < kCaps; ++i)
            caps[(size_t)i] = std::min<int64_t>(lo + width * i, total + 1);
        if ((s = count(kCaps, every)) != GILA_OK) return s;
        pick = 0;
        while (pick < kCaps && counts[(size_t)pick] > target) ++pick;
        lo = caps[kCaps - 1];
        if (pick == kCaps && lo == total + 1) return fail(GILA_ESTATE, "block partition");  // cannot happen
    }
    size_t slot = (size_t)pick;
    if (!every) {
        caps[0] = caps[(size_t)pick];
        if ((s = count(1, true)) != GILA_OK) return s;
        slot = 0;
    }
    std::vector<int> tiles((size_t)nt);
    std::vector<int32_t> cuts((size_t)(nt * stride));
    GILA_CUDA(cudaMemcpyAsync(tiles.data(), d_tiles + slot * (size_t)nt, sizeof(int) * (size_t)nt,
                              cudaMemcpyDeviceToHost, g->stream));
    GILA_CUDA(cudaMemcpyAsync(cuts.data(), d_cuts + slot * (size_t)(nt * stride), per_cap,
                              cudaMemcpyDeviceToHost, g->stream));
    GILA_CUDA(cudaStreamSynchronize(g->stream));
    rs.resize((size_t)nt);
    for (int64_t j = 0; j < nt; ++j)
        rs[(size_t)j].assign(cuts.begin() + j * stride, cuts.begin() + j * stride + tiles[(size_t)j] + 1);
    return GILA_OK;
}

// Shared memory a window-mode CTA needs: the window with the far slot, the
// row directory, and two position-type cells per row.
size_t window_smem(int64_t wmax, int64_t rmax, size_t esz)
{
    return (((size_t)(wmax + 1) * esz + (size_t)(rmax + 1) * 4 + 15) & ~size_t(15)) +
           (size_t)rmax * 2 * esz;
}

// Window mode with a row per lane (rows_kernel): ranges of whole slices with
// a window each, where every window fits, the slices' padding stays within
// kRowPadding of the lists (rows of about equal length), no adjacency row is
// longer than kRowMaxDeg, and every row's neighbours are among its k-hop ids
// (checked while the slices are filled). *done = false leaves the graph to
// the shares of blocked_kernel. krow and span: the lists' offsets and the
// rows' first and last ids, on the host.
gila_status plan_rows(gila_graph* g, size_t esz, TilePlan& P, const std::vector<int64_t>& krow,
                      const std::vector<int32_t>& span, bool* done)
{
    *done = false;
    const int64_t n = g->n, nsl = (n + 31) / 32;
    std::vector<int64_t> arow((size_t)n + 1);
    GILA_CUDA(cudaMemcpyAsync(arow.data(), g->row, sizeof(int64_t) * (n + 1),
                              cudaMemcpyDeviceToHost, g->stream));
    GILA_CUDA(cudaStreamSynchronize(g->stream));
    std::vector<int32_t> sd(4 * (size_t)nsl);
    std::vector<int64_t> pre((size_t)nsl + 1, 0);
    int64_t units = 0;
    for (int64_t s = 0; s < nsl; ++s) {
        int64_t most = 0;
        for (int64_t u = s * 32; u < std::min<int64_t>(n, s * 32 + 32); ++u) {
            most = std::max<int64_t>(most, krow[(size_t)u + 1] - krow[(size_t)u]);
            if (arow[(size_t)u + 1] - arow[(size_t)u] > kRowMaxDeg) return GILA_OK;
        }
        const int64_t steps = (most + 3) / 4;
        if (units + steps > INT32_MAX) return GILA_OK;
        sd[4 * (size_t)s] = (int32_t)units;
        sd[4 * (size_t)s + 1] = (int32_t)steps;
        units += steps;
        // a slice costs its steps and about two more (positions, the move)
        pre[(size_t)s + 1] = pre[(size_t)s] + steps + 2;
    }
    if ((double)units * 128.0 > kRowPadding * (double)g->nnz_khop) return GILA_OK;
    const bool automatic = g->tune.tiled < 0;
    if (automatic && (double)g->nnz_khop > kRowMeanLen * (double)n) return GILA_OK;
    // two CTAs per SM, resident together, at least about 16 steps per warp of
    // a CTA; more and shorter ranges where their windows are too wide for two
    // CTAs' shared memory, or, failing that, for one's
    const int64_t by_work = std::max<int64_t>(1, pre[(size_t)nsl] / (kRowWarps * 16));
    const int64_t base_target = std::min<int64_t>(blocks_target(g, true), by_work);
    std::vector<int32_t> rs;
    std::vector<int64_t> wb;
    int64_t nr = 0, wmax = 0, wsum = 0;
    auto windows = [&](int64_t target) {
        rs = partition_rows(pre, nsl, target, nsl);
        nr = (int64_t)rs.size() - 1;
        wb.assign(2 * (size_t)nr, 0);
        wmax = wsum = 0;
        for (int64_t r = 0; r < nr; ++r) {
            const int64_t u0 = (int64_t)rs[(size_t)r] * 32;
            const int64_t u1 = std::min<int64_t>(n, (int64_t)rs[(size_t)r + 1] * 32);
            int64_t lo = INT64_MAX, hi = -1;
            for (int64_t u = u0; u < u1; ++u) {
                lo = std::min<int64_t>(lo, span[2 * (size_t)u]);
                hi = std::max<int64_t>(hi, span[2 * (size_t)u + 1]);
            }
            if (hi < 0) lo = hi = u0;  // no entries: a one-id window
            const int64_t base = lo & ~int64_t(1);  // even: a 16-byte aligned float2 window
            wb[2 * (size_t)r] = base;
            wb[2 * (size_t)r + 1] = hi - base + 1;
            wmax = std::max<int64_t>(wmax, hi - base + 1);
            wsum += hi - base + 1;
        }
    };
    bool fits = false;
    for (int one = 0; one < 2 && !fits; ++one)
        for (int64_t m = 1; m <= 16 && !fits; m *= 2) {
            windows(base_target * m);
            fits = wmax <= kMaxTile &&  // 16-bit relative ids
                   (size_t)(wmax + 1) * esz <= (one ? (size_t)(kSmemCap - 4096) : kRowWindow);
        }
    if (!fits) return GILA_OK;
    // the windows (from L2) against the id stream
    if (automatic && wsum * (int64_t)esz > kRowWindowBytes * g->nnz_khop) return GILA_OK;
    std::vector<int32_t> bdesc(4 * (size_t)nr, 0);
    for (int64_t r = 0; r < nr; ++r) {
        bdesc[4 * (size_t)r] = rs[(size_t)r] * 32;
        bdesc[4 * (size_t)r + 1] =
            (int32_t)std::min<int64_t>(n, (int64_t)rs[(size_t)r + 1] * 32);
        for (int64_t s = rs[(size_t)r]; s < rs[(size_t)r + 1]; ++s) {
            sd[4 * (size_t)s + 2] = (int32_t)wb[2 * (size_t)r];
            sd[4 * (size_t)s + 3] = (int32_t)wb[2 * (size_t)r + 1];
        }
    }
    gila_status s;
    const size_t sd_bytes = sizeof(int32_t) * sd.size();
    if ((s = ensure((void**)&P.sdesc, &P.sdesc_cap, sd_bytes + 16)) != GILA_OK ||
        (s = ensure((void**)&P.deg, &P.deg_cap, sizeof(uint16_t) * (size_t)n)) != GILA_OK ||
        (s = ensure((void**)&P.tk, &P.tk_cap, (size_t)units * 256 + 16)) != GILA_OK ||
        (s = ensure((void**)&P.bdesc, &P.bdesc_cap, sizeof(int32_t) * bdesc.size())) != GILA_OK ||
        (s = ensure((void**)&P.wtile, &P.wtile_cap, sizeof(int64_t) * wb.size())) != GILA_OK)
        return s;
    int* bad = reinterpret_cast<int*>(reinterpret_cast<char*>(P.sdesc) + sd_bytes);
    GILA_CUDA(cudaMemcpyAsync(P.sdesc, sd.data(), sd_bytes, cudaMemcpyHostToDevice, g->stream));
    GILA_CUDA(cudaMemcpyAsync(P.bdesc, bdesc.data(), sizeof(int32_t) * bdesc.size(),
                              cudaMemcpyHostToDevice, g->stream));
    GILA_CUDA(cudaMemcpyAsync(P.wtile, wb.data(), sizeof(int64_t) * wb.size(),
                              cudaMemcpyHostToDevice, g->stream));
    GILA_CUDA(cudaMemsetAsync(bad, 0, sizeof(int), g->stream));
    rows_fill_kernel<<<(unsigned)((nsl + 3) / 4), 128, 0, g->stream>>>(
        n, nsl, g->row, g->col, g->krow, g->kcol, reinterpret_cast<const int4*>(P.sdesc), P.tk,
        P.deg, bad);
    count_launch();
    GILA_CUDA(cudaGetLastError());
    int h_bad = 0;
    GILA_CUDA(cudaMemcpyAsync(&h_bad, bad, sizeof(int), cudaMemcpyDeviceToHost, g->stream));
    GILA_CUDA(cudaStreamSynchronize(g->stream));  // the host vectors go out of scope too
    if (h_bad) return GILA_OK;
    P.nt = 1;
    P.nb = (int32_t)nr;
    P.tv = (int32_t)wmax;
    P.rmax = 0;
    P.window = P.rows = P.use = true;
    *done = true;
    return GILA_OK;
}

// Window mode: rows are cut into ranges, and each range's rows, whose k-hop
// ids span a window [b, b + len) of consecutive ids narrow enough for
// shared memory (meshes, grids, locality-preserving orders, and every graph
// small enough to fit whole), read their positions from that window. Each
// row then lies wholly in its range's block, so the CTA finishes its rows
// itself (no partials, no second kernel). *fits tells whether every range's
// window fits; `rs` receives the ranges, `wb` the windows (2 nr: first id,
// length).
gila_status plan_window(gila_graph* g, size_t esz, TilePlan& P, bool* fits,
                        std::vector<int32_t>& rs, std::vector<int64_t>& wb, int64_t* wmax_out,
                        int64_t* rmax_out)
{
    *fits = false;
    const int64_t n = g->n;
    gila_status s = ensure((void**)&P.rowspan, &P.rowspan_cap, sizeof(int32_t) * (2 * (size_t)n + 1));
    if (s != GILA_OK) return s;
    int32_t* widest = P.rowspan + 2 * n;
    GILA_CUDA(cudaMemsetAsync(widest, 0, sizeof(int32_t), g->stream));
    rowspan_kernel<<<(unsigned)((n + 255) / 256), 256, 0, g->stream>>>(n, g->krow, g->kcol,
                                                                      P.rowspan, widest);
    count_launch();
    GILA_CUDA(cudaGetLastError());
    // a window holds at least its widest row's ids: most graphs end here
    int32_t span_max = 0;
    GILA_CUDA(cudaMemcpyAsync(&span_max, widest, sizeof(int32_t), cudaMemcpyDeviceToHost, g->stream));
    GILA_CUDA(cudaStreamSynchronize(g->stream));
    if (span_max > kMaxTile || ((size_t)span_max + 1) * esz > (size_t)(kSmemCap - 4096))
        return GILA_OK;
    std::vector<int64_t> krow((size_t)n + 1);
    GILA_CUDA(cudaMemcpyAsync(krow.data(), g->krow, sizeof(int64_t) * (n + 1),
                              cudaMemcpyDeviceToHost, g->stream));
    std::vector<int32_t> span(2 * (size_t)n);
    GILA_CUDA(cudaMemcpyAsync(span.data(), P.rowspan, sizeof(int32_t) * 2 * n,
                              cudaMemcpyDeviceToHost, g->stream));
    GILA_CUDA(cudaStreamSynchronize(g->stream));
    bool done = false;
    if ((s = plan_rows(g, esz, P, krow, span, &done)) != GILA_OK || done) return s;
    std::vector<int64_t> pre((size_t)n + 1, 0);
    for (int64_t u = 0; u < n; ++u)
        pre[(size_t)u + 1] = pre[(size_t)u] + row_cost(krow[(size_t)u + 1] - krow[(size_t)u]);
    // enough ranges for several CTAs per SM, but at least about 16 entries
    // per thread of a CTA (a small graph is one or a few ranges)
    const int64_t by_work = std::max<int64_t>(1, pre[(size_t)n] / ((int64_t)kBThreads * 16));
    rs = partition_rows(pre, n, std::min<int64_t>(blocks_target(g, true), by_work), kMaxRows);
    const int64_t nr = (int64_t)rs.size() - 1;
    wb.assign(2 * (size_t)nr, 0);
    int64_t wmax = 0, rmax = 0;
    for (int64_t r = 0; r < nr; ++r) {
        int64_t lo = INT64_MAX, hi = -1;
        for (int64_t u = rs[(size_t)r]; u < rs[(size_t)r + 1]; ++u) {
            lo = std::min<int64_t>(lo, span[2 * (size_t)u]);
            hi = std::max<int64_t>(hi, span[2 * (size_t)u + 1]);
        }
        if (hi < 0) lo = hi = rs[(size_t)r];  // no entries: a one-id window
        const int64_t base = lo & ~int64_t(1);  // even first id: a 16-byte aligned float2 window
        wb[2 * (size_t)r] = base;
        wb[2 * (size_t)r + 1] = hi - base + 1;
        wmax = std::max<int64_t>(wmax, hi - base + 1);
        rmax = std::max<int64_t>(rmax, (int64_t)(rs[(size_t)r + 1] - rs[(size_t)r]));
        if (wmax > kMaxTile) return GILA_OK;  // 16-bit relative ids
    }
    if (window_smem(wmax, rmax, esz) > (size_t)(kSmemCap - 4096)) return GILA_OK;
    // windows pay where they are narrow: the positions all CTAs load stay
    // below half the bytes of the 16-bit id stream (the mesh: 22 MB of
    // windows for 75 MB of ids, 0.086 ms per iteration against 0.150 plain;
    // a Barabasi-Albert graph of 10,000 vertices at k = 3, whose every range
    // needs the whole graph, about as many window bytes as id bytes: 0.039
    // against 0.030 plain)
    int64_t wsum = 0;
    for (int64_t r = 0; r < nr; ++r) wsum += wb[2 * (size_t)r + 1];
    if (g->tune.tiled < 0 && wsum * (int64_t)esz > g->nnz_khop) return GILA_OK;
    *wmax_out = wmax;
    *rmax_out = rmax;
    *fits = true;
    return GILA_OK;
}

// The block layout shared by tiles and windows: blocks (j, r) for each
// tile j's ranges rs[j], each in share storage (lane_len(L) slots per
// thread; block starts are multiples of 8 slots, 16 bytes); segments padded
// to multiples of 8 entries; segment starts within their block; ids
// rearranged into 16-bit relative ids. wb (window mode, one tile) gives each
// range's window; tiles are [j tv, (j + 1) tv). Blocks are numbered (and
// launched) costliest first, so that in a grid of several waves the CTAs
// that start last are short ones.
gila_status build_layout(gila_graph* g, size_t esz, TilePlan& P, int64_t nt, int64_t tv,
                         const std::vector<std::vector<int32_t>>& rs,
                         const std::vector<int64_t>* wb)
{
    const int64_t n = g->n;
    const int64_t cells = n * nt;
    gila_status s;
    struct Blk {
        int32_t j, r, u0, u1;
        int64_t L, cost;
    };
    std::vector<Blk> bl;
    for (int64_t j = 0; j < nt; ++j) {
        const std::vector<int32_t>& c = rs[(size_t)j];
        for (size_t r = 0; r + 1 < c.size(); ++r)
            bl.push_back({(int32_t)j, (int32_t)r, c[r], c[r + 1], 0, 0});
    }
    {
        // the blocks' entries and costs from the prefix sums
        const size_t m = bl.size();
        std::vector<int32_t> at(4 * m, 0);
        for (size_t b = 0; b < m; ++b) {
            at[4 * b] = bl[b].u0;
            at[4 * b + 1] = bl[b].u1;
            at[4 * b + 2] = bl[b].j;
        }
        std::vector<int64_t> sums(2 * m);
        if ((s = ensure(&P.cut, &P.cut_cap, 32 * m + 32)) != GILA_OK) return s;
        int4* d_at = (int4*)P.cut;
        int64_t* d_sums = (int64_t*)(d_at + m);
        GILA_CUDA(cudaMemcpyAsync(d_at, at.data(), 16 * m, cudaMemcpyHostToDevice, g->stream));
        block_sums_kernel<<<(unsigned)((m + 127) / 128), 128, 0, g->stream>>>(n, cells, (int64_t)m, d_at,
                                                                             P.pre, d_sums);
        count_launch();
        GILA_CUDA(cudaGetLastError());
        GILA_CUDA(cudaMemcpyAsync(sums.data(), d_sums, 16 * m, cudaMemcpyDeviceToHost, g->stream));
        GILA_CUDA(cudaStreamSynchronize(g->stream));
        for (size_t b = 0; b < m; ++b) {
            bl[b].L = sums[2 * b];
            bl[b].cost = sums[2 * b + 1];
        }
    }
    const int64_t nb = (int64_t)bl.size();
    std::vector<int32_t> order((size_t)nb);
    for (int64_t b = 0; b < nb; ++b) order[(size_t)b] = (int32_t)b;
    std::stable_sort(order.begin(), order.end(),
                     [&](int32_t x, int32_t y) { return bl[(size_t)x].cost > bl[(size_t)y].cost; });
    std::vector<int64_t> blk(2 * (size_t)nb), wbb(wb ? 2 * (size_t)nb : 0);
    std::vector<int32_t> bdesc(4 * (size_t)nb);
    int64_t slots = 0;
    for (int64_t b = 0; b < nb; ++b) {
        const Blk& x = bl[(size_t)order[(size_t)b]];
        blk[2 * (size_t)b] = slots;
        blk[2 * (size_t)b + 1] = x.L;
        slots += (int64_t)kBThreads * lane_len((int32_t)x.L);
        bdesc[4 * (size_t)b] = x.u0;
        bdesc[4 * (size_t)b + 1] = x.u1;
        bdesc[4 * (size_t)b + 2] = x.j;
        bdesc[4 * (size_t)b + 3] = 0;
        if (wb) {
            wbb[2 * (size_t)b] = (*wb)[2 * (size_t)x.r];
            wbb[2 * (size_t)b + 1] = (*wb)[2 * (size_t)x.r + 1];
        }
    }
    const int64_t tk_len = slots + kStep + 256 * 4;  // slack: the kernel's ring reads ahead
    if ((s = ensure((void**)&P.toff, &P.toff_cap, sizeof(int32_t) * (size_t)cells)) != GILA_OK)
        return s;
    if ((s = ensure((void**)&P.blk, &P.blk_cap, sizeof(int64_t) * blk.size())) != GILA_OK) return s;
    if ((s = ensure((void**)&P.bdesc, &P.bdesc_cap, sizeof(int32_t) * bdesc.size())) != GILA_OK)
        return s;
    if ((s = ensure((void**)&P.tk, &P.tk_cap, sizeof(uint16_t) * (size_t)tk_len)) != GILA_OK)
        return s;
    if (wb) {
        if ((s = ensure((void**)&P.wtile, &P.wtile_cap, sizeof(int64_t) * wbb.size())) != GILA_OK)
            return s;
        GILA_CUDA(cudaMemcpyAsync(P.wtile, wbb.data(), sizeof(int64_t) * wbb.size(),
                                  cudaMemcpyHostToDevice, g->stream));
    } else if ((s = ensure(&P.part, &P.part_cap, 2 * esz * (size_t)cells)) != GILA_OK) {
        return s;
    }
    GILA_CUDA(cudaMemcpyAsync(P.blk, blk.data(), sizeof(int64_t) * blk.size(),
                              cudaMemcpyHostToDevice, g->stream));
    GILA_CUDA(cudaMemcpyAsync(P.bdesc, bdesc.data(), sizeof(int32_t) * bdesc.size(),
                              cudaMemcpyHostToDevice, g->stream));
    // the slots past each share set to the block's padding id, then the ids
    // ordered for conflict-free gathers, or in ascending order; the slack
    // after the last block (read ahead by the kernel's ring, never used) is zeroed
    const int64_t* wdev = wb ? P.wtile : nullptr;
    const int shorts = g->nnz_khop < 32 * cells ? 1 : 0;  // most segments short
    GILA_CUDA(cudaMemsetAsync(P.tk + slots, 0, sizeof(uint16_t) * (size_t)(tk_len - slots),
                              g->stream));
    if (nb > 0) {
        toff_kernel<<<(unsigned)nb, 256, 0, g->stream>>>(n, reinterpret_cast<const int4*>(P.bdesc),
                                                         P.pre, P.toff);
        count_launch();
        pad_shares_kernel<<<(unsigned)nb, kBThreads, 0, g->stream>>>(P.tk, P.blk, wdev, (int)tv, shorts);
        count_launch();
        GILA_CUDA(cudaGetLastError());
    }
    // CTAs per block, for about 48 per SM
    constexpr int64_t kParts = 48;
    const unsigned parts = (unsigned)std::max<int64_t>(
        1, std::min<int64_t>(64, ((int64_t)sm_count(g->device) * kParts + nb - 1) / std::max<int64_t>(nb, 1)));
    auto layout = [&](auto kernel) -> cudaError_t {
        const size_t smem = sizeof(SpreadSmem) * kSpreadWarps;
        cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        kernel<<<dim3((unsigned)nb, parts), kSpreadWarps * 32, smem, g->stream>>>(
            n, g->krow, g->kcol, (int)tv, wdev, P.len, P.len + cells, P.toff, P.blk,
            reinterpret_cast<const int4*>(P.bdesc), P.tk);
        count_launch();
        return cudaGetLastError();
    };
    if (nb > 0)
        GILA_CUDA(g->tune.bank_spread < 0
                      ? layout(shorts ? block_layout_kernel<16, false, true>
                                      : block_layout_kernel<16, false, false>)
                  : esz == 8 ? layout(shorts ? block_layout_kernel<16, true, true>
                                             : block_layout_kernel<16, true, false>)
                             : layout(shorts ? block_layout_kernel<8, true, true>
                                             : block_layout_kernel<8, true, false>));
    if (!wb) {
        // hubs of the adjacency for the combine kernel (synchronises)
        if ((s = plan_hubs(g, P)) != GILA_OK) return s;
    }
    // the host vectors above go out of scope
    GILA_CUDA(cudaStreamSynchronize(g->stream));
    P.nt = (int32_t)nt;
    P.nb = (int32_t)nb;
    P.use = true;
    return GILA_OK;
}

// Decide whether the blocked path serves g for positions of `esz` bytes and
// build its layout: a window per row range (window mode), or tiles, row
// ranges, block offsets and rearranged ids.
gila_status plan_tiles(gila_graph* g, size_t esz, TilePlan& P)
{
    P.ready = true;
    P.use = false;
    P.window = false;
    P.rows = false;
    const int64_t n = g->n;
    if (n == 0 || g->nnz_khop == 0 || g->tune.tiled == 0) return GILA_OK;
    // tiles for a row directory of rmax entries: positions per tile (one
    // slot for the padding's position) and the number of tiles
    int64_t tv = 0, nt = 0;
    const bool weighted = g->wt64 != nullptr;
    auto geometry = [&](int64_t rmax) {
        // with weights: half a position more per vertex, tiles of a multiple
        // of four vertices (their first weight on a 16-byte boundary)
        const int64_t step = weighted ? 4 : 2;
        const int64_t bytes = (int64_t)esz + (weighted ? (int64_t)esz / 2 : 0);
        int64_t tv_max = (kSmemCap - (rmax + 1) * 4 - 4096) / bytes - 1 - (weighted ? 2 : 0);
        if (g->tune.tile_vertices > 0) tv_max = std::min<int64_t>(tv_max, g->tune.tile_vertices);
        tv_max = std::max<int64_t>(step, std::min<int64_t>(tv_max, kMaxTile) & ~(step - 1));
        nt = (n + tv_max - 1) / tv_max;
        tv = std::min<int64_t>(tv_max, ((n + nt - 1) / nt + step - 1) & ~(step - 1));
    };
    geometry(kMaxRows);
    const int min_seg = g->tune.min_segment;  // 0: no limit
    const double avg_seg = (double)g->nnz_khop / ((double)n * (double)nt);
    {
        // window mode wherever every range's window fits shared memory (a
        // tile size set by the tuning asks for tiles instead); automatic mode
        // leaves lists below 4 10^6 entries to the plain kernel, which
        // spreads small graphs over more SMs (32 x 32 grid, FP64: 0.017 ms
        // plain, 0.105 ms in one window; triangulated 200 x 200 mesh, k = 3:
        // 0.015 against 0.021)
        if (!weighted && g->tune.tile_vertices <= 0 &&
            (g->tune.tiled > 0 || g->nnz_khop >= kBlockedMinNnz)) {
            bool fits = false;
            std::vector<int64_t> wb;
            std::vector<int32_t> rs;
            int64_t wmax = 0, rmax = 0;
            gila_status s = plan_window(g, esz, P, &fits, rs, wb, &wmax, &rmax);
            if (s != GILA_OK || P.rows) return s;
            if (fits) {
                if ((s = ensure((void**)&P.len, &P.len_cap, 2 * sizeof(int32_t) * (size_t)n)) != GILA_OK)
                    return s;
                rowlen_kernel<<<(unsigned)((n + 255) / 256), 256, 0, g->stream>>>(n, g->krow, P.len,
                                                                                P.len + n);
                count_launch();
                if ((s = prefix_cells(g, P, n, esz, false)) != GILA_OK) return s;
                if ((s = build_layout(g, esz, P, 1, 0, {rs}, &wb)) != GILA_OK) return s;
                P.window = true;
                P.tv = (int32_t)wmax;
                P.rmax = (int32_t)rmax;
                return GILA_OK;
            }
        }
    }
    // automatic mode: tiles from 4 10^6 k-hop entries on (BA n = 100,000,
    // k = 2, 1.4e7 entries in segments of 36: 0.0493 ms per iteration
    // against 0.0609 plain; BA n = 333,334, k = 2, segments of 12: 0.183
    // against 0.209). FP64 follows the same rule (its tiles hold half as
    // many positions): on BA k = 3 blocked 5.14 ms vs plain 6.03 ms
    // (weighted graphs, whose windows are not tried, stay with the plain
    // kernel where most segments would be nearly empty)
    const bool tiles_pay = !(g->tune.tiled < 0 && avg_seg < std::max(min_seg, weighted ? kWeightedMinSeg : 0));
    if (!tiles_pay || (g->tune.tiled < 0 && g->nnz_khop < kBlockedMinNnz)) return GILA_OK;
    // many rows: where 4096-row ranges alone make more blocks than the CTA
    // target, a larger directory (smaller tiles) gives fewer blocks, each
    // loading its tile once; but only for segments long enough that the
    // extra tiles add little padding (BA n = 333,334, k = 3, 323 entries a
    // segment: 0.702 -> 0.588 ms per iteration with 8192-row ranges; k = 2,
    // 12 entries: 0.148 -> 0.170 ms, so it keeps 4096)
    int64_t rmax = kMaxRows;
    const int64_t target = blocks_target(g, false);
    while (rmax < kMaxRowsTiles && (n + rmax - 1) / rmax * nt > target &&
           (double)g->nnz_khop >= 64.0 * (double)n * (double)nt) {
        rmax *= 2;
        geometry(rmax);
    }
    const int64_t cells = n * nt;
    gila_status s = ensure((void**)&P.len, &P.len_cap, 2 * sizeof(int32_t) * (size_t)cells);
    if (s != GILA_OK) return s;
    seglen_kernel<<<(unsigned)((cells + 255) / 256), 256, 0, g->stream>>>(
        n, g->krow, g->kcol, (int)nt, (int)tv, P.len, P.len + cells);
    count_launch();
    GILA_CUDA(cudaGetLastError());
    // each tile's row ranges: blocks of about equal cost (padded entries +
    // a per-row term), at most rmax rows each, about ctas_per_sm per SM
    if ((s = prefix_cells(g, P, cells, esz, true)) != GILA_OK) return s;
    // the block count: at least 5% above what the row limit alone makes,
    // so that a tile with more entries than the others (the hubs' ids) can
    // still be cut finer, and whole waves of one CTA per SM, since blocks of
    // equal cost end together (BA n = 333,334, k = 3: 574 row-limited blocks
    // against a target of 456: 1.27 ms per iteration with no room, 0.63 with
    // 631 blocks, 0.59 with 608)
    const int64_t sms = sm_count(g->device);
    const int64_t floor_blocks = (n + rmax - 1) / rmax * nt;
    const int64_t want = std::max<int64_t>(target, (floor_blocks * 21 + 19) / 20);
    const int64_t tgt = (want + sms - 1) / sms * sms;
    std::vector<std::vector<int32_t>> rs;
    if ((s = partition_tiles(g, P, n, nt, tgt, rmax, rs)) != GILA_OK) return s;
    if ((s = build_layout(g, esz, P, nt, tv, rs, nullptr)) != GILA_OK) return s;
    P.tv = (int32_t)tv;
    P.rmax = (int32_t)rmax;
    return GILA_OK;
}

bool blocked_auto_applies(int64_t n, int64_t nnz_khop, size_t esz, const gila_tuning& tune)
{
    if (n == 0 || nnz_khop == 0 || tune.tiled == 0) return tune.tiled == 1 && n > 0;
    if (tune.tiled == 1) return true;
    int64_t tv_max = kTileBudget / (int64_t)esz - 1;  // one slot for the padding's position
    if (tune.tile_vertices > 0) tv_max = std::min<int64_t>(tv_max, tune.tile_vertices);
    tv_max = std::max<int64_t>(2, std::min<int64_t>(tv_max, kMaxTile) & ~int64_t(1));
    const int64_t nt = (n + tv_max - 1) / tv_max;
    return nnz_khop >= kBlockedMinNnz &&
           (double)nnz_khop / ((double)n * (double)nt) >= (double)tune.min_segment;
}

// Repulsion weights with exponents other than Fruchterman-Reingold's are
// applied by the plain kernel only.
static bool plain_weights(const gila_graph* g, const gila_params* prm)
{
    return g->wt64 && !(prm->p == 2 && prm->q == 1);
}

gila_status prepare_iteration(gila_graph* g, const gila_params* prm)
{
    if (prm->precision == GILA_FP64_ORDERED || g->n == 0 || plain_weights(g, prm)) return GILA_OK;
    TilePlan& P = g->tplan[is_f64(prm->precision) ? 1 : 0];
    return P.ready ? GILA_OK : plan_tiles(g, is_f64(prm->precision) ? 16 : 8, P);
}

gila_status launch_blocked(gila_graph* g, const gila_params* prm, double t, const void* pos_in,
                           void* pos_out, void* disp_out, bool* handled)
{
    *handled = false;
    if (prm->precision == GILA_FP64_ORDERED || g->n == 0 || plain_weights(g, prm)) return GILA_OK;
    const size_t esz = is_f64(prm->precision) ? 16 : 8;
    TilePlan& P = g->tplan[esz == 16 ? 1 : 0];
    if (!P.ready) {
        gila_status s = plan_tiles(g, esz, P);
        if (s != GILA_OK) return s;
    }
    if (!P.use || ((uintptr_t)pos_in & 15) != 0) return GILA_OK;
    if (P.rows) {
        RowsArgs R;
        R.tk = P.tk;
        R.sdesc = reinterpret_cast<const int4*>(P.sdesc);
        R.deg = P.deg;
        R.bdesc = reinterpret_cast<const int4*>(P.bdesc);
        R.wbase = P.wtile;
        R.n = g->n;
        R.q = prm->q;
        R.p = prm->p;
        R.c = force_consts(prm->d, t);
        R.pos = pos_in;
        R.pos_out = pos_out;
        R.disp_out = disp_out;
        R.wait_ns = g->wait_test ? kTestWaitNs : kWaitNs;
        R.skip_copy = g->wait_test ? 1 : 0;
        const bool fr = prm->p == 2 && prm->q == 1;
        cudaError_t e;
        switch (prm->precision) {
        case GILA_FP64:
            e = fr ? launch_rows<double, kFR, false>(g, R, P) : launch_rows<double, kGeneric, false>(g, R, P);
            break;
        case GILA_FP32_COMPENSATED:
            e = fr ? launch_rows<float, kFR, true>(g, R, P) : launch_rows<float, kGeneric, true>(g, R, P);
            break;
        default:
            e = fr ? launch_rows<float, kFR, false>(g, R, P) : launch_rows<float, kGeneric, false>(g, R, P);
            break;
        }
        if (e != cudaSuccess) return cuda_fail(e, "rows_kernel");
        *handled = true;
        return GILA_OK;
    }
    BlockedArgs B;
    B.tk = P.tk;
    B.toff = P.toff;
    B.blk = P.blk;
    B.bdesc = reinterpret_cast<const int4*>(P.bdesc);
    B.n = g->n;
    B.nt = P.nt;
    B.tv = P.tv;
    B.q = prm->q;
    B.pos = pos_in;
    B.part = P.part;
    B.wait_ns = g->wait_test ? kTestWaitNs : kWaitNs;
    B.skip_copy = g->wait_test ? 1 : 0;
    B.wbase = P.window ? P.wtile : nullptr;
    B.wmax = P.window ? P.tv : 0;
    B.rmax = P.rmax;
    B.row = g->row;
    B.col = g->col;
    B.c = force_consts(prm->d, t);
    B.p = prm->p;
    B.pos_out = pos_out;
    B.disp_out = disp_out;
    // FP32 steps warp-uniform by default (measured against the divergent
    // schedule: Chung-Lu n = 250,000, k = 3, 4.88 vs 4.96 ms per launch;
    // Barabasi-Albert n = 100,000, k = 3, 0.172 vs 0.186 ms). The kernel
    // keeps both schedules: with the divergent one compiled beside it the
    // uniform schedule itself measured faster (4.88 vs 5.08 ms on Chung-Lu)
    B.uniform = g->tune.step_schedule >= 0 ? 1 : 0;
    B.wt = !g->wt64 ? nullptr : esz == 16 ? (const void*)g->wt64 : (const void*)g->wt32;
    CombineArgs C;
    C.row = g->row;
    C.col = g->col;
    C.n = g->n;
    C.nt = P.nt;
    C.c = B.c;
    if (B.wt) C.c.d2 = C.c.d2f = 1;  // in the weighted terms already
    C.p = prm->p;
    C.pos_in = pos_in;
    C.part = P.part;
    C.pos_out = pos_out;
    C.disp_out = disp_out;
    C.hubs = P.hubs;
    C.nhub = P.nhub;
    C.nreg = (int32_t)((g->n * kCombineLanes + kCombineThreads - 1) / kCombineThreads);
    const int grid = P.nb;
    const size_t smem = P.window ? window_smem(P.tv, P.rmax, esz)
                        : B.wt   ? weights_at(P.tv, P.rmax, esz) + (size_t)(P.tv + 1) * (esz / 2)
                                 : (size_t)(P.tv + 1) * esz + (size_t)(P.rmax + 1) * 4;
    const bool fr = (prm->p == 2 && prm->q == 1);
    const bool w = P.window;
    cudaError_t e;
    switch (prm->precision) {
    case GILA_FP64:
        e = fr ? launch_pair<double, kFR, false>(g, B, C, grid, smem, g->stream, g->device, w)
               : launch_pair<double, kGeneric, false>(g, B, C, grid, smem, g->stream, g->device, w);
        break;
    case GILA_FP32_COMPENSATED:
        e = fr ? launch_pair<float, kFR, true>(g, B, C, grid, smem, g->stream, g->device, w)
               : launch_pair<float, kGeneric, true>(g, B, C, grid, smem, g->stream, g->device, w);
        break;
    default:
        e = fr ? launch_pair<float, kFR, false>(g, B, C, grid, smem, g->stream, g->device, w)
               : launch_pair<float, kGeneric, false>(g, B, C, grid, smem, g->stream, g->device, w);
        break;
    }
    if (e != cudaSuccess) return cuda_fail(e, "blocked_kernel");
    *handled = true;
    return GILA_OK;
}

int64_t blocked_metric_partials(const gila_graph* g, const gila_params* prm, const void* pos)
{
    const TilePlan& P = g->tplan[0];
    if (is_f64(prm->precision) || !P.ready || !P.use || g->n == 0 || g->wt64) return 0;
    if (((uintptr_t)pos & 15) != 0) return 0;
    // the tile (or window) beside the kernel's own shared arrays; a larger
    // window leaves the term to the generic reduction
    if (((size_t)P.tv + 1) * sizeof(float2) > (size_t)kMetSmemMax) return 0;
    return P.nb;
}

gila_status blocked_khop_metric(gila_graph* g, const gila_params* prm, const void* pos,
                                double* partials, double* rep_total)
{
    const TilePlan& P = g->tplan[0];
    const size_t smem = ((size_t)P.tv + 1) * sizeof(float2);
    const int grid = P.nb;
    const double d2 = prm->d * prm->d;
    MetricArgs M;
    M.krow = g->krow;
    M.len = P.window ? nullptr : P.len;
    M.start = P.window ? nullptr : P.len + g->n * P.nt;
    M.kcol = g->kcol;
    M.bdesc = reinterpret_cast<const int4*>(P.bdesc);
    M.wbase = P.window ? P.wtile : nullptr;
    M.n = g->n;
    M.nt = P.nt;
    M.tv = P.tv;
    M.d2 = d2;
    M.d2hi = (float)d2;
    M.d2lo = (float)(d2 - (double)M.d2hi);
    M.unit = prm->d == 1.0 && prm->q == 1;
    M.q = prm->q;
    M.pos = reinterpret_cast<const float2*>(pos);
    M.partial = partials;
    M.wait_ns = kWaitNs;
    static std::atomic<uint64_t> configured{0};
    const uint64_t bit = 1ull << (g->device & 63);
    if (!(configured.load() & bit)) {
        GILA_CUDA(cudaFuncSetAttribute(khop_metric_kernel,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       kMetSmemMax));
        configured.fetch_or(bit);
    }
    khop_metric_kernel<<<grid, kMetThreads, smem, g->stream>>>(M);
    count_launch();
    sum_partials_kernel<<<1, 256, 0, g->stream>>>(partials, grid, rep_total);
    count_launch();
    GILA_CUDA(cudaGetLastError());
    return GILA_OK;
}

}  // namespace gila
