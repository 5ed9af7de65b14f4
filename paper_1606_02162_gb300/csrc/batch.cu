// Batched layouts: many graphs in one persistent launch.
//
// A batch is the disjoint union of its graphs (ids offset per graph), so one
// k-hop build serves all of them. The layout of every graph then runs inside
// a single CTA, or a cluster of CTAs, from its first to its last iteration:
// the placement is staged in shared memory (two buffers, Jacobi), the graph's
// k-hop rows are streamed (small enough to stay in L2 across iterations), and
// iterations are separated by a block barrier or an exchange within the
// cluster, so no grid-wide barrier and no per-iteration launch exists. CTAs
// take graphs from global counters, largest first. Graphs of short rows take
// a lane per row (batch_rows_kernel); the others take 4, 8, 16 or 32 lanes per
// vertex by their own mean row length (batch_kernel), and those too large for
// shared memory iterate on two global buffers in the same way. A graph's
// result does not depend on the other graphs of the batch. The temperature of
// each graph follows its own schedule: the default t0 uses that graph's n
// (and, for geometric cooling, the aspect of its own initial bounding box).
#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstring>
#include <numeric>
#include <string>
#include <type_traits>
#include <vector>

#include "device_util.cuh"
#include "force.cuh"
#include "gila_impl.h"

struct gila_batch {
    gila_graph* g = nullptr;  // disjoint union of the graphs
    int32_t count = 0;
    std::vector<int64_t> voff_h;  // vertex offsets, count + 1
    std::vector<int32_t> order_h; // graphs, largest first
    int64_t* voff = nullptr;
    int32_t* order = nullptr;     // graphs in processing order
    int* work = nullptr;          // next position in `order`
    double* geo = nullptr;        // 0.93^i table
    size_t geo_cap = 0;
    void* tmp = nullptr;          // second global placement for graphs beyond shared memory
    size_t tmp_cap = 0;
    void* pos[2] = {nullptr, nullptr};  // placement buffers of the host-memory calls
    size_t pos_cap[2] = {0, 0};
    double* stage = nullptr;
    size_t stage_cap = 0;
    int64_t max_n = 0;
    cudaStream_t user = nullptr;   // caller's stream
    cudaStream_t own = nullptr;    // capture stream
    cudaEvent_t ev_in = nullptr, ev_out = nullptr;
    cudaGraphExec_t exec = nullptr;
    std::vector<unsigned char> exec_key;  // arguments the captured graph was made with
    gila_batch_tuning tune = {0, 0, 0, 0, 0};
    // row-per-lane plan of the current k-hop lists, by position width
    // (0: float2, 1: double2; the widths share the arrays, see batch_plan)
    int64_t plan_serial = -1;      // the build it was made for
    std::vector<int32_t> big[2], small[2], rest[2];  // graphs by the form that serves them
    int64_t max_rows_n[2] = {0, 0};                  // largest graph of big and small
    int cluster[2] = {1, 1};                         // CTAs of a cluster
    int32_t* rorder[2] = {nullptr, nullptr};         // big, small, rest
    int32_t* soff = nullptr;
    int32_t* sgraph = nullptr;
    int32_t* base = nullptr;
    int32_t* units = nullptr;
    uint8_t* skip = nullptr;       // 2 count: skip, bad
    int2* sdesc = nullptr;
    uint16_t* deg = nullptr;
    uint16_t* perm = nullptr;
    uint16_t* rank = nullptr;
    uint16_t* cuts = nullptr;
    uint16_t* tk = nullptr;
    size_t tk_cap = 0;
    int* wait_failed = nullptr;    // host memory the kernel writes: a cluster's wait ran out
    int wait_test = 0;             // test hook: clusters push nothing, so that their waits run out
    cudaStream_t side = nullptr;   // capture fork: the group kernel beside the row-per-lane one
    cudaEvent_t ev_fork = nullptr, ev_join = nullptr;
};

namespace gila {

namespace {

struct BatchArgs {
    const int64_t* voff;
    const int32_t* order;
    int32_t count;
    const int64_t* row;
    const int32_t* col;
    const int64_t* krow;
    const uint32_t* kcol;
    int* work;
    const double* geo;
    int iters, schedule;
    double d, t0;
    int p, q;
    void* pos;
    void* tmp;
    int smem_verts;
    int g4_max, g8_max, g16_max;
};

template <class T>
__device__ __forceinline__ void capped(T t, T fx, T fy, T& mx, T& my)
{
    const T fn = sqrt(fx * fx + fy * fy);
    mx = fx;
    my = fy;
    if (fn > t) {
        const T sc = t / fn;
        mx = fx * sc;
        my = fy * sc;
    }
}

// One CTA lays out one graph at a time; see the file comment.
template <class T, int MODEL, bool COMP>
__global__ void __launch_bounds__(1024) batch_kernel(const BatchArgs A)
{
    using P2 = typename V2<T>::type;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ int s_g;
    __shared__ double s_box[32][4];
    P2* sbuf0 = reinterpret_cast<P2*>(smem_raw);
    P2* sbuf1 = sbuf0 + A.smem_verts;
    P2* gpos = reinterpret_cast<P2*>(A.pos);
    P2* gtmp = reinterpret_cast<P2*>(A.tmp);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (;;) {
        if (threadIdx.x == 0) s_g = atomicAdd(A.work, 1);
        __syncthreads();
        const int gi = s_g;
        __syncthreads();
        if (gi >= A.count) break;
        const int gid = A.order[gi];
        const int64_t v0 = A.voff[gid];
        const int64_t n = A.voff[gid + 1] - v0;
        if (n == 0) continue;
        const int64_t nnz = A.krow[v0 + n] - A.krow[v0];
        const int64_t avg = nnz / n;
        const int G = avg <= A.g4_max ? 4 : avg <= A.g8_max ? 8 : avg <= A.g16_max ? 16 : 32;
        const bool in_smem = n <= A.smem_verts;
        P2* cur = in_smem ? sbuf0 : gpos + v0;
        P2* nxt = in_smem ? sbuf1 : gtmp + v0;
        if (in_smem)
            for (int64_t i = threadIdx.x; i < n; i += blockDim.x) cur[i] = gpos[v0 + i];
        __syncthreads();
        // initial temperature of this graph
        double t0 = A.t0;
        if (!(t0 > 0.0)) {
            if (A.schedule != GILA_COOL_GEOMETRIC) {
                t0 = 0.1 * sqrt((double)n);
            } else {
                double x0 = INFINITY, x1 = -INFINITY, y0 = INFINITY, y1 = -INFINITY;
                for (int64_t i = threadIdx.x; i < n; i += blockDim.x) {
                    const P2 p = cur[i];
                    x0 = fmin(x0, (double)p.x);
                    x1 = fmax(x1, (double)p.x);
                    y0 = fmin(y0, (double)p.y);
                    y1 = fmax(y1, (double)p.y);
                }
                for (int o = 16; o > 0; o >>= 1) {
                    x0 = fmin(x0, __shfl_xor_sync(kFull, x0, o));
                    x1 = fmax(x1, __shfl_xor_sync(kFull, x1, o));
                    y0 = fmin(y0, __shfl_xor_sync(kFull, y0, o));
                    y1 = fmax(y1, __shfl_xor_sync(kFull, y1, o));
                }
                if (lane == 0) {
                    s_box[warp][0] = x0;
                    s_box[warp][1] = x1;
                    s_box[warp][2] = y0;
                    s_box[warp][3] = y1;
                }
                __syncthreads();
                x0 = s_box[0][0];
                x1 = s_box[0][1];
                y0 = s_box[0][2];
                y1 = s_box[0][3];
                for (int w = 1; w < (int)(blockDim.x >> 5); ++w) {
                    x0 = fmin(x0, s_box[w][0]);
                    x1 = fmax(x1, s_box[w][1]);
                    y0 = fmin(y0, s_box[w][2]);
                    y1 = fmax(y1, s_box[w][3]);
                }
                __syncthreads();
                const double w = x1 - x0, h = y1 - y0;
                const double a = (w > 0.0 && h > 0.0) ? h / w : 1.0;
                t0 = sqrt((double)n * A.d / a);
            }
        }
        Rep<T, MODEL, COMP, kSrcGeneric> f;
        f.src.base = (uint32_t)v0;
        f.d2 = (T)(A.d * A.d);
        f.q = A.q;
        Att<T, MODEL, COMP, kSrcGeneric> att;
        att.src.base = (uint32_t)v0;
        att.inv_d = (T)(1.0 / A.d);
        att.p = A.p;
        const int groups = blockDim.x / G;
        const int grp = threadIdx.x / G, gl = threadIdx.x % G;
        for (int it = 0; it < A.iters; ++it) {
            const double td = A.schedule == GILA_COOL_GEOMETRIC
                                  ? t0 * A.geo[it]
                                  : t0 * (double)(A.iters - it) / (double)A.iters;
            const T t = (T)td;
            // ids are global; the buffer holds this graph's vertices from 0
            f.src.pos = cur;
            att.src.pos = cur;
            for (int64_t vb = 0; vb < n; vb += groups) {
                const int64_t v = vb + grp;
                const bool live = v < n;
                Acc<T, COMP> a;
                P2 pu;
                pu.x = T(0);
                pu.y = T(0);
                if (live) {
                    pu = cur[v];
                    f.xu = pu.x;
                    f.yu = pu.y;
                    att.xu = pu.x;
                    att.yu = pu.y;
                    // lanes take entries by their place in the row, so the
                    // order does not depend on where the row sits in the batch
                    row_sum_rel(A.kcol, A.krow[v0 + v], A.krow[v0 + v + 1], gl, G, f, a);
                    row_sum_rel(reinterpret_cast<const uint32_t*>(A.col), A.row[v0 + v],
                                A.row[v0 + v + 1], gl, G, att, a);
                }
                a.group_reduce(G);
                if (live && gl == 0) {
                    T mx, my;
                    capped<T>(t, a.fx(), a.fy(), mx, my);
                    P2 o;
                    o.x = pu.x + mx;
                    o.y = pu.y + my;
                    nxt[v] = o;
                }
            }
            __syncthreads();
            P2* s = cur;
            cur = nxt;
            nxt = s;
        }
        // the result goes to the caller's buffer
        if (in_smem || cur != gpos + v0)
            for (int64_t i = threadIdx.x; i < n; i += blockDim.x) gpos[v0 + i] = cur[i];
        __syncthreads();
    }
}

// Row-per-lane form of the batched layout, for graphs of short rows. At plan
// time (once per k-hop build) each graph's vertices are sorted by row length,
// and 32 consecutive ones of that order form a slice, stored step-major (four
// 16-bit ids of every lane, 256 bytes a step) and padded to the slice's
// longest row with the row's own id (at distance 0, where a term is zero,
// whatever the coordinates). A row's first ids are its neighbours,
// whose attraction is formed from the same shared-memory positions. A lane
// sums its row in registers and moves its vertex: no reduction over lanes, no
// lane without a row in the finish (a square root and a division per vertex,
// which a group of eight lanes issued for four vertices at a time), and ids
// that arrive as 16-byte-aligned streams ahead of their use.
//
// In the compensated mode every term goes through a two-sum, as in the group
// kernel (sixteen terms summed plainly before each had three times its error).
// In FP32 a row is added in four sums that are joined after sixteen ids, as many
// partial sums as the group kernel's lanes keep: one sum over a row loses more
// (a row of 2^24 and 63 ones loses 63 with one sum, 3 here, at 0.6% of the time).
//
// CTAs come in clusters of 1, 2, 4 or 8. A graph that would keep one CTA busy
// for longer than its share of the batch is taken by a whole cluster: every
// CTA with slices holds the placement, computes a contiguous part of the slices
// (equal steps), and pushes its new positions into the others' shared memory
// with bulk copies that complete on their mbarriers, one mbarrier per parity
// of the iteration. A CTA needs the positions of every other one to go on, so
// that it is at most one iteration ahead of any: two mbarriers suffice, and a
// buffer is overwritten only after its last reader. A CTA whose part is empty
// (fewer slices than CTAs, or one slice that outweighs several shares) pushes
// nothing, so that nobody would wait for it: it takes no part in the graph and
// nothing is pushed to it. After the large graphs each CTA
// takes small ones on its own. The order of a row's additions is the same in
// every case and depends on the graph alone.
//
// Against groups of lanes per vertex (batch_kernel, which the longer rows
// keep), whose bound was the latency of one group's chain (offsets, ids,
// positions, reduction) and, in FP64, lanes without work on the two FP64
// operations a clock of an SM: 500 graphs of 50..5000 vertices, k = 2, 50
// iterations in FP32 6.5 -> 0.62 ms, 3000 graphs 9.2 -> 1.6 ms (30
// iterations), 250 graphs in FP64 20.8 -> 3.6 ms (20 iterations; its FP64
// pipe is 63% busy, the FP32 form issues in 52% of the cycles, the rest mostly
// the barrier between iterations).
constexpr int kBrCluster = 8;             // largest cluster
constexpr int kBrBins = 1024;             // row lengths told apart by the sort
constexpr int64_t kBrMeanLen = 64;        // longest mean row taken
constexpr double kBrPadding = 2.0;        // most slots per entry
constexpr int kBrAhead = 4;               // steps of ids in registers ahead
constexpr int kBrSmem = 227 * 1024 - 2048;
// fewest slices worth a cluster: below, an exchange an iteration costs more
// than the split saves (FP64 slices take about ten times as long)
constexpr int64_t kBrBigSlices[2] = {16, 4};
constexpr uint64_t kBrWaitNs = 1000000000ull;    // bound on a wait for peers' positions
constexpr uint64_t kBrTestWaitNs = 1000000ull;   // ... while the wait test hook is on

struct BatchRowsArgs {
    const int64_t* voff;
    const int32_t* order;    // large graphs, then small ones, largest first
    int32_t nbig, nall;
    const int32_t* soff;     // first slice of every graph
    const int2* sdesc;       // per slice: start in tk (units of 128 ids), steps
    const uint16_t* deg;     // adjacency degrees in sorted order
    const uint16_t* perm;    // vertex of each place of the sorted order
    const uint16_t* cuts;    // kBrCluster + 1 slice bounds per graph
    const uint16_t* tk;
    int* work;               // next large, next small
    const double* geo;
    int iters, schedule;
    double d, t0;
    ForceConsts c;           // its t is unused: every graph cools on its own
    int p, q;
    void* pos;
    int stride;              // positions per buffer, far slot included (even)
    uint64_t wait_ns;
    int skip_push;           // test hook: announce the peers' positions but push none
    int* wait_failed;        // the batch's, in host memory: set when a wait ran out
};

__device__ __forceinline__ uint32_t cluster_rank()
{
    uint32_t r;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}

__device__ __forceinline__ void cluster_sync()
{
    asm volatile("barrier.cluster.arrive.release;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
}

__device__ __forceinline__ uint32_t cluster_size()
{
    uint32_t r;
    asm("mov.u32 %0, %%cluster_nctaid.x;" : "=r"(r));
    return r;
}

// Address in CTA `rank`'s shared memory of the same place as `a` in this one's.
__device__ __forceinline__ uint32_t cluster_map(uint32_t a, uint32_t rank)
{
    uint32_t r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
    return r;
}

// Bulk copy from this CTA's shared memory to another's, completing on the
// other's mbarrier.
__device__ __forceinline__ void bulk_s2s(uint32_t dst_cluster, uint32_t src, uint32_t bytes,
                                         uint32_t bar_cluster)
{
    asm volatile(
        "cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::
            "r"(dst_cluster),
        "r"(src), "r"(bytes), "r"(bar_cluster)
        : "memory");
}

template <class T, int MODEL, bool COMP>
__global__ void __launch_bounds__(1024) batch_rows_kernel(const BatchRowsArgs A)
{
    using P2 = typename V2<T>::type;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ __align__(8) uint64_t s_bar[2];
    __shared__ int s_g;
    __shared__ double s_t0;
    __shared__ T s_t[2];  // this and the next iteration's temperature
    __shared__ double s_box[32][4];
    P2* const buf0 = reinterpret_cast<P2*>(smem_raw);
    P2* const buf1 = buf0 + A.stride;
    P2* const gpos = reinterpret_cast<P2*>(A.pos);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    const uint32_t rank = cluster_rank(), csize = cluster_size();
    if (threadIdx.x == 0) {
        mbar_init(&s_bar[0], 1);
        mbar_init(&s_bar[1], 1);
    }
    uint32_t phase = 0;  // bit i: parity of the phase of s_bar[i] that this CTA waits for next
    bool gave_up = false;  // a wait of this thread ran out

    // one graph, its slices [s0 + ca, s0 + cb) on this CTA
    auto layout = [&](int gid, bool big) {
        const int64_t v0 = A.voff[gid];
        const int n = (int)(A.voff[gid + 1] - v0);
        const int npad = (n + 31) & ~31;
        const int s0 = A.soff[gid];
        const int ns = npad >> 5;
        const uint16_t* cuts = A.cuts + (kBrCluster + 1) * (int64_t)gid;
        const int part = kBrCluster / (int)csize;  // eighths of the graph per CTA
        const int ca = big ? cuts[rank * part] : 0;
        const int cb = big ? cuts[(rank + 1) * part] : ns;
        if (ca == cb) return;  // no slices: no part in the exchange below
        uint32_t peers = 0;    // the other CTAs of the cluster that have slices, a bit each
        for (uint32_t r = 0; big && r < csize; ++r)
            if (r != rank && cuts[(r + 1) * part] > cuts[r * part]) peers |= 1u << r;
        const uint16_t* perm = A.perm + v0;
        for (int i = threadIdx.x; i < n; i += blockDim.x) buf0[i] = gpos[v0 + perm[i]];
        if (threadIdx.x == 0) {
            P2 far;
            far.x = FarSlot<T>::v;
            far.y = FarSlot<T>::v;
            buf0[npad] = far;
            buf1[npad] = far;
        }
        __syncthreads();
        // initial temperature of this graph
        if (!(A.t0 > 0.0) && A.schedule == GILA_COOL_GEOMETRIC) {
            double x0 = INFINITY, x1 = -INFINITY, y0 = INFINITY, y1 = -INFINITY;
            for (int i = threadIdx.x; i < n; i += blockDim.x) {
                const P2 p = buf0[i];
                x0 = fmin(x0, (double)p.x);
                x1 = fmax(x1, (double)p.x);
                y0 = fmin(y0, (double)p.y);
                y1 = fmax(y1, (double)p.y);
            }
            for (int o = 16; o > 0; o >>= 1) {
                x0 = fmin(x0, __shfl_xor_sync(kFull, x0, o));
                x1 = fmax(x1, __shfl_xor_sync(kFull, x1, o));
                y0 = fmin(y0, __shfl_xor_sync(kFull, y0, o));
                y1 = fmax(y1, __shfl_xor_sync(kFull, y1, o));
            }
            if (lane == 0) {
                s_box[warp][0] = x0;
                s_box[warp][1] = x1;
                s_box[warp][2] = y0;
                s_box[warp][3] = y1;
            }
            __syncthreads();
        }
        if (threadIdx.x == 0) {
            double t0 = A.t0;
            if (!(t0 > 0.0)) {
                t0 = 0.1 * sqrt((double)n);
                if (A.schedule == GILA_COOL_GEOMETRIC) {
                    double x0 = s_box[0][0], x1 = s_box[0][1], y0 = s_box[0][2], y1 = s_box[0][3];
                    for (int w = 1; w < nwarps; ++w) {
                        x0 = fmin(x0, s_box[w][0]);
                        x1 = fmax(x1, s_box[w][1]);
                        y0 = fmin(y0, s_box[w][2]);
                        y1 = fmax(y1, s_box[w][3]);
                    }
                    const double w = x1 - x0, h = y1 - y0;
                    const double a = (w > 0.0 && h > 0.0) ? h / w : 1.0;
                    t0 = sqrt((double)n * A.d / a);
                }
            }
            s_t0 = t0;
            s_t[0] = (T)(A.schedule == GILA_COOL_GEOMETRIC
                             ? t0 * A.geo[0]
                             : t0 * (double)A.iters / (double)A.iters);
        }
        __syncthreads();
        Rep<T, MODEL, COMP, kSrcShared, true, false, true> f;  // right at the smallest distances too
        f.d2 = T(1);
        f.q = A.q;
        Att<T, MODEL, COMP, kSrcShared> att;
        att.inv_d = const_inv_d<T>(A.c);
        att.p = A.p;
        const T d2 = const_d2<T>(A.c);
        P2* cur = buf0;
        P2* nxt = buf1;
        const uint2* ids = reinterpret_cast<const uint2*>(A.tk) + lane;
        const int first = ca + warp;  // this warp's slices: first, first + nwarps, ...
        int2 sd = make_int2(0, 0);
        uint2 next[kBrAhead];
        if (first < cb) {
            sd = A.sdesc[s0 + first];
#pragma unroll
            for (int i = 0; i < kBrAhead; ++i)
                if (i < sd.y) next[i] = ld_ids2(ids + 32 * ((int64_t)sd.x + i));
        }
        for (int it = 0; it < A.iters; ++it) {
            const T t = s_t[it & 1];
            if (threadIdx.x == 0 && it + 1 < A.iters)
                s_t[(it + 1) & 1] = (T)(A.schedule == GILA_COOL_GEOMETRIC
                                            ? s_t0 * A.geo[it + 1]
                                            : s_t0 * (double)(A.iters - it - 1) / (double)A.iters);
            f.src.set_shared(cur, 0u);
            att.src.set_shared(cur, 0u);
            for (int s = first; s < cb; s += nwarps) {
                const int i = s * 32 + lane;
                const bool live = i < n;
                P2 pu;
                pu.x = T(0);
                pu.y = T(0);
                int deg = 0;
                if (live) {
                    pu = cur[i];
                    deg = A.deg[v0 + i];
                }
                f.xu = att.xu = pu.x;
                f.yu = att.yu = pu.y;
                const int dmax = __reduce_max_sync(kFull, deg);
                const int steps = sd.y;
                const int64_t start = sd.x;
                // the slice after this one: the warp's next, or its first
                // again for the next iteration
                const int2 sn = A.sdesc[s0 + (s + nwarps < cb ? s + nwarps : first)];
                // FP32: four sums, one of each id of a step, added after sixteen ids
                constexpr bool FOUR = sizeof(T) == 4 && !COMP;
                constexpr int M = FOUR ? 3 : 0;
                Acc<T, COMP> acc, at, part[M + 1];
                for (int k0 = 0; k0 < steps || k0 == 0; k0 += kBrAhead) {
                    uint2 c4[kBrAhead];
#pragma unroll
                    for (int x = 0; x < kBrAhead; ++x) c4[x] = next[x];
                    const bool more = k0 + kBrAhead < steps;
                    const int64_t from = more ? start + k0 + kBrAhead : (int64_t)sn.x;
                    const int left = more ? steps - k0 - kBrAhead : sn.y;
#pragma unroll
                    for (int x = 0; x < kBrAhead; ++x)
                        if (x < left) next[x] = ld_ids2(ids + 32 * (from + x));
#pragma unroll
                    for (int x = 0; x < kBrAhead; ++x) {
                        if (k0 + x >= steps) break;
                        const uint32_t i0 = c4[x].x & 0xffffu, i1 = c4[x].x >> 16;
                        const uint32_t i2 = c4[x].y & 0xffffu, i3 = c4[x].y >> 16;
                        const int e = 4 * (k0 + x);
                        if constexpr (sizeof(T) == 4 && MODEL == kFR) {
                            if (e < dmax) {  // the rows' first ids are their neighbours
                                fr_entry(cur[i0], pu.x, pu.y, att.inv_d, e < deg, part[0], at);
                                fr_entry(cur[i1], pu.x, pu.y, att.inv_d, e + 1 < deg, part[1 & M], at);
                                fr_entry(cur[i2], pu.x, pu.y, att.inv_d, e + 2 < deg, part[2 & M], at);
                                fr_entry(cur[i3], pu.x, pu.y, att.inv_d, e + 3 < deg, part[3 & M], at);
                                continue;
                            }
                        }
                        f(i0, part[0]);
                        f(i1, part[1 & M]);
                        f(i2, part[2 & M]);
                        f(i3, part[3 & M]);
                        if (e < dmax) {
                            if (e < deg) att(i0, at);
                            if (e + 1 < deg) att(i1, at);
                            if (e + 2 < deg) att(i2, at);
                            if (e + 3 < deg) att(i3, at);
                        }
                    }
                    if constexpr (FOUR) {
                        part[0].merge(part[1].sx, part[1].sy, T(0), T(0));
                        part[2].merge(part[3].sx, part[3].sy, T(0), T(0));
                        part[0].merge(part[2].sx, part[2].sy, T(0), T(0));
                        acc.merge(part[0].sx, part[0].sy, T(0), T(0));
#pragma unroll
                        for (int i = 0; i < 4; ++i) part[i] = Acc<T, COMP>();
                    }
                }
                if constexpr (!FOUR) acc = part[0];
                scale(acc, d2);
                acc.merge(at.sx, at.sy, at.cx, at.cy);
                T mx, my;
                capped<T>(t, acc.fx(), acc.fy(), mx, my);
                // (padding is all an isolated vertex has: 0 at a finite place)
                P2 o;
                o.x = deg > 0 ? pu.x + mx : pu.x;
                o.y = deg > 0 ? pu.y + my : pu.y;
                nxt[i] = o;
                sd = sn;
            }
            if (big) {
                // push this CTA's new positions to its peers and wait for theirs
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                // once a thread of the CTA has given up, the CTA neither
                // announces, pushes nor waits any more
                const bool failed = __syncthreads_or(gave_up) != 0;
                uint64_t* bar = &s_bar[it & 1];
                const uint32_t parity = (phase >> (it & 1)) & 1;
                const uint32_t mine = (uint32_t)(cb - ca) * 32u * (uint32_t)sizeof(P2);
                if (threadIdx.x == 0 && !failed) {
                    mbar_arrive_expect_tx(bar, (uint32_t)npad * (uint32_t)sizeof(P2) - mine);
                    const uint32_t src = smem_addr(nxt + ca * 32), b = smem_addr(bar);
                    for (uint32_t r = 1; r < csize && !A.skip_push; ++r) {
                        const uint32_t to = (rank + r) & (csize - 1);
                        if ((peers >> to) & 1)
                            bulk_s2s(cluster_map(src, to), src, mine, cluster_map(b, to));
                    }
                }
                if (!failed && !mbar_wait(bar, parity, A.wait_ns)) {
                    // give up: flag it, let what is in flight land (bounded);
                    // the cluster leaves together
                    gave_up = true;
                    *(volatile int*)A.wait_failed = 1;
                    __threadfence_system();
                    mbar_wait(bar, parity, A.wait_ns);
                }
                phase ^= 1u << (it & 1);
                // s_t of the next iteration is visible: written before the
                // __syncthreads above
            } else {
                __syncthreads();
            }
            P2* x = cur;
            cur = nxt;
            nxt = x;
        }
        for (int i = ca * 32 + threadIdx.x; i < n && i < cb * 32; i += blockDim.x)
            gpos[v0 + perm[i]] = cur[i];
    };

    // large graphs, a cluster each
    for (;;) {
        cluster_sync();  // mbarriers initialised; every CTA is done with the graph before
        if (rank == 0 && threadIdx.x == 0) {
            const int g = atomicAdd(&A.work[0], 1);
            const uint32_t a = smem_addr(&s_g);
            for (uint32_t r = 0; r < csize; ++r)
                asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(cluster_map(a, r)), "r"(g)
                             : "memory");
        }
        cluster_sync();
        const int gi = s_g;
        if (gi >= A.nbig) break;  // uniform over the cluster
        layout(A.order[gi], true);
    }
    // small graphs, a CTA each
    for (;;) {
        __syncthreads();
        if (threadIdx.x == 0) s_g = atomicAdd(&A.work[1], 1);
        __syncthreads();
        const int gi = A.nbig + s_g;
        if (gi >= A.nall) break;
        layout(A.order[gi], false);
    }
}

// First k-hop entry of every graph (count + 1 values).
__global__ void graph_bounds_kernel(int32_t count, const int64_t* __restrict__ voff,
                                    const int64_t* __restrict__ krow, int64_t* __restrict__ out)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i <= count) out[i] = krow[voff[i]];
}

// Plan, one block per graph: its vertices sorted by row length (longest
// first; a counting sort, the order within a length left to the atomics: no
// result depends on it), the steps of every slice and their starts within the
// graph, the total, and the slice bounds of a cluster's CTAs (equal steps,
// two more a slice for its positions and moves). Graphs with skip[g] set are
// left out.
__global__ void __launch_bounds__(256)
batch_sort_kernel(const int64_t* __restrict__ voff, const int32_t* __restrict__ soff,
                  const uint8_t* __restrict__ skip, const int64_t* __restrict__ krow,
                  uint16_t* __restrict__ perm, uint16_t* __restrict__ rank,
                  int2* __restrict__ sdesc, int32_t* __restrict__ units,
                  uint16_t* __restrict__ cuts)
{
    __shared__ int hist[kBrBins];
    __shared__ int wt[256 / 32 + 1];
    const int g = blockIdx.x, tid = threadIdx.x;
    if (skip[g]) return;
    const int64_t v0 = voff[g];
    const int n = (int)(voff[g + 1] - v0);
    for (int b = tid; b < kBrBins; b += 256) hist[b] = 0;
    __syncthreads();
    auto bin = [&](int i) {
        const int64_t len = krow[v0 + i + 1] - krow[v0 + i];
        return kBrBins - 1 - (len < kBrBins ? (int)len : kBrBins - 1);
    };
    for (int i = tid; i < n; i += 256) atomicAdd(&hist[bin(i)], 1);
    __syncthreads();
    int carry = 0;
    for (int b0 = 0; b0 < kBrBins; b0 += 256) {
        const int c = hist[b0 + tid];
        int total;
        const int incl = block_inclusive_scan<int, 256>(c, wt, &total);
        hist[b0 + tid] = carry + incl - c;
        carry += total;
    }
    __syncthreads();
    for (int i = tid; i < n; i += 256) {
        const int at = atomicAdd(&hist[bin(i)], 1);
        perm[v0 + at] = (uint16_t)i;
        rank[v0 + i] = (uint16_t)at;
    }
    __syncthreads();
    const int ns = (n + 31) >> 5;
    int2* sd = sdesc + soff[g];
    carry = 0;
    for (int b0 = 0; b0 < ns; b0 += 256) {
        const int s = b0 + tid;
        int steps = 0;
        if (s < ns) {
            int64_t most = 0;
            for (int i = s * 32; i < n && i < s * 32 + 32; ++i) {
                const int64_t v = v0 + perm[v0 + i];
                const int64_t len = krow[v + 1] - krow[v];
                most = len > most ? len : most;
            }
            steps = (int)((most + 3) >> 2);
        }
        int total;
        const int incl = block_inclusive_scan<int, 256>(steps, wt, &total);
        if (s < ns) sd[s] = make_int2(carry + incl - steps, steps);
        carry += total;
    }
    if (tid == 0) units[g] = carry;
    __syncthreads();
    if (tid <= kBrCluster) {
        // the first slice whose cost before it reaches the share
        const int64_t want = (int64_t)(carry + 2 * ns) * tid / kBrCluster;
        int lo = 0, hi = ns;
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if (sd[mid].x + 2 * mid < want) lo = mid + 1; else hi = mid;
        }
        cuts[(kBrCluster + 1) * g + tid] = (uint16_t)(tid == kBrCluster ? ns : lo);
    }
}

// Plan, a warp per slice and a row per lane: the slice's start becomes its
// place in tk, and its ids are written, neighbours first (both lists
// ascending, one merge), then the rest, then its own as padding (the far slot's
// in lanes without a row). A row whose
// neighbours are not all among its k-hop ids (an unsorted or repeated
// adjacency, a self-loop) sets bad[g]: the graph keeps the group kernel.
__global__ void __launch_bounds__(128)
batch_fill_kernel(int64_t nslices, const int32_t* __restrict__ sgraph,
                  const int64_t* __restrict__ voff, const int32_t* __restrict__ soff,
                  const int32_t* __restrict__ base, const uint8_t* __restrict__ skip,
                  const int64_t* __restrict__ row, const int32_t* __restrict__ col,
                  const int64_t* __restrict__ krow, const uint32_t* __restrict__ kcol,
                  const uint16_t* __restrict__ perm, const uint16_t* __restrict__ rank,
                  int2* __restrict__ sdesc, uint16_t* __restrict__ deg_out,
                  uint16_t* __restrict__ tk, uint8_t* __restrict__ bad)
{
    const int lane = threadIdx.x & 31;
    const int64_t s = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (s >= nslices) return;  // warp-uniform
    const int g = sgraph[s];
    if (skip[g]) return;
    const int64_t v0 = voff[g];
    const int n = (int)(voff[g + 1] - v0);
    const int npad = (n + 31) & ~31;
    int2 sd = sdesc[s];
    __syncwarp();
    sd.x += base[g];
    if (lane == 0) sdesc[s] = sd;
    const int i = (int)(s - soff[g]) * 32 + lane;
    int64_t kb = 0, ke = 0, ab = 0;
    int deg = 0;
    if (i < n) {
        const int64_t u = v0 + perm[v0 + i];
        kb = krow[u];
        ke = krow[u + 1];
        ab = row[u];
        const int64_t d64 = row[u + 1] - ab;
        deg = d64 <= ke - kb ? (int)d64 : 0;
        if (d64 != deg) bad[g] = 1;
        deg_out[v0 + i] = (uint16_t)deg;
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
    for (int a = 0; a < deg; ++a) put(rank[col[ab + a]]);
    int a = 0, found = 0;
    for (int64_t x = kb; x < ke; ++x) {
        const uint32_t id = kcol[x];
        while (a < deg && (uint32_t)col[ab + a] < id) ++a;
        if (a < deg && (uint32_t)col[ab + a] == id) ++found;
        else put(rank[id]);
    }
    if (found != deg) bad[g] = 1;
    while (w < slots) put((uint32_t)(i < n ? i : npad));
}

// Pack graphs given as device CSRs into the union CSR (one block per graph).
struct PackSrc {
    const int64_t* row;
    const int32_t* col;
    int64_t n, voff, eoff;
};

__global__ void pack_kernel(const PackSrc* __restrict__ src, int64_t* __restrict__ row,
                            int32_t* __restrict__ col)
{
    const PackSrc s = src[blockIdx.x];
    for (int64_t i = threadIdx.x; i < s.n; i += blockDim.x) row[s.voff + i] = s.eoff + s.row[i];
    const int64_t nnz = s.row[s.n] - s.row[0];
    for (int64_t i = threadIdx.x; i < nnz; i += blockDim.x)
        col[s.eoff + i] = (int32_t)(s.voff + s.col[s.row[0] + i]);
}

// Whether the tuning asks for lane groups on every graph.
bool wants_groups(const gila_batch_tuning& t)
{
    return t.group4_max > 0 || t.group8_max > 0 || t.group16_max > 0;
}

// The tuning as a caller reads it back: what it leaves to the library stays 0
// (filled in, the lane groups would ask for the group kernel on every graph), so
// that setting it again changes nothing.
gila_batch_tuning reported(const gila_batch_tuning& set)
{
    gila_batch_tuning t = set;
    if (t.threads == 0) t.threads = 512;
    if (wants_groups(t)) {
        if (t.group4_max <= 0) t.group4_max = 8;
        if (t.group8_max <= 0) t.group8_max = 24;
        if (t.group16_max <= 0) t.group16_max = 64;
    }
    return t;
}

// The tuning that the group kernel runs with.
gila_batch_tuning resolved(const gila_batch* b, size_t esz)
{
    gila_batch_tuning t = b->tune;
    if (t.threads != 256 && t.threads != 512 && t.threads != 1024) t.threads = 512;
    if (t.group4_max <= 0) t.group4_max = 8;
    if (t.group8_max <= 0) t.group8_max = 24;
    if (t.group16_max <= 0) t.group16_max = 64;
    const int64_t smem_cap = 227 * 1024 - 2048;  // opt-in limit less the static arrays
    if (t.ctas_per_sm <= 0) {
        // two CTAs per SM unless a graph then no longer fits
        const int64_t need = 2 * b->max_n * (int64_t)esz;
        t.ctas_per_sm = (need * 2 <= smem_cap) ? 2 : 1;
    }
    t.ctas_per_sm = std::max(1, std::min(t.ctas_per_sm, 2048 / t.threads));
    return t;
}

template <class T, int MODEL, bool COMP>
cudaError_t launch_batch(const BatchArgs& A, int grid, int threads, size_t smem, cudaStream_t st)
{
    batch_kernel<T, MODEL, COMP><<<grid, threads, smem, st>>>(A);
    count_launch();
    return cudaGetLastError();
}

template <class T, bool COMP>
struct Form {
    using type = T;
    static constexpr bool comp = COMP;
};

template <class T, int MODEL, bool COMP>
cudaError_t launch_batch_rows(const BatchRowsArgs& R, int grid, int cluster, int threads,
                              size_t smem, cudaStream_t st)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at = {};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = (unsigned)cluster;
    at.val.clusterDim.y = 1;
    at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    cudaError_t e = cudaLaunchKernelEx(&cfg, batch_rows_kernel<T, MODEL, COMP>, R);
    count_launch();
    return e != cudaSuccess ? e : cudaGetLastError();
}

// Shared-memory opt-in for every instantiation on the current device
// (outside any stream capture); once per device, callers may race.
cudaError_t configure_batch_kernels()
{
    static std::atomic<uint64_t> done{0};
    int device = 0;
    cudaError_t de = cudaGetDevice(&device);
    if (de != cudaSuccess) return de;
    const uint64_t bit = 1ull << (device & 63);
    if (done.load() & bit) return cudaSuccess;
    const int lim = 227 * 1024;
    cudaError_t e = cudaSuccess;
#define GILA_OPT_IN(T, M, C)                                                                 \
    if (e == cudaSuccess)                                                                    \
        e = cudaFuncSetAttribute(batch_kernel<T, M, C>,                                      \
                                 cudaFuncAttributeMaxDynamicSharedMemorySize, lim - 2048);   \
    if (e == cudaSuccess)                                                                    \
        e = cudaFuncSetAttribute(batch_rows_kernel<T, M, C>,                                 \
                                 cudaFuncAttributeMaxDynamicSharedMemorySize, kBrSmem);
    GILA_OPT_IN(float, kFR, false)
    GILA_OPT_IN(float, kGeneric, false)
    GILA_OPT_IN(float, kFR, true)
    GILA_OPT_IN(float, kGeneric, true)
    GILA_OPT_IN(double, kFR, false)
    GILA_OPT_IN(double, kGeneric, false)
#undef GILA_OPT_IN
    if (e == cudaSuccess) done.fetch_or(bit);
    return e;
}

gila_status batch_finish_create(gila_batch* b)
{
    const int32_t count = b->count;
    // processing order: largest graphs first
    std::vector<int32_t> order(count);
    std::iota(order.begin(), order.end(), 0);
    std::stable_sort(order.begin(), order.end(), [&](int32_t a, int32_t c) {
        return b->voff_h[a + 1] - b->voff_h[a] > b->voff_h[c + 1] - b->voff_h[c];
    });
    b->order_h = order;
    b->max_n = 0;
    for (int32_t i = 0; i < count; ++i)
        b->max_n = std::max<int64_t>(b->max_n, b->voff_h[i + 1] - b->voff_h[i]);
    GILA_CUDA(cudaMalloc(&b->voff, sizeof(int64_t) * (count + 1)));
    GILA_CUDA(cudaMalloc(&b->order, sizeof(int32_t) * std::max(count, 1)));
    GILA_CUDA(cudaMalloc(&b->work, sizeof(int) * 3));  // group kernel, large, small graphs
    GILA_CUDA(cudaMemcpy(b->voff, b->voff_h.data(), sizeof(int64_t) * (count + 1),
                         cudaMemcpyHostToDevice));
    if (count > 0)
        GILA_CUDA(cudaMemcpy(b->order, order.data(), sizeof(int32_t) * count,
                             cudaMemcpyHostToDevice));
    GILA_CUDA(cudaHostAlloc((void**)&b->wait_failed, sizeof(int), cudaHostAllocMapped));
    *b->wait_failed = 0;
    GILA_CUDA(cudaStreamCreateWithFlags(&b->own, cudaStreamNonBlocking));
    GILA_CUDA(cudaStreamCreateWithFlags(&b->side, cudaStreamNonBlocking));
    GILA_CUDA(cudaEventCreateWithFlags(&b->ev_fork, cudaEventDisableTiming));
    GILA_CUDA(cudaEventCreateWithFlags(&b->ev_join, cudaEventDisableTiming));
    GILA_CUDA(cudaEventCreateWithFlags(&b->ev_in, cudaEventDisableTiming));
    GILA_CUDA(cudaEventCreateWithFlags(&b->ev_out, cudaEventDisableTiming));
    return GILA_OK;
}

gila_status check_batch_params(const gila_params* p)
{
    if (!p) return fail(GILA_EINVAL, "params is NULL");
    if (p->k < 1 || p->k > 64) return fail(GILA_EINVAL, "k must be in [1, 64]");
    if (p->iters < 0) return fail(GILA_EINVAL, "iters must be >= 0");
    if (!(p->d > 0.0) || !std::isfinite(p->d)) return fail(GILA_EINVAL, "d must be finite and > 0");
    if (!std::isfinite(p->t0)) return fail(GILA_EINVAL, "t0 must be finite");
    if (p->schedule != GILA_COOL_LINEAR && p->schedule != GILA_COOL_GEOMETRIC)
        return fail(GILA_EINVAL, "unknown cooling schedule");
    if (p->p < 0 || p->p > 8 || p->q < 0 || p->q > 8)
        return fail(GILA_EINVAL, "p and q must be in [0, 8]");
    if (p->precision != GILA_FP32 && p->precision != GILA_FP64 &&
        p->precision != GILA_FP32_COMPENSATED)
        return fail(GILA_EINVAL, "batched layouts support GILA_FP32, GILA_FP32_COMPENSATED and "
                                 "GILA_FP64");
    return GILA_OK;
}

// The row-per-lane plan (see batch_rows_kernel), made once per k-hop build.
// A graph takes it when its rows are short (mean at most kBrMeanLen: longer
// rows keep groups of lanes), its slots at most kBrPadding per entry, its two
// buffers fit shared memory, and its neighbours are among its k-hop ids. All
// of that depends on the graph alone.
gila_status batch_plan(gila_batch* b)
{
    gila_graph* g = b->g;
    if (b->plan_serial == g->khop_serial) return GILA_OK;
    b->plan_serial = -1;
    const int32_t count = b->count;
    cudaStream_t st = b->user;
    const std::vector<int64_t>& vo = b->voff_h;
    std::vector<int32_t> soff((size_t)count + 1, 0);
    for (int32_t i = 0; i < count; ++i)
        soff[(size_t)i + 1] = soff[(size_t)i] + (int32_t)((vo[(size_t)i + 1] - vo[(size_t)i] + 31) / 32);
    const int64_t nsl = soff[(size_t)count];
    if (!b->soff) {
        std::vector<int32_t> sg((size_t)nsl);
        for (int32_t i = 0; i < count; ++i)
            std::fill(sg.begin() + soff[(size_t)i], sg.begin() + soff[(size_t)i + 1], i);
        const size_t n1 = (size_t)std::max<int64_t>(g->n, 1), s1 = (size_t)std::max<int64_t>(nsl, 1);
        // (what an earlier call that ran out of memory left is kept)
        auto need = [](auto** p, size_t bytes) -> gila_status {
            if (!*p) GILA_CUDA(cudaMalloc(p, bytes));
            return GILA_OK;
        };
        gila_status s;
        if ((s = need(&b->sgraph, sizeof(int32_t) * s1)) || (s = need(&b->sdesc, sizeof(int2) * s1)) ||
            (s = need(&b->base, sizeof(int32_t) * (size_t)count)) ||
            (s = need(&b->units, sizeof(int32_t) * (size_t)count)) ||
            (s = need(&b->skip, 2 * (size_t)count)) || (s = need(&b->deg, sizeof(uint16_t) * n1)) ||
            (s = need(&b->perm, sizeof(uint16_t) * n1)) ||
            (s = need(&b->rank, sizeof(uint16_t) * n1)) ||
            (s = need(&b->cuts, sizeof(uint16_t) * (kBrCluster + 1) * (size_t)count)) ||
            (s = need(&b->rorder[0], sizeof(int32_t) * (size_t)count)) ||
            (s = need(&b->rorder[1], sizeof(int32_t) * (size_t)count)))
            return s;
        GILA_CUDA(cudaMemcpyAsync(b->sgraph, sg.data(), sizeof(int32_t) * (size_t)nsl,
                                  cudaMemcpyHostToDevice, st));
        int32_t* so = nullptr;
        GILA_CUDA(cudaMalloc(&so, sizeof(int32_t) * ((size_t)count + 1)));
        b->soff = so;  // last: marks the set complete
        GILA_CUDA(cudaMemcpyAsync(so, soff.data(), sizeof(int32_t) * soff.size(),
                                  cudaMemcpyHostToDevice, st));
        GILA_CUDA(cudaStreamSynchronize(st));  // the host vectors go out of scope
    }
    // rows' totals per graph
    std::vector<int64_t> koff((size_t)count + 1);
    int64_t* dk = nullptr;
    GILA_CUDA(cudaMalloc(&dk, sizeof(int64_t) * ((size_t)count + 1)));
    graph_bounds_kernel<<<(unsigned)((count + 256) / 256), 256, 0, st>>>(count, b->voff, g->krow, dk);
    count_launch();
    cudaMemcpyAsync(koff.data(), dk, sizeof(int64_t) * koff.size(), cudaMemcpyDeviceToHost, st);
    cudaError_t e = cudaStreamSynchronize(st);
    cudaFree(dk);
    if (e != cudaSuccess) return cuda_fail(e, "batch plan");
    constexpr int64_t max_n = kBrSmem / 16 - 64;  // float2, two buffers and their far slots
    std::vector<uint8_t> skip(2 * (size_t)count, 0);
    for (int32_t i = 0; i < count; ++i) {
        const int64_t n = vo[(size_t)i + 1] - vo[(size_t)i];
        const int64_t nnz = koff[(size_t)i + 1] - koff[(size_t)i];
        skip[(size_t)i] = n == 0 || n > max_n || nnz > kBrMeanLen * n;
    }
    std::vector<int32_t> units((size_t)count, 0), base((size_t)count, 0);
    GILA_CUDA(cudaMemcpyAsync(b->skip, skip.data(), skip.size(), cudaMemcpyHostToDevice, st));
    GILA_CUDA(cudaMemsetAsync(b->units, 0, sizeof(int32_t) * (size_t)count, st));
    batch_sort_kernel<<<(unsigned)count, 256, 0, st>>>(b->voff, b->soff, b->skip, g->krow, b->perm,
                                                       b->rank, b->sdesc, b->units, b->cuts);
    count_launch();
    GILA_CUDA(cudaGetLastError());
    GILA_CUDA(cudaMemcpyAsync(units.data(), b->units, sizeof(int32_t) * (size_t)count,
                              cudaMemcpyDeviceToHost, st));
    GILA_CUDA(cudaStreamSynchronize(st));
    int64_t total = 0;
    for (int32_t i = 0; i < count; ++i) {
        const int64_t nnz = koff[(size_t)i + 1] - koff[(size_t)i];
        const int64_t n = vo[(size_t)i + 1] - vo[(size_t)i];
        if (!skip[(size_t)i] &&
            ((double)units[(size_t)i] * 128.0 > kBrPadding * (double)nnz + 128.0 * (double)((n + 31) / 32) ||
             total + units[(size_t)i] > INT32_MAX))
            skip[(size_t)i] = 1;
        base[(size_t)i] = (int32_t)total;
        if (!skip[(size_t)i]) total += units[(size_t)i];
    }
    gila_status s = ensure((void**)&b->tk, &b->tk_cap, (size_t)total * 256 + 16);
    if (s != GILA_OK) return s;
    GILA_CUDA(cudaMemcpyAsync(b->skip, skip.data(), skip.size(), cudaMemcpyHostToDevice, st));
    GILA_CUDA(cudaMemcpyAsync(b->base, base.data(), sizeof(int32_t) * (size_t)count,
                              cudaMemcpyHostToDevice, st));
    if (nsl > 0) {
        batch_fill_kernel<<<(unsigned)((nsl + 3) / 4), 128, 0, st>>>(
            nsl, b->sgraph, b->voff, b->soff, b->base, b->skip, g->row, g->col, g->krow, g->kcol,
            b->perm, b->rank, b->sdesc, b->deg, b->tk, b->skip + count);
        count_launch();
        GILA_CUDA(cudaGetLastError());
    }
    std::vector<uint8_t> bad((size_t)count);
    GILA_CUDA(cudaMemcpyAsync(bad.data(), b->skip + count, (size_t)count, cudaMemcpyDeviceToHost, st));
    GILA_CUDA(cudaStreamSynchronize(st));
    // by width: large graphs, small ones, and the rest, each by falling work
    for (int w = 0; w < 2; ++w) {
        const int64_t lim = w == 0 ? max_n : kBrSmem / 32 - 64;
        std::vector<int32_t> rows;
        b->rest[w].clear();
        b->big[w].clear();
        b->small[w].clear();
        b->max_rows_n[w] = 0;
        for (int32_t i : b->order_h) {
            const int64_t n = vo[(size_t)i + 1] - vo[(size_t)i];
            if (skip[(size_t)i] || bad[(size_t)i] || n > lim) {
                b->rest[w].push_back(i);
                continue;
            }
            b->max_rows_n[w] = std::max(b->max_rows_n[w], n);
            rows.push_back(i);
        }
        std::stable_sort(rows.begin(), rows.end(), [&](int32_t x, int32_t y) {
            return units[(size_t)x] > units[(size_t)y];
        });
        // An SM's share of the batch (steps, two more a slice), the cluster
        // that brings the largest graph below it, and the graphs it takes:
        // 500 graphs of 50..5000 vertices in FP32 6.5 -> 0.90, 0.73, 0.60 ms
        // with clusters of 8, 4, 2 (the share asks for 2); 250 in FP64 20.8
        // -> 5.8, 4.1, 5.1 (4); 30 in FP64 0.69, 1.21, 2.22 (8); 1500 in FP64
        // 6.5, 4.2, 3.4 (1: an SM left over in a GPC, or waiting for a peer,
        // is then lost). Graphs from about a third of the share on.
        auto cost = [&](int32_t i) {
            return units[(size_t)i] + 2 * ((vo[(size_t)i + 1] - vo[(size_t)i] + 31) / 32);
        };
        int64_t all_cost = 0;
        for (int32_t i : rows) all_cost += cost(i);
        const int64_t share = all_cost / std::max(1, sm_count(g->device)) + 1;
        b->cluster[w] = 1;
        if (!rows.empty())
            while (b->cluster[w] < kBrCluster && cost(rows[0]) > share * b->cluster[w])
                b->cluster[w] *= 2;
        for (int32_t i : rows) {
            const bool large = b->cluster[w] > 1 && 3 * cost(i) > share &&
                               (vo[(size_t)i + 1] - vo[(size_t)i] + 31) / 32 >= kBrBigSlices[w];
            (large ? b->big[w] : b->small[w]).push_back(i);
        }
        std::vector<int32_t> all(b->big[w]);
        all.insert(all.end(), b->small[w].begin(), b->small[w].end());
        all.insert(all.end(), b->rest[w].begin(), b->rest[w].end());
        GILA_CUDA(cudaMemcpyAsync(b->rorder[w], all.data(), sizeof(int32_t) * all.size(),
                                  cudaMemcpyHostToDevice, st));
        GILA_CUDA(cudaStreamSynchronize(st));
    }
    b->plan_serial = g->khop_serial;
    return GILA_OK;
}

// GILA_ECUDA (and clears the flag) when a cluster of a launch of this batch
// gave up waiting for its peers' positions since the last call. Does not
// synchronise: launches that have not ended are told of by a later call.
gila_status batch_wait_failed(gila_batch* b)
{
    if (!*(volatile int*)b->wait_failed) return GILA_OK;
    *(volatile int*)b->wait_failed = 0;
    return fail(GILA_ECUDA, "a cluster of the batch kernel did not receive its positions in time");
}

// Launch (or replay) the persistent kernel on the batch's capture stream,
// ordered after and before the caller's stream.
gila_status batch_run(gila_batch* b, const gila_params* prm, void* pos)
{
    gila_graph* g = b->g;
    const size_t esz = is_f64(prm->precision) ? 16 : 8;
    gila_status s = batch_wait_failed(b);  // of an earlier launch
    if (s != GILA_OK) return s;
    if (b->count == 0 || g->n == 0 || prm->iters == 0) return GILA_OK;
    if (prm->schedule == GILA_COOL_GEOMETRIC) {
        s = ensure((void**)&b->geo, &b->geo_cap, sizeof(double) * (size_t)prm->iters);
        if (s != GILA_OK) return s;
        std::vector<double> geo((size_t)prm->iters);
        for (int i = 0; i < prm->iters; ++i) geo[i] = std::pow(0.93, (double)i);
        GILA_CUDA(cudaMemcpy(b->geo, geo.data(), sizeof(double) * geo.size(),
                             cudaMemcpyHostToDevice));
    }
    // without memory for the plan every graph keeps the group kernel
    s = batch_plan(b);
    if (s != GILA_OK && s != GILA_ENOMEM) return s;
    const bool planned = s == GILA_OK;
    const int sms = sm_count(g->device);
    const gila_batch_tuning tu = resolved(b, esz);
    // lane groups set by the tuning ask for the group kernel on every graph
    const int w = esz == 16 ? 1 : 0;
    const bool groups = !planned || wants_groups(b->tune);
    const int nbig = groups ? 0 : (int)b->big[w].size();
    const int nrows = groups ? 0 : nbig + (int)b->small[w].size();
    const int nrest = b->count - nrows;
    const int64_t smem_cap = 227 * 1024 - 2048;
    int64_t per_cta = smem_cap / tu.ctas_per_sm;
    int64_t smem_verts = std::min<int64_t>(b->max_n, per_cta / (2 * (int64_t)esz));
    if (smem_verts < 2) smem_verts = 2;
    const size_t smem = (size_t)smem_verts * 2 * esz;
    if (b->max_n > smem_verts) {
        s = ensure(&b->tmp, &b->tmp_cap, esz * (size_t)g->n);
        if (s != GILA_OK) return s;
    }
    BatchArgs A;
    memset(&A, 0, sizeof(A));  // padding too: the bytes are part of the captured graph's key
    A.voff = b->voff;
    A.order = groups ? b->order : b->rorder[w] + nrows;
    A.count = nrest;
    A.row = g->row;
    A.col = g->col;
    A.krow = g->krow;
    A.kcol = g->kcol;
    A.work = b->work;
    A.geo = b->geo;
    A.iters = prm->iters;
    A.schedule = prm->schedule;
    A.d = prm->d;
    A.t0 = prm->t0;
    A.p = prm->p;
    A.q = prm->q;
    A.pos = pos;
    A.tmp = b->tmp;
    A.smem_verts = (int)smem_verts;
    A.g4_max = tu.group4_max;
    A.g8_max = tu.group8_max;
    A.g16_max = tu.group16_max;
    const int grid = std::max(1, std::min<int>(sms * tu.ctas_per_sm, nrest));
    BatchRowsArgs R;
    memset(&R, 0, sizeof(R));
    R.voff = b->voff;
    R.order = b->rorder[w];
    R.nbig = nbig;
    R.nall = nrows;
    R.soff = b->soff;
    R.sdesc = b->sdesc;
    R.deg = b->deg;
    R.perm = b->perm;
    R.cuts = b->cuts;
    R.tk = b->tk;
    R.work = b->work + 1;
    R.geo = b->geo;
    R.iters = prm->iters;
    R.schedule = prm->schedule;
    R.d = prm->d;
    R.t0 = prm->t0;
    R.c = force_consts(prm->d, 0.0);
    R.p = prm->p;
    R.q = prm->q;
    R.pos = pos;
    R.stride = (int)((b->max_rows_n[w] + 31) / 32 * 32 + 2);
    R.wait_ns = b->wait_test ? kBrTestWaitNs : kBrWaitNs;
    R.skip_push = b->wait_test;
    R.wait_failed = b->wait_failed;
    const size_t rsmem = 2 * (size_t)R.stride * esz;
    // as many CTAs per SM as the tuning and the buffers allow, in clusters
    const int64_t fit = std::max<int64_t>(1, (kBrSmem + 2048) / (int64_t)(rsmem + 2048));
    const int64_t per_sm = std::min<int64_t>(fit, b->tune.ctas_per_sm > 0 ? tu.ctas_per_sm
                                                                          : 2048 / tu.threads);
    const int cl = b->cluster[w];
    const int64_t want = std::min<int64_t>(sms * per_sm, (int64_t)nbig * cl + nrows - nbig);
    const int rgrid = (int)((std::max<int64_t>(want, 1) + cl - 1) / cl * cl);
    // the captured graph is reused while every argument is the same
    const int extra[7] = {grid, tu.threads, prm->precision, nrows, nrest, rgrid, cl};
    std::vector<unsigned char> key(sizeof(A) + sizeof(R) + sizeof(extra));
    memcpy(key.data(), &A, sizeof(A));
    memcpy(key.data() + sizeof(A), &R, sizeof(R));
    memcpy(key.data() + sizeof(A) + sizeof(R), extra, sizeof(extra));
    GILA_CUDA(configure_batch_kernels());
    GILA_CUDA(cudaEventRecord(b->ev_in, b->user));
    GILA_CUDA(cudaStreamWaitEvent(b->own, b->ev_in, 0));
    if (!b->exec || key != b->exec_key) {
        if (b->exec) {
            cudaGraphExecDestroy(b->exec);
            b->exec = nullptr;
        }
        cudaGraph_t graph = nullptr;
        GILA_CUDA(cudaStreamBeginCapture(b->own, cudaStreamCaptureModeThreadLocal));
        cudaError_t e = cudaMemsetAsync(b->work, 0, sizeof(int) * 3, b->own);
        const bool fr = (prm->p == 2 && prm->q == 1);
        const bool fork = nrows > 0 && nrest > 0;
        cudaStream_t gst = fork ? b->side : b->own;
        if (e == cudaSuccess && fork) e = cudaEventRecord(b->ev_fork, b->own);
        if (e == cudaSuccess && fork) e = cudaStreamWaitEvent(b->side, b->ev_fork, 0);
        auto launch = [&](auto model, auto one) {
            // `one`: a value of the force type; its second field the compensation
            using T = typename decltype(one)::type;
            constexpr bool comp = decltype(one)::comp;
            constexpr int M = decltype(model)::value;
            if (e == cudaSuccess && nrows > 0)
                e = launch_batch_rows<T, M, comp>(R, rgrid, cl, tu.threads, rsmem, b->own);
            if (e == cudaSuccess && nrest > 0)
                e = launch_batch<T, M, comp>(A, grid, tu.threads, smem, gst);
        };
        auto by_type = [&](auto model) {
            switch (prm->precision) {
            case GILA_FP64: launch(model, Form<double, false>()); break;
            case GILA_FP32_COMPENSATED: launch(model, Form<float, true>()); break;
            default: launch(model, Form<float, false>()); break;
            }
        };
        if (fr) by_type(std::integral_constant<int, kFR>());
        else by_type(std::integral_constant<int, kGeneric>());
        if (e == cudaSuccess && fork) e = cudaEventRecord(b->ev_join, b->side);
        if (e == cudaSuccess && fork) e = cudaStreamWaitEvent(b->own, b->ev_join, 0);
        cudaError_t e2 = cudaStreamEndCapture(b->own, &graph);
        if (e != cudaSuccess) {
            if (graph) cudaGraphDestroy(graph);
            return cuda_fail(e, "batch_kernel");
        }
        if (e2 != cudaSuccess) return cuda_fail(e2, "cudaStreamEndCapture");
        cudaError_t e3 = cudaGraphInstantiate(&b->exec, graph, 0);
        cudaGraphDestroy(graph);
        if (e3 != cudaSuccess) {
            b->exec = nullptr;
            return cuda_fail(e3, "cudaGraphInstantiate");
        }
        b->exec_key = key;
    }
    GILA_CUDA(cudaGraphLaunch(b->exec, b->own));
    GILA_CUDA(cudaEventRecord(b->ev_out, b->own));
    GILA_CUDA(cudaStreamWaitEvent(b->user, b->ev_out, 0));
    return GILA_OK;
}

}  // namespace
}  // namespace gila

using namespace gila;

extern "C" {

gila_status gila_batch_create(int32_t count, const int64_t* n, const int64_t* const* row_ptr,
                              const int32_t* const* col_idx, int32_t flags, gila_batch** out)
{
    if (!out) return fail(GILA_EINVAL, "out is NULL");
    *out = nullptr;
    if (count < 0) return fail(GILA_EINVAL, "count must be >= 0");
    if (count > 0 && (!n || !row_ptr || !col_idx)) return fail(GILA_EINVAL, "array is NULL");
    std::vector<int64_t> voff(count + 1, 0), eoff(count + 1, 0);
    for (int32_t i = 0; i < count; ++i) {
        if (n[i] < 0 || !row_ptr[i]) return fail(GILA_EINVAL, "graph " + std::to_string(i) + ": bad n or row_ptr");
        if (flags & GILA_GRAPH_VALIDATE) {
            gila_status s = gila_csr_validate(n[i], row_ptr[i], col_idx[i]);
            if (s != GILA_OK) return fail(s, "graph " + std::to_string(i) + ": " + gila_last_error());
        } else {
            gila_status s = check_csr_bounds(n[i], row_ptr[i], col_idx[i]);
            if (s != GILA_OK) return fail(s, "graph " + std::to_string(i) + ": " + gila_last_error());
        }
        voff[i + 1] = voff[i] + n[i];
        eoff[i + 1] = eoff[i] + (row_ptr[i][n[i]] - row_ptr[i][0]);
    }
    if (voff[count] >= ((int64_t)1 << 31)) return fail(GILA_EINVAL, "batch has too many vertices");
    // union CSR on the host, uploaded once
    std::vector<int64_t> row((size_t)voff[count] + 1);
    std::vector<int32_t> col((size_t)eoff[count]);
    for (int32_t i = 0; i < count; ++i) {
        const int64_t b0 = row_ptr[i][0];
        for (int64_t u = 0; u < n[i]; ++u) row[voff[i] + u] = eoff[i] + (row_ptr[i][u] - b0);
        for (int64_t j = 0; j < eoff[i + 1] - eoff[i]; ++j)
            col[eoff[i] + j] = (int32_t)(voff[i] + col_idx[i][b0 + j]);
    }
    row[voff[count]] = eoff[count];
    gila_batch* b = new (std::nothrow) gila_batch();
    if (!b) return fail(GILA_ENOMEM, "host allocation");
    gila_status s = gila_graph_create(voff[count], row.data(), col.data(), 0, &b->g);
    if (s != GILA_OK) {
        delete b;
        return s;
    }
    b->count = count;
    b->voff_h = voff;
    s = batch_finish_create(b);
    if (s != GILA_OK) {
        gila_batch_destroy(b);
        return s;
    }
    *out = b;
    return GILA_OK;
}

void gila_batch_destroy(gila_batch* b)
{
    if (!b) return;
    if (b->g) cudaSetDevice(b->g->device);
    if (b->own) cudaStreamSynchronize(b->own);
    if (b->exec) cudaGraphExecDestroy(b->exec);
    if (b->own) cudaStreamDestroy(b->own);
    if (b->side) cudaStreamDestroy(b->side);
    if (b->ev_fork) cudaEventDestroy(b->ev_fork);
    if (b->ev_join) cudaEventDestroy(b->ev_join);
    if (b->ev_in) cudaEventDestroy(b->ev_in);
    if (b->ev_out) cudaEventDestroy(b->ev_out);
    cudaFree(b->voff);
    cudaFree(b->order);
    cudaFree(b->work);
    cudaFree(b->geo);
    for (void* p : {(void*)b->rorder[0], (void*)b->rorder[1], (void*)b->soff, (void*)b->sgraph,
                    (void*)b->base, (void*)b->units, (void*)b->skip, (void*)b->sdesc,
                    (void*)b->deg, (void*)b->perm, (void*)b->rank, (void*)b->cuts, (void*)b->tk})
        cudaFree(p);
    if (b->wait_failed) cudaFreeHost(b->wait_failed);
    cudaFree(b->tmp);
    cudaFree(b->pos[0]);
    cudaFree(b->pos[1]);
    cudaFree(b->stage);
    gila_graph_destroy(b->g);
    delete b;
}

gila_status gila_batch_set_stream(gila_batch* b, void* cuda_stream)
{
    if (!b) return fail(GILA_EINVAL, "batch is NULL");
    b->user = (cudaStream_t)cuda_stream;
    return gila_graph_set_stream(b->g, cuda_stream);
}

gila_status gila_batch_set_wait_test(gila_batch* b, int32_t on)
{
    if (!b) return fail(GILA_EINVAL, "batch is NULL");
    b->wait_test = on ? 1 : 0;
    return GILA_OK;
}

gila_status gila_batch_info(const gila_batch* b, int32_t* count, int64_t* total_n,
                            int64_t* nnz_khop)
{
    if (!b) return fail(GILA_EINVAL, "batch is NULL");
    if (count) *count = b->count;
    if (total_n) *total_n = b->g->n;
    if (nnz_khop) *nnz_khop = b->g->k_built ? b->g->nnz_khop : 0;
    return GILA_OK;
}

gila_status gila_batch_build_khop(gila_batch* b, int32_t k, int64_t* nnz_out)
{
    if (!b) return fail(GILA_EINVAL, "batch is NULL");
    return gila_build_khop(b->g, k, nnz_out);
}

gila_status gila_batch_khop_reset(gila_batch* b)
{
    if (!b) return fail(GILA_EINVAL, "batch is NULL");
    return gila_khop_reset(b->g);
}

gila_status gila_batch_khop_export(const gila_batch* b, int64_t* krow_host, int32_t* kcol_host)
{
    if (!b) return fail(GILA_EINVAL, "batch is NULL");
    return gila_khop_export(b->g, krow_host, kcol_host);
}

gila_status gila_batch_tune(gila_batch* b, const gila_batch_tuning* t)
{
    if (!b || !t) return fail(GILA_EINVAL, "batch or tuning is NULL");
    if (t->threads != 0 && t->threads != 256 && t->threads != 512 && t->threads != 1024)
        return fail(GILA_EINVAL, "threads must be 256, 512 or 1024");
    if (t->ctas_per_sm < 0 || t->ctas_per_sm > 8) return fail(GILA_EINVAL, "ctas_per_sm in [0, 8]");
    b->tune = *t;
    return GILA_OK;
}

gila_status gila_batch_get_tuning(const gila_batch* b, int32_t precision, gila_batch_tuning* out)
{
    if (!b || !out) return fail(GILA_EINVAL, "batch or out is NULL");
    (void)precision;
    *out = reported(b->tune);
    return GILA_OK;
}

gila_status gila_batch_autotune(gila_batch* b, const gila_params* prm, const void* pos_dev,
                                int32_t probe_iters, gila_batch_tuning* chosen)
{
    if (!b) return fail(GILA_EINVAL, "batch is NULL");
    gila_status s = check_batch_params(prm);
    if (s != GILA_OK) return s;
    if (probe_iters < 1) return fail(GILA_EINVAL, "probe_iters must be >= 1");
    gila_graph* g = b->g;
    if (g->n > 0 && !pos_dev) return fail(GILA_EINVAL, "placement is NULL");
    GILA_CUDA(cudaSetDevice(g->device));
    s = gila_build_khop(g, prm->k, nullptr);
    if (s != GILA_OK) return s;
    const size_t esz = is_f64(prm->precision) ? 16 : 8;
    const size_t bytes = esz * (size_t)g->n;
    if ((s = ensure(&b->pos[1], &b->pos_cap[1], bytes)) != GILA_OK) return s;
    gila_params q = *prm;
    q.iters = probe_iters;
    static const int kThreadsSet[3] = {256, 512, 1024};
    static const int kCtasSet[4] = {1, 2, 4, 8};
    // no groups set: rows per lane where they apply
    static const int kGroups[4][3] = {{0, 0, 0}, {8, 24, 64}, {4, 12, 32}, {16, 48, 128}};
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    GILA_CUDA(cudaEventCreate(&e0));
    GILA_CUDA(cudaEventCreate(&e1));
    const gila_batch_tuning saved = b->tune;
    gila_batch_tuning best = saved;
    float best_ms = INFINITY;
    s = GILA_OK;
    for (int ti = 0; ti < 3 && s == GILA_OK; ++ti)
        for (int ci = 0; ci < 4 && s == GILA_OK; ++ci) {
            if (kCtasSet[ci] * kThreadsSet[ti] > 2048) continue;
            for (int gi = 0; gi < 4 && s == GILA_OK; ++gi) {
                gila_batch_tuning c = {kThreadsSet[ti], kCtasSet[ci], kGroups[gi][0],
                                       kGroups[gi][1], kGroups[gi][2]};
                b->tune = c;
                float ms = 0.0f;
                for (int rep = 0; rep < 2 && s == GILA_OK; ++rep) {  // first run captures
                    if (bytes)
                        cudaMemcpyAsync(b->pos[1], pos_dev, bytes, cudaMemcpyDeviceToDevice,
                                        b->user);
                    cudaEventRecord(e0, b->user);
                    s = batch_run(b, &q, b->pos[1]);
                    cudaEventRecord(e1, b->user);
                }
                if (s != GILA_OK) break;
                cudaError_t e = cudaEventSynchronize(e1);
                if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, e0, e1);
                if (e != cudaSuccess) {
                    s = cuda_fail(e, "autotune timing");
                    break;
                }
                if ((s = batch_wait_failed(b)) != GILA_OK) break;
                if (ms < best_ms) {
                    best_ms = ms;
                    best = c;
                }
            }
        }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    b->tune = (s == GILA_OK) ? best : saved;
    if (s != GILA_OK) return s;
    if (chosen) *chosen = reported(b->tune);
    return GILA_OK;
}

gila_status gila_layout_batch_device(gila_batch* b, const gila_params* prm, void* pos_dev_inout)
{
    if (!b) return fail(GILA_EINVAL, "batch is NULL");
    gila_status s = check_batch_params(prm);
    if (s != GILA_OK) return s;
    if (b->g->n > 0 && !pos_dev_inout) return fail(GILA_EINVAL, "placement is NULL");
    GILA_CUDA(cudaSetDevice(b->g->device));
    s = gila_build_khop(b->g, prm->k, nullptr);
    if (s != GILA_OK) return s;
    return batch_run(b, prm, pos_dev_inout);
}

gila_status gila_layout_batch_run(gila_batch* b, const gila_params* prm, const double* pos_in_host,
                                  double* pos_out_host)
{
    if (!b) return fail(GILA_EINVAL, "batch is NULL");
    gila_status s = check_batch_params(prm);
    if (s != GILA_OK) return s;
    gila_graph* g = b->g;
    if (g->n > 0 && (!pos_in_host || !pos_out_host)) return fail(GILA_EINVAL, "placement is NULL");
    GILA_CUDA(cudaSetDevice(g->device));
    s = gila_build_khop(g, prm->k, nullptr);
    if (s != GILA_OK) return s;
    if (g->n == 0) return GILA_OK;
    const size_t n = (size_t)g->n;
    const bool f64 = is_f64(prm->precision);
    const size_t esz = f64 ? 16 : 8;
    if ((s = ensure(&b->pos[0], &b->pos_cap[0], esz * n)) != GILA_OK) return s;
    if (!f64 && (s = ensure((void**)&b->stage, &b->stage_cap, 16 * n)) != GILA_OK) return s;
    if (f64) {
        GILA_CUDA(cudaMemcpyAsync(b->pos[0], pos_in_host, 16 * n, cudaMemcpyHostToDevice, b->user));
    } else {
        GILA_CUDA(cudaMemcpyAsync(b->stage, pos_in_host, 16 * n, cudaMemcpyHostToDevice, b->user));
        if ((s = convert_positions(g, prm->precision, b->stage, b->pos[0], true)) != GILA_OK)
            return s;
    }
    if ((s = batch_run(b, prm, b->pos[0])) != GILA_OK) return s;
    if (f64) {
        GILA_CUDA(cudaMemcpyAsync(pos_out_host, b->pos[0], 16 * n, cudaMemcpyDeviceToHost, b->user));
    } else {
        if ((s = convert_positions(g, prm->precision, b->stage, b->pos[0], false)) != GILA_OK)
            return s;
        GILA_CUDA(cudaMemcpyAsync(pos_out_host, b->stage, 16 * n, cudaMemcpyDeviceToHost, b->user));
    }
    GILA_CUDA(cudaStreamSynchronize(b->user));
    return batch_wait_failed(b);
}

gila_status gila_layout_batch(gila_graph* const* gs, int32_t count, const gila_params* prm,
                              const double* const* pos_in, double* const* pos_out)
{
    if (count < 0) return fail(GILA_EINVAL, "count must be >= 0");
    if (count > 0 && (!gs || !pos_in || !pos_out)) return fail(GILA_EINVAL, "array is NULL");
    gila_status s = check_batch_params(prm);
    if (s != GILA_OK) return s;
    if (count == 0) return GILA_OK;
    for (int32_t i = 0; i < count; ++i)
        if (!gs[i] || gs[i]->device != gs[0]->device)
            return fail(GILA_EINVAL, "graphs must be non-NULL and on one device");
    GILA_CUDA(cudaSetDevice(gs[0]->device));
    cudaStream_t st = gs[0]->stream;
    // pack the graphs' device CSRs into one union graph
    std::vector<int64_t> voff(count + 1, 0), eoff(count + 1, 0);
    std::vector<PackSrc> src(count);
    for (int32_t i = 0; i < count; ++i) {
        voff[i + 1] = voff[i] + gs[i]->n;
        eoff[i + 1] = eoff[i] + gs[i]->nnz_adj;
        src[i] = PackSrc{gs[i]->row, gs[i]->col, gs[i]->n, voff[i], eoff[i]};
    }
    if (voff[count] >= ((int64_t)1 << 31)) return fail(GILA_EINVAL, "batch has too many vertices");
    gila_batch* b = new (std::nothrow) gila_batch();
    if (!b) return fail(GILA_ENOMEM, "host allocation");
    b->g = new (std::nothrow) gila_graph();
    if (!b->g) {
        delete b;
        return fail(GILA_ENOMEM, "host allocation");
    }
    gila_graph* g = b->g;
    g->device = gs[0]->device;
    g->n = voff[count];
    g->nnz_adj = eoff[count];
    g->stream = st;
    b->user = st;
    b->count = count;
    b->voff_h = voff;
    PackSrc* dsrc = nullptr;
    cudaError_t e = cudaMalloc(&g->row, sizeof(int64_t) * (size_t)(g->n + 1));
    if (e == cudaSuccess) e = cudaMalloc(&g->col, sizeof(int32_t) * (size_t)std::max<int64_t>(g->nnz_adj, 1));
    if (e == cudaSuccess) e = cudaMalloc(&dsrc, sizeof(PackSrc) * count);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(dsrc, src.data(), sizeof(PackSrc) * count, cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) {
        pack_kernel<<<count, 256, 0, st>>>(dsrc, g->row, g->col);
        count_launch();
        e = cudaGetLastError();
    }
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(g->row + g->n, &eoff[count], sizeof(int64_t), cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    cudaFree(dsrc);
    if (e != cudaSuccess) {
        gila_batch_destroy(b);
        return cuda_fail(e, "batch pack");
    }
    s = batch_finish_create(b);
    std::vector<double> in, outv;
    if (s == GILA_OK) {
        in.resize(2 * (size_t)g->n);
        outv.resize(2 * (size_t)g->n);
        for (int32_t i = 0; i < count; ++i)
            if (gs[i]->n > 0)
                memcpy(in.data() + 2 * voff[i], pos_in[i], sizeof(double) * 2 * gs[i]->n);
        s = gila_layout_batch_run(b, prm, in.data(), outv.data());
    }
    if (s == GILA_OK)
        for (int32_t i = 0; i < count; ++i)
            if (gs[i]->n > 0)
                memcpy(pos_out[i], outv.data() + 2 * voff[i], sizeof(double) * 2 * gs[i]->n);
    gila_batch_destroy(b);
    return s;
}

}  // extern "C"
