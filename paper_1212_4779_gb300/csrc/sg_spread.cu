// sg_spread.cu -- seed-set spread snapshot by snapshot: a block walks one
// snapshot at a time with one visited bit per node in shared memory.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "sg_internal.cuh"

namespace sgi {

namespace {

constexpr unsigned FULL_WARP = 0xffffffffu;
constexpr int SPREAD_U = 4;                         // arcs in flight per lane
constexpr int SPREAD_ROW = 64;                      // arcs from which a row is read straight
constexpr int SPREAD_HUB = 512;                     // ... and from which the whole block shares it
constexpr int SPREAD_HUBS = 128;                    // such rows remembered per level
constexpr size_t SPREAD_SMEM = (size_t)216 << 10;   // shared memory of one SM for visited bits ...
constexpr size_t SPREAD_FIXED = 3200;               // ... and what a block takes beside them
constexpr size_t SPREAD_DYNAMIC = SPREAD_SMEM - SPREAD_FIXED + 1024 * 4;  // most a launch asks for

struct SpreadView {
    int32_t n, R, ns, words, none_live;
    const int32_t *rp, *col;
    const uint2 *fw;
    uint64_t seed;
    uint32_t uic_tm1;
    const int32_t *S;
    int32_t *queue;              // [blocks][n]
    unsigned long long *next;    // snapshot counter
    long long *total;
    unsigned long long *edges;
};

// One arc's coin in the snapshot whose seed word is s = seed ^ (r << 40),
// then its destination's visited bit; fresh destinations go to the queue.
template <int MODEL, int U>
__device__ __forceinline__ void spread_arcs(const SpreadView &a, uint64_t s, const int (&e)[U], uint32_t *seen,
                                            int32_t *queue, int *tail)
{
    int y[U];
    uint32_t tm1[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
        y[u] = 0;
        tm1[u] = a.uic_tm1;
        if (e[u] < 0) continue;
        if (MODEL == MODEL_WIC) {
            const uint2 w = __ldg(a.fw + e[u]);
            y[u] = (int)w.x;
            tm1[u] = w.y;
        } else {
            y[u] = __ldg(a.col + e[u]);
        }
    }
    bool live[U];
#pragma unroll
    for (int u = 0; u < U; ++u)
        live[u] = e[u] >= 0 && !a.none_live && coin_hi32(s ^ (uint64_t)(uint32_t)e[u], 0u) <= tm1[u];
    // one arc in twenty is live here: a lane's own push is cheaper than a
    // ballot for every arc
#pragma unroll
    for (int u = 0; u < U; ++u) {
        if (!live[u]) continue;
        const uint32_t bit = 1u << (y[u] & 31);
        if (!(atomicOr(&seen[y[u] >> 5], bit) & bit)) queue[atomicAdd(tail, 1)] = y[u];
    }
}

// Reached nodes and their out-degrees over the R snapshots.  The walk draws
// the coins of every reached node's arcs once per snapshot, which is what it
// cannot do without: R-MAT 20, its 50 largest out-degrees as seeds and 20,000
// snapshots draw 40 G coins (53 ms at the rate snap_coins_kernel draws them),
// in 136 ms here against 319 ms bit-sliced, where most of the time went into
// scattered records (R = 100: 1.2 against 155 ms, one block per word).  Bound
// by issue (65 %), a third of it the coins.  A snapshot at a time keeps the
// whole visited set on the SM (128 KB for a million nodes) and the arcs in L2;
// the bit-sliced walks it replaces kept 16 bytes a node and word for all words
// in flight, 5 GB of scattered records.  A warp takes
// 32 nodes of the level: their short rows spread over the lanes, a longer
// one by the whole warp; hub rows wait for the next level, where all warps
// share them (left to the warp that met them, the others waited two thirds
// of the time).
template <int MODEL>
__global__ void __launch_bounds__(1024) spread_snapshots_kernel(SpreadView a)
{
    extern __shared__ __align__(16) uint32_t seen[];
    __shared__ int head, tail, snap, nhub[2];
    __shared__ int2 hub[2][SPREAD_HUBS];  // (first arc, arcs)
    const int tid = threadIdx.x, lane = tid & 31, T = blockDim.x, wid = tid >> 5, nw = T >> 5;
    // per warp: first arc minus offset of the batch's nonempty rows
    int *first = reinterpret_cast<int *>(seen + a.words) + 32 * wid;
    int32_t *queue = a.queue + (size_t)blockIdx.x * (size_t)a.n;
    unsigned long long edges = 0;
    long long total = 0;
    while (true) {
        __syncthreads();
        if (tid == 0) {
            snap = (int)min(atomicAdd(a.next, 1ull), (unsigned long long)a.R);
            tail = 0;
            nhub[0] = 0;
            nhub[1] = 0;
        }
        int4 *s4 = reinterpret_cast<int4 *>(seen);
        for (int i = tid; i < a.words / 4; i += T) s4[i] = make_int4(0, 0, 0, 0);
        __syncthreads();
        const int r = snap;
        if (r >= a.R) break;
        const uint64_t s = a.seed ^ ((uint64_t)(uint32_t)r << 40);
        // arcs t .. t + 32 SPREAD_U - 1 (below end) of the row at arc p
        auto straight = [&](int p, int t, int end) {
            int e[SPREAD_U];
#pragma unroll
            for (int u = 0; u < SPREAD_U; ++u) e[u] = t + 32 * u + lane < end ? p + t + 32 * u + lane : -1;
            spread_arcs<MODEL, SPREAD_U>(a, s, e, seen, queue, &tail);
        };
        for (int j = tid; j < a.ns; j += T) {
            const int x = __ldg(a.S + j);
            const uint32_t bit = 1u << (x & 31);
            if (!(atomicOr(&seen[x >> 5], bit) & bit)) queue[atomicAdd(&tail, 1)] = x;  // repeated seeds count once
        }
        int par = 0;
        for (int lo = 0;; par ^= 1) {
            __syncthreads();
            const int hi = tail, nh = min(nhub[par], SPREAD_HUBS);
            if (tid == 0) head = lo;
            __syncthreads();
            if (lo >= hi && nh == 0) break;
            if (tid == 0) nhub[par] = 0;  // read by all before the barrier; filled again two levels on
            int before = 0;  // chunks of the hub rows before this one
            for (int k = 0; k < nh; ++k) {
                const int2 h = hub[par][k];
                const int chunks = (h.y + SPREAD_HUB - 1) / SPREAD_HUB;
                for (int c = (wid + nw - before % nw) % nw; c < chunks; c += nw) {
                    const int end = min(h.y, (c + 1) * SPREAD_HUB);
                    for (int t = c * SPREAD_HUB; t < end; t += 32 * SPREAD_U) straight(h.x, t, end);
                }
                before += chunks;
            }
            while (true) {
                int b = 0;
                if (lane == 0) b = atomicAdd(&head, 32);
                b = __shfl_sync(FULL_WARP, b, 0);
                if (b >= hi) break;
                int beg = 0, deg = 0;
                if (b + lane < hi) {
                    const int x = queue[b + lane];
                    beg = __ldg(a.rp + x);
                    deg = __ldg(a.rp + x + 1) - beg;
                }
                edges += (unsigned long long)deg;
                bool own = deg >= SPREAD_ROW;  // a row the warp reads straight
                if (deg > SPREAD_HUB) {
                    const int h = atomicAdd(&nhub[par ^ 1], 1);
                    if (h < SPREAD_HUBS) {
                        hub[par ^ 1][h] = make_int2(beg, deg);
                        own = false;
                    }
                }
                for (unsigned big = __ballot_sync(FULL_WARP, own); big; big &= big - 1u) {
                    const int k = __ffs(big) - 1;
                    const int p = __shfl_sync(FULL_WARP, beg, k), d = __shfl_sync(FULL_WARP, deg, k);
                    for (int t = 0; t < d; t += 32 * SPREAD_U) straight(p, t, d);
                }
                const int small = deg < SPREAD_ROW ? deg : 0;
                int inc = small;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int v = __shfl_up_sync(FULL_WARP, inc, o);
                    if (lane >= o) inc += v;
                }
                const int all = __shfl_sync(FULL_WARP, inc, 31), ex = inc - small;
                // Short rows: arc j of the batch belongs to the last nonempty
                // row starting at or before j.  The rows' starts within 32
                // arcs are a bit mask, so that is a population count.
                const unsigned ne = __ballot_sync(FULL_WARP, small > 0);
                if (small > 0) first[__popc(ne & ((1u << lane) - 1u))] = beg - ex;
                __syncwarp();
                int rows = 0;  // nonempty rows starting before the window
                for (int t = 0; t < all; t += 32 * SPREAD_U) {
                    int e[SPREAD_U];
#pragma unroll
                    for (int u = 0; u < SPREAD_U; ++u) {
                        const int j = t + 32 * u + lane, at = ex - t - 32 * u;
                        const unsigned starts =
                            __reduce_or_sync(FULL_WARP, small > 0 && (unsigned)at < 32u ? 1u << at : 0u);
                        const int k = rows + __popc(starts & (FULL_WARP >> (31 - lane))) - 1;
                        e[u] = j < all ? first[k] + j : -1;
                        rows += __popc(starts);
                    }
                    spread_arcs<MODEL, SPREAD_U>(a, s, e, seen, queue, &tail);
                }
                __syncwarp();
            }
            lo = hi;
        }
        total += tail;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) edges += __shfl_xor_sync(FULL_WARP, edges, o);
    if (lane == 0 && edges) atomicAdd(a.edges, edges);
    if (tid == 0 && total) atomicAdd((unsigned long long *)a.total, (unsigned long long)total);
}

}  // namespace

// LT draws per node, not per arc; above 1.7 M nodes the bits do not fit.  A
// snapshot takes a block a few microseconds however little it reaches, so many
// snapshots of a small graph go faster 64 at a time.  Six cascades (mean live
// degree 0.1 to 2.5) from 1, 10 and 100 seeds on uniform and power-law graphs,
// bit-sliced time over this one's, geometric means:
//       R =      4,000  20,000  100,000
//   n =    200    1.26    0.85     0.57
//   n =  1,000    1.64    1.06     0.75
//   n =  4,000    2.17    1.28     0.92
//   n = 16,000    2.74    1.52     1.14
// so the line lies at R = 800 sqrt(n).
bool spread_by_snapshot(const sg_graph *g, const Coins &co)
{
    return !co.lt && ((size_t)g->n + 127) / 128 * 16 + SPREAD_FIXED <= SPREAD_SMEM &&
           (double)co.R * co.R <= 640000.0 * (double)g->n;
}

sg_status run_spread_snapshots(sg_graph *g, const Coins &co, int model, const int32_t *d_S, int32_t ns,
                               long long *d_total, unsigned long long *d_edges, cudaStream_t st)
{
    SpreadView a{};
    a.n = (int32_t)g->n;
    a.R = co.R;
    a.ns = ns;
    a.none_live = co.none_live;
    a.words = (int32_t)((g->n + 127) / 128 * 4);
    a.rp = g->rp.p;
    a.col = g->col.p;
    a.fw = g->fw.p;
    a.seed = co.seed;
    a.uic_tm1 = co.uic_tm1;
    a.S = d_S;
    a.total = d_total;
    a.edges = d_edges;
    // as many blocks per SM as their bits allow, sharing 2048 threads
    const size_t bits = (size_t)a.words * 4;
    const int per = (int)std::max<size_t>(1, std::min<size_t>(16, SPREAD_SMEM / (bits + SPREAD_FIXED)));
    const int T = std::min(1024, 2048 / per / 32 * 32);
    const int blocks = std::min(g->num_sms * per, co.R);
    const size_t smem = bits + (size_t)T * 4;
    DBuf<int32_t> queue;
    DBuf<unsigned long long> next;
    sg_status rc = SG_OK;
    if ((rc = dbuf_alloc(queue, (size_t)blocks * (size_t)g->n, st)) != SG_OK) return rc;
    if ((rc = dbuf_alloc(next, 1, st)) != SG_OK) {
        dbuf_free(queue, st);
        return rc;
    }
    a.queue = queue.p;
    a.next = next.p;
    // The limit belongs to the kernel, not to the call: every call sets the same,
    // so that none lowers it between another thread's set-up and launch.
    auto kern = model == MODEL_WIC ? spread_snapshots_kernel<MODEL_WIC> : spread_snapshots_kernel<MODEL_UIC>;
    if (cudaMemsetAsync(next.p, 0, 8, st) != cudaSuccess ||
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SPREAD_DYNAMIC) != cudaSuccess) {
        set_error("sg_spread: launch set-up failed");
        rc = SG_ECUDA;
    } else {
        kern<<<blocks, T, smem, st>>>(a);
        if (cudaGetLastError() != cudaSuccess) {
            set_error("sg_spread: launch failed");
            rc = SG_ECUDA;
        }
        ++g_launches;
    }
    dbuf_free(queue, st);
    dbuf_free(next, st);
    return rc;
}

}  // namespace sgi
