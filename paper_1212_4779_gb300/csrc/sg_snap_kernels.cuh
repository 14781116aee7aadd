// sg_snap_kernels.cuh -- device kernels of the compact snapshot graphs (the
// default route of a selection; sg_snap.cu launches them).
//
// Every snapshot's live graph is laid out once per query and contracted to
// what reachability counts need.  In snapshot r:
//   internal node   a node with a live out-arc (others reach only themselves)
//   join            a node with two or more live in-arcs, or the lowest node
//                   of a cycle of nodes with one live in-arc each
//   tree            every other node has at most one live in-arc, so below
//                   each join (and each node without in-arcs) hangs a tree;
//                   T(v) is the subtree of v in it
// T(v) is entered only through v, so |R(v)| = |T(v)| + the sizes |T(j)| of
// the joins j reachable from v.  Tree nodes are laid out so that the arcs
// leaving T(v) towards joins are one contiguous range J(v) of the snapshot's
// join-arc list; a count is a closure walk over join ids alone, with one
// visited bit per join.
// On R-MAT 20 under the weighted cascade a snapshot's 450 K live arcs leave
// 80 K joins (62 K of them with no join arc of their own), 179 K join arcs
// and 28 K ranges to walk, 3 M arc visits in all, where walking the nodes
// themselves visits 22 M; the snapshot takes about 4 MB, so the walks of a
// few snapshots at a time stay in L2 and their visited bits in shared
// memory.  The initial gains of R = 256 snapshots take 38 ms so, bitmaps and
// graphs included, where the tiered engines take 347 ms.
//
// A selection round covers R(v*) in each snapshot (closed under
// reachability, so later walks skip covered joins), marks the uncovered
// nodes that reach a newly covered join, and subtracts from each of them
// the newly covered nodes it reaches: all of them for the ancestors of v*,
// else a closure walk restricted to the marked and newly covered joins.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "sg_internal.cuh"

namespace sgi {
namespace {

constexpr unsigned SN_FULL = 0xffffffffu;
constexpr int SN_T = 1024;      // most threads of the one-block-per-snapshot kernels
constexpr int EX_U = 4;         // most elements a thread of sn_expand_n has in flight
constexpr int SN_TILE = 256;    // arcs or nodes per block pass of the bit transposes
constexpr int WK_T = 512;       // threads of the closure walks
constexpr int WK_W = WK_T / 32;
constexpr int WK_QS = 128;      // queue entries of a walk in shared memory
constexpr int WK_QG = 8192;     // ... and in global memory
constexpr int WK_TS = 128;      // visited joins remembered for a cheap undo
constexpr int WK_CH = 16;       // most tasks a warp claims at a time (initial gains; rounds: one per lane)
constexpr int SW_CAP = 16;      // joins a one-thread walk may visit
constexpr int SW_ARCS = 96;     // ... and arcs it may scan
constexpr int SW_U = 4;         // ... several at a time
constexpr int WK_U = 4;         // arcs in flight per lane
constexpr int ROUND_ONE = 2;    // tasks per chunk from which a round walks with single threads first
constexpr int LMK_LONG = 64;    // in-arcs of a join from which warps share their sum ...
constexpr int LMK_CHUNK = 2048; // ... this many a warp
constexpr int LMK_MORE = 512;  // joins of a landmark's component from which another landmark is looked for ...
constexpr int LMK_FAR = 64;    // ... with at least this part of the first one's score
constexpr int ROUND_LMK = 512;  // newly covered joins from which a round has a landmark
constexpr uint32_t CV_CYCLE = 0x80000000u;
constexpr uint32_t ARC_LEAF = 0x80000000u;  // jarc: the join has no live out-arc (weight 1, nothing below)

__device__ __forceinline__ uint64_t sn_word_mask(int word, int R)
{
    const int rem = R - word * 64;
    return rem >= 64 ? ~0ull : ((1ull << rem) - 1ull);
}

__device__ __forceinline__ bool sn_bit(const uint32_t *b, int i) { return (b[i >> 5] >> (i & 31)) & 1u; }

// number of set bits of bitmap b below position i (p: exclusive prefix per word)
__device__ __forceinline__ int sn_rank(const uint32_t *b, const int32_t *p, int i)
{
    return p[i >> 5] + __popc(b[i >> 5] & ((1u << (i & 31)) - 1u));
}

// (j+1)-th lowest set bit of m, j < popc(m)
__device__ __forceinline__ int sn_nth_bit(uint32_t m, int j)
{
    int pos = 0;
#pragma unroll
    for (int w = 16; w >= 1; w >>= 1) {
        const int c = __popc(m & ((1u << w) - 1u));
        if (j >= c) {
            j -= c;
            m >>= w;
            pos += w;
        }
    }
    return pos;
}

__device__ __forceinline__ int sn_warp_incl(int v, int lane)
{
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(SN_FULL, v, o);
        if (lane >= o) v += u;
    }
    return v;
}

__device__ __forceinline__ unsigned long long sn_pack(int hi, uint32_t lo)
{
    return ((unsigned long long)(uint32_t)hi << 32) | lo;
}
__device__ __forceinline__ int sn_hi(unsigned long long w) { return (int)(w >> 32); }
__device__ __forceinline__ uint32_t sn_lo(unsigned long long w) { return (uint32_t)w; }
__device__ __forceinline__ unsigned long long sn_vol(const unsigned long long *p)
{
    return *(const volatile unsigned long long *)p;
}
__device__ __forceinline__ int sn_vol(const int32_t *p) { return *(const volatile int32_t *)p; }

// Exclusive block scan of v; sh[33].
__device__ __forceinline__ int sn_block_excl(int v, int *sh, int &total)
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int inc = sn_warp_incl(v, lane);
    __syncthreads();
    if (lane == 31) sh[wid] = inc;
    __syncthreads();
    const int wi = sn_warp_incl(lane < nw ? sh[lane] : 0, lane);
    total = __shfl_sync(SN_FULL, wi, 31);
    const int before = __shfl_sync(SN_FULL, wi, (wid + 31) & 31);
    return (wid ? before : 0) + inc - v;
}

// Exclusive offset of one int per warp; sh[33].
__device__ __forceinline__ int sn_warp_offset(int v, int *sh, int &total)
{
    const int lane = threadIdx.x & 31;
    const int ex = sn_block_excl(lane == 0 ? v : 0, sh, total);
    return __shfl_sync(SN_FULL, ex, 0);
}

// Ranges of queue entries [q0, q1), spread evenly over the block: range(q)
// gives (first, length) of an entry, body(q, k) is called for each of its
// elements k.  Few entries hold most elements (hubs), so one warp per entry
// left most of the block idle.  The body may push to the queue: every thread
// has read its entries by then.  Ends with a barrier.
struct ExpandShared {
    int sh[33];
    int ex[SN_T];
    int first[SN_T];
    int aux[SN_T];  // an entry's own word, where range() leaves one
};
// Up to 32 entries, most levels of most searches, need no scan over the block:
// each warp reads them all and finds its elements with shuffles, two barriers a
// level in place of four (15k nodes, WIC, k = 50: 5.36 -> 5.02 ms).  False, with
// nothing done, past `limit` elements.
template <class Range, class Body>
__device__ __forceinline__ bool sn_expand_short(int q0, int q1, int limit, Range range, Body body)
{
    const int lane = threadIdx.x & 31;
    int first = 0, len = 0;
    if (q0 + lane < q1) range(q0 + lane, first, len);
    const int inc = sn_warp_incl(len, lane), ex = inc - len;
    const int total = __shfl_sync(SN_FULL, inc, 31);
    __syncthreads();
    if (total > limit) return false;
    for (int a0 = threadIdx.x - lane; a0 < total; a0 += blockDim.x) {
        const int a = a0 + lane;
        int k = 0;
#pragma unroll
        for (int step = 16; step >= 1; step >>= 1)
            if (__shfl_sync(SN_FULL, ex, k + step) <= a) k += step;  // k + step <= 31
        const int f = __shfl_sync(SN_FULL, first, k), e = __shfl_sync(SN_FULL, ex, k);
        if (a < total) body(q0 + k, f + a - e);
        __syncwarp();
    }
    __syncthreads();
    return true;
}
template <class Range, class Body>
__device__ __forceinline__ void sn_expand(ExpandShared &S, int q0, int q1, Range range, Body body)
{
    const int tid = threadIdx.x, T = blockDim.x;
    if (q1 == q0) return;
    if (q1 - q0 <= 32 && sn_expand_short(q0, q1, INT32_MAX, range, body)) return;
    for (int b = q0; b < q1; b += T) {
        int first = 0, len = 0, total;
        if (b + tid < q1) range(b + tid, first, len);
        const int ex = sn_block_excl(len, S.sh, total);
        S.ex[tid] = ex;
        S.first[tid] = first;
        __syncthreads();
        const int n = min(T, q1 - b);
        for (int a = tid; a < total; a += T) {
            int lo = 0, hi = n - 1;
            while (lo < hi) {
                const int mid = (lo + hi + 1) >> 1;
                if (S.ex[mid] <= a) lo = mid;
                else hi = mid - 1;
            }
            body(b + lo, S.first[lo] + a - S.ex[lo]);
        }
        __syncthreads();
    }
}

// The same with U elements a thread at a time: body(q, k) takes arrays of U (q
// negative: no element) and can have the loads of all in flight, where one
// element after another is a chain of dependent accesses each.  U is EX_U, or 1
// where the block has a thread for every element (cover's node, landmark and
// arc passes; select: R-MAT 20 102.2 -> 92.4 ms, LT on 60k nodes 4.51 -> 3.91).
template <int U, class Body>
__device__ __forceinline__ void sn_expand_pass(const ExpandShared &S, int b, int n, int total, Body body)
{
    const int tid = threadIdx.x, T = blockDim.x;
    const int top = n > 1 ? 1 << (31 - __clz(n - 1)) : 0;
    for (int a = tid; a < total; a += U * T) {
        int q[U], k[U];
#pragma unroll
        for (int u = 0; u < U; ++u) q[u] = 0;
        for (int step = top; step; step >>= 1) {
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (q[u] + step < n && S.ex[q[u] + step] <= a + u * T) q[u] += step;
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            k[u] = S.first[q[u]] + a + u * T - S.ex[q[u]];
            q[u] = a + u * T < total ? b + q[u] : -1;
        }
        body(q, k);
    }
}
template <class Range, class Body>
__device__ __forceinline__ void sn_expand_n(ExpandShared &S, int q0, int q1, Range range, Body body)
{
    const int tid = threadIdx.x, T = blockDim.x;
    if (q1 == q0) return;
    if (q1 - q0 <= 32 && sn_expand_short(q0, q1, T, range, [&](int q, int k) {
            const int qa[1] = {q}, ka[1] = {k};
            body(qa, ka);
        }))
        return;
    for (int b = q0; b < q1; b += T) {
        int first = 0, len = 0, total;
        if (b + tid < q1) range(b + tid, first, len);
        const int ex = sn_block_excl(len, S.sh, total);
        S.ex[tid] = ex;
        S.first[tid] = first;
        __syncthreads();
        if (total <= T) sn_expand_pass<1>(S, b, min(T, q1 - b), total, body);
        else sn_expand_pass<EX_U>(S, b, min(T, q1 - b), total, body);
        __syncthreads();
    }
}

// A level-synchronous search over a queue in global memory.  Whoever pushes
// an entry also loads its range, beside the atomic that claims the entry, and
// leaves it in shared memory: a level is then two dependent memory accesses
// (element, claim) where reading queue and range first made it four.
struct QueueShared {
    int tail;
    int2 range[SN_T];
};
__device__ __forceinline__ void sn_push(QueueShared &Q, int32_t *queue, int x, int2 range)
{
    const int p = atomicAdd(&Q.tail, 1);
    queue[p] = x;
    Q.range[p & (SN_T - 1)] = range;
}
// Upward searches over internal nodes: the arcs into a join root as its
// range; a tree node has none, its marker goes on to the parent itself
// (a tree path is then one level, not one per node).
__device__ __forceinline__ int2 joins_above(int2 up) { return up.x < 0 ? make_int2(0, 0) : up; }
__device__ __forceinline__ void mark_path(QueueShared &Q, const int2 *up, uint32_t *marks, int32_t *queue, int i)
{
    while (true) {
        const uint32_t bit = 1u << (i & 31);
        const int2 e = up[i];
        if (atomicOr(&marks[i >> 5], bit) & bit) return;
        sn_push(Q, queue, i, joins_above(e));
        if (e.x >= 0) return;
        i = ~e.x;
    }
}
// Expands the queue from entry `from` until no level adds to it (entry(x)
// gives an entry's range where a level is too long for shared memory,
// body(k) takes the elements and may push); returns the queue's length.
// Starts and ends with a barrier.
template <class Entry, class Body>
__device__ __forceinline__ int sn_search(ExpandShared &S, QueueShared &Q, const int32_t *queue, int from, Entry entry,
                                         Body body)
{
    int h = from;
    __syncthreads();
    while (true) {
        const int t = Q.tail;
        if (h >= t) break;
        const bool held = t - h <= (int)blockDim.x;  // then all are read before any push
        sn_expand(
            S, h, t,
            [&](int q, int &first, int &len) {
                const int2 e = held ? Q.range[q & (SN_T - 1)] : entry(queue[q]);
                first = e.x;
                len = e.y;
            },
            [&](int, int k) { body(k); });
        h = t;
    }
    __syncthreads();
    return h;
}

// ------------------------------------------------------- coins to bitmaps

// Live bits of arcs, transposed to one bitmap over the arcs per snapshot,
// and per (word, node) the snapshots with a live out-arc (oany), a live
// in-arc (any) and two or more (join).  FROM 0: uniform coins, 1: weighted
// coins, 2: masks already drawn (lm [W][m]).  Each warp evaluates 32 arcs
// of one word, 64 coins per lane, and turns the 64 x 32 bits with ballots;
// rows leave the block 32 bytes at a time.  Bound by the coins' integer
// arithmetic (R-MAT 20, R = 256: 2.1 G coins in 2.9 ms); they are drawn once
// for both directions.
template <int FROM>
__global__ void __launch_bounds__(SN_TILE) snap_coins_kernel(SnapView v, Coins co, const uint2 *fw,
                                                             const unsigned long long *lm)
{
    __shared__ uint32_t tile[64][SN_TILE / 32];
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const long long tiles = (v.m + SN_TILE - 1) / SN_TILE;
    for (long long t = blockIdx.x; t < tiles; t += gridDim.x) {
        const long long e = t * SN_TILE + tid;
        const bool in = e < v.m;
        int y = 0, x = 0;
        uint32_t tm1 = co.uic_tm1;
        if (in) {
            x = __ldg(v.esrc + e);
            if (FROM == 1) {
                const uint2 a = __ldg(fw + e);
                y = (int)a.x;
                tm1 = a.y;
            } else {
                y = __ldg(v.col + e);
            }
        }
        const uint64_t base = co.seed ^ (uint64_t)e;
        for (int w = 0; w < v.W; ++w) {
            uint64_t mk = 0;
            if (in) {
                if (FROM == 2) {
                    mk = __ldg(lm + (long long)w * v.m + e);
                } else if (!co.none_live) {
                    const int nb = min(64, v.R - 64 * w);
                    uint32_t lo = 0, hi = 0;
#pragma unroll 8
                    for (int b = 0; b < min(32, nb); ++b)
                        lo |= (uint32_t)(coin_hi32(base, (uint32_t)(64 * w + b)) <= tm1) << b;
#pragma unroll 8
                    for (int b = 32; b < nb; ++b)
                        hi |= (uint32_t)(coin_hi32(base, (uint32_t)(64 * w + b)) <= tm1) << (b - 32);
                    mk = ((uint64_t)hi << 32) | lo;
                }
                if (mk) {
                    const size_t o = (size_t)w * (size_t)v.n;
                    atomicOr(&v.oany[o + x], (unsigned long long)mk);
                    const uint64_t dup = mk & atomicOr(&v.any[o + y], (unsigned long long)mk);
                    if (dup) atomicOr(&v.join[o + y], (unsigned long long)dup);
                }
            }
            uint32_t r0 = 0, r1 = 0;
            const uint32_t ml = (uint32_t)mk, mh = (uint32_t)(mk >> 32);
#pragma unroll
            for (int b = 0; b < 32; ++b) {
                const uint32_t b0 = __ballot_sync(SN_FULL, (ml >> b) & 1u), b1 = __ballot_sync(SN_FULL, (mh >> b) & 1u);
                if (lane == b) {
                    r0 = b0;
                    r1 = b1;
                }
            }
            tile[lane][wid] = r0;
            tile[lane + 32][wid] = r1;
            __syncthreads();
            for (int i = tid; i < 64 * (SN_TILE / 32); i += SN_TILE) {
                const int b = i / (SN_TILE / 32), k = i % (SN_TILE / 32);
                const int r = 64 * w + b;
                if (r < v.R) v.lb[(size_t)r * v.m32 + (size_t)t * (SN_TILE / 32) + k] = tile[b][k];
            }
            __syncthreads();
        }
    }
}

// Node bitmaps per snapshot (internal nodes, joins) from the bit-sliced
// words, and the part of the initial gains and of their edge count that
// needs no walk: a node without a live out-arc reaches itself.  A pass over
// memory (0.18 ms, R-MAT 20, R = 256).
__global__ void __launch_bounds__(SN_TILE) snap_nodes_kernel(SnapView v, Ctl *ctl, long long *s)
{
    __shared__ uint32_t to[64][SN_TILE / 32], tj[64][SN_TILE / 32];
    chain_start();
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int tiles = (v.n + SN_TILE - 1) / SN_TILE;
    unsigned long long ed = 0;
    for (int t = blockIdx.x; t < tiles; t += gridDim.x) {
        const int x = t * SN_TILE + tid;  // t * SN_TILE <= n < 2^31
        const bool in = x < v.n && x >= 0;
        long long own = 0;
        for (int w = 0; w < v.W; ++w) {
            uint64_t o = 0, j = 0;
            if (in) {
                o = v.oany[(size_t)w * (size_t)v.n + x];
                j = v.join[(size_t)w * (size_t)v.n + x];
                own += __popcll(sn_word_mask(w, v.R) & ~o);
            }
            uint32_t o0 = 0, o1 = 0, j0 = 0, j1 = 0;
#pragma unroll
            for (int b = 0; b < 32; ++b) {
                const uint32_t a0 = __ballot_sync(SN_FULL, (o >> b) & 1ull), a1 = __ballot_sync(SN_FULL, (o >> (b + 32)) & 1ull);
                const uint32_t c0 = __ballot_sync(SN_FULL, (j >> b) & 1ull), c1 = __ballot_sync(SN_FULL, (j >> (b + 32)) & 1ull);
                if (lane == b) {
                    o0 = a0;
                    o1 = a1;
                    j0 = c0;
                    j1 = c1;
                }
            }
            to[lane][wid] = o0;
            to[lane + 32][wid] = o1;
            tj[lane][wid] = j0;
            tj[lane + 32][wid] = j1;
            __syncthreads();
            for (int i = tid; i < 64 * (SN_TILE / 32); i += SN_TILE) {
                const int b = i / (SN_TILE / 32), k = i % (SN_TILE / 32);
                const int r = 64 * w + b;
                if (r < v.R) {
                    const size_t q = (size_t)r * v.n32 + (size_t)t * (SN_TILE / 32) + k;
                    v.outb[q] = to[b][k];
                    v.joinb[q] = tj[b][k];
                }
            }
            __syncthreads();
        }
        if (in) {
            s[x] = own;
            ed += (unsigned long long)own * (unsigned long long)(__ldg(v.rp + x + 1) - __ldg(v.rp + x));
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) ed += __shfl_xor_sync(SN_FULL, ed, o);
    if (lane == 0 && ed) atomicAdd(&ctl->init_edges, ed);
}

// ---------------------------------------------------------- per snapshot

// Set bits of a bitmap: totals per warp chunk of words.  Chunks are
// contiguous and a multiple of 32 words, so the order is kept.
__device__ __forceinline__ void sn_chunk(long long words, long long &lo, long long &hi)
{
    const int wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const long long per = ((words + nw - 1) / nw + 31) / 32 * 32;
    lo = min((long long)wid * per, words);
    hi = min(lo + per, words);
}

__device__ __forceinline__ int sn_chunk_count(const uint32_t *b, long long lo, long long hi)
{
    const int lane = threadIdx.x & 31;
    int c = 0;
    for (long long i = lo + lane; i < hi; i += 32) c += __popc(b[i]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(SN_FULL, c, o);
    return c;
}

// Internal nodes and live arcs of one snapshot, in node and arc order, with
// the direct counts of every internal node: itself and its leaf children
// (low half of acc), its arcs to joins (high half), their out-degrees, and
// the parent of every internal tree node.  One block a snapshot, as in all
// kernels that build and cover: its maps and lists are its own, so the steps
// need block barriers only.  Bound by scattered accesses to the node maps
// (115 M live arcs in 4.2 ms, R-MAT 20, R = 256).
__global__ void __launch_bounds__(SN_T) snap_compact_kernel(SnapView v, Ctl *ctl)
{
    __shared__ int sh[33];
    chain_start();
    const int r = blockIdx.x, tid = threadIdx.x, lane = tid & 31;
    const uint32_t *outb = v.outb + (size_t)r * v.n32, *joinb = v.joinb + (size_t)r * v.n32;
    const uint32_t *lb = v.lb + (size_t)r * v.m32;
    int32_t *outp = v.outp + (size_t)r * v.n32;
    const size_t io = (size_t)r * v.icap;
    SnapInfo *info = v.info + r;
    long long lo, hi, alo, ahi;
    sn_chunk(v.n32, lo, hi);
    sn_chunk(v.m32, alo, ahi);
    int nI, L;
    int off = sn_warp_offset(sn_chunk_count(outb, lo, hi), sh, nI);
    int aoff = sn_warp_offset(sn_chunk_count(lb, alo, ahi), sh, L);
    const bool bad = nI > v.icap || L > v.cap;
    if (tid == 0) {
        SnapInfo z{};
        z.nI = bad ? 0 : nI;
        z.L = bad ? 0 : L;
        z.bad = bad;
        *info = z;
        if (bad) atomicOr(&ctl->flags, FLAG_SNAPSHOT);
    }
    for (long long i0 = lo; i0 < hi; i0 += 32) {
        const long long i = i0 + lane;
        uint32_t b = i < hi ? outb[i] : 0u;
        const int c = __popc(b);
        const int inc = sn_warp_incl(c, lane);
        int p = off + inc - c;
        if (i < hi) outp[i] = p;
        off += __shfl_sync(SN_FULL, inc, 31);
        while (b && !bad) {
            const int x = (int)(i * 32) + __ffs(b) - 1;
            b &= b - 1;
            v.inode[io + p] = x;
            v.acc[io + p] = 1ull;
            v.deg[io + p] = (uint32_t)(__ldg(v.rp + x + 1) - __ldg(v.rp + x));
            v.par[io + p] = -1;
            v.pend[io + p] = 1;
            v.share[io + p] = -1;
            v.jid[io + p] = -1;
            v.cv[io + p] = 0;
            ++p;
        }
    }
    if (bad) return;
    __syncthreads();
    // live arcs: 32 words (1024 arcs) per warp step, spread over the lanes
    int2 *arc = v.arc + (size_t)r * v.cap;
    for (long long i0 = alo; i0 < ahi; i0 += 32) {
        const long long i = i0 + lane;
        const uint32_t b = i < ahi ? lb[i] : 0u;
        const int c = __popc(b);
        const int inc = sn_warp_incl(c, lane);
        const int total = __shfl_sync(SN_FULL, inc, 31), ex = inc - c;
        for (int j0 = 0; j0 < total; j0 += 32) {
            const int j = j0 + lane;
            int k = 0;
#pragma unroll
            for (int step = 16; step >= 1; step >>= 1)
                if (__shfl_sync(SN_FULL, ex, k + step) <= j) k += step;  // k + step <= 31
            const uint32_t wb = __shfl_sync(SN_FULL, b, k);
            const int wex = __shfl_sync(SN_FULL, ex, k);
            if (j < total) {
                const long long e = (i0 + k) * 32 + sn_nth_bit(wb, j - wex);
                const int y = __ldg(v.col + e);
                const int x = __ldg(v.esrc + e);
                const int xi = sn_rank(outb, outp, x);
                arc[aoff + j] = make_int2(xi, y);
                if (sn_bit(joinb, y)) {
                    atomicAdd(&v.acc[io + xi], 1ull << 32);
                } else if (sn_bit(outb, y)) {
                    v.par[io + sn_rank(outb, outp, y)] = xi;
                } else {
                    atomicAdd(&v.acc[io + xi], 1ull);
                    atomicAdd(&v.deg[io + xi], (uint32_t)(__ldg(v.rp + y + 1) - __ldg(v.rp + y)));
                }
            }
        }
        aoff += total;
    }
}

// Trees of one snapshot: cycles of one-parent nodes are cut at their lowest
// node (which becomes a join), subtree totals are summed towards the roots,
// and every node gets its absolute positions in the join-arc and node lists.
// Pointer doubling in place of level passes: a step is one dependent load for
// every node, and depth counts by its logarithm (4.2 ms, R-MAT 20, R = 256).
__global__ void __launch_bounds__(SN_T) snap_trees_kernel(SnapView v, Ctl *ctl)
{
    __shared__ int sh[33];
    __shared__ int changed, ncut;
    chain_start();
    const int r = blockIdx.x, tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, T = blockDim.x;
    SnapInfo *info = v.info + r;
    if (info->bad) return;
    const int nI = info->nI;
    const size_t io = (size_t)r * v.icap;
    const int32_t *inode = v.inode + io;
    int32_t *par = v.par + io, *pend = v.pend + io, *share = v.share + io;
    unsigned long long *acc = v.acc + io, *pj = v.pj + io, *pn = v.pn + io;
    uint32_t *deg = v.deg + io;
    uint32_t *joinb = v.joinb + (size_t)r * v.n32;
    int32_t *cut = v.apos + (size_t)r * v.cap;  // scratch here
    // Pointer doubling: pj = (an ancestor, lowest index on the path up to
    // it).  A round without a change leaves exactly the nodes above which
    // lies a cycle unrooted, each with the cycle's lowest index.
    for (int i = tid; i < nI; i += T) pj[i] = sn_pack(par[i] >= 0 ? par[i] : i, (uint32_t)i);
    if (tid == 0) ncut = 0;
    int rounds = 0;
    while (true) {
        __syncthreads();
        if (tid == 0) changed = 0;
        __syncthreads();
        for (int i = tid; i < nI; i += T) {
            if (par[i] < 0) continue;
            const unsigned long long w = pj[i];
            const int p = sn_hi(w);
            if (par[p] < 0) continue;  // rooted
            const unsigned long long q = sn_vol(pj + p);
            const uint32_t mn = min(sn_lo(w), sn_lo(q));
            *(volatile unsigned long long *)(pj + i) = sn_pack(sn_hi(q), mn);
            if (mn != sn_lo(w) || par[sn_hi(q)] < 0) changed = 1;
        }
        __syncthreads();
        if (!changed) break;
        if (++rounds > 64) {
            if (tid == 0) atomicOr(&ctl->flags, FLAG_SNAPSHOT);
            break;
        }
    }
    for (int i = tid; i < nI; i += T) {
        if (par[i] < 0) continue;
        const int p = sn_hi(pj[i]);
        if (par[p] < 0) continue;
        const int c = (int)sn_lo(pj[p]);
        const int x = inode[c];
        const uint32_t bit = 1u << (x & 31);
        if (!(atomicOr(&joinb[x >> 5], bit) & bit)) cut[atomicAdd(&ncut, 1)] = c;
    }
    __syncthreads();
    for (int k = tid; k < ncut; k += T) {
        const int c = cut[k];
        atomicAdd(&acc[par[c]], 1ull << 32);  // its in-arc leads to a join now
    }
    __syncthreads();
    for (int k = tid; k < ncut; k += T) par[cut[k]] = -1;
    __syncthreads();
    for (int i = tid; i < nI; i += T)
        if (par[i] >= 0) atomicAdd(&pend[par[i]], 1);
    __syncthreads();
    // Subtree sums: the last of a node's own thread and its children's
    // carries on upwards; what the parent had before is the child's offset.
    for (int i = tid; i < nI; i += T) {
        int c = i;
        while (atomicSub(&pend[c], 1) == 1) {
            const int p = par[c];
            if (p < 0) break;
            __threadfence_block();
            const unsigned long long a = sn_vol(acc + c);
            const uint32_t d = *(volatile uint32_t *)(deg + c);
            const unsigned long long old = atomicAdd(&acc[p], a);
            pj[c] = sn_pack(p, (uint32_t)sn_hi(old));
            pn[c] = sn_pack(p, sn_lo(old));
            atomicAdd(&deg[p], d);
            __threadfence_block();
            c = p;
        }
    }
    __syncthreads();
    // roots in index order
    {
        const int nw = T >> 5, per = ((nI + nw - 1) / nw + 31) / 32 * 32;
        const int lo = min(wid * per, nI), hi = min(lo + per, nI);
        int cj = 0, cn = 0;
        for (int i = lo + lane; i < hi; i += 32)
            if (par[i] < 0) {
                cj += sn_hi(acc[i]);
                cn += (int)sn_lo(acc[i]);
            }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            cj += __shfl_xor_sync(SN_FULL, cj, o);
            cn += __shfl_xor_sync(SN_FULL, cn, o);
        }
        int JA, N;
        int oj = sn_warp_offset(cj, sh, JA), on = sn_warp_offset(cn, sh, N);
        for (int i0 = lo; i0 < hi; i0 += 32) {
            const int i = i0 + lane;
            const bool root = i < hi && par[i] < 0;
            const int a = root ? sn_hi(acc[i]) : 0, b = root ? (int)sn_lo(acc[i]) : 0;
            const int ia = sn_warp_incl(a, lane), ib = sn_warp_incl(b, lane);
            if (root) {
                pj[i] = sn_pack(~i, (uint32_t)(oj + ia - a));
                pn[i] = sn_pack(~i, (uint32_t)(on + ib - b));
            }
            oj += __shfl_sync(SN_FULL, ia, 31);
            on += __shfl_sync(SN_FULL, ib, 31);
        }
        if (tid == 0) {
            info->JA = JA;
            info->N = N;
        }
    }
    // absolute positions: (ancestor or ~root, offset below it)
    rounds = 0;
    while (true) {
        __syncthreads();
        if (tid == 0) changed = 0;
        __syncthreads();
        for (int i = tid; i < nI; i += T) {
            const unsigned long long a = pj[i], b = pn[i];
            if (sn_hi(a) >= 0) {
                const unsigned long long q = sn_vol(pj + sn_hi(a));
                *(volatile unsigned long long *)(pj + i) = sn_pack(sn_hi(q), sn_lo(a) + sn_lo(q));
                changed = 1;
            }
            if (sn_hi(b) >= 0) {
                const unsigned long long q = sn_vol(pn + sn_hi(b));
                *(volatile unsigned long long *)(pn + i) = sn_pack(sn_hi(q), sn_lo(b) + sn_lo(q));
                changed = 1;
            }
        }
        __syncthreads();
        if (!changed) break;
        if (++rounds > 64) {
            if (tid == 0) atomicOr(&ctl->flags, FLAG_SNAPSHOT);
            break;
        }
    }
    // a child with its parent's whole range shares the parent's closure
    for (int i = tid; i < nI; i += T) {
        const int p = par[i], sj = sn_hi(acc[i]);
        if (p >= 0 && sj > 0 && sj == sn_hi(acc[p])) share[p] = i;
    }
    // joins in node order
    int32_t *joinp = v.joinp + (size_t)r * v.n32;
    long long lo, hi;
    sn_chunk(v.n32, lo, hi);
    int C;
    int off = sn_warp_offset(sn_chunk_count(joinb, lo, hi), sh, C);
    if (tid == 0) info->C = C;
    for (long long i0 = lo; i0 < hi; i0 += 32) {
        const long long i = i0 + lane;
        uint32_t b = i < hi ? joinb[i] : 0u;
        const int c = __popc(b);
        const int inc = sn_warp_incl(c, lane);
        int p = off + inc - c;
        if (i < hi) joinp[i] = p;
        off += __shfl_sync(SN_FULL, inc, 31);
        while (b) {
            v.jnode[(size_t)r * v.jcap + p] = (int)(i * 32) + __ffs(b) - 1;
            b &= b - 1;
            ++p;
        }
    }
}

// The chunks of tasks of every snapshot's two task segments, in order, and
// the most bits a walk needs (one block; cnt(r, seg) gives the lengths,
// ids(r) the bits).  A chunk is `chunk` tasks, fewer (not below `least`) when
// there would not be several chunks for each walking warp.
template <class F, class G>
__device__ __forceinline__ void sn_plan(const SnapView &v, int *sh, int least, int chunk, F cnt, G ids)
{
    const int tid = threadIdx.x, T = blockDim.x;
    __shared__ int most;
    __shared__ unsigned long long all;
    if (tid == 0) {
        most = 0;
        all = 0;
    }
    __syncthreads();
    for (int r = tid; r < v.R; r += T) {
        const int c = cnt(r, 0) + cnt(r, 1);
        if (c > 0) {
            atomicAdd(&all, (unsigned long long)c);
            atomicMax(&most, ids(r));
        }
    }
    __syncthreads();
    const int ch = (int)max((unsigned long long)least, min((unsigned long long)chunk, all / (unsigned long long)(8 * v.wwarps)));
    int carry = 0;
    for (int base = 0; base < 2 * v.R; base += T) {
        const int q = base + tid;
        int total;
        const int ex = sn_block_excl(q < 2 * v.R ? (cnt(q >> 1, q & 1) + ch - 1) / ch : 0, sh, total);
        if (q < 2 * v.R) v.cstart[q] = carry + ex;
        carry += total;
        __syncthreads();
    }
    if (tid == 0) {
        v.cstart[2 * v.R] = carry;
        v.cstart[2 * v.R + 1] = most;
        v.cstart[2 * v.R + 2] = ch;
        v.cstart[2 * v.R + 3] = 0;
        *v.cnext = 0;
    }
}

// Join-arc, join in-arc and node lists and join records of one snapshot,
// then its landmarks: joins x with many arcs below and many above.  Every
// node that reaches x reaches all of R(x), so those walks start from a copy of
// R(x)'s bits and total.  Bound by chains of an
// arc's map, rank and counter accesses (9 ms, R-MAT 20, R = 256); four arcs a
// thread in stages gave 1.6 % of a selection there and cost 3 % on a dense
// cascade of 97k nodes.  32 registers, so that two blocks share an SM (48 took
// that cascade from 10.5 to 10.7 ms).
__global__ void __launch_bounds__(SN_T, 2) snap_place_kernel(SnapView v)
{
    __shared__ ExpandShared S;
    __shared__ QueueShared Q;
    __shared__ unsigned long long best;
    __shared__ unsigned int lc, ld;
    __shared__ int nlong, inside;
    chain_start();
    const int r = blockIdx.x, tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, T = blockDim.x;
    SnapInfo *info = v.info + r;
    const int nI = info->nI, L = info->L, C = info->C;
    const size_t io = (size_t)r * v.icap, jo = (size_t)r * v.jcap, ao = (size_t)r * v.cap;
    const uint32_t *outb = v.outb + (size_t)r * v.n32, *joinb = v.joinb + (size_t)r * v.n32;
    const int32_t *outp = v.outp + (size_t)r * v.n32, *joinp = v.joinp + (size_t)r * v.n32;
    const unsigned long long *acc = v.acc + io, *pj = v.pj + io, *pn = v.pn + io;
    unsigned long long *fill = v.cv + io;
    int32_t *inoff = v.inoff + (size_t)r * (v.jcap + 1);
    uint32_t *jarc = v.jarc + ao;
    int2 *jin = v.jin + ao, *tn = v.tn + (size_t)r * v.tcap;
    int4 *rec = v.rec + jo;
    for (int c = tid; c <= C; c += T) inoff[c] = 0;
    if (tid == 0) {
        best = 0;
        lc = 0;
        ld = 0;
        Q.tail = 0;
    }
    for (int i = tid; i < nI; i += T) tn[sn_lo(pn[i])] = make_int2(v.inode[io + i], i);
    __syncthreads();
    for (int j = tid; j < L; j += T) {
        const int2 a = v.arc[ao + j];
        const bool out = sn_bit(outb, a.y);
        if (sn_bit(joinb, a.y)) {
            const int c = sn_rank(joinb, joinp, a.y);
            const int k = sn_hi(atomicAdd(&fill[a.x], 1ull << 32)) + (int)sn_lo(pj[a.x]);
            jarc[k] = (uint32_t)c | (out ? 0u : ARC_LEAF);
            v.apos[ao + j] = k;
            atomicAdd(&inoff[c + 1], 1);
        } else if (!out) {
            const int k = (int)sn_lo(atomicAdd(&fill[a.x], 1ull));
            tn[sn_lo(pn[a.x]) + 1 + k] = make_int2(a.y, -1);
        }
    }
    __syncthreads();
    // inoff[c + 1] = in-arcs of join c -> its start (shifted by one: the
    // fill below moves each to the join's end, the next one's start)
    {
        const int nw = T >> 5, per = ((C + nw - 1) / nw + 31) / 32 * 32;
        const int lo = min(wid * per, C), hi = min(lo + per, C);
        int s = 0, all;
        for (int c = lo + lane; c < hi; c += 32) s += inoff[c + 1];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(SN_FULL, s, o);
        int off = sn_warp_offset(s, S.sh, all);
        for (int c0 = lo; c0 < hi; c0 += 32) {
            const int c = c0 + lane;
            const int x = c < hi ? inoff[c + 1] : 0;
            const int inc = sn_warp_incl(x, lane);
            if (c < hi) inoff[c + 1] = off + inc - x;
            off += __shfl_sync(SN_FULL, inc, 31);
        }
    }
    // joins without out-arcs follow the trees in the node list
    const int trees = info->N;
    if (tid == 0) ld = 0;
    __syncthreads();
    for (int c = tid; c < C; c += T) {
        const int y = v.jnode[jo + c];
        if (sn_bit(outb, y)) {
            const int i = sn_rank(outb, outp, y);
            v.jid[io + i] = c;
            v.jtn[jo + c] = make_int2((int)sn_lo(pn[i]), (int)sn_lo(acc[i]));
            rec[c] = make_int4((int)sn_lo(acc[i]), (int)v.deg[io + i], (int)sn_lo(pj[i]), sn_hi(acc[i]));
        } else {
            const int p = trees + (int)atomicAdd(&ld, 1u);
            tn[p] = make_int2(y, -1);
            v.jtn[jo + c] = make_int2(p, 1);
            rec[c] = make_int4(1, __ldg(v.rp + y + 1) - __ldg(v.rp + y), 0, 0);
        }
    }
    __syncthreads();
    for (int j = tid; j < L; j += T) {
        const int2 a = v.arc[ao + j];
        if (sn_bit(joinb, a.y))
            jin[atomicAdd(&inoff[sn_rank(joinb, joinp, a.y) + 1], 1)] = make_int2(a.x, v.apos[ao + j]);
    }
    __syncthreads();
    int2 *up = v.up + io;
    for (int i = tid; i < nI; i += T) {
        const int p = v.par[io + i], j = v.jid[io + i];
        up[i] = p >= 0 ? make_int2(~p, 1) : (j >= 0 ? make_int2(inoff[j], inoff[j + 1] - inoff[j]) : make_int2(0, 0));
    }
    // landmarks: join arcs below times in-arcs up to two steps above.  A join
    // with many in-arcs is left to the warps: with one thread each, the 200,000
    // in-arcs of one join took 33 ms.
    auto above2 = [&](int k) -> unsigned long long {
        const int j = v.jid[io + ~sn_hi(pj[jin[k].x])];
        return 1ull + (j >= 0 ? (unsigned long long)(inoff[j + 1] - inoff[j]) : 0ull);
    };
    int32_t *scores = v.fb + io;
    auto score = [&](int c, unsigned long long up) {
        const unsigned long long sc = min(up * (unsigned long long)rec[c].w, (1ull << 31) - 1ull);
        if (C >= LMK_MORE) scores[c] = (int)sc;
        atomicMax(&best, (sc << 32) | (uint32_t)c);
    };
    unsigned long long *sums = reinterpret_cast<unsigned long long *>(Q.range);  // of the joins in S.aux
    if (tid == 0) nlong = 0;
    __syncthreads();
    for (int c = tid; c < C; c += T) {
        if (rec[c].w < 2) {
            if (C >= LMK_MORE) scores[c] = 0;
            continue;
        }
        if (inoff[c + 1] - inoff[c] > LMK_LONG) {
            const int q = atomicAdd(&nlong, 1);
            if (q < SN_T) {
                S.aux[q] = c;
                sums[q] = 0;
                continue;
            }
        }
        unsigned long long up = 0;
        for (int k = inoff[c]; k < inoff[c + 1]; ++k) up += above2(k);
        score(c, up);
    }
    __syncthreads();
    {
        const int nl = min(nlong, SN_T), nw = T >> 5;
        int before = 0;  // chunks of the joins before this one
        for (int q = 0; q < nl; ++q) {
            const int c = S.aux[q], k0 = inoff[c], k1 = inoff[c + 1];
            const int chunks = (k1 - k0 + LMK_CHUNK - 1) / LMK_CHUNK;
            for (int h = (wid + nw - before % nw) % nw; h < chunks; h += nw) {
                const int end = min(k1 - k0, (h + 1) * LMK_CHUNK);
                unsigned long long up = 0;
                for (int k = h * LMK_CHUNK + lane; k < end; k += 32) up += above2(k0 + k);
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) up += __shfl_xor_sync(SN_FULL, up, o);
                if (lane == 0) atomicAdd(&sums[q], up);
            }
            before += chunks;
        }
        __syncthreads();
        for (int q = tid; q < nl; q += T) score(S.aux[q], sums[q]);
    }
    __syncthreads();
    // Several large components need a landmark each: while the last one lies in
    // a component of many joins, the join with the best score among those that
    // reach none so far is the next.  A node's landmark is the first it reaches.
    const unsigned long long first = best >> 32;
    const int cw = (C + 31) >> 5, iw = (nI + 31) >> 5;
    uint32_t *lu = v.marki + (size_t)r * v.iw;
    int32_t *ql = v.jlist + jo, *qi = v.ilist + io;
    for (int i = tid; i < iw; i += T) lu[i] = 0;
    int from = 0, marks = 0;  // nodes above the landmarks before this one; landmarks
    for (int l = 0; l < SN_LMK; ++l) {
        if (l > 0) {
            __syncthreads();
            if (tid == 0) best = 0;
            __syncthreads();
            for (int c = tid; c < C; c += T) {
                const unsigned long long sc = (unsigned long long)scores[c];
                if (sc * LMK_FAR < first || sn_bit(lu, sn_rank(outb, outp, v.jnode[jo + c]))) continue;
                atomicMax(&best, (sc << 32) | (uint32_t)c);
            }
            __syncthreads();
        }
        if (!best) break;
        const int x = (int)(uint32_t)best;
        uint32_t *lr = l ? v.lmi + ((size_t)r * SN_LMK + l) * v.jw : v.lmr + (size_t)r * v.jw;
        for (int i = tid; i < cw; i += T) lr[i] = 0;
        if (tid == 0) {
            lc = 0;
            ld = 0;
            inside = 0;
            Q.tail = 0;
        }
        __syncthreads();
        auto below = [&](int j) {
            const int4 e = rec[j];
            return make_int2(e.z, e.w);
        };
        if (tid == 0) {
            lr[x >> 5] = 1u << (x & 31);
            sn_push(Q, ql, x, below(x));
        }
        const int nl = sn_search(S, Q, ql, 0, below, [&](int k) {  // R(x): joins
            const uint32_t a = jarc[k];
            const int j = (int)(a & ~ARC_LEAF);
            const uint32_t bit = 1u << (j & 31);
            const int2 e = a & ARC_LEAF ? make_int2(0, 0) : below(j);
            if (!(atomicOr(&lr[j >> 5], bit) & bit)) sn_push(Q, ql, j, e);
        });
        for (int q = tid; q < nl; q += T) {
            const int4 e = rec[ql[q]];
            atomicAdd(&lc, (unsigned)e.x);
            atomicAdd(&ld, (unsigned)e.y);
        }
        if (tid == 0) Q.tail = from;
        __syncthreads();
        // U(x): internal nodes that reach x
        auto mark = [&](int i) { mark_path(Q, up, lu, qi, i); };
        for (int k = inoff[x] + tid; k < inoff[x + 1]; k += T) mark(jin[k].x);
        auto above = [&](int i) { return joins_above(up[i]); };
        const int to = sn_search(S, Q, qi, from, above, [&](int k) { mark(jin[k].x); });
        if (tid == 0) {
            if (l) {
                v.lmt[(size_t)r * SN_LMK + l] = make_int2((int)lc, (int)ld);
            } else {
                info->lmk_cnt = (int)lc;
                info->lmk_deg = (int)ld;
            }
            S.aux[l] = to;
        }
        ++marks;
        if (to - from < LMK_MORE) break;
        for (int q = from + tid; q < to; q += T) {
            const int j = v.jid[io + qi[q]];
            if (j >= 0 && sn_bit(lr, j)) atomicAdd(&inside, 1);
        }
        from = to;
        __syncthreads();
        if (inside < LMK_MORE) break;
    }
    if (tid == 0) info->marks = marks;
    if (marks > 1) {
        __syncthreads();
        for (int l = 0; l < marks; ++l)
            for (int q = (l ? S.aux[l - 1] : 0) + tid; q < S.aux[l]; q += T) v.pend[io + qi[q]] = l;
    }
}

// ------------------------------------------------------------- the walks

// One thread's closure walk, for the many ranges that reach only a few
// joins (on R-MAT 20 three in four): the visited joins are a short list,
// looked through only when a 64-bit filter says that one may be there.
// skip: joins left out (NULL: none).  Returns false, with the totals
// meaningless, when the walk is too large; n: visited joins.
template <bool EDGES>
__device__ __forceinline__ bool small_walk(uint32_t *list, int stride, const uint32_t *jarc, const int4 *rec,
                                           const uint32_t *skip, int pos, int wd, unsigned int &cnt, unsigned int &deg,
                                           int &n)
{
    n = 0;
    int h = 0, p = pos, e = pos + wd, scanned = 0;
    unsigned long long seen = 0;
    if (wd > SW_ARCS) return false;
    while (true) {
        if (p < e) {
            uint32_t a[SW_U];  // several loads in flight
            bool in[SW_U];
#pragma unroll
            for (int u = 0; u < SW_U; ++u) {
                in[u] = p + u < e;
                a[u] = in[u] ? jarc[p + u] : 0u;
            }
#pragma unroll
            for (int u = 0; u < SW_U; ++u) {
                const int j = (int)(a[u] & ~ARC_LEAF);
                if (skip && in[u]) in[u] = !sn_bit(skip, j);
            }
            p += SW_U;
#pragma unroll
            for (int u = 0; u < SW_U; ++u) {
                if (!in[u]) continue;
                const int j = (int)(a[u] & ~ARC_LEAF);
                const unsigned long long f = 1ull << (((uint32_t)j * 2654435761u) >> 26);
                if (seen & f) {
                    bool found = false;
                    for (int k = 0; k < n; ++k) found |= list[k * stride] == a[u];
                    if (found) continue;
                }
                if (n == SW_CAP) return false;
                seen |= f;
                list[n * stride] = a[u];
                ++n;
                if (a[u] & ARC_LEAF) {
                    cnt += 1u;
                    if (EDGES) deg += (unsigned)rec[j].y;
                }
            }
        } else {
            while (h < n && (list[h * stride] & ARC_LEAF)) ++h;
            if (h == n) return true;
            const int j = (int)list[h * stride];
            ++h;
            const int4 r = rec[j];
            cnt += (unsigned)r.x;
            if (EDGES) deg += (unsigned)r.y;
            scanned += r.w;
            if (scanned > SW_ARCS) return false;
            p = r.z;
            e = p + r.w;
        }
    }
}

// What snapshot r's landmark l reaches, and its totals (count, out-degrees).
__device__ __forceinline__ uint32_t *snap_reach(const SnapView &v, int r, int l)
{
    return l ? v.lmi + ((size_t)r * SN_LMK + l) * v.jw : v.lmr + (size_t)r * v.jw;
}
__device__ __forceinline__ int2 snap_total(const SnapView &v, int r, int l)
{
    return l ? v.lmt[(size_t)r * SN_LMK + l] : make_int2(v.info[r].lmk_cnt, v.info[r].lmk_deg);
}

// Internal node i's landmark in the initial gains: the bits of what it reaches
// (NULL: none) and its totals.  lu: nodes that have one, pend: which, with
// several (one more dependent load for every walk otherwise).
__device__ __forceinline__ const uint32_t *snap_landmark(const SnapView &v, int r, int i, const uint32_t *lu, size_t io,
                                                         bool several, unsigned int &cnt, unsigned int &deg)
{
    cnt = 0;
    deg = 0;
    if (!sn_bit(lu, i)) return nullptr;
    const int l = several ? v.pend[io + i] : 0;
    const int2 t = snap_total(v, r, l);
    cnt = (unsigned)t.x;
    deg = (unsigned)t.y;
    return snap_reach(v, r, l);
}

// The initial gains' ranges by one thread each; those that are too large go
// to the task lists of the warp walks (in place of all tasks).  R-MAT 20, R =
// 256: 4.2 ms here and 13.5 ms of warp walks; all ranges by warps took 20 and 7
// ms with them.
template <bool EDGES>
__global__ void __launch_bounds__(256) snap_small_kernel(SnapView v)
{
    __shared__ uint32_t list[SW_CAP][256];
    __shared__ int sh[33];
    __shared__ int last;
    chain_start();
    const int tid = threadIdx.x;
    const int per = gridDim.x / v.R > 0 ? gridDim.x / v.R : 1;  // blocks per snapshot
    for (int b = blockIdx.x; b < per * v.R; b += gridDim.x) {
        const int r = b / per, part = b - r * per;
        SnapInfo *info = v.info + r;
        const int nI = info->nI;
        const size_t io = (size_t)r * v.icap, jo = (size_t)r * v.jcap;
        const uint32_t *lu = v.marki + (size_t)r * v.iw;
        const bool several = info->marks > 1;
        for (int i = part * 256 + tid; i < nI; i += per * 256) {
            const int wd = sn_hi(v.acc[io + i]);
            if (wd < 2 || v.share[io + i] >= 0) continue;
            const unsigned long long pj = v.pj[io + i];
            unsigned int c = 0, d = 0;
            const uint32_t *l = snap_landmark(v, r, i, lu, io, several, c, d);
            int n;
            if (small_walk<EDGES>(&list[0][tid], 256, v.jarc + (size_t)r * v.cap, v.rec + jo, l, (int)sn_lo(pj), wd, c,
                                  d, n)) {
                const int rj = v.jid[io + ~sn_hi(pj)];
                bool cyc = rj >= 0 && l && sn_bit(l, rj);
                for (int k = 0; k < n; ++k) cyc |= (int)(list[k][tid] & ~ARC_LEAF) == rj;
                v.cv[io + i] = sn_pack((int)(c | (cyc ? CV_CYCLE : 0u)), d);
            } else if (l) {
                v.task[io + v.icap - 1 - atomicAdd(&info->t1, 1)] = i;
            } else {
                v.task[io + atomicAdd(&info->t0, 1)] = i;
            }
        }
    }
    __syncthreads();
    if (tid == 0) {
        __threadfence();
        last = atomicAdd(v.arrive, 1) == (int)gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    sn_plan(v, sh, 1, WK_CH, [&](int q, int seg) { return sn_vol(seg ? &v.info[q].t1 : &v.info[q].t0); },
            [&](int q) { return sn_vol(&v.info[q].C); });
    if (tid == 0) *v.arrive = 0;
}

// One warp's closure walk over join ids.  A join found for the first time
// adds its totals and, with join arcs of its own, is queued.  Each lane
// keeps WK_U arcs in flight: the walk is a chain of dependent loads from
// L2 (arc, record), so loads in flight set its rate.  The queue's first
// entries lie in shared memory; entries past its end are dropped and the
// walk then re-expands every join it visited (which changes nothing for
// those already expanded) until no entry was dropped.
template <bool SH>
struct Walk {
    int off;             // the warp's shared memory: queue, undo list, bits (SH)
    uint32_t *gvis;      // bits in global memory (not SH)
    int32_t *qg;         // global queue
    const uint32_t *jarc;
    const int4 *rec;
    int count;           // joins
    int qt, nt, na;      // queued, visited, arcs scanned
    bool lost;
    unsigned int cnt, deg;

    // addressed from the shared array itself, so that the accesses compile to
    // shared-memory instructions
    __device__ __forceinline__ int32_t *qs() const
    {
        extern __shared__ __align__(16) unsigned char smem_raw[];
        return reinterpret_cast<int32_t *>(smem_raw + off);
    }
    __device__ __forceinline__ int32_t *ts() const { return qs() + WK_QS; }
    __device__ __forceinline__ uint32_t *vis() const
    {
        return SH ? reinterpret_cast<uint32_t *>(qs() + WK_QS + WK_TS) : gvis;
    }
    // arcs a[u] of this lane, valid where act[u]
    template <bool EDGES, int U>
    __device__ __forceinline__ void arcs(const uint32_t (&a)[U], const bool (&act)[U], int lane)
    {
        int id[U];
        bool fresh[U], push[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            id[u] = (int)(a[u] & ~ARC_LEAF);
            fresh[u] = act[u];
            if (fresh[u]) {
                const uint32_t bit = 1u << (id[u] & 31);
                fresh[u] = !(atomicOr(&vis()[id[u] >> 5], bit) & bit);
            }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            push[u] = false;
            if (!fresh[u]) continue;
            if (!EDGES && (a[u] & ARC_LEAF)) {
                cnt += 1u;
            } else {
                const int4 e = rec[id[u]];
                cnt += (unsigned)e.x;
                if (EDGES) deg += (unsigned)e.y;
                push[u] = e.w > 0;
            }
        }
        const unsigned lt = (1u << lane) - 1u;
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const unsigned bf = __ballot_sync(SN_FULL, fresh[u]);
            if (!bf) continue;
            if (fresh[u]) {
                const int p = nt + __popc(bf & lt);
                if (p < WK_TS) ts()[p] = id[u];
            }
            nt += __popc(bf);
            const unsigned bp = __ballot_sync(SN_FULL, push[u]);
            if (push[u]) {
                const int p = qt + __popc(bp & lt);
                if (p < WK_QS) qs()[p] = id[u];
                else if (p < WK_QS + WK_QG) qg[p - WK_QS] = id[u];
            }
            qt += __popc(bp);
        }
        if (qt > WK_QS + WK_QG) {
            qt = WK_QS + WK_QG;
            lost = true;
        }
    }

    // arcs a0 + 32u + lane of the batch of ranges the lanes hold (none is
    // empty; ex: a range's offset in the batch): arc t belongs to the last
    // range starting at or before t; the starts within 32 arcs are a bit
    // mask, so that is a population count.  rows: ranges starting before a0.
    template <bool EDGES, int U>
    __device__ __forceinline__ void spread(int a0, int total, int base, int ex, bool has, int &rows, int lane)
    {
        uint32_t a[U];
        bool act[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int t = a0 + 32 * u + lane, at = ex - a0 - 32 * u;
            const unsigned starts = __reduce_or_sync(SN_FULL, has && (unsigned)at < 32u ? 1u << at : 0u);
            const int k = rows + __popc(starts & (SN_FULL >> (31 - lane))) - 1;
            rows += __popc(starts);
            const int b = __shfl_sync(SN_FULL, base, k);
            act[u] = t < total;
            a[u] = act[u] ? jarc[b + t] : 0u;
        }
        arcs<EDGES, U>(a, act, lane);
    }

    template <bool EDGES, int U>
    __device__ __forceinline__ void straight(int pos, int left, int lane)
    {
        uint32_t a[U];
        bool act[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            act[u] = 32 * u + lane < left;
            a[u] = act[u] ? jarc[pos + 32 * u + lane] : 0u;
        }
        arcs<EDGES, U>(a, act, lane);
    }

    template <bool EDGES>
    __device__ __forceinline__ void queue(int lane)
    {
        int qh = 0;
        __syncwarp();
        while (qh < qt) {
            const int nb = min(32, qt - qh);
            int pos = 0, wd = 0;
            if (lane < nb) {
                const int p = qh + lane;
                const int4 e = rec[p < WK_QS ? qs()[p] : qg[p - WK_QS]];
                pos = e.z;
                wd = e.w;
            }
            qh += nb;
            const int inc = sn_warp_incl(wd, lane);
            const int total = __shfl_sync(SN_FULL, inc, 31), ex = inc - wd;
            na += total;
            if (qh == qt && qt > WK_QS) {  // drained: start over at the front
                __syncwarp();
                qh = 0;
                qt = 0;
            }
            int rows = 0;
            for (int a0 = 0; a0 < total;) {
                if (total - a0 > 32) {
                    spread<EDGES, WK_U>(a0, total, pos - ex, ex, lane < nb, rows, lane);
                    a0 += 32 * WK_U;
                } else {
                    spread<EDGES, 1>(a0, total, pos - ex, ex, lane < nb, rows, lane);
                    a0 += 32;
                }
            }
            __syncwarp();
        }
        qt = 0;
    }

    // Closure of the join-arc range [pos, pos + wd); base: bits set in vis
    // before the walk (NULL: none).
    template <bool EDGES>
    __device__ __forceinline__ void range(int pos, int wd, const uint32_t *base, int lane)
    {
        qt = 0;
        nt = 0;
        na = wd;
        lost = false;
        cnt = 0;
        deg = 0;
        for (int a0 = 0; a0 < wd;) {
            if (wd - a0 > 32) {
                straight<EDGES, WK_U>(pos + a0, wd - a0, lane);
                a0 += 32 * WK_U;
            } else {
                straight<EDGES, 1>(pos + a0, wd - a0, lane);
                a0 += 32;
            }
        }
        queue<EDGES>(lane);
        while (lost) {
            lost = false;
            const int words = (count + 31) >> 5;
            for (int i = 0; i < words; ++i) {
                const uint32_t b = *(volatile uint32_t *)&vis()[i] & ~(base ? base[i] : 0u);
                const int j = i * 32 + lane;
                const bool act = ((b >> lane) & 1u) && j < count && rec[j].w > 0;
                const unsigned bp = __ballot_sync(SN_FULL, act);
                if (!bp) continue;
                if (act) qs()[__popc(bp & ((1u << lane) - 1u))] = j;  // at most 32 <= WK_QS
                qt = __popc(bp);
                queue<EDGES>(lane);
            }
        }
    }

    // vis back to the base
    __device__ __forceinline__ void undo(const uint32_t *base, int lane)
    {
        __syncwarp();
        if (nt <= WK_TS) {
            for (int t = lane; t < nt; t += 32) atomicAnd(&vis()[ts()[t] >> 5], ~(1u << (ts()[t] & 31)));
            __syncwarp();
        } else {
            load(base, lane);
        }
    }

    __device__ __forceinline__ void load(const uint32_t *base, int lane)
    {
        const int words = (count + 31) >> 5;
        // vis areas and bases are 16-byte aligned and padded to 16 bytes
        int4 *d = reinterpret_cast<int4 *>(vis());
        const int4 *b = reinterpret_cast<const int4 *>(base);
#pragma unroll 4
        for (int i = lane; i < (words + 3) >> 2; i += 32) d[i] = base ? b[i] : make_int4(0, 0, 0, 0);
        __syncwarp();
    }
};

// Internal node i and the tree ancestors that share its range lose c;
// returns the reverse edges.
template <bool EDGES>
__device__ __forceinline__ unsigned long long snap_lose(const SnapView &v, long long *s, size_t io, int i,
                                                        unsigned int c)
{
    unsigned long long edges = 0;
    for (int u = i;;) {
        const int x = v.inode[io + u];
        v.cnt[io + u] -= c;
        atomicAdd((unsigned long long *)&s[x], (unsigned long long)(-(long long)c));
        if (EDGES) edges += (unsigned long long)c * (unsigned long long)(__ldg(v.crp + x + 1) - __ldg(v.crp + x));
        const int p = v.par[io + u];
        if (p < 0 || v.share[io + p] != u) return edges;
        u = p;
    }
}

// Largest q in [0, count) with start[q] <= t (non-decreasing, start[0] = 0);
// the whole warp searches, 32 ways a step.
__device__ __forceinline__ int find_chunk(const int32_t *start, int count, int t)
{
    const int lane = threadIdx.x & 31;
    int lo = 0, n = count;
    while (n > 1) {
        const int step = (n + 31) / 32, at = lo + lane * step;
        const unsigned le = __ballot_sync(SN_FULL, at < lo + n && start[at] <= t);
        const int k = 31 - __clz((int)le);
        const int end = lo + n;
        lo += k * step;
        n = min(step, end - lo);
    }
    return lo;
}

// MODE 0: initial gains, the distinct ranges (result kept in cv).
// MODE 1: initial gains, sources whose count needs their own walk.
// MODE 2: a round's marked ranges: the newly covered nodes each reaches,
//         subtracted from it and from the tree ancestors that share its range.
// EDGES: also the out-degree sums / reverse edges.
// Warps claim chunks of tasks in snapshot order, so the graphs of the few
// snapshots in flight stay in L2.  (Chunks claimed per block, with a barrier
// after each, left warps waiting for the block's longest walk 40 % of the
// time.)  Each warp keeps its bits in shared memory (in global memory, one
// warp per block, when they are more than that holds) and undoes a small
// walk's bits one by one instead of clearing all.  R-MAT 20, R = 256: 13.5 ms
// (MODE 0, 0.8 G join arcs), 18 ms (MODE 2, all rounds, 6 of them the first).
template <int MODE, bool EDGES, bool SH>
__device__ __forceinline__ void walk_tasks(const SnapView &v, Ctl *ctl, long long *s, int area)
{
    constexpr bool ROUND = MODE == 2;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int total = v.cstart[2 * v.R], per = v.cstart[2 * v.R + 2];
    const bool all = ROUND && v.cstart[2 * v.R + 3];  // no one-thread walks ran before
    Walk<SH> w;
    w.off = SH ? wid * area : 0;
    w.gvis = v.gbm + (size_t)blockIdx.x * v.jw;
    w.qg = v.wq + ((size_t)blockIdx.x * WK_W + wid) * WK_QG;
    int q = -1, qbeg = 0, qend = 0;  // (snapshot, segment) at hand: its base is in vis
    int cnt = 0, lcnt = 0, ldeg = 0, mark = -1;
    size_t io = 0;
    const uint32_t *base = nullptr;
    const int32_t *list = nullptr;
    unsigned long long edges = 0, arcs = 0, joins = 0;
    while (true) {
        int ch = 0;
        if (lane == 0) ch = atomicAdd(v.cnext, 1);
        ch = __shfl_sync(SN_FULL, ch, 0);
        if (ch >= total) break;
        if (ch >= qend) {
            q = find_chunk(v.cstart, 2 * v.R, ch);
            qbeg = v.cstart[q];
            qend = v.cstart[q + 1];
            const int r = q >> 1, seg = q & 1;
            const SnapInfo *in = v.info + r;
            cnt = MODE == 0 || all ? (seg ? in->t1 : in->t0) : (seg ? in->f1 : in->f0);
            lcnt = seg && ROUND ? in->lmk_cnt : 0;
            ldeg = 0;
            mark = -1;
            io = (size_t)r * v.icap;
            w.count = ROUND ? in->nrel : in->C;
            w.jarc = (ROUND ? v.rarc : v.jarc) + (size_t)r * v.cap;
            w.rec = (ROUND ? v.rrec : v.rec) + (size_t)r * v.jcap;
            base = seg && ROUND ? v.lmc + (size_t)r * v.jw : nullptr;
            list = (MODE == 0 || all ? v.task : (MODE == 1 ? v.fb : v.ilist)) + io;
            if (ROUND || !seg) w.load(base, lane);
        }
        const int k0 = (ch - qbeg) * per, nk = min(cnt - k0, per);
        int ti = 0, tp = 0, tw = 0, tr = 0, tl = 0;  // the chunk's tasks, one per lane
        if (lane < nk) {
            ti = list[(q & 1) ? v.icap - 1 - (k0 + lane) : k0 + lane];
            if (ROUND) {
                const int2 a = v.rrange[io + ti];
                tp = a.x;
                tw = a.y;
            } else {
                const unsigned long long pj = v.pj[io + ti];
                tp = (int)sn_lo(pj);
                tw = sn_hi(v.acc[io + ti]);
                tr = v.jid[io + ~sn_hi(pj)];
                if ((q & 1) && v.info[q >> 1].marks > 1) tl = v.pend[io + ti];
            }
        }
        for (int k = 0; k < nk; ++k) {
            if (!ROUND && (q & 1)) {
                const int l = __shfl_sync(SN_FULL, tl, k);
                if (l != mark) {  // another landmark than the last task's
                    mark = l;
                    const int2 t = snap_total(v, q >> 1, l);
                    lcnt = t.x;
                    ldeg = t.y;
                    base = snap_reach(v, q >> 1, l);
                    w.load(base, lane);
                }
            }
            const int i = __shfl_sync(SN_FULL, ti, k), rj = __shfl_sync(SN_FULL, tr, k);
            w.template range<EDGES && !ROUND>(__shfl_sync(SN_FULL, tp, k), __shfl_sync(SN_FULL, tw, k), base, lane);
            unsigned int c = w.cnt, d = w.deg;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                c += __shfl_xor_sync(SN_FULL, c, o);
                if (EDGES) d += __shfl_xor_sync(SN_FULL, d, o);
            }
            if (lane == 0) {
                c += (unsigned)lcnt;
                d += (unsigned)ldeg;
                if (MODE != 2) {
                    const bool cyc = rj >= 0 && (*(volatile uint32_t *)&w.vis()[rj >> 5] >> (rj & 31) & 1u);
                    if (MODE == 0) {
                        v.cv[io + i] = sn_pack((int)(c | (cyc ? CV_CYCLE : 0u)), d);
                    } else {
                        if (!cyc) {
                            c += sn_lo(v.acc[io + i]);
                            d += v.deg[io + i];
                        }
                        v.cnt[io + i] = c;
                        atomicAdd((unsigned long long *)&s[v.inode[io + i]], (unsigned long long)c);
                        edges += d;
                    }
                } else {
                    edges += snap_lose<EDGES>(v, s, io, i, c);
                }
            }
            arcs += (unsigned long long)w.na;
            joins += (unsigned long long)w.nt;
            w.undo(base, lane);
        }
    }
    if (EDGES && lane == 0 && edges) atomicAdd(MODE == 2 ? &ctl->rev_edges : &ctl->init_edges, edges);
    if (lane == 0 && arcs) {
        atomicAdd(&ctl->work_elems[MODE == 2 ? 1 : 0][MODE == 0 ? 0 : 2], arcs);
        atomicAdd(&ctl->work_keys[MODE == 2 ? 1 : 0][MODE == 0 ? 0 : 2], joins);
    }
}

template <int MODE, bool EDGES>
__global__ void __launch_bounds__(WK_T, 2) snap_walk_kernel(SnapView v, Ctl *ctl, long long *s, int smem_bytes)
{
    chain_start();
    const int wid = threadIdx.x >> 5;
    const int area = ((((v.cstart[2 * v.R + 1] + 31) >> 5) * 4 + 15) & ~15) + (WK_QS + WK_TS) * 4;
    const int nact = smem_bytes / area;
    if (wid < nact) walk_tasks<MODE, EDGES, true>(v, ctl, s, area);
    else if (nact == 0 && wid == 0) walk_tasks<MODE, EDGES, false>(v, ctl, s, area);
}

// Counts of all internal nodes from the walked ranges.  A node's closure is
// that of the lowest tree node with the same range; a range of one join arc
// is followed to the join's own closure.  Where that closure runs through a
// cycle (so that it might hold the node's own tree) the node gets a walk of
// its own, by this thread or, when too large, by a warp (list fb, planned
// for MODE 1 by the last block).  Bound by loads in flight: five blocks an SM
// (four, 57 registers: LT on 60k nodes 146 -> 198 us).
template <bool EDGES>
__global__ void __launch_bounds__(256, EDGES ? 4 : 5) snap_resolve_kernel(SnapView v, Ctl *ctl, long long *s)
{
    __shared__ uint32_t list[SW_CAP][256];
    __shared__ int sh[33];
    __shared__ int last;
    chain_start();
    const int tid = threadIdx.x, lane = tid & 31;
    unsigned long long edges = 0;
    const int per = gridDim.x / v.R > 0 ? gridDim.x / v.R : 1;  // blocks per snapshot
    for (int b = blockIdx.x; b < per * v.R; b += gridDim.x) {
        const int r = b / per, part = b - r * per;
        SnapInfo *info = v.info + r;
        const int nI = info->nI;
        const size_t io = (size_t)r * v.icap, jo = (size_t)r * v.jcap;
        const uint32_t *jarc = v.jarc + (size_t)r * v.cap;
        const uint32_t *lu = v.marki + (size_t)r * v.iw;
        const uint32_t *outb = v.outb + (size_t)r * v.n32;
        const int32_t *outp = v.outp + (size_t)r * v.n32;
        for (int i = part * 256 + tid; i < nI; i += per * 256) {
            const unsigned long long a = v.acc[io + i];
            unsigned int c = sn_lo(a), d = v.deg[io + i];
            bool walk = false;
            if (sn_hi(a) > 0) {
                int o = i;
                while (v.share[io + o] >= 0) o = v.share[io + o];
                int wd = sn_hi(a), pos = (int)sn_lo(v.pj[io + o]), before = -1;
                for (int step = 0;; ++step) {
                    if (wd >= 2) {
                        const unsigned long long cv = v.cv[io + o];
                        if ((uint32_t)sn_hi(cv) & CV_CYCLE) {
                            if (step > 0) {
                                walk = true;
                                break;
                            }
                            c = 0;  // its own tree is among the joins found
                            d = 0;
                        }
                        c += (uint32_t)sn_hi(cv) & ~CV_CYCLE;
                        d += sn_lo(cv);
                        break;
                    }
                    const int j = (int)(jarc[pos] & ~ARC_LEAF);
                    const int4 e = v.rec[jo + j];
                    c += (unsigned)e.x;
                    d += (unsigned)e.y;
                    if (e.w == 0) break;
                    if (step >= 32 || j == before) {  // a cycle of one-arc joins, or perhaps one
                        walk = true;
                        break;
                    }
                    before = j;
                    o = sn_rank(outb, outp, v.jnode[jo + j]);
                    while (v.share[io + o] >= 0) o = v.share[io + o];
                    wd = e.w;
                    pos = e.z;
                }
            }
            if (walk) {
                const unsigned long long pj = v.pj[io + i];
                const uint32_t *l = snap_landmark(v, r, i, lu, io, info->marks > 1, c, d);
                int n;
                if (small_walk<EDGES>(&list[0][tid], 256, jarc, v.rec + jo, l, (int)sn_lo(pj), sn_hi(a), c, d, n)) {
                    const int rj = v.jid[io + ~sn_hi(pj)];
                    bool cyc = rj >= 0 && l && sn_bit(l, rj);
                    for (int k = 0; k < n; ++k) cyc |= (int)(list[k][tid] & ~ARC_LEAF) == rj;
                    if (!cyc) {
                        c += sn_lo(a);
                        d += v.deg[io + i];
                    }
                    walk = false;
                }
            }
            if (walk) {
                if (sn_bit(lu, i)) v.fb[io + v.icap - 1 - atomicAdd(&info->f1, 1)] = i;
                else v.fb[io + atomicAdd(&info->f0, 1)] = i;
            } else {
                v.cnt[io + i] = c;
                atomicAdd((unsigned long long *)&s[v.inode[io + i]], (unsigned long long)c);
                edges += d;
            }
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) edges += __shfl_xor_sync(SN_FULL, edges, o);
    if (lane == 0 && edges) atomicAdd(&ctl->init_edges, edges);
    __syncthreads();
    if (tid == 0) {
        __threadfence();
        last = atomicAdd(v.arrive, 1) == (int)gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    sn_plan(v, sh, 1, WK_CH, [&](int q, int seg) { return sn_vol(seg ? &v.info[q].f1 : &v.info[q].f0); },
            [&](int q) { return sn_vol(&v.info[q].C); });
    if (tid == 0) *v.arrive = 0;
}

// ------------------------------------------------------------- a round

// One block per snapshot.  Bound by the slowest block's chain of levels: each is
// two or three dependent accesses and two or four barriers, with few entries
// (R-MAT 18: 27 warp cycles an instruction at barriers, 13 on loads, L2 at 6 %).
// R-MAT 20, R = 256: 2.6 ms in the first round, 0.57 ms on average, 28 ms of a
// selection's 92; 15k nodes, R = 100, UIC: 20 us.  1024 threads a block, or 256
// where snapshots have few live arcs; 512 in place of 1024 cost 11 %.
// Cover R(v*) in one snapshot, subtract from the ancestors of v*, and list
// the ranges whose counts need a walk (Algorithm 2, inner loops), with the
// joins such a walk may enter: the newly covered ones and the marked ones
// above them.  With many newly covered joins one of them serves as the
// round's landmark, as in the initial gains.
// DU false: cover only (no gain is kept current).  direct: every task goes
// to the warp walks (the caller launches no one-thread walks).
template <bool EDGES, bool DU>
__global__ void __launch_bounds__(SN_T)
    snap_cover_kernel(SnapView v, Ctl *ctl, long long *s, unsigned long long *cov, int direct)
{
    __shared__ ExpandShared S;
    __shared__ QueueShared Q;
    __shared__ int nnew, tnew, nt0, nt1, last, pleaf, around;
    __shared__ unsigned int lw;
    __shared__ unsigned long long best;
    chain_start();
    const int r = blockIdx.x, tid = threadIdx.x, lane = tid & 31, T = blockDim.x;
    SnapInfo *info = v.info + r;
    const int x = sn_vol(&ctl->vstar);
    const int C = info->C;
    const size_t io = (size_t)r * v.icap, jo = (size_t)r * v.jcap;
    const uint32_t *outb = v.outb + (size_t)r * v.n32, *joinb = v.joinb + (size_t)r * v.n32;
    const int32_t *outp = v.outp + (size_t)r * v.n32, *joinp = v.joinp + (size_t)r * v.n32;
    const uint32_t *lb = v.lb + (size_t)r * v.m32;
    unsigned long long *covw = cov + (size_t)(r >> 6) * (size_t)v.n;
    const unsigned long long cbit = 1ull << (r & 63);
    const uint32_t *jarc = v.jarc + (size_t)r * v.cap;
    const int2 *jin = v.jin + (size_t)r * v.cap;
    const int32_t *inoff = v.inoff + (size_t)r * (v.jcap + 1);
    const int2 *tn = v.tn + (size_t)r * v.tcap, *up = v.up + io;
    const int32_t *par = v.par + io, *jid = v.jid + io;
    const int4 *rec = v.rec + jo;
    uint32_t *covj = v.covj + (size_t)r * v.jw, *rel = v.rel + (size_t)r * v.jw, *lmr = v.lmr + (size_t)r * v.jw;
    uint2 *rel2 = v.rel2 + (size_t)r * v.jw;
    // mk: covered or marked in this round; covi: covered
    uint32_t *covi = v.covi + (size_t)r * v.iw, *mk = v.marki + (size_t)r * v.iw;
    int32_t *ql = v.jlist + jo, *qi = v.ilist + io, *qr = v.fb + io;  // fb is free after the initial gains
    uint32_t *abit = v.abit + (size_t)r * v.aw;  // arcs to relevant joins, by position in jarc
    uint2 *abit2 = v.abit2 + (size_t)r * v.aw;
    const int cw = (C + 31) >> 5, aw = (info->JA + 31) >> 5;
    unsigned long long fwd = 0, rev = 0;
    const bool run = x >= 0 && !info->bad && !(covw[x] & cbit);
    int nrel = 0;
    if (tid == 0) {
        Q.tail = 0;
        nnew = 0;
        tnew = 0;
        nt0 = 0;
        nt1 = 0;
        pleaf = -1;
        around = 0;
        lw = 0;
        best = 0;
    }
    if (run) {
        const bool internal = sn_bit(outb, x), isj = sn_bit(joinb, x);
        const int xi = internal ? sn_rank(outb, outp, x) : -1;
        const int xj = isj ? sn_rank(joinb, joinp, x) : -1;
        for (int i = tid; i < cw; i += T) rel[i] = 0;
        for (int i = tid; i < aw; i += T) abit[i] = 0;
        __syncthreads();
        // newly covered joins: closure from v* over uncovered joins
        auto below = [&](int j) {
            const int4 e = rec[j];
            return make_int2(e.z, e.w);
        };
        auto cover = [&](uint32_t a) {
            const int j = (int)(a & ~ARC_LEAF);
            const uint32_t bit = 1u << (j & 31);
            const int2 e = a & ARC_LEAF ? make_int2(0, 0) : below(j);
            if (!(atomicOr(&covj[j >> 5], bit) & bit)) {
                atomicOr(&rel[j >> 5], bit);
                sn_push(Q, ql, j, e);
            }
        };
        if (isj) {
            if (tid == 0) cover((uint32_t)xj);
        } else if (internal) {
            const int p0 = (int)sn_lo(v.pj[io + xi]), wd = sn_hi(v.acc[io + xi]);
            for (int k = tid; k < wd; k += T) cover(jarc[p0 + k]);
        }
        const int nd = sn_search(S, Q, ql, 0, below, [&](int k) { cover(jarc[k]); });
        // Ancestors of v*: uncovered internal nodes above it, through newly
        // covered nodes too (v* may lie in a component with them).  A leaf
        // keeps no parent: its live in-arc is looked up among its canonical
        // ones.
        auto mark = [&](int i) { mark_path(Q, up, mk, qi, i); };
        auto mark_up = [&](int k) { mark(jin[k].x); };
        auto mark_arc = [&](int k) {
            const int2 a = jin[k];
            atomicOr(&abit[a.y >> 5], 1u << (a.y & 31));
            mark(a.x);
        };
        auto above = [&](int i) { return joins_above(up[i]); };
        if (tid == 0) Q.tail = 0;
        __syncthreads();
        if (isj) {
            if (DU)
                for (int k = inoff[xj] + tid; k < inoff[xj + 1]; k += T) mark(jin[k].x);
        } else if (internal) {
            if (tid == 0 && par[xi] >= 0) {
                pleaf = par[xi];
                if (DU) mark(par[xi]);
            }
        } else {
            for (int k = __ldg(v.crp + x) + tid; k < __ldg(v.crp + x + 1); k += T) {
                const int2 a = __ldg(v.cin + k);
                if ((lb[(uint32_t)a.y >> 5] >> (a.y & 31)) & 1u) {
                    const int i = sn_rank(outb, outp, a.x);
                    pleaf = i;
                    if (DU) mark(i);
                }
            }
        }
        const int na = DU ? sn_search(S, Q, qi, 0, above, mark_up) : 0;
        // The round's landmark: the newly covered join with the most arcs
        // below times in-arcs from uncovered non-ancestors, two steps up.  Where
        // it lies on a cycle, the nodes above it are looked for before any is
        // marked as covered, since the way up leads through newly covered ones:
        // v* may lie above a large component that others reach at joins of their
        // own (R-MAT 18, p = 0.2, R = 64: a million walks of 36,000 joins each in
        // round one otherwise).  Elsewhere the few more nodes found so are not
        // worth the longer way (R-MAT 20, WIC: 2 % of a selection).
        int nu = na, nl = 0, lj = -1;
        auto climb = [&]() {
            if (tid == 0) Q.tail = na;
            __syncthreads();
            for (int k = inoff[lj] + tid; k < inoff[lj + 1]; k += T) mark(jin[k].x);
            nu = sn_search(S, Q, qi, na, above, mark_arc);
        };
        if (DU && nd >= ROUND_LMK) {
            for (int i = tid; i < cw; i += T) lmr[i] = 0;
            for (int q = tid; q < nd; q += T) qr[q] = 0;
            __syncthreads();
            sn_expand_n(
                S, 0, nd,
                [&](int q, int &first, int &len) {
                    const int j = ql[q];
                    if (rec[j].w < 2) return;
                    first = inoff[j];
                    len = inoff[j + 1] - first;
                },
                [&](const auto &q, const auto &k) {
                    constexpr int U = sizeof(q) / sizeof(int);
                    int i[U], rj[U];
#pragma unroll
                    for (int u = 0; u < U; ++u) i[u] = q[u] >= 0 ? jin[k[u]].x : -1;
#pragma unroll
                    for (int u = 0; u < U; ++u)
                        if (i[u] >= 0) rj[u] = sn_bit(mk, i[u]) ? -2 : ~sn_hi(v.pj[io + i[u]]);
#pragma unroll
                    for (int u = 0; u < U; ++u)
                        if (i[u] >= 0 && rj[u] != -2) rj[u] = jid[rj[u]];
#pragma unroll
                    for (int u = 0; u < U; ++u) {
                        if (i[u] < 0 || rj[u] == -2 || (rj[u] >= 0 && sn_bit(rel, rj[u]))) continue;
                        atomicAdd(&qr[q[u]], 1 + (rj[u] >= 0 ? inoff[rj[u] + 1] - inoff[rj[u]] : 0));
                    }
                });
            for (int q = tid; q < nd; q += T) {
                const unsigned long long a = (unsigned long long)(uint32_t)qr[q];
                if (a)
                    atomicMax(&best, (min(a * (unsigned long long)rec[ql[q]].w, (1ull << 31) - 1ull) << 32) |
                                         (uint32_t)ql[q]);
            }
            __syncthreads();
            lj = best ? (int)(uint32_t)best : -1;
            if (lj >= 0) {
                if (tid == 0) {
                    Q.tail = 0;
                    lmr[lj >> 5] = 1u << (lj & 31);
                    sn_push(Q, qr, lj, below(lj));
                }
                nl = sn_search(S, Q, qr, 0, below, [&](int k) {
                    const uint32_t a = jarc[k];
                    const int j = (int)(a & ~ARC_LEAF);
                    const uint32_t bit = 1u << (j & 31);
                    const int2 e = a & ARC_LEAF ? make_int2(0, 0) : below(j);
                    if (!(rel[j >> 5] & bit)) return;  // covered before
                    if (j == lj) around = 1;
                    if (!(atomicOr(&lmr[j >> 5], bit) & bit)) sn_push(Q, qr, j, e);
                });
                for (int q = tid; q < nl; q += T) atomicAdd(&lw, (unsigned)rec[qr[q]].x);
                if (around) climb();
            }
        }
        // newly covered nodes: the trees of those joins and T(v*)
        // (a node stands once in a list, so its bit is looked up before it is
        // set and the loads of EX_U nodes go out together)
        auto nodes = [&](const auto &a) -> int {
            constexpr int U = sizeof(a) / sizeof(int2);
            bool fresh[U];
            unsigned int c[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                fresh[u] = a[u].x >= 0 && !(*(volatile unsigned long long *)&covw[a[u].x] & cbit);
                c[u] = DU && a[u].x >= 0 && a[u].y >= 0 ? v.cnt[io + a[u].y] : 1u;
            }
            int got = 0;
#pragma unroll
            for (int u = 0; u < U; ++u) {
                if (!fresh[u]) continue;
                const int y = a[u].x, i = a[u].y;
                ++got;
                atomicOr(&covw[y], cbit);
                if (DU && i >= 0) {
                    atomicOr(&covi[i >> 5], 1u << (i & 31));
                    atomicOr(&mk[i >> 5], 1u << (i & 31));
                    v.cnt[io + i] = 0;
                }
                if (DU) atomicAdd((unsigned long long *)&s[y], (unsigned long long)(-(long long)c[u]));
                if (EDGES) {
                    fwd += (unsigned long long)(__ldg(v.rp + y + 1) - __ldg(v.rp + y));
                    rev += (unsigned long long)c[u] * (unsigned long long)(__ldg(v.crp + y + 1) - __ldg(v.crp + y));
                }
            }
            return got;
        };
        const int2 none = make_int2(-1, -1);
        int got = 0, gott = 0;
        if (!isj) {
            const int p0 = internal ? (int)sn_lo(v.pn[io + xi]) : 0, len = internal ? (int)sn_lo(v.acc[io + xi]) : 1;
            auto own = [&](auto &a, int k) {
                constexpr int U = sizeof(a) / sizeof(int2);
#pragma unroll
                for (int u = 0; u < U; ++u)
                    a[u] = k + u * T >= len ? none : internal ? tn[p0 + k + u * T] : make_int2(x, -1);
                gott += nodes(a);
            };
            if (len <= T) {
                int2 a[1];
                if (tid < len) own(a, tid);
            } else {
                int2 a[EX_U];
                for (int k = tid; k < len; k += EX_U * T) own(a, k);
            }
        }
        sn_expand_n(
            S, 0, nd,
            [&](int q, int &first, int &len) {
                const int2 e = v.jtn[jo + ql[q]];
                first = e.x;
                len = e.y;
            },
            [&](const auto &q, const auto &k) {
                    constexpr int U = sizeof(q) / sizeof(int);
                int2 a[U];
#pragma unroll
                for (int u = 0; u < U; ++u) a[u] = q[u] >= 0 ? tn[k[u]] : none;
                got += nodes(a);
            });
        if (gott) atomicAdd(&tnew, gott);
        if (got + gott) atomicAdd(&nnew, got + gott);
        __syncthreads();
        const int N = nnew;
        for (int q = tid; q < na; q += T) {
            const int i = qi[q];
            if (sn_bit(covi, i)) continue;
            const int y = v.inode[io + i];
            v.cnt[io + i] -= (unsigned)N;
            atomicAdd((unsigned long long *)&s[y], (unsigned long long)(-(long long)N));
            if (EDGES) rev += (unsigned long long)N * (unsigned long long)(__ldg(v.crp + y + 1) - __ldg(v.crp + y));
        }
        if (tid == 0 && pleaf >= 0 && tnew) {
            // the tree v* hangs in lost T(v*)
            const int j = jid[~sn_hi(v.pj[io + pleaf])];
            if (j >= 0 && !sn_bit(covj, j)) v.rec[jo + j].x -= tnew;
        }
        int32_t *task = v.task + io;
        if (DU && lj >= 0) {
            if (!around) {
                climb();
            } else {  // covered nodes leave the list
                for (int q = na + tid; q < nu; q += T)
                    if (!sn_bit(covi, qi[q])) task[atomicAdd(&nt0, 1)] = qi[q];
                __syncthreads();
                nu = na + nt0;
                for (int q = na + tid; q < nu; q += T) qi[q] = task[q - na];
                __syncthreads();
                if (tid == 0) nt0 = 0;
            }
        }
        int ni = 0;
        if (DU) {
            if (tid == 0) Q.tail = nu;
            // the other nodes that reach a newly covered join
            sn_expand(
                S, 0, nd,
                [&](int q, int &first, int &len) {
                    const int j = ql[q];
                    first = inoff[j];
                    len = inoff[j + 1] - first;
                },
                [&](int, int k) { mark_arc(k); });
            ni = sn_search(S, Q, qi, nu, above, mark_arc);
        }
        // their ranges are tasks, the joins among them relevant too
        for (int q = na + tid; q < ni; q += T) {
            const int i = qi[q];
            const int j = jid[i];
            if (j >= 0) atomicOr(&rel[j >> 5], 1u << (j & 31));
            if (v.share[io + i] >= 0) continue;  // with the child that has its range
            if (q < nu) task[v.icap - 1 - atomicAdd(&nt1, 1)] = i;
            else task[atomicAdd(&nt0, 1)] = i;
        }
        for (int q = tid; q < ni; q += T) {
            const int i = qi[q];
            if (!sn_bit(covi, i)) atomicAnd(&mk[i >> 5], ~(1u << (i & 31)));
        }
        __syncthreads();
        if (nt0 + nt1) {
            // The round's own closure graph: relevant joins by rank, the arcs
            // to them in order; a range of join arcs is again a range.
            for (int b = 0; b < cw; b += T) {
                const int i = b + tid;
                int tot;
                const uint32_t w = i < cw ? rel[i] : 0u;
                const int ex = sn_block_excl(__popc(w), S.sh, tot);
                if (i < cw) rel2[i] = make_uint2(w, (unsigned)(nrel + ex));
                nrel += tot;
            }
            int na2 = 0;
            for (int b = 0; b < aw; b += T) {
                const int i = b + tid;
                int tot;
                const uint32_t w = i < aw ? abit[i] : 0u;
                const int ex = sn_block_excl(__popc(w), S.sh, tot);
                if (i < aw) abit2[i] = make_uint2(w, (unsigned)(na2 + ex));
                na2 += tot;
            }
            __syncthreads();
            int4 *rrec = v.rrec + jo;
            int2 *rrange = v.rrange + io;
            uint32_t *rarc = v.rarc + (size_t)r * v.cap;
            auto rank2 = [](const uint2 *b, int j) {
                const uint2 w = b[j >> 5];
                return (int)w.y + __popc(w.x & ((1u << (j & 31)) - 1u));
            };
            auto range2 = [&](int pos, int wd) {
                if (wd == 0) return make_int2(0, 0);
                const int a = rank2(abit2, pos);
                const int l = pos + wd - 1;  // the last position: its own bit counts too
                return make_int2(a, rank2(abit2, l) + (int)((abit2[l >> 5].x >> (l & 31)) & 1u) - a);
            };
            auto record = [&](int j, bool covered) {
                const int4 e = rec[j];
                const int2 a = range2(e.z, e.w);
                rrec[rank2(rel2, j)] = make_int4(covered ? e.x : 0, 0, a.x, a.y);
            };
            for (int q = na + tid; q < ni; q += T) {
                const int i = qi[q], j = jid[i];
                if (j >= 0) record(j, false);
                if (v.share[io + i] < 0) rrange[i] = range2((int)sn_lo(v.pj[io + i]), sn_hi(v.acc[io + i]));
            }
            sn_expand_n(
                S, 0, nd + ni - na,
                [&](int q, int &first, int &len) {
                    const int j = q < nd ? ql[q] : jid[qi[na + q - nd]];
                    if (j < 0) return;
                    if (q < nd) record(j, true);
                    S.aux[tid] = rank2(rel2, j);
                    first = inoff[j];
                    len = inoff[j + 1] - first;
                },
                [&](const auto &q, const auto &k) {
                    constexpr int U = sizeof(q) / sizeof(int);
                    int p[U];
                    uint32_t leaf[U];
#pragma unroll
                    for (int u = 0; u < U; ++u) p[u] = q[u] >= 0 ? jin[k[u]].y : -1;
#pragma unroll
                    for (int u = 0; u < U; ++u) {
                        if (p[u] < 0) continue;
                        leaf[u] = jarc[p[u]] & ARC_LEAF;
                        p[u] = rank2(abit2, p[u]);
                    }
#pragma unroll
                    for (int u = 0; u < U; ++u)
                        if (p[u] >= 0) rarc[p[u]] = (uint32_t)S.aux[q[u] & (T - 1)] | leaf[u];
                });
            if (nt1) {
                // the landmark's reach by rank
                uint32_t *lmc = v.lmc + (size_t)r * v.jw;
                for (int i = tid; i < v.jw && i * 32 < nrel + 128; i += T) lmc[i] = 0;
                __syncthreads();
                for (int q = tid; q < nl; q += T) {
                    const int k = rank2(rel2, qr[q]);
                    atomicOr(&lmc[k >> 5], 1u << (k & 31));
                }
            }
        }
    }
    if (EDGES) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            fwd += __shfl_xor_sync(SN_FULL, fwd, o);
            rev += __shfl_xor_sync(SN_FULL, rev, o);
        }
        if (lane == 0 && fwd) atomicAdd(&ctl->fwd_edges, fwd);
        if (lane == 0 && rev) atomicAdd(&ctl->rev_edges, rev);
    }
    __syncthreads();
    if (tid == 0) {
        info->t0 = nt0;
        info->t1 = nt1;
        info->f0 = 0;
        info->f1 = 0;
        info->nrel = nrel;
        info->lmk_cnt = (int)lw;
        if (nt0 + nt1) atomicAdd(&ctl->rev_tasks, (unsigned long long)(nt0 + nt1));
        if (nnew) atomicAdd(&ctl->du_entries, (unsigned long long)nnew);
        chain_next();
        __threadfence();
        last = atomicAdd(v.arrive, 1) == (int)gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    if (!DU) {
        if (tid == 0) *v.arrive = 0;
        return;
    }
    __threadfence();
    // few tasks: one warp each at once, without the one-thread walks
    auto tasks = [&](int q, int seg) { return sn_vol(seg ? &v.info[q].t1 : &v.info[q].t0); };
    auto ids = [&](int q) { return sn_vol(&v.info[q].nrel); };
    sn_plan(v, S.sh, 1, WK_CH, tasks, ids);
    __syncthreads();
    if (!direct && v.cstart[2 * v.R + 2] >= ROUND_ONE) {
        __syncthreads();
        sn_plan(v, S.sh, 32, 32, tasks, ids);
    } else if (tid == 0) {
        v.cstart[2 * v.R + 3] = 1;
    }
    if (tid == 0) *v.arrive = 0;
}

// Marginal gains of up to EV_MAX candidates (lazy evaluation): block (r, b)
// adds to out[b] the nodes candidate b would newly cover in snapshot r, a
// closure over uncovered joins like the cover's, with nothing written back.
// bits [EV_MAX][R][jw], queues [EV_MAX][R][jcap]: scratch.  One candidate a
// launch left the chip idle and the host waiting (15k nodes, WIC, k = 50: CELF
// 83.6 ms on the tiered walks, 6.5 ms so).
constexpr int EV_MAX = 16;
struct EvalArgs {
    int32_t v[EV_MAX];
    uint32_t *bits;
    int32_t *queue;
    unsigned long long *out;
};
__global__ void __launch_bounds__(256) snap_eval_kernel(SnapView v, EvalArgs ev, const unsigned long long *cov)
{
    __shared__ ExpandShared S;
    __shared__ QueueShared Q;
    __shared__ unsigned int sum;
    const int r = blockIdx.x, tid = threadIdx.x, lane = tid & 31, T = blockDim.x;
    const int x = ev.v[blockIdx.y];
    const unsigned long long *covw = cov + (size_t)(r >> 6) * (size_t)v.n;
    const unsigned long long cbit = 1ull << (r & 63);
    const SnapInfo *info = v.info + r;
    if (info->bad || (covw[x] & cbit)) return;
    const size_t io = (size_t)r * v.icap, jo = (size_t)r * v.jcap;
    const uint32_t *outb = v.outb + (size_t)r * v.n32, *joinb = v.joinb + (size_t)r * v.n32;
    const uint32_t *jarc = v.jarc + (size_t)r * v.cap;
    const int4 *rec = v.rec + jo;
    const size_t slot = (size_t)blockIdx.y * v.R + r;
    uint32_t *bits = ev.bits + slot * v.jw;
    int32_t *ql = ev.queue + slot * v.jcap;
    const bool internal = sn_bit(outb, x), isj = sn_bit(joinb, x);
    unsigned int c = 0;
    if (tid == 0) {
        sum = 0;
        Q.tail = 0;
    }
    if (internal || isj) {
        const uint32_t *covj = v.covj + (size_t)r * v.jw;
        const int cw = (info->C + 31) >> 5;
        for (int i = tid; i < cw; i += T) bits[i] = covj[i];
        __syncthreads();
        auto below = [&](int j) {
            const int4 e = rec[j];
            return make_int2(e.z, e.w);
        };
        auto found = [&](uint32_t a) {
            const int j = (int)(a & ~ARC_LEAF);
            const uint32_t bit = 1u << (j & 31);
            const int2 e = a & ARC_LEAF ? make_int2(0, 0) : below(j);
            if (!(atomicOr(&bits[j >> 5], bit) & bit)) sn_push(Q, ql, j, e);
        };
        const int xi = internal ? sn_rank(outb, v.outp + (size_t)r * v.n32, x) : -1;
        if (isj) {
            if (tid == 0) found((uint32_t)sn_rank(joinb, v.joinp + (size_t)r * v.n32, x));
        } else {
            const int p0 = (int)sn_lo(v.pj[io + xi]), wd = sn_hi(v.acc[io + xi]);
            for (int k = tid; k < wd; k += T) found(jarc[p0 + k]);
        }
        const int nd = sn_search(S, Q, ql, 0, below, [&](int k) { found(jarc[k]); });
        for (int q = tid; q < nd; q += T) c += (unsigned)rec[ql[q]].x;
        if (!isj) {
            // T(x), unless its tree is among those found
            const int rj = v.jid[io + ~sn_hi(v.pj[io + xi])];
            if (rj < 0 || !sn_bit(bits, rj)) {
                const int2 *tn = v.tn + (size_t)r * v.tcap + (int)sn_lo(v.pn[io + xi]);
                const int len = (int)sn_lo(v.acc[io + xi]);
                for (int k = tid; k < len; k += T) c += !(covw[tn[k].x] & cbit);
            }
        }
    } else {
        __syncthreads();
        c = tid == 0;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(SN_FULL, c, o);
    if (lane == 0 && c) atomicAdd(&sum, c);
    __syncthreads();
    if (tid == 0) atomicAdd(&ev.out[blockIdx.y], (unsigned long long)sum);
}

__global__ void snap_choose_kernel(Ctl *ctl, int32_t x, long long *before)
{
    ctl->vstar = x;
    *before = (long long)ctl->du_entries;
}

// What the nodes marked in a round lose, one thread each (a warp claims 32
// tasks of a snapshot); ranges that are too large go to the warp walks.  R-MAT
// 20, R = 256: 6 ms a selection; with these walks as the first stage of the warp
// kernel, whose lanes then waited for the chunk's large ones, its 43 ms became 71.
template <bool EDGES>
__global__ void __launch_bounds__(256) snap_lose_kernel(SnapView v, Ctl *ctl, long long *s)
{
    __shared__ uint32_t list[SW_CAP][256];
    __shared__ int sh[33];
    __shared__ int last;
    chain_start();
    const int tid = threadIdx.x, lane = tid & 31;
    const int total = v.cstart[2 * v.R];
    if (v.cstart[2 * v.R + 3] || total == 0) return;
    unsigned long long edges = 0;
    while (true) {
        int ch = 0;
        if (lane == 0) ch = atomicAdd(v.cnext, 1);
        ch = __shfl_sync(SN_FULL, ch, 0);
        if (ch >= total) break;
        const int q = find_chunk(v.cstart, 2 * v.R, ch);
        const int r = q >> 1, seg = q & 1;
        SnapInfo *info = v.info + r;
        const int k = (ch - v.cstart[q]) * 32 + lane;
        if (k >= (seg ? info->t1 : info->t0)) continue;
        const size_t io = (size_t)r * v.icap, jw = (size_t)r * v.jw;
        const int i = v.task[io + (seg ? v.icap - 1 - k : k)];
        unsigned int c = seg ? (unsigned)info->lmk_cnt : 0u, d = 0;
        int n;
        const int2 a = v.rrange[io + i];
        if (small_walk<false>(&list[0][tid], 256, v.rarc + (size_t)r * v.cap, v.rrec + (size_t)r * v.jcap,
                              seg ? v.lmc + jw : nullptr, a.x, a.y, c, d, n))
            edges += snap_lose<EDGES>(v, s, io, i, c);
        else if (seg)
            v.ilist[io + v.icap - 1 - atomicAdd(&info->f1, 1)] = i;
        else
            v.ilist[io + atomicAdd(&info->f0, 1)] = i;
    }
    if (EDGES) {
        __syncwarp();
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) edges += __shfl_xor_sync(SN_FULL, edges, o);
        if (lane == 0 && edges) atomicAdd(&ctl->rev_edges, edges);
    }
    __syncthreads();
    if (tid == 0) {
        __threadfence();
        last = atomicAdd(v.arrive, 1) == (int)gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    sn_plan(v, sh, 1, WK_CH, [&](int q, int seg) { return sn_vol(seg ? &v.info[q].f1 : &v.info[q].f0); },
            [&](int q) { return sn_vol(&v.info[q].nrel); });
    if (tid == 0) *v.arrive = 0;
}

}  // namespace
}  // namespace sgi
