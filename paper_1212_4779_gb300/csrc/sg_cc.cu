// sg_cc.cu -- the undirected variant: uniform cascade on a symmetric graph
// with one coin per undirected edge (both arcs hash the lower of their two
// canonical arc ids).  Each snapshot is then an undirected graph, as Section
// 3.4.1 treats undirected snapshots, and R(G'_r, v) is v's connected
// component.  So Algorithm 2 reduces to component bookkeeping:
//   initial gains   s_v = sum_r |C_r(v)| (union-find per snapshot);
//   a round's seed  v*: in every snapshot where C_r(v*) is not yet covered,
//                   its |C_r(v*)| nodes are newly covered, and each of them
//                   (each reaches every newly covered node) loses |C_r(v*)|.
// The snapshot-edge counters follow from per-component sizes and degree
// sums, equal to the dynamic update's counts: init = sum_{v,r} degsum(C_r(v));
// forward = sum over newly covered components of degsum; reverse = sum over
// them of |C| * degsum (every node of C is reached backwards from each of the
// |C| newly covered nodes, and in-degree = out-degree).
#include <cuda_runtime.h>
#include <stdint.h>
#include <string.h>

#include <algorithm>

#include "sg_internal.cuh"

using namespace sgi;

namespace {

constexpr int CC_T = 256;
constexpr long long CC_SPIN = 1LL << 24;


// Source of every arc and the lower id of each arc and its reverse;
// *asym is set if some arc has no reverse.
__global__ void cc_coupling_kernel(int n, long long m, const int32_t *rp, const int32_t *col, int32_t *esrc,
                                   int32_t *pmin, int32_t *asym)
{
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < m; e += (long long)gridDim.x * blockDim.x) {
        int lo = 0, hi = n - 1;  // the row holding arc e: largest u with rp[u] <= e
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (__ldg(rp + mid) <= e) lo = mid;
            else hi = mid - 1;
        }
        const int u = lo, v = __ldg(col + e);
        int a = __ldg(rp + v), b = __ldg(rp + v + 1);
        while (a < b) {
            const int mid = (a + b) >> 1;
            if (__ldg(col + mid) < u) a = mid + 1;
            else b = mid;
        }
        const bool found = a < __ldg(rp + v + 1) && __ldg(col + a) == u;
        if (!found) *asym = 1;
        esrc[e] = u;
        pmin[e] = found ? (int32_t)min((long long)a, e) : (int32_t)e;
    }
}

__device__ __forceinline__ int cc_find(int32_t *lab, int x)
{
    // path halving; the shortcuts written are ancestors, so races only
    // leave longer paths, never wrong roots
    while (true) {
        const int p = *(volatile int32_t *)&lab[x];
        if (p == x) return x;
        const int gp = *(volatile int32_t *)&lab[p];
        if (gp != p) *(volatile int32_t *)&lab[x] = gp;
        x = gp;
    }
}

// Root without writing: used once hooking is over, while other threads
// store their final roots (a shortcut written then could overwrite a final
// root with an intermediate ancestor).
__device__ __forceinline__ int cc_root(const int32_t *lab, int x)
{
    while (true) {
        const int p = *(volatile const int32_t *)&lab[x];
        if (p == x) return x;
        x = p;
    }
}

__global__ void cc_init_kernel(int n, long long total, int32_t *lab)
{
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total;
         i += (long long)gridDim.x * blockDim.x)
        lab[i] = (int32_t)(i % n);
}

// Union the endpoints of every live undirected edge {u, v} (u < v, arc
// u->v is the lower id) in every snapshot; the larger root is hooked under
// the smaller by compare-and-swap.  A bounded number of retries per edge;
// on expiry the error flag is set.  A union is a chain of dependent reads of
// the labels, so a warp that tosses 32 coins and then waits for the one or two
// lanes whose coin landed spends its time idle: a block tosses the coins of
// CC_T edges in CC_RB snapshots first and unions from a list of those that
// landed, one a thread.  241 -> 92 us (37k nodes, 463k arcs, 100 snapshots).
constexpr int CC_RB = 32;
__global__ void __launch_bounds__(CC_T) cc_hook_kernel(int n, long long m, int R, uint64_t seed, uint32_t tm1,
                                                       int none_live, const int32_t *esrc, const int32_t *col,
                                                       int32_t *lab, int32_t *flags)
{
    static_assert(CC_T * CC_RB <= 65536, "a list entry is 16 bits");
    __shared__ uint16_t landed[CC_T * CC_RB];
    __shared__ int su[CC_T], sw[CC_T];
    __shared__ int count;
    if (none_live) return;
    const int tid = threadIdx.x;
    const long long tiles = (m + CC_T - 1) / CC_T;
    const int rb = (R + CC_RB - 1) / CC_RB;
    for (long long t = blockIdx.x; t < tiles * rb; t += gridDim.x) {
        const int r0 = (int)(t % rb) * CC_RB, nr = min(R - r0, CC_RB);
        const long long e = t / rb * CC_T + tid;
        __syncthreads();  // the list of the last tile is done with
        if (tid == 0) count = 0;
        int u = 0, w = 0;
        if (e < m) {
            u = __ldg(esrc + e);
            w = __ldg(col + e);
        }
        su[tid] = u;
        sw[tid] = w;
        uint32_t mine = 0;
        if (u < w)
            for (int r = 0; r < nr; ++r)
                mine |= (uint32_t)(coin_hi32(seed ^ (uint64_t)e, (uint32_t)(r0 + r)) <= tm1) << r;
        __syncthreads();
        int at = mine ? atomicAdd(&count, __popc(mine)) : 0;
        for (; mine; mine &= mine - 1) landed[at++] = (uint16_t)(tid * CC_RB + __ffs(mine) - 1);
        __syncthreads();
        for (int q = tid; q < count; q += CC_T) {
            int32_t *L = lab + (size_t)(r0 + landed[q] % CC_RB) * n;
            int a = su[landed[q] / CC_RB], b = sw[landed[q] / CC_RB];
            long long tries = 0;
            while (true) {
                a = cc_find(L, a);
                b = cc_find(L, b);
                if (a == b) break;
                if (a > b) {
                    const int x = a;
                    a = b;
                    b = x;
                }
                const int old = atomicCAS(&L[b], b, a);
                if (old == b) break;
                b = old;
                if (++tries > CC_SPIN) {
                    atomicOr(flags, 8);
                    break;
                }
            }
        }
    }
}

// lab[r][v] = its root; component sizes and out-degree sums at the roots
// (csz, cdg zero on entry).  The nodes of a warp that share a root add to it
// once: a giant component's root otherwise takes one atomic per node (124 ->
// 48 us, same graph).
__global__ void __launch_bounds__(CC_T) cc_compress_kernel(int n, int R, const int32_t *rp, int32_t *lab,
                                                           int32_t *csz, unsigned long long *cdg)
{
    const int tiles = (n + CC_T - 1) / CC_T, lane = threadIdx.x & 31;
    for (long long t = blockIdx.x; t < (long long)tiles * R; t += gridDim.x) {
        const int r = (int)(t / tiles);
        const int v = (int)(t % tiles) * CC_T + threadIdx.x;
        int32_t *L = lab + (size_t)r * n;
        int root = -1 - lane;  // past the last node: a group of its own
        uint32_t deg = 0;
        if (v < n) {
            root = cc_root(L, v);
            L[v] = root;  // only this thread writes L[v] here
            deg = (uint32_t)(__ldg(rp + v + 1) - __ldg(rp + v));
        }
        const unsigned same = __match_any_sync(0xffffffffu, root);
        uint32_t lo = deg & 0xffffu, hi = deg >> 16;  // 32 of either cannot overflow
        if (same & (same - 1)) {
            lo = __reduce_add_sync(same, lo);
            hi = __reduce_add_sync(same, hi);
        }
        if (root >= 0 && lane == __ffs(same) - 1) {
            atomicAdd(&csz[(size_t)r * n + root], __popc(same));
            atomicAdd(&cdg[(size_t)r * n + root], ((unsigned long long)hi << 16) + lo);
        }
    }
}

// s_v = sum_r |C_r(v)|; the initial snapshot-edge count.
__global__ void __launch_bounds__(CC_T) cc_gains_kernel(int n, int R, const int32_t *lab, const int32_t *csz,
                                                        const unsigned long long *cdg, long long *s,
                                                        unsigned long long *init_edges)
{
    __shared__ unsigned long long red[CC_T / 32];
    unsigned long long ed = 0;
    for (long long v = (long long)blockIdx.x * CC_T + threadIdx.x; v < n; v += (long long)gridDim.x * CC_T) {
        long long acc = 0;
        for (int r = 0; r < R; ++r) {
            const size_t q = (size_t)r * n + __ldg(lab + (size_t)r * n + v);
            acc += __ldg(csz + q);
            ed += __ldg(cdg + q);
        }
        s[v] = acc;
    }
    for (int o = 16; o > 0; o >>= 1) ed += __shfl_xor_sync(0xffffffffu, ed, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = ed;
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned long long t = 0;
        for (int w = 0; w < CC_T / 32; ++w) t += red[w];
        if (t) atomicAdd(init_edges, t);
    }
}

// One round after the seed v* (ctl->vstar) is chosen, and the choice of the
// next: in every snapshot where v*'s component is not yet covered, each of its
// nodes loses its size; the same pass over the nodes takes the largest
// remaining gain (lowest id on ties), which the last block publishes.  Rounds
// as three launches (cover, decrement, argmax) spent much of their time between
// them: the whole selection of 50 seeds on 37k nodes and 100 snapshots took
// 1.81 ms, with one launch a round 1.06 ms.
// Every block finds the newly covered components itself, so none may be
// flagged while others look: block 0 notes a round's roots in proot (by the
// round's parity, -1: none) and sets their flags one round later.  Snapshots
// are taken CC_R at a time.
constexpr int CC_R = 512;
__global__ void __launch_bounds__(CC_T) cc_round_kernel(int n, int R, int round, int last_round, const int32_t *lab,
                                                        const int32_t *csz, const unsigned long long *cdg,
                                                        uint8_t *cov, int32_t *proot, Ctl *ctl, long long *s,
                                                        long long *pg, int *pi,
                                                        int32_t *out_seeds, long long *out_gains)
{
    __shared__ int root[CC_R], nsz[CC_R], snap[CC_R];
    __shared__ int live;
    __shared__ long long sg[CC_T / 32];
    __shared__ int si[CC_T / 32];
    __shared__ int sh_last;
    chain_start();
    const int vs = *(volatile int32_t *)&ctl->vstar;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    unsigned long long fwd = 0, rev = 0;
    for (int r0 = 0; r0 < R; r0 += CC_R) {
        __syncthreads();
        if (tid == 0) live = 0;
        __syncthreads();
        for (int r = r0 + tid; r < min(R, r0 + CC_R); r += CC_T) {
            const int before = proot[(size_t)(~round & 1) * R + r];
            const int c = vs >= 0 ? __ldg(lab + (size_t)r * n + vs) : -1;
            const size_t q = (size_t)r * n + max(c, 0);
            const bool fresh = c >= 0 && c != before && !*(volatile uint8_t *)&cov[q];
            if (blockIdx.x == 0) {
                if (before >= 0) cov[(size_t)r * n + before] = 1;
                proot[(size_t)(round & 1) * R + r] = fresh ? c : -1;
            }
            if (!fresh) continue;
            const int sz = csz[q];
            if (blockIdx.x == 0) {
                fwd += cdg[q];
                rev += (unsigned long long)sz * cdg[q];
            }
            const int k = atomicAdd(&live, 1);
            root[k] = c;
            nsz[k] = sz;
            snap[k] = r;
        }
        __syncthreads();
        const int nl = live;
        if (nl == 0) continue;
        for (long long v = (long long)blockIdx.x * CC_T + tid; v < n; v += (long long)gridDim.x * CC_T) {
            long long dec = 0;
#pragma unroll 4
            for (int k = 0; k < nl; ++k)
                if (__ldg(lab + (size_t)snap[k] * n + v) == root[k]) dec += nsz[k];
            if (dec) s[v] -= dec;
        }
    }
    if (fwd) atomicAdd(&ctl->fwd_edges, fwd);
    if (rev) atomicAdd(&ctl->rev_edges, rev);
    if (last_round) return;
    auto better = [](long long g1, int i1, long long g2, int i2) {
        return g1 > g2 || (g1 == g2 && (unsigned)i1 < (unsigned)i2);
    };
    long long bg = -1;
    int bi = -1;
    for (long long v = (long long)blockIdx.x * CC_T + tid; v < n; v += (long long)gridDim.x * CC_T) {
        const long long x = s[v];  // seeds are negative
        if (x > bg) {
            bg = x;
            bi = (int)v;
        }
    }
    auto reduce = [&]() {  // (bg, bi) of the block in thread 0
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const long long og = __shfl_xor_sync(0xffffffffu, bg, o);
            const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
            if (better(og, oi, bg, bi)) {
                bg = og;
                bi = oi;
            }
        }
        __syncthreads();
        if (lane == 0) {
            sg[wid] = bg;
            si[wid] = bi;
        }
        __syncthreads();
        if (tid == 0)
            for (int w = 1; w < CC_T / 32; ++w)
                if (better(sg[w], si[w], bg, bi)) {
                    bg = sg[w];
                    bi = si[w];
                }
    };
    reduce();
    if (tid == 0) {
        pg[blockIdx.x] = bg;
        pi[blockIdx.x] = bi;
        chain_next();
        __threadfence();
        sh_last = atomicAdd(&ctl->argmax_arrivals, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!sh_last) return;
    __threadfence();
    bg = -1;
    bi = -1;
    for (int b = tid; b < (int)gridDim.x; b += CC_T) {
        const long long og = *(volatile long long *)&pg[b];
        const int oi = *(volatile int *)&pi[b];
        if (better(og, oi, bg, bi)) {
            bg = og;
            bi = oi;
        }
    }
    reduce();
    if (tid == 0) {
        out_seeds[round + 1] = bi;
        out_gains[round + 1] = bg;
        ctl->vstar = bi;
        if (bi >= 0) s[bi] = -(1LL << 62);
        else ctl->flags |= FLAG_NO_CANDIDATE;
        ctl->argmax_arrivals = 0;
    }
}

// Spread of S: per snapshot, the sizes of the distinct components S meets
// (mark zero on entry, reused as the "counted" flags).
__global__ void __launch_bounds__(CC_T) cc_spread_kernel(int n, int R, const int32_t *lab, const int32_t *csz,
                                                         const unsigned long long *cdg, const int32_t *S, int ns,
                                                         uint8_t *mark, long long *total, unsigned long long *edges)
{
    __shared__ long long rt[CC_T / 32];
    __shared__ unsigned long long re[CC_T / 32];
    long long t = 0;
    unsigned long long ed = 0;
    const long long work = (long long)R * ns;
    for (long long i = blockIdx.x * (long long)CC_T + threadIdx.x; i < work; i += (long long)gridDim.x * CC_T) {
        const int r = (int)(i / ns);
        const int v = __ldg(S + (i - (long long)r * ns));
        const size_t q = (size_t)r * n + __ldg(lab + (size_t)r * n + v);
        // one byte flag per (r, root): claim it with an atomic on its word
        unsigned int *wordp = (unsigned int *)(mark + (q & ~(size_t)3));
        const unsigned int bit = 1u << (8 * (q & 3));
        if (!(atomicOr(wordp, bit) & bit)) {
            t += __ldg(csz + q);
            ed += __ldg(cdg + q);
        }
    }
    for (int o = 16; o > 0; o >>= 1) {
        t += __shfl_xor_sync(0xffffffffu, t, o);
        ed += __shfl_xor_sync(0xffffffffu, ed, o);
    }
    if ((threadIdx.x & 31) == 0) {
        rt[threadIdx.x >> 5] = t;
        re[threadIdx.x >> 5] = ed;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        long long a = 0;
        unsigned long long b = 0;
        for (int w = 0; w < CC_T / 32; ++w) {
            a += rt[w];
            b += re[w];
        }
        if (a) atomicAdd((unsigned long long *)total, (unsigned long long)a);
        if (b) atomicAdd(edges, b);
    }
}

int grid_for(const sg_graph *g, long long work)
{
    return (int)std::max<long long>(1, std::min<long long>((work + CC_T - 1) / CC_T, (long long)g->num_sms * 16));
}

}  // namespace

namespace sgi {

// Coupling arrays of a symmetric graph, built on first use; SG_EINVAL for a
// graph with an arc whose reverse is missing.
sg_status cc_prepare_graph(sg_graph *g, cudaStream_t st)
{
    if (g->cc_sym == 0) {
        set_error("the undirected cascade needs a symmetric graph (every arc's reverse present)");
        return SG_EINVAL;
    }
    if (g->cc_sym == 1) return SG_OK;
    const long long m = g->m;
    DBuf<int32_t> flag;
    SG_TRY(dbuf_alloc(g->cc_esrc, (size_t)std::max<long long>(1, m), st));
    SG_TRY(dbuf_alloc(g->cc_pmin, (size_t)std::max<long long>(1, m), st));
    SG_TRY(dbuf_alloc(flag, 1, st));
    SG_CUDA_TRY(cudaMemsetAsync(flag.p, 0, 4, st));
    if (m > 0) {
        cc_coupling_kernel<<<grid_for(g, m), CC_T, 0, st>>>((int)g->n, m, g->rp.p, g->col.p, g->cc_esrc.p,
                                                            g->cc_pmin.p, flag.p);
        SG_CUDA_TRY(cudaGetLastError());
        ++g_launches;
    }
    int32_t h = 0;
    SG_CUDA_TRY(cudaMemcpyAsync(&h, flag.p, 4, cudaMemcpyDeviceToHost, st));
    SG_CUDA_TRY(cudaStreamSynchronize(st));
    dbuf_free(flag, st);
    g->cc_sym = h ? 0 : 1;
    if (!g->cc_sym) {
        set_error("the undirected cascade needs a symmetric graph (every arc's reverse present)");
        return SG_EINVAL;
    }
    return SG_OK;
}

size_t cc_workspace_bytes(const sg_graph *g, int32_t R)
{
    const size_t rn = (size_t)R * (size_t)g->n;
    return rn * (4 + 4 + 8 + 1) + (size_t)R * 8 + 64;
}

sg_status cc_ensure(sg_graph *g, sg_workspace &ws, int32_t R, cudaStream_t st)
{
    const size_t rn = (size_t)R * (size_t)g->n;
    if (ws.cc_cap < rn || ws.cc_rcap < R) {
        dbuf_free(ws.cc_lab, st);
        dbuf_free(ws.cc_size, st);
        dbuf_free(ws.cc_deg, st);
        dbuf_free(ws.cc_cov, st);
        dbuf_free(ws.cc_root, st);
        ws.cc_cap = 0;
        ws.cc_rcap = 0;
        SG_TRY(dbuf_alloc(ws.cc_lab, rn, st));
        SG_TRY(dbuf_alloc(ws.cc_size, rn, st));
        SG_TRY(dbuf_alloc(ws.cc_deg, rn, st));
        SG_TRY(dbuf_alloc(ws.cc_cov, rn + 8, st));
        SG_TRY(dbuf_alloc(ws.cc_root, (size_t)R * 2, st));
        ws.cc_cap = rn;
        ws.cc_rcap = R;
    }
    return SG_OK;
}

// Components of every snapshot (lab, csz, cdg) for R snapshots of `seed`.
sg_status cc_components(sg_graph *g, sg_workspace &ws, const Coins &co, cudaStream_t st)
{
    const long long total = (long long)co.R * g->n;
    SG_CUDA_TRY(cudaMemsetAsync(ws.cc_size.p, 0, (size_t)total * 4, st));
    SG_CUDA_TRY(cudaMemsetAsync(ws.cc_deg.p, 0, (size_t)total * 8, st));
    cc_init_kernel<<<grid_for(g, total), CC_T, 0, st>>>((int)g->n, total, ws.cc_lab.p);
    if (g->m > 0)
        cc_hook_kernel<<<grid_for(g, (long long)co.R * g->m), CC_T, 0, st>>>(
            (int)g->n, g->m, co.R, co.seed, co.uic_tm1, co.none_live, g->cc_esrc.p, g->col.p, ws.cc_lab.p,
            &ws.ctl.p->flags);
    cc_compress_kernel<<<grid_for(g, total), CC_T, 0, st>>>((int)g->n, co.R, g->rp.p, ws.cc_lab.p, ws.cc_size.p,
                                                             reinterpret_cast<unsigned long long *>(ws.cc_deg.p));
    SG_CUDA_TRY(cudaGetLastError());
    g_launches += 3;
    return SG_OK;
}

// Initial gains into ws.s and the init counter (ctl zeroed by the caller).
sg_status cc_init_gains(sg_graph *g, sg_workspace &ws, const Coins &co, cudaStream_t st)
{
    SG_TRY(cc_components(g, ws, co, st));
    cc_gains_kernel<<<grid_for(g, g->n), CC_T, 0, st>>>((int)g->n, co.R, ws.cc_lab.p, ws.cc_size.p,
                                                         reinterpret_cast<const unsigned long long *>(ws.cc_deg.p),
                                                         ws.s.p, &ws.ctl.p->init_edges);
    SG_CUDA_TRY(cudaGetLastError());
    ++g_launches;
    return SG_OK;
}

// Rounds 0 .. k - 1 (the first seed by the common argmax).
sg_status cc_rounds(sg_graph *g, sg_workspace &ws, const Coins &co, int32_t k, cudaStream_t st)
{
    SG_TRY(run_argmax(g, ws, co, 0, st));
    // one partial maximum per block
    const int blocks = std::min(ws.am_blocks, grid_for(g, g->n));
    for (int32_t i = 0; i < k; ++i) {
        SG_CUDA_TRY(launch_chained(cc_round_kernel, blocks, CC_T, 0, st, (int)g->n, co.R, i, i + 1 == k, ws.cc_lab.p,
                                   ws.cc_size.p, reinterpret_cast<const unsigned long long *>(ws.cc_deg.p),
                                   ws.cc_cov.p, ws.cc_root.p, ws.ctl.p, ws.s.p, ws.am_gain.p, ws.am_id.p,
                                   ws.out_seeds.p, ws.out_gains.p));
        ++g_launches;
    }
    return SG_OK;
}

sg_status cc_clear_cover(sg_graph *g, sg_workspace &ws, const Coins &co, cudaStream_t st)
{
    SG_CUDA_TRY(cudaMemsetAsync(ws.cc_cov.p, 0, (size_t)co.R * (size_t)g->n + 8, st));
    SG_CUDA_TRY(cudaMemsetAsync(ws.cc_root.p, 0xff, (size_t)co.R * 8, st));
    return SG_OK;
}

// sum_r |union of the components S meets|, and their degree sums.
sg_status cc_spread(sg_graph *g, sg_workspace &ws, const Coins &co, const int32_t *d_S, int32_t ns, long long *d_total,
                    unsigned long long *d_edges, cudaStream_t st)
{
    SG_TRY(cc_components(g, ws, co, st));
    SG_TRY(cc_clear_cover(g, ws, co, st));
    cc_spread_kernel<<<grid_for(g, (long long)co.R * ns), CC_T, 0, st>>>(
        (int)g->n, co.R, ws.cc_lab.p, ws.cc_size.p, reinterpret_cast<const unsigned long long *>(ws.cc_deg.p), d_S,
        ns, ws.cc_cov.p, d_total, d_edges);
    SG_CUDA_TRY(cudaGetLastError());
    ++g_launches;
    return SG_OK;
}

}  // namespace sgi
