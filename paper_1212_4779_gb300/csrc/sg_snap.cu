// sg_snap.cu -- the compact snapshot graphs: when a query takes them, their
// device memory, and the launches (kernels in sg_snap_kernels.cuh).
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <cmath>

#include "sg_snap_kernels.cuh"

namespace sgi {

namespace {

constexpr size_t SNAP_BYTES_MAX = (size_t)64 << 30;
constexpr int WALK_BLOCKS = 2;                // closure-walk blocks per SM
// Their shared memory for bitmaps and queues: over all joins (initial
// gains), over the relevant ones (rounds, which leave more of the SM to L1
// for the relevance bitmaps).
constexpr int WALK_SMEM = 108 << 10;
constexpr int ROUND_SMEM = 64 << 10;

// Live arcs reserved per snapshot.  Their number is a sum of independent
// coins: the mean plus 16 standard deviations (and a constant for small
// means) is passed with a probability below e^-120; a snapshot that does
// pass it is reported (FLAG_SNAPSHOT), never truncated.  LT keeps at most
// one in-arc per node.
int64_t live_cap(const sg_graph *g, const Coins &co, int model)
{
    double mean;
    if (co.lt) return std::max<int64_t>(1, std::min(g->m, g->n_in));
    if (model == MODEL_WIC) mean = (double)g->n_in;
    else mean = co.none_live ? 0.0 : (double)g->m * (((double)co.uic_tm1 + 1.0) / 4294967296.0);
    const double c = mean + 16.0 * std::sqrt(mean) + 256.0;
    return std::max<int64_t>(1, std::min<int64_t>(g->m, (int64_t)c));
}

struct Carve {
    unsigned char *base;
    size_t off = 0;
    template <class T>
    void take(T *&p, size_t count)
    {
        off = (off + 255) & ~(size_t)255;
        p = base ? reinterpret_cast<T *>(base + off) : nullptr;
        off += count * sizeof(T);
    }
};

// Lays the arrays out from `base` (NULL: sizes only); returns the bytes.
// `clear` / `clear_bytes`: the leading part a query starts from zero.
size_t carve(const sg_graph *g, const Coins &co, int model, unsigned char *base, SnapView &v,
             unsigned long long **lm, size_t *clear_bytes)
{
    v = SnapView{};
    v.n = (int32_t)g->n;
    v.m = g->m;
    v.R = co.R;
    v.W = co.W;
    v.cap = (int32_t)live_cap(g, co, model);
    v.icap = (int32_t)std::min<int64_t>(g->n, v.cap);
    v.jcap = v.icap;
    v.tcap = (int32_t)std::min<int64_t>(g->n, 2 * (int64_t)v.cap);
    v.iw = (v.icap + 31) / 32;
    v.jw = (v.jcap + 127) / 128 * 4;  // copied 16 bytes at a time
    v.aw = (v.cap + 31) / 32;
    v.n32 = (g->n + 255) / 256 * 8;
    v.m32 = (g->m + 255) / 256 * 8;
    v.wwarps = g->num_sms * WALK_BLOCKS * WK_W;
    v.rp = g->rp.p;
    v.col = g->col.p;
    v.esrc = g->esrc.p;
    v.crp = g->crp.p;
    v.cin = g->cin.p;
    const size_t R = (size_t)co.R, nw = (size_t)g->n * co.W;
    const size_t ri = R * v.icap, rj = R * v.jcap, rc = R * v.cap;
    const size_t wb = (size_t)g->num_sms * WALK_BLOCKS;
    Carve c{base};
    c.take(v.cnext, 1);
    c.take(v.arrive, 1);
    c.take(v.any, nw);
    c.take(v.join, nw);
    c.take(v.oany, nw);
    c.take(v.covi, R * v.iw);
    c.take(v.covj, R * v.jw);
    if (clear_bytes) *clear_bytes = c.off;
    c.take(v.lb, R * v.m32);
    c.take(v.outb, R * v.n32);
    c.take(v.joinb, R * v.n32);
    c.take(v.outp, R * v.n32);
    c.take(v.joinp, R * v.n32);
    c.take(v.info, R);
    c.take(v.arc, rc);
    c.take(v.inode, ri);
    c.take(v.par, ri);
    c.take(v.pend, ri);
    c.take(v.share, ri);
    c.take(v.jid, ri);
    c.take(v.deg, ri);
    c.take(v.cnt, ri);
    c.take(v.acc, ri);
    c.take(v.pj, ri);
    c.take(v.pn, ri);
    c.take(v.up, ri);
    // the rounds' ranges lie where the initial gains' landmarks were
    c.take(v.rrange, std::max(ri, (R * SN_LMK * v.jw + 1) / 2));
    v.lmi = reinterpret_cast<uint32_t *>(v.rrange);
    c.take(v.cv, ri);
    c.take(v.task, ri);
    c.take(v.fb, ri);
    c.take(v.ilist, ri);
    c.take(v.rec, rj);
    c.take(v.jnode, rj);
    c.take(v.jtn, rj);
    c.take(v.jlist, rj);
    c.take(v.inoff, R * ((size_t)v.jcap + 1));
    c.take(v.jarc, rc);
    c.take(v.jin, rc);
    c.take(v.tn, R * v.tcap);
    c.take(v.marki, R * v.iw);
    c.take(v.rel, R * v.jw);
    c.take(v.rel2, R * v.jw);
    c.take(v.lmr, R * v.jw);
    c.take(v.lmc, R * v.jw);
    c.take(v.rrec, rj);
    c.take(v.rarc, rc);
    c.take(v.apos, rc);
    c.take(v.abit, R * v.aw);
    c.take(v.abit2, R * v.aw);
    c.take(v.cstart, 2 * R + 4);
    c.take(v.wq, wb * WK_W * WK_QG);
    c.take(v.gbm, wb * v.jw);
    c.take(v.lmt, R * SN_LMK);
    unsigned long long *masks = nullptr;
    if (co.lt) c.take(masks, (size_t)g->m * co.W);
    if (lm) *lm = masks;
    return c.off;
}

__global__ void __launch_bounds__(256) arc_sources_kernel(int n, const int32_t *rp, int32_t *esrc)
{
    // one warp per row
    const int lane = threadIdx.x & 31;
    const long long nw = ((long long)gridDim.x * blockDim.x) >> 5;
    for (long long u = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5; u < n; u += nw)
        for (int e = __ldg(rp + u) + lane; e < __ldg(rp + u + 1); e += 32) esrc[e] = (int32_t)u;
}

}  // namespace

// The compact snapshot graphs serve every directed cascade and LT.  The
// tiered engines remain for the calls that set one of their knobs (whoever
// asks for a tier, a landmark count or a cache gets it), for graphs without
// arcs, and where the graphs would pass SNAP_BYTES_MAX.  Per place reserved, a
// snapshot takes 28 bytes for a live arc, 88 for an internal node, 52 for a join
// and 8 for a tree node, and nodes and joins have as many places as live arcs
// have, up to n.  Under WIC and LT that is 184 to 200 bytes per live arc (R-MAT
// 20, R = 256: 21 GiB; a weighted R-MAT 22 passes the limit near R = 175); where
// the live arcs far outnumber the nodes it comes near 28.
bool snap_route(const sg_graph *g, const Coins &co, int model)
{
    const Knobs k = knobs();
    if (k.walk_groups != 64 || k.bu_mode != 1 || k.bu_div != 4 || k.t1_keys != 64 || k.t2_keys != 2048 ||
        k.landmarks != 8 || k.scc != 1 || k.fwd_lists != 1 || k.word_major != 1 || k.t1_direct != 16)
        return false;
    if (g_mask_cache || !g_snapshot_lists || g->heavy_min_deg != 2 || g->m == 0) return false;
    return snap_bytes(g, co, model) <= SNAP_BYTES_MAX;
}

size_t snap_bytes(const sg_graph *g, const Coins &co, int model)
{
    SnapView v;
    return carve(g, co, model, nullptr, v, nullptr, nullptr);
}

sg_status build_arc_sources(sg_graph *g, cudaStream_t st)
{
    if (g->esrc.p || g->m == 0) return SG_OK;
    SG_TRY(dbuf_alloc(g->esrc, (size_t)g->m, st));
    const int blocks = (int)std::min<long long>((g->n * 32 + 255) / 256, (long long)g->num_sms * 16);
    arc_sources_kernel<<<blocks, 256, 0, st>>>((int)g->n, g->rp.p, g->esrc.p);
    SG_CUDA_TRY(cudaGetLastError());
    ++g_launches;
    return SG_OK;
}

static size_t free_device_memory()
{
    size_t fr = 0, all = 0;
    if (cudaMemGetInfo(&fr, &all) != cudaSuccess) cudaGetLastError();
    return fr;
}

// Whether a size that was refused is asked for again: when the device has
// clearly more room than it had then, else (memory behind the allocator hooks
// does not show there) after 4 more queries, then 8, 16, ... 64, since a
// refused request can be dear to whoever refuses it (a caching allocator gives
// up its cache first).  A stream that is being captured takes the route its
// query was sized for.
static bool snap_ask(sg_workspace &ws, size_t need, cudaStream_t st)
{
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(st, &cs) != cudaSuccess) cudaGetLastError();
    if (cs != cudaStreamCaptureStatusNone) return false;
    if (free_device_memory() > ws.snap_free + need / 8) return true;
    if (--ws.snap_wait > 0) return false;
    return true;
}

// Sizes ws for a query on the compact graphs; *snap false, with nothing more
// done, where it goes to the tiered engines: by snap_route, or because the
// graphs do not fit into the device's memory (dense cascades: the engines'
// arrays do not grow with the live arcs).
sg_status ensure_snap(sg_graph *g, sg_workspace &ws, const Coins &co, int model, int32_t k, cudaStream_t st,
                      bool *snap)
{
    const size_t need = snap_bytes(g, co, model);
    *snap = !ws.engines_only && snap_route(g, co, model) && (need < ws.snap_limit || snap_ask(ws, need, st));
    if (!*snap) return SG_OK;
    SG_TRY(ensure_core(g, ws, co.W, k, st));
    if (ws.snap.bytes >= need) return SG_OK;
    dbuf_free(ws.snap, st);
    if (dbuf_alloc(ws.snap, need, st) != SG_OK) {
        clear_error();
        ws.snap_gap = ws.snap_limit == SIZE_MAX ? 4 : std::min(64, 2 * ws.snap_gap);
        ws.snap_wait = ws.snap_gap;
        ws.snap_limit = need;
        ws.snap_free = free_device_memory();
        *snap = false;
    } else if (need >= ws.snap_limit) {
        ws.snap_limit = SIZE_MAX;
    }
    return SG_OK;
}

namespace {

template <int MODE, bool EDGES>
sg_status launch_walk(sg_graph *g, sg_workspace &ws, const SnapView &v, cudaStream_t st)
{
    auto kern = snap_walk_kernel<MODE, EDGES>;
    constexpr int smem = MODE == 2 ? ROUND_SMEM : WALK_SMEM;
    SG_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    SG_CUDA_TRY(launch_chained(kern, g->num_sms * WALK_BLOCKS, WK_T, smem, st, v, ws.ctl.p, ws.s.p, smem));
    ++g_launches;
    return SG_OK;
}

}  // namespace

// Threads of the kernels that give each snapshot one block.
static int snap_threads(const SnapView &v) { return v.cap >= 8192 ? 1024 : 256; }

// Coins and compact graphs of every snapshot.
sg_status run_snap_build(sg_graph *g, sg_workspace &ws, const Coins &co, int model, cudaStream_t st)
{
    SnapView v;
    unsigned long long *lm = nullptr;
    size_t clear = 0;
    carve(g, co, model, ws.snap.p, v, &lm, &clear);
    SG_CUDA_TRY(cudaMemsetAsync(ws.snap.p, 0, clear, st));
    const int tiles = (int)std::min<long long>((v.m + SN_TILE - 1) / SN_TILE, (long long)g->num_sms * 8);
    if (co.lt) {
        SG_CUDA_TRY(cudaMemsetAsync(lm, 0, (size_t)g->m * co.W * 8, st));
        SG_TRY(run_lt_masks(g, co, 0, co.W, nullptr, lm, nullptr, 0, st));
        snap_coins_kernel<2><<<tiles, SN_TILE, 0, st>>>(v, co, nullptr, lm);
    } else if (model == MODEL_WIC) {
        snap_coins_kernel<1><<<tiles, SN_TILE, 0, st>>>(v, co, g->fw.p, nullptr);
    } else {
        snap_coins_kernel<0><<<tiles, SN_TILE, 0, st>>>(v, co, nullptr, nullptr);
    }
    SG_CUDA_TRY(cudaGetLastError());
    const int ntiles = (int)std::min<long long>(((long long)v.n + SN_TILE - 1) / SN_TILE, (long long)g->num_sms * 8);
    SG_CUDA_TRY(launch_chained(snap_nodes_kernel, ntiles, SN_TILE, 0, st, v, ws.ctl.p, ws.s.p));
    SG_CUDA_TRY(launch_chained(snap_compact_kernel, v.R, snap_threads(v), 0, st, v, ws.ctl.p));
    SG_CUDA_TRY(launch_chained(snap_trees_kernel, v.R, snap_threads(v), 0, st, v, ws.ctl.p));
    SG_CUDA_TRY(launch_chained(snap_place_kernel, v.R, snap_threads(v), 0, st, v));
    g_launches += 5;
    return SG_OK;
}

// Initial gains into ws.s; their edge count only if `edges`.
sg_status run_snap_init(sg_graph *g, sg_workspace &ws, const Coins &co, int model, bool edges, cudaStream_t st,
                        const TierEvents *ev)
{
    SnapView v;
    carve(g, co, model, ws.snap.p, v, nullptr, nullptr);
    if (ev && ev->start) SG_CUDA_TRY(cudaEventRecord(ev->start, st));
    // blocks per snapshot of the kernels that give each internal node a thread
    const int per = (int)std::max<long long>(1, std::min<long long>((v.icap + 1023) / 1024, (8LL * g->num_sms + v.R - 1) / v.R));
    SG_CUDA_TRY(launch_chained(edges ? snap_small_kernel<true> : snap_small_kernel<false>, v.R * per, 256, 0, st, v));
    if (edges) SG_TRY((launch_walk<0, true>(g, ws, v, st)));
    else SG_TRY((launch_walk<0, false>(g, ws, v, st)));
    if (ev && ev->t1) SG_CUDA_TRY(cudaEventRecord(ev->t1, st));
    SG_CUDA_TRY(launch_chained(edges ? snap_resolve_kernel<true> : snap_resolve_kernel<false>, v.R * per, 256, 0, st, v,
                               ws.ctl.p, ws.s.p));
    g_launches += 2;
    if (ev && ev->t2) SG_CUDA_TRY(cudaEventRecord(ev->t2, st));
    if (edges) SG_TRY((launch_walk<1, true>(g, ws, v, st)));
    else SG_TRY((launch_walk<1, false>(g, ws, v, st)));
    // the landmark marks give way to the rounds' marks
    SG_CUDA_TRY(cudaMemsetAsync(v.marki, 0, (size_t)v.R * v.iw * 4, st));
    if (ev && ev->t3) SG_CUDA_TRY(cudaEventRecord(ev->t3, st));
    return SG_OK;
}

// Candidates one evaluation launch takes: their scratch within 8 GiB.
int32_t snap_eval_count(const sg_graph *g, const Coins &co, int model)
{
    SnapView v;
    carve(g, co, model, nullptr, v, nullptr, nullptr);
    const size_t each = (size_t)v.R * ((size_t)v.jcap + v.jw) * 4;
    return (int32_t)std::max<size_t>(1, std::min<size_t>(EV_MAX, ((size_t)8 << 30) / each));
}

size_t snap_eval_words(const sg_graph *g, const Coins &co, int model, int32_t count)
{
    SnapView v;
    carve(g, co, model, nullptr, v, nullptr, nullptr);
    return (size_t)count * v.R * ((size_t)v.jcap + v.jw);
}

// out[b] = marginal gain of cand[b], b < count <= room (scratch: snap_eval_words
// of room).
sg_status run_snap_eval(sg_graph *g, sg_workspace &ws, const Coins &co, int model, const int32_t *cand, int32_t count,
                        int32_t room, uint32_t *scratch, unsigned long long *out, cudaStream_t st)
{
    SnapView v;
    carve(g, co, model, ws.snap.p, v, nullptr, nullptr);
    EvalArgs ev{};
    for (int32_t b = 0; b < count; ++b) ev.v[b] = cand[b];
    ev.bits = scratch;
    ev.queue = reinterpret_cast<int32_t *>(scratch + (size_t)room * v.R * v.jw);
    ev.out = out;
    SG_CUDA_TRY(cudaMemsetAsync(out, 0, (size_t)count * 8, st));
    snap_eval_kernel<<<dim3((unsigned)v.R, (unsigned)count), 256, 0, st>>>(v, ev, ws.cov.p);
    SG_CUDA_TRY(cudaGetLastError());
    ++g_launches;
    return SG_OK;
}

// Covers what x reaches (forward edges and newly covered pairs into ctl);
// *before: the pairs covered until then.
sg_status run_snap_cover(sg_graph *g, sg_workspace &ws, const Coins &co, int model, int32_t x, long long *before,
                         cudaStream_t st)
{
    SnapView v;
    carve(g, co, model, ws.snap.p, v, nullptr, nullptr);
    snap_choose_kernel<<<1, 1, 0, st>>>(ws.ctl.p, x, before);
    snap_cover_kernel<true, false><<<v.R, snap_threads(v), 0, st>>>(v, ws.ctl.p, ws.s.p, ws.cov.p, 1);
    SG_CUDA_TRY(cudaGetLastError());
    g_launches += 2;
    return SG_OK;
}

// One selection round: argmax, cover, update; the edge counts only if `edges`.
sg_status run_snap_round(sg_graph *g, sg_workspace &ws, const Coins &co, int model, bool edges, int32_t round,
                         cudaStream_t st, cudaEvent_t after_cover)
{
    SnapView v;
    carve(g, co, model, ws.snap.p, v, nullptr, nullptr);
    SG_TRY(run_argmax(g, ws, co, round, st));
    // Small queries (at most 2^18 internal nodes over all snapshots) mark a
    // few hundred nodes a round; walking those by warps at once saves a launch.
    const int direct = (long long)v.R * v.icap <= (1 << 18);
    SG_CUDA_TRY(launch_chained(edges ? snap_cover_kernel<true, true> : snap_cover_kernel<false, true>, v.R,
                               snap_threads(v), 0, st, v, ws.ctl.p, ws.s.p, ws.cov.p, direct));
    ++g_launches;
    if (after_cover) SG_CUDA_TRY(cudaEventRecord(after_cover, st));
    if (!direct) {
        const int blocks = g->num_sms * 6;
        SG_CUDA_TRY(launch_chained(edges ? snap_lose_kernel<true> : snap_lose_kernel<false>, blocks, 256, 0, st, v,
                                   ws.ctl.p, ws.s.p));
        ++g_launches;
    }
    if (edges) return launch_walk<2, true>(g, ws, v, st);
    return launch_walk<2, false>(g, ws, v, st);
}

}  // namespace sgi
