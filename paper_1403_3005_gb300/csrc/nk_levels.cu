// Closeness sweeps: the levels of B = 64*W breadth-first searches at once, as bitsets, without
// path counts.  Closeness from one search per node, exact or for sampled sources (Table 1), needs
// only the distance of every vertex from every source: v is at distance d from the sources whose
// bit joins v's visited set at level d.
//
// State of one batch (q = word 0..W-1): F[d % 3][v][q] the sources with v on level d, vis[v][q]
// the union so far.  Level d, either
//   bottom-up  every vertex with unvisited sources ORs F_d of its neighbours, and stops reading
//              once every source it waits for has turned up;  or
//   top-down   every frontier vertex pushes its bits into its neighbours' F_{d+1} (atomicOr) and
//              queues each once per level.
// A vertex that joins level d+1 for c sources adds c (d+1) to its distance sum and c to its reach
// count at once, so no more than three levels are kept and a search may be as deep as the graph.
//
// What bounds it: a level reads a column id and a 32-byte bitset (W = 4) per arc of the vertices
// not yet complete, from L2 while the bitsets fit there.  The sums came from the betweenness
// sweep's forward half before, which gathers a row of path counts per arc and source.
#include <cooperative_groups.h>

#include <algorithm>
#include <vector>

#include "nk_device.cuh"
#include "nk_internal.h"
#include "nk_sweep.cuh"

namespace cg = cooperative_groups;

namespace nk {
namespace {

using namespace sweep;

constexpr int kThreads = 256;

struct LArgs {
    int32_t n;
    int64_t A;
    const int32_t *rp, *col;
    const int32_t *src;
    int32_t nsrc;
    unsigned long long *F;       // [3][n][W]
    unsigned long long *vis;     // [n][W]
    int32_t *qmark;              // [n] last level a vertex was queued for
    int32_t *queue;              // [2][n] entries of an even and of an odd level
    int32_t *vcnt, *qcnt;        // [4] vertices and queue entries of level d % 4
    unsigned long long *mfv;     // [4] sum of degrees of the level's vertices
    unsigned long long *dmu;     // [4] degrees of the vertices completed at the level
    int32_t *wq;                 // [4][8] work counters
    unsigned long long *far, *reach;  // [n] += sums of distances, number of sources
    Ctrl *ctrl;
    uint64_t limit_ns;
    double alpha;
    int dir;
    int32_t chunk;
    const int32_t *hv, *hfirst, *chunk_h;
    int32_t H, C;

    __device__ __forceinline__ Ctrl *status() const { return ctrl; }
};

// One warp's shared memory: a group's vertices.
template <int W> struct GroupBuf {
    unsigned long long t[32][W];  // bits a vertex waits for (bottom-up) or pushes (top-down)
    unsigned long long f[32][W];  // bits found so far
    int off[32];                  // first arc, less the arcs of the vertices before
    Hand hand;
};

// Lane L's vertex w (where `on`) joins level d+1 for the sources nb.
template <int W>
__device__ __forceinline__ void join(const LArgs &a, bool on, int w, int d, const Bits<W> &nb, const Bits<W> &act,
                                     BlockCnt *bc)
{
    bool full = on;
    unsigned dg = 0;
    if (on) {
        Bits<W> nv = load_bits<W>(a.vis + (size_t)w * W);
        int c = 0;
#pragma unroll
        for (int q = 0; q < W; ++q) {
            nv.w[q] |= nb.w[q];
            full &= nv.w[q] == act.w[q];
            c += __popcll(nb.w[q]);
        }
        store_bits<W>(a.vis + (size_t)w * W, nv);
        // one vertex, one lane, one batch at a time: additions that nobody waits for
        atomicAdd(a.far + w, (unsigned long long)c * (unsigned)(d + 1));
        atomicAdd(a.reach + w, (unsigned long long)c);
        dg = (unsigned)deg_of(a.rp, w);
    }
    const unsigned m = __ballot_sync(FULL, on);
    if (!m) return;
    unsigned long long df = dg, dd = full ? dg : 0;
    df = dev::group_sum<32>(df);
    dd = dev::group_sum<32>(dd);
    if ((threadIdx.x & 31) == 0) {
        atomicAdd(&bc->v, __popc(m));
        atomicAdd(&bc->mf, df);
        if (dd) atomicAdd(&bc->dmu, dd);
    }
}

template <int W> __global__ void __launch_bounds__(kThreads, 4) k_levels(LArgs a)
{
    __shared__ BlockCnt bc;
    __shared__ GroupBuf<W> bufs[kThreads / 32];
    GroupBuf<W> &st = bufs[threadIdx.x >> 5];
    const long long tid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const long long nthr = (long long)gridDim.x * blockDim.x;
    const int lane = threadIdx.x & 31;
    const size_t slab = (size_t)a.n * W;
    Bits<W> act;
#pragma unroll
    for (int q = 0; q < W; ++q) {
        const int left = a.nsrc - 64 * q;
        act.w[q] = left >= 64 ? ~0ull : (left <= 0 ? 0ull : ((1ull << left) - 1));
    }
    for (size_t i = tid; i < slab; i += nthr) {
        a.vis[i] = 0;
        a.F[i] = 0;
        a.F[slab + i] = 0;
    }
    for (long long i = tid; i < a.n; i += nthr) a.qmark[i] = -1;
    if (tid < 4 * 8) a.wq[tid] = 0;
    if (tid < 4) {
        a.vcnt[tid] = 0;
        a.qcnt[tid] = 0;
        a.mfv[tid] = 0;
        a.dmu[tid] = 0;
    }
    if (!dev::grid_barrier(a.ctrl, a.limit_ns)) return;
    if (tid < a.nsrc) {
        const int s = __ldg(a.src + tid);
        const unsigned long long bit = 1ull << (tid & 63);
        atomicOr(a.F + (size_t)s * W + (tid >> 6), bit);
        atomicOr(a.vis + (size_t)s * W + (tid >> 6), bit);
        a.queue[tid] = s;
        atomicAdd(a.mfv, (unsigned long long)deg_of(a.rp, s));
    }
    if (!dev::grid_barrier(a.ctrl, a.limit_ns)) return;

    long long mu = a.A, mf = (long long)__ldcg(a.mfv);
    int d = 0, td = 0, bu = 0, nq = min(a.nsrc, a.n);
    bool queued = a.nsrc <= a.n;  // else (a list with repetitions) level 0 is scanned
    for (;; ++d) {
        const int s1 = (d + 1) & 3, s2 = (d + 2) & 3;
        if (threadIdx.x == 0) {
            bc.v = 0;
            bc.mf = 0;
            bc.dmu = 0;
        }
        if (tid == 0) {
            a.vcnt[s2] = 0;
            a.qcnt[s2] = 0;
            a.mfv[s2] = 0;
            a.dmu[s2] = 0;
        }
        if (tid < 8) a.wq[s2 * 8 + tid] = 0;
        {
            unsigned long long *Fz = a.F + (size_t)((d + 2) % 3) * slab;
            for (size_t i = tid; i < slab; i += nthr) Fz[i] = 0;
        }
        __syncthreads();
        const unsigned long long *Fd = a.F + (size_t)(d % 3) * slab;
        unsigned long long *Fn = a.F + (size_t)((d + 1) % 3) * slab;
        int32_t *wq = a.wq + (d & 3) * 8;
        const bool use_bu = a.dir == NK_DIR_BOTTOM_UP ||
                            (a.dir == NK_DIR_AUTO && a.alpha * (double)mf > (double)mu);
        if (use_bu) {
            for_work(a, {nullptr, a.n}, wq + WQ_BU, st.hand, [&](bool on, int v, int beg, int dg, int chunk) {
                Bits<W> t;
                if (on) {
                    t = andnot<W>(act, load_bits<W>(a.vis + (size_t)v * W));
                    on = any_bits<W>(t);
                }
                if (!__any_sync(FULL, on)) return;
                Rows rows(on ? dg : 0);
                const int pos = rows.place();
                __syncwarp();
                if (pos >= 0) {
                    st.off[pos] = beg - rows.pre;
#pragma unroll
                    for (int q = 0; q < W; ++q) {
                        st.t[pos][q] = t.w[q];
                        st.f[pos][q] = 0;
                    }
                }
                __syncwarp();
                for (int base = 0; base < rows.total; base += 32) {
                    const int o = rows.owner(base);
                    Bits<W> m;
#pragma unroll
                    for (int q = 0; q < W; ++q) m.w[q] = 0;
                    if (base + lane < rows.total) {
                        // what the vertex still waits for (a bit another lane is just adding may
                        // be found twice, which changes nothing)
#pragma unroll
                        for (int q = 0; q < W; ++q) m.w[q] = st.t[o][q] & ~st.f[o][q];
                        if (any_bits<W>(m)) {
                            const int c = __ldg(a.col + st.off[o] + base + lane);
                            const Bits<W> fc = load_bits<W>(Fd + (size_t)c * W);
#pragma unroll
                            for (int q = 0; q < W; ++q) m.w[q] &= fc.w[q];
                        }
                    }
                    __syncwarp();  // the bits found so far are read before they change
                    if (!__any_sync(FULL, any_bits<W>(m))) continue;
                    if (__shfl_sync(FULL, o, 0) == __shfl_sync(FULL, o, 31)) {
                        // a window of one row: the lanes' bits joined in registers
#pragma unroll
                        for (int q = 0; q < W; ++q) {
                            const unsigned lo = __reduce_or_sync(FULL, (unsigned)m.w[q]);
                            const unsigned hi = __reduce_or_sync(FULL, (unsigned)(m.w[q] >> 32));
                            if (lane == q) st.f[o][q] |= (unsigned long long)hi << 32 | lo;
                        }
                    } else {
#pragma unroll
                        for (int q = 0; q < W; ++q) {
                            unsigned *f = reinterpret_cast<unsigned *>(&st.f[o][q]);
                            if ((unsigned)m.w[q]) atomicOr(f, (unsigned)m.w[q]);
                            if (m.w[q] >> 32) atomicOr(f + 1, (unsigned)(m.w[q] >> 32));
                        }
                    }
                    __syncwarp();
                }
                Bits<W> nb;
#pragma unroll
                for (int q = 0; q < W; ++q) nb.w[q] = pos >= 0 ? st.f[pos][q] : 0ull;
                const bool hit = any_bits<W>(nb);
                if (chunk >= 0) {
                    if (hit)
#pragma unroll
                        for (int q = 0; q < W; ++q)
                            if (nb.w[q]) atomicOr(Fn + (size_t)v * W + q, nb.w[q]);
                    return;
                }
                if (hit) store_bits<W>(Fn + (size_t)v * W, nb);
                join<W>(a, hit, v, d, nb, act, &bc);
            });
            if (a.H > 0) {
                if (!dev::grid_barrier(a.ctrl, a.limit_ns)) return;
                for (long long i0 = tid - lane; i0 < a.H; i0 += nthr) {
                    const bool in = i0 + lane < a.H;
                    const int h = in ? __ldg(a.hv + i0 + lane) : 0;
                    Bits<W> nb;
                    if (in) nb = load_bits<W>(Fn + (size_t)h * W);
                    join<W>(a, in && any_bits<W>(nb), h, d, nb, act, &bc);
                }
            }
            ++bu;
        } else {
            int32_t *qnext = a.queue + (size_t)((d + 1) & 1) * a.n;
            for_work(a, {queued ? a.queue + (size_t)(d & 1) * a.n : nullptr, nq}, wq + WQ_PUSH, st.hand,
                     [&](bool on, int v, int beg, int dg, int) {
                Bits<W> t;
                if (on) {
                    t = load_bits<W>(Fd + (size_t)v * W);
                    on = any_bits<W>(t);
                }
                Rows rows(on ? dg : 0);
                const int pos = rows.place();
                __syncwarp();
                if (pos >= 0) {
                    st.off[pos] = beg - rows.pre;
#pragma unroll
                    for (int q = 0; q < W; ++q) st.t[pos][q] = t.w[q];
                }
                __syncwarp();
                for (int base = 0; base < rows.total; base += 32) {
                    const int o = rows.owner(base);
                    if (base + lane >= rows.total) continue;
                    const int c = __ldg(a.col + st.off[o] + base + lane);
                    const Bits<W> vc = load_bits<W>(a.vis + (size_t)c * W);
                    bool any = false;
#pragma unroll
                    for (int q = 0; q < W; ++q) {
                        const unsigned long long m = st.t[o][q] & ~vc.w[q];
                        any |= m != 0;
                        if (m) atomicOr(Fn + (size_t)c * W + q, m);
                    }
                    if (any && __ldcg(a.qmark + c) != d + 1 && atomicExch(a.qmark + c, d + 1) != d + 1) {
                        cg::coalesced_group g = cg::coalesced_threads();
                        int at = 0;
                        if (g.thread_rank() == 0) at = atomicAdd(a.qcnt + s1, (int)g.size());
                        at = g.shfl(at, 0) + (int)g.thread_rank();
                        if (at < a.n) qnext[at] = c;  // always: a vertex is queued once per level
                    }
                }
            });
            if (!dev::grid_barrier(a.ctrl, a.limit_ns)) return;
            nq = min(__ldcg(a.qcnt + s1), a.n);
            for (long long i0 = tid - lane; i0 < nq; i0 += nthr) {
                bool in = i0 + lane < nq;
                const int w = in ? __ldcg(qnext + i0 + lane) : 0;
                if (in && (unsigned)w >= (unsigned)a.n) {
                    check_failed(a.status(), kErrCheck, 4, w);
                    in = false;
                }
                Bits<W> nb;
                if (in) nb = load_bits<W>(Fn + (size_t)w * W);
                join<W>(a, in, w, d, nb, act, &bc);
            }
            ++td;
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            if (bc.v) atomicAdd(a.vcnt + s1, bc.v);
            if (bc.mf) atomicAdd(a.mfv + s1, bc.mf);
            if (bc.dmu) atomicAdd(a.dmu + s1, bc.dmu);
        }
        if (!dev::grid_barrier(a.ctrl, a.limit_ns)) return;
        const int c = __ldcg(a.vcnt + s1);
        if (c == 0) break;
        queued = !use_bu;
        if (use_bu) nq = c;
        mu -= (long long)__ldcg(a.dmu + s1);
        mf = (long long)__ldcg(a.mfv + s1);
    }
    if (tid == 0) {
        a.ctrl->depth = d;
        a.ctrl->td_levels = td;
        a.ctrl->bu_levels = bu;
    }
}

enum { WS_BATCH = 5, WS_BCTRL = 6 };

template <int W>
int run_levels_w(nk_graph *g, const int32_t *d_src, int32_t k, const int32_t *d_count, const RunCfg &cfg, RunStats *st, cudaStream_t s)
{
    constexpr int B = 64 * W;
    Tmp osrc, okey;
    if (k > B) {  // similar sources share a batch and its bottom-up levels
        NK_TRY(osrc.alloc(sizeof(int32_t) * (size_t)k, s));
        NK_TRY(okey.alloc(sizeof(unsigned long long) * (size_t)k, s));
        NK_TRY(order_sources(g, d_src, k, d_count, okey.as<unsigned long long>(), osrc.as<int32_t>(), s));
        d_src = osrc.as<int32_t>();
    }
    HeavyView hw;
    NK_TRY(heavy_view(g, cfg.chunk, s, &hw));
    DevBuf *ws = scratch(cfg, g);
    const int nb = (k + B - 1) / B;
    NK_TRY(ws[WS_BCTRL].ensure(sizeof(Ctrl) * nb));
    const size_t n = (size_t)g->n;
    auto al = [](size_t x) { return (x + 255) & ~(size_t)255; };
    const size_t o_vis = al(3 * n * W * 8), o_mark = o_vis + al(n * W * 8), o_queue = o_mark + al(n * 4),
                 o_cnt = o_queue + al(2 * std::max<size_t>(n, B) * 4), bytes = o_cnt + 4 * (2 * 8 + 2 * 4 + 8 * 4);
    NK_TRY(ws[WS_BATCH].ensure(bytes));
    char *p = ws[WS_BATCH].as<char>();
    LArgs a{};
    a.n = g->n;
    a.A = g->A;
    a.rp = g->rp.as<int32_t>();
    a.col = g->col.as<int32_t>();
    a.F = reinterpret_cast<unsigned long long *>(p);
    a.vis = reinterpret_cast<unsigned long long *>(p + o_vis);
    a.qmark = reinterpret_cast<int32_t *>(p + o_mark);
    a.queue = reinterpret_cast<int32_t *>(p + o_queue);
    a.mfv = reinterpret_cast<unsigned long long *>(p + o_cnt);
    a.dmu = a.mfv + 4;
    a.vcnt = reinterpret_cast<int32_t *>(a.dmu + 4);
    a.qcnt = a.vcnt + 4;
    a.wq = a.qcnt + 4;
    a.far = cfg.far;
    a.reach = cfg.reach;
    a.limit_ns = cfg.limit_ns ? cfg.limit_ns : wait_limit_ns();
    a.alpha = cfg.alpha > 0 ? cfg.alpha : 1.0;
    a.dir = cfg.direction;
    a.chunk = hw.chunk;
    a.hv = hw.hv;
    a.hfirst = hw.hfirst;
    a.chunk_h = hw.chunk_h;
    a.H = hw.H;
    a.C = hw.C;
    static const int bps = [] {
        int v = 0;
        return cudaOccupancyMaxActiveBlocksPerMultiprocessor(&v, k_levels<W>, kThreads, 0) == cudaSuccess ? v : 0;
    }();
    if (bps < 1) return set_error(NK_ERR_CUDA, "closeness kernel cannot be resident");
    int grid = std::max(1, bps * num_sms() / std::max(1, cfg.grid_div));
    if (cfg.grid_ctas > 0) grid = std::min(grid, cfg.grid_ctas);
    Ctrl *ctrls = ws[WS_BCTRL].as<Ctrl>();
    NK_CUDA(cudaMemsetAsync(ctrls, 0, sizeof(Ctrl) * nb, s));
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    if (cfg.time_kernels) {
        NK_CUDA(cudaEventCreate(&e0));
        NK_CUDA(cudaEventCreate(&e1));
        NK_CUDA(cudaEventRecord(e0, s));
    }
    for (int bi = 0; bi < nb; ++bi) {
        a.src = d_src + (size_t)bi * B;
        a.nsrc = std::min(B, k - bi * B);
        a.ctrl = ctrls + bi;
        void *args[] = {&a};
        NK_CUDA(cudaLaunchCooperativeKernel((const void *)k_levels<W>, dim3(grid), dim3(kThreads), args, 0, s));
        ::nk::count_launch();
    }
    if (cfg.time_kernels) NK_CUDA(cudaEventRecord(e1, s));
    std::vector<Ctrl> h(nb);
    NK_CUDA(cudaMemcpyAsync(h.data(), ctrls, sizeof(Ctrl) * nb, cudaMemcpyDeviceToHost, s));
    const int rc = host_wait(s, nb, a.limit_ns);
    if (rc == NK_OK && cfg.time_kernels) {
        float ms = 0;
        cudaEventElapsedTime(&ms, e0, e1);
        st->kernel_ms += ms;
    }
    if (e0) cudaEventDestroy(e0);
    if (e1) cudaEventDestroy(e1);
    NK_TRY(rc);
    st->tpv = 32;
    st->launches += nb;
    st->kernel_launches += nb;
    st->alpha = a.alpha;
    for (const Ctrl &c : h) {
        if (c.err == NK_ERR_TIMEOUT)
            return set_error(NK_ERR_TIMEOUT, "closeness sweep aborted: a bounded device-side wait or phase ran out (check %d, value %d)", c.where, c.bad_id);
        if (c.err) return set_error(NK_ERR_CUDA, "closeness sweep aborted: device range check %d failed (value %d)", c.where, c.bad_id);
        st->max_depth = std::max(st->max_depth, c.depth);
        st->td_levels += c.td_levels;
        st->bu_levels += c.bu_levels;
    }
    return NK_OK;
}

}  // namespace

int run_levels(nk_graph *g, const int32_t *d_src, int32_t k, const RunCfg &cfg, RunStats *st, cudaStream_t s)
{
    Tmp list, count;
    NK_TRY(compact_list(g, &d_src, &k, list, count, s));
    // without a width from the caller: the narrowest that takes all sources (with arcs) in one launch,
    // up to 256
    const int B = cfg.batch ? cfg.batch : k > 128 ? 256 : k > 64 ? 128 : 64;
    st->mode = NK_MODE_BATCHED;
    st->batch = B;
    if (k == 0) return NK_OK;
    switch (B) {
    case 64: return run_levels_w<1>(g, d_src, k, count.as<int32_t>(), cfg, st, s);
    case 128: return run_levels_w<2>(g, d_src, k, count.as<int32_t>(), cfg, st, s);
    case 256: return run_levels_w<4>(g, d_src, k, count.as<int32_t>(), cfg, st, s);
    default: return set_error(NK_ERR_ARG, "batch must be 64, 128 or 256 (got %d)", B);
    }
}

}  // namespace nk
