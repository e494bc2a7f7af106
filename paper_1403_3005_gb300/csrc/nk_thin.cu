// Betweenness for a handful of sources: up to 8 per batch, one byte of source bits per vertex and
// level, rows of 8 entries (64 bytes) of path counts or dependencies per vertex.  The 64-source
// sweep of nk_batch.cu spends a warp's instruction on every neighbour however few of its slots are
// in use; here 8 lanes are a neighbour's 8 sources, and the four parts of a warp work on four
// vertices (rows of up to kShortRow arcs) or on four stretches of one row at a time.
//
// Same steps as nk_batch.cu: direction-optimising BFS levels, kept as slabs of n bytes; top-down
// levels push bits and queue the new vertices, then those pull their path counts; bottom-up levels
// pull at every vertex with unvisited sources.  Backward, deepest level first, a vertex pulls psi =
// (1 + delta) / sigma of its successors; psi replaces sigma in the row.  Path counts are 64-bit
// throughout (an overflow is reported).  Rows longer than the hub chunk are summed from per-chunk
// partials in chunk order, so results do not depend on timing.  Several batches run side by side,
// one per row of the grid.  Sums of psi, and of a vertex's dependencies over its sources, are rounded once
// (ff_sum): added step by step in double-single, scores of 2 to 15 sources were up to twice as far
// from FP64 as the per-source form's (ER 112063, degree 22, 13 sources, 2-norm: 3.5e-15 against 1.5e-15,
// now 5e-16).  It costs 2 to 3 % (R-MAT 20, 8 sources, 3.37 -> 3.44 ms); FP64 sums are as exact and cost
// 10 to 17 %.
//
// What bounds it: the latency of the dependent reads column id -> level byte -> row entry (48
// registers for 40 warps an SM: 5 blocks 3.4 ms on R-MAT 20 with 8 sources, 4 3.6, 6 3.4, R-MAT 22
// 12.1, 13.2, 13.8), and on R-MAT graphs the instructions per arc: reading only a part's relevant
// arcs, 4 at a time, instead of 8 of 8 took R-MAT 20 from 3.3 to 3.1 ms.
#include <cooperative_groups.h>

#include <algorithm>
#include <climits>
#include <vector>

#include "nk_device.cuh"
#include "nk_internal.h"
#include "nk_sweep.cuh"

namespace cg = cooperative_groups;

namespace nk {
namespace {

using namespace sweep;

constexpr int kThreads = 256;
constexpr int kT = 8;            // sources per batch
constexpr int kShortRow = 32;    // arcs up to which a row is one part's work
constexpr int kErrDepth = 100;   // internal status: BFS deeper than the level slabs
constexpr int kStartLevels = 48;

struct TArgs {
    int32_t n;
    int64_t A;
    const int32_t *rp, *col;
    const int32_t *src;
    int32_t nsrc, b0;
    int32_t lcap;                // levels 0..lcap may be non-empty; slabs 0..lcap+1
    int64_t nw8;                 // bytes of a slab of source bits (n rounded up to 16)
    unsigned char *F;            // [lcap+2][teams][nw8]
    unsigned char *vis;          // [teams][nw8]
    unsigned long long *sp;      // [teams][n][8] sigma, then psi
    int32_t *qmark;              // [teams][n]
    int32_t *queue;              // [teams][2][n] entries of an even and of an odd level
    int32_t *vcnt, *qcnt;        // [teams][lcap+3]
    unsigned long long *mfv, *dmu;  // [teams][lcap+3]
    int32_t *wq;                 // [teams][lcap+3][8]
    unsigned long long *part;    // [teams][C][8] a hub chunk's path counts, or its psi (double)
    double *scores;              // [teams][n]
    Ctrl *ctrl;
    uint64_t limit_ns;
    double alpha;
    int dir;
    int32_t chunk;
    const int32_t *hv, *hfirst, *chunk_h;
    int32_t H, C;

    __device__ __forceinline__ Ctrl *status() const { return ctrl + b0 + blockIdx.y; }
    __device__ __forceinline__ unsigned char *level(int d) const { return F + ((size_t)d * gridDim.y + blockIdx.y) * nw8; }
};

// One warp's shared memory: the short rows of a group.
struct ThinBuf {
    int v[32], beg[32], dg[32];
    unsigned char t[32], nb[32];
    Hand hand;
};

// The sum over the arcs [beg, beg + dg) of the entry `slot` of the neighbours' rows whose bit is set
// in Fsel and in t, over lanes of a part (stride 8) or, with `parts` = 4, of all parts of the warp
// (each takes every fourth stretch of 8 arcs).  Lane `slot` of a part reads one arc's column id and
// bits for the part, then the part reads the 8 arcs' entries together.  All lanes of the warp call
// it; a part without work has dg = 0.
template <bool PSI>
__device__ __forceinline__ void thin_gather(const TArgs &a, int beg, int dg, unsigned t, const unsigned char *Fsel,
                                            int parts, unsigned long long &acc, dev::ff_sum &facc, bool &ovf)
{
    const int lane = threadIdx.x & 31, slot = lane & 7;
    const unsigned long long *rows = a.sp + (size_t)blockIdx.y * a.n * kT + slot;
    const int first = parts == 1 ? 0 : (lane >> 3) * 8, step = 8 * parts;
    const int longest = __reduce_max_sync(FULL, dg);
    for (int base = first; base - first < longest; base += step) {  // the same number of steps for every lane
        int c = 0;
        unsigned f = 0;
        if (base + slot < dg) {
            c = __ldg(a.col + beg + base + slot);
            f = __ldcg(Fsel + c) & t;
        }
        // the part's relevant arcs, four at a time
        unsigned m = (__ballot_sync(FULL, f != 0) >> (lane & 24)) & 0xffu;
        for (int left = __reduce_max_sync(FULL, __popc(m)); left > 0; left -= 4) {
            unsigned long long x[4];
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const int i = __ffs(m) - 1;  // -1: none left in this part
                m &= m - 1;
                const int ci = __shfl_sync(FULL, c, i & 7, 8);
                const unsigned fi = __shfl_sync(FULL, f, i & 7, 8);
                x[r] = 0;
                if (i >= 0 && ((fi >> slot) & 1u)) x[r] = __ldcg(rows + (size_t)ci * kT);
            }
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                if constexpr (PSI) {
                    if (r < left) facc.add(dev::ff_unpack(x[r]));  // uniform
                } else {
                    acc += x[r];
                    ovf |= acc < x[r];
                }
            }
        }
    }
    if (parts > 1) {
#pragma unroll
        for (int o = 8; o < 32; o <<= 1) {
            if constexpr (PSI) {
                facc.join(o);
            } else {
                const unsigned long long y = __shfl_xor_sync(FULL, acc, o);
                acc += y;
                ovf |= acc < y;
            }
        }
    }
}

__global__ void __launch_bounds__(kThreads, 5) k_thin(TArgs a)
{
    __shared__ BlockCnt bc;
    __shared__ struct {              // kept by thread 0 from level to level
        long long mu, mf;            // arcs of vertices not yet visited by every source, of the level's
        int nq, td, bu;
    } lv;
    __shared__ ThinBuf bufs[kThreads / 32];
    ThinBuf &st = bufs[threadIdx.x >> 5];
    const long long tid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const long long nthr = (long long)gridDim.x * blockDim.x;
    const int lane = threadIdx.x & 31, slot = lane & 7, part = lane >> 3;
    const int nsrc = min(kT, a.nsrc - (a.b0 + (int)blockIdx.y) * kT);
    const unsigned act = (1u << nsrc) - 1u;
    const size_t tn = (size_t)blockIdx.y * a.n;
    const size_t lv0 = (size_t)blockIdx.y * (a.lcap + 3);
    unsigned char *vis = a.vis + (size_t)blockIdx.y * a.nw8;
    unsigned long long *rows = a.sp + tn * kT;
    bool ovf = false;

    auto clear = [&](unsigned char *p) {
        for (long long i = tid; i < a.nw8 / 16; i += nthr) reinterpret_cast<uint4 *>(p)[i] = make_uint4(0, 0, 0, 0);
    };
    clear(vis);
    clear(a.level(0));
    clear(a.level(1));
    for (long long i = tid; i < a.n; i += nthr) a.qmark[tn + i] = -1;
    if (tid < 3 * 8) a.wq[lv0 * 8 + tid] = 0;
    if (tid < 3) {
        a.vcnt[lv0 + tid] = 0;
        a.qcnt[lv0 + tid] = 0;
        a.mfv[lv0 + tid] = 0;
        a.dmu[lv0 + tid] = 0;
    }
    if (!dev::grid_barrier(a.status(), a.limit_ns)) return;
    auto set_bits = [](unsigned char *p, size_t v, unsigned m) {
        atomicOr(reinterpret_cast<unsigned *>(p) + (v >> 2), m << (8 * (v & 3)));
    };
    if (tid < nsrc) {
        const int s = __ldg(a.src + (size_t)(a.b0 + blockIdx.y) * kT + tid);
        set_bits(a.level(0), s, 1u << tid);
        set_bits(vis, s, 1u << tid);
        rows[(size_t)s * kT + tid] = 1ull;
        atomicAdd(a.mfv + lv0, (unsigned long long)deg_of(a.rp, s));
    }
    if (!dev::grid_barrier(a.status(), a.limit_ns)) return;

    // Lane L's vertex w (where `on`) joins level d + 1 for the sources nb.
    auto join = [&](bool on, int w, unsigned nb, unsigned char *Fn) {
        unsigned long long df = 0, dd = 0;
        if (on) {
            const unsigned nv = __ldcg(vis + w) | nb;
            vis[w] = (unsigned char)nv;
            Fn[w] = (unsigned char)nb;
            df = (unsigned)deg_of(a.rp, w);
            if (nv == act) dd = df;
        }
        const unsigned m = __ballot_sync(FULL, on);
        if (!m) return;
        df = dev::group_sum<32>(df);
        dd = dev::group_sum<32>(dd);
        if (lane == 0) {
            atomicAdd(&bc.v, __popc(m));
            atomicAdd(&bc.mf, df);
            if (dd) atomicAdd(&bc.dmu, dd);
        }
    };
    // The group's members (lanes `on`, with their row and bits t): short rows are listed and taken
    // four at a time by body(o, v, beg, dg, t, 1), longer ones one by one by body(o, ..., 4), where o
    // is the member's lane.
    auto each_row = [&](bool on, int v, int beg, int dg, unsigned t, auto body) {
        const unsigned shrt = __ballot_sync(FULL, on && dg <= kShortRow);
        __syncwarp();
        if (on) {
            st.v[lane] = v;
            st.beg[lane] = beg;
            st.dg[lane] = dg;
            st.t[lane] = (unsigned char)t;
        }
        __syncwarp();
        for (unsigned m = shrt; m;) {
            int o = -1;  // the part's member: the part-th set bit of m
#pragma unroll
            for (int p = 0; p < 4; ++p) {
                const int b = __ffs(m) - 1;
                if (p == part) o = b;
                m &= m - 1;  // 0 stays 0
            }
            const bool in = o >= 0;
            const int i = in ? o : 0;
            body(o, in ? st.v[i] : 0, in ? st.beg[i] : 0, in ? st.dg[i] : 0, in ? (unsigned)st.t[i] : 0u, 1);
        }
        for (unsigned m = __ballot_sync(FULL, on && dg > kShortRow); m; m &= m - 1) {
            const int o = __ffs(m) - 1;
            body(o, st.v[o], st.beg[o], st.dg[o], (unsigned)st.t[o], 4);
        }
    };

    if (threadIdx.x == 0) {
        lv.mu = a.A;
        lv.mf = (long long)__ldcg(a.mfv + lv0);
        lv.nq = lv.td = lv.bu = 0;
    }
    int d = 0;
    bool queued = false;  // level 0 (at most 8 vertices) is scanned
    for (;;) {
        if (threadIdx.x == 0) {
            bc.v = 0;
            bc.mf = 0;
            bc.dmu = 0;
        }
        if (tid == 0) {
            a.vcnt[lv0 + d + 2] = 0;
            a.qcnt[lv0 + d + 2] = 0;
            a.mfv[lv0 + d + 2] = 0;
            a.dmu[lv0 + d + 2] = 0;
        }
        if (tid < 8) a.wq[(lv0 + d + 2) * 8 + tid] = 0;
        clear(a.level(d + 2));
        __syncthreads();
        const unsigned char *Fd = a.level(d);
        unsigned char *Fn = a.level(d + 1);
        int32_t *wq = a.wq + (lv0 + d) * 8;
        int32_t *qnext = a.queue + (2 * (size_t)blockIdx.y + ((d + 1) & 1)) * a.n;
        const bool use_bu = a.dir == NK_DIR_BOTTOM_UP ||
                            (a.dir == NK_DIR_AUTO && a.alpha * (double)lv.mf > (double)lv.mu);
        int nq1 = 0;
        if (!use_bu) {
            const int32_t *qd = a.queue + (2 * (size_t)blockIdx.y + (d & 1)) * a.n;
            for_work(a, {queued ? qd : nullptr, lv.nq}, wq + WQ_PUSH, st.hand, [&](bool on, int v, int beg, int dg, int) {
                unsigned t = 0;
                if (on) t = __ldcg(Fd + v);
                on = t != 0;
                Rows rws(on ? dg : 0);
                const int pos = rws.place();
                __syncwarp();
                if (pos >= 0) {
                    st.beg[pos] = beg - rws.pre;
                    st.t[pos] = (unsigned char)t;
                }
                __syncwarp();
                for (int base = 0; base < rws.total; base += 32) {
                    const int o = rws.owner(base);
                    if (base + lane >= rws.total) continue;
                    const int c = __ldg(a.col + st.beg[o] + base + lane);
                    const unsigned m = st.t[o] & ~(unsigned)__ldcg(vis + c);
                    if (!m) continue;
                    set_bits(Fn, c, m);
                    if (__ldcg(a.qmark + tn + c) != d + 1 && atomicExch(a.qmark + tn + c, d + 1) != d + 1) {
                        cg::coalesced_group g = cg::coalesced_threads();
                        int at = 0;
                        if (g.thread_rank() == 0) at = atomicAdd(a.qcnt + lv0 + d + 1, (int)g.size());
                        at = g.shfl(at, 0) + (int)g.thread_rank();
                        if (at < a.n) qnext[at] = c;  // always: a vertex is queued once per level
                    }
                }
            });
            if (!dev::grid_barrier(a.status(), a.limit_ns)) return;
            nq1 = __ldcg(a.qcnt + lv0 + d + 1);
        }
        // pull sigma from level d
        for_work(a, use_bu ? Level{nullptr, a.n} : Level{qnext, nq1}, wq + (use_bu ? WQ_BU : WQ_PULL), st.hand,
                 [&](bool on, int v, int beg, int dg, int chunk) {
            unsigned t = 0;
            if (on) t = use_bu ? act & ~(unsigned)__ldcg(vis + v) : (unsigned)__ldcg(Fn + v);
            on = t != 0;
            if (!__any_sync(FULL, on)) return;
            if (chunk >= 0) {
                unsigned long long acc = 0;
                dev::ff_sum facc;
                thin_gather<false>(a, beg, dg, __shfl_sync(FULL, t, 0), Fd, 4, acc, facc, ovf);
                if (part == 0) a.part[((size_t)blockIdx.y * a.C + chunk) * kT + slot] = acc;
                return;
            }
            unsigned done = 0;
            each_row(on, v, beg, dg, t, [&](int o, int w, int b, int g, unsigned tw, int parts) {
                unsigned long long acc = 0;
                dev::ff_sum facc;
                thin_gather<false>(a, b, g, tw, Fd, parts, acc, facc, ovf);
                const bool mine = o >= 0 && (parts == 1 || part == 0) && acc != 0;
                if (mine) rows[(size_t)w * kT + slot] = acc;
                const unsigned got = __ballot_sync(FULL, mine);
                if (o >= 0 && (parts == 1 || part == 0) && slot == 0) st.nb[o] = (unsigned char)(got >> (part * 8));
                done |= __reduce_or_sync(FULL, o >= 0 ? 1u << o : 0u);
            });
            __syncwarp();
            const unsigned nb = (done >> lane) & 1u ? (unsigned)st.nb[lane] : 0u;
            join(nb != 0, v, nb, Fn);
        });
        if (a.H > 0) {
            if (!dev::grid_barrier(a.status(), a.limit_ns)) return;
            for_heavy(a, [&](int, int h, int c0, int c1) {
                const unsigned t = use_bu ? act & ~(unsigned)__ldcg(vis + h) : (unsigned)__ldcg(Fn + h);
                if (!t) return;
                unsigned long long acc = 0;
                for (int c = c0 + part; c < c1; c += 4) {  // integer sums: any order
                    const unsigned long long x = __ldcg(a.part + ((size_t)blockIdx.y * a.C + c) * kT + slot);
                    acc += x;
                    ovf |= acc < x;
                }
#pragma unroll
                for (int o = 8; o < 32; o <<= 1) {
                    const unsigned long long y = __shfl_xor_sync(FULL, acc, o);
                    acc += y;
                    ovf |= acc < y;
                }
                const unsigned nb = __ballot_sync(FULL, acc != 0) & 0xffu;
                if (part == 0 && acc != 0) rows[(size_t)h * kT + slot] = acc;
                join(lane == 0 && nb != 0, h, nb, Fn);
            });
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            if (bc.v) atomicAdd(a.vcnt + lv0 + d + 1, bc.v);
            if (bc.mf) atomicAdd(a.mfv + lv0 + d + 1, bc.mf);
            if (bc.dmu) atomicAdd(a.dmu + lv0 + d + 1, bc.dmu);
        }
        if (!dev::grid_barrier(a.status(), a.limit_ns)) return;
        const int c = __ldcg(a.vcnt + lv0 + d + 1);
        if (threadIdx.x == 0) {
            use_bu ? ++lv.bu : ++lv.td;
            lv.nq = use_bu ? c : nq1;
            lv.mu -= (long long)__ldcg(a.dmu + lv0 + d + 1);
            lv.mf = (long long)__ldcg(a.mfv + lv0 + d + 1);
        }
        queued = !use_bu;
        ++d;
        if (c == 0) break;
        if (d + 1 > a.lcap) {
            if (tid == 0) atomicCAS(&a.status()->err, 0, kErrDepth);
            return;
        }
    }
    const int D = d - 1;
    if (tid == 0) {
        a.status()->depth = D;
        a.status()->td_levels = lv.td;
        a.status()->bu_levels = lv.bu;
    }
    if (ovf) atomicOr(&a.status()->ovf, 1);

    // backward: psi and delta of vertex v from its successor sums (the lane's slot), delta summed
    // over the part's 8 lanes into the score; one warp adds to a vertex's score per level
    auto finish = [&](bool in, int v, const dev::ff_sum &acc) {
        dev::ff_sum delta;
        if (in) {
            const dev::ff s = dev::ff_from_u64(__ldcg(rows + (size_t)v * kT + slot));
            rows[(size_t)v * kT + slot] = dev::ff_pack(dev::ff_add(dev::ff_rcp(s), acc.value()));
            delta = acc.times(s);
        }
#pragma unroll
        for (int o = 1; o < kT; o <<= 1) delta.join(o);
        if (slot == 0 && delta.s != 0.0f) atomicAdd(a.scores + tn + v, delta.to_double());
    };
    for (int l = D; l >= 1; --l) {
        const unsigned char *Fl = a.level(l), *Fs = a.level(l + 1);
        // bottom-up and top-down levels alike are found by a scan of their bytes
        for_work(a, {nullptr, __ldcg(a.vcnt + lv0 + l)}, a.wq + (lv0 + l) * 8 + WQ_BACK, st.hand,
                 [&](bool on, int v, int beg, int dg, int chunk) {
            unsigned t = 0;
            if (on) t = __ldcg(Fl + v);
            on = t != 0;
            if (!__any_sync(FULL, on)) return;
            unsigned long long acc = 0;
            bool dummy = false;
            if (chunk >= 0) {
                dev::ff_sum facc;
                thin_gather<true>(a, beg, dg, __shfl_sync(FULL, t, 0), Fs, 4, acc, facc, dummy);
                if (part == 0) a.part[((size_t)blockIdx.y * a.C + chunk) * kT + slot] = (unsigned long long)__double_as_longlong(facc.to_double());
                return;
            }
            each_row(on, v, beg, dg, t, [&](int o, int w, int b, int g, unsigned tw, int parts) {
                dev::ff_sum facc;
                thin_gather<true>(a, b, g, tw, Fs, parts, acc, facc, dummy);
                finish(o >= 0 && (parts == 1 || part == 0) && ((tw >> slot) & 1u), w, facc);
            });
        });
        if (a.H > 0) {
            if (!dev::grid_barrier(a.status(), a.limit_ns)) return;
            for_heavy(a, [&](int, int h, int c0, int c1) {
                const unsigned t = __ldcg(Fl + h);
                if (!t) return;
                double facc = 0.0;
                for (int c = c0 + part; c < c1; c += 4)
                    facc += __longlong_as_double((long long)__ldcg(a.part + ((size_t)blockIdx.y * a.C + c) * kT + slot));
#pragma unroll
                for (int o = 8; o < 32; o <<= 1) facc += __shfl_xor_sync(FULL, facc, o);
                finish(part == 0 && ((t >> slot) & 1u), h, dev::ff_sum(facc));
            });
        }
        if (!dev::grid_barrier(a.status(), a.limit_ns)) return;
    }
}

enum { WS_BATCH = 5, WS_BCTRL = 6 };

}  // namespace

int run_thin(nk_graph *g, const int32_t *d_src, int32_t k, double *d_scores, const RunCfg &cfg, RunStats *st,
             cudaStream_t s)
{
    Tmp csrc, ccnt;
    NK_TRY(compact_list(g, &d_src, &k, csrc, ccnt, s));
    st->mode = NK_MODE_BATCHED;
    st->batch = kT;
    if (k == 0) return NK_OK;
    HeavyView hw;
    NK_TRY(heavy_view(g, cfg.chunk, s, &hw));
    // a single source, and two or three on large graphs most of whose arcs are hubs', go one by one: a
    // hub's chunk then is a warp's for one source, without the parts.  Per-source against 8 at once, ms,
    // for 1, 2, 3, 4, 8 sources: ER 200003 0.41 / 0.57, 0.74 / 0.64, 1.0 / 0.70, ..., 2.7 / 0.82; BA 10^6 1.1 /
    // 1.4, 2.1 / 1.8, ..., 8.2 / 2.3; R-MAT 16 0.38 / 0.61, 0.71 / 0.64, 1.0 / 0.64; R-MAT 18 0.53 / 0.91, 1.1 / 1.1,
    // 1.6 / 1.2; R-MAT 20 1.0 / 2.4, 2.0 / 2.6, 3.3 / 3.0, 4.4 / 3.0, 7.8 / 3.4; R-MAT 22 3.0 / 7.4, 5.1 / 8.0, 8.5 / 9.5,
    // 11.6 / 9.7, 21.7 / 12.2
    const bool hubs = (int64_t)hw.C * hw.chunk > g->A / 4;
    RunCfg pc = cfg;  // of the per-source form
    pc.compacted = true;
    if (k == 1 || (hubs && ((k == 2 && g->A >= (4 << 20)) || (k == 3 && g->A >= (64 << 20)))))
        return run_per_source(g, d_src, k, d_scores, pc, st, s);
    DevBuf *ws = scratch(cfg, g);
    const int nb = (k + kT - 1) / kT;
    NK_TRY(ws[WS_BCTRL].ensure(sizeof(Ctrl) * nb));
    static const int bps = [] {
        int v = 0;
        return cudaOccupancyMaxActiveBlocksPerMultiprocessor(&v, k_thin, kThreads, 0) == cudaSuccess ? v : 0;
    }();
    if (bps < 1) return set_error(NK_ERR_CUDA, "sweep kernel cannot be resident");
    int grid = std::max(1, bps * num_sms() / std::max(1, cfg.grid_div));
    if (cfg.grid_ctas > 0) grid = std::min(grid, cfg.grid_ctas);
    const int teams = std::min(std::min(nb, 4), grid);
    const size_t n = (size_t)g->n;
    auto al = [](size_t x) { return (x + 255) & ~(size_t)255; };
    Ctrl *ctrls = ws[WS_BCTRL].as<Ctrl>();
    std::vector<int> todo(nb);
    for (int i = 0; i < nb; ++i) todo[i] = i;
    // level slabs: 48 at first; deeper searches run again with those that an eighth of the free memory,
    // 8 GB at most, holds for the batches side by side together
    size_t free_b = 0, total_b = 0;
    cudaMemGetInfo(&free_b, &total_b);
    const size_t slabs = std::min<size_t>(free_b / 8, (size_t)8 << 30) / std::max<size_t>(n, 1), deepest = std::max<size_t>(n, 4);
    int lcap = (int)std::min<size_t>(deepest, kStartLevels), side = teams;
    for (;;) {
        TArgs a{};
        a.nw8 = (int64_t)((n + 15) / 16 * 16);
        const size_t lv = (size_t)(lcap + 3) * side;
        const size_t o_vis = al((size_t)(lcap + 2) * side * a.nw8), o_sp = o_vis + al(side * (size_t)a.nw8),
                     o_mark = o_sp + al(n * kT * 8 * side), o_queue = o_mark + al(n * 4 * side),
                     o_cnt = o_queue + al(2 * n * 4 * side), o_part = o_cnt + al(lv * (2 * 8 + 2 * 4 + 8 * 4)),
                     bytes = o_part + al((size_t)std::max(hw.C, 1) * kT * 8 * side);
        NK_TRY(ws[WS_BATCH].ensure(bytes));
        char *p = ws[WS_BATCH].as<char>();
        a.n = g->n;
        a.A = g->A;
        a.rp = g->rp.as<int32_t>();
        a.col = g->col.as<int32_t>();
        a.src = d_src;
        a.nsrc = k;
        a.lcap = lcap;
        a.F = reinterpret_cast<unsigned char *>(p);
        a.vis = reinterpret_cast<unsigned char *>(p + o_vis);
        a.sp = reinterpret_cast<unsigned long long *>(p + o_sp);
        a.qmark = reinterpret_cast<int32_t *>(p + o_mark);
        a.queue = reinterpret_cast<int32_t *>(p + o_queue);
        a.mfv = reinterpret_cast<unsigned long long *>(p + o_cnt);
        a.dmu = a.mfv + lv;
        a.vcnt = reinterpret_cast<int32_t *>(a.dmu + lv);
        a.qcnt = a.vcnt + lv;
        a.wq = a.qcnt + lv;
        a.part = reinterpret_cast<unsigned long long *>(p + o_part);
        a.ctrl = ctrls;
        a.limit_ns = cfg.limit_ns ? cfg.limit_ns : wait_limit_ns();
        a.alpha = cfg.alpha > 0 ? cfg.alpha : 1.0;
        a.dir = cfg.direction;
        a.chunk = hw.chunk;
        a.hv = hw.hv;
        a.hfirst = hw.hfirst;
        a.chunk_h = hw.chunk_h;
        a.H = hw.H;
        a.C = hw.C;
        a.scores = d_scores;
        Tmp outs;
        if (side > 1) {
            NK_TRY(outs.alloc(sizeof(double) * n * side, s));
            NK_CUDA(cudaMemsetAsync(outs.p, 0, sizeof(double) * n * side, s));
            a.scores = outs.as<double>();
        }
        NK_CUDA(cudaMemsetAsync(ctrls, 0, sizeof(Ctrl) * nb, s));
        cudaEvent_t e0 = nullptr, e1 = nullptr;
        if (cfg.time_kernels) {
            NK_CUDA(cudaEventCreate(&e0));
            NK_CUDA(cudaEventCreate(&e1));
            NK_CUDA(cudaEventRecord(e0, s));
        }
        for (size_t t = 0; t < todo.size(); t += side) {
            a.b0 = todo[t];
            const int now = std::min<int>(side, (int)(todo.size() - t));
            // a small graph's barriers get dearer with every block (as in nk_batch.cu)
            const int ctas = std::min(grid / now, std::max(128, g->n / 64));
            void *args[] = {&a};
            NK_CUDA(cudaLaunchCooperativeKernel((const void *)k_thin, dim3(ctas, now), dim3(kThreads), args, 0, s));
            ::nk::count_launch();
        }
        if (side > 1) NK_TRY(add_vectors(outs.as<double>(), side, (int64_t)n, d_scores, s));
        if (cfg.time_kernels) NK_CUDA(cudaEventRecord(e1, s));
        std::vector<Ctrl> h(nb);
        NK_CUDA(cudaMemcpyAsync(h.data(), ctrls, sizeof(Ctrl) * nb, cudaMemcpyDeviceToHost, s));
        const int rc = host_wait(s, (int64_t)todo.size(), a.limit_ns);
        if (rc == NK_OK && cfg.time_kernels) {
            float ms = 0;
            cudaEventElapsedTime(&ms, e0, e1);
            st->kernel_ms += ms;
        }
        if (e0) cudaEventDestroy(e0);
        if (e1) cudaEventDestroy(e1);
        NK_TRY(rc);
        st->tpv = 8;
        st->launches += (int64_t)todo.size();
        st->kernel_launches += ((int64_t)todo.size() + side - 1) / side;
        st->alpha = a.alpha;
        std::vector<int> deep;
        bool ovf = false;
        for (int bi : todo) {
            const Ctrl &c = h[bi];
            if (c.err == NK_ERR_TIMEOUT)
                return set_error(NK_ERR_TIMEOUT, "sweep aborted: a bounded device-side wait or phase ran out (check %d, value %d)", c.where, c.bad_id);
            if (c.err == kErrDepth) deep.push_back(bi);
            else if (c.err) return set_error(NK_ERR_CUDA, "sweep aborted: device range check %d failed (value %d)", c.where, c.bad_id);
            ovf |= c.ovf != 0;
            st->max_depth = std::max(st->max_depth, c.depth);
            st->td_levels += c.td_levels;
            st->bu_levels += c.bu_levels;
        }
        if (ovf) return set_error(NK_ERR_OVERFLOW, "a shortest-path count exceeded 2^64 - 1");
        if (deep.empty()) return NK_OK;
        side = (int)deep.size() == nb ? teams : 1;  // reruns of some of the batches go one by one
        const int lmax = (int)std::min(deepest, slabs / side);
        if (lcap < lmax) {
            todo = deep;
            lcap = lmax;
            continue;
        }
        // deeper than any level cap: the per-source form takes these sources
        for (int bi : deep)
            NK_TRY(run_per_source(g, d_src + (size_t)bi * kT, std::min(kT, k - bi * kT), d_scores, pc, st, s));
        return NK_OK;
    }
}

}  // namespace nk
