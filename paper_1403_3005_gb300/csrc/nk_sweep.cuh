// Parts shared by the kernels that sweep a graph level by level for a batch of sources: bitsets
// of W 64-bit words (one bit per source), the hand-out of a phase's work to warps, and the walk
// over the concatenated arcs of a group of vertices.  `Args` is a kernel's argument structure;
// the members used here are n, A, rp, limit_ns, the chunk table (chunk, hv, hfirst, chunk_h, H, C)
// and status(), the control words of the block's sweep.  The warps that share a sweep are those of gridDim.x blocks (a team, blockIdx.y).
#pragma once

#include "nk_device.cuh"
#include "nk_internal.h"

namespace nk {
namespace sweep {

constexpr unsigned FULL = 0xffffffffu;
constexpr int kErrCheck = 101;       // internal status: a device-side range check failed
constexpr int kGrabV = 32;           // most vertices a warp takes at a time (one per lane)
constexpr int kGrabArcs = 256;       // arcs, by the graph's average, a warp takes at a time
constexpr int kGrabShare = 4;        // a warp takes at most 1/kGrabShare of its share of a phase
constexpr int kGrabCMax = 16;        // most heavy chunks a warp takes at a time
// work-counter slots of a level
enum { WQ_BU = 0, WQ_BU_C, WQ_PUSH, WQ_PUSH_C, WQ_PULL, WQ_PULL_C, WQ_BACK, WQ_BACK_C };

template <int W> struct Bits {
    unsigned long long w[W];
};

template <int W> __device__ __forceinline__ Bits<W> load_bits(const unsigned long long *p)
{
    Bits<W> r;
    if constexpr (W == 1) {
        r.w[0] = __ldcg(p);
    } else {
#pragma unroll
        for (int q = 0; q < W; q += 2) {
            const ulonglong2 x = __ldcg(reinterpret_cast<const ulonglong2 *>(p + q));
            r.w[q] = x.x;
            r.w[q + 1] = x.y;
        }
    }
    return r;
}

template <int W> __device__ __forceinline__ bool any_bits(const Bits<W> &b)
{
    unsigned long long o = 0;
#pragma unroll
    for (int q = 0; q < W; ++q) o |= b.w[q];
    return o != 0;
}

template <int W> __device__ __forceinline__ Bits<W> andnot(const Bits<W> &x, const Bits<W> &y)
{
    Bits<W> r;
#pragma unroll
    for (int q = 0; q < W; ++q) r.w[q] = x.w[q] & ~y.w[q];
    return r;
}

__device__ __forceinline__ int deg_of(const int32_t *rp, int v) { return __ldg(rp + v + 1) - __ldg(rp + v); }

// Records the first failed device-side check (code, where, offending value); every CTA
// then leaves at its next grid barrier and the host reports the status.
__device__ __forceinline__ void check_failed(Ctrl *ctrl, int code, int where, int value)
{
    if (atomicCAS(&ctrl->err, 0, code) == 0) {
        ctrl->where = where;
        ctrl->bad_id = value;
    }
}

struct BlockCnt {
    int v;
    unsigned long long mf, dmu;
};

template <int W> __device__ __forceinline__ void store_bits(unsigned long long *p, const Bits<W> &b)
{
    if constexpr (W == 1) {
        *p = b.w[0];
    } else {
#pragma unroll
        for (int q = 0; q < W; q += 2) *reinterpret_cast<ulonglong2 *>(p + q) = make_ulonglong2(b.w[q], b.w[q + 1]);
    }
}

// Vertices a warp takes at a time (a power of two up to the 32 lanes) of the n of a phase: about
// kGrabArcs arcs by the graph's average, and at most 1/kGrabShare of the warp's share.  Always 32
// vertices left most warps idle on small graphs (63 of 4864 worked on ER 2000: a launch of 64
// sources 680 us, now 200) and made long tails on others: BA 10^6 (16 arcs a vertex), 128 sources,
// 128 arcs a grab 34.1 ms, 256 33.7, 512 42.6; R-MAT 24 (31) 398, 372, 361 (the counter's atomics).
template <class Args> __device__ __forceinline__ int grab_size(const Args &a, int n, int nw)
{
    const int by_arcs = (int)((long long)a.n * kGrabArcs / max((long long)a.A, 1ll));
    const int most = min(by_arcs, n / (kGrabShare * nw));
    return most >= kGrabV ? kGrabV : most <= 1 ? 1 : 1 << (31 - __clz(most));
}

// How a phase finds its vertices: the nq entries of a queue, or (null) a scan of all vertices, whose
// bits the callee looks at (nq: the number of vertices expected).
struct Level {
    const int32_t *queue;
    int nq;
};

// A warp's place in the hand-out of a phase's work, in shared memory (lane 0 writes it).
struct Hand {
    unsigned long long until;  // deadline of the phase
    int c, cend;               // the grabbed chunks left
};

// Calls fn(on, v, beg, dg, chunk) with the whole warp for all work of a phase.  First the
// chunks of the heavy vertices, whose work is largest (chunk >= 0: lane 0 holds the vertex and
// the chunk's arcs), then groups of light vertices, one per lane (chunk = -1).  Warps take work
// dynamically from two zeroed counters (ctr[0] vertices, ctr[1] chunks), each grab requested while the one before is worked
// on; scans of sparse levels (under n/32 vertices) are static.  Loops are bounded in time: lane
// 0 checks the phase's deadline once per item and the warp leaves together (the status is read
// at the next barrier).
template <class Args, class Fn>
__device__ __forceinline__ void for_work(const Args &a, Level lv, int32_t *ctr, Hand &hand, Fn fn)
{
    const int lane = threadIdx.x & 31;
    const int nw = (int)(((long long)gridDim.x * blockDim.x) >> 5);
    if (lane == 0) {
        hand.until = dev::globaltimer() + a.limit_ns;
        hand.c = hand.cend = 0;
    }
    __syncwarp();
    // about C / (32 warps) chunks per grab, 1..16: few chunks stay spread over many warps,
    // millions of chunks cost few atomics
    auto chunk_grab = [&]() { return max(1, min(kGrabCMax, a.C / (32 * nw))); };
    const bool fixed = !lv.queue && lv.nq < a.n / 32;
    const int gv = fixed ? kGrabV : grab_size(a, lv.queue ? lv.nq : a.n, nw);
    const unsigned end = lv.queue ? lv.nq : a.n;
    unsigned next = 0;  // lane 0: the grab under way
    bool chunks = a.C > 0;
    auto grab = [&]() {
        if (lane == 0) {
            if (chunks) next = (unsigned)atomicAdd(ctr + 1, chunk_grab());
            else next = fixed ? next + nw * kGrabV : (unsigned)atomicAdd(ctr, gv);
        }
    };
    auto first = [&]() {  // of the vertices
        if (lane == 0) next = fixed ? (unsigned)(((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * kGrabV
                                    : (unsigned)atomicAdd(ctr, gv);
    };
    if (chunks) grab();
    else first();
    for (;;) {
        bool on = false;
        int v = 0, beg = 0, dg = 0, chunk = -1;
        if (chunks) {
            int c = hand.c;
            if (c >= hand.cend) {
                c = __shfl_sync(FULL, (int)next, 0);
                if (c >= a.C) {
                    chunks = false;
                    first();
                    continue;
                }
                __syncwarp();
                if (lane == 0) hand.cend = min(c + chunk_grab(), a.C);
                grab();
            }
            __syncwarp();
            if (lane == 0) hand.c = c + 1;
            __syncwarp();
            const int i = __ldg(a.chunk_h + c);
            v = __ldg(a.hv + i);
            beg = __ldg(a.rp + v) + (c - __ldg(a.hfirst + i)) * a.chunk;
            dg = min(a.chunk, __ldg(a.rp + v + 1) - beg);
            on = lane == 0;
            chunk = c;
        } else {
            const unsigned i = __shfl_sync(FULL, next, 0) + lane;
            if (i - lane >= end) break;
            grab();
            on = lane < gv && i < end;
            if (on) v = lv.queue ? __ldcg(lv.queue + i) : (int)i;
            if (on && (unsigned)v >= (unsigned)a.n) {
                check_failed(a.status(), kErrCheck, 3, v);
                on = false;
            }
            if (on) {
                beg = __ldg(a.rp + v);
                dg = __ldg(a.rp + v + 1) - beg;
                on = dg > 0 && dg <= a.chunk;
            }
        }
        int late = 0;
        if (lane == 0 && dev::globaltimer() > hand.until) {
            check_failed(a.status(), NK_ERR_TIMEOUT, 2, lv.nq);
            late = 1;
        }
        if (__shfl_sync(FULL, late, 0)) break;
        fn(on, v, beg, dg, chunk);
    }
}

// fn(i, h, c0, c1) per heavy vertex (chunks [c0, c1)), with the whole warp.
template <class Args, class Fn> __device__ __forceinline__ void for_heavy(const Args &a, Fn fn)
{
    const long long wid = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const long long nw = ((long long)gridDim.x * blockDim.x) >> 5;
    for (long long i = wid; i < a.H; i += nw)
        fn((int)i, __ldg(a.hv + i), __ldg(a.hfirst + i), __ldg(a.hfirst + i + 1));
}

// The concatenated arcs of a group of up to 32 vertices, one per lane (d0: the lane's arcs, 0 where
// it has none): lane L's arcs are numbers [pre, pre + d0) of `total`, and the vertices with arcs
// have places 0, 1, ... in the order of the lanes.
struct Rows {
    int d0, pre, total, before;
    unsigned members;
    __device__ __forceinline__ explicit Rows(int d) : d0(d), before(0)
    {
        const int lane = threadIdx.x & 31;
        int incl = d;
#pragma unroll
        for (int s = 1; s < 32; s <<= 1) {
            const int y = __shfl_up_sync(FULL, incl, s);
            if (lane >= s) incl += y;
        }
        total = __shfl_sync(FULL, incl, 31);
        pre = incl - d;
        members = __ballot_sync(FULL, d > 0);
    }
    // the lane's vertex's place, -1 without arcs
    __device__ __forceinline__ int place() const { return d0 > 0 ? __popc(members & dev::lanemask_lt()) : -1; }
    // the place of arc base + lane's vertex, for windows taken in order: the vertices whose arcs
    // start in a window mark their first arc, an arc's vertex is the number of marks up to it
    __device__ __forceinline__ int owner(int base)
    {
        const unsigned marks = __reduce_or_sync(FULL, d0 > 0 && (unsigned)(pre - base) < 32u ? 1u << (pre - base) : 0u);
        const int o = before + __popc(marks & (dev::lanemask_lt() << 1 | 1u)) - 1;
        before += __popc(marks);
        return o;
    }
};

}  // namespace sweep
}  // namespace nk
