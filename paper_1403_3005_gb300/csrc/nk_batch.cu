// Batched multi-source betweenness: B = 64*W sources share one sweep, and several such batches
// one persistent cooperative launch, a row of the grid each.  The paper parallelises Brandes'
// algorithm over sources with one dependency array per thread, summed at the end (Section 3.2);
// on the GPU the sources of a batch instead share every pass over the CSR, so the adjacency of a level is read once for
// all B shortest-path trees.
//
// State of one batch, all in HBM (b = source slot 0..B-1, q = word 0..W-1):
//   F_d[v][q]   bitset of the sources for which v is at BFS level d (one slab per
//               level, kept for the backward sweep)
//   vis[v][q]   union of F_0..F_d
//   sp[v][b]    sigma_b(v) (uint64) during the forward sweep; replaced by
//               psi_b(v) = (1 + delta_b(v)) / sigma_b(v) in the backward sweep (a
//               double-single pair of floats, see nk_device.cuh)
//   queue       vertices of the levels found top-down (levels found bottom-up are
//               iterated by scanning F_d)
// Forward level d, either
//   bottom-up  every vertex w with unvisited sources u = act & ~vis[w] gathers F_d of
//              its neighbours (a warp per group of vertices, lanes over their arcs); for
//              every neighbour c with F_d[c] & u != 0 the lanes switch to the source slots
//              and add sigma_b(c) (the sigma row of c is contiguous, so the gather reads
//              only the sectors of the sources that need it);
//              F_{d+1}[w] = the bits whose sum is non-zero;  or
//   top-down   (a) every frontier vertex v pushes m = F_d[v] & ~vis[c] into F_{d+1}[c]
//              (atomicOr) and queues c once per level; (b) every queued vertex w pulls
//              sigma for exactly its new bits F_{d+1}[w], as above.  sigma is never
//              updated atomically, so sp needs no zeroing.
// Backward level d (deepest first): every v with F_d[v] != 0 gathers, per source bit b
// of F_d[v], acc_b = sum of psi_b(c) over neighbours c with bit b in F_{d+1}[c]; then
// delta_b(v) = sigma_b(v) * acc_b (Brandes' recurrence with sigma_v factored out), psi
// overwrites sigma, and scores[v] += sum_b delta_b(v).
// Bottom-up is chosen when alpha * (arcs of frontier vertices) > (arcs of vertices not
// yet visited by every source).  A BFS deeper than the level slabs aborts the batch
// before its backward sweep (scores untouched); the host re-runs those sources with
// the per-source form.
#include <cooperative_groups.h>

#include <algorithm>
#include <climits>
#include <cstdio>
#include <cstdlib>
#include <vector>

#include "nk_device.cuh"
#include "nk_internal.h"
#include "nk_sweep.cuh"

namespace cg = cooperative_groups;

namespace nk {
namespace {

using namespace sweep;

constexpr int kThreads = 256;
constexpr int kErrDepth = 100;  // internal status: BFS deeper than the level slabs
constexpr int kErrWide = 102;   // internal status: a path count did not fit the 32-bit sigma rows
constexpr int kStartLevels = 48; // level slabs of a first attempt
constexpr int kTraceCap = 1024;
constexpr int kChunk = kHeavyChunk;  // default arcs per work item; longer rows are split
// The arrays below hold the state of every team (blockIdx.y) side by side: [n] stands for
// [teams][n], and a team's row of vertex v is row team * n + v.
struct BArgs {
    int32_t n;
    int64_t A;
    const int32_t *rp, *col;
    const int32_t *src;
    int32_t nsrc;                // sources of the whole run
    int32_t b0;                  // this launch's first batch
    // when set (captured calls), the number of sources of the whole run is *ksrc, read on
    // the device
    const int32_t *ksrc;
    int32_t lcap;                // levels 0..lcap may be non-empty; slabs 0..lcap+1
    unsigned long long *F;       // [lcap+2][teams][n][W]
    unsigned long long *vis;     // [n][W]
    unsigned long long *sp;      // [n][B]
    unsigned *sp32;              // [n][B] sigma in 32 bits during the forward sweep (kernels with S32)
    int32_t *qmark;              // [n] last level a vertex was queued for
    int32_t *queue;              // [qcap]
    int64_t qcap;
    int32_t *vcnt;               // [lcap+3] vertices with F_d != 0
    int32_t *qcnt;               // [lcap+3] queue entries of level d
    int32_t *qoff;               // [lcap+3] start of level d in queue, -1 if not queued
    unsigned long long *mfv;     // [lcap+3] sum of degrees of the level-d vertices
    unsigned long long *dmu;     // [lcap+3] degrees of vertices completed at level d
    int32_t *wq;                 // [lcap+3][8] work counters of the phases of level d
    double *scores;
    Ctrl *ctrl;                  // [batches of the run]
    uint64_t limit_ns;
    double alpha;
    int dir;
    // vertices of degree > chunk are split into chunks of `chunk` arcs (kChunk unless the
    // caller or the autotuner chose another size)
    int32_t chunk;
    const int32_t *hv;           // [H] heavy vertices
    const int32_t *hfirst;       // [H+1] first chunk of each heavy vertex
    const int32_t *chunk_h;      // [C] heavy index of each chunk
    int32_t H, C;
    unsigned long long *part;    // [C][B] per-chunk partial sums (uint64 or double)
    unsigned long long *trace;   // [kTraceCap][2] (code, globaltimer) after each barrier, or null
    int backward;                // 0: forward sweep only (error-bounded estimate)
    double *edge;                // [A] edge betweenness: per-arc shares, or null
    // error-bounded estimate (forward sweep only): per source slot, the target of its
    // random shortest path and the key of the walk's stream; counts of interior vertices
    const int32_t *rk_t;
    const unsigned long long *rk_key;
    unsigned long long *rk_count;

    __device__ __forceinline__ Ctrl *status() const { return ctrl + b0 + blockIdx.y; }
};

// Source slots of a lane: lane L owns the G = 2W consecutive sources [G L, G L + G) of the
// batch.  Slot k of lane L is source G L + k: bit G L + k of the batch's bitsets (word
// (G L + k) / 64) and entry G L + k of a vertex's row of B values, so that one contiguous load
// moves all of a lane's values of a row, and the lane's bits of a bitset are one field of one
// byte.
template <int W> __device__ __forceinline__ int slot_off(int k, int lane) { return 2 * W * lane + k; }

// The word of a bitset that holds the lane's slots (selected without indexing the register
// array by a run-time value, which would move it to local memory).
template <int W> __device__ __forceinline__ unsigned long long lane_word(const Bits<W> &b, int lane)
{
    // mask-and-or over the words: a select chain can be turned into an indexed access
    const int qi = (2 * W * lane) >> 6;
    unsigned long long w = 0ull;
#pragma unroll
    for (int q = 0; q < W; ++q) w |= b.w[q] & (0ull - (unsigned long long)(qi == q));
    return w;
}

// The lane's 2W bits of a bitset of W words in shared memory: a field of one byte.
template <int W> __device__ __forceinline__ unsigned lane_bits(const unsigned long long *w, int lane)
{
    const int s = 2 * W * lane;
    return ((unsigned)reinterpret_cast<const unsigned char *>(w)[s >> 3] >> (s & 7)) & ((1u << (2 * W)) - 1u);
}

// Every lane's 2W bits stored as a bitset of W words in shared memory: the lanes of a byte
// join their fields, the first of them stores it.
template <int W> __device__ __forceinline__ void store_lane_bits(unsigned long long *w, unsigned f, int lane)
{
    constexpr int LPB = 8 / (2 * W);  // lanes of a byte: 4, 2, 1
#pragma unroll
    for (int o = 1; o < LPB; o <<= 1) f |= __shfl_down_sync(FULL, f, o) << (2 * W * o);
    if (lane % LPB == 0) reinterpret_cast<unsigned char *>(w)[lane / LPB] = (unsigned char)f;
}

// acc += x with the carry out of bit 63 counted in carry (a path-count overflow).
__device__ __forceinline__ void add_carry(unsigned long long &acc, unsigned &carry, unsigned long long x)
{
    asm("add.cc.u64 %0, %0, %2;\n\taddc.u32 %1, %1, 0;" : "+l"(acc), "+r"(carry) : "l"(x));
}

// One warp's shared memory: the group of vertices it works on, and the list of the relevant
// neighbours of the current window of 32 arcs.
template <int W, bool EDGE> struct WarpBuf {
    unsigned long long f[32][W];  // list: bits the neighbour shares with its vertex
    unsigned long long t[32][W];  // group: the bits a vertex gathers (a pull leaves its new bits here)
    unsigned c[32];               // list: the neighbour's row
    int o[32];                    // list: its vertex's place in the group
    int off[32];                  // group: first arc, less the arcs of the vertices before
    unsigned v[32];               // group: the vertex's row
    Hand hand;
    double e[EDGE ? 32 : 1];      // list, edge variant: the arc's share
};

// sum_k sv[k] * x[k] over the lane's G slots (x: double-single pairs, zero for slots that are
// not relevant), as a compensated dot product (Ogita, Rump and Oishi's Dot2): the leading
// products hi*hi are summed by TwoSum, and their exact FMA errors, the cross terms hi*lo and
// lo*hi and the TwoSum errors are gathered in one float instead of renormalising the pair
// after every term.  All terms are non-negative (sigma and psi are), so the gathered float
// stays a small fraction of the sum.
template <int G>
__device__ __forceinline__ dev::ff edge_dot(const dev::ff (&sv)[G], const dev::ff (&x)[G])
{
    float s = 0.0f, c = 0.0f;
#pragma unroll
    for (int k = 0; k < G; ++k) {
        const dev::ff b = x[k];
        const float p = __fmul_rn(sv[k].hi, b.hi);
        c = __fmaf_rn(sv[k].hi, b.lo, __fmaf_rn(sv[k].lo, b.hi, __fadd_rn(c, __fmaf_rn(sv[k].hi, b.hi, -p))));
        const float t = __fadd_rn(s, p);
        const float z = __fsub_rn(t, s);
        c = __fadd_rn(c, __fadd_rn(__fsub_rn(s, __fsub_rn(t, z)), __fsub_rn(p, z)));  // TwoSum error
        s = t;
    }
    return {s, c};  // not renormalised: edge_sum2 and ff_to_double take the pair as it is
}

// a + b for pairs whose second parts are small non-negative corrections (edge_dot's
// results): the leading parts by TwoSum, its error and both corrections into the second
// part, without renormalising
__device__ __forceinline__ dev::ff edge_sum2(dev::ff a, dev::ff b)
{
    const float t = __fadd_rn(a.hi, b.hi);
    const float z = __fsub_rn(t, a.hi);
    const float e = __fadd_rn(__fsub_rn(a.hi, __fsub_rn(t, z)), __fsub_rn(b.hi, z));
    return {t, __fadd_rn(__fadd_rn(a.lo, b.lo), e)};
}

// 16- and 8-byte loads that bypass L1, zeros where `on` is zero.  Written out so that a load is
// predicated: the compiler made it a branch, and R-MAT 18 took 13.6 instead of 12.5 ms.  (Reading
// a dummy address instead takes 33 ms: the lanes of all warps meet in one L2 slice.)
// "memory" keeps them in order with the plain stores to the rows that they read; with it and without
// it every form of the kernel takes the same registers and spills.
__device__ __forceinline__ void load16_if(unsigned on, const void *p, unsigned &x, unsigned &y, unsigned &z, unsigned &w)
{
    x = y = z = w = 0;
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %4, 0;\n\t@p ld.global.cg.v4.u32 {%0, %1, %2, %3}, [%5];\n\t}"
                 : "+r"(x), "+r"(y), "+r"(z), "+r"(w) : "r"(on), "l"(p) : "memory");
}
__device__ __forceinline__ void load8_if(unsigned on, const void *p, unsigned &x, unsigned &y)
{
    x = y = 0;
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %2, 0;\n\t@p ld.global.cg.v2.u32 {%0, %1}, [%3];\n\t}"
                 : "+r"(x), "+r"(y) : "r"(on), "l"(p) : "memory");
}

// acc += x where on is not zero
__device__ __forceinline__ void add_if(unsigned on, unsigned long long &acc, unsigned x)
{
    asm("{\n\t.reg .pred p;\n\t.reg .b64 t;\n\tsetp.ne.u32 p, %1, 0;\n\tcvt.u64.u32 t, %2;\n\t@p add.u64 %0, %0, t;\n\t}"
        : "+l"(acc) : "r"(on), "r"(x));
}

// dev::ff_add(a, {hi, lo}), operation by operation, where on is not zero: only the two results
// are predicated, which replaces the two selections of an addition of zero
__device__ __forceinline__ void ff_add_if(unsigned on, dev::ff &a, unsigned hi, unsigned lo)
{
    asm("{\n\t.reg .pred p;\n\t.reg .f32 s, v, e, t;\n\t"
        "setp.ne.u32 p, %2, 0;\n\t"
        "add.rn.f32 s, %0, %3;\n\t"
        "sub.rn.f32 v, s, %0;\n\t"
        "sub.rn.f32 e, s, v;\n\t"
        "sub.rn.f32 e, %0, e;\n\t"
        "sub.rn.f32 v, %3, v;\n\t"
        "add.rn.f32 e, e, v;\n\t"
        "add.rn.f32 t, %1, %4;\n\t"
        "add.rn.f32 t, e, t;\n\t"
        "@p add.rn.f32 %0, s, t;\n\t"
        "sub.rn.f32 v, %0, s;\n\t"
        "@p sub.rn.f32 %1, t, v;\n\t}"
        : "+f"(a.hi), "+f"(a.lo) : "r"(on), "f"(__uint_as_float(hi)), "f"(__uint_as_float(lo)));
}

// F_d of the block's team, and its queue
__device__ __forceinline__ unsigned long long *level_bits(const BArgs &a, int d, size_t slab)
{
    return a.F + ((size_t)d * gridDim.y + blockIdx.y) * slab;
}
__device__ __forceinline__ int32_t *queue_of(const BArgs &a) { return a.queue + (size_t)blockIdx.y * a.qcap; }

// A lane's 2W values of a vertex's row, loaded in 16-byte pieces, each only if one of its
// entries is relevant (nib); the values of other entries are undefined.
template <int W, bool S32> struct RowPart {
    static constexpr int G = 2 * W;
    unsigned u[S32 ? G : 2 * G];
    __device__ __forceinline__ void load(const BArgs &a, unsigned c, int lane, unsigned nib)
    {
        if constexpr (S32) {
            const unsigned *row = a.sp32 + (size_t)c * (64 * W) + G * lane;
            if constexpr (G == 2) {
                load8_if(nib, row, u[0], u[1]);
            } else {
#pragma unroll
                for (int h = 0; h < G / 4; ++h)
                    load16_if(nib & (15u << (4 * h)), row + 4 * h, u[4 * h], u[4 * h + 1], u[4 * h + 2], u[4 * h + 3]);
            }
        } else {
            const unsigned long long *row = a.sp + (size_t)c * (64 * W) + G * lane;
#pragma unroll
            for (int h = 0; h < G / 2; ++h)
                load16_if(nib & (3u << (2 * h)), row + 2 * h, u[4 * h], u[4 * h + 1], u[4 * h + 2], u[4 * h + 3]);
        }
    }
    __device__ __forceinline__ unsigned long long u64(int k) const
    {
        if constexpr (S32) return u[k];
        else return ((unsigned long long)u[2 * k + 1] << 32) | u[2 * k];
    }
    // a path count as a double-single number
    __device__ __forceinline__ dev::ff count(int k) const
    {
        if constexpr (S32) return dev::ff_from_u32(u[k]);
        else return dev::ff_from_u64(u64(k));
    }
};

// Gathers, for a group of up to 32 vertices (lane L's vertex v with arcs [beg, beg + dg) and
// bits t, where `on`), per source slot the sum of sp over the neighbours c whose Fsel[c] & t
// holds that source's bit: uint64 sums (sigma, with carry detection) or double-single sums
// (psi).  The warp walks the concatenated arcs of the group in windows of 32, lanes over arcs:
// a window's column ids, then their level bits, are read in one step whatever the rows'
// lengths, and the neighbours that share a bit with their vertex are listed in shared memory
// in the order of the arcs.  Then the lanes, each on its own source slots, read the rows of
// NB listed neighbours at a time (all of their loads in flight together) and add the relevant
// entries.  When the list comes to another vertex, flush(o) takes the sums of the vertex at
// place o and clears them, and begin(o) is called for the next.  One vertex at a time, a row
// of 8 arcs used 8 of 32 lanes and paid the chain of column, bits and row reads by itself: ER
// 200003 (degree 8) k = 300 in batches of 128 takes 5.1 ms in groups, 8.0 ms without.  What bounds
// it is instruction issue and the latency of its reads (R-MAT 20: issue active 56 %, DRAM 7 %).
// Vertices without a relevant neighbour are never flushed.  Returns the places flushed; pos:
// the lane's vertex's place, or -1.
// With EDGE (psi only) every relevant arc (v, c) also gets its share sum_b sigma_b(v) *
// psi_b(c) (sv: sigma_b of the vertex's slots, set by begin): a warp sum per neighbour, parked
// in shared memory, then added to edge[j] by the lane that listed the arc, which loaded the old
// value when it listed it.  The arc is owned by this warp at this level: no atomics.
template <int W, bool PSI, bool EDGE, bool S32, class Buf, class Begin, class Flush>
__device__ __forceinline__ unsigned gather(const BArgs &a, bool on, int v, int beg, int dg, const Bits<W> &t,
                                           const unsigned long long *Fsel, Buf &st,
                                           unsigned long long (&acc)[2 * W], dev::ff (&facc)[2 * W],
                                           dev::ff (&sv)[2 * W], int &pos, Begin begin, Flush flush)
{
    // rows in flight.  With 2 instead of 4 rows of 32-bit counts R-MAT 18 and BA 10^6 (128 sources)
    // go from 13.2 to 13.5 and 33.5 to 35.7 ms; with 4 rows of psi the W = 2 and 4 kernels run out of
    // registers (256 sources: 12.7 -> 14.7, 33.0 -> 45.6 ms), the W = 1 one gains (15.9 -> 15.4,
    // 41.5 -> 36.0 ms)
    constexpr int G = 2 * W, NB = S32 || (PSI && !EDGE && W == 1) ? 4 : 2;
    const int lane = threadIdx.x & 31;
    const unsigned tn = blockIdx.y * (unsigned)a.n;
    unsigned carry = 0;
    if (on && (beg < 0 || dg < 0 || (long long)beg + dg > a.A)) {
        check_failed(a.status(), kErrCheck, 1, beg);
        on = false;
    }
    Rows rows(on ? dg : 0);
    pos = rows.place();
    __syncwarp();  // the group before is done with the buffer
    if (pos >= 0) {
        st.v[pos] = tn + v;
        st.off[pos] = beg - rows.pre;
#pragma unroll
        for (int q = 0; q < W; ++q) st.t[pos][q] = t.w[q];
    }
    __syncwarp();
    int cur = -1;
    unsigned done = 0;
    for (int base = 0; base < rows.total; base += 32) {
        const int o = rows.owner(base);
        int c = 0, j = 0;
        Bits<W> f;
#pragma unroll
        for (int q = 0; q < W; ++q) f.w[q] = 0;
        if (base + lane < rows.total) {
            j = st.off[o] + base + lane;
            c = __ldg(a.col + j);
            const Bits<W> fc = load_bits<W>(Fsel + (size_t)c * W);
#pragma unroll
            for (int q = 0; q < W; ++q) f.w[q] = fc.w[q] & st.t[o][q];
        }
        const bool mine = any_bits<W>(f);
        const unsigned rel = __ballot_sync(FULL, mine);
        if (!rel) continue;
        const int at = __popc(rel & dev::lanemask_lt()), cnt = __popc(rel);
        // list entries whose vertex is not that of the entry before
        const int lead = __shfl_sync(FULL, o, 31 - __clz(rel & dev::lanemask_lt()));
        const unsigned fresh = __reduce_or_sync(FULL, mine && o != (at ? lead : cur) ? 1u << at : 0u);
        double eold = 0.0;
        if (mine) {
            st.c[at] = tn + c;
            st.o[at] = o;
#pragma unroll
            for (int q = 0; q < W; ++q) st.f[at][q] = f.w[q];
            if constexpr (EDGE) eold = __ldcg(a.edge + (size_t)blockIdx.y * a.A + j);
        }
        if (lane >= cnt && lane < ((cnt + NB - 1) & ~(NB - 1))) {  // the last round's empty places
            st.c[lane] = 0;
#pragma unroll
            for (int q = 0; q < W; ++q) st.f[lane][q] = 0;
        }
        __syncwarp();
        for (int i = 0; i < cnt; i += NB) {
            unsigned nib[NB];
            RowPart<W, S32> x[NB];
#pragma unroll
            for (int r = 0; r < NB; ++r) {
                nib[r] = lane_bits<W>(st.f[i + r], lane);
                x[r].load(a, st.c[i + r], lane, nib[r]);
            }
            dev::ff e[NB];
            auto add = [&](int r) {
                if constexpr (PSI && EDGE) {
                    dev::ff y[G];
#pragma unroll
                    for (int k = 0; k < G; ++k) {
                        y[k] = (nib[r] >> k) & 1u ? dev::ff_unpack(x[r].u64(k)) : dev::ff_zero();
                        facc[k] = dev::ff_add(facc[k], y[k]);
                    }
                    e[r] = edge_dot<G>(sv, y);
                } else if constexpr (PSI) {
#pragma unroll
                    for (int k = 0; k < G; ++k) ff_add_if(nib[r] & (1u << k), facc[k], x[r].u[2 * k], x[r].u[2 * k + 1]);
                } else {
#pragma unroll
                    for (int k = 0; k < G; ++k) {
                        // 32-bit counts: a row of under 2^31 of them cannot overflow 64 bits
                        if constexpr (S32) add_if(nib[r] & (1u << k), acc[k], x[r].u[k]);
                        else add_carry(acc[k], carry, (nib[r] >> k) & 1u ? x[r].u64(k) : 0ull);
                    }
                }
            };
            if (!((fresh >> i) & ((1u << NB) - 1u))) {  // warp-uniform: all of one vertex
#pragma unroll
                for (int r = 0; r < NB; ++r) add(r);
            } else {
#pragma unroll
                for (int r = 0; r < NB; ++r) {
                    if ((fresh >> i) & (1u << r)) {
                        if (cur >= 0) {
                            flush(cur);
                            done |= 1u << cur;
                        }
                        cur = st.o[i + r];
                        begin(cur);
                    }
                    add(r);
                }
            }
            if constexpr (EDGE) {
                // both sums at once: one exchange leaves neighbour 0's partials in the low
                // half-warp and neighbour 1's in the high half, then each half reduces alone
                const bool lo = lane < 16;
                dev::ff own = lo ? e[0] : e[1], other = lo ? e[1] : e[0];
                dev::ff recv;
                recv.hi = __shfl_xor_sync(FULL, other.hi, 16);
                recv.lo = __shfl_xor_sync(FULL, other.lo, 16);
                own = edge_sum2(own, recv);
#pragma unroll
                for (int s = 8; s > 0; s >>= 1) {
                    dev::ff y;
                    y.hi = __shfl_xor_sync(FULL, own.hi, s);
                    y.lo = __shfl_xor_sync(FULL, own.lo, s);
                    own = edge_sum2(own, y);
                }
                if (lane == 0) st.e[i] = dev::ff_to_double(own);
                if (i + 1 < cnt && lane == 16) st.e[i + 1] = dev::ff_to_double(own);
            }
        }
        __syncwarp();
        if constexpr (EDGE) {
            if (mine) a.edge[(size_t)blockIdx.y * a.A + j] = eold + st.e[at];
        }
    }
    if (cur >= 0) {
        flush(cur);
        done |= 1u << cur;
    }
    if (!PSI && !S32 && carry != 0) atomicOr(&a.status()->ovf, 1);
    return done;
}

// Writes the new counts acc of the lane's slots nib of vertex w's sigma row.
template <int W, bool S32>
__device__ __forceinline__ void store_sigma(const BArgs &a, unsigned w, unsigned nib, int lane,
                                            const unsigned long long (&acc)[2 * W])
{
    constexpr int B = 64 * W;
    if constexpr (S32) {
        // a count that does not fit 32 bits sends the batch back to the 64-bit kernel
        unsigned *row = a.sp32 + (size_t)w * B;
        unsigned wide = 0;
#pragma unroll
        for (int k = 0; k < 2 * W; ++k)
            if ((nib >> k) & 1u) {
                row[slot_off<W>(k, lane)] = (unsigned)acc[k];
                wide |= (unsigned)(acc[k] >> 32);
            }
        if (wide) atomicCAS(&a.status()->err, 0, kErrWide);
    } else {
        unsigned long long *row = a.sp + (size_t)w * B;
#pragma unroll
        for (int k = 0; k < 2 * W; ++k)
            if ((nib >> k) & 1u) row[slot_off<W>(k, lane)] = acc[k];
    }
}

// Lane L's vertex w (where `on`) joined level d+1 for the sources nb: writes its visited set
// and F_{d+1}, and counts the warp's vertices in the block's counters.
template <int W>
__device__ __forceinline__ void join_level(const BArgs &a, bool on, int w, int dg, const Bits<W> &nb,
                                           const Bits<W> &act, unsigned long long *Fn, BlockCnt *bc)
{
    const unsigned tn = blockIdx.y * (unsigned)a.n;
    bool full = on;
    if (on) {
        Bits<W> nv = load_bits<W>(a.vis + (size_t)(tn + w) * W);
#pragma unroll
        for (int q = 0; q < W; ++q) {
            nv.w[q] |= nb.w[q];
            full &= nv.w[q] == act.w[q];
        }
        store_bits<W>(a.vis + (size_t)(tn + w) * W, nv);
        store_bits<W>(Fn + (size_t)w * W, nb);
    }
    const unsigned m = __ballot_sync(FULL, on);
    const unsigned df = __reduce_add_sync(FULL, on ? (unsigned)dg : 0u);
    const unsigned dd = __reduce_add_sync(FULL, full ? (unsigned)dg : 0u);
    if ((threadIdx.x & 31) == 0 && m) {
        atomicAdd(&bc->v, __popc(m));
        atomicAdd(&bc->mf, (unsigned long long)df);
        if (dd) atomicAdd(&bc->dmu, (unsigned long long)dd);
    }
}

// Phase trace (diagnostics): CTA 0 records (code, %globaltimer) after a grid barrier.
// code = level * 16 + phase.
enum { PH_INIT = 1, PH_BU_A, PH_BU_B, PH_TD_A, PH_TD_B, PH_TD_C, PH_BK_A, PH_BK_B };

__device__ __forceinline__ void trace_mark(const BArgs &a, int &ti, int level, int phase)
{
    if (a.trace && blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0 && ti < kTraceCap) {
        a.trace[2 * ti] = (unsigned long long)(level * 16 + phase);
        a.trace[2 * ti + 1] = dev::globaltimer();
        ++ti;
    }
}

template <int W>
__device__ __forceinline__ void store_part(const BArgs &a, int c, const unsigned long long (&acc)[2 * W])
{
    unsigned long long *row = a.part + (size_t)(blockIdx.y * (unsigned)a.C + c) * (64 * W);
#pragma unroll
    for (int k = 0; k < 2 * W; ++k) row[slot_off<W>(k, threadIdx.x & 31)] = acc[k];
}

// Sums of a heavy vertex's chunks [c0, c1) in chunk order, four loads in flight at a time.
template <int W, class Add> __device__ __forceinline__ void sum_parts(const BArgs &a, int c0, int c1, Add add)
{
    const unsigned long long *p = a.part + (size_t)(blockIdx.y * (unsigned)a.C + c0) * (64 * W) + slot_off<W>(0, threadIdx.x & 31);
    constexpr int U = W == 1 ? 4 : 2;
    int c = c0;
    for (; c + U <= c1; c += U, p += U * 64 * W) {
        ulonglong2 y[U][W];
#pragma unroll
        for (int r = 0; r < U; ++r)
#pragma unroll
            for (int h = 0; h < W; ++h) y[r][h] = __ldcg(reinterpret_cast<const ulonglong2 *>(p + r * 64 * W) + h);
#pragma unroll
        for (int r = 0; r < U; ++r)
#pragma unroll
            for (int h = 0; h < W; ++h) {
                add(2 * h, y[r][h].x);
                add(2 * h + 1, y[r][h].y);
            }
    }
    for (; c < c1; ++c, p += 64 * W)
#pragma unroll
        for (int k = 0; k < 2 * W; ++k) add(k, __ldcg(p + k));
}

// CTAs per SM that the launch bounds ask for: 4 for 64 and 128 sources (64 registers), 3 for
// the 128-source edge sweep (its per-arc shares need 80 registers, which 64 would spill), 2
// for 256 sources
template <int W, bool EDGE> constexpr int min_ctas() { return W >= 4 ? 2 : (EDGE && W == 2) ? 3 : 4; }

// One batch per team: batch b0 + blockIdx.y by the gridDim.x blocks of that row of the grid.
template <int W, bool EDGE, bool S32>
__global__ void __launch_bounds__(kThreads, min_ctas<W, EDGE>()) k_batch(BArgs a)
{
    constexpr int B = 64 * W;
    // what changes from level to level, kept by thread 0 (in registers it would cost every thread of
    // the gathers about twenty)
    __shared__ BlockCnt bc;
    __shared__ struct {
        unsigned long long act[W];  // bits of the batch's sources
        long long mu, mf;           // arcs of vertices not yet visited by every source, of the level's
        long long qtail;            // queue entries of all levels so far
        int qo, nq;                 // the level's queue entries (qo < 0: found by a scan)
        int td, bu, ti;
    } lv;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int bi = a.b0 + blockIdx.y;
    WarpBuf<W, EDGE> &st = reinterpret_cast<WarpBuf<W, EDGE> *>(smem_raw)[threadIdx.x >> 5];
    const long long tid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const long long nthr = (long long)gridDim.x * blockDim.x;
    const int lane = threadIdx.x & 31;
    const size_t slab = (size_t)a.n * W;
    const unsigned tn = blockIdx.y * (unsigned)a.n;           // the team's first row
    const size_t lv0 = (size_t)blockIdx.y * (a.lcap + 3);      // its first level counter
    const int nsrc = max(0, min(B, (a.ksrc ? __ldg(a.ksrc) : a.nsrc) - bi * B));
    if (nsrc == 0) return;  // uniform over the team: no barrier is entered
    if (threadIdx.x < W) {
        const int left = nsrc - 64 * (int)threadIdx.x;
        lv.act[threadIdx.x] = left >= 64 ? ~0ull : (left <= 0 ? 0ull : ((1ull << left) - 1));
    }
    if (threadIdx.x == 0) lv.ti = 0;
    auto active = [&]() {
        Bits<W> r;
#pragma unroll
        for (int q = 0; q < W; ++q) r.w[q] = lv.act[q];
        return r;
    };
    trace_mark(a, lv.ti, 0, 0);
    auto flush_counts = [&](int lvl) {
        __syncthreads();
        if (threadIdx.x == 0) {
            if (bc.v) atomicAdd(a.vcnt + lv0 + lvl, bc.v);
            if (bc.mf) atomicAdd(a.mfv + lv0 + lvl, bc.mf);
            if (bc.dmu) atomicAdd(a.dmu + lv0 + lvl, bc.dmu);
        }
    };

    // ---- init: empty visited sets, F_0 and F_1, queue marks, level-0..2 counters
    for (size_t i = tid; i < slab; i += nthr) {
        a.vis[(size_t)tn * W + i] = 0;
        level_bits(a, 0, slab)[i] = 0;
        level_bits(a, 1, slab)[i] = 0;
    }
    for (long long i = tid; i < a.n; i += nthr) a.qmark[tn + i] = -1;
    if (tid < 3 * 8) a.wq[lv0 * 8 + tid] = 0;
    if (tid < 3) {
        a.vcnt[lv0 + tid] = 0;
        a.qcnt[lv0 + tid] = 0;
        a.qoff[lv0 + tid] = -1;
        a.mfv[lv0 + tid] = 0;
        a.dmu[lv0 + tid] = 0;
    }
    if (!dev::grid_barrier(a.status(), a.limit_ns)) return;
    trace_mark(a, lv.ti, 0, PH_INIT);
    if (tid < nsrc) {
        const int s = __ldg(a.src + (size_t)bi * B + tid);
        const unsigned long long bit = 1ull << (tid & 63);
        atomicOr(level_bits(a, 0, slab) + (size_t)s * W + (tid >> 6), bit);
        atomicOr(a.vis + (size_t)(tn + s) * W + (tid >> 6), bit);
        if constexpr (S32) a.sp32[(size_t)(tn + s) * B + tid] = 1u;
        else a.sp[(size_t)(tn + s) * B + tid] = 1ull;
        queue_of(a)[tid] = s;
        atomicAdd(a.mfv + lv0, (unsigned long long)deg_of(a.rp, s));
        if (nsrc == 1) a.dmu[lv0] = (unsigned long long)deg_of(a.rp, s);
    }
    if (tid == 0) {
        a.vcnt[lv0] = nsrc;
        a.qcnt[lv0] = nsrc;
        a.qoff[lv0] = 0;
    }
    if (!dev::grid_barrier(a.status(), a.limit_ns)) return;

    if (threadIdx.x == 0) {
        lv.mu = a.A - (long long)__ldcg(a.dmu + lv0);
        lv.mf = (long long)__ldcg(a.mfv + lv0);
        lv.qtail = lv.nq = nsrc;
        lv.qo = lv.td = lv.bu = 0;
    }
    int d = 0;
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
        {
            unsigned long long *Fz = level_bits(a, d + 2, slab);
            for (size_t i = tid; i < slab; i += nthr) Fz[i] = 0;
        }
        __syncthreads();
        const unsigned long long *Fd = level_bits(a, d, slab);
        unsigned long long *Fn = level_bits(a, d + 1, slab);
        const bool use_bu = a.dir == NK_DIR_BOTTOM_UP ||
                            (a.dir == NK_DIR_AUTO && a.alpha * (double)lv.mf > (double)lv.mu);
        bool queued = false;
        int nq1 = 0;
        int32_t *wq = a.wq + (lv0 + d) * 8;
        if (!use_bu) {
            // ---- top-down (a): push the frontier's bits, queue each new vertex once; lanes over
            //      the concatenated arcs of a group of frontier vertices, or of a heavy one's chunk
            for_work(a, {lv.qo >= 0 ? queue_of(a) + lv.qo : nullptr, lv.nq}, wq + WQ_PUSH, st.hand, [&](bool on, int v, int beg, int dg, int) {
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
                    const Bits<W> vc = load_bits<W>(a.vis + (size_t)(tn + c) * W);
                    bool any = false;
#pragma unroll
                    for (int q = 0; q < W; ++q) {
                        const unsigned long long m = st.t[o][q] & ~vc.w[q];
                        any |= m != 0;
                        if (m) atomicOr(Fn + (size_t)c * W + q, m);
                    }
                    if (any && __ldcg(a.qmark + tn + c) != d + 1 && atomicExch(a.qmark + tn + c, d + 1) != d + 1) {
                        cg::coalesced_group g = cg::coalesced_threads();
                        int pos = 0;
                        if (g.thread_rank() == 0) pos = atomicAdd(a.qcnt + lv0 + d + 1, (int)g.size());
                        pos = g.shfl(pos, 0) + (int)g.thread_rank();
                        if (lv.qtail + pos < a.qcap) queue_of(a)[lv.qtail + pos] = c;
                    }
                }
            });
            if (!dev::grid_barrier(a.status(), a.limit_ns)) return;
            trace_mark(a, lv.ti, d, PH_TD_A);
            nq1 = __ldcg(a.qcnt + lv0 + d + 1);
            queued = lv.qtail + nq1 <= a.qcap;
        }
        // ---- pull sigma from level d: bottom-up every vertex with unvisited sources, for all of
        //      them; top-down (b) every new vertex for its new bits.  Chunks of heavy vertices
        //      store partial sums.
        const Level pull = use_bu ? Level{nullptr, a.n} : Level{queued ? queue_of(a) + lv.qtail : nullptr, nq1};
        for_work(a, pull, wq + (use_bu ? WQ_BU : WQ_PULL), st.hand,
                 [&](bool on, int v, int beg, int dg, int chunk) {
            Bits<W> t;
            if (on) {
                t = load_bits<W>(use_bu ? a.vis + (size_t)(tn + v) * W : Fn + (size_t)v * W);
                if (use_bu) t = andnot<W>(active(), t);
                on = any_bits<W>(t);
            }
            if (!__any_sync(FULL, on)) return;
            unsigned long long acc[2 * W];
            dev::ff facc[2 * W];
#pragma unroll
            for (int k = 0; k < 2 * W; ++k) acc[k] = 0;
            int pos;
            const unsigned done = gather<W, false, false, S32>(
                a, on, v, beg, dg, t, Fd, st, acc, facc, facc, pos, [](int) {},
                [&](int o) {
                    if (chunk >= 0) return;  // stored below
                    unsigned nib = 0;
#pragma unroll
                    for (int k = 0; k < 2 * W; ++k) nib |= (acc[k] != 0ull ? 1u : 0u) << k;
                    store_sigma<W, S32>(a, st.v[o], nib, lane, acc);
                    store_lane_bits<W>(st.t[o], nib, lane);
#pragma unroll
                    for (int k = 0; k < 2 * W; ++k) acc[k] = 0;
                });
            if (chunk >= 0) {
                store_part<W>(a, chunk, acc);
                return;
            }
            __syncwarp();
            Bits<W> nb;
#pragma unroll
            for (int q = 0; q < W; ++q) nb.w[q] = 0;
            if (pos >= 0 && ((done >> pos) & 1u))
#pragma unroll
                for (int q = 0; q < W; ++q) nb.w[q] = st.t[pos][q];
            join_level<W>(a, any_bits<W>(nb), v, dg, nb, active(), Fn, &bc);
        });
        if (a.H > 0 && !dev::grid_barrier(a.status(), a.limit_ns)) return;
        trace_mark(a, lv.ti, d, use_bu ? PH_BU_A : PH_TD_B);
        // ---- heavy vertices sum their chunks in chunk order
        for_heavy(a, [&](int i, int h, int c0, int c1) {
            const Bits<W> t = use_bu ? andnot<W>(active(), load_bits<W>(a.vis + (size_t)(tn + h) * W)) : load_bits<W>(Fn + (size_t)h * W);
            if (!any_bits<W>(t)) return;
            unsigned long long acc[2 * W];
#pragma unroll
            for (int k = 0; k < 2 * W; ++k) acc[k] = 0;
            bool ovf = false;
            sum_parts<W>(a, c0, c1, [&](int k, unsigned long long x) {
                const unsigned long long y = acc[k] + x;
                ovf |= y < x;
                acc[k] = y;
            });
            if (ovf) atomicOr(&a.status()->ovf, 1);
            unsigned nib = 0;
#pragma unroll
            for (int k = 0; k < 2 * W; ++k) nib |= (acc[k] != 0ull ? 1u : 0u) << k;
            store_sigma<W, S32>(a, tn + h, nib, lane, acc);
            __syncwarp();
            store_lane_bits<W>(st.t[0], nib, lane);
            __syncwarp();
            Bits<W> nb;
#pragma unroll
            for (int q = 0; q < W; ++q) nb.w[q] = st.t[0][q];
            join_level<W>(a, lane == 0 && any_bits<W>(nb), h, deg_of(a.rp, h), nb, active(), Fn, &bc);
        });
        flush_counts(d + 1);
        if (tid == 0) a.qoff[lv0 + d + 1] = queued ? (int)lv.qtail : -1;
        if (!dev::grid_barrier(a.status(), a.limit_ns)) return;
        trace_mark(a, lv.ti, d, use_bu ? PH_BU_B : PH_TD_C);
        const int c = __ldcg(a.vcnt + lv0 + d + 1);
        if (threadIdx.x == 0) {
            use_bu ? ++lv.bu : ++lv.td;
            lv.qo = queued ? (int)lv.qtail : -1;
            lv.nq = queued ? nq1 : c;
            if (queued) lv.qtail += nq1;
            lv.mu -= (long long)__ldcg(a.dmu + lv0 + d + 1);
            lv.mf = (long long)__ldcg(a.mfv + lv0 + d + 1);
        }
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
    if (a.rk_t) {
        // error-bounded estimate: one warp per source slot b walks one shortest path back
        // from its target, choosing each predecessor z of w with probability
        // sigma_b(z) / sigma_b(w): t = below(stream(key, step), sigma_b(w)) falls in the
        // run of z when the predecessors' sigma values are laid end to end in adjacency
        // order.  Every vertex strictly between the source and the target is counted.
        // The slabs and sigma rows are complete: the last level ended with a grid barrier.
        const long long wid = tid >> 5, nw = nthr >> 5;
        for (long long b = wid; b < nsrc; b += nw) {
            const int v = __ldg(a.rk_t + (size_t)bi * B + b);
            const int q = (int)(b >> 6);
            const unsigned long long bit = 1ull << (b & 63);
            int L = -1;
            for (int l0 = 1; l0 <= D && L < 0; l0 += 32) {
                const int l = l0 + lane;
                const bool hit = l <= D && (__ldcg(level_bits(a, l, slab) + (size_t)v * W + q) & bit) != 0;
                const unsigned m = __ballot_sync(FULL, hit);
                if (m) L = l0 + __ffs(m) - 1;
            }
            if (L < 0) continue;  // the target is not reachable from the source
            const unsigned long long key = __ldg(a.rk_key + (size_t)bi * B + b);
            int w = v;
            for (int l = L, step = 0; l > 1; --l, ++step) {
                const unsigned long long sw = S32 ? (unsigned long long)__ldcg(a.sp32 + (size_t)(tn + w) * B + b)
                                                  : __ldcg(a.sp + (size_t)(tn + w) * B + b);
                const unsigned long long t = dev::below(dev::stream_at(key, (uint64_t)step), sw);
                const unsigned long long *Fp = level_bits(a, l - 1, slab);
                const int end = __ldg(a.rp + w + 1);
                unsigned long long run = 0;
                int z = -1;
                for (int base = __ldg(a.rp + w); base < end && z < 0; base += 32) {
                    const int j = base + lane;
                    int c = -1;
                    unsigned long long x = 0;
                    if (j < end) {
                        c = __ldg(a.col + j);
                        if (__ldcg(Fp + (size_t)c * W + q) & bit)
                            x = S32 ? (unsigned long long)__ldcg(a.sp32 + (size_t)(tn + c) * B + b) : __ldcg(a.sp + (size_t)(tn + c) * B + b);
                    }
                    unsigned long long incl = x;  // inclusive prefix over the lanes
#pragma unroll
                    for (int o = 1; o < 32; o <<= 1) {
                        const unsigned long long y = __shfl_up_sync(FULL, incl, o);
                        if (lane >= o) incl += y;
                    }
                    const unsigned m = __ballot_sync(FULL, x != 0 && run + incl > t);
                    if (m) z = __shfl_sync(FULL, c, __ffs(m) - 1);
                    else run += __shfl_sync(FULL, incl, 31);
                }
                if (z < 0) break;  // only with a wrapped path count (reported as an overflow)
                if (lane == 0) atomicAdd(a.rk_count + z, 1ull);
                w = z;
            }
        }
    }
    if (!a.backward) return;

    // ---- backward sweep, deepest level first (edge betweenness also needs level 0: the
    //      arcs from the sources carry shares, although the sources get no score)
    for (int l = D; l >= (EDGE ? 0 : 1); --l) {
        const unsigned long long *Fl = level_bits(a, l, slab);
        const unsigned long long *Fs = level_bits(a, l + 1, slab);
        const int ql = __ldcg(a.qoff + lv0 + l);
        const int nl = ql >= 0 ? __ldcg(a.qcnt + lv0 + l) : __ldcg(a.vcnt + lv0 + l);
        // delta/psi/score of vertex v from its successor sums facc (whole warp; the lane's slots
        // nib, its path counts sg): psi_v = 1/sigma_v + acc and delta_v = sigma_v * acc (Brandes'
        // recurrence with sigma_v factored out), in double-single; the vertex's delta summed over
        // its source slots (exactly, over the lanes) goes to the FP64 score once per vertex and level.  One warp adds to a
        // vertex's score per level, so the atomic addition, which returns nothing and is not
        // waited for, keeps the order of the additions.
        auto finish = [&](unsigned v, unsigned nib, const RowPart<W, S32> &sg, const dev::ff (&facc)[2 * W]) {
            dev::ff part = dev::ff_zero();
            unsigned long long *row = a.sp + (size_t)v * B;
#pragma unroll
            for (int k = 0; k < 2 * W; ++k) {
                if ((nib >> k) & 1u) {
                    const dev::ff s = sg.count(k);
                    row[slot_off<W>(k, lane)] = dev::ff_pack(dev::ff_add(dev::ff_rcp(s), facc[k]));
                    part = dev::ff_add(part, dev::ff_mul(s, facc[k]));
                }
            }
            if constexpr (!EDGE) {
                const double sum = dev::warp_sum(part);
                if (lane == 0 && sum != 0.0) atomicAdd(a.scores + v, sum);
            }
        };
        for_work(a, {ql >= 0 ? queue_of(a) + ql : nullptr, nl}, a.wq + (lv0 + l) * 8 + WQ_BACK, st.hand,
                 [&](bool on, int v, int beg, int dg, int chunk) {
            Bits<W> t;
            if (on) {
                t = load_bits<W>(Fl + (size_t)v * W);
                on = any_bits<W>(t);
            }
            const unsigned members = __ballot_sync(FULL, on);
            if (!members) return;
            unsigned long long acc[2 * W];
            dev::ff facc[2 * W], sv[2 * W];
            RowPart<W, S32> sg;
#pragma unroll
            for (int k = 0; k < 2 * W; ++k) facc[k] = dev::ff_zero();
            int pos;
            const unsigned done = gather<W, true, EDGE, false>(
                a, on, v, beg, dg, t, Fs, st, acc, facc, sv, pos,
                [&](int o) {
                    if (!EDGE && chunk >= 0) return;
                    const unsigned nib = lane_bits<W>(st.t[o], lane);
                    sg.load(a, st.v[o], lane, nib);  // in flight while the vertex's rows are gathered
                    if constexpr (EDGE) {
#pragma unroll
                        for (int k = 0; k < 2 * W; ++k) sv[k] = (nib >> k) & 1u ? sg.count(k) : dev::ff_zero();
                    }
                },
                [&](int o) {
                    if (chunk >= 0) return;  // stored below
                    finish(st.v[o], lane_bits<W>(st.t[o], lane), sg, facc);
#pragma unroll
                    for (int k = 0; k < 2 * W; ++k) facc[k] = dev::ff_zero();
                });
            if (chunk >= 0) {
#pragma unroll
                for (int k = 0; k < 2 * W; ++k) acc[k] = dev::ff_pack(facc[k]);
                store_part<W>(a, chunk, acc);
                return;
            }
            // vertices without successors: psi = 1 / sigma
            unsigned rest = ((2u << (__popc(members) - 1)) - 1u) & ~done;
            while (rest) {
                const int o = __ffs(rest) - 1;
                rest &= rest - 1;
                const unsigned nib = lane_bits<W>(st.t[o], lane);
                unsigned long long *row = a.sp + (size_t)st.v[o] * B;
                sg.load(a, st.v[o], lane, nib);
#pragma unroll
                for (int k = 0; k < 2 * W; ++k)
                    if ((nib >> k) & 1u) row[slot_off<W>(k, lane)] = dev::ff_pack(dev::ff_rcp(sg.count(k)));
            }
        });
        if (a.H > 0 && !dev::grid_barrier(a.status(), a.limit_ns)) return;
        trace_mark(a, lv.ti, l, PH_BK_A);
        for_heavy(a, [&](int i, int h, int c0, int c1) {
            const Bits<W> mv = load_bits<W>(Fl + (size_t)h * W);
            if (!any_bits<W>(mv)) return;
            const unsigned nib = (unsigned)(lane_word<W>(mv, lane) >> ((2 * W * lane) & 63)) & ((1u << (2 * W)) - 1u);
            RowPart<W, S32> sg;
            sg.load(a, tn + h, lane, nib);
            dev::ff facc[2 * W];
#pragma unroll
            for (int k = 0; k < 2 * W; ++k) facc[k] = dev::ff_zero();
            sum_parts<W>(a, c0, c1, [&](int k, unsigned long long x) { facc[k] = dev::ff_add(facc[k], dev::ff_unpack(x)); });
            finish(tn + h, nib, sg, facc);
        });
        if (!dev::grid_barrier(a.status(), a.limit_ns)) return;
        trace_mark(a, lv.ti, l, PH_BK_B);
    }
}

// ------------------------------------------------------------------ host side
// Dynamic shared memory of one CTA: a neighbour list per warp.
template <int W, bool EDGE> constexpr size_t smem_bytes() { return (size_t)(kThreads / 32) * sizeof(WarpBuf<W, EDGE>); }

// Co-resident CTAs per SM of k_batch<W, EDGE> with its shared memory (the shared-memory
// attribute is set on the first call, outside any stream capture).
template <int W, bool EDGE = false, bool S32 = false> int blocks_per_sm()
{
    static int b = -1;
    if (b < 0) {
        NK_CUDA(cudaFuncSetAttribute(k_batch<W, EDGE, S32>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_bytes<W, EDGE>()));
        int v = 0;
        NK_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&v, k_batch<W, EDGE, S32>, kThreads, smem_bytes<W, EDGE>()));
        b = v;
    }
    return b;
}

struct Layout {
    int W, B, lcap;
    int64_t qcap;
    size_t off_F, off_vis, off_sp, off_sp32, off_qmark, off_queue, off_cnt, off_part, total;
};

size_t align_up(size_t x) { return (x + 255) & ~(size_t)255; }

// chunk count of the heavy table for `chunk` arcs per chunk (an upper bound before the
// table is built)
int64_t chunk_count(const nk_graph *g, int chunk)
{
    if (chunk <= 0) chunk = kChunk;
    if (chunk == kChunk && g->heavy_H >= 0) return g->heavy_C;
    if (chunk != kChunk && g->heavy_alt_H >= 0 && g->heavy_alt_chunk == chunk) return g->heavy_alt_C;
    return g->A / chunk + (g->max_deg > chunk ? g->n : 0);
}

// The workspace of `teams` teams, array by array (so that a team's rows are an offset of the row
// number and not of a pointer).
Layout layout(const nk_graph *g, int B, int lcap, int chunk = 0, int teams = 1)
{
    Layout L;
    L.B = B;
    L.W = B / 64;
    L.lcap = lcap;
    L.qcap = 2 * (int64_t)g->n + B;  // level 0 may hold a vertex several times (drawn pairs)
    const size_t n = (size_t)g->n * teams;
    size_t o = 0;
    L.off_F = o;
    o = align_up(o + (size_t)(lcap + 2) * n * L.W * 8);
    L.off_vis = o;
    o = align_up(o + n * L.W * 8);
    L.off_sp = o;
    o = align_up(o + n * (size_t)B * 8);
    L.off_sp32 = o;
    o = align_up(o + n * (size_t)B * 4);
    L.off_qmark = o;
    o = align_up(o + n * 4);
    L.off_queue = o;
    o = align_up(o + (size_t)L.qcap * 4 * teams);
    L.off_cnt = o;
    o = align_up(o + (size_t)(lcap + 3) * (3 * 4 + 2 * 8 + 8 * 4) * teams);
    L.off_part = o;
    o = align_up(o + (size_t)chunk_count(g, chunk) * B * 8 * teams);
    L.total = o;
    return L;
}

int choose_lcap(const nk_graph *g, int B, const DevBuf *ws, int chunk = 0)
{
    size_t free_b = 0, total_b = 0;
    cudaMemGetInfo(&free_b, &total_b);
    const size_t slab = (size_t)g->n * (B / 64) * 8;
    const Layout base = layout(g, B, 0, chunk);
    // level slabs may use up to half of what is free after the rest of the batch state
    const size_t have = free_b + ws[5].bytes;
    size_t budget = have > base.total ? (have - base.total) / 2 : 0;
    int64_t l = slab ? (int64_t)(budget / slab) - 2 : 1022;
    l = std::min<int64_t>(l, 1022);
    l = std::min<int64_t>(l, std::max<int64_t>(g->n, 4));  // a BFS has at most n levels; 4 at least
    return (int)std::max<int64_t>(l, 0);
}

enum { WS_BATCH = 5, WS_BCTRL = 6 };

constexpr int kMaxTeams = 64;
constexpr size_t kTeamRows = 3300u << 20;  // bytes of sigma and psi rows from which on no team is added
constexpr int kTeamCtas = 128, kTeamVertices = 64;

// Batches run side by side, each by a team of blocks with its own state: one batch of a small graph
// cannot use the GPU, and on the others teams fill the tails of each other's phases.  As many as
// there are batches until their rows reach kTeamRows together (the last team may go beyond it, to at
// most twice that), from where on they only take memory and cache from each other.  1, 2, 4, 8 and all batches at once, 128 sources each: ER 2000
// exact 3.3, 1.7, 0.87, 0.60, 0.46 ms; R-MAT 14 3.7, 2.3, 1.25, 0.98; R-MAT 18 (6) 13.2, 10.6,
// 10.0, -, 9.8; BA 10^6 (4) 31.5, 29.9, 30.0; R-MAT 20 36.2, 34.4, 35.8, 40.3; R-MAT 22 133, 132,
// 136, 146; R-MAT 24 320, 320.  Stopping short of kTeamRows, with 2 instead of 3 teams on 2^20 vertices
// (k = 600, 1000): R-MAT 20 of 31M arcs 24.0 against 26.3 ms and 36.6 / 37.5, of 16M arcs 15.7 / 14.2 and 23.4 / 21.2;
// ER 900000 39.6 / 39.8 and 64.9 / 65.3; on 2^21, 1 against 2, R-MAT 21 of 32M arcs 28.9 / 28.0 and 38.8 / 38.2.
// The number of teams per launch is evened out; the batches stay full and
// the last one short (made equal, R-MAT 18 takes 12.9 instead of 11.3 ms: a row read serves fewer).  Callers with their
// own workspace or grid (captured graphs) run one batch at a time unless they say how many at most (servers).
//
// The sums are kept apart from how many run at once: batch i of a call adds to vector i mod P, in the
// order of the batches, and the P vectors are added up in their order, where P is the number of teams
// that the graph and the batches ask for.  Free memory, or a server's load, may make the teams fewer
// without changing a bit of the scores.
int choose_partials(const nk_graph *g, int B, int nb, const RunCfg &cfg)
{
    if (nb < 2 || (cfg.teams <= 0 && (cfg.ws || cfg.grid_ctas > 0))) return 1;
    return batch_partials(g->n, B, nb);
}

// Teams of a launch: `partials` of them if a quarter of the memory holds their state beside the vectors
// (`outs` sums each), and no more than the caller asks for.
int choose_teams(size_t state, int partials, int grid, const RunCfg &cfg, const DevBuf *ws, int64_t outs)
{
    int want = std::min(partials, grid);
    if (cfg.teams > 0) want = std::min(want, cfg.teams);
    const size_t free_b = free_bytes(ws[WS_BATCH].stream_ordered);
    const size_t sums = sizeof(double) * (size_t)outs * partials;
    while (want > 1 && state * want + sums > (free_b + ws[WS_BATCH].bytes) / 4) --want;
    return want;
}

// Blocks of a team: its share of the grid, but no more than a small graph can use, whose barriers get
// dearer with every block (ER 2000, one batch of 64: 128 blocks 0.185 ms, 608 0.209; R-MAT 14:
// 256 0.459, 608 0.509; ER 50000: 256 0.650, 608 0.596).
int team_ctas(const nk_graph *g, int grid, int teams) { return std::min(grid / teams, std::max(kTeamCtas, g->n / kTeamVertices)); }

// Sources per batch where neither the caller nor the autotuner chose: 128 if there are more than 128
// and their state fits, else 64 (64 against 128, ms: ER 200003 k = 300 4.53 / 4.30, R-MAT 16 3.54 /
// 3.44, R-MAT 18 11.1 / 9.8, BA 20000 1.68 / 1.58, R-MAT 20 40.3 / 34.4: the 128-source kernel
// gathers 64 % of the rows; but up to 128 sources two batches of 64 side by side are better than
// one: R-MAT 18 from its edge list with k = 128 7.3 / 8.0).
int default_width(const nk_graph *g, int32_t k, const RunCfg &cfg)
{
    return k > 128 && choose_lcap(g, 128, scratch(cfg, const_cast<nk_graph *>(g)), cfg.chunk) >= std::min(kStartLevels, std::max(g->n, 4)) ? 128 : 64;
}

// The arguments that do not depend on the batch: graph, workspace at `base`, options.
BArgs make_args(const nk_graph *g, const Layout &L, int teams, const HeavyView &hw, char *base, double *d_scores,
                const RunCfg &cfg)
{
    BArgs a{};
    a.n = g->n;
    a.A = g->A;
    a.rp = g->rp.as<int32_t>();
    a.col = g->col.as<int32_t>();
    a.lcap = L.lcap;
    a.F = reinterpret_cast<unsigned long long *>(base + L.off_F);
    a.vis = reinterpret_cast<unsigned long long *>(base + L.off_vis);
    a.sp = reinterpret_cast<unsigned long long *>(base + L.off_sp);
    a.sp32 = reinterpret_cast<unsigned *>(base + L.off_sp32);
    a.qmark = reinterpret_cast<int32_t *>(base + L.off_qmark);
    a.queue = reinterpret_cast<int32_t *>(base + L.off_queue);
    a.qcap = L.qcap;
    const size_t lv = ((size_t)L.lcap + 3) * teams;
    char *cb = base + L.off_cnt;
    a.mfv = reinterpret_cast<unsigned long long *>(cb);
    a.dmu = a.mfv + lv;
    a.vcnt = reinterpret_cast<int32_t *>(a.dmu + lv);
    a.qcnt = a.vcnt + lv;
    a.qoff = a.qcnt + lv;
    a.wq = a.qoff + lv;
    a.scores = d_scores;
    a.hv = hw.hv;
    a.hfirst = hw.hfirst;
    a.chunk_h = hw.chunk_h;
    a.H = hw.H;
    a.C = hw.C;
    a.chunk = hw.chunk;
    a.part = reinterpret_cast<unsigned long long *>(base + L.off_part);
    a.backward = cfg.backward ? 1 : 0;
    a.edge = cfg.edge && cfg.backward ? cfg.edge : nullptr;
    a.rk_t = cfg.rk_t;
    a.rk_key = cfg.rk_key;
    a.rk_count = cfg.rk_count;
    a.limit_ns = cfg.limit_ns ? cfg.limit_ns : wait_limit_ns();
    a.alpha = cfg.alpha > 0 ? cfg.alpha : 1.0;
    a.dir = cfg.direction;
    return a;
}

// d_count: the number of sources on the device, if they may be put in another order (all have arcs)
template <int W>
int launch_batches(nk_graph *g, const int32_t *d_src, int32_t k, const int32_t *d_count, double *d_scores,
                   const RunCfg &cfg, RunStats *st, cudaStream_t s)
{
    constexpr int B = 64 * W;
    // more than one batch: similar sources share one.  R-MAT 18, 670 sources by 128: 65.2M
    // rows gathered in the order of the ids, 42.8M in this order, 18.3 -> 13.4 ms; R-MAT 24,
    // 271 sources: 493 -> 348 ms; BA 10^6, 512 sources: 40.2 -> 36.9 ms; ER (no hubs) equal
    // (both sides one batch at a time, with the gather of that time: the calls now take 10.7, 300 and 29.4)
    Tmp osrc, okey;
    if (d_count && k > B && !cfg.keep_order) {
        NK_TRY(osrc.alloc(sizeof(int32_t) * (size_t)k, s));
        NK_TRY(okey.alloc(sizeof(unsigned long long) * (size_t)k, s));
        NK_TRY(order_sources(g, d_src, k, d_count, okey.as<unsigned long long>(), osrc.as<int32_t>(), s));
        d_src = osrc.as<int32_t>();
    }
    HeavyView hw;
    NK_TRY(heavy_view(g, cfg.chunk, s, &hw));
    DevBuf *ws = scratch(cfg, g);
    // level slabs: start small; batches whose BFS is deeper are rerun once with the
    // largest cap that free memory allows, then (if still deeper) by the per-source form
    const int lmax = cfg.lcap > 0 ? std::min(cfg.lcap, std::max(g->n, 4)) : choose_lcap(g, B, ws, hw.chunk);
    if (lmax < 4) return set_error(NK_ERR_NOMEM, "not enough device memory for a batch of %d sources", B);
    const int lstart = cfg.lcap > 0 ? lmax : std::min(lmax, std::max(kStartLevels, 4));
    const int nb = (k + B - 1) / B;
    NK_TRY(ws[WS_BCTRL].ensure(sizeof(Ctrl) * nb));
    const bool edge = cfg.edge && cfg.backward;
    // sigma in 32-bit rows unless a batch's counts do not fit (then that batch is rerun with
    // 64-bit rows)
    bool s32 = true;
    auto pick = [&](const void *&kfn, int &grid) -> int {
        const int bps = edge ? (s32 ? blocks_per_sm<W, true, true>() : blocks_per_sm<W, true, false>())
                             : (s32 ? blocks_per_sm<W, false, true>() : blocks_per_sm<W, false, false>());
        if (bps < 1) return set_error(NK_ERR_CUDA, "batched kernel cannot be resident");
        kfn = edge ? (s32 ? (const void *)k_batch<W, true, true> : (const void *)k_batch<W, true, false>)
                   : (s32 ? (const void *)k_batch<W, false, true> : (const void *)k_batch<W, false, false>);
        grid = std::max(1, bps * num_sms() / std::max(1, cfg.grid_div));
        if (cfg.grid_ctas > 0) grid = std::min(grid, cfg.grid_ctas);
        return NK_OK;
    };
    const void *kfn = nullptr;
    int grid = 0;
    NK_TRY(pick(kfn, grid));
    Ctrl *ctrls = ws[WS_BCTRL].as<Ctrl>();
    std::vector<int> todo(nb);
    for (int bi = 0; bi < nb; ++bi) todo[bi] = bi;
    const double alpha_used = cfg.alpha > 0 ? cfg.alpha : 1.0;
    // entries of the sums that the batches add to: per-arc shares, scores, or none
    const int64_t a_out = edge ? g->A : cfg.backward ? g->n : 0;
    static const bool trace_on = std::getenv("NK_TRACE") != nullptr;
    Tmp trace_buf;
    if (trace_on) {
        NK_TRY(trace_buf.alloc(sizeof(unsigned long long) * 2 * kTraceCap, s));
        NK_CUDA(cudaMemsetAsync(trace_buf.p, 0, sizeof(unsigned long long) * 2 * kTraceCap, s));
    }
    for (int lcap = lstart;;) {
        // reruns of some of the batches go one by one
        int partials = (int)todo.size() == nb ? choose_partials(g, B, nb, cfg) : 1;
        Tmp outs;
        if (partials > 1 && a_out > 0 && outs.alloc(sizeof(double) * (size_t)a_out * partials, s) != NK_OK)
            partials = 1;  // no room for the vectors: batch after batch into one
        const int teams = choose_teams(layout(g, B, lcap, hw.chunk).total, partials, grid, cfg, ws, a_out);
        const Layout L = layout(g, B, lcap, hw.chunk, teams);
        NK_TRY(ws[WS_BATCH].ensure(L.total));
        BArgs a = make_args(g, L, teams, hw, ws[WS_BATCH].as<char>(), d_scores, cfg);
        a.src = d_src;
        a.nsrc = k;
        a.ctrl = ctrls;
        if (outs.p) NK_CUDA(cudaMemsetAsync(outs.p, 0, sizeof(double) * (size_t)a_out * partials, s));
        int64_t sweep_launches = 0;
        NK_CUDA(cudaMemsetAsync(ctrls, 0, sizeof(Ctrl) * nb, s));
        cudaEvent_t e0 = nullptr, e1 = nullptr;
        if (cfg.time_kernels) {
            NK_CUDA(cudaEventCreate(&e0));
            NK_CUDA(cudaEventCreate(&e1));
            NK_CUDA(cudaEventRecord(e0, s));
        }
        for (size_t t = 0; t < todo.size();) {
            a.b0 = todo[t];
            a.trace = (trace_on && t == 0) ? trace_buf.as<unsigned long long>() : nullptr;
            // the last launch's teams are larger; a launch's batches add to vectors in a row
            const int at = a.b0 % partials;
            const int now = std::min<int>(std::min(teams, partials - at), (int)(todo.size() - t));
            if (outs.p) (edge ? a.edge : a.scores) = outs.as<double>() + (size_t)at * a_out;
            void *args[] = {&a};
            NK_CUDA(cudaLaunchCooperativeKernel(kfn, dim3(team_ctas(g, grid, now), now), dim3(kThreads), args, edge ? smem_bytes<W, true>() : smem_bytes<W, false>(), s));
            ::nk::count_launch();
            ++sweep_launches;
            t += now;
        }
        if (outs.p) NK_TRY(add_vectors(outs.as<double>(), partials, a_out, edge ? cfg.edge : d_scores, s));
        if (cfg.time_kernels) NK_CUDA(cudaEventRecord(e1, s));
        std::vector<Ctrl> h(nb);
        NK_CUDA(cudaMemcpyAsync(h.data(), ctrls, sizeof(Ctrl) * nb, cudaMemcpyDeviceToHost, s));
        NK_TRY(host_wait(s, (int64_t)todo.size(), a.limit_ns));
        if (st) {
            st->mode = NK_MODE_BATCHED;
            st->batch = B;
            st->tpv = 32;
            st->launches += (int64_t)todo.size();
            st->kernel_launches += sweep_launches;
            st->alpha = alpha_used;
            for (int bi : todo) {
                st->max_depth = std::max(st->max_depth, h[bi].depth);
                st->td_levels += h[bi].td_levels;
                st->bu_levels += h[bi].bu_levels;
            }
            if (cfg.time_kernels) {
                float ms = 0;
                cudaEventElapsedTime(&ms, e0, e1);
                st->kernel_ms += ms;
            }
        }
        if (e0) cudaEventDestroy(e0);
        if (e1) cudaEventDestroy(e1);
        if (trace_on) {
            static const char *names[] = {"start", "init", "bu-pull", "bu-hubs", "td-push", "td-pull", "td-hubs", "back", "back-hubs"};
            std::vector<unsigned long long> t(2 * kTraceCap);
            NK_CUDA(cudaMemcpyAsync(t.data(), trace_buf.p, sizeof(unsigned long long) * t.size(), cudaMemcpyDeviceToHost, s));
            NK_CUDA(cudaStreamSynchronize(s));
            for (int i = 1; i < kTraceCap && t[2 * i + 1]; ++i)
                fprintf(stderr, "nk-trace B=%d level=%llu phase=%s us=%.1f\n", B, t[2 * i] / 16,
                        names[std::min<unsigned long long>(t[2 * i] % 16, 8)], (t[2 * i + 1] - t[2 * i - 1]) * 1e-3);
        }
        bool ovf = false;
        std::vector<int> deep, wide;
        for (int bi : todo) {
            if (h[bi].err == NK_ERR_TIMEOUT)
                return set_error(NK_ERR_TIMEOUT, "batched sweep aborted: a bounded device-side wait or phase ran out (check %d, value %d)",
                                 h[bi].where, h[bi].bad_id);
            if (h[bi].err == kErrCheck)
                return set_error(NK_ERR_CUDA, "batched sweep aborted: device range check %d failed (value %d)",
                                 h[bi].where, h[bi].bad_id);
        }
        for (int bi : todo)
            if (h[bi].err == kErrWide) wide.push_back(bi);
        if (!wide.empty()) {
            // counts beyond 32 bits: these batches again with 64-bit sigma rows, together with
            // any that ran out of level slabs (an aborted batch never reaches the backward
            // sweep, so it has added nothing to the scores)
            for (int bi : todo)
                if (h[bi].err == kErrDepth) wide.push_back(bi);
            std::sort(wide.begin(), wide.end());
            s32 = false;
            NK_TRY(pick(kfn, grid));
            todo = wide;
            continue;
        }
        for (int bi : todo) {
            ovf |= h[bi].ovf != 0;
            if (h[bi].err == kErrDepth) deep.push_back(bi);
        }
        if (ovf) return set_error(NK_ERR_OVERFLOW, "a shortest-path count exceeded 2^64 - 1");
        if (deep.empty()) return NK_OK;
        if (lcap < lmax) {
            todo = deep;
            lcap = lmax;
            continue;
        }
        // deeper than any level cap that fits: the per-source form takes these sources
        for (int bi : deep) {
            RunCfg pc = cfg;
            pc.tpv = 0;
            pc.compacted = true;
            if (pc.rk_t) {
                pc.rk_t += (size_t)bi * B;
                pc.rk_key += (size_t)bi * B;
            }
            NK_TRY(run_per_source(g, d_src + (size_t)bi * B, std::min(B, k - bi * B), d_scores, pc, st, s));
        }
        return NK_OK;
    }
}

// Capturable form of one pass of launch_batches: no host synchronisation and no
// allocation once prepared.  With prepare_only it sizes and allocates the workspace (call
// it before a stream capture); otherwise it enqueues the status reset and the cooperative
// launches (cudaLaunchKernelExC with the cooperative attribute, which stream capture
// records as kernel nodes) and returns the per-batch status words for the caller to read.
template <int W>
int enqueue_batches(nk_graph *g, const int32_t *d_src, int32_t k, double *d_scores,
                    const RunCfg &cfg, cudaStream_t s, bool prepare_only, Ctrl **ctrls_out, int *nb_out)
{
    constexpr int B = 64 * W;
    DevBuf *ws = scratch(cfg, g);
    HeavyView hw;
    NK_TRY(heavy_view(g, cfg.chunk, s, &hw));
    const int lcap = cfg.lcap > 0 ? std::min(cfg.lcap, std::max(g->n, 4)) : std::min(choose_lcap(g, B, ws, hw.chunk), std::max(kStartLevels, 4));
    if (lcap < 4) return set_error(NK_ERR_NOMEM, "not enough device memory for a batch of %d sources", B);
    const int nb = (k + B - 1) / B;
    const Layout L = layout(g, B, lcap, hw.chunk);
    // status words of the nb batches, then the compacted sources and their count; with more
    // than one batch also the ordered sources and their keys
    const size_t ctrl_bytes = align_up(sizeof(Ctrl) * nb), src_bytes = align_up(sizeof(int32_t) * (size_t)k);
    const size_t bctrl_bytes = ctrl_bytes + src_bytes + 256 + (nb > 1 ? src_bytes + sizeof(unsigned long long) * (size_t)k : 0);
    if (prepare_only) {
        NK_TRY(ws[WS_BATCH].ensure(L.total));
        NK_TRY(ws[WS_BCTRL].ensure(bctrl_bytes));
        if (blocks_per_sm<W, false, true>() < 1) return set_error(NK_ERR_CUDA, "batched kernel cannot be resident");
        return NK_OK;
    }
    if (ws[WS_BATCH].bytes < L.total || ws[WS_BCTRL].bytes < bctrl_bytes)
        return set_error(NK_ERR_ARG, "batched workspace not prepared");
    const int bps = blocks_per_sm<W, false, true>();
    if (bps < 1) return set_error(NK_ERR_CUDA, "batched kernel cannot be resident");
    int grid = std::max(1, bps * num_sms() / std::max(1, cfg.grid_div));
    if (cfg.grid_ctas > 0) grid = std::min(grid, cfg.grid_ctas);
    BArgs a = make_args(g, L, 1, hw, ws[WS_BATCH].as<char>(), d_scores, cfg);
    a.edge = nullptr;  // the captured form serves vertex scores only
    Ctrl *ctrls = ws[WS_BCTRL].as<Ctrl>();
    int32_t *csrc = reinterpret_cast<int32_t *>(ws[WS_BCTRL].as<char>() + ctrl_bytes);
    int32_t *ccnt = reinterpret_cast<int32_t *>(ws[WS_BCTRL].as<char>() + ctrl_bytes + src_bytes);
    NK_CUDA(cudaMemsetAsync(ctrls, 0, sizeof(Ctrl) * nb, s));
    // sources without arcs add nothing: compacted on the device, each batch reads the count
    NK_TRY(compact_sources(g, d_src, k, csrc, ccnt, s));
    if (nb > 1) {
        char *ob = ws[WS_BCTRL].as<char>() + ctrl_bytes + src_bytes + 256;
        int32_t *osrc = reinterpret_cast<int32_t *>(ob);
        NK_TRY(order_sources(g, csrc, k, ccnt, reinterpret_cast<unsigned long long *>(ob + src_bytes), osrc, s));
        csrc = osrc;
    }
    a.src = csrc;
    a.nsrc = k;
    a.ksrc = ccnt;
    a.ctrl = ctrls;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeCooperative;
    attr.val.cooperative = 1;
    cudaLaunchConfig_t lc = {};
    lc.gridDim = dim3(grid);
    lc.blockDim = dim3(kThreads);
    lc.dynamicSmemBytes = smem_bytes<W, false>();
    lc.stream = s;
    lc.attrs = &attr;
    lc.numAttrs = 1;
    for (int bi = 0; bi < nb; ++bi) {
        a.b0 = bi;
        void *args[] = {&a};
        NK_CUDA(cudaLaunchKernelExC(&lc, (const void *)k_batch<W, false, true>, args));
        ::nk::count_launch();
    }
    *ctrls_out = ctrls;
    *nb_out = nb;
    return NK_OK;
}

}  // namespace

int batch_partials(int32_t n, int B, int nb)
{
    const size_t rows = (size_t)n * B * 12;
    int want = (int)std::min<size_t>(std::min(nb, kMaxTeams), (kTeamRows + rows - 1) / rows);
    while (want > 1 && (int64_t)n * want > INT32_MAX) --want;  // rows are numbered in 32 bits
    const int rounds = (nb + want - 1) / want;
    return (nb + rounds - 1) / rounds;
}

size_t batched_bytes(const nk_graph *g, int B) { return layout(g, B, 16).total; }

size_t batched_bytes_lcap(const nk_graph *g, int B, int lcap) { return layout(g, B, lcap).total; }

int run_batched(nk_graph *g, const int32_t *d_src, int32_t k, double *d_scores,
                const RunCfg &cfg, RunStats *st, cudaStream_t s)
{
    // sources without arcs add nothing: the batches, and the choice of their width, take the others
    // (the error-bounded estimate keeps its slots, which are tied to their targets)
    Tmp list, count;
    if (!cfg.rk_t) NK_TRY(compact_list(g, &d_src, &k, list, count, s));
    int B = cfg.batch;
    if (B == 0) B = g->tuned.valid ? g->tuned.batch : default_width(g, k, cfg);
    if (k == 0) {
        if (st) {
            st->mode = NK_MODE_BATCHED;
            st->batch = B;
        }
        return NK_OK;
    }
    switch (B) {
    case 64: return launch_batches<1>(g, d_src, k, count.as<int32_t>(), d_scores, cfg, st, s);
    case 128: return launch_batches<2>(g, d_src, k, count.as<int32_t>(), d_scores, cfg, st, s);
    case 256: return launch_batches<4>(g, d_src, k, count.as<int32_t>(), d_scores, cfg, st, s);
    default: return set_error(NK_ERR_ARG, "batch must be 64, 128 or 256 (got %d)", B);
    }
}

int enqueue_batched(nk_graph *g, const int32_t *d_src, int32_t k, double *d_scores,
                    const RunCfg &cfg, cudaStream_t s, bool prepare_only, Ctrl **ctrls, int *nb)
{
    int B = cfg.batch;
    if (B == 0) B = g->tuned.valid ? g->tuned.batch : 64;
    switch (B) {
    case 64: return enqueue_batches<1>(g, d_src, k, d_scores, cfg, s, prepare_only, ctrls, nb);
    case 128: return enqueue_batches<2>(g, d_src, k, d_scores, cfg, s, prepare_only, ctrls, nb);
    case 256: return enqueue_batches<4>(g, d_src, k, d_scores, cfg, s, prepare_only, ctrls, nb);
    default: return set_error(NK_ERR_ARG, "batch must be 64, 128 or 256 (got %d)", B);
    }
}

}  // namespace nk
