// Source sampler for the sampled betweenness estimate (Section 3.2: betweenness from a
// small number of randomly chosen shortest-path trees, after Geisberger et al.).
//
// Rule: k distinct sources uniformly without replacement = the k vertices with the
// smallest key(v) = v-th output of the SplitMix64 stream seeded with `seed`.  The keys
// are distinct (v -> seed + (v+1)*gamma is a bijection mod 2^64 for odd gamma, and the
// finaliser is a bijection), so the selection is a threshold: key(v) <= T where T is
// the k-th smallest key.  T is found by a radix select over 11-bit digits (keys are
// recomputed, never stored); the chosen ids are then written in ascending
// order by an order-preserving compaction.  No sort is needed.
#include <algorithm>

#include "nk_device.cuh"
#include "nk_internal.h"

namespace nk {
namespace {

constexpr int kDigit = 11;        // bits of a digit
constexpr int kBins = 1 << kDigit;
constexpr int kSelThreads = 256;
constexpr int kPerThread = kBins / kSelThreads;

struct SelState {
    uint64_t prefix;  // digits of T fixed so far; T itself once done
    uint64_t mask;    // which bits of the prefix are fixed
    int64_t krem;     // rank of T among the keys that match the prefix (1-based)
    unsigned blocks;  // blocks of the running pass that have added their counts
    int done;         // T is known
};

__global__ void k_sel_init(SelState *s, int64_t k, unsigned *hist)
{
    s->prefix = 0;
    s->mask = 0;
    s->krem = k;
    s->blocks = 0;
    s->done = 0;
    for (int i = threadIdx.x; i < kBins; i += blockDim.x) hist[i] = 0;
}

// One digit of T: counts the keys with the prefix found so far by their digit; the last block to add
// its counts chooses the digit that holds the krem-th key and clears the counts.  Once a digit's keys
// all belong to the sample, T is the largest key with that prefix and the passes left return at once:
// usually after two or three of six.  (Eight passes of eight bits, each with a second kernel whose one
// thread walked the counts, took 175 us of every sampled call.)
__global__ void __launch_bounds__(kSelThreads)
k_sel_pass(int32_t n, uint64_t seed, SelState *s, int shift, int bits, unsigned *hist)
{
    __shared__ unsigned h[kBins];
    __shared__ unsigned warp_sum[kSelThreads / 32];
    __shared__ bool last;
    if (s->done) return;  // uniform: set by an earlier pass
    for (int i = threadIdx.x; i < kBins; i += kSelThreads) h[i] = 0;
    __syncthreads();
    const uint64_t prefix = s->prefix, mask = s->mask;
    const unsigned low = (1u << bits) - 1u;
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n;
         v += (int64_t)gridDim.x * blockDim.x) {
        const uint64_t key = dev::stream_at(seed, (uint64_t)v);
        if ((key & mask) == prefix) atomicAdd(&h[(unsigned)(key >> shift) & low], 1u);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < kBins; i += kSelThreads)
        if (h[i]) atomicAdd(&hist[i], h[i]);
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(&s->blocks, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!last) return;
    __threadfence();
    // the last block: each thread's kPerThread bins, a scan over the block, and the one thread whose
    // bins hold the krem-th key
    unsigned c[kPerThread], mine = 0;
#pragma unroll
    for (int q = 0; q < kPerThread; ++q) mine += c[q] = __ldcg(hist + threadIdx.x * kPerThread + q);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    unsigned incl = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    if (lane == 31) warp_sum[wid] = incl;
    const int64_t krem = s->krem;
    __syncthreads();
    int64_t before = (int64_t)incl - mine;
    for (int w = 0; w < wid; ++w) before += warp_sum[w];
    if (before < krem && before + mine >= krem) {
        int q = 0;
        while (before + c[q] < krem) before += c[q++];
        const uint64_t digit = (uint64_t)(threadIdx.x * kPerThread + q);
        s->krem = krem - before;
        s->prefix = prefix | digit << shift;
        s->mask = mask | (uint64_t)low << shift;
        if ((int64_t)c[q] == krem - before) {
            s->prefix |= (1ull << shift) - 1ull;
            s->done = 1;
        }
        s->blocks = 0;
    }
    __syncthreads();
    for (int i = threadIdx.x; i < kBins; i += kSelThreads) hist[i] = 0;
}

constexpr int kTileV = 1024;

__global__ void __launch_bounds__(kTileV)
k_sel_count(int32_t n, uint64_t seed, const SelState *s, int64_t *tile_cnt)
{
    __shared__ int wc[32];
    const int64_t v = (int64_t)blockIdx.x * kTileV + threadIdx.x;
    const bool pick = v < n && dev::stream_at(seed, (uint64_t)v) <= s->prefix;
    const unsigned bal = __ballot_sync(0xffffffffu, pick);
    if ((threadIdx.x & 31) == 0) wc[threadIdx.x >> 5] = __popc(bal);
    __syncthreads();
    if (threadIdx.x == 0) {
        int t = 0;
        for (int i = 0; i < 32; ++i) t += wc[i];
        tile_cnt[blockIdx.x] = t;
    }
}

__global__ void __launch_bounds__(kTileV)
k_sel_write(int32_t n, uint64_t seed, const SelState *s, const int64_t *tile_off,
            int32_t *src)
{
    __shared__ int wc[32];
    const int64_t v = (int64_t)blockIdx.x * kTileV + threadIdx.x;
    const bool pick = v < n && dev::stream_at(seed, (uint64_t)v) <= s->prefix;
    const unsigned bal = __ballot_sync(0xffffffffu, pick);
    const int wid = threadIdx.x >> 5;
    if ((threadIdx.x & 31) == 0) wc[wid] = __popc(bal);
    __syncthreads();
    int before = 0;
    for (int i = 0; i < wid; ++i) before += wc[i];
    if (pick) src[tile_off[blockIdx.x] + before + __popc(bal & dev::lanemask_lt())] = (int32_t)v;
}

}  // namespace

int sample_sources_device(int32_t n, uint64_t seed, int32_t k, int32_t *d_src, cudaStream_t st)
{
    if (n < 1 || k < 1 || k > n) return set_error(NK_ERR_ARG, "need 1 <= k <= n (k=%d, n=%d)", k, n);
    Tmp state, hist, tiles;
    NK_TRY(state.alloc(sizeof(SelState), st));
    NK_TRY(hist.alloc(kBins * sizeof(unsigned), st));
    const int64_t ntiles = ((int64_t)n + kTileV - 1) / kTileV;
    NK_TRY(tiles.alloc(sizeof(int64_t) * ntiles, st));
    SelState *S = state.as<SelState>();
    unsigned *H = hist.as<unsigned>();
    k_sel_init<<<1, 256, 0, st>>>(S, k, H);
    ::nk::count_launch();
    NK_CUDA(cudaGetLastError());
    int blocks = (int)std::min<int64_t>(((int64_t)n + 255) / 256, 4LL * num_sms());
    for (int top = 64; top > 0; top -= kDigit) {
        const int bits = std::min(top, kDigit);
        k_sel_pass<<<blocks, kSelThreads, 0, st>>>(n, seed, S, top - bits, bits, H);
        ::nk::count_launch();
    }
    NK_CUDA(cudaGetLastError());
    k_sel_count<<<(unsigned)ntiles, kTileV, 0, st>>>(n, seed, S, tiles.as<int64_t>());
    ::nk::count_launch();
    NK_CUDA(cudaGetLastError());
    NK_TRY(scan_exclusive_i64(tiles.as<int64_t>(), tiles.as<int64_t>(), ntiles, nullptr, st));
    k_sel_write<<<(unsigned)ntiles, kTileV, 0, st>>>(n, seed, S, tiles.as<int64_t>(), d_src);
    ::nk::count_launch();
    NK_CUDA(cudaGetLastError());
    return NK_OK;
}

}  // namespace nk

using namespace nk;

extern "C" int nk_sample_sources(int32_t n, uint64_t seed, int32_t k, int32_t *src, uint32_t flags)
{
    if (!src) return set_error(NK_ERR_ARG, "src is null");
    if (n < 1 || k < 1 || k > n) return set_error(NK_ERR_ARG, "need 1 <= k <= n (k=%d, n=%d)", k, n);
    cudaStream_t st = stream();
    if (flags & NK_RUN_DEVICE_PTRS) {
        NK_TRY(sample_sources_device(n, seed, k, src, st));
        NK_CUDA(cudaStreamSynchronize(st));
        return NK_OK;
    }
    Tmp d;
    NK_TRY(d.alloc(sizeof(int32_t) * k, st));
    NK_TRY(sample_sources_device(n, seed, k, d.as<int32_t>(), st));
    NK_CUDA(cudaMemcpyAsync(src, d.p, sizeof(int32_t) * k, cudaMemcpyDeviceToHost, st));
    NK_CUDA(cudaStreamSynchronize(st));
    return NK_OK;
}
