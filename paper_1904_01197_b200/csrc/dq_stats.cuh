// Histogram of the codes of a packed message: the input of the paper's rate accounting (entropy of the index
// stream, Section 4, tables of raw and entropy-coded bits).  One pass over the packed words.
//
// One and two bits are counted by population counts of whole words; wider codes one by one into shared memory.
// Messages of one- and two-bit codes up to kHistClusterBytes are counted by a single cluster of CTAs, whose partial
// counts meet in the first CTA's shared memory: the counters are written once, so they need not be cleared first, and
// one launch is all (2 bits, n = 65,536: 6.2 us with a memset, 2.4 us).  Longer messages take the whole GPU and a small
// kernel before it that clears the counters: the count can begin to launch while it runs, which it cannot behind a
// memset.
#pragma once

#include "dq_device.cuh"

namespace dq {

constexpr int kHistThreads = 256;
constexpr int kHistClusterThreads = 1024;
constexpr int kHistCluster = 16;                       // 8 where a cluster of 16 cannot be resident
constexpr uint64_t kHistClusterBytes = 3ull << 19;

__global__ void __launch_bounds__(kHistThreads) clear_histogram_kernel(unsigned long long* hist)
{
    grid_dependency_wait();
    grid_dependency_launch_next();
    hist[threadIdx.x] = 0ull;
}

// Counts of the codes 1, 2 and 3 (of the code 1 with one bit) in a stretch of words.
struct FewCounts { uint32_t c1, c2, c3; };

// Two words of 2-bit codes: three population counts, the codes of the second word beside those of the first.
__device__ __forceinline__ void count2(uint32_t a, uint32_t b, FewCounts& f)
{
    const uint32_t m = 0x55555555u;
    const uint32_t lo = (a & m) | ((b & m) << 1), hi = ((a >> 1) & m) | (b & ~m);
    f.c1 += __popc(lo & ~hi);
    f.c2 += __popc(hi & ~lo);
    f.c3 += __popc(lo & hi);
}

template <int BITS>
__device__ __forceinline__ void count_words(const uint32_t* __restrict__ packed, uint64_t n, uint64_t first, uint64_t stride,
                                            FewCounts& f)
{
    const uint64_t quads = (n * BITS) >> 7;            // 16-byte pieces without pad bits
    auto count = [&](const uint4& v) {
        if constexpr (BITS == 1) {
            f.c1 += __popc(v.x) + __popc(v.y) + __popc(v.z) + __popc(v.w);
        } else {
            count2(v.x, v.y, f);
            count2(v.z, v.w, f);
        }
    };
    const uint4* p = reinterpret_cast<const uint4*>(packed);
    constexpr int kFlight = 4;                         // loads in flight: a short message is two or three latencies
    for (uint64_t i = first; i < quads; i += kFlight * stride) {
        uint4 v[kFlight];
#pragma unroll
        for (int j = 0; j < kFlight; ++j)
            if (i + (uint64_t)j * stride < quads) v[j] = __ldg(p + i + (uint64_t)j * stride);
#pragma unroll
        for (int j = 0; j < kFlight; ++j)
            if (i + (uint64_t)j * stride < quads) count(v[j]);
    }
    if (first == 0u) {                                 // what is left: at most four words, the last one partly pad
        for (uint64_t w = quads * 4u; w * 32u < n * BITS; ++w) {
            const uint64_t left = n * BITS - w * 32u;
            uint4 v = make_uint4(__ldg(packed + w) & (left >= 32u ? 0xFFFFFFFFu : (1u << (uint32_t)left) - 1u), 0u, 0u, 0u);
            count(v);
        }
    }
}

// Adds every thread's counts into sums[0..2] (shared memory, zero on entry; the caller synchronises before and after).
__device__ __forceinline__ void add_counts(const FewCounts& f, uint32_t* sums)
{
    const uint32_t a = __reduce_add_sync(0xFFFFFFFFu, f.c1), b = __reduce_add_sync(0xFFFFFFFFu, f.c2),
                   c = __reduce_add_sync(0xFFFFFFFFu, f.c3);
    if ((threadIdx.x & 31u) == 0u) {
        atomicAdd(sums, a);
        atomicAdd(sums + 1, b);
        atomicAdd(sums + 2, c);
    }
}

// One cluster counts everything and writes the counters (fewer than 2^32 codes).
template <int BITS>
__global__ void __launch_bounds__(kHistClusterThreads)
code_histogram_cluster_kernel(const uint32_t* __restrict__ packed, uint64_t n, unsigned long long* hist)
{
    __shared__ uint32_t sums[3], total[3];
    if (threadIdx.x < 3u) sums[threadIdx.x] = total[threadIdx.x] = 0u;
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    grid_dependency_wait();
    grid_dependency_launch_next();
    FewCounts f = {0u, 0u, 0u};
    count_words<BITS>(packed, n, (uint64_t)blockIdx.x * kHistClusterThreads + threadIdx.x,
                      (uint64_t)gridDim.x * kHistClusterThreads, f);
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");        // total[] of CTA 0 is zero
    add_counts(f, sums);
    __syncthreads();
    if (threadIdx.x < 3u) {
        uint32_t remote;
        asm volatile("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(remote) : "r"(smem_u32(total + threadIdx.x)));
        asm volatile("red.relaxed.cluster.shared::cluster.add.u32 [%0], %1;" ::"r"(remote), "r"(sums[threadIdx.x]) : "memory");
    }
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    if (blockIdx.x == 0u && threadIdx.x < (1u << BITS))
        hist[threadIdx.x] = threadIdx.x == 0u ? n - total[0] - total[1] - total[2] : total[threadIdx.x - 1u];
}

// Longer messages of one- and two-bit codes; hist has been cleared.
template <int BITS>
__global__ void __launch_bounds__(kHistThreads)
code_histogram_words_kernel(const uint32_t* __restrict__ packed, uint64_t n, unsigned long long* hist)
{
    __shared__ uint32_t sums[3];
    if (threadIdx.x < 3u) sums[threadIdx.x] = 0u;
    grid_dependency_wait();
    grid_dependency_launch_next();
    FewCounts f = {0u, 0u, 0u};
    count_words<BITS>(packed, n, (uint64_t)blockIdx.x * kHistThreads + threadIdx.x, (uint64_t)gridDim.x * kHistThreads, f);
    __syncthreads();
    add_counts(f, sums);
    __syncthreads();
    if (threadIdx.x < (1u << BITS) - 1u) {
        atomicAdd(hist + 1 + threadIdx.x, (unsigned long long)sums[threadIdx.x]);
        atomicAdd(hist, 0ull - (unsigned long long)sums[threadIdx.x]);          // (modulo 2^64)
    }
    if (blockIdx.x == 0u && threadIdx.x == 31u) atomicAdd(hist, (unsigned long long)n);
}

// Wider codes; hist has been cleared.  A thread handles one row (32 codes, BITS words) at a time.  Each warp has counters
// of its own; with OWN (four and five bits, very long messages: see dq_code_histogram) each thread has, so that no two
// lanes of a warp meet in a shared-memory bank, but 32 KB have to be cleared and added up per CTA.
template <int BITS, bool OWN>
__global__ void __launch_bounds__(kHistThreads)
code_histogram_kernel(const uint32_t* __restrict__ packed, uint64_t n, unsigned long long* hist)
{
    constexpr uint32_t kBins = 1u << BITS, kWarps = kHistThreads / 32;
    constexpr uint32_t kStep = OWN ? (uint32_t)kHistThreads : 1u;
    __shared__ uint32_t bins[OWN ? kBins * kHistThreads : kBins * kWarps];
    for (uint32_t i = threadIdx.x; i < sizeof(bins) / 4u; i += kHistThreads) bins[i] = 0u;
    __syncthreads();
    grid_dependency_wait();
    grid_dependency_launch_next();
    uint32_t* mine = bins + (OWN ? threadIdx.x : (threadIdx.x >> 5) * kBins);

    const uint64_t rows = (n + 31u) >> 5;
    const uint64_t num_words = (n * BITS + 31u) >> 5;
    for (uint64_t row = (uint64_t)blockIdx.x * kHistThreads + threadIdx.x; row < rows;
         row += (uint64_t)gridDim.x * kHistThreads) {
        const uint32_t valid = (row * 32u + 32u <= n) ? 32u : (uint32_t)(n - row * 32u);
        uint32_t w[BITS];
#pragma unroll
        for (int j = 0; j < BITS; ++j) w[j] = (row * BITS + j < num_words) ? __ldg(packed + row * BITS + j) : 0u;
#pragma unroll
        for (int e = 0; e < 32; ++e) {
            const int bit = e * BITS, wi = bit >> 5, sh = bit & 31;
            const uint32_t v = (sh + BITS <= 32) ? (w[wi] >> sh) : __funnelshift_r(w[wi], w[(wi + 1) % BITS], sh);
            if ((uint32_t)e < valid) atomicAdd(mine + (v & (kBins - 1u)) * kStep, 1u);
        }
    }
    __syncthreads();
    if constexpr (OWN) {
        // a warp adds up the counters of one code at a time
        for (uint32_t b = threadIdx.x >> 5; b < kBins; b += kWarps) {
            uint32_t s = 0u;
#pragma unroll
            for (uint32_t t = 0; t < (uint32_t)kHistThreads; t += 32u) s += bins[b * kHistThreads + t + (threadIdx.x & 31u)];
            s = __reduce_add_sync(0xFFFFFFFFu, s);
            if ((threadIdx.x & 31u) == 0u && s != 0u) atomicAdd(hist + b, (unsigned long long)s);
        }
    } else {
        for (uint32_t b = threadIdx.x; b < kBins; b += kHistThreads) {
            unsigned long long s = 0ull;
#pragma unroll
            for (uint32_t w = 0; w < kWarps; ++w) s += bins[w * kBins + b];
            if (s) atomicAdd(hist + b, s);
        }
    }
}

}  // namespace dq
