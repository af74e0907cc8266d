// Encode kernel for every bucket size: per-bucket scale, dither, quantize, (coset), pack -- one pass over the gradient
// (Eq. (DQSG) and Algorithm 1, worker steps; nested encoder equation and Algorithm 2, workers in P2).
//
// A group is 8 consecutive elements: two Philox blocks (one of the 16-bit stream), 32 bytes of the gradient and exactly
// `bits` bytes of the stream, and it never straddles a bucket.  A lane takes R groups that lie 32 groups apart, so every
// load and store of a warp is contiguous.  A CTA owns a window of whole buckets, or a cluster of CTAs owns one bucket
// that is too large for a CTA; the lanes' maxima meet in the bucket's scale (within the warp, through shared memory, or
// over the cluster's distributed shared memory), then every lane quantizes its groups from registers.  The gradient is
// read once, whatever the bucket size, and the hardware's block scheduler balances the load.
//   R = 1 for gradients that do not fill the GPU: the most lanes, the shortest chain per lane.
//   R = 4 for longer ones: what a warp costs once (indices, round keys, reduction, gain) is
//     spread over 32 elements per lane.
//
// What bounds it at large n: the multiplier pipe (about four wide multiplies of four cycles each per dither value) and
// instruction issue; at small n the latency of launch, load and one Philox chain.  Against a tile pipeline with a row
// of 32 elements per lane (plain loads where the tiles do not fit): n = 124.4 M, B = 4096, 3 bits 123.0 -> 112.4 us;
// n = 11.7 M, B = 2048 17.8 -> 14.3 us; n = 25.6 M, B = 1536 46.1 -> 34.2 us; n = 1.66 M, B = 16384, K = 3
// 11.7 -> 5.0 us; n = 266,610 3.9 -> 2.6 us.
#pragma once

#include "dq_device.cuh"
#include "dq_encode.cuh"

namespace dq {

template <int R> constexpr int kDirectMaxThreads = R == 1 ? 1024 : 256;
template <int R> constexpr int kDirectMaxCluster = 65536 / (8 * R * kDirectMaxThreads<R>);

// The kernels come in two kinds.  kDirectAhead makes most dithers before the first use of the elements and takes 80 registers
// (R = 1: 48); kDirectDense makes two at most and is held to 64 (40), for more resident CTAs where the shape leaves the GPU
// waiting for latency or for a second wave: see the dispatch.
enum DirectKind : int { kDirectAhead = 0, kDirectDense = 1 };
template <int R> constexpr uint32_t kDenseMaxThreads = R == 1 ? 768 : 256;
constexpr uint32_t direct_registers(int R, int kind)
{
    return R == 1 ? (kind == kDirectAhead ? 48u : 40u) : kind == kDirectAhead ? 80u : 64u;
}

// Groups of a lane whose dither is made before the first use of its elements.  With none, a CTA computes nothing while it
// waits for memory, and then for the maxima of its other warps (n = 11.7 M, B = 2048, 2 bits: 14.1 us with none, 13.4 with one,
// 13.1 two, 12.7 three, 12.8 four; 25.6 M: 25.4, 24.5, 24.1, 23.7, 23.7; B = 8192: 27.2, 25.6, 25.0, 24.3, 24.3; n = 124.4 M,
// 3 bits: 112.2, 109.4, 109.0, 107.8, 108.3).  All four fit beside the elements with the 16-bit stream (25.6 M: 19.7 us
// with none, 18.8 three, 18.4 four).  Two groups per Philox pass instead of one: no difference (23.8).  In the dense kernels two
// fit beside the elements but for 8 bytes; a draw of 490 encodes with four groups per lane takes 1.03 of the time with none, 1.006
// with one.  One-group lanes: n = 1.2 M, B = 2048 2.65 us with none, 2.50 with its one; 0.6 M, B = 16384 3.53 and 3.28.
template <int R, int DITH, int KIND> constexpr int kDitherAhead = R == 1 ? 1 : KIND == kDirectDense ? 2 : DITH == 16 ? 4 : 3;

// How the lanes' maxima meet in a bucket's scale.  Where a bucket is a power-of-two number of chunks the warp needs
// neither a barrier nor a gain (a division) per chunk: n = 25.6 M, 2 bits: bucket 1024 28.8 -> 26.5 us, 512 29.0 -> 28.0,
// 256 30.6 -> 28.7 (one redux per chunk instead of five shuffles).
enum DirectReduce : uint32_t {
    kPartOfWarp = 0,      // a bucket is an aligned power-of-two part of a chunk of 32 groups
    kTwoChunks = 1,       // a bucket is two of a warp's four chunks
    kWarpIsBucket = 2,    // a bucket is what a warp takes: no barrier, one gain
    kWarpInBucket = 3,    // a warp lies within one bucket: shared memory, one gain
    kAnywhere = 4         // anything else: shared memory, lane by lane
};

struct DirectArgs {
    const float* grad;
    uint32_t* packed;
    float* scale;
    uint64_t n;                   // elements in the gradient
    uint64_t num_bytes;           // 4 * packed words of the gradient
    uint32_t num_groups;          // groups that touch a packed word (a multiple of 4)
    uint32_t whole_groups;        // n / 8
    uint32_t groups_per_bucket;
    uint32_t groups_per_window;   // groups_per_bucket * buckets_per_window
    uint32_t buckets_per_window;  // 1 when a cluster shares a bucket
    uint32_t cluster;             // CTAs per bucket, 1 unless a bucket is larger than a CTA
    uint32_t bucket_magic;        // group of the window -> bucket: (group * bucket_magic) >> 22
    uint32_t reduce;              // DirectReduce
    uint32_t gains;               // further gains than the first chunk's: 0 none, 1 the third's, 2 every chunk's (a count,
                                  // not the enum, in the loop over chunks: tests of `reduce` there made 2048 1.5 % slower)
    uint32_t grad_align32;        // grad is 32-byte aligned
    float gain_num;               // DQSG: s = (L-1)/2;  NDQSG: A = alpha * M1
    int32_t kmax;                 // DQSG: L - 1
    uint32_t K;                   // NDQSG: coarse ratio
    uint32_t K_offset;            // NDQSG any K: multiple of K that is >= 2^22
    uint32_t K_magic;             // NDQSG any K: ceil(2^32 / K)
    uint32_t first_group;         // index of grad[0]'s group in the whole gradient (0 unless a bucket range is encoded):
                                  // only the dither counters see it
    uint32_t late_launch;         // the next kernel is let in at the end of this one and not right after the wait
    uint32_t early_read;          // } see the kernel and EncodeArgs
    uint32_t early_store;         // }
    f32x2 shift, magic, two, off; // pairs of equal values: DQSG s; 1.5 * 2^23; scale and offset of the dither
    PhiloxStream ps;
};

// Threads per CTA, buckets per CTA and CTAs per bucket for buckets of `g` groups.  Among the CTAs of 128 threads and
// more the one with the fewest idle lanes is taken, the smallest of equals; a bucket that does not fit one CTA is cut
// evenly over a cluster.
struct DirectShape { uint32_t threads, buckets, cluster; };

inline DirectShape direct_shape(uint32_t g, int R)
{
    const uint32_t per_warp = 32u * (uint32_t)R;
    const uint32_t most = (uint32_t)(R == 1 ? kDirectMaxThreads<1> : kDirectMaxThreads<4>);
    auto threads_for = [&](uint32_t groups) { return (groups + per_warp - 1u) / per_warp * 32u; };
    if (threads_for(g) > most) {
        uint32_t size = 2u;                     // (cluster sizes are powers of two)
        while (threads_for((g + size - 1u) / size) > most) size *= 2u;
        return {threads_for((g + size - 1u) / size), 1u, size};
    }
    DirectShape best = {0u, 0u, 1u};
    for (uint32_t k = 1u; threads_for(k * g) <= most; ++k) {
        const uint32_t t = threads_for(k * g);
        if (t < 128u && threads_for((k + 1u) * g) <= most) continue;
        // more groups per thread than the best so far
        if (best.threads == 0u || (uint64_t)k * best.threads > (uint64_t)best.buckets * t) best = {t, k, 1u};
        if (t / 32u * per_warp == k * g) break;
    }
    return best;
}

// The dither values of a group as pairs.  p0: first Philox product (M0 * counter) of the group's first block.
template <int DITH>
__device__ __forceinline__ void dither_group8(uint64_t p0, const DirectArgs& args, f32x2 (&delta)[4])
{
    constexpr int N = (DITH == 16) ? 1 : 2;
    uint32_t hi[N], lo[N], rnd[N][4];
#pragma unroll
    for (int j = 0; j < N; ++j) {
        const uint64_t p = p0 + (uint64_t)j * kPhiloxM0;
        hi[j] = (uint32_t)(p >> 32);
        lo[j] = (uint32_t)p;
    }
    philox4x32_10_after_first<N>(hi, lo, args.ps, rnd);
#pragma unroll
    for (int e = 0; e < 4; ++e) delta[e] = fma2(dither_bits2<DITH>(rnd, 2 * e), args.two, args.off);
}

// The codes of a group: 8 * BITS bits in ceil(BITS / 4) words.  x: the elements as pairs; aa: the bucket's gain twice.
template <int BITS, int MODE>
__device__ __forceinline__ void encode_group8(const f32x2* x, const f32x2 (&delta)[4], f32x2 aa, const DirectArgs& args,
                                              uint32_t (&out)[(BITS + 3) / 4])
{
    uint32_t sr = 0u;
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        // v = fma(g, a, delta); DQSG: w = v + s; then round to nearest even
        f32x2 v = fma2(x[e], aa, delta[e]);
        if constexpr (MODE == kEncDqsg) v = add2(v, args.shift);
        float t0, t1;
        unpack2(add2(v, args.magic), t0, t1);
        push_code<BITS>(sr, code_of<MODE>(t0, args), 2 * e, out);
        push_code<BITS>(sr, code_of<MODE>(t1, args), 2 * e + 1, out);
    }
    if constexpr (BITS % 4 != 0) out[BITS / 4] = sr >> (32 - 8 * BITS % 32);
}

// The BITS bytes of a whole group.
template <int BITS, int NW>
__device__ __forceinline__ void store_group8(uint8_t* dst, const uint32_t (&out)[NW])
{
    if constexpr (BITS == 8) {
        *reinterpret_cast<uint2*>(dst) = make_uint2(out[0], out[1]);
    } else if constexpr (BITS == 4) {
        *reinterpret_cast<uint32_t*>(dst) = out[0];
    } else if constexpr (BITS % 2 == 0) {
#pragma unroll
        for (int j = 0; j < BITS / 2; ++j)
            reinterpret_cast<uint16_t*>(dst)[j] = (uint16_t)(out[j >> 1] >> (16 * (j & 1)));
    } else {
#pragma unroll
        for (int j = 0; j < BITS; ++j) dst[j] = (uint8_t)(out[j >> 2] >> (8 * (j & 3)));
    }
}

// The last group(s): codes past the end are cleared, and only bytes of existing words are written.
template <int BITS, int NW>
__device__ __forceinline__ void store_group8_tail(uint8_t* packed, uint64_t byte, const uint32_t (&out)[NW], uint32_t nvalid,
                                                  uint64_t num_bytes)
{
#pragma unroll
    for (int j = 0; j < BITS; ++j) {
        const int32_t keep = (int32_t)(nvalid * BITS) - 8 * j;
        const uint32_t m = (keep >= 8) ? 0xFFu : (keep <= 0) ? 0u : ((1u << keep) - 1u);
        if (byte + j < num_bytes) packed[byte + j] = (uint8_t)((out[j >> 2] >> (8 * (j & 3))) & m);
    }
}

// max over the warp of non-negative floats (their bit patterns order like the values).
__device__ __forceinline__ uint32_t warp_max(uint32_t v) { return __reduce_max_sync(0xFFFFFFFFu, v); }

// The maximum over the CTAs of a cluster of their values `mine`; called by every thread.  part_max: this CTA's copy of
// the values.  The caller has executed barrier.cluster.arrive.
__device__ __forceinline__ uint32_t cluster_max(uint32_t mine, uint32_t part, uint32_t* part_max, uint32_t cluster)
{
    asm volatile("barrier.cluster.wait.aligned;" ::: "memory");          // every CTA is here: tell each of them
    if (threadIdx.x < cluster) {
        uint32_t remote;
        asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(smem_u32(part_max + part)), "r"(threadIdx.x));
        asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(remote), "r"(mine) : "memory");
    }
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    uint32_t m = 0u;
    for (uint32_t c = 0; c < cluster; ++c) m = max(m, part_max[c]);
    return m;
}

template <int BITS, int MODE, int DITH, int R, int KIND>
__global__ void __launch_bounds__(KIND == kDirectDense ? kDenseMaxThreads<R> : kDirectMaxThreads<R>,
                                  R == 1 ? (KIND == kDirectDense ? 2 : 1) : (KIND == kDirectDense ? 4 : 3))
encode_direct_kernel(const __grid_constant__ DirectArgs args)
{
    constexpr int NW = (BITS + 3) / 4;
    constexpr uint32_t kBlocks = (DITH == 16) ? 1u : 2u;       // Philox blocks of a group
    __shared__ uint32_t slot[kDirectMaxThreads<R> * R / 4];    // per bucket of the window (a bucket has 4 groups or more)
    __shared__ uint32_t part_max[kDirectMaxCluster<R>];

    const uint32_t tid = threadIdx.x, lane = tid & 31u;
    const uint32_t gpb = args.groups_per_bucket, gpw = args.groups_per_window;
    // A launch that overlaps with its predecessor by the caller's flags lets its successor in at once, but for its last
    // cluster, which has no work: that one waits for the predecessor first.  The successor, which may store without
    // waiting, therefore starts only when everything before this grid is complete (see launch_overlapped), and this grid
    // does not complete before its predecessor, on which a later kernel relies.
    if (args.early_read != 0u) {
        if (blockIdx.x >= gridDim.x - args.cluster) {
            grid_dependency_wait();
            grid_dependency_launch_next();
            return;
        }
        grid_dependency_launch_next();
    }
    uint32_t window = blockIdx.x, part = 0u;
    if (args.cluster > 1u) {
        window = blockIdx.x / args.cluster;
        part = blockIdx.x % args.cluster;
    }
    // the lane's groups: group + 32 c, c < R; `local` in the window, of which the warp's end at warp_end
    const uint32_t local = part * (blockDim.x * (uint32_t)R) + (tid >> 5) * (32u * R) + lane;
    const uint32_t group = window * gpw + local;
    const uint32_t warp_end = local - lane + 32u * (uint32_t)R;
    const bool whole = warp_end <= gpw && group - lane + 32u * (uint32_t)R <= args.whole_groups;     // (uniform in a warp)

    // first product of the lane's first block; those of its other blocks follow by 64-bit additions (M0 (k + j) is
    // M0 k + M0 j), which are cheaper than wide multiplies on the pipe that bounds the kernel
    const uint64_t p0 = (uint64_t)kPhiloxM0 * ((args.first_group + group) * kBlocks);
    // The dither does not depend on the gradient: the dithers of kAhead groups are made while the elements are on their way.
    constexpr int kAhead = kDitherAhead<R, DITH, KIND>;
    f32x2 delta[R][4];
    auto dither = [&](int c) { dither_group8<DITH>(p0 + (uint64_t)(32u * c * kBlocks) * kPhiloxM0, args, delta[c]); };
    // (a value that is used here is not computed further down)
    auto made = [&](int c) { asm volatile("" ::"l"(delta[c][0]), "l"(delta[c][1]), "l"(delta[c][2]), "l"(delta[c][3])); };
    if (args.early_read == 0u) {
        grid_dependency_wait();
        if (args.late_launch == 0u) grid_dependency_launch_next();
    }
    f32x2 x[4 * R];
    uint32_t mb[R];
    const float* g = args.grad + (uint64_t)group * 8u;
    auto nvalid_of = [&](int c) {
        const uint64_t i0 = (uint64_t)(group + 32u * c) * 8u;
        return (local + 32u * c >= gpw || i0 >= args.n) ? 0u : (uint32_t)min((uint64_t)8u, args.n - i0);
    };
    if (whole) {
#pragma unroll
        for (int c = 0; c < R; ++c) {
            if (args.grad_align32 != 0u) {
                asm volatile("ld.global.v4.b64 {%0, %1, %2, %3}, [%4];"
                             : "=l"(x[4 * c]), "=l"(x[4 * c + 1]), "=l"(x[4 * c + 2]), "=l"(x[4 * c + 3])
                             : "l"(g + 256 * c));
            } else {
                asm volatile("ld.global.v2.b64 {%0, %1}, [%2];" : "=l"(x[4 * c]), "=l"(x[4 * c + 1]) : "l"(g + 256 * c));
                asm volatile("ld.global.v2.b64 {%0, %1}, [%2];" : "=l"(x[4 * c + 2]), "=l"(x[4 * c + 3]) : "l"(g + 256 * c + 4));
            }
        }
    } else {
#pragma unroll
        for (int c = 0; c < R; ++c) {
            const uint32_t nvalid = nvalid_of(c);
#pragma unroll
            for (uint32_t e = 0; e < 4u; ++e)
                x[4 * c + e] = pack2(2u * e < nvalid ? __ldg(g + 256 * c + 2u * e) : 0.0f,
                                     2u * e + 1u < nvalid ? __ldg(g + 256 * c + 2u * e + 1u) : 0.0f);
        }
    }
#pragma unroll
    for (int c = 0; c < kAhead; ++c) {
        dither(c);
        made(c);
    }
    if (args.reduce >= kWarpInBucket) {
        for (uint32_t i = tid; i < args.buckets_per_window; i += blockDim.x) slot[i] = 0u;
        if (args.cluster > 1u) asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
        __syncthreads();
    }
#pragma unroll
    for (int c = 0; c < R; ++c) {
        float mx = 0.0f;
#pragma unroll
        for (int e = 0; e < 4; ++e) mx = max_pair(mx, x[4 * c + e]);
        mb[c] = __float_as_uint(mx);
    }
    if (args.reduce == kWarpInBucket) {
        uint32_t m = mb[0];
#pragma unroll
        for (int c = 1; c < R; ++c) m = max(m, mb[c]);
        m = warp_max(m);
        const uint32_t b = (args.cluster > 1u) ? 0u : (local * args.bucket_magic) >> 22;
        if (lane == 0u) atomicMax(slot + b, m);
        __syncthreads();
        m = slot[b];
        if (args.cluster > 1u) m = cluster_max(m, part, part_max, args.cluster);
#pragma unroll
        for (int c = 0; c < R; ++c) mb[c] = m;
    } else if (args.reduce == kPartOfWarp) {
        if (gpb == 32u) {
#pragma unroll
            for (int c = 0; c < R; ++c) mb[c] = warp_max(mb[c]);
        } else {
            for (uint32_t step = 1u; step < gpb; step <<= 1) {
#pragma unroll
                for (int c = 0; c < R; ++c) mb[c] = max(mb[c], __shfl_xor_sync(0xFFFFFFFFu, mb[c], step));
            }
        }
    } else if (R == 4 && args.reduce == kWarpIsBucket) {
        mb[0] = mb[1 % R] = mb[2 % R] = mb[3 % R] = warp_max(max(max(mb[0], mb[1 % R]), max(mb[2 % R], mb[3 % R])));
    } else if (R == 4 && args.reduce == kTwoChunks) {
        mb[0] = mb[1 % R] = warp_max(max(mb[0], mb[1 % R]));
        mb[2 % R] = mb[3 % R] = warp_max(max(mb[2 % R], mb[3 % R]));
    } else {
#pragma unroll
        for (int c = 0; c < R; ++c) {
            const uint32_t at = local + 32u * c;
            if ((gpb & 31u) == 0u) {             // the chunk lies within one bucket
                const uint32_t m = warp_max(mb[c]);
                if (lane == 0u && at < gpw) atomicMax(slot + ((at * args.bucket_magic) >> 22), m);
            } else if (at < gpw) {
                atomicMax(slot + ((at * args.bucket_magic) >> 22), mb[c]);
            }
        }
        __syncthreads();
#pragma unroll
        for (int c = 0; c < R; ++c) {
            const uint32_t at = local + 32u * c;
            mb[c] = at < gpw ? slot[(at * args.bucket_magic) >> 22] : 0u;
        }
    }
    uint32_t out[R][NW];
    f32x2 aa = both(bucket_gain(args.gain_num, __uint_as_float(mb[0])));
#pragma unroll
    for (int c = 0; c < R; ++c) {
        if (c > 0 && args.gains > (uint32_t)(c % 2)) aa = both(bucket_gain(args.gain_num, __uint_as_float(mb[c])));
        if (c >= kAhead) dither(c);
        encode_group8<BITS, MODE>(x + 4 * c, delta[c], aa, args, out[c]);
    }
    if (args.early_read == 0u) grid_dependency_launch_next();
    else if (args.early_store == 0u) grid_dependency_wait();
    const uint64_t byte = (uint64_t)group * (uint32_t)BITS;
    uint8_t* dst = reinterpret_cast<uint8_t*>(args.packed) + byte;
    if (whole) {
#pragma unroll
        for (int c = 0; c < R; ++c) store_group8<BITS>(dst + 32 * c * BITS, out[c]);
    } else {
#pragma unroll
        for (int c = 0; c < R; ++c)
            if (local + 32u * c < gpw && group + 32u * c < args.num_groups)
                store_group8_tail<BITS>(reinterpret_cast<uint8_t*>(args.packed), byte + 32u * c * BITS, out[c], nvalid_of(c),
                                        args.num_bytes);
    }
    // the scale leaves with the first group of a bucket
#pragma unroll
    for (int c = 0; c < R; ++c) {
        if (c > 0 && args.gains == 0u) break;    // a warp's first group is the only candidate
        const uint32_t at = local + 32u * c;
        const uint32_t b = (args.cluster > 1u) ? 0u : (at * args.bucket_magic) >> 22;
        if (at == b * gpb && at < gpw && group + 32u * c < args.num_groups)
            args.scale[(uint64_t)window * args.buckets_per_window + b] = __uint_as_float(mb[c]);
    }
}

}  // namespace dq
