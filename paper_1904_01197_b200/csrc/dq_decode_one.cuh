// Decoder of a single DQSG message (Algorithm 1, server steps 1 and 2, for one worker): what a server runs to have one
// worker's gradient, e.g. as a side information vector.
//
// A group is 8 consecutive elements, as in the direct encoder: two Philox blocks (one of the 16-bit stream) and exactly
// `bits` bytes of the stream.  A lane takes R groups that lie 32 groups apart, so the loads and stores of a warp are
// contiguous, every address but the first is a constant further on, and what a lane costs once is spread over 8 R elements;
// it requests the codes and scales of all of them, and the generator of the first group hides their latency.
//
// What bounds it: the multiplier pipe (82 %) and instruction issue (21 instructions per element, nine of them the generator).
// Against the general decoder with 16 elements per lane (28 instructions per element, issue slots 67 % used): n = 25.6 M,
// 3 bits 30.6 -> 25.2 us; 16-bit stream 28.4 -> 19.5; n = 4 M 6.2 -> 5.1; n = 266,037 1.71 -> 1.30.
#pragma once

#include "dq_decode.cuh"

namespace dq {

constexpr int kOneThreads = 128;

// kappa / s, by multiplication where s is a power of two.
__device__ __forceinline__ float one_gain(const DecWorker& wk, float kappa)
{
    return (wk.step_mul != 0.0f) ? __fmul_rn(kappa, wk.step_mul) : __fdiv_rn(kappa, wk.s);
}

// The R groups from `group` on; WHOLE: none of them touches the end of the range (else: up to `end`, the last group).
template <int DITH, int BITS, int R, bool WHOLE>
__device__ __forceinline__ void decode_one_chunk(const DecodeArgsOf<1>& args, uint32_t group, uint32_t last)
{
    constexpr int N = (DITH == 16) ? 1 : 2;                    // Philox blocks of a group
    constexpr int FORM = dec_form(kDecDqsg, BITS, DITH, 8), SHIFT = dec_shift(kDecDqsg, BITS, DITH, 8);
    const DecWorker& wk = args.w[0];
    using F = Field<BITS, 8>;
    auto bucket_of = [&](uint32_t g) {
        const uint32_t row = g >> 2;
        return (args.bucket_magic != 0u) ? (__umulhi(row, args.bucket_magic) >> args.bucket_shift) : (row >> args.bucket_shift);
    };
    // groups past the end repeat the last one and are not stored
    auto group_of = [&](int c) { return WHOLE ? group + 32u * (uint32_t)c : min(group + 32u * (uint32_t)c, last); };

    F field[R];
    float kappa[R];
    const uint32_t* words = wk.packed + (((uint64_t)group * (uint32_t)F::kBits) >> 5);
#pragma unroll
    for (int c = 0; c < R; ++c) {
        if constexpr (WHOLE) field[c].load_from(words + 8 * BITS * c);       // 32 groups are 8 * BITS words
        else field[c].load(wk.packed, group_of(c), true, args.n);
    }
    const uint32_t first_bucket = bucket_of(group_of(0));
    const bool one_bucket = WHOLE && R > 1 && first_bucket == bucket_of(group_of(R - 1));
    kappa[0] = __ldg(wk.scale + first_bucket);
    if (!one_bucket) {
#pragma unroll
        for (int c = 1; c < R; ++c) kappa[c] = __ldg(wk.scale + bucket_of(group_of(c)));
    }
    const uint64_t p0 = (uint64_t)kPhiloxM0 * (group * (uint32_t)N);
    float* const out = args.out + (uint64_t)group * 8u;
    uint32_t kappa_bits_max = 0u;
    f32x2 cc = 0ull;
    float up = 1.0f;
#pragma unroll
    for (int c = 0; c < R; ++c) {
        uint32_t hi[N], lo[N], rnd[N][4];
#pragma unroll
        for (int j = 0; j < N; ++j) {
            const uint64_t p = WHOLE ? p0 + (uint64_t)(32 * N * c + j) * kPhiloxM0
                                     : (uint64_t)kPhiloxM0 * (group_of(c) * (uint32_t)N + (uint32_t)j);
            hi[j] = (uint32_t)(p >> 32);
            lo[j] = (uint32_t)p;
        }
        philox4x32_10_after_first<N>(hi, lo, wk.ps, rnd);
        if (c == 0 || !one_bucket) {
            const uint32_t kb = __float_as_uint(kappa[c]) & 0x7FFFFFFFu;
            kappa_bits_max = max(kappa_bits_max, kb);
            float k = one_gain(wk, kappa[c]);
            // the scaled form's factor goes to the gain, or to the product where the gain might overflow
            if constexpr (SHIFT != 0) {
                const bool large = kb > args.kappa_limit;
                up = large ? pow2f(SHIFT) : 1.0f;
                k = large ? k : __fmul_rn(k, pow2f(SHIFT));
            }
            cc = both(k);
        }
        uint32_t f[F::kWords];
        field[c].align(WHOLE ? group : group_of(c), f);        // (32 groups do not change the position in a word)
        const f32x2 nz = args.neg_zero;
        f32x2 v[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int t = 2 * e;
            f32x2 x;
            if constexpr (FORM == kFormJoined && DITH == 16) {
                x = fma2(pack2(join16<BITS>(f, t, rnd[0][e], 0), join16<BITS>(f, t + 1, rnd[0][e], 1)), both(-kTwo127), wk.offset);
            } else if constexpr (FORM == kFormJoined) {
                x = fma2(pack2(join32<BITS>(f, t, rnd[t >> 2][t & 3], args.low22),
                               join32<BITS>(f, t + 1, rnd[t >> 2][(t & 3) + 1], args.low22)),
                         both(kTwo127), wk.offset);
            } else {
                const f32x2 nf = DITH == 16 ? fma2(dither_bits2<DITH>(rnd, t), both(-kTwo125), both(-kF16Offset))
                                            : fma2(dither_bits2<DITH>(rnd, t), both(-kTwo127), both(-kF32Offset));
                x = add2(add2(pack2(unpack_half_biased<BITS>(f, t, args.half_bias_bits),
                                    unpack_half_biased<BITS>(f, t + 1, args.half_bias_bits)), wk.offset), nf);
            }
            // (a sum that starts at +0: no negative zeros)
            v[e] = SHIFT != 0 ? fma2(fma2(cc, x, nz), both(up), 0ull) : add2(fma2(cc, x, nz), 0ull);
        }
        if constexpr (WHOLE) {
            store8(out + 256 * c, v, args.out_align32 != 0u);
        } else if (group + 32u * (uint32_t)c <= last) {
            const uint64_t i0 = (uint64_t)group_of(c) * 8u;
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                float a, b;
                unpack2(v[e], a, b);
                if (i0 + 2u * e < args.n) args.out[i0 + 2u * e] = a;
                if (i0 + 2u * e + 1u < args.n) args.out[i0 + 2u * e + 1u] = b;
            }
        }
    }
    if (args.status != nullptr && kappa_bits_max >= 0x7F800000u) atomicOr(args.status, 0x1u);
    grid_dependency_launch_next();                             // (late, as in the general decoder)
}

template <int DITH, int BITS, int R>
__global__ void __launch_bounds__(kOneThreads)
decode_one_kernel(const __grid_constant__ DecodeArgsOf<1> args)
{
    const uint32_t first_group = args.first_row * 4u, last = first_group + (uint32_t)args.num_groups - 1u;
    const uint32_t chunk = first_group + (blockIdx.x * (uint32_t)(kOneThreads / 32) + (threadIdx.x >> 5)) * (32u * R);
    const uint32_t group = chunk + (threadIdx.x & 31u);
    grid_dependency_wait();
    // the fields of a whole chunk end well before the stream does (uniform in a warp)
    if (((uint64_t)chunk + 32u * R) * 8u + 64u <= args.n) decode_one_chunk<DITH, BITS, R, true>(args, group, last);
    else decode_one_chunk<DITH, BITS, R, false>(args, group, last);
}

}  // namespace dq
