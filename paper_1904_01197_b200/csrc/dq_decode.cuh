// Fused decode-and-average kernel (Algorithm 1, server steps; nested decoder equation and Algorithm 2,
// server loop with the side information given as a vector, taken as the running mean, or taken as the
// reconstruction of message 0).
//
// One lane owns E consecutive elements (a group): E fp32 accumulators in registers, and per worker exactly E * bits
// packed bits.  A group never straddles a bucket (buckets are multiples of 32 elements), so a lane needs one scale
// per worker.  For every worker, in array order, the lane regenerates its E dithers (E / 4 Philox blocks, E / 8 with
// the 16-bit stream), reconstructs and accumulates; the packed words are requested before the Philox work (or one
// worker ahead), which hides their latency, the scale one worker ahead.  Side information is read once into the
// lane's own shared-memory slots, and so are the first Philox products, which are the same for every worker; the
// mean is written once in full 32-byte sectors.  Nothing is shared between lanes: there is no barrier, and the
// hardware's block scheduler balances the load.
//
// What bounds it: the multiplier pipe and instruction issue.  Each (element, worker) pair needs a quarter of a
// Philox block, 4.25 wide multiplies of four cycles each, before any reconstruction arithmetic; that arithmetic runs
// on packed pairs of fp32 values (half the instructions).
#pragma once

#include "dq_device.cuh"

namespace dq {

// Where the side information of the nested messages comes from: a vector given by the caller (or none at all: only
// DQSG messages), the running mean of the messages decoded so far, or the reconstruction of message 0.
enum DecSide : int { kSideGiven = 0, kSideRunning = 1, kSideFirst = 2 };

enum DecKind : uint32_t {
    kDecDqsg = 0, kDecNdqsgPow2 = 1, kDecNdqsgPow2Shrink = 2, kDecNdqsgAnyK = 3, kDecNdqsgAnyKShrink = 4
};

struct DecWorker {
    const uint32_t* packed;   // } addresses of the (virtual) whole-gradient buffers, see DecodeArgs
    const float* scale;       // }
    // Pairs of equal values (one 64-bit load each), for the form in which the routine works (DecForm; u = 2^-shift):
    f32x2 offset;         // joined: see there; biased: minus (DQSG: 4194304 + s - 1.5, NDQSG: 4194304 - 1.5)
    f32x2 neg_K;          // -K u
    f32x2 neg_K_code;     // -K in units of the tiny code
    f32x2 inv_K;          // 1/K rounded to nearest (exact when K is a power of two), over u
    PhiloxStream ps;
    uint32_t variant;     // DecKind * 8 + bits - 1: one jump selects the routine
    uint32_t group_end;   // index after the last worker of the run of equal variants that this worker belongs to
    float step_mul;       // DQSG: 1/s, NDQSG: 1/M1, when that divisor is a power of two (the division is then an
                          // exact multiplication); 0 otherwise
    float s;              // DQSG (L-1)/2
    float A;              // NDQSG alpha * M1 * u
    float M1;
    float alpha;
    float one_m_alpha2;   // 1 - alpha*alpha
    float rcp_count;      // running-mean mode: 1 / (number of workers before this one)
    float K;
};

struct DecodeHead {
    const float* side;
    float* out;
    uint32_t* status;
    // A call may cover the elements [first, n) of a longer gradient (first a multiple of the bucket size, 0 for a
    // whole gradient).  Groups, elements and buckets are then numbered as in the whole gradient -- which is what the
    // dither counters need -- and every pointer above and in w[] is the buffer's address minus the range's offset,
    // so that "pointer + global index" lands in the caller's buffer.
    uint64_t n;               // end of the range (element index)
    uint32_t first_row;       // first / 32
    uint32_t W;
    uint64_t num_groups;      // groups of E elements in the range (E = the launched instantiation's)
    uint32_t rows_per_bucket; // B / 32
    uint32_t bucket_shift;    // row -> bucket: (row * bucket_magic) >> 32 >> bucket_shift, or row >> bucket_shift
    uint32_t bucket_magic;    // when bucket_magic is 0 (power-of-two buckets); see set_bucket_division
    uint32_t has_side;        // the side information vector is read
    uint32_t out_align32;     // out is 32-byte aligned: whole groups leave in 32-byte stores
    uint32_t half_bias_bits;  // 0x4A800000 (bit pattern of 2^22), passed in so that it lives in a register
    uint32_t low22;           // 2^22 - 1, likewise
    uint32_t kappa_limit;     // bit pattern of the largest scale that the scaled forms of these messages take (see DecForm)
    float Wf;
    f32x2 neg_zero;           // -0.0 twice (see f32x2)           } constants that would otherwise be assembled from
    f32x2 magic, neg_magic;   // +-1.5 * 2^23 twice               } immediates again and again
    float invW;               // 1/W when W is a power of two, else 0
};

// Kernel parameters for up to MAXW workers.  A launch copies all of them: 0.8 us more for 64 workers (11 KB) than for 8,
// which counts for short gradients (kDecFewWorkers).
template <int MAXW>
struct DecodeArgsOf : DecodeHead {
    DecWorker w[MAXW];
};
using DecodeArgs = DecodeArgsOf<64>;
constexpr int kDecFewWorkers = 8;

// Division of a row index below 2^29 by rows_per_bucket as a multiplication: with s = floor(log2 d) and
// m = ceil(2^(32+s) / d), m d - 2^(32+s) < d < 2^(s+1) <= 2^(32+s) / 2^29, which is what makes
// floor(row m / 2^(32+s)) exact.
inline void set_bucket_division(DecodeHead& a)
{
    const uint32_t d = a.rows_per_bucket;
    uint32_t s = 0u;
    while ((2u << s) <= d) ++s;
    a.bucket_shift = s;
    a.bucket_magic = (d & (d - 1u)) == 0u ? 0u : (uint32_t)(((1ull << (32u + s)) + d - 1u) / d);
}

constexpr int kDecThreads = 128;
// Which variants a kernel holds.  With all forty routines in one kernel the compiler's register allocation and its
// choice between uniform and per-lane loads of a worker's constants cost routines up to 5 %, so the usual variants
// (DQSG, and NDQSG with a power-of-two K and no shrinkage, up to 4 bits) and the odd ones (the same with another K, the
// paper's K = 3 among them) have kernels of their own, and for long gradients every pair of one DQSG and one NDQSG width has
// (n = 25.6 M, W = 16, 3 bits and a vector 362 us with all, 375 with the usual ones, 348 with the pair; W = 8, 3 and 2 bits, side
// information from message 0 181, 181 and 179; running mean, W = 8, K = 3, n = 266,010 5.6 us with all, 5.4 with the odd ones,
// 2.4 M 22.6 and 21.8; but 11.7 M, in groups of 32, 91.5 and 92.3).
constexpr int kSetAll = 0, kSetUsual = 1, kSetOdd = 2, kSetAllFull = 3;      // (kSetAllFull: see dec_ctas_per_sm)
constexpr int pair_set(int dqsg_bits, int ndqsg_bits) { return 16 * dqsg_bits + ndqsg_bits; }

// Resident CTAs per SM that the register budget is set for.  E = 32 takes 80 registers (24 warps per SM) in the pair
// kernels: what a worker costs per lane (scale, gain, constants, loop: about 65 instructions) is spread over the most
// elements.  96 registers are 3 % faster for a given side information vector but 2 to 8 % slower otherwise (the compiler
// then loads a worker's constants lane by lane), 128 registers 7 % slower; the kernel with all routines wants 96.
// E = 16 and 8 take 64 registers (32 warps), but for 72 (28 warps) where all routines in one kernel spill at 64 and are faster
// without (E = 16, 32-bit stream: running mean, W = 8, 8 and 3 bits, n = 1.7 M 18.0 us with 64, 17.4 with 72; E = 8, 16-bit
// stream, W = 16, up to 1 M: 64 is 3 to 6 % slower).  The same routines at 64 (kSetAllFull) serve a grid that is one wave of
// eight CTAs per SM and would be two of seven (W = 2, n = 1.2 M, 16-bit stream and a vector 4.4 us, with 72 registers 5.1), and
// messages of 5 to 7 bits against a vector or none in groups of 8 (32-bit stream, W = 16, 5 bits, n = 128,073 8.7 us and 11.0;
// but 8 bits, 266,610 9.5 and 8.9).
constexpr int dec_ctas_per_sm(int dith, int E, int set)
{
    if (E == 32) return set == kSetAll ? 5 : 6;
    return set == kSetAll && (E == 16 ? dith == 32 : dith != 0) ? 7 : 8;
}

// How a routine forms k - s - delta (DQSG) and m - delta, q - delta (NDQSG) from the code and the random bits.  All forms
// round the same real numbers once, so they give the same bits; they differ in the number of packed instructions.
//   biased:  X = k - s + 1.5 from the float 2^22 + k, f = delta + 1.5 from the random bits, X - f.
//   joined:  code and random bits side by side in one mantissa, one multiply-add for both.  The join is an integer below
//            2^24, read as a (subnormal or small) float; with the 16-bit stream always possible (up to seven bits), with
//            the 32-bit stream where 22 + bits <= 24 and (NDQSG) m - delta is representable, so that q - delta follows
//            from it by another multiply-add.  Not in groups of 32 for DQSG with the 32-bit stream, where the biased form is
//            ahead in its own routines (W = 8, 2 bits, n = 25.6 M: joined 166.5 us, biased 158.6; in groups of 8, 266,610
//            4.45 and 4.56) and in the others of their kernel (side information from message 0, six bits, 11.7 M: 99.6 and
//            92.1).
//   tiny:    NDQSG up to four bits: the code in bits 23.. downwards of a float is an exact multiple of 2^-149, so that
//            m - delta and q - delta are one multiply-add each and no bias has to be taken off.
// The values of the last two forms are smaller than the real ones by 2^shift, because a multiply-add cannot scale by more than
// 2^127; gain and 1/K carry the factor, and groups with a scale where that could overflow or lose bits (kappa_limit, far
// above any gradient) are decoded again by decode_group_plain.
enum DecForm : int { kFormBiased = 0, kFormJoined = 1, kFormTiny = 2 };

__host__ __device__ constexpr int dec_form(uint32_t kind, int bits, int dith, int group)
{
    if (dith == 16) return bits <= 7 ? kFormJoined : kFormBiased;
    if (dith == 32 && kind == kDecDqsg) return bits <= 2 && group < 32 ? kFormJoined : kFormBiased;
    if (dith == 32) return bits == 1 ? kFormJoined : bits <= 4 ? kFormTiny : kFormBiased;
    return kFormBiased;
}

__host__ __device__ constexpr int dec_shift(uint32_t kind, int bits, int dith, int group)
{
    const int form = dec_form(kind, bits, dith, group);
    return form == kFormTiny ? bits - 2 : (form == kFormJoined && dith == 16) ? 6 : 0;
}

// Whether a kernel calls decode_group_plain.  Not where none of its routines is scaled: against a vector the call costs registers
// there (the pair of 3 and 2 bits spills 52 bytes with it; W = 8, n = 25.6 M 0.4 % slower).  Against message 0 and the running
// mean the compiler's allocation comes out better with the call, although it is never taken (the same pair 2 % faster).
__host__ __device__ constexpr bool may_be_plain(int set, int dith, int side, int group)
{
    return dith != 0 && (side != kSideGiven || set <= kSetAllFull || dec_shift(kDecDqsg, set / 16, dith, group) != 0 ||
                         dec_shift(kDecNdqsgPow2, set % 16, dith, group) != 0);
}

__host__ __device__ constexpr float pow2f(int e)
{
    float v = 1.0f;
    for (; e > 0; --e) v *= 2.0f;
    for (; e < 0; ++e) v *= 0.5f;
    return v;
}

// BITS bits of the stream from bit `start` on (a compile-time constant after unrolling) and what follows them.
template <int NF>
__device__ __forceinline__ uint32_t stream_from(const uint32_t (&f)[NF], int start, int bits)
{
    const int wi = start >> 5, sh = start & 31;
    if (sh == 0) return f[wi];
    if (sh + bits <= 32) return f[wi] >> sh;
    return __funnelshift_r(f[wi], f[(wi + 1) % NF], sh);
}

// Code of element `idx` of a group as the float 2^22 + code: the bit pattern of 2^22 with the code in mantissa
// bits 1.. (floats in [2^22, 2^23) step by 1/2).  Subtracting a constant then gives code - c exactly.
template <int BITS, int NF>
__device__ __forceinline__ float unpack_half_biased(const uint32_t (&f)[NF], int idx, uint32_t bias_bits)
{
    const int bit = idx * BITS;
    const int wi = bit >> 5;
    const int sh = bit & 31;
    constexpr uint32_t mask2 = ((1u << BITS) - 1u) << 1;
    uint32_t v;
    if (sh + BITS <= 32) {
        v = (sh == 0) ? (f[wi] << 1) : (f[wi] >> (sh - 1));
    } else {
        v = __funnelshift_r(f[wi], f[(wi + 1) % NF], sh - 1);
    }
    return __uint_as_float((v & mask2) | bias_bits);          // one logic op: (v & immediate) | register
}

// 16-bit stream, joined form: the complement of the code above the half-word.  Codes that share a shift are masked
// together, and one byte permutation takes the two bytes of the half-word, the code's byte, and zeros (the copies of that
// byte's clear top bit).
template <int BITS, int NF>
__device__ __forceinline__ float join16(const uint32_t (&f)[NF], int idx, uint32_t word, int high)
{
    constexpr uint32_t mask = (1u << BITS) - 1u;
    uint32_t v;
    int byte;
    if constexpr (8 % BITS == 0) {
        const int bit = idx * BITS;
        v = ~(f[bit >> 5] >> (bit & 7)) & (mask * 0x01010101u);
        byte = (bit >> 3) & 3;
    } else if constexpr (BITS == 3 || BITS == 6) {            // codes 24 bits apart
        constexpr int step = 24 / BITS;
        const int first = idx / (2 * step) * (2 * step) + idx % step;
        v = ~stream_from(f, first * BITS, (NF * 32 - first * BITS >= 24 + BITS) ? 24 + BITS : BITS) & (mask * 0x01000001u);
        byte = idx % (2 * step) >= step ? 3 : 0;
    } else {
        v = ~stream_from(f, idx * BITS, BITS) & mask;
        byte = 0;
    }
    const uint32_t b = 4u + (uint32_t)byte;
    uint32_t d;
    asm("prmt.b32 %0, %1, %2, %3;" : "=r"(d) : "r"(word), "r"(v), "r"((high ? 0x32u : 0x10u) | (b << 8) | ((b | 8u) << 12)));
    return __uint_as_float(d);
}

// 32-bit stream, joined form: the code above the complement of the 22 random bits.
template <int BITS, int NF>
__device__ __forceinline__ float join32(const uint32_t (&f)[NF], int idx, uint32_t word, uint32_t low22)
{
    const uint32_t v = __funnelshift_r(word, f[(idx * BITS) >> 5] >> ((idx * BITS) & 31), 10);
    return __uint_as_float((v & ((1u << (22 + BITS)) - 1u)) ^ low22);      // one logic op: (v & immediate) ^ register
}

// The code in the BITS bits below bit 24 (one bit: below bit 23).
template <int BITS, int NF>
__device__ __forceinline__ float tiny_code(const uint32_t (&f)[NF], int idx)
{
    constexpr uint32_t mask = (1u << BITS) - 1u;
    const int bit = idx * BITS;
    if constexpr (8 % BITS == 0) {
        const int up = 8 - BITS - (bit & 7);                  // to the top of its byte
        const uint32_t v = (up >= 0 ? f[bit >> 5] << up : f[bit >> 5] >> -up) & ((mask << (8 - BITS)) * 0x01010101u);
        return __uint_as_float(__byte_perm(v, 0u, 0x4044u | (uint32_t)(((bit >> 3) & 3) << 8)));
    } else {
        const int sh = (bit & 31) - (24 - BITS), wi = bit >> 5;
        const uint32_t v = (bit & 31) + BITS > 32 ? __funnelshift_r(f[wi], f[(wi + 1) % NF], sh)
                           : sh >= 0              ? f[wi] >> sh
                                                  : f[wi] << -sh;
        return __uint_as_float(v & (mask << (24 - BITS)));
    }
}

constexpr int gcd_of(int a, int b) { return b == 0 ? a : gcd_of(b, a % b); }

// The E * BITS bits of group `g`, aligned to bit 0 of f[0].  With `careful` (the last groups of the gradient) every
// word is checked against the end of the stream.
template <int BITS, int E>
struct Field {
    static constexpr int kBits = E * BITS;
    static constexpr int kWords = (kBits + 31) / 32;
    static constexpr int kAlign = gcd_of(kBits, 32);                       // a field starts at a multiple of this
    static constexpr int kLoads = (32 - kAlign + kBits + 31) / 32;         // words that a field can touch
    uint32_t w[kLoads];

    __device__ __forceinline__ void load(const uint32_t* packed, uint32_t g, bool careful, uint64_t n)
    {
        const uint64_t wi = ((uint64_t)g * (uint32_t)kBits) >> 5;
        const uint32_t* p = packed + wi;
        if (careful) {
            const uint64_t num_words = (n * (uint32_t)BITS + 31u) >> 5;
#pragma unroll
            for (int j = 0; j < kLoads; ++j) w[j] = (wi + j < num_words) ? __ldg(p + j) : 0u;
            return;
        }
        load_from(p);
    }

    // (p: the word that holds the field's first bit; every word that a field can touch is there)
    __device__ __forceinline__ void load_from(const uint32_t* p)
    {
        if constexpr (kAlign == 32 && kLoads % 4 == 0) {
#pragma unroll
            for (int j = 0; j < kLoads; j += 4) {
                const uint4 v = __ldg(reinterpret_cast<const uint4*>(p + j));
                w[j] = v.x; w[j + 1] = v.y; w[j + 2] = v.z; w[j + 3] = v.w;
            }
        } else if constexpr (kAlign == 32 && kLoads % 2 == 0) {
#pragma unroll
            for (int j = 0; j < kLoads; j += 2) {
                const uint2 v = __ldg(reinterpret_cast<const uint2*>(p + j));
                w[j] = v.x; w[j + 1] = v.y;
            }
        } else {
#pragma unroll
            for (int j = 0; j < kLoads; ++j) w[j] = __ldg(p + j);
        }
    }

    __device__ __forceinline__ void align(uint32_t g, uint32_t (&f)[kWords]) const
    {
        const uint32_t sh = (kAlign == 32) ? 0u : ((g * (uint32_t)kBits) & 31u);
#pragma unroll
        for (int j = 0; j < kWords; ++j) {
            if (kAlign == 32) f[j] = w[j];
            else if (j + 1 < kLoads) f[j] = __funnelshift_r(w[j], w[j + 1], sh);
            else f[j] = w[j] >> sh;
        }
    }
};

// State of a lane while it walks over the workers.
struct DecLane {
    uint32_t group, bucket, kappa_bits_max;
    uint32_t slot;              // shared-memory address of the lane's first 16-byte slot (slots are kDecThreads apart)
    uint32_t first[2];          // first Philox product (hi, lo) of a lane with one block
    float kappa_next;
    bool careful;
};

// Decodes one group and stores its mean, element by element and with nothing scaled: for groups with a scale near the end of
// the fp32 range (kappa_limit).  (It stores its results
// itself: an array in local memory for them cost every call of the kernel, n = 266,610, W = 8 6.5 us instead of 6.3.)
template <int DITH, int SIDE, int E, typename Args>
__device__ __noinline__ void decode_group_plain(const Args& args, uint32_t group, uint32_t bucket)
{
#pragma unroll 1
    for (uint32_t e = 0; e < (uint32_t)E; ++e) {
        const uint64_t i = (uint64_t)group * (uint32_t)E + e;
        if (i >= args.n) return;
        float acc = 0.0f, y = (SIDE == kSideGiven && args.has_side != 0u) ? __ldg(args.side + i) : 0.0f;
#pragma unroll 1
        for (uint32_t w = 0; w < args.W; ++w) {
            const DecWorker& wk = args.w[w];
            const uint32_t bits = (wk.variant & 7u) + 1u, kind = wk.variant >> 3;
            const uint64_t bit = i * bits;
            const uint32_t sh = (uint32_t)bit & 31u;
            uint32_t code = __ldg(wk.packed + (bit >> 5)) >> sh;
            if (sh + bits > 32u) code |= __ldg(wk.packed + (bit >> 5) + 1u) << (32u - sh);
            const float k = (float)(code & ((1u << bits) - 1u)), kappa = __ldg(wk.scale + bucket);
            const uint64_t p = (uint64_t)kPhiloxM0 * (uint32_t)(i / (DITH == 16 ? 8u : 4u));
            const uint32_t hi[1] = {(uint32_t)(p >> 32)}, lo[1] = {(uint32_t)p};
            uint32_t rnd[1][4];
            philox4x32_10_after_first<1>(hi, lo, wk.ps, rnd);
            const uint32_t at = (uint32_t)i & (DITH == 16 ? 7u : 3u), which = DITH == 16 ? at >> 1 : at;
            const uint32_t word = which == 0u ? rnd[0][0] : which == 1u ? rnd[0][1] : which == 2u ? rnd[0][2] : rnd[0][3];
            const float delta = DITH == 16 ? __fmaf_rn((float)((word >> (16u * (at & 1u))) & 0xFFFFu), 0x1p-16f, -kD16Offset)
                                           : __fmaf_rn((float)(word >> 10), 0x1p-22f, -kD32Offset);
            float gt;
            if (kind == kDecDqsg) {
                gt = __fmul_rn(__fdiv_rn(kappa, wk.s), __fsub_rn(__fsub_rn(k, wk.s), delta));
            } else {
                const float a = (kappa >= 0x1p-100f) ? __fdiv_rn(__fmul_rn(wk.alpha, wk.M1), kappa) : 0.0f;
                const float c = __fdiv_rn(__fmul_rn(wk.alpha, kappa), wk.M1);
                if (SIDE == kSideRunning) y = __fmul_rn(acc, wk.rcp_count);
                const float r = __fmaf_rn(-y, a, __fsub_rn(k, delta));
                const float d = __fsub_rn(__fmaf_rn(-wk.K, rintf(__fdiv_rn(r, wk.K)), k), delta);
                gt = wk.alpha == 1.0f ? __fmul_rn(c, d) : __fmaf_rn(c, d, __fmul_rn(wk.one_m_alpha2, y));
            }
            acc = __fadd_rn(acc, gt);
            if (SIDE == kSideFirst && w == 0u) y = acc;
        }
        if (args.W > 1u) acc = (args.invW != 0.0f) ? __fmul_rn(acc, args.invW) : __fdiv_rn(acc, args.Wf);
        args.out[i] = acc;
    }
}

// The contributions of the workers [w, w_end), a run of equal variants: the same routine for each, so the jump on the
// variant is taken once per run and not once per worker (Algorithm 2's groups P1 and P2 are two runs).
//   DQSG:  g~ = (kappa/s) ((k - s) - delta)
//   NDQSG: r = (m - delta) - y a;  jj = rint(r / K);  q1^ = m - K jj;  g~ = beta (q1^ - delta) [+ (1-alpha^2) y]
// AHEAD: the packed words are requested one worker ahead (see kWordsAhead).
//
// Requesting the words a worker ahead costs registers and pays only where a worker is done soonest: the 16-bit stream's
// DQSG messages (W = 8, n = 11.7 M: 54.9 -> 52.4 us); elsewhere the Philox work hides the latency.
template <int DITH, uint32_t KIND, int E, int SET>
constexpr bool kWordsAhead = DITH == 16 && KIND == kDecDqsg && E == 32 && SET != kSetAll;

template <int BITS, uint32_t KIND, int DITH, int SIDE, int E, bool AHEAD, typename Args>
__device__ __forceinline__ void decode_run(const Args& args, uint32_t w, uint32_t w_end, DecLane& ln,
                                           f32x2 (&acc)[E / 2])
{
    constexpr bool RUN = SIDE == kSideRunning;
    constexpr bool ANY_K = KIND == kDecNdqsgAnyK || KIND == kDecNdqsgAnyKShrink;
    constexpr bool SHRINK = KIND == kDecNdqsgPow2Shrink || KIND == kDecNdqsgAnyKShrink;
    constexpr int FORM = dec_form(KIND, BITS, DITH, E), SHIFT = dec_shift(KIND, BITS, DITH, E);
    constexpr int EPB = (DITH == 16) ? 8 : 4;       // elements per Philox block
    constexpr int N = E / EPB;                      // blocks of the group
    constexpr int P = N < 2 ? N : 2;                // blocks in flight
    Field<BITS, E> field;
    if constexpr (AHEAD) field.load(args.w[w].packed, ln.group, ln.careful, args.n);
#pragma unroll 1
    for (; w < w_end; ++w) {
        const DecWorker& wk = args.w[w];
        if constexpr (!AHEAD) field.load(wk.packed, ln.group, ln.careful, args.n);
        uint32_t f[Field<BITS, E>::kWords];
        f32x2 cc, na = 0ull;
        const f32x2 nz = args.neg_zero;
#pragma unroll
        for (int h = 0; h < N / P; ++h) {
            uint32_t rnd[P][4];
            if constexpr (DITH != 0) {
                uint32_t hi[P], lo[P];
                if constexpr (N == 1) {
                    hi[0] = ln.first[0];
                    lo[0] = ln.first[1];
                } else {
                    asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];"
                                 : "=r"(hi[0]), "=r"(lo[0]), "=r"(hi[1]), "=r"(lo[1])
                                 : "r"(ln.slot + (uint32_t)((E / 4 + h) * kDecThreads * 16)));
                }
                philox4x32_10_after_first<P>(hi, lo, wk.ps, rnd);
            }
            if (h == 0) {
                // the Philox work above hides the latency of the words; the scale was requested a worker ago
                field.align(ln.group, f);
                if constexpr (AHEAD) {
                    if (w + 1u < w_end) field.load(args.w[w + 1u].packed, ln.group, ln.careful, args.n);
                }
                const float kappa = ln.kappa_next;
                if (w + 1u < args.W) ln.kappa_next = __ldg(args.w[w + 1u].scale + ln.bucket);
                const uint32_t kb = __float_as_uint(kappa) & 0x7FFFFFFFu;
                ln.kappa_bits_max = (kb > ln.kappa_bits_max) ? kb : ln.kappa_bits_max;
                // kappa / s and alpha kappa / M1: a division by a power of two is an exact multiplication
                float c;
                if constexpr (KIND == kDecDqsg) {
                    c = (wk.step_mul != 0.0f) ? __fmul_rn(kappa, wk.step_mul) : __fdiv_rn(kappa, wk.s);
                } else {
                    na = both((kappa >= 0x1p-100f) ? -__fdiv_rn(wk.A, kappa) : -0.0f);
                    const float ak = __fmul_rn(wk.alpha, kappa);
                    c = (wk.step_mul != 0.0f) ? __fmul_rn(ak, wk.step_mul) : __fdiv_rn(ak, wk.M1);        // beta
                }
                if constexpr (SHIFT != 0) c = __fmul_rn(c, pow2f(SHIFT));
                cc = both(c);
            }
#pragma unroll
            for (int qq = 0; qq < P * EPB / 4; ++qq) {      // four elements at a time (one 16-byte slot of y)
                const int q = h * (P * EPB / 4) + qq;
                f32x2 y[2] = {0ull, 0ull};
                if constexpr (KIND != kDecDqsg && !RUN)
                    asm volatile("ld.shared.v2.b64 {%0, %1}, [%2];"
                                 : "=l"(y[0]), "=l"(y[1])
                                 : "r"(ln.slot + (uint32_t)(q * kDecThreads * 16))
                                 : "memory");
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const int t = 4 * q + 2 * e;                           // element of the group
                    const int tr = 4 * qq + 2 * e;                         // ... of the blocks in rnd
                    // x = u (k - s - delta) or u (m - delta); biased: X and nf with x = X + nf; tiny: code and nf
                    f32x2 x, X = 0ull, nf = 0ull;
                    if constexpr (FORM == kFormJoined && DITH == 16) {
                        const uint32_t word = rnd[tr >> 3][(tr & 7) >> 1];
                        x = fma2(pack2(join16<BITS>(f, t, word, 0), join16<BITS>(f, t + 1, word, 1)), both(-kTwo127), wk.offset);
                    } else if constexpr (FORM == kFormJoined) {
                        x = fma2(pack2(join32<BITS>(f, t, rnd[tr >> 2][tr & 3], args.low22),
                                          join32<BITS>(f, t + 1, rnd[tr >> 2][(tr & 3) + 1], args.low22)),
                                 both(kTwo127), wk.offset);
                    } else if constexpr (FORM == kFormTiny) {
                        nf = fma2(dither_bits2<32>(rnd, tr), both(-kTwo127 * pow2f(-SHIFT)), both(kD32Offset * pow2f(-SHIFT)));
                        X = pack2(tiny_code<BITS>(f, t), tiny_code<BITS>(f, t + 1));
                        x = fma2(X, both(kTwo127), nf);
                    } else {
                        if constexpr (DITH == 0) nf = both(-1.5f);
                        else if constexpr (DITH == 16) nf = fma2(dither_bits2<16>(rnd, tr), both(-kTwo125), both(-kF16Offset));
                        else nf = fma2(dither_bits2<32>(rnd, tr), both(-kTwo127), both(-kF32Offset));
                        X = add2(pack2(unpack_half_biased<BITS>(f, t, args.half_bias_bits),
                                       unpack_half_biased<BITS>(f, t + 1, args.half_bias_bits)), wk.offset);
                        x = add2(X, nf);
                    }
                    f32x2 gt;
                    if constexpr (KIND == kDecDqsg) {
                        gt = fma2(cc, x, nz);                              // c ((k - s) - delta)
                    } else {
                        // side information: the given vector, the reconstruction of message 0, or (Algorithm 2 as
                        // written) the mean of the reconstructions accumulated so far
                        const f32x2 yy = RUN ? fma2(acc[t >> 1], both(wk.rcp_count), nz) : y[e];
                        const f32x2 r = fma2(yy, na, x);
                        f32x2 jj;
                        if constexpr (ANY_K) {
                            // r / K rounded to nearest from the correctly rounded 1/K: one residual correction leaves
                            // a relative error below 2^-46 before the last rounding, while r / K (24-bit r, 8-bit K)
                            // is either representable or at least 2^-33 away from every rounding boundary
                            const f32x2 q0 = fma2(r, wk.inv_K, nz);
                            const f32x2 rem = fma2(wk.neg_K, q0, r);
                            jj = add2(add2(fma2(rem, wk.inv_K, q0), args.magic), args.neg_magic);
                        } else {
                            // K is a power of two: r * (1/K) is exact, so one rounding gives rint(r / K)
                            jj = add2(fma2(r, wk.inv_K, args.magic), args.neg_magic);
                        }
                        f32x2 d;                                           // u (q1^ - delta)
                        if constexpr (FORM == kFormJoined) d = fma2(wk.neg_K, jj, x);
                        else if constexpr (FORM == kFormTiny) d = fma2(fma2(wk.neg_K_code, jj, X), both(kTwo127), nf);
                        else d = add2(fma2(wk.neg_K, jj, X), nf);          // (q1^ + 1.5 is exact)
                        gt = SHRINK ? fma2(cc, d, fma2(both(wk.one_m_alpha2), yy, nz)) : fma2(cc, d, nz);
                    }
                    acc[t >> 1] = add2(acc[t >> 1], gt);
                }
            }
        }
        if (SIDE == kSideFirst && w == 0u) {
            // the accumulators are now the reconstruction of message 0: the side information of the nested messages
#pragma unroll
            for (int q = 0; q < E / 4; ++q)
                asm volatile("st.shared.v2.b64 [%0], {%1, %2};"
                             ::"r"(ln.slot + (uint32_t)(q * kDecThreads * 16)), "l"(acc[2 * q]), "l"(acc[2 * q + 1])
                             : "memory");
        }
    }
}

inline bool is_usual_variant(uint32_t variant) { return (variant >> 3) <= kDecNdqsgPow2 && (variant & 7u) < 4u; }
// (one bit has no K but two)
inline bool is_odd_variant(uint32_t variant)
{
    return ((variant >> 3) == kDecDqsg || (variant >> 3) == kDecNdqsgAnyK) && (variant & 7u) < 4u;
}

// All W workers, run by run; dispatch on (kind, bits) with one jump per run.
template <int DITH, int SIDE, int E, int SET, typename Args>
__device__ __forceinline__ void decode_workers(const Args& args, DecLane& ln, f32x2 (&acc)[E / 2])
{
#define DQ_DEC_CASE(KIND, BITS)                                                                                    \
    case (KIND) * 8u + (BITS) - 1u:                                                                                \
        decode_run<BITS, KIND, DITH, SIDE, E, kWordsAhead<DITH, KIND, E, SET>>(args, w, w_end, ln, acc);        \
        break;
#define DQ_DEC_LOW(KIND)                                                                                           \
    DQ_DEC_CASE(KIND, 1) DQ_DEC_CASE(KIND, 2) DQ_DEC_CASE(KIND, 3) DQ_DEC_CASE(KIND, 4)
#define DQ_DEC_KIND(KIND)                                                                                          \
    DQ_DEC_LOW(KIND)                                                                                               \
    DQ_DEC_CASE(KIND, 5) DQ_DEC_CASE(KIND, 6) DQ_DEC_CASE(KIND, 7) DQ_DEC_CASE(KIND, 8)
#pragma unroll 1
    for (uint32_t w = 0; w < args.W;) {
        const uint32_t w_end = args.w[w].group_end;
        if constexpr (SET == kSetAll || SET == kSetAllFull) {
            switch (args.w[w].variant) {
                DQ_DEC_KIND(kDecDqsg)
                DQ_DEC_KIND(kDecNdqsgPow2)
                DQ_DEC_KIND(kDecNdqsgPow2Shrink)
                DQ_DEC_KIND(kDecNdqsgAnyK)
                DQ_DEC_KIND(kDecNdqsgAnyKShrink)
                default: break;
            }
        } else if constexpr (SET == kSetOdd) {
            switch (args.w[w].variant) {
                DQ_DEC_LOW(kDecDqsg)
                DQ_DEC_CASE(kDecNdqsgAnyK, 2) DQ_DEC_CASE(kDecNdqsgAnyK, 3) DQ_DEC_CASE(kDecNdqsgAnyK, 4)
                default: break;
            }
        } else if constexpr (SET == kSetUsual) {
            switch (args.w[w].variant) {
                DQ_DEC_LOW(kDecDqsg)
                DQ_DEC_LOW(kDecNdqsgPow2)
                default: break;
            }
        } else {
            switch (args.w[w].variant) {
                DQ_DEC_CASE(kDecDqsg, SET / 16)
                DQ_DEC_CASE(kDecNdqsgPow2, SET % 16)
                default: break;
            }
        }
        w = w_end;
    }
#undef DQ_DEC_KIND
#undef DQ_DEC_LOW
#undef DQ_DEC_CASE
}

__device__ __forceinline__ void store8(float* p, const f32x2 (&v)[4], bool align32)
{
    if (align32) {
        asm volatile("st.global.v4.b64 [%0], {%1, %2, %3, %4};" ::"l"(p), "l"(v[0]), "l"(v[1]), "l"(v[2]), "l"(v[3])
                     : "memory");
    } else {
        asm volatile("st.global.v2.b64 [%0], {%1, %2};" ::"l"(p), "l"(v[0]), "l"(v[1]) : "memory");
        asm volatile("st.global.v2.b64 [%0], {%1, %2};" ::"l"(p + 4), "l"(v[2]), "l"(v[3]) : "memory");
    }
}

// ---------------------------------------------------------------------------------------------------
// The decode kernel: one group of E elements per lane.
// ---------------------------------------------------------------------------------------------------
// Shared memory, per lane: E / 4 slots of side information, then the first Philox products (two blocks per slot).
template <int DITH, int E>
constexpr int kDecBlocks = (DITH == 16) ? E / 8 : E / 4;
template <int DITH, int E>
constexpr int kDecSlots = E / 4 + (DITH != 0 && kDecBlocks<DITH, E> > 1 ? kDecBlocks<DITH, E> / 2 : 0);

// The kernel's work, for the lane's group `local`.
template <int DITH, int SIDE, int E, int SET, typename Args>
__device__ __forceinline__ void decode_group(const Args& args, float4 (*slots)[kDecThreads], uint64_t local)
{
    constexpr int N = kDecBlocks<DITH, E>;
    // Lanes past the end either leave (there is no barrier below), or repeat the last group and store nothing: then the
    // control flow stays uniform for the compiler and a worker's constants take the uniform data path, which gains 1 to 2 %
    // with long chains per lane and loses as much in the shorter ones.
    constexpr bool kClamp = E == 32 || (E == 16 && SET <= kSetOdd);
    const bool live = local < args.num_groups;
    if constexpr (!kClamp) {
        if (!live) return;
    }
    DecLane ln;
    ln.group = args.first_row * (32u / E) + (uint32_t)(!kClamp || live ? local : args.num_groups - 1u);
    const uint64_t i0 = (uint64_t)ln.group * (uint32_t)E;
    const uint32_t row = ln.group / (32u / E);
    ln.bucket = (args.bucket_magic != 0u) ? (__umulhi(row, args.bucket_magic) >> args.bucket_shift)
                                          : (row >> args.bucket_shift);
    ln.slot = smem_u32(&slots[0][threadIdx.x]);
    ln.kappa_bits_max = 0u;
    ln.careful = i0 + 64u > args.n;             // the words of a field may reach past the stream's end
    const bool whole = i0 + (uint32_t)E <= args.n;
    ln.first[0] = ln.first[1] = 0u;
    if constexpr (DITH != 0) {
        uint32_t p[2 * N];
#pragma unroll
        for (int j = 0; j < N; ++j) {
            const uint64_t p0 = (uint64_t)kPhiloxM0 * (ln.group * (uint32_t)N + (uint32_t)j);
            p[2 * j] = (uint32_t)(p0 >> 32);
            p[2 * j + 1] = (uint32_t)p0;
        }
        ln.first[0] = p[0];
        ln.first[1] = p[1];
        if constexpr (N > 1) {
#pragma unroll
            for (int j = 0; j < N / 2; ++j)
                slots[E / 4 + j][threadIdx.x] = make_float4(__uint_as_float(p[4 * j]), __uint_as_float(p[4 * j + 1]),
                                                            __uint_as_float(p[4 * j + 2]), __uint_as_float(p[4 * j + 3]));
        }
    }
    // the messages (and the side information) may be the previous kernel's output
    grid_dependency_wait();
    ln.kappa_next = __ldg(args.w[0].scale + ln.bucket);

    if (SIDE == kSideGiven && args.has_side != 0u) {
        const float* s = args.side + i0;
#pragma unroll
        for (int q = 0; q < E / 4; ++q) {
            float4 v = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            if (whole) {
                v = __ldg(reinterpret_cast<const float4*>(s) + q);
            } else {
                if (i0 + 4 * q < args.n) v.x = __ldg(s + 4 * q);
                if (i0 + 4 * q + 1 < args.n) v.y = __ldg(s + 4 * q + 1);
                if (i0 + 4 * q + 2 < args.n) v.z = __ldg(s + 4 * q + 2);
                if (i0 + 4 * q + 3 < args.n) v.w = __ldg(s + 4 * q + 3);
            }
            slots[q][threadIdx.x] = v;
        }
    }

    f32x2 acc[E / 2];
#pragma unroll
    for (int e = 0; e < E / 2; ++e) acc[e] = 0ull;
    decode_workers<DITH, SIDE, E, SET>(args, ln, acc);
    // the mean (of one message: the message itself)
    if (args.W > 1u) {
        const f32x2 nz = args.neg_zero;
#pragma unroll
        for (int e = 0; e < E / 2; ++e) {
            if (args.invW != 0.0f) {
                acc[e] = fma2(acc[e], both(args.invW), nz);
            } else {
                float u, v;
                unpack2(acc[e], u, v);
                acc[e] = pack2(__fdiv_rn(u, args.Wf), __fdiv_rn(v, args.Wf));
            }
        }
    }
    float* o = args.out + i0;
    if (kClamp && !live) return;
    if (may_be_plain(SET, DITH, SIDE, E) && ln.kappa_bits_max > args.kappa_limit) {
        decode_group_plain<DITH, SIDE, E>(args, ln.group, ln.bucket);
    } else if (whole) {
#pragma unroll
        for (int k = 0; k < E / 8; ++k) {
            const f32x2 v[4] = {acc[4 * k], acc[4 * k + 1], acc[4 * k + 2], acc[4 * k + 3]};
            store8(o + 8 * k, v, args.out_align32 != 0u);
        }
    } else {
#pragma unroll
        for (int e = 0; e < E / 2; ++e) {
            float u, v;
            unpack2(acc[e], u, v);
            if (i0 + 2 * e < args.n) o[2 * e] = u;
            if (i0 + 2 * e + 1 < args.n) o[2 * e + 1] = v;
        }
    }
    if (args.status != nullptr && ln.kappa_bits_max >= 0x7F800000u) atomicOr(args.status, 0x1u);
    // The next kernel may become resident when every CTA of this one has stored.  Let in right after the wait, its CTAs would
    // take the slots that this kernel leaves free, and what does not fit would be placed when these end, several CTAs on one
    // SM and none on others, as soon as a grid takes more than half the slots (W = 8 and a vector: n = 1.3 M 19.7 us per call,
    // here 14.3; 266,610 5.9 and 5.5; from a few waves on there is no difference).  Let in before the stores, the last CTAs to
    // store still make the placement uneven (W = 8, n = 266,610: running mean 5.6 us per call, here 5.3; vector 5.9 and 5.5).
    grid_dependency_launch_next();
}

template <int DITH, int SIDE, int E, int SET, int MAXW>
__global__ void __launch_bounds__(kDecThreads, dec_ctas_per_sm(DITH, E, SET))
decode_aggregate_kernel(const __grid_constant__ DecodeArgsOf<MAXW> args)
{
    __shared__ __align__(16) float4 slots[kDecSlots<DITH, E>][kDecThreads];
    decode_group<DITH, SIDE, E, SET>(args, slots, (uint64_t)blockIdx.x * (uint32_t)kDecThreads + threadIdx.x);
}

}  // namespace dq
