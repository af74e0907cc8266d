// Host side of the C ABI declared in include/dq.h: argument checks, tensor-map set-up, kernel launches.
// Everything numerical happens in the kernels of dq_encode.cuh / dq_decode.cuh.
#include "dq.h"

#include <atomic>
#include <cmath>
#include <cstring>
#include <limits>
#include <mutex>
#include <utility>

#include "dq_decode.cuh"
#include "dq_encode.cuh"
#include "dq_encode_direct.cuh"
#include "dq_host_memory.h"
#include "dq_launch.h"
#include "dq_stats.cuh"
#include "dq_ternary.cuh"

// The device's error word: kernels OR DQ_ERR_* bits into it through the address they are given.  In host code
// the name is a handle for the runtime, not an address.
static __device__ unsigned int g_dq_error_flags = 0u;

namespace {

using dq::launch_overlapped;

std::atomic<uint64_t> g_launches{0};

bool is_pow2(uint32_t v) { return v && !(v & (v - 1u)); }

// Address of element 0 of the virtual whole-gradient array whose element `first` is p[0] (integer arithmetic: the
// result may lie outside any allocation and is only ever used with indices >= first).
template <typename T>
T* virtual_base(T* p, uint64_t first)
{
    return reinterpret_cast<T*>(reinterpret_cast<uintptr_t>(p) - first * sizeof(T));
}
bool float_is_pow2(float v)
{
    uint32_t u;
    std::memcpy(&u, &v, sizeof(u));
    return v > 0.0f && (u & 0x007FFFFFu) == 0u && (u >> 23) != 0u && (u >> 23) != 0xFFu;
}
bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0u; }

void fill_philox(dq::PhiloxStream& ps, uint64_t seed, uint32_t worker, uint64_t step)
{
    uint32_t k[10][2] = {{(uint32_t)(seed & 0xFFFFFFFFull), (uint32_t)(seed >> 32)}};
    for (int r = 1; r < 10; ++r) {
        k[r][0] = k[r - 1][0] + dq::kPhiloxW0;
        k[r][1] = k[r - 1][1] + dq::kPhiloxW1;
    }
    const uint32_t c1 = worker, c2 = (uint32_t)(step & 0xFFFFFFFFull), c3 = (uint32_t)(step >> 32);
    // the block-independent parts of rounds 0..2 (see PhiloxStream)
    const uint64_t p1 = (uint64_t)dq::kPhiloxM1 * (uint64_t)c2;
    const uint32_t u0 = (uint32_t)(p1 >> 32) ^ c1 ^ k[0][0];
    const uint64_t p0 = (uint64_t)dq::kPhiloxM0 * (uint64_t)u0;
    ps.v0 = c3 ^ k[0][1];
    ps.v1 = (uint32_t)p1 ^ k[1][0];
    ps.v2 = (uint32_t)(p0 >> 32) ^ k[1][1];
    ps.v3 = (uint32_t)p0 ^ k[2][1];
    ps.k2 = k[2][0];
    std::memcpy(ps.rk, k + 3, sizeof(ps.rk));
}

int device_sm_count()
{
    static thread_local int cached_dev = -1, cached_sms = 0;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 0;
    if (dev != cached_dev) {
        int sms = 0;
        if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 0;
        cached_dev = dev;
        cached_sms = sms;
    }
    return cached_sms;
}

dq_status check_params(const dq_params* p, dq_kind kind, uint32_t* levels_out, float* alpha_out)
{
    if (!p) return DQ_ERR_INVALID_ARG;
    if (p->bucket < 32u || p->bucket > 65536u || (p->bucket % 32u) != 0u) return DQ_ERR_INVALID_ARG;
    if (p->bits < 1u || p->bits > 8u) return DQ_ERR_INVALID_ARG;
    if (p->dither_bits != 0u && p->dither_bits != 32u && p->dither_bits != 16u) return DQ_ERR_INVALID_ARG;
    if (kind == DQ_KIND_DQSG) {
        const uint32_t L = p->levels ? p->levels : dq_default_levels(p->bits);
        if (L < 2u || L > (1u << p->bits)) return DQ_ERR_INVALID_ARG;
        *levels_out = L;
        *alpha_out = 1.0f;
    } else if (kind == DQ_KIND_NDQSG) {
        const float alpha = (p->alpha == 0.0f) ? 1.0f : p->alpha;
        if (p->coarse_K < 2u || p->coarse_K > (1u << p->bits)) return DQ_ERR_INVALID_ARG;
        if (!(p->fine_M > 0.0f) || !(alpha > 0.0f) || alpha > 1.0f) return DQ_ERR_INVALID_ARG;
        const float A = alpha * p->fine_M;
        if (!(A > 0.0f)) return DQ_ERR_INVALID_ARG;
        if (A > 1048576.0f) return DQ_ERR_UNSUPPORTED;
        *levels_out = 0u;
        *alpha_out = alpha;
    } else {
        return DQ_ERR_INVALID_ARG;
    }
    return DQ_OK;
}

// cuTensorMapEncodeTiled, looked up at run time so the library loads on machines without a driver.
typedef CUresult (*encode_tiled_fn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                    const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                    CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

encode_tiled_fn get_encode_tiled()
{
    static encode_tiled_fn fn = []() -> encode_tiled_fn {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult qres;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &qres) != cudaSuccess ||
            qres != cudaDriverEntryPointSuccess)
            return nullptr;
        return reinterpret_cast<encode_tiled_fn>(p);
    }();
    return fn;
}

// [rows x 32 fp32] view of a flat vector, boxes of `box_rows` rows, 128-byte swizzle.
bool make_row_map(CUtensorMap* map, const void* base, uint64_t rows, uint32_t box_rows)
{
    encode_tiled_fn fn = get_encode_tiled();
    if (!fn) return false;
    const cuuint64_t dims[2] = {32u, rows};
    const cuuint64_t strides[1] = {128u};
    const cuuint32_t box[2] = {32u, box_rows};
    const cuuint32_t estr[2] = {1u, 1u};
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2u, const_cast<void*>(base), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

constexpr int kMaxDevices = 64;

// Device address of g_dq_error_flags on the current device; looked up once per device.
unsigned int* error_flags_address()
{
    static std::mutex mu;
    static unsigned int* addr[kMaxDevices] = {};
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return nullptr;
    std::lock_guard<std::mutex> lock(mu);
    if (addr[dev] == nullptr) {
        void* ptr = nullptr;
        if (cudaGetSymbolAddress(&ptr, g_dq_error_flags) != cudaSuccess) return nullptr;
        addr[dev] = static_cast<unsigned int*>(ptr);
    }
    return addr[dev];
}

cudaError_t launch_encode(int mode, uint32_t bits, bool dither16, const CUtensorMap& map, const dq::EncodeArgs& a,
                          uint32_t grid, cudaStream_t st)
{
    switch (mode * 2 + (dither16 ? 1 : 0)) {
        case 0: return dq::launch_encode_m0_d32(bits, map, a, grid, st);
        case 1: return dq::launch_encode_m0_d16(bits, map, a, grid, st);
        case 2: return dq::launch_encode_m1_d32(bits, map, a, grid, st);
        case 3: return dq::launch_encode_m1_d16(bits, map, a, grid, st);
        case 4: return dq::launch_encode_m2_d32(bits, map, a, grid, st);
        case 5: return dq::launch_encode_m2_d16(bits, map, a, grid, st);
        case 6: return dq::launch_encode_m3_d32(bits, map, a, grid, st);
        default: return dq::launch_encode_m3_d16(bits, map, a, grid, st);
    }
}

uint32_t bits_of(float v)
{
    uint32_t u;
    std::memcpy(&u, &v, sizeof(u));
    return u;
}

dq::f32x2 twice(float v) { return ((dq::f32x2)bits_of(v) << 32) | bits_of(v); }

cudaError_t launch_direct(int mode, uint32_t bits, bool dither16, int R, int kind, const dq::DirectArgs& a, uint32_t grid,
                          uint32_t threads, cudaStream_t st)
{
    switch (mode * 2 + (dither16 ? 1 : 0)) {
        case 0: return dq::launch_direct_m0_d32(bits, R, kind, a, grid, threads, st);
        case 1: return dq::launch_direct_m0_d16(bits, R, kind, a, grid, threads, st);
        case 2: return dq::launch_direct_m1_d32(bits, R, kind, a, grid, threads, st);
        case 3: return dq::launch_direct_m1_d16(bits, R, kind, a, grid, threads, st);
        case 4: return dq::launch_direct_m2_d32(bits, R, kind, a, grid, threads, st);
        case 5: return dq::launch_direct_m2_d16(bits, R, kind, a, grid, threads, st);
        case 6: return dq::launch_direct_m3_d32(bits, R, kind, a, grid, threads, st);
        default: return dq::launch_direct_m3_d16(bits, R, kind, a, grid, threads, st);
    }
}

// Launches the direct encoder (dq_encode_direct.cuh).  `e` holds what both encoders need.
cudaError_t encode_direct(int mode, const dq_params& p, const dq::EncodeArgs& e, uint64_t n, int sms, cudaStream_t st)
{
    dq::DirectArgs a;
    std::memset(&a, 0, sizeof(a));
    a.grad = e.grad;
    a.packed = e.packed;
    a.scale = e.scale;
    a.n = n;
    a.num_bytes = e.num_words * 4u;
    a.num_groups = (uint32_t)((n + 31u) / 32u * 4u);
    a.whole_groups = (uint32_t)(n / 8u);
    // Up to one wave of one-group lanes (1.2 M elements on 148 SMs) the GPU is not full and the shortest chain per lane
    // wins (B = 2048: n = 266,610 1.6 us with one group, 2.7 with four; 1.2 M 2.5 and 2.8).  Past it large buckets want four at
    // once (B = 16384: 1.3 M 5.9 and 4.3 us), small ones from 1.7 M on (B = 2048: 1.3 M 2.8 and 3.2, 1.7 M 3.4 and 3.3, 2.4 M
    // 4.6 and 4.2).
    const int R = n <= (uint64_t)sms * 1024u * 8u ? 1 : 4;
    const uint32_t gpb = p.bucket / 8u;
    const dq::DirectShape shape = dq::direct_shape(gpb, R);
    a.groups_per_bucket = gpb;
    a.buckets_per_window = shape.buckets;
    a.groups_per_window = gpb * shape.buckets;
    a.cluster = shape.cluster;
    // group / gpb for the (at most 1024) groups of a window: exact because group (magic gpb - 2^22) < 1024 gpb <= 2^22
    // while gpb <= 1024, and larger buckets are alone in their window
    a.bucket_magic = ((1u << 22) + gpb - 1u) / gpb;
    a.reduce = (gpb <= 32u && is_pow2(gpb))                            ? dq::kPartOfWarp
               : (R == 4 && gpb == 64u)                                ? dq::kTwoChunks
               : (R == 4 && gpb == 128u)                               ? dq::kWarpIsBucket
               : (shape.cluster > 1u || gpb % (32u * (uint32_t)R) == 0u) ? dq::kWarpInBucket
                                                                       : dq::kAnywhere;
    a.gains = (a.reduce == dq::kWarpIsBucket || a.reduce == dq::kWarpInBucket) ? 0u
              : a.reduce == dq::kTwoChunks                                     ? 1u
                                                                               : 2u;
    a.grad_align32 = (reinterpret_cast<uintptr_t>(e.grad) & 31u) == 0u ? 1u : 0u;
    a.gain_num = e.gain_num;
    a.kmax = e.kmax;
    a.K = e.K;
    a.K_offset = e.K_offset;
    a.K_magic = e.K_magic;
    a.first_group = e.row_offset * 4u;
    a.early_read = e.early_read;
    a.early_store = e.early_store;
    a.shift = e.shift2;
    a.magic = e.magic;
    a.two = e.two;
    a.off = e.off;
    a.ps = e.ps;
    // A grid of up to two waves lets the next kernel in late: beside it, the CTAs of the next one would be placed unevenly
    // (see the decoder; n = 2.4 M, B = 2048: 4.9 us per call, late 4.2; 1.9 M, B = 16384: 5.1 and 4.4; 1.2 M, B = 2048: 2.8
    // and 2.5).  With more waves it does not matter and the early launch hides a little more (11.7 M: 13.3 us, late 13.4), and
    // so it does where clusters of one-group lanes leave the GPU half empty (0.6 M, B = 16384: 3.31 us, late 3.36).
    a.late_launch = (R == 4 ? n <= (uint64_t)sms * 768u * 32u * 2u : shape.cluster == 1u) ? 1u : 0u;
    // (with early_read one cluster more: see the kernel)
    const uint64_t grid = ((dq_num_buckets(n, p.bucket) + shape.buckets - 1u) / shape.buckets + (a.early_read ? 1u : 0u)) *
                          shape.cluster;
    // More resident CTAs instead of more dithers ahead (times of calls in a stream, ahead and dense):
    //   - where they make one wave of two: n = 4.2 M, B = 4096, 2 bits, flagged 5.4 and 4.6 us; 3.7 M, B = 1504, K = 15 8.5 and
    //     6.5; one-group lanes in CTAs of 656 to 768 threads, of which the ahead kernels run one to an SM: 1.2 M, B = 12288,
    //     4 bits 5.1 and 3.7.  (Clusters of four and eight CTAs, which must find room together, do not fill every slot: B = 65536,
    //     16-bit stream, 3.3 M, 0.94 of the slots 4.9 and 4.1; but 0.82 of them 4 % slower.  Where the buckets of a window share
    //     warps the second wave has to hold a sixteenth of the CTAs, but for flagged calls: B = 1504, 3.6 M 7.5 and 8.0.  Not the
    //     16-bit stream unflagged, whose four dithers ahead hide more: B = 4096, 4.4 M from HBM 5.1 and 5.4);
    //   - from 1.75 waves on where the CTAs of a cluster wait for one another's maxima: B = 65536, 16-bit stream, 11.7 M 13.3 and
    //     12.0; B = 8224, K = 3, 11.7 M 19.5 and 18.3; but 6 M, B = 65536, 2 bits, 1.66 waves 9.7 and 10.2;
    //   - where the buckets of a window share warps, from four waves on 3 to 5 %, from 2.25 on flagged or with codes that are
    //     stored in many bytes (B = 1504, 11.7 M, 7 bits, 16-bit stream 23.7 and 21.9, but 3 bits 17.8 and 18.4).
    // Else the dithers ahead win: 11.7 M, B = 2048, 2 bits 12.5 and 12.6; B = 4096, 1 bit, 16-bit stream 10.2 and 10.8; 2.4 M
    // 3 to 5 %.
    auto slots = [&](int kind) { return (uint64_t)sms * (65536u / (dq::direct_registers(R, kind) * shape.threads)); };
    const uint64_t ahead = slots(dq::kDirectAhead), fits = slots(dq::kDirectDense);
    const bool shared = R == 4 && a.reduce == dq::kAnywhere;
    const uint64_t full = R == 1                               ? ahead
                          : shape.cluster == 8u                ? ahead * 7u / 8u
                          : shape.cluster == 4u                ? ahead * 15u / 16u
                          : (shared && a.early_read == 0u)     ? ahead * 17u / 16u
                                                               : ahead;
    bool dense = grid > full && grid <= fits &&
                 (R == 1 || shape.cluster > 1u || shared || a.early_read != 0u || p.dither_bits != 16u);
    if (R == 4 && shape.cluster > 1u) dense = dense || 4u * grid > 7u * ahead;
    if (shared)
        dense = dense || grid > 4u * ahead || (4u * grid > 9u * ahead && (a.early_read != 0u || p.bits >= 5u));
    dense = dense && shape.threads <= (R == 1 ? dq::kDenseMaxThreads<1> : dq::kDenseMaxThreads<4>);
    return launch_direct(mode, p.bits, p.dither_bits == 16u, R, dense ? dq::kDirectDense : dq::kDirectAhead, a, (uint32_t)grid,
                         shape.threads, st);
}

// The tile kernel streams back-to-back encodes of long gradients, whose launches overlap by the caller's flags, through
// persistent CTAs, a row of 32 elements per lane.  From 16 M elements on it is ahead of the direct kernel (times of calls in a
// stream, tile and direct)
//   - in small buckets, where a lane of the direct kernel computes a gain per group: B = 128, 16.8 M, 2 bits 17.0 and 18.1 us,
//     67 M 57.6 and 65.3; B = 256 2 to 8 %; B = 512 only from 33 M on (16.8 M 16.0 and 15.7, 67 M, 3 bits 61.9 and 65.7);
//   - where a direct lane's codes leave as single bytes and the tile kernel's as words, at seven bits (B = 8192, 16.8 M, 16-bit
//     stream 15.5 and 19.6, 67 M 49.0 and 78.7; B = 2048, 25.6 M 20.7 and 23.8; B = 4096, 16.8 M 14.9 and 16.1) and, B = 8192, at
//     five and six (67 M, 5 bits 46.9 and 52.6, 6 bits 49.8 and 51.5);
//   - in very long gradients in buckets of 1024 and 2048: B = 2048, 124 M, 2 bits 108 and 115, 3 bits 117 and 126; 67 M, 3 bits
//     57.3 and 58.7; B = 1024, 124 M, 3 bits 112 and 115, 67 M, 2 bits, 16-bit stream 42.5 and 41.1.
// Not elsewhere: B = 4096, 25.6 M 7 % slower, B = 1024 and 8192, 16.8 M 7 to 12 %.
bool tile_encoder_pays(uint64_t n, uint32_t bucket, uint32_t bits)
{
    if (n < (1ull << 24)) return false;
    if (bucket <= 256u || bits == 7u) return true;
    switch (bucket) {
        case 512u: return n >= (1ull << 25);
        case 1024u: return n >= 3ull * (1ull << 25);
        case 2048u: return n >= (1ull << 26);
        case 8192u: return (bits == 5u || bits == 6u) && n >= 3ull * (1ull << 23);
        default: return false;
    }
}

dq_status encode_common(dq_kind kind, const float* grad, uint64_t n, uint64_t seed, uint32_t worker,
                        uint64_t step, const dq_params* p, uint32_t* out_packed, float* out_scale,
                        cudaStream_t st, uint64_t first_element = 0u)
{
    uint32_t L = 0;
    float alpha = 1.0f;
    dq_status s = check_params(p, kind, &L, &alpha);
    if (s != DQ_OK) return s;
    if (first_element % p->bucket != 0u) return DQ_ERR_INVALID_ARG;      // a range starts at a bucket boundary
    if (n == 0) return DQ_OK;
    if (n >= (1ull << 34) || first_element >= (1ull << 34) || first_element + n >= (1ull << 34))
        return DQ_ERR_UNSUPPORTED;
    if (!grad || !out_packed || !out_scale) return DQ_ERR_INVALID_ARG;
    if (!aligned16(grad) || !aligned16(out_packed) || !aligned16(out_scale)) return DQ_ERR_ALIGNMENT;

    dq::EncodeArgs a;
    std::memset(&a, 0, sizeof(a));
    a.grad = grad;
    a.packed = out_packed;
    a.scale = out_scale;
    a.n = n;
    a.row_offset = (uint32_t)(first_element / 32u);
    a.bucket = p->bucket;
    a.num_buckets = dq_num_buckets(n, p->bucket);
    a.num_words = dq_packed_words(n, p->bits);
    int mode;
    if (kind == DQ_KIND_DQSG) {
        mode = dq::kEncDqsg;
        a.shift = (float)(L - 1u) / 2.0f;
        a.gain_num = a.shift;
        a.kmax = (int32_t)(L - 1u);
    } else {
        // K = 2^bits: the coset is the low `bits` bits of the fine index; a smaller power of two: one mask more;
        // any other K: the remainder
        mode = (p->coarse_K == (1u << p->bits)) ? dq::kEncNdqsgPow2
               : is_pow2(p->coarse_K)           ? dq::kEncNdqsgPow2Mask
                                                : dq::kEncNdqsgAnyK;
        a.gain_num = alpha * p->fine_M;
        a.K = p->coarse_K;
        a.K_offset = ((4194304u + p->coarse_K - 1u) / p->coarse_K) * p->coarse_K;
        a.K_magic = (uint32_t)(((1ull << 32) + p->coarse_K - 1u) / p->coarse_K);
    }
    const bool d16 = (p->dither_bits == 16u);
    a.shift2 = twice(a.shift);
    a.magic = twice(dq::kMagic);
    a.two = twice(d16 ? dq::kTwo125 : dq::kTwo127);
    a.off = twice(d16 ? -dq::kD16Offset : -dq::kD32Offset);
    fill_philox(a.ps, seed, worker, step);
    a.early_read = (p->flags & DQ_FLAG_INPUT_READY) ? 1u : 0u;
    a.early_store = (a.early_read && (p->flags & DQ_FLAG_OUTPUT_FREE)) ? 1u : 0u;
    a.all_lanes = 0xFFFFFFFFu;
    a.test_drop_copy = (p->flags & DQ_FLAG_TEST_DROP_COPY) ? 1u : 0u;
    a.error_flags = error_flags_address();
    if (!a.error_flags) return DQ_ERR_CUDA;

    const int sms = device_sm_count();
    if (sms <= 0) return DQ_ERR_CUDA;
    const bool tiles_wanted = is_pow2(p->bucket) && p->bucket <= 8192u &&
                              (a.test_drop_copy != 0u || (a.early_store != 0u && tile_encoder_pays(n, p->bucket, p->bits)));
    if (!tiles_wanted) {
        if (encode_direct(mode, *p, a, n, sms, st) != cudaSuccess) return DQ_ERR_CUDA;
        g_launches.fetch_add(1);
        return DQ_OK;
    }
    // whole work units (a bucket, or 1024 elements for smaller buckets) go through the tile path of the kernel, the rest
    // through its plain-load part, in the same launch
    const uint32_t B = p->bucket;
    const uint32_t U = (B < 1024u) ? 1024u : B;                     // elements per work unit
    const uint64_t tiles = n / U;                                   // whole units
    if (tiles > 0xFFFFFFFFull) return DQ_ERR_UNSUPPORTED;
    CUtensorMap map;
    std::memset(&map, 0, sizeof(map));
    const bool pair = (B == 2048u || B == 4096u || B == 8192u);     // a warp takes 2048 elements, two halves in time
    const uint32_t wpb = pair ? (B / 2048u) : (B < 1024u) ? 1u : (B / 1024u);
    a.pair_in_time = pair ? 1u : 0u;
    if (tiles > 0) {
        if (!make_row_map(&map, grad, tiles * (U / 32u), 32u)) return DQ_ERR_CUDA;
        a.num_units = (uint32_t)tiles;
        a.lanes_per_bucket = (B < 1024u) ? (B / 32u) : 32u;
        a.warps_per_bucket = wpb;
        uint32_t lg = 0;
        while ((1u << lg) < B) ++lg;
        a.bucket_log2 = lg;
    }
    a.first_bucket = tiles * (U / B);
    const uint64_t rest = a.num_buckets - a.first_bucket;
    const uint32_t slots = (uint32_t)dq::kEncCtasPerSm * (uint32_t)sms;   // resident CTAs
    uint32_t plain = 0;
    if (rest > 0) {
        // buckets of at most 32 rows: a warp takes a window of whole buckets; up to 128 rows: a warp per bucket;
        // larger ones: a CTA per bucket
        uint64_t want = rest;
        if (B <= 1024u) {
            const uint64_t rpb = B / 32u, rows_per_window = (32u / rpb) * rpb;
            const uint64_t rest_rows = (n + 31u) / 32u - a.first_bucket * rpb;
            a.plain_windows = (rest_rows + rows_per_window - 1u) / rows_per_window;
            want = (a.plain_windows + dq::kConsumerWarps - 1u) / dq::kConsumerWarps;
        } else if (B <= dq::kPlainWarpBucketMax) {
            want = (rest + dq::kConsumerWarps - 1u) / dq::kConsumerWarps;           // a warp per bucket
        }
        const uint64_t cap = (tiles > 0) ? (slots / 4u) : (4ull * slots);
        plain = (uint32_t)(want < cap ? want : cap);
        if (plain == 0u) plain = 1u;
    }
    a.plain_ctas = plain;
    uint32_t tile_ctas = 0;
    if (tiles > 0) {
        const uint32_t room = (slots > plain) ? (slots - plain) : 1u;
        const uint64_t groups_per_cta = (uint64_t)dq::kConsumerWarps / wpb;
        const uint64_t want_ctas = (tiles + groups_per_cta - 1u) / groups_per_cta;
        tile_ctas = (uint32_t)(want_ctas < room ? want_ctas : room);
    }
    if (launch_encode(mode, p->bits, d16, map, a, plain + tile_ctas, st) != cudaSuccess) return DQ_ERR_CUDA;
    g_launches.fetch_add(1);
    return DQ_OK;
}

// Elements per lane of the decoder.  Up to one wave of 8-element lanes (1.2 M elements on 148 SMs) the GPU is not
// full and the shortest chain per lane wins (W = 8, running mean: n = 266,610 5.3 us with 8, 6.7 with 16, 9.1 with 32).  Beyond
// it 16 and then 32 elements amortise what a worker costs per lane.  32 pays from about two and a half of its own waves, a
// little before or after with the side information (W = 8: first 3.3 M +2 %, 4.2 M -5 %, 7.4 M -4 %; running mean +1, -5, -4 %;
// a vector +10, +2, +1 %; 7.6 M W = 4 -5 %, W = 2 0 %; W = 8, 11.7 M -7 %), and not for one nested message, or two messages and
// a vector, where memory latency matters more and 16 has more warps to hide it (n = 25.6 M: W = 1 45.5 us with 16, 55.6 with
// 32; W = 2 with a vector 62.9 and 69.3, without 51.3 and 48.1).  (One DQSG message has a kernel of its own.)  In the kernel with
// all routines, whose routines are longer, 32 pays from one wave of 16-element lanes on if there are eight messages (`usual`
// false; six bits, W = 8: n = 2.4 M 23.5 us with 16, 23.0 with 32; 3 M 28.3 and 26.3; 4.2 M 38.3 and 35.2; W = 32, 4.2 M 147
// and 134; but W = 3 and a vector, 4.2 M 18.9 and 22.9).  From 48 messages on, whose parameters do not stay in the caches between
// a warp's steps, 32 pays from 1.33 waves of 16-element lanes on (W = 64, one nested bit: running mean 3.3 M 228 and 200 us, 4.2 M
// 296 and 234; first 3.3 M 243 and 203; two bits, running mean 4.2 M 249 and 235, but 2.5 M 162 and 167).
int decode_group_size(uint64_t n, uint32_t W, bool reads_side, bool usual, int sms)
{
    const uint64_t lanes = (uint64_t)sms * dq::kDecThreads;
    const uint64_t wave8 = 8u * lanes * 8u, wave16 = 16u * lanes * 8u, wave32 = 32u * lanes * 5u;
    if (n <= wave8) return 8;
    if (!usual && W >= 8u && n > wave16) return 32;
    if (W >= 48u && 3u * n > 4u * wave16) return 32;
    if (W <= (reads_side ? 2u : 1u) || 2u * n < 5u * wave32) return 16;
    return 32;
}

// The constants of a worker that depend on the form its routine works in (see DecForm).  Returns the largest scale that the
// form takes.
float set_decode_form(dq::DecWorker& d, int dith, int group)
{
    const uint32_t kind = d.variant >> 3;
    const int bits = (int)(d.variant & 7u) + 1;
    const int form = dq::dec_form(kind, bits, dith, group), shift = dq::dec_shift(kind, bits, dith, group);
    const float u = 1.0f / (float)(1u << shift);
    if (form == dq::kFormJoined && dith == 16)
        d.offset = twice(((float)((1u << bits) - 1u) - d.s + dq::kD16Offset) * u);          // J = (2^bits - 1 - k) 2^16 + h
    else if (form == dq::kFormJoined)
        d.offset = twice(-(d.s + dq::kD32Offset));                                          // J = k 2^22 + (2^22 - 1 - j)
    else
        d.offset = twice(-(4194304.0f + d.s - 1.5f));
    if (kind != dq::kDecDqsg) {
        d.neg_K = twice(-d.K * u);
        if (form == dq::kFormTiny) d.neg_K_code = twice(-d.K * 0x1p-125f / (float)(1u << bits));
        d.inv_K = twice(1.0f / d.K / u);
        d.A *= u;
    }
    if (shift == 0) return std::numeric_limits<float>::infinity();
    // kappa / s / u and alpha kappa / M1 / u below 2^127, alpha M1 u / kappa normal, and alpha M1 u too: a subnormal number
    // has lost bits
    if (kind == dq::kDecDqsg) return 0x1p119f;
    if (d.A < 0x1p-126f) return 0.0f;
    const float most = std::fmin(d.M1 / d.alpha * 0x1p-6f, d.A);
    return most >= 1.0f ? 0x1p120f : most * 0x1p120f;
}

dq_status decode_common(const dq_msg* msgs, uint32_t W, uint64_t n, uint64_t step, const float* side_info,
                        float* out_avg, uint32_t* status_word, bool allow_nested, cudaStream_t st,
                        bool running = false, bool half_dithered = false, uint64_t first_element = 0u,
                        bool side_first = false)
{
    if (!msgs || W == 0u || W > DQ_MAX_WORKERS) return DQ_ERR_INVALID_ARG;
    static thread_local dq::DecodeArgs a;    // ~11 KB: keep it off the stack; the first W entries of a.w are filled
    std::memset(static_cast<dq::DecodeHead*>(&a), 0, sizeof(dq::DecodeHead));
    bool any_nested = false;
    for (uint32_t w = 0; w < W; ++w) {
        const dq_msg& m = msgs[w];
        uint32_t L = 0;
        float alpha = 1.0f;
        dq_status s = check_params(&m.p, m.kind, &L, &alpha);
        if (s != DQ_OK) return s;
        if (m.kind == DQ_KIND_NDQSG && !allow_nested) return DQ_ERR_INVALID_ARG;
        if (m.p.bucket != msgs[0].p.bucket) return DQ_ERR_UNSUPPORTED;
        if (!half_dithered && (m.p.dither_bits == 16u) != (msgs[0].p.dither_bits == 16u)) return DQ_ERR_UNSUPPORTED;
        dq::DecWorker& d = a.w[w];
        std::memset(&d, 0, sizeof(d));
        // addresses of the (virtual) whole-gradient buffers: see DecodeArgs
        d.packed = virtual_base(m.packed, first_element / 32u * m.p.bits);
        d.scale = virtual_base(m.scale, first_element / m.p.bucket);
        fill_philox(d.ps, m.seed, m.worker, step);
        uint32_t kind;
        if (m.kind == DQ_KIND_DQSG) {
            kind = dq::kDecDqsg;
            d.s = (float)(L - 1u) / 2.0f;
            d.step_mul = is_pow2(L - 1u) && L >= 3u ? 2.0f / (float)(L - 1u) : (L == 2u ? 2.0f : 0.0f);
        } else {
            any_nested = true;
            if (is_pow2(m.p.coarse_K)) kind = (alpha == 1.0f) ? dq::kDecNdqsgPow2 : dq::kDecNdqsgPow2Shrink;
            else kind = (alpha == 1.0f) ? dq::kDecNdqsgAnyK : dq::kDecNdqsgAnyKShrink;
            d.A = alpha * m.p.fine_M;
            d.M1 = m.p.fine_M;
            d.alpha = alpha;
            const float a2 = alpha * alpha;
            d.one_m_alpha2 = 1.0f - a2;
            d.K = (float)m.p.coarse_K;
            d.step_mul = float_is_pow2(m.p.fine_M) ? 1.0f / m.p.fine_M : 0.0f;
            if (running) {
                if (w == 0u) return DQ_ERR_INVALID_ARG;      // nothing decoded yet to serve as side information
                d.rcp_count = 1.0f / (float)w;
            }
        }
        d.variant = kind * 8u + m.p.bits - 1u;
    }
    // runs of equal variants (one routine per run, see decode_workers)
    for (uint32_t w = W; w-- > 0u;)
        a.w[w].group_end = (w + 1u < W && a.w[w + 1u].variant == a.w[w].variant) ? a.w[w + 1u].group_end : w + 1u;
    if (first_element % msgs[0].p.bucket != 0u) return DQ_ERR_INVALID_ARG;   // a range starts at a bucket boundary
    if (n == 0) return DQ_OK;
    if (n >= (1ull << 34) || first_element >= (1ull << 34) || first_element + n >= (1ull << 34))
        return DQ_ERR_UNSUPPORTED;
    if (!out_avg) return DQ_ERR_INVALID_ARG;
    if (side_first && msgs[0].kind != DQ_KIND_DQSG) return DQ_ERR_INVALID_ARG;   // message 0 is decoded on its own
    if (any_nested && !running && !side_first && !side_info) return DQ_ERR_INVALID_ARG;
    if (!aligned16(out_avg) || (side_info && !aligned16(side_info))) return DQ_ERR_ALIGNMENT;
    for (uint32_t w = 0; w < W; ++w) {
        if (!msgs[w].packed || !msgs[w].scale) return DQ_ERR_INVALID_ARG;
        if (!aligned16(msgs[w].packed) || !aligned16(msgs[w].scale)) return DQ_ERR_ALIGNMENT;
    }
    const bool reads_side = any_nested && !running && !side_first;
    const bool from_first = any_nested && !running && side_first;
    a.side = reads_side ? virtual_base(side_info, first_element) : nullptr;
    a.out = virtual_base(out_avg, first_element);
    a.status = status_word;
    a.n = first_element + n;
    a.first_row = (uint32_t)(first_element / 32u);
    a.W = W;
    a.rows_per_bucket = msgs[0].p.bucket / 32u;
    dq::set_bucket_division(a);
    a.has_side = reads_side ? 1u : 0u;
    a.out_align32 = (reinterpret_cast<uintptr_t>(out_avg) & 31u) == 0u ? 1u : 0u;
    a.half_bias_bits = 0x4A800000u;
    a.low22 = 0x003FFFFFu;
    a.neg_zero = twice(-0.0f);
    a.magic = twice(dq::kMagic);
    a.neg_magic = twice(-dq::kMagic);
    a.Wf = (float)W;
    a.invW = is_pow2(W) ? 1.0f / (float)W : 0.0f;
    const int sms = device_sm_count();
    if (sms <= 0) return DQ_ERR_CUDA;
    const bool d16 = (msgs[0].p.dither_bits == 16u);
    // (a single nested message needs a side information vector and goes the general way)
    const bool one_message = W == 1u && !half_dithered && !any_nested;
    bool usual = true;
    for (uint32_t w = 0; w < W; ++w) usual = usual && dq::is_usual_variant(a.w[w].variant);
    const int E = one_message ? 8 : decode_group_size(n, W, reads_side, usual, sms);
    a.num_groups = (n + (uint32_t)E - 1u) / (uint32_t)E;
    const int side = from_first ? dq::kSideFirst : (running && any_nested) ? dq::kSideRunning : dq::kSideGiven;
    float kappa_most = std::numeric_limits<float>::infinity();
    for (uint32_t w = 0; w < W; ++w)
        kappa_most = std::fmin(kappa_most, set_decode_form(a.w[w], half_dithered ? 0 : d16 ? 16 : 32, E));
    // (no limit: above the pattern of any NaN)
    a.kappa_limit = std::isinf(kappa_most) ? 0xFFFFFFFFu : bits_of(kappa_most);
    if (one_message) {
        static thread_local dq::DecodeArgsOf<1> one;
        static_cast<dq::DecodeHead&>(one) = a;
        one.w[0] = a.w[0];
        // up to one wave of one-group lanes the shortest chain wins, with the 32-bit stream to a quarter more (calls in a
        // stream, 3 bits: n = 266,037 1.25 us with one group, 1.86 with four; 1.3 M 2.75 and 3.06; 1.5 M 3.02 and 3.12; 1.7 M
        // 3.28 and 3.07; 2.4 M 3.99 and 3.69; 16-bit stream: 1.25 M 2.56 and 2.51; 1.7 M 3.06 and 2.60)
        const int R = n <= (uint64_t)sms * 1024u * (d16 ? 8u : 10u) ? 1 : 4;
        const cudaError_t e = d16 ? dq::launch_decode_one_d16(one, R, st) : dq::launch_decode_one_d32(one, R, st);
        if (e != cudaSuccess) return DQ_ERR_CUDA;
        g_launches.fetch_add(1);
        return DQ_OK;
    }
    cudaError_t le;
    if (half_dithered) le = dq::launch_decode_d0_r0(a, E, sms, st);
    else if (side == dq::kSideRunning) le = d16 ? dq::launch_decode_d16_r1(a, E, sms, st) : dq::launch_decode_d32_r1(a, E, sms, st);
    else if (side == dq::kSideFirst) le = d16 ? dq::launch_decode_d16_r2(a, E, sms, st) : dq::launch_decode_d32_r2(a, E, sms, st);
    else le = d16 ? dq::launch_decode_d16_r0(a, E, sms, st) : dq::launch_decode_d32_r0(a, E, sms, st);
    if (le != cudaSuccess) return DQ_ERR_CUDA;
    g_launches.fetch_add(1);
    return DQ_OK;
}

// CTAs in the histogram's cluster: 16 (which needs an attribute per kernel and device) where one can be resident, else
// the portable 8; 0 on a CUDA error.
uint32_t hist_cluster_size()
{
    static std::mutex mu;
    static uint32_t size[kMaxDevices] = {};
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return 0u;
    std::lock_guard<std::mutex> lock(mu);
    if (size[dev] == 0u) {
        uint32_t s = 8u;
        bool ok = true;
        for (auto k : {dq::code_histogram_cluster_kernel<1>, dq::code_histogram_cluster_kernel<2>})
            ok = ok && cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess;
        if (ok) {
            cudaLaunchConfig_t cfg = {};
            cfg.gridDim = dim3(dq::kHistCluster);
            cfg.blockDim = dim3(dq::kHistClusterThreads);
            cudaLaunchAttribute attr[1];
            attr[0].id = cudaLaunchAttributeClusterDimension;
            attr[0].val.clusterDim.x = dq::kHistCluster;
            attr[0].val.clusterDim.y = 1;
            attr[0].val.clusterDim.z = 1;
            cfg.attrs = attr;
            cfg.numAttrs = 1;
            int clusters = 0;
            if (cudaOccupancyMaxActiveClusters(&clusters, dq::code_histogram_cluster_kernel<2>, &cfg) == cudaSuccess &&
                clusters > 0)
                s = (uint32_t)dq::kHistCluster;
        }
        cudaGetLastError();
        size[dev] = s;
    }
    return size[dev];
}

uint64_t align_up(uint64_t v, uint64_t a) { return (v + a - 1u) / a * a; }

}  // namespace

namespace {

// The *_host calls move their data in one of three ways:
//   - short gradients in pinned memory: no copies at all, the kernels read and write the host buffers over the bus (a
//     copy costs 4 us of set-up, and a decode has two per message);
//   - long ones: in two pieces, so that the copies of one direction run beside the kernel and the copies of the other.
//     The bus moves 55 GB/s in each direction at once, but a change between copies, events and kernels costs some 20 us,
//     so more pieces than two gain nothing (n = 11.7 M: encode 942 us in one piece, 893 in two, 892 in three; decode of
//     four messages 1183, 1102 and 1115);
//   - everything else: copy in, kernel, copy out.
constexpr uint64_t kHostDirectElements = 1ull << 20;       // up to here without copies
constexpr uint64_t kHostPieceElements = 1ull << 22;        // from here in pieces
constexpr int kHostPieces = 2;

// cuPointerGetAttributes, looked up like cuTensorMapEncodeTiled.
typedef CUresult (*pointer_attributes_fn)(unsigned int, CUpointer_attribute*, void**, CUdeviceptr);

pointer_attributes_fn get_pointer_attributes()
{
    static pointer_attributes_fn fn = []() -> pointer_attributes_fn {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult qres;
        if (cudaGetDriverEntryPoint("cuPointerGetAttributes", &p, cudaEnableDefault, &qres) != cudaSuccess ||
            qres != cudaDriverEntryPointSuccess)
            return nullptr;
        return reinterpret_cast<pointer_attributes_fn>(p);
    }();
    return fn;
}

// The page-locked range that `host` lies in; false when it is not page-locked (or managed memory).
bool pinned_range(const void* host, dq::PinnedRange* out)
{
    pointer_attributes_fn fn = get_pointer_attributes();
    if (!fn) return false;
    CUpointer_attribute what[] = {CU_POINTER_ATTRIBUTE_MEMORY_TYPE, CU_POINTER_ATTRIBUTE_IS_MANAGED,
                                  CU_POINTER_ATTRIBUTE_DEVICE_POINTER, CU_POINTER_ATTRIBUTE_RANGE_START_ADDR,
                                  CU_POINTER_ATTRIBUTE_RANGE_SIZE};
    unsigned int type = 0u;
    int managed = 0;
    CUdeviceptr device = 0u, start = 0u;
    size_t size = 0u;
    void* values[] = {&type, &managed, &device, &start, &size};
    const CUdeviceptr p = static_cast<CUdeviceptr>(reinterpret_cast<uintptr_t>(host));
    if (fn(5u, what, values, p) != CUDA_SUCCESS) {
        // a host thread that has no context yet gets the runtime's by this call
        cudaPointerAttributes at;
        if (cudaPointerGetAttributes(&at, host) != cudaSuccess) {
            cudaGetLastError();
            return false;
        }
        if (fn(5u, what, values, p) != CUDA_SUCCESS) return false;
    }
    if (type != (unsigned int)CU_MEMORYTYPE_HOST || managed || device == 0u) return false;
    *out = {(uint64_t)device, (uint64_t)start, (uint64_t)size};
    return true;
}

// Device address of `count` values in page-locked host memory, null where the kernels cannot work on them.
template <typename T>
T* pinned_view(T* host, uint64_t count)
{
    return reinterpret_cast<T*>(static_cast<uintptr_t>(dq::pinned_device_address(host, count * sizeof(T), pinned_range)));
}

// A second stream and the events that tie it to the caller's: one set per host thread and device, made at the thread's
// first long *_host call on the device and given back when the thread ends.
struct HostPipe {
    cudaStream_t stream = nullptr;
    cudaEvent_t arrived[kHostPieces] = {};       // (piece i is ready for the second stream)
    bool make()
    {
        if (stream) return true;
        for (cudaEvent_t& e : arrived)
            if (!e && cudaEventCreateWithFlags(&e, cudaEventDisableTiming) != cudaSuccess) return false;
        return cudaStreamCreateWithFlags(&stream, cudaStreamNonBlocking) == cudaSuccess;
    }
    ~HostPipe()
    {
        for (cudaEvent_t e : arrived)
            if (e) cudaEventDestroy(e);
        if (stream) cudaStreamDestroy(stream);
    }
};

HostPipe* host_pipe()
{
    static thread_local HostPipe pipes[kMaxDevices];
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return nullptr;
    return pipes[dev].make() ? &pipes[dev] : nullptr;
}

// Start of piece i when n elements are cut at `sixteenths[i]` sixteenths: a multiple of four buckets, so that every
// buffer's piece is 16-byte aligned.
uint64_t piece_start(uint64_t n, uint32_t bucket, uint32_t sixteenths)
{
    return sixteenths >= 16u ? n : n / 16u * sixteenths / (4u * bucket) * (4u * bucket);
}

}  // namespace

extern "C" {

uint64_t dq_packed_words(uint64_t n, uint32_t bits) { return (n * (uint64_t)bits + 31u) / 32u; }
uint64_t dq_num_buckets(uint64_t n, uint32_t bucket) { return bucket ? (n + bucket - 1u) / bucket : 0u; }
uint32_t dq_default_levels(uint32_t bits) { return bits == 1u ? 2u : (1u << bits) - 1u; }

const char* dq_status_string(dq_status s)
{
    switch (s) {
        case DQ_OK: return "ok";
        case DQ_ERR_INVALID_ARG: return "invalid argument";
        case DQ_ERR_UNSUPPORTED: return "unsupported configuration";
        case DQ_ERR_ALIGNMENT: return "device pointer not 16-byte aligned";
        case DQ_ERR_CUDA: return "CUDA call failed";
        case DQ_ERR_TOO_LARGE: return "input larger than the built-in scratch buffer";
    }
    return "unknown status";
}

dq_status dqsg_encode(const float* grad, uint64_t n, uint64_t seed, uint32_t worker, uint64_t step,
                      const dq_params* p, uint32_t* out_packed, float* out_scale, void* cuda_stream)
{
    return encode_common(DQ_KIND_DQSG, grad, n, seed, worker, step, p, out_packed, out_scale,
                         static_cast<cudaStream_t>(cuda_stream));
}

dq_status ndqsg_encode(const float* grad, uint64_t n, uint64_t seed, uint32_t worker, uint64_t step,
                       const dq_params* p, uint32_t* out_packed, float* out_scale, void* cuda_stream)
{
    return encode_common(DQ_KIND_NDQSG, grad, n, seed, worker, step, p, out_packed, out_scale,
                         static_cast<cudaStream_t>(cuda_stream));
}

dq_status dqsg_decode_aggregate(const dq_msg* msgs, uint32_t W, uint64_t n, uint64_t step, float* out_avg,
                                void* cuda_stream)
{
    return decode_common(msgs, W, n, step, nullptr, out_avg, nullptr, false, static_cast<cudaStream_t>(cuda_stream));
}

dq_status ndqsg_decode_aggregate(const dq_msg* msgs, uint32_t W, uint64_t n, uint64_t step,
                                 const float* side_info, float* out_avg, uint32_t* status_word, void* cuda_stream)
{
    return decode_common(msgs, W, n, step, side_info, out_avg, status_word, true,
                         static_cast<cudaStream_t>(cuda_stream));
}

dq_status ndqsg_decode_aggregate_side_first(const dq_msg* msgs, uint32_t W, uint64_t n, uint64_t step, float* out_avg,
                                            uint32_t* status_word, void* cuda_stream)
{
    return decode_common(msgs, W, n, step, nullptr, out_avg, status_word, true,
                         static_cast<cudaStream_t>(cuda_stream), false, false, 0u, true);
}

dq_status dqsg_decode_aggregate_half_dithered(const dq_msg* msgs, uint32_t W, uint64_t n, float* out_avg,
                                              void* cuda_stream)
{
    return decode_common(msgs, W, n, 0u, nullptr, out_avg, nullptr, false, static_cast<cudaStream_t>(cuda_stream),
                         false, true);
}

dq_status ndqsg_decode_aggregate_running(const dq_msg* msgs, uint32_t W, uint64_t n, uint64_t step, float* out_avg,
                                         uint32_t* status_word, void* cuda_stream)
{
    return decode_common(msgs, W, n, step, nullptr, out_avg, status_word, true,
                         static_cast<cudaStream_t>(cuda_stream), true);
}

// ------------------------------------------------------------------------------------------------ bucket ranges
dq_status dqsg_encode_range(const float* grad, uint64_t n, uint64_t first_element, uint64_t seed, uint32_t worker,
                            uint64_t step, const dq_params* p, uint32_t* out_packed, float* out_scale,
                            void* cuda_stream)
{
    return encode_common(DQ_KIND_DQSG, grad, n, seed, worker, step, p, out_packed, out_scale,
                         static_cast<cudaStream_t>(cuda_stream), first_element);
}

dq_status ndqsg_encode_range(const float* grad, uint64_t n, uint64_t first_element, uint64_t seed, uint32_t worker,
                             uint64_t step, const dq_params* p, uint32_t* out_packed, float* out_scale,
                             void* cuda_stream)
{
    return encode_common(DQ_KIND_NDQSG, grad, n, seed, worker, step, p, out_packed, out_scale,
                         static_cast<cudaStream_t>(cuda_stream), first_element);
}

dq_status ndqsg_decode_aggregate_range(const dq_msg* msgs, uint32_t W, uint64_t n, uint64_t first_element,
                                       uint64_t step, const float* side_info, float* out_avg,
                                       uint32_t* status_word, void* cuda_stream)
{
    return decode_common(msgs, W, n, step, side_info, out_avg, status_word, true,
                         static_cast<cudaStream_t>(cuda_stream), false, false, first_element);
}

dq_status dq_code_histogram(const uint32_t* packed, uint64_t n, uint32_t bits, uint64_t* hist, void* cuda_stream)
{
    if (bits < 1u || bits > 8u) return DQ_ERR_INVALID_ARG;
    if (!hist) return DQ_ERR_INVALID_ARG;
    if (n >= (1ull << 34)) return DQ_ERR_UNSUPPORTED;
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    if (n != 0 && !packed) return DQ_ERR_INVALID_ARG;
    if (n != 0 && (!aligned16(packed) || (reinterpret_cast<uintptr_t>(hist) & 7u) != 0u)) return DQ_ERR_ALIGNMENT;
    static_assert(sizeof(unsigned long long) == sizeof(uint64_t), "histogram counters are 64-bit");
    unsigned long long* h = reinterpret_cast<unsigned long long*>(hist);
    if (n != 0 && bits <= 2u && n * bits <= 8u * dq::kHistClusterBytes) {
        const uint32_t cluster = hist_cluster_size();
        if (cluster == 0u) return DQ_ERR_CUDA;
        // no CTA without at least two 16-byte pieces per warp
        uint32_t ctas = 1u;
        while (ctas < cluster && n * bits > 128u * 64u * ctas) ctas *= 2u;
        auto k = bits == 1u ? dq::code_histogram_cluster_kernel<1> : dq::code_histogram_cluster_kernel<2>;
        if (launch_overlapped(k, ctas, (uint32_t)dq::kHistClusterThreads, 0, st, ctas, packed, n, h) != cudaSuccess)
            return DQ_ERR_CUDA;
        g_launches.fetch_add(1);
        return DQ_OK;
    }
    if (n == 0) return cudaMemsetAsync(hist, 0, sizeof(uint64_t) << bits, st) == cudaSuccess ? DQ_OK : DQ_ERR_CUDA;
    if (launch_overlapped(dq::clear_histogram_kernel, 1u, 1u << bits, 0, st, 1u, h) != cudaSuccess) return DQ_ERR_CUDA;
    g_launches.fetch_add(1);
    const int sms = device_sm_count();
    if (sms <= 0) return DQ_ERR_CUDA;
    const uint64_t rows = (n + 31u) / 32u;
    uint64_t grid = (rows + dq::kHistThreads - 1u) / dq::kHistThreads;
    if (grid > (uint64_t)sms * 4u) grid = (uint64_t)sms * 4u;
    const uint32_t g = (uint32_t)grid, t = (uint32_t)dq::kHistThreads;
    // counters per thread pay from about 80 M codes on (5 bits: n = 7 M 15.2 us with them, 5.6 with counters per warp;
    // n = 30 M 21.3 and 14.5; n = 120 M 45.2 and 50.2; 4 bits, n = 120 M: 43.8 and 48.6; 3 bits: 54.8 and 48.4)
    const bool own = n >= 80000000u;
    auto k4 = own ? dq::code_histogram_kernel<4, true> : dq::code_histogram_kernel<4, false>;
    auto k5 = own ? dq::code_histogram_kernel<5, true> : dq::code_histogram_kernel<5, false>;
    cudaError_t e = cudaErrorInvalidValue;
    switch (bits) {
        case 1: e = launch_overlapped(dq::code_histogram_words_kernel<1>, g, t, 0, st, 1u, packed, n, h); break;
        case 2: e = launch_overlapped(dq::code_histogram_words_kernel<2>, g, t, 0, st, 1u, packed, n, h); break;
        case 3: e = launch_overlapped(dq::code_histogram_kernel<3, false>, g, t, 0, st, 1u, packed, n, h); break;
        case 4: e = launch_overlapped(k4, g, t, 0, st, 1u, packed, n, h); break;
        case 5: e = launch_overlapped(k5, g, t, 0, st, 1u, packed, n, h); break;
        case 6: e = launch_overlapped(dq::code_histogram_kernel<6, false>, g, t, 0, st, 1u, packed, n, h); break;
        case 7: e = launch_overlapped(dq::code_histogram_kernel<7, false>, g, t, 0, st, 1u, packed, n, h); break;
        default: e = launch_overlapped(dq::code_histogram_kernel<8, false>, g, t, 0, st, 1u, packed, n, h); break;
    }
    if (e != cudaSuccess) return DQ_ERR_CUDA;
    g_launches.fetch_add(1);
    return DQ_OK;
}

dq_status dq_code_entropy(const uint64_t* hist_host, uint32_t bits, double* out_bits_per_element)
{
    if (!hist_host || !out_bits_per_element || bits < 1u || bits > 8u) return DQ_ERR_INVALID_ARG;
    long double total = 0.0L;
    for (uint32_t c = 0; c < (1u << bits); ++c) total += (long double)hist_host[c];
    long double h = 0.0L;
    if (total > 0.0L) {
        for (uint32_t c = 0; c < (1u << bits); ++c) {
            if (hist_host[c] == 0u) continue;
            const long double pc = (long double)hist_host[c] / total;
            h -= pc * log2l(pc);
        }
    }
    *out_bits_per_element = (double)h;
    return DQ_OK;
}

// ------------------------------------------------------------------------------------------------ radix-3 container
uint64_t dq_ternary_bytes(uint64_t n) { return (n + 4u) / 5u; }

static_assert(dq::kWarnCodeRange == DQ_WARN_CODE_RANGE, "status bit of the container kernels");

dq_status dq_ternary_pack(const uint32_t* packed, uint64_t n, uint8_t* out_radix, uint32_t* status_word,
                          void* cuda_stream)
{
    if (n >= (1ull << 34)) return DQ_ERR_UNSUPPORTED;
    if (n == 0) return DQ_OK;
    if (!packed || !out_radix) return DQ_ERR_INVALID_ARG;
    if (!aligned16(packed) || !aligned16(out_radix)) return DQ_ERR_ALIGNMENT;
    const uint64_t units = (n + 79u) / 80u;
    const uint64_t grid = (units + dq::kTernaryThreads - 1u) / dq::kTernaryThreads;
    if (launch_overlapped(dq::ternary_pack_kernel, (uint32_t)grid, (uint32_t)dq::kTernaryThreads, 0,
                          static_cast<cudaStream_t>(cuda_stream), 1u, packed, n, out_radix, status_word) != cudaSuccess)
        return DQ_ERR_CUDA;
    g_launches.fetch_add(1);
    return DQ_OK;
}

dq_status dq_ternary_unpack(const uint8_t* radix, uint64_t n, uint32_t* out_packed, void* cuda_stream)
{
    if (n >= (1ull << 34)) return DQ_ERR_UNSUPPORTED;
    if (n == 0) return DQ_OK;
    if (!radix || !out_packed) return DQ_ERR_INVALID_ARG;
    if (!aligned16(radix) || !aligned16(out_packed)) return DQ_ERR_ALIGNMENT;
    const uint64_t units = (n + 79u) / 80u;
    const uint64_t grid = (units + dq::kTernaryThreads - 1u) / dq::kTernaryThreads;
    if (launch_overlapped(dq::ternary_unpack_kernel, (uint32_t)grid, (uint32_t)dq::kTernaryThreads, 0,
                          static_cast<cudaStream_t>(cuda_stream), 1u, radix, n, out_packed) != cudaSuccess)
        return DQ_ERR_CUDA;
    g_launches.fetch_add(1);
    return DQ_OK;
}

// ------------------------------------------------------------------------------------------------ host buffers
uint64_t dq_encode_workspace_bytes(uint64_t n, const dq_params* p)
{
    if (!p || p->bucket == 0u) return 0u;
    return align_up(n * 4u, 256u) + align_up(dq_packed_words(n, p->bits) * 4u, 256u) +
           align_up(dq_num_buckets(n, p->bucket) * 4u, 256u);
}

uint64_t dq_decode_workspace_bytes(const dq_msg* msgs, uint32_t W, uint64_t n, int has_side_info)
{
    if (!msgs) return 0u;
    uint64_t total = align_up(n * 4u, 256u) * (has_side_info ? 2u : 1u);
    for (uint32_t w = 0; w < W; ++w) {
        if (msgs[w].p.bucket == 0u) return 0u;
        total += align_up(dq_packed_words(n, msgs[w].p.bits) * 4u, 256u) +
                 align_up(dq_num_buckets(n, msgs[w].p.bucket) * 4u, 256u);
    }
    return total;
}

// may_pipe: long gradients may go in pieces over the host thread's second stream, which the first such call creates.
static dq_status encode_host(dq_kind kind, const float* grad, uint64_t n, uint64_t seed, uint32_t worker,
                             uint64_t step, const dq_params* p, uint32_t* out_packed, float* out_scale,
                             void* workspace, uint64_t workspace_bytes, void* cuda_stream, bool may_pipe = true)
{
    uint32_t L;
    float alpha;
    dq_status s = check_params(p, kind, &L, &alpha);
    if (s != DQ_OK) return s;
    if (n == 0) return DQ_OK;
    if (n >= (1ull << 34)) return DQ_ERR_UNSUPPORTED;
    if (!grad || !out_packed || !out_scale || !workspace) return DQ_ERR_INVALID_ARG;
    if ((reinterpret_cast<uintptr_t>(workspace) & 255u) != 0u) return DQ_ERR_ALIGNMENT;
    if (workspace_bytes < dq_encode_workspace_bytes(n, p)) return DQ_ERR_INVALID_ARG;
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    const bool plain = (p->flags & DQ_FLAG_TEST_DROP_COPY) != 0u;        // (the hook is about one launch)
    // The launch flags say nothing about host buffers and the workspace, which the caller's previous kernel may use.
    dq_params unflagged = *p;
    unflagged.flags &= ~(DQ_FLAG_INPUT_READY | DQ_FLAG_OUTPUT_FREE);
    p = &unflagged;
    if (!plain && n <= kHostDirectElements) {
        const float* h_grad = pinned_view(grad, n);
        uint32_t* h_packed = h_grad ? pinned_view(out_packed, dq_packed_words(n, p->bits)) : nullptr;
        float* h_scale = h_packed ? pinned_view(out_scale, dq_num_buckets(n, p->bucket)) : nullptr;
        if (h_scale) {
            // Codes of 3, 5, 6 and 7 bits leave the kernel in pieces with gaps between them (store_group8), each a
            // transaction of its own on the bus: they go through the workspace (n = 1 M: 2 bits in place 105 us; 3 bits
            // in place 159 us, through the workspace 121; 7 bits 719 and 130).
            const bool staged = !is_pow2(p->bits);
            uint32_t* d_packed = staged ? static_cast<uint32_t*>(workspace) : h_packed;
            s = encode_common(kind, h_grad, n, seed, worker, step, p, d_packed, h_scale, st);
            if (s != DQ_OK) return s;
            const bool sent = !staged || cudaMemcpyAsync(out_packed, d_packed, dq_packed_words(n, p->bits) * 4u,
                                                         cudaMemcpyDeviceToHost, st) == cudaSuccess;
            return cudaStreamSynchronize(st) == cudaSuccess && sent ? DQ_OK : DQ_ERR_CUDA;
        }
    }
    uint8_t* ws = static_cast<uint8_t*>(workspace);
    float* d_grad = reinterpret_cast<float*>(ws);
    ws += align_up(n * 4u, 256u);
    uint32_t* d_packed = reinterpret_cast<uint32_t*>(ws);
    const uint64_t pbytes = dq_packed_words(n, p->bits) * 4u;
    ws += align_up(pbytes, 256u);
    float* d_scale = reinterpret_cast<float*>(ws);
    const uint64_t sbytes = dq_num_buckets(n, p->bucket) * 4u;
    HostPipe* pipe = (may_pipe && !plain && n >= kHostPieceElements) ? host_pipe() : nullptr;
    if (pipe) {
        // The gradient is what takes long: a small last piece, so that little is left to do when it arrives.
        static constexpr uint32_t cuts[kHostPieces + 1] = {0u, 14u, 16u};
        bool ok = true;
        s = DQ_OK;
        for (int i = 0; i < kHostPieces && ok && s == DQ_OK; ++i) {
            const uint64_t lo = piece_start(n, p->bucket, cuts[i]), hi = piece_start(n, p->bucket, cuts[i + 1]);
            if (lo == hi) continue;
            ok = cudaMemcpyAsync(d_grad + lo, grad + lo, (hi - lo) * 4u, cudaMemcpyHostToDevice, st) == cudaSuccess &&
                 cudaEventRecord(pipe->arrived[i], st) == cudaSuccess &&
                 cudaStreamWaitEvent(pipe->stream, pipe->arrived[i], 0) == cudaSuccess;
            if (!ok) break;
            const uint64_t w0 = lo / 32u * p->bits, w1 = hi == n ? pbytes / 4u : hi / 32u * p->bits;
            s = encode_common(kind, d_grad + lo, hi - lo, seed, worker, step, p, d_packed + w0, d_scale + lo / p->bucket,
                              pipe->stream, lo);
            ok = s != DQ_OK || cudaMemcpyAsync(out_packed + w0, d_packed + w0, (w1 - w0) * 4u, cudaMemcpyDeviceToHost,
                                               pipe->stream) == cudaSuccess;
        }
        if (ok && s == DQ_OK)
            ok = cudaMemcpyAsync(out_scale, d_scale, sbytes, cudaMemcpyDeviceToHost, pipe->stream) == cudaSuccess;
        // both streams, also after an error: copies that are queued use the caller's buffers
        const bool done = cudaStreamSynchronize(st) == cudaSuccess && cudaStreamSynchronize(pipe->stream) == cudaSuccess;
        return s != DQ_OK ? s : (ok && done) ? DQ_OK : DQ_ERR_CUDA;
    }
    if (cudaMemcpyAsync(d_grad, grad, n * 4u, cudaMemcpyHostToDevice, st) != cudaSuccess) return DQ_ERR_CUDA;
    s = encode_common(kind, d_grad, n, seed, worker, step, p, d_packed, d_scale, st);
    if (s != DQ_OK) {
        cudaStreamSynchronize(st);          // the copy above may still be reading the caller's buffer
        return s;
    }
    if (cudaMemcpyAsync(out_packed, d_packed, pbytes, cudaMemcpyDeviceToHost, st) != cudaSuccess) return DQ_ERR_CUDA;
    if (cudaMemcpyAsync(out_scale, d_scale, sbytes, cudaMemcpyDeviceToHost, st) != cudaSuccess) return DQ_ERR_CUDA;
    if (cudaStreamSynchronize(st) != cudaSuccess) return DQ_ERR_CUDA;
    return DQ_OK;
}

dq_status dqsg_encode_host(const float* grad, uint64_t n, uint64_t seed, uint32_t worker, uint64_t step,
                           const dq_params* p, uint32_t* out_packed, float* out_scale, void* workspace,
                           uint64_t workspace_bytes, void* cuda_stream)
{
    return encode_host(DQ_KIND_DQSG, grad, n, seed, worker, step, p, out_packed, out_scale, workspace,
                       workspace_bytes, cuda_stream);
}

dq_status ndqsg_encode_host(const float* grad, uint64_t n, uint64_t seed, uint32_t worker, uint64_t step,
                            const dq_params* p, uint32_t* out_packed, float* out_scale, void* workspace,
                            uint64_t workspace_bytes, void* cuda_stream)
{
    return encode_host(DQ_KIND_NDQSG, grad, n, seed, worker, step, p, out_packed, out_scale, workspace,
                       workspace_bytes, cuda_stream);
}

static dq_status decode_host(const dq_msg* msgs, uint32_t W, uint64_t n, uint64_t step, const float* side_info,
                             bool side_first, float* out_avg, void* workspace, uint64_t workspace_bytes,
                             void* cuda_stream)
{
    if (!msgs || W == 0u || W > DQ_MAX_WORKERS) return DQ_ERR_INVALID_ARG;
    if (side_first && msgs[0].kind != DQ_KIND_DQSG) return DQ_ERR_INVALID_ARG;
    for (uint32_t w = 0; w < W; ++w) {
        uint32_t L;
        float alpha;
        dq_status s = check_params(&msgs[w].p, msgs[w].kind, &L, &alpha);
        if (s != DQ_OK) return s;
        if (!msgs[w].packed || !msgs[w].scale) return DQ_ERR_INVALID_ARG;
        // what decode_common would reject, checked here before any copy is queued
        if (msgs[w].p.bucket != msgs[0].p.bucket) return DQ_ERR_UNSUPPORTED;
        if ((msgs[w].p.dither_bits == 16u) != (msgs[0].p.dither_bits == 16u)) return DQ_ERR_UNSUPPORTED;
        if (msgs[w].kind == DQ_KIND_NDQSG && !side_info && !side_first) return DQ_ERR_INVALID_ARG;
    }
    if (n == 0) return DQ_OK;
    if (n >= (1ull << 34)) return DQ_ERR_UNSUPPORTED;
    if (!out_avg || !workspace) return DQ_ERR_INVALID_ARG;
    if ((reinterpret_cast<uintptr_t>(workspace) & 255u) != 0u) return DQ_ERR_ALIGNMENT;
    if (workspace_bytes < dq_decode_workspace_bytes(msgs, W, n, side_info != nullptr)) return DQ_ERR_INVALID_ARG;
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    dq_msg dev_msgs[DQ_MAX_WORKERS];
    if (n <= kHostDirectElements) {
        float* h_out = pinned_view(out_avg, n);
        const float* h_side = (h_out && side_info) ? pinned_view(side_info, n) : nullptr;
        bool direct = h_out != nullptr && (!side_info || h_side);
        for (uint32_t w = 0; w < W && direct; ++w) {
            dev_msgs[w] = msgs[w];
            dev_msgs[w].packed = pinned_view(msgs[w].packed, dq_packed_words(n, msgs[w].p.bits));
            dev_msgs[w].scale = pinned_view(msgs[w].scale, dq_num_buckets(n, msgs[w].p.bucket));
            direct = dev_msgs[w].packed && dev_msgs[w].scale;
        }
        if (direct) {
            const dq_status s = decode_common(dev_msgs, W, n, step, h_side, h_out, nullptr, true, st, false, false, 0u,
                                              side_first);
            if (s != DQ_OK) return s;
            return cudaStreamSynchronize(st) == cudaSuccess ? DQ_OK : DQ_ERR_CUDA;
        }
    }
    uint8_t* ws = static_cast<uint8_t*>(workspace);
    float* d_out = reinterpret_cast<float*>(ws);
    ws += align_up(n * 4u, 256u);
    float* d_side = nullptr;
    if (side_info) {
        d_side = reinterpret_cast<float*>(ws);
        ws += align_up(n * 4u, 256u);
    }
    uint32_t* d_packed[DQ_MAX_WORKERS];
    float* d_scale[DQ_MAX_WORKERS];
    for (uint32_t w = 0; w < W; ++w) {
        dev_msgs[w] = msgs[w];
        d_packed[w] = reinterpret_cast<uint32_t*>(ws);
        ws += align_up(dq_packed_words(n, msgs[w].p.bits) * 4u, 256u);
        d_scale[w] = reinterpret_cast<float*>(ws);
        ws += align_up(dq_num_buckets(n, msgs[w].p.bucket) * 4u, 256u);
    }
    const uint32_t bucket = msgs[0].p.bucket;
    HostPipe* pipe = n >= kHostPieceElements ? host_pipe() : nullptr;
    // The mean is what takes long (a side information vector as long): a small first piece, so that it starts early.
    // Without the second stream there is one piece.
    static constexpr uint32_t two[kHostPieces + 1] = {0u, 5u, 16u}, one[2] = {0u, 16u};
    const uint32_t* cuts = pipe ? two : one;
    const int pieces = pipe ? kHostPieces : 1;
    cudaStream_t out_st = pipe ? pipe->stream : st;
    bool ok = true;
    dq_status s = DQ_OK;
    for (uint32_t w = 0; w < W && ok; ++w)
        ok = cudaMemcpyAsync(d_scale[w], msgs[w].scale, dq_num_buckets(n, bucket) * 4u, cudaMemcpyHostToDevice, st) ==
             cudaSuccess;
    for (int i = 0; i < pieces && ok && s == DQ_OK; ++i) {
        const uint64_t lo = piece_start(n, bucket, cuts[i]), hi = piece_start(n, bucket, cuts[i + 1]);
        if (lo == hi) continue;
        if (side_info)
            ok = cudaMemcpyAsync(d_side + lo, side_info + lo, (hi - lo) * 4u, cudaMemcpyHostToDevice, st) == cudaSuccess;
        for (uint32_t w = 0; w < W && ok; ++w) {
            const uint32_t bits = msgs[w].p.bits;
            const uint64_t w0 = lo / 32u * bits, w1 = hi == n ? dq_packed_words(n, bits) : hi / 32u * bits;
            ok = cudaMemcpyAsync(d_packed[w] + w0, msgs[w].packed + w0, (w1 - w0) * 4u, cudaMemcpyHostToDevice, st) ==
                 cudaSuccess;
            dev_msgs[w].packed = d_packed[w] + w0;
            dev_msgs[w].scale = d_scale[w] + lo / bucket;
        }
        if (!ok) break;
        // the kernel runs between two copies in: those have time, while the copies out follow each other without a gap
        s = decode_common(dev_msgs, W, hi - lo, step, side_info ? d_side + lo : nullptr, d_out + lo, nullptr, true, st,
                          false, false, lo, side_first);
        if (s != DQ_OK) break;
        if (pipe)
            ok = cudaEventRecord(pipe->arrived[i], st) == cudaSuccess &&
                 cudaStreamWaitEvent(out_st, pipe->arrived[i], 0) == cudaSuccess;
        ok = ok && cudaMemcpyAsync(out_avg + lo, d_out + lo, (hi - lo) * 4u, cudaMemcpyDeviceToHost, out_st) == cudaSuccess;
    }
    // both streams, also after an error: copies that are queued use the caller's buffers
    const bool done = cudaStreamSynchronize(st) == cudaSuccess && (!pipe || cudaStreamSynchronize(out_st) == cudaSuccess);
    return s != DQ_OK ? s : (ok && done) ? DQ_OK : DQ_ERR_CUDA;
}

dq_status ndqsg_decode_aggregate_host(const dq_msg* msgs, uint32_t W, uint64_t n, uint64_t step,
                                      const float* side_info, float* out_avg, void* workspace,
                                      uint64_t workspace_bytes, void* cuda_stream)
{
    return decode_host(msgs, W, n, step, side_info, false, out_avg, workspace, workspace_bytes, cuda_stream);
}

dq_status ndqsg_decode_aggregate_side_first_host(const dq_msg* msgs, uint32_t W, uint64_t n, uint64_t step,
                                                 float* out_avg, void* workspace, uint64_t workspace_bytes,
                                                 void* cuda_stream)
{
    return decode_host(msgs, W, n, step, nullptr, true, out_avg, workspace, workspace_bytes, cuda_stream);
}

// ------------------------------------------------------------------------------------------------ no allocation
// Staging area of dqsg_encode_host_static.  In host code this name is only a handle for the runtime, not a
// device address: the address the kernels and copies use is looked up with cudaGetSymbolAddress.
static __device__ __align__(256) unsigned char g_static_scratch[DQ_STATIC_SCRATCH_BYTES];

namespace {
std::mutex g_static_scratch_mutex;
void* g_static_scratch_addr[kMaxDevices] = {};

// Device address of g_static_scratch on the current device; looked up once per device.
dq_status static_scratch_address(void** out)
{
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return DQ_ERR_CUDA;
    std::lock_guard<std::mutex> lock(g_static_scratch_mutex);
    if (g_static_scratch_addr[dev] == nullptr) {
        void* ptr = nullptr;
        if (cudaGetSymbolAddress(&ptr, g_static_scratch) != cudaSuccess || ptr == nullptr) return DQ_ERR_CUDA;
        g_static_scratch_addr[dev] = ptr;
    }
    *out = g_static_scratch_addr[dev];
    return DQ_OK;
}
}  // namespace

dq_status dqsg_encode_host_static(const float* grad, uint64_t n, uint64_t seed, uint32_t worker, uint64_t step,
                                  const dq_params* p, uint32_t* out_packed, float* out_scale, void* cuda_stream)
{
    uint32_t L;
    float alpha;
    dq_status s = check_params(p, DQ_KIND_DQSG, &L, &alpha);
    if (s != DQ_OK) return s;
    if (n == 0) return DQ_OK;
    if (!grad || !out_packed || !out_scale) return DQ_ERR_INVALID_ARG;
    if (n >= (1ull << 34) || dq_encode_workspace_bytes(n, p) > (uint64_t)DQ_STATIC_SCRATCH_BYTES)
        return DQ_ERR_TOO_LARGE;
    void* scratch = nullptr;
    s = static_scratch_address(&scratch);
    if (s != DQ_OK) return s;
    // (no second stream: this call creates nothing, on whichever thread)
    return encode_host(DQ_KIND_DQSG, grad, n, seed, worker, step, p, out_packed, out_scale, scratch,
                       (uint64_t)DQ_STATIC_SCRATCH_BYTES, cuda_stream, false);
}

dq_status dq_device_error_flags(uint32_t* out_flags)
{
    if (!out_flags) return DQ_ERR_INVALID_ARG;
    unsigned int v = 0u, zero = 0u;
    if (cudaDeviceSynchronize() != cudaSuccess) return DQ_ERR_CUDA;
    if (cudaMemcpyFromSymbol(&v, g_dq_error_flags, sizeof(v)) != cudaSuccess) return DQ_ERR_CUDA;
    if (cudaMemcpyToSymbol(g_dq_error_flags, &zero, sizeof(zero)) != cudaSuccess) return DQ_ERR_CUDA;
    *out_flags = v;
    return DQ_OK;
}

uint64_t dq_launch_count(void) { return g_launches.load(); }

}  // extern "C"
