// Launch interface between the host side of the C ABI (dq_b200.cu) and the translation units that hold the
// kernel instantiations.  The encode and decode kernels are templates with dozens of instantiations; they are
// compiled as separate translation units (one per encoder mode and dither width, one per decoder variant) so that
// the library builds in parallel.
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <utility>

namespace dq {

struct EncodeArgs;
struct DirectArgs;
template <int MAXW> struct DecodeArgsOf;
using DecodeArgs = DecodeArgsOf<64>;

// Launch with programmatic stream serialization allowed: a kernel may become resident while the previous one of the
// stream drains, which hides launch latency.  Every kernel executes griddepcontrol.wait before it writes anything, and
// before it reads anything that the previous kernel may have produced -- unless the caller's flags say that an encode
// need not (EncodeArgs::early_read, early_store), which they say about the previous kernel only.  Therefore at least one
// CTA of every kernel executes griddepcontrol.launch_dependents only after its own wait: a kernel then starts when
// everything before its predecessor is complete, and no more than two kernels ever overlap.
template <typename... KArgs, typename... Args>
cudaError_t launch_overlapped(void (*kernel)(KArgs...), uint32_t grid, uint32_t block, size_t smem, cudaStream_t st,
                              uint32_t cluster, Args&&... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (cluster > 1u) {
        attr[1].id = cudaLaunchAttributeClusterDimension;
        attr[1].val.clusterDim.x = cluster;
        attr[1].val.clusterDim.y = 1;
        attr[1].val.clusterDim.z = 1;
        cfg.numAttrs = 2;
    }
    return cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}

// Encoder: mode = EncMode, dith = 32 or 16.  One function per (mode, dith) translation unit; launch_encode picks.
#define DQ_DECLARE_ENCODE(MODE, DITH)                                                                              \
    cudaError_t launch_encode_m##MODE##_d##DITH(uint32_t bits, const CUtensorMap& map, const EncodeArgs& a,        \
                                                uint32_t grid, cudaStream_t st);
DQ_DECLARE_ENCODE(0, 32) DQ_DECLARE_ENCODE(1, 32) DQ_DECLARE_ENCODE(2, 32) DQ_DECLARE_ENCODE(3, 32)
DQ_DECLARE_ENCODE(0, 16) DQ_DECLARE_ENCODE(1, 16) DQ_DECLARE_ENCODE(2, 16) DQ_DECLARE_ENCODE(3, 16)
#undef DQ_DECLARE_ENCODE

// The same for the direct encoder; R = groups per lane, 1 or 4; kind = DirectKind.
#define DQ_DECLARE_DIRECT(MODE, DITH)                                                                              \
    cudaError_t launch_direct_m##MODE##_d##DITH(uint32_t bits, int R, int kind, const DirectArgs& a,               \
                                                uint32_t grid, uint32_t threads, cudaStream_t st);
DQ_DECLARE_DIRECT(0, 32) DQ_DECLARE_DIRECT(1, 32) DQ_DECLARE_DIRECT(2, 32) DQ_DECLARE_DIRECT(3, 32)
DQ_DECLARE_DIRECT(0, 16) DQ_DECLARE_DIRECT(1, 16) DQ_DECLARE_DIRECT(2, 16) DQ_DECLARE_DIRECT(3, 16)
#undef DQ_DECLARE_DIRECT

// Decoder: dith = 32, 16 or 0 (no dither at the receiver); run = DecSide (0 given vector or none, 1 running mean,
// 2 reconstruction of message 0).
// group_size: elements per lane, 32, 16 or 8; the grid follows from a.num_groups.  sms: the device's SMs.
#define DQ_DECLARE_DECODE(DITH, RUN)                                                                               \
    cudaError_t launch_decode_d##DITH##_r##RUN##_e32(const DecodeArgs& a, int sms, cudaStream_t st);               \
    cudaError_t launch_decode_d##DITH##_r##RUN##_e16(const DecodeArgs& a, int sms, cudaStream_t st);               \
    cudaError_t launch_decode_d##DITH##_r##RUN##_e8(const DecodeArgs& a, int sms, cudaStream_t st);                \
    inline cudaError_t launch_decode_d##DITH##_r##RUN(const DecodeArgs& a, int group_size, int sms, cudaStream_t st) \
    {                                                                                                              \
        return group_size == 32   ? launch_decode_d##DITH##_r##RUN##_e32(a, sms, st)                               \
               : group_size == 16 ? launch_decode_d##DITH##_r##RUN##_e16(a, sms, st)                               \
                                  : launch_decode_d##DITH##_r##RUN##_e8(a, sms, st);                               \
    }
DQ_DECLARE_DECODE(32, 0) DQ_DECLARE_DECODE(32, 1) DQ_DECLARE_DECODE(16, 0) DQ_DECLARE_DECODE(16, 1)
DQ_DECLARE_DECODE(32, 2) DQ_DECLARE_DECODE(16, 2)
DQ_DECLARE_DECODE(0, 0)
#undef DQ_DECLARE_DECODE

// Decoder of one DQSG message; R = groups of 8 elements per lane, 1 or 4.
cudaError_t launch_decode_one_d32(const DecodeArgsOf<1>& a, int R, cudaStream_t st);
cudaError_t launch_decode_one_d16(const DecodeArgsOf<1>& a, int R, cudaStream_t st);

}  // namespace dq
