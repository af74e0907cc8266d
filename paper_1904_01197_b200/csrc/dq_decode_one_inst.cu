// Instantiations of decode_one_kernel for one dither width (DQ_INST_DITH, given on the compiler's command line) and all
// code widths.
#include "dq_decode_one.cuh"
#include "dq_launch.h"

#ifndef DQ_INST_DITH
#error "compile with -DDQ_INST_DITH=<32|16>"
#endif

namespace dq {
namespace {

template <int BITS, int R>
cudaError_t launch_one(const DecodeArgsOf<1>& a, cudaStream_t st)
{
    constexpr uint32_t per_cta = kOneThreads * R;
    return launch_overlapped(decode_one_kernel<DQ_INST_DITH, BITS, R>, (uint32_t)((a.num_groups + per_cta - 1u) / per_cta),
                             (uint32_t)kOneThreads, 0, st, 1u, a);
}

template <int BITS>
cudaError_t launch_bits(const DecodeArgsOf<1>& a, int R, cudaStream_t st)
{
    return R == 1 ? launch_one<BITS, 1>(a, st) : launch_one<BITS, 4>(a, st);
}

}  // namespace

#define DQ_NAME2(D) launch_decode_one_d##D
#define DQ_NAME(D) DQ_NAME2(D)

cudaError_t DQ_NAME(DQ_INST_DITH)(const DecodeArgsOf<1>& a, int R, cudaStream_t st)
{
    switch (a.w[0].variant & 7u) {
        case 0: return launch_bits<1>(a, R, st);
        case 1: return launch_bits<2>(a, R, st);
        case 2: return launch_bits<3>(a, R, st);
        case 3: return launch_bits<4>(a, R, st);
        case 4: return launch_bits<5>(a, R, st);
        case 5: return launch_bits<6>(a, R, st);
        case 6: return launch_bits<7>(a, R, st);
        default: return launch_bits<8>(a, R, st);
    }
}

}  // namespace dq
