// Instantiations of decode_aggregate_kernel for one dither width and one side-information mode (DQ_INST_DITH,
// DQ_INST_RUN = a DecSide value, given on the compiler's command line), all group sizes and both sets of variants.
#include <cstring>

#include "dq_decode.cuh"
#include "dq_launch.h"

#ifndef DQ_INST_DITH
#error "compile with -DDQ_INST_DITH=<32|16|0> -DDQ_INST_RUN=<0|1|2>"
#endif

namespace dq {

#define DQ_NAME2(D, R) launch_decode_d##D##_r##R
#define DQ_NAME(D, R) DQ_NAME2(D, R)

namespace {

template <int E>
cudaError_t launch_groups_of(const DecodeArgs& a, cudaStream_t st)
{
    const uint32_t grid = (uint32_t)((a.num_groups + kDecThreads - 1u) / kDecThreads);
    bool usual = true;
    for (uint32_t w = 0; w < a.W; ++w) usual = usual && is_usual_variant(a.w[w].variant);
    if constexpr (E == 8) {
        // short gradients: the launch itself counts
        if (a.W <= (uint32_t)kDecFewWorkers) {
            auto k = usual ? decode_aggregate_kernel<DQ_INST_DITH, DQ_INST_RUN, E, false, kDecFewWorkers>
                           : decode_aggregate_kernel<DQ_INST_DITH, DQ_INST_RUN, E, true, kDecFewWorkers>;
            DecodeArgsOf<kDecFewWorkers> few;
            static_cast<DecodeHead&>(few) = a;
            std::memcpy(few.w, a.w, a.W * sizeof(DecWorker));
            return launch_overlapped(k, grid, (uint32_t)kDecThreads, 0, st, 1u, few);
        }
    }
    auto k = usual ? decode_aggregate_kernel<DQ_INST_DITH, DQ_INST_RUN, E, false, 64>
                   : decode_aggregate_kernel<DQ_INST_DITH, DQ_INST_RUN, E, true, 64>;
    return launch_overlapped(k, grid, (uint32_t)kDecThreads, 0, st, 1u, a);
}

}  // namespace

cudaError_t DQ_NAME(DQ_INST_DITH, DQ_INST_RUN)(const DecodeArgs& a, int group_size, cudaStream_t st)
{
    if (group_size == 32) return launch_groups_of<32>(a, st);
    if (group_size == 16) return launch_groups_of<16>(a, st);
    return launch_groups_of<8>(a, st);
}

}  // namespace dq
