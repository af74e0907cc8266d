// Instantiations of decode_aggregate_kernel for one dither width, one side-information mode and one group size
// (DQ_INST_DITH, DQ_INST_RUN = a DecSide value, DQ_INST_E, given on the compiler's command line) and all sets of variants.
#include <cstring>

#include "dq_decode.cuh"
#include "dq_launch.h"

#ifndef DQ_INST_DITH
#error "compile with -DDQ_INST_DITH=<32|16|0> -DDQ_INST_RUN=<0|1|2> -DDQ_INST_E=<32|16|8>"
#endif

namespace dq {

#define DQ_NAME2(D, R, E) launch_decode_d##D##_r##R##_e##E
#define DQ_NAME(D, R, E) DQ_NAME2(D, R, E)

namespace {

template <int E, int SET, int MAXW = 64>
cudaError_t launch_set(const DecodeArgsOf<MAXW>& a, uint32_t grid, cudaStream_t st)
{
    return launch_overlapped(decode_aggregate_kernel<DQ_INST_DITH, DQ_INST_RUN, E, SET, MAXW>, grid, (uint32_t)kDecThreads, 0,
                             st, 1u, a);
}

// All routines: with the registers that they want, or held to eight CTAs per SM (see dec_ctas_per_sm).
template <int E, int MAXW>
cudaError_t launch_all(const DecodeArgsOf<MAXW>& a, uint32_t grid, int sms, cudaStream_t st)
{
    constexpr uint32_t fits = dec_ctas_per_sm(DQ_INST_DITH, E, kSetAll);
    if constexpr (E < 32 && fits < 8u) {
        bool full = grid > fits * (uint32_t)sms && grid <= 8u * (uint32_t)sms;
        if constexpr (E == 8 && DQ_INST_DITH == 32 && DQ_INST_RUN == kSideGiven) {
            for (uint32_t w = 0; w < a.W; ++w) full = full || ((a.w[w].variant & 7u) >= 4u && (a.w[w].variant & 7u) < 7u);
        }
        if (full) return launch_set<E, kSetAllFull>(a, grid, st);
    }
    return launch_set<E, kSetAll>(a, grid, st);
}

template <int E, int A>
cudaError_t launch_pair(int b, const DecodeArgs& a, uint32_t grid, cudaStream_t st)
{
    if constexpr (DQ_INST_DITH == 0) {        // (the receiver without the dither takes DQSG messages only)
        return launch_set<E, pair_set(A, A)>(a, grid, st);
    } else {
        switch (b) {
            case 1: return launch_set<E, pair_set(A, 1)>(a, grid, st);
            case 2: return launch_set<E, pair_set(A, 2)>(a, grid, st);
            case 3: return launch_set<E, pair_set(A, 3)>(a, grid, st);
            default: return launch_set<E, pair_set(A, 4)>(a, grid, st);
        }
    }
}

template <int E>
cudaError_t launch_groups_of(const DecodeArgs& a, int sms, cudaStream_t st)
{
    const uint32_t grid = (uint32_t)((a.num_groups + kDecThreads - 1u) / kDecThreads);
    bool usual = true, one_pair = true;
    int width[2] = {0, 0};              // code widths of the DQSG and of the NDQSG messages
    for (uint32_t w = 0; w < a.W; ++w) {
        const uint32_t v = a.w[w].variant;
        usual = usual && is_usual_variant(v);
        if (!usual) break;
        int& have = width[v >> 3];
        one_pair = one_pair && (have == 0 || have == (int)(v & 7u) + 1);
        have = (int)(v & 7u) + 1;
    }
    if constexpr (E >= 16) {
        // (not for one message in groups of 16, where it is 4 % faster or 2 % slower; two messages of the 32-bit stream against
        // message 0, the running mean or nothing take 1 to 5 % less, against a vector 2 % less to 3 % more; of the 16-bit stream
        // up to 13 % more with messages from HBM: running mean, 3 and 2 bits, n = 1.7 M 4.7 and 5.3 us)
        const bool two_gain = DQ_INST_DITH == 32 && (DQ_INST_RUN != kSideGiven || width[1] == 0);
        if (usual && one_pair && (E == 32 || a.W > 2u || (a.W == 2u && two_gain))) {
            if (width[0] == 0) width[0] = width[1];
            if (width[1] == 0) width[1] = width[0];
            switch (width[0]) {
                case 1: return launch_pair<E, 1>(width[1], a, grid, st);
                case 2: return launch_pair<E, 2>(width[1], a, grid, st);
                case 3: return launch_pair<E, 3>(width[1], a, grid, st);
                default: return launch_pair<E, 4>(width[1], a, grid, st);
            }
        }
    }
    bool odd = DQ_INST_DITH != 0 && !usual;       // (the receiver without the dither takes DQSG messages only: usual or wide)
    for (uint32_t w = 0; w < a.W; ++w) odd = odd && is_odd_variant(a.w[w].variant);
    if constexpr (E == 8) {
        // short gradients: the launch itself counts
        if (a.W <= (uint32_t)kDecFewWorkers) {
            DecodeArgsOf<kDecFewWorkers> few;
            static_cast<DecodeHead&>(few) = a;
            std::memcpy(few.w, a.w, a.W * sizeof(DecWorker));
            if constexpr (DQ_INST_DITH != 0) {
                if (odd) return launch_set<E, kSetOdd, kDecFewWorkers>(few, grid, st);
            }
            return usual ? launch_set<E, kSetUsual, kDecFewWorkers>(few, grid, st) : launch_all<E>(few, grid, sms, st);
        }
    }
    if constexpr (E < 32 && DQ_INST_DITH != 0) {
        if (odd) return launch_set<E, kSetOdd>(a, grid, st);
    }
    return usual ? launch_set<E, kSetUsual>(a, grid, st) : launch_all<E>(a, grid, sms, st);
}

}  // namespace

cudaError_t DQ_NAME(DQ_INST_DITH, DQ_INST_RUN, DQ_INST_E)(const DecodeArgs& a, int sms, cudaStream_t st)
{
    return launch_groups_of<DQ_INST_E>(a, sms, st);
}

}  // namespace dq
