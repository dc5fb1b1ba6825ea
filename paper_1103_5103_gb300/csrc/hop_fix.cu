// Instantiations of the fixed-point FP64 hop (hop_fix.cuh).
#include "hop_fix.cuh"

namespace wl {

int hop_fix_launch(int dagger, const HopArgs &a, const EpiStore &e, int blocks_per_sm, cudaStream_t s)
{
    if (dagger) launch_k_hop_fix<true>(a, e, blocks_per_sm, s);
    else launch_k_hop_fix<false>(a, e, blocks_per_sm, s);
    WL_CUDA_TRY(cudaGetLastError());
    return WL_OK;
}

template <int KIND>
static void reduce_kind(int dagger, const HopArgs &a, const void *epi, cudaStream_t s)
{
    const auto &e = *static_cast<const EpiReduce<KIND> *>(epi);
    if (dagger) launch_k_hop_fix_reduce<true, KIND>(a, e, s);
    else launch_k_hop_fix_reduce<false, KIND>(a, e, s);
}

int hop_fix_reduce_launch(int kind, int dagger, const HopArgs &a, const void *epi, cudaStream_t s)
{
    switch (kind) {
    case 0: reduce_kind<0>(dagger, a, epi, s); break;
    case 1: reduce_kind<1>(dagger, a, epi, s); break;
    case 2: reduce_kind<2>(dagger, a, epi, s); break;
    default: reduce_kind<3>(dagger, a, epi, s); break;
    }
    WL_CUDA_TRY(cudaGetLastError());
    return WL_OK;
}

}  // namespace wl
