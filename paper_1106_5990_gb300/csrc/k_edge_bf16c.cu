// k_edge_bf16c.cu -- instantiations of the edge pass (k_edge.cuh) for BF16 storage, compensated
// FP32 sums
#include "k_edge.cuh"

namespace amgd {

cudaError_t launch_edge_bf16_comp(bool in_place, bool unit_w, const EdgeArgs &a, cudaStream_t s)
{
    return edge_impl::dispatch<__nv_bfloat16, true>(in_place, unit_w, a, s);
}

}  // namespace amgd
