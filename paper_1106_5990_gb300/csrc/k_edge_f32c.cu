// k_edge_f32c.cu -- instantiations of the edge pass (k_edge.cuh) for FP32 storage, compensated
// FP32 sums
#include "k_edge.cuh"

namespace amgd {

cudaError_t launch_edge_f32_comp(bool in_place, bool unit_w, const EdgeArgs &a, cudaStream_t s)
{
    return edge_impl::dispatch<float, true>(in_place, unit_w, a, s);
}

}  // namespace amgd
