// k_edge_f32.cu -- instantiations of the edge pass (k_edge.cuh) for FP32 storage, plain FP32
// sums
#include "k_edge.cuh"

namespace amgd {

cudaError_t launch_edge_f32_comp(bool in_place, bool unit_w, const EdgeArgs &a, cudaStream_t s);

cudaError_t launch_edge_f32(bool in_place, bool unit_w, const EdgeArgs &a, cudaStream_t s)
{
    const cudaError_t e = cudaMemsetAsync(a.defer_count, 0, sizeof(uint32_t), s);
    if (e != cudaSuccess) return e;
    return a.compensated ? launch_edge_f32_comp(in_place, unit_w, a, s)
                         : edge_impl::dispatch<float, false>(in_place, unit_w, a, s);
}

}  // namespace amgd
