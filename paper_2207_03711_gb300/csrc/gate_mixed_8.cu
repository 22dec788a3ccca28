// Instances of the gate engine (gate_kernel.cuh): mixed precision, eight and four blocks a slot.
#include "gate_kernel.cuh"

namespace mpsvqe {
template cudaError_t launch_cluster<float, 256, 8, 1, false, false>(const DevMPS&, const CircDev&, int64_t, int64_t, int, int,
    const double*, double, int, cudaStream_t);
template int max_clusters<float, 256, 8, 1, false, false>(int);
template cudaError_t launch_cluster<float, 256, 4, 2, false, false>(const DevMPS&, const CircDev&, int64_t, int64_t, int, int,
    const double*, double, int, cudaStream_t);
template int max_clusters<float, 256, 4, 2, false, false>(int);
}  // namespace mpsvqe
