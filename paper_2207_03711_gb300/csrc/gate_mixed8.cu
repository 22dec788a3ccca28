// Instances of the gate engine (gate_kernel.cuh): mixed precision, eight blocks a slot.
#include "gate_kernel.cuh"

namespace mpsvqe {
template cudaError_t launch_cluster<float, 256, 8, 1, false>(const DevMPS&, const CircDev&, int64_t, int64_t, int, int,
    const double*, double, int, cudaStream_t);
template int max_clusters<float, 256, 8, 1, false>(int);
}  // namespace mpsvqe
