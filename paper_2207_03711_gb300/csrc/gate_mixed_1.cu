// Instances of the gate engine (gate_kernel.cuh): mixed precision, one block a slot.
#include "gate_kernel.cuh"

namespace mpsvqe {
template cudaError_t launch_cluster<float, 512, 1, 8, false, false>(const DevMPS&, const CircDev&, int64_t, int64_t, int, int,
    const double*, double, int, cudaStream_t);
template int max_clusters<float, 512, 1, 8, false, false>(int);
}  // namespace mpsvqe
