// Instances of the gate engine (gate_kernel.cuh): FP64, two blocks a slot.
#include "gate_kernel.cuh"

namespace mpsvqe {
template cudaError_t launch_cluster<double, 256, 2, 4, false, false>(const DevMPS&, const CircDev&, int64_t, int64_t, int, int,
    const double*, double, int, cudaStream_t);
template int max_clusters<double, 256, 2, 4, false, false>(int);
}  // namespace mpsvqe
