// Instances of the gate engine (gate_kernel.cuh): caller-owned tensors (mixed precision).
#include "gate_kernel.cuh"

namespace mpsvqe {
template cudaError_t launch_cluster<float, 256, 1, 2, true, false>(const DevMPS&, const CircDev&, int64_t, int64_t, int, int,
    const double*, double, int, cudaStream_t);
template cudaError_t launch_cluster<float, 256, 8, 1, true, false>(const DevMPS&, const CircDev&, int64_t, int64_t, int, int,
    const double*, double, int, cudaStream_t);
}  // namespace mpsvqe
