// Instances of the gate engine (gate_kernel.cuh): FP64, eight blocks a slot.
#include "gate_kernel.cuh"

namespace mpsvqe {
template cudaError_t launch_cluster<double, 256, 8, 1, false>(const DevMPS&, const CircDev&, int64_t, int64_t, int, int,
    const double*, double, int, cudaStream_t);
}  // namespace mpsvqe
