// Instances of the gate engine (gate_kernel.cuh): mixed precision, bond caps up to 16.
#include "gate_kernel.cuh"

namespace mpsvqe {
template cudaError_t launch_cluster<float, 256, 1, 2, false, false>(const DevMPS&, const CircDev&, int64_t, int64_t, int, int,
    const double*, double, int, cudaStream_t);
}  // namespace mpsvqe
