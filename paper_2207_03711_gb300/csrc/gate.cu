// Host side of the gate engine: how many blocks a slot gets, and the entry point for
// caller-owned memory. The kernel is gate_kernel.cuh.
#include <cmath>
#include <cstring>
#include <mutex>

#include "../../include/mpsvqe.h"
#include "kernels.cuh"

namespace mpsvqe {

template <class R, int NT, int C, int VG, bool RAW>
cudaError_t launch_cluster(const DevMPS& m, const CircDev& c, int64_t g0, int64_t g1, int slot0, int count,
                           const double* theta, double cutoff, int max_sweeps, cudaStream_t st);
// Slots that run at once on the current device (one thread block per SM).
template <class R, int NT, int C, int VG, bool RAW>
int max_clusters(int chi);

// Blocks per slot in mixed precision. chi <= 16: one (a step of these sizes is shorter than
// a cluster barrier is worth). chi 17..64: the most of 8, 4, 2, 1 with which all running slots
// (of all calls in progress) still run at once, with the same bits for each (8 virtual ranks).
// A chi = 64 gate takes 263 us with 8 blocks (up to 14 slots), 294 with 4, 342 with 2 and 477
// with 1 (152 slots); one block alone took 746 us before clusters, and 415 and 442 us a gate at
// 73 and 152 slots. Serving 152 single slots with 8 blocks each would run 14 at a time: 2 860 us
// a round of gates instead of 477. chi > 64: 8, M' needs their shared memory.
template <bool RAW>
static cudaError_t launch_mixed(const DevMPS& m, const CircDev& c, int64_t g0, int64_t g1, int slot0, int count,
                                int running, const double* theta, double cutoff, int max_sweeps, cudaStream_t st) {
  if (m.chi <= 16)
    return launch_cluster<float, 256, 1, 2, RAW>(m, c, g0, g1, slot0, count, theta, cutoff, max_sweeps, st);
  if constexpr (!RAW) {
    if (m.chi <= 64 && running > max_clusters<float, 256, 8, 1, RAW>(m.chi)) {
      if (running <= max_clusters<float, 256, 4, 2, RAW>(m.chi))
        return launch_cluster<float, 256, 4, 2, RAW>(m, c, g0, g1, slot0, count, theta, cutoff, max_sweeps, st);
      if (running <= max_clusters<float, 256, 2, 4, RAW>(m.chi))
        return launch_cluster<float, 256, 2, 4, RAW>(m, c, g0, g1, slot0, count, theta, cutoff, max_sweeps, st);
      return launch_cluster<float, 512, 1, 8, RAW>(m, c, g0, g1, slot0, count, theta, cutoff, max_sweeps, st);
    }
  }
  return launch_cluster<float, 256, 8, 1, RAW>(m, c, g0, g1, slot0, count, theta, cutoff, max_sweeps, st);
}

cudaError_t launch_circuit(const DevMPS& m, int prec, const CircDev& c, int64_t g0, int64_t g1, int slot0, int count,
                           int running, const double* theta, double cutoff, int max_sweeps, cudaStream_t st) {
  if (prec == MPS_PREC_FP64)
    return launch_cluster<double, 256, 8, 1, false>(m, c, g0, g1, slot0, count, theta, cutoff, max_sweeps, st);
  return launch_mixed<false>(m, c, g0, g1, slot0, count, running, theta, cutoff, max_sweeps, st);
}

}  // namespace mpsvqe

// ------------------------------------------------------------------------------
// Allocation-free variant of the gate engine for callers that cannot allocate device
// memory themselves or through this library (the paper has no counterpart; see the
// declaration of mps_apply_gates_noalloc in include/mpsvqe.h). Its workspace lives in
// the file-scope array below, which every GPU that loads the library keeps until the
// process exits; all calls share it.
namespace mpsvqe {
namespace {
constexpr size_t kNoAllocScratchBytes = size_t(1) << 20;   // 1 MiB
constexpr int kNoAllocMaxChi = 64;
}  // namespace
}  // namespace mpsvqe

static __device__ __align__(256) unsigned char g_noalloc_scratch[mpsvqe::kNoAllocScratchBytes];

namespace {
std::mutex g_noalloc_mu;
void* g_noalloc_ptr[64] = {nullptr};
}  // namespace

extern "C" int mps_apply_gates_noalloc(int n_qubits, int chi, void* site_tensors, const int64_t* site_offsets,
                                       double* lambdas, int32_t* ranks, int64_t n_gates, const int32_t* bonds,
                                       const double* gates, void* cuda_stream, double* discarded_weight) {
  using namespace mpsvqe;
  if (!site_tensors || !site_offsets || !lambdas || !ranks || (n_gates > 0 && (!bonds || !gates))) {
    set_error_message("mps_apply_gates_noalloc: null device pointer");
    return MPS_EINVAL;
  }
  if (n_qubits < 2 || n_qubits > kMaxQubits || chi < 1 || chi > kNoAllocMaxChi || n_gates < 0) {
    set_error_message("mps_apply_gates_noalloc: needs 2 <= n_qubits <= 128, 1 <= chi <= 64 and n_gates >= 0 "
                      "(the fixed 1 MiB device workspace holds one chi <= 64 gate step)");
    return MPS_EINVAL;
  }
  const size_t mm = 2 * (size_t)chi;
  const size_t off_M = 0;
  const size_t off_X = off_M + ((mm * mm * 8 + 255) & ~(size_t)255);
  const size_t off_S = off_X + ((mm * (mm + 16) * 8 + 255) & ~(size_t)255);
  const size_t off_dw = off_S + ((16 * (size_t)chi * chi * 8 + 255) & ~(size_t)255);
  const size_t off_end = off_dw + 256;
  if (off_end > kNoAllocScratchBytes) {
    set_error_message("mps_apply_gates_noalloc: workspace larger than the 1 MiB device array");
    return MPS_EINVAL;
  }
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) {
    set_error_message("mps_apply_gates_noalloc: no current CUDA device");
    return MPS_ECUDA;
  }
  unsigned char* base = nullptr;
  {
    std::lock_guard<std::mutex> lock(g_noalloc_mu);
    if (!g_noalloc_ptr[dev]) {
      void* p = nullptr;
      if (cudaGetSymbolAddress(&p, g_noalloc_scratch) != cudaSuccess || !p) {
        set_error_message("mps_apply_gates_noalloc: cudaGetSymbolAddress of the device workspace failed");
        return MPS_ECUDA;
      }
      g_noalloc_ptr[dev] = p;
    }
    base = (unsigned char*)g_noalloc_ptr[dev];
  }
  cudaStream_t st = (cudaStream_t)cuda_stream;
  DevMPS d{};
  d.n = n_qubits;
  d.chi = chi;
  d.n_slots = 1;
  d.slot_elems = 0;
  d.site_off = site_offsets;
  d.B = site_tensors;
  d.lam = lambdas;
  d.rank = ranks;
  d.work_M = base + off_M;
  d.work_X = base + off_X;
  d.work_S = base + off_S;
  d.dw = (double*)(base + off_dw);
  d.stat = (int*)(base + off_dw + 8);
  d.prof = (unsigned long long*)(base + off_dw + 64);
  // the shared array keeps the previous call's contents: clear the accumulators
  if (cudaMemsetAsync(base + off_dw, 0, 256, st) != cudaSuccess) return MPS_ECUDA;
  CircDev c{};
  c.gates = nullptr;
  c.n_gates = n_gates;
  c.mats = gates;
  c.n_params = 1;
  c.raw_bond = bonds;
  const double* theta = (const double*)(base + off_dw + 128);   // never read: every gate is fixed
  for (int64_t g0 = 0; g0 < n_gates; g0 += 16384) {
    const int64_t g1 = g0 + 16384 < n_gates ? g0 + 16384 : n_gates;
    if (launch_mixed<true>(d, c, g0, g1, 0, 1, 1, theta, std::ldexp(1.0, -20), 60, st) != cudaSuccess) return MPS_ECUDA;
  }
  if (discarded_weight) {
    // the discarded weight and the status words sit next to each other in the array:
    // one copy brings both back
    unsigned char host[8 + 4 * kStatWords];
    if (cudaMemcpyAsync(host, d.dw, sizeof(host), cudaMemcpyDeviceToHost, st) != cudaSuccess) return MPS_ECUDA;
    if (cudaStreamSynchronize(st) != cudaSuccess) return MPS_ECUDA;
    int stat[kStatWords];
    std::memcpy(discarded_weight, host, 8);
    std::memcpy(stat, host + 8, sizeof(stat));
    if (stat[5]) {
      set_error_message("mps_apply_gates_noalloc: a bond outside [0, n-2] or a rank outside its capacity "
                        "reached the device; gates from there on were not applied");
      return MPS_EINVAL;
    }
    if (stat[4] > 0) {
      set_error_message("mps_apply_gates_noalloc: a gate's M' held a NaN or Inf; the gate was skipped");
      return MPS_ENONFINITE;
    }
    if (stat[1] > 0) {
      set_error_message("mps_apply_gates_noalloc: a Jacobi SVD fallback reached its sweep cap");
      return MPS_ENOCONV;
    }
  }
  return MPS_OK;
}
