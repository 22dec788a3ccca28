// Host side of the gate engine: how many blocks a slot gets, and the entry point for
// caller-owned memory. The kernel is gate_kernel.cuh.
#include <cmath>
#include <cstring>
#include <mutex>

#include "../../include/mpsvqe.h"
#include "kernels.cuh"

namespace mpsvqe {

template <class R, int NT, int C, int VG, bool RAW, bool TG>
cudaError_t launch_cluster(const DevMPS& m, const CircDev& c, int64_t g0, int64_t g1, int slot0, int count,
                           const double* theta, double cutoff, int max_sweeps, cudaStream_t st);
// Slots that run at once on the current device (one thread block per SM); 0 where chi does not fit.
template <class R, int NT, int C, int VG, bool RAW, bool TG>
int max_clusters(int chi);

namespace {
struct Engine {
  decltype(&launch_cluster<float, 256, 8, 1, false, false>) launch;
  int (*slots)(int chi);
};
template <class R, int NT, int C, int VG, bool TG>
constexpr Engine engine() {
  return {launch_cluster<R, NT, C, VG, false, TG>, max_clusters<R, NT, C, VG, false, TG>};
}
// Blocks per slot: the most with which all running slots (of all calls in progress) still run at
// once, else the instance that runs most of them; each has the same bits (8 virtual ranks). One
// slot finishes soonest on eight blocks, but a gate costs the fewest SM cycles in one. Time of a
// gate of a UCCSD circuit in us, at 14 / 76 / 152 / 304 slots, and with one block a slot before
// clusters (any number up to 152 / 304):
//   mixed  chi = 33  114 / 158 / 218 / 433       209 - 212 / 423
//          chi = 64  197 / 315 / 423 / 820       415 - 442 / 849
//          chi = 72  161 / 276 / 542 / 1 060     569 - 601 / 1 157
//          chi = 128 252 / 590 / 1 078 / 1 953   1 186 - 1 275 / 2 351
//   FP64   chi = 16  185 / 206 / 402 / 792       1 545 - 1 599 / 3 116 (random rotations)
//          chi = 64  694 / 924 / 1 820           3 963 - 4 062
// (From 77 slots on caps of 33 are 2 %, of 65 to 67 8 % behind the one-block engine of old.)
// Eight blocks for all in FP64 and above chi = 64 took 1 876 and 6 158 us (FP64), 2 900 - 7 200 us
// (mixed, chi = 65 - 128) at 152 slots. One block holds M' up to chi = 70, two up to 96 (FP64 72);
// above, two blocks keep part of it in L2. Mixed chi <= 16 takes one block always: a step of
// these sizes is shorter than a cluster barrier is worth.
constexpr Engine kMixed[] = {engine<float, 256, 8, 1, false>(), engine<float, 256, 4, 2, false>(),
                             engine<float, 256, 2, 4, false>(), engine<float, 256, 2, 4, true>(),
                             engine<float, 512, 1, 8, false>()};
constexpr Engine kFp64[] = {engine<double, 256, 8, 1, false>(), engine<double, 256, 4, 2, false>(),
                            engine<double, 256, 2, 4, false>(), engine<double, 256, 2, 4, true>()};
template <int N>
const Engine& choose(const Engine (&of)[N], int chi, int running) {
  const Engine* best = &of[0];
  int most = 0;
  for (const Engine& e : of) {
    const int n = e.slots(chi);
    if (n > most) {
      best = &e;
      most = n;
    }
    if (n >= running) break;
  }
  return *best;
}
}  // namespace

cudaError_t launch_circuit(const DevMPS& m, int prec, const CircDev& c, int64_t g0, int64_t g1, int slot0, int count,
                           int running, const double* theta, double cutoff, int max_sweeps, cudaStream_t st) {
  if (prec != MPS_PREC_FP64 && m.chi <= 16)
    return launch_cluster<float, 256, 1, 2, false, false>(m, c, g0, g1, slot0, count, theta, cutoff, max_sweeps, st);
  const Engine& e = prec == MPS_PREC_FP64 ? choose(kFp64, m.chi, running) : choose(kMixed, m.chi, running);
  return e.launch(m, c, g0, g1, slot0, count, theta, cutoff, max_sweeps, st);
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
    const auto launch = chi <= 16 ? launch_cluster<float, 256, 1, 2, true, false> : launch_cluster<float, 256, 8, 1, true, false>;
    if (launch(d, c, g0, g1, 0, 1, theta, std::ldexp(1.0, -20), 60, st) != cudaSuccess) return MPS_ECUDA;
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
