// FP64 environment contractions of the trie measurement on the tensor cores; see
// env_fp64_tc.cu for the method.
#pragma once
#include <cuda_runtime.h>
#include <cstdint>

#include "cx.cuh"
#include "kernels.cuh"

namespace mpsvqe {

// Scratch of one handle at bond cap chi: the site's shared operands and a batch of nodes.
struct EnvFp64 {
  char* scratch = nullptr;   // env_fp64_scratch(chi, batch) bytes, 256-byte aligned
  int* err = nullptr;        // device int: set by a tensor-core pipeline wait that ran out
  int* bal = nullptr;        // [sites][chi]: balance of each site's left bond (env_fp64_balance)
  int chi = 0, batch = 0;
};

int env_fp64_batch(int chi);        // nodes of a batch at most (128 bytes x chi^2 each, 512 MiB in all)
size_t env_fp64_scratch(int chi, int batch);

// Balance of all bonds of a slot from its right environments (largest bond: top), once per
// measurement.
cudaError_t env_fp64_balance(const EnvFp64& s, const DevMPS& m, int slot, int top, const Cx<double>* Renv, cudaStream_t st);
// Shared operands of site k (D = left bond, Dp = right bond), once per level chunk.
cudaError_t env_fp64_site(const EnvFp64& s, const Cx<double>* Bk, int k, int D, int Dp, cudaStream_t st);
// T_j[u] = L[u] B^j of U <= batch nodes (dense L) at site k, into the scratch. e0 / e1 (optional)
// are recorded on st right before and after the tensor-core GEMM.
cudaError_t env_fp64_T(const EnvFp64& s, const Cx<double>* L, int k, int U, int D, int Dp, cudaStream_t st,
                       cudaEvent_t e0 = nullptr, cudaEvent_t e1 = nullptr);
// L[child] = sum_ij P_ij (B^i)^+ T_j[parent] for nc children of the batch of U nodes that starts
// at trie node node_base, dense.
cudaError_t env_fp64_children(const EnvFp64& s, const int32_t* parent, const uint8_t* edge, int nc, int node_base, int U, int D,
                              int Dp, Cx<double>* Lout, cudaStream_t st, cudaEvent_t e0 = nullptr, cudaEvent_t e1 = nullptr);

}  // namespace mpsvqe
