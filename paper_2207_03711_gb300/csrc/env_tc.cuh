// Environment contractions of the trie measurement on the tensor cores (mixed
// precision); see env_tc.cu for the GEMM formulation.
#pragma once
#include <cuda_runtime.h>
#include <cstdint>

#include "cx.cuh"

namespace mpsvqe {

// Scratch of one handle at bond cap chi: the shared operands of one site.
struct EnvTc {
  float* scratch = nullptr;   // env_tc_scratch_floats(chi) floats, 256-byte aligned
  int* err = nullptr;         // device int: set by a tensor-core pipeline wait that ran out
  int chi = 0;
};

size_t env_tc_scratch_floats(int chi);

// Shared operands of site k (D = left bond, Dp = right bond), once per level chunk.
cudaError_t env_tc_site(const EnvTc& s, const Cx<float>* Bk, int D, int Dp, cudaStream_t st);
// T_j[u] = L[u] B^j for the U nodes of a level chunk (L[u] at u env_node(D)), as T^T:
// 4 Dp rows (j, re/im, c) over columns (u, a), env_rows(D) floats per node.
// e0 / e1 (optional) are recorded on st right before and after the tensor-core GEMM.
cudaError_t env_tc_T(const EnvTc& s, const Cx<float>* L, float* Tt, int U, int D, int Dp, cudaStream_t st,
                     cudaEvent_t e0 = nullptr, cudaEvent_t e1 = nullptr);
// L[child] = sum_ij P_ij (B^i)^+ T_j[parent] for nc children (parent: trie node indices,
// node_base = the trie index of T^T's entry 0; edge: the letters P), child c at
// c env_node(D').
cudaError_t env_tc_children(const EnvTc& s, const float* Tt, const int32_t* parent, const uint8_t* edge, int nc,
                            int node_base, int U, int D, int Dp, Cx<float>* Lout, cudaStream_t st,
                            cudaEvent_t e0 = nullptr, cudaEvent_t e1 = nullptr);

}  // namespace mpsvqe
