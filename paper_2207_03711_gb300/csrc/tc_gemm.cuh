// Tensor-core (tcgen05) GEMM with compensated TF32 splits: the contraction primitive of
// the environment sweeps in mixed precision (see tc_gemm.cu).
#pragma once
#include <cuda_runtime.h>
#include <cstdint>

#include "cx.cuh"

namespace mpsvqe {
namespace tc {

// An FP32 operand, row-major with K contiguous and leading dimension ld (floats, a
// multiple of 4), 16-byte aligned.
struct Plane {
  const float* p;
  int64_t ld;
};

// Copy of an M x K row-major plane (leading dimension ld_in) into one of leading
// dimension ld_out; columns K..ld_out-1 become zero.
cudaError_t launch_pad_rows(const float* x, int64_t ld_in, int M, int K, float* out, int64_t ld_out,
                            cudaStream_t st);

// C (M x N, leading dimension ldc) = A (M x K) . B (N x K)^T on the tensor cores as
// A_hi B_hi + A_hi B_lo + A_lo B_hi (hi/lo TF32 splits made in shared memory) with
// round-to-nearest FP32 sums of per-K-tile accumulations. *err (device int) receives a
// non-zero code if a bounded pipeline wait ran out. Returns cudaErrorInvalidValue for
// misaligned planes.
cudaError_t launch_gemm_tf32x3(const Plane& A, const Plane& B, int M, int N, int K, float* C, int64_t ldc, int* err,
                               cudaStream_t st);

// The same with A given as hi plane A and lo plane a_lo (same leading dimension).
cudaError_t launch_gemm_presplit(const Plane& A, const float* a_lo, const Plane& B, int M, int N, int K, float* C,
                                 int64_t ldc, int* err, cudaStream_t st);

// Environments of nc trie children: L[child][c'][c] = sum over (i, a) of conj(B^i[a][c'])
// W_i[a][c], W_i = sum_j P_ij T_j[parent]. A, a_lo: planes of 2 Dp rows (c', re/im) over
// inner indices (i, re/im, a), a padded with zeros to a multiple of 32; Tt: T^T, rows
// (j, re/im, c) over columns (node, a) of U nodes at a stride of Dn >= D (a multiple of 4).
cudaError_t launch_gemm_children(const Plane& A, const float* a_lo, const Plane& Tt, int U, int D, int Dn, int Dp,
                                 const int32_t* parent, const uint8_t* edge, int node_base, int nc, Cx<float>* L,
                                 int* err, cudaStream_t st);

}  // namespace tc
}  // namespace mpsvqe
