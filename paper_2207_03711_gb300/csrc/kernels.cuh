// Device-side entry points of the MPS-VQE engine (launchers called by api.cu).
#pragma once
#include <cuda_runtime.h>
#include <cstdint>

#include "host.hpp"

namespace mpsvqe {

enum { MPS_PREC_FP64 = 0, MPS_PREC_MIXED = 1 };

// Per-slot status words written by the gate engine: [0] most bisection passes of one
// gate, [1] Jacobi fallbacks that hit their sweep cap, [2] largest rank reached,
// [3] Jacobi fallbacks taken, [4] gates skipped because M' held a NaN or Inf,
// [5] set when a caller-owned bond or rank array was out of range (raw-gate launches),
// [6..7] unused.
constexpr int kStatWords = 8;

// Device view of n_slots MPS states that share one layout.
struct DevMPS {
  int n;                    // sites
  int chi;                  // bond cap
  int n_slots;
  int64_t slot_elems;       // complex entries of B per slot
  const int64_t* site_off;  // [n] entry offset of site k inside a slot
  void* B;                  // complex<R> [n_slots][slot_elems], site k = (r_{k-1}, 2, r_k) row-major
  double* lam;              // [n_slots][n-1][chi]
  int* rank;                // [n_slots][n+1]; rank[0] = rank[n] = 1, rank[b+1] = rank of bond b
  void* work_M;             // complex<R> [n_slots][(2chi)^2]  gate workspace (unscaled M)
  void* work_X;             // complex<R> [n_slots][2chi (2chi+16)]  reflector vectors
  void* work_S;             // double [n_slots][16 chi^2]  SVD scratch (vectors; columns of M' that do not fit in smem)
  double* dw;               // [n_slots] accumulated discarded weight
  int* stat;                // [n_slots][kStatWords] status words (see kStatWords)
  unsigned long long* prof; // [n_slots][8] clock cycles per gate-engine phase (thread 0)
};

struct CircDev {
  const GateRec* gates;
  int64_t n_gates;
  const double* mats;  // 32 doubles per matrix (16 complex)
  int n_params;
  const int32_t* raw_bond = nullptr;  // raw-gate launches only: bond of gate g, matrix g of mats
  // Optional per-block arrays (index blockIdx.x, i.e. slot - slot0): the first gate the
  // block applies, and a shift added to the rotation angle phi of one parametric gate
  // (parameter-shift evaluations forked from a shared prefix).
  const int64_t* start_gate = nullptr;
  const int64_t* shift_gate = nullptr;
  const double* shift_phi = nullptr;
};

// Reset slots [slot0, slot0+count) to product states; occ: [count][n] bytes (0/1).
cudaError_t launch_reset(const DevMPS& m, int prec, int slot0, int count, const uint8_t* occ_dev,
                         cudaStream_t st);

// Apply gates [g0, g1) to slots [slot0, slot0+count); theta_dev: [count][n_params]. running:
// slots that share the device, these included (it decides the speed only).
cudaError_t launch_circuit(const DevMPS& m, int prec, const CircDev& c, int64_t g0, int64_t g1,
                           int slot0, int count, int running, const double* theta_dev, double cutoff,
                           int max_sweeps, cudaStream_t st);

// Measurement workspace (device) for one slot at a time.
struct MeasDev {
  void* R;          // complex<R> [n+1][chi*chi] right identity environments R_k
  void* Bhat;       // complex<R> like one slot of B: B_k^i R_{k+1}
  void* Q;          // complex<R> [n][4][chi env_ld(chi)]: Q_k^P = sum_ij conj(P_ij) Bhat_k^i (B_k^j)^+ per letter P
  double* vals;     // [n_terms][2] re, im of unnormalised <P>
  double* out;      // [4 + n_terms*2]: E, norm, ...
  double* part;     // [energy_sum_blocks][2]: (sum, correction) per block of the energy sum
  unsigned* done;   // blocks of the energy sum that have finished (zero between calls)
};


// Thread-local message returned by mps_last_error() (defined with the C ABI).
void set_error_message(const char* msg);

// ranks: the slot's n+1 bond ranks on the host (ranks[k] = left dimension of site k).
cudaError_t launch_right_envs(const DevMPS& m, int prec, int slot, const int* ranks, MeasDev& w, cudaStream_t st,
                              int* launches);
// Leading dimension of a D x D environment L: an FP32 row starts on a 16-byte boundary, so
// that the tensor-core route can read it in place; the entry an odd D leaves over is zero.
// The per-letter right blocks have the same layout.
template <class R>
__host__ __device__ constexpr int env_ld(int D) {
  return sizeof(R) == 4 ? D + (D & 1) : D;
}
// Entries from one node's L to the next. FP32 rounds the rows up to a multiple of 4, zeros
// below the D-th, so that the columns (node, row) of T^T start on 16-byte boundaries too.
__host__ __device__ constexpr int env_rows(int D) { return (D + 3) & ~3; }
template <class R>
__host__ __device__ constexpr int64_t env_node(int D) {
  return sizeof(R) == 4 ? (int64_t)env_rows(D) * env_ld<R>(D) : (int64_t)D * D;
}
// Chunked trie levels. Environment buffers: L holds node u's D_k x D_k block (row-major,
// leading dimension env_ld(D_k)) at u env_node(D_k) complex entries; T holds T_j[u] =
// L[u] B_k^j (D_k x D_{k+1}, dense) at (2u + j) D_k D_{k+1}. Node indices in cnode /
// parent are absolute trie indices; node_base is the trie index of buffer entry 0.
// cb: first child of each of the n_nodes nodes (nodes without children are left out).
cudaError_t launch_env_T(const DevMPS& m, int prec, int slot, int k, const void* L, void* T, int n_nodes,
                         const int32_t* cb, cudaStream_t st);
// A level whose bonds are both <= kFusedMax: T in shared memory, children [c_lo, c_hi) of
// parents [u_lo, u_hi) (trie indices; cb[u] = first child of node u) into Lout.
constexpr int kFusedMax = 64;
cudaError_t launch_level_fused(const DevMPS& m, int prec, int slot, int k, int D, int Dp, int u_lo, int u_hi,
                               int node_base, int c_lo, int c_hi, const int32_t* cb, const int32_t* parent,
                               const uint8_t* edge, const void* L, void* Lout, cudaStream_t st);
cudaError_t launch_env_close(const DevMPS& m, int prec, int slot, int k, const void* L, const void* Q,
                             const int32_t* cnode, const uint8_t* cletter, const int32_t* cterm, int n_closes,
                             int node_base, double* vals, cudaStream_t st);
cudaError_t launch_env_child(const DevMPS& m, int prec, int slot, int k, const void* T, const int32_t* parent,
                             const uint8_t* edge, int n_children, int node_base, void* Lout, cudaStream_t st);
// E = sum_t coeff_t Re(vals_t) / norm + id_coeff (compensated, fixed order); also writes
// normalised <P_t> to out[4 + 2t], out[0] = E, out[1] = norm.
int64_t energy_sum_blocks(int64_t n_terms);
cudaError_t launch_energy_sum(int prec, MeasDev& w, int64_t n_terms, const double* coeff_dev, double id_coeff,
                              int64_t id_term, cudaStream_t st);

}  // namespace mpsvqe
