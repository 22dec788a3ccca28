// Environment contractions of the trie measurement on the tensor cores (mixed precision).
//
// One trie level k (site k, left bond D = D_k, right bond D' = D_{k+1}) does two dense
// complex contractions (Eq. 11 generalised to Pauli strings, Sec. III-C):
//   T_j[u] = L[u] B^j                               (D x D)(D x D'),  j = 0, 1
//   L[child] = sum_ij P_ij (B^i)^+ T_j[u]          P = the edge letter of the child
// The second is formed per child, not per parent: with W_i = sum_j P_ij T_j[u] (for
// I: (T_0, T_1); X: (T_1, T_0); Y: (-i T_1, i T_0); Z: (T_0, -T_1)) it is one product
// sum_i (B^i)^+ W_i with the i sum stacked along K. In a Jordan-Wigner trie almost every
// parent has a single child (the next letter of a Z chain), and computing the four
// C_ij = (B^i)^+ T_j of every parent, as a per-parent form would, doubles that work.
// Over a chunk both become single real GEMMs with a shared operand built from the site
// tensor, which comes to the GEMM already split into TF32 hi and lo planes:
//   GEMM-T: BT (4D' x 2D) times the rows (u, a) of L[u] read as interleaved floats (re, im
//           per entry; the level buffer itself),
//           BT row (j, re, c) = [ Re B^j[b, c], -Im B^j[b, c] ]_b   (interleaved per b),
//           BT row (j, im, c) = [ Im B^j[b, c],  Re B^j[b, c] ]_b,
//           so that the product is T^T: rows (j, re/im, c) over columns (u, a).
//   GEMM-C: A2 (2D' rows (c', re/im)) times columns (child, c) over inner indices
//           (i, re/im, a): those of W_i are rows of T^T at the child's parent, up to a swap
//           of blocks and a sign that the letter gives, so the GEMM loads them from T^T
//           directly and applies the sign where it splits the tile,
//           A2 row (c', re) = [ Re B^0[:, c'],  Im B^0[:, c'],  Re B^1[:, c'],  Im B^1[:, c'] ],
//           A2 row (c', im) = [-Im B^0[:, c'],  Re B^0[:, c'], -Im B^1[:, c'],  Re B^1[:, c'] ],
//           each a range padded with zeros to a multiple of 32; the product goes to the
//           children's L as complex entries. Bonds up to 64 put two children into one
//           tile of 128 columns.
// No layout pass is left around the GEMMs: packing W and placing the children took 12 % of
// a 64-qubit chi = 256 measurement (11.5 + 7.6 of 148 ms, a 10-orbital Hamiltonian).
// Both run on tc_gemm.cu (tcgen05, compensated TF32 splits). L[u] has an even leading
// dimension (env_ld) and Dn rows, D rounded up to a multiple of 4, zeros in the ones added;
// so T^T has Dn columns per node (TMA rows and boxes start on 16-byte boundaries).
#include <cstdint>

#include "cx.cuh"
#include "env_tc.cuh"
#include "kernels.cuh"
#include "tc_gemm.cuh"

namespace mpsvqe {

static inline int pad32(int d) { return (d + 31) / 32 * 32; }

// The tensor core truncates its accumulator after each product. A truncation takes half a
// unit in the last place on average, 2^-23 / 2 / m of a value with mantissa m, so a K tile
// with its four products at full size loses (1 + 2 + 3 + 4) / 4 of that: a fixed fraction
// kLoss of the sum whatever its terms, which two products a level over dozens of levels
// add up. The operand that all tiles share carries the inverse factor.
constexpr float kLoss = 9.0e-8f;
__device__ __forceinline__ void split_store(float z, float* hi, float* lo) {
  uint32_t b;
  asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(b) : "f"(z));
  const float h = __uint_as_float(b);
  asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(b) : "f"(fmaf(z, kLoss, z - h)));
  *hi = h;
  *lo = __uint_as_float(b);
}

// BT (4D' x 2D, leading dimension 2 env_ld(D)) and A2 (2D' x 4 Dk, Dk = D rounded up to 32) from site k (B[b][j][c] at
// (b 2 + j) D' + c), hi and lo planes.
__global__ void k_tc_site_operands(const Cx<float>* Bk, int D, int Dp, int Dk, float* bt, float* bt_lo, float* a2,
                                   float* a2_lo) {
  const int ldb = 2 * env_ld<float>(D);
  const int64_t nbt = (int64_t)4 * Dp * ldb, na2 = (int64_t)2 * Dp * 4 * Dk;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < nbt + na2;
       i += (int64_t)gridDim.x * blockDim.x) {
    if (i < nbt) {
      const int64_t row = i / ldb;
      const int col = (int)(i - row * ldb);
      if (col >= 2 * D) continue;   // never loaded
      const int c = (int)(row % Dp), ro = (int)(row / Dp) & 1, j = (int)(row / Dp) >> 1;
      const int b = col >> 1, ri = col & 1;
      const Cx<float> z = Bk[((size_t)b * 2 + j) * Dp + c];   // B^j[b][c]
      // re row: (Br, -Bi) per b; im row: (Bi, Br) per b
      split_store(ro == 0 ? (ri == 0 ? z.x : -z.y) : (ri == 0 ? z.y : z.x), bt + i, bt_lo + i);
    } else {
      const int64_t e = i - nbt, row = e / (4 * Dk);
      const int col = (int)(e - row * 4 * Dk);
      const int ro = (int)(row & 1), cp = (int)(row >> 1);
      const int ii = col / (2 * Dk), ri = (col / Dk) & 1, a = col % Dk;
      const Cx<float> z = a < D ? Bk[((size_t)a * 2 + ii) * Dp + cp] : cx<float>(0.f, 0.f);   // B^i[a][c']
      // re row [Br, Bi] per i, im row [-Bi, Br] per i
      split_store(ro == 0 ? (ri == 0 ? z.x : z.y) : (ri == 0 ? -z.y : z.x), a2 + e, a2_lo + e);
    }
  }
}

static inline int grid_for(int64_t total) {
  const int64_t b = (total + 255) / 256;
  return (int)(b < 152 * 32 ? (b > 0 ? b : 1) : 152 * 32);
}

namespace {
struct Parts {
  float *bt, *bt_lo, *a2, *a2_lo;
};
int64_t part_bt(int chi) { return ((int64_t)8 * chi * env_ld<float>(chi) + 63) & ~(int64_t)63; }
int64_t part_a2(int chi) { return ((int64_t)8 * chi * pad32(chi) + 63) & ~(int64_t)63; }
Parts carve(float* base, int chi) {
  return {base, base + part_bt(chi), base + 2 * part_bt(chi), base + 2 * part_bt(chi) + part_a2(chi)};
}
}  // namespace

size_t env_tc_scratch_floats(int chi) { return (size_t)(2 * part_bt(chi) + 2 * part_a2(chi)); }

cudaError_t env_tc_site(const EnvTc& s, const Cx<float>* Bk, int D, int Dp, cudaStream_t st) {
  const Parts p = carve(s.scratch, s.chi);
  const int Dk = pad32(D);
  k_tc_site_operands<<<grid_for(8 * (int64_t)Dp * (D + Dk)), 256, 0, st>>>(Bk, D, Dp, Dk, p.bt, p.bt_lo, p.a2, p.a2_lo);
  return cudaGetLastError();
}

cudaError_t env_tc_T(const EnvTc& s, const Cx<float>* L, float* Tt, int U, int D, int Dp, cudaStream_t st,
                     cudaEvent_t e0, cudaEvent_t e1) {
  if (U <= 0) return cudaSuccess;
  const Parts p = carve(s.scratch, s.chi);
  const int Dn = env_rows(D);
  const int64_t ld = 2 * env_ld<float>(D);
  cudaError_t e;
  if (e0 && (e = cudaEventRecord(e0, st)) != cudaSuccess) return e;
  e = tc::launch_gemm_presplit(tc::Plane{p.bt, ld}, p.bt_lo, tc::Plane{(const float*)L, ld},
                               4 * Dp, U * Dn, 2 * D, Tt, (int64_t)U * Dn, s.err, st);
  if (e != cudaSuccess) return e;
  if (e1 && (e = cudaEventRecord(e1, st)) != cudaSuccess) return e;
  return cudaSuccess;
}

cudaError_t env_tc_children(const EnvTc& s, const float* Tt, const int32_t* parent, const uint8_t* edge, int nc,
                            int node_base, int U, int D, int Dp, Cx<float>* Lout, cudaStream_t st, cudaEvent_t e0,
                            cudaEvent_t e1) {
  if (nc <= 0) return cudaSuccess;
  const Parts p = carve(s.scratch, s.chi);
  const int Dn = env_rows(D);
  cudaError_t e;
  if (e0 && (e = cudaEventRecord(e0, st)) != cudaSuccess) return e;
  e = tc::launch_gemm_children(tc::Plane{p.a2, 4 * (int64_t)pad32(D)}, p.a2_lo, tc::Plane{Tt, (int64_t)U * Dn}, U, D,
                               Dn, Dp, parent, edge, node_base, nc, Lout, s.err, st);
  if (e != cudaSuccess) return e;
  if (e1 && (e = cudaEventRecord(e1, st)) != cudaSuccess) return e;
  return cudaSuccess;
}

}  // namespace mpsvqe
