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
#include <algorithm>
#include <cstdint>

#include "cx.cuh"
#include "env_tc.cuh"
#include "kernels.cuh"
#include "tc_gemm.cuh"

namespace mpsvqe {

static inline int pad32(int d) { return (d + 31) / 32 * 32; }

// The tensor core truncates its accumulator after each product of 8 inner indices: half a unit
// in the last place on average, 2^-24 / m of a sum with mantissa m, which two products a level
// over dozens of levels add up. With mantissas spread evenly over their logarithm that is the
// fraction 2/3 2^-24 = 4.0e-8 of the sum (least squares: E[m] / E[m^2]). In a 32-wide K tile a
// term loses it once for its own group of 8, measured 3.7e-8, and again for each later group
// of the tile, less where that group has few entries n in the shared operand's row (few terms
// leave few bits to cut): 1.2e-8 for n = 1, 1.9 for 2, 2.9 for 4, 3.3 for 8, which kLater (1 -
// 0.62^n) follows. A tile whose only entry is a power of two (sites that pass an index through)
// has exact products and loses nothing. The operand that all tiles share carries the
// inverse factor entry by entry. One factor of 9.0e-8 for every entry, right for dense rows, moved <P> by 1.5e-5 over 100
// sites that pass the bond through.
constexpr float kOwn = 3.7e-8f, kLater = 3.3e-8f;
// One row of a K tile by a warp, an entry a lane: hi and lo planes of z (1 + loss).
__device__ __forceinline__ void split_store(float z, float* hi, float* lo, bool store) {
  const unsigned nz = __ballot_sync(0xffffffffu, z != 0.f);
  float loss = kOwn;
#pragma unroll
  for (int g = 1; g < 4; ++g)
    if (g > (int)(threadIdx.x & 31) / 8) loss += kLater * (1.0f - exp2f(-0.69f * (float)__popc(nz >> (8 * g) & 255u)));
  const bool exact = __popc(nz) == 1 && (__float_as_uint(z) & 0x7fffffu) == 0;
  uint32_t b;
  asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(b) : "f"(z));
  const float h = __uint_as_float(b);
  asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(b) : "f"(fmaf(z, exact ? 0.f : loss, z - h)));
  if (store) {
    *hi = h;
    *lo = __uint_as_float(b);
  }
}

// BT (4D' x 2D, leading dimension 2 env_ld(D)) and A2 (2D' x 4 Dk, Dk = D rounded up to 32) from site k (B[b][j][c] at
// (b 2 + j) D' + c), hi and lo planes. One warp a row of a K tile, rows fastest: neighbouring
// warps share the sectors that they read.
__global__ void __launch_bounds__(256) k_tc_site_operands(const Cx<float>* Bk, int D, int Dp, int Dk, float* bt, float* bt_lo,
                                                          float* a2, float* a2_lo) {
  const int ldb = 2 * env_ld<float>(D), lane = threadIdx.x & 31;
  const int64_t nbt = (int64_t)4 * Dp * ((2 * D + 31) / 32), na2 = (int64_t)2 * Dp * (4 * Dk / 32);
  for (int64_t i = blockIdx.x * (int64_t)8 + (threadIdx.x >> 5); i < nbt + na2; i += (int64_t)gridDim.x * 8) {
    if (i < nbt) {
      const int64_t row = i % (4 * Dp);
      const int col = (int)(i / (4 * Dp)) * 32 + lane;
      const int c = (int)(row % Dp), ro = (int)(row / Dp) & 1, j = (int)(row / Dp) >> 1;
      const int b = col >> 1, ri = col & 1;
      const Cx<float> z = b < D ? Bk[((size_t)b * 2 + j) * Dp + c] : cx<float>(0.f, 0.f);   // B^j[b][c]
      // re row: (Br, -Bi) per b; im row: (Bi, Br) per b
      const int64_t o = row * ldb + col;
      split_store(ro == 0 ? (ri == 0 ? z.x : -z.y) : (ri == 0 ? z.y : z.x), bt + o, bt_lo + o, b < D);
    } else {
      const int64_t e = i - nbt, row = e % (2 * Dp);
      const int col = (int)(e / (2 * Dp)) * 32 + lane;
      const int ro = (int)(row & 1), cp = (int)(row >> 1);
      const int ii = col / (2 * Dk), ri = (col / Dk) & 1, a = col % Dk;
      const Cx<float> z = a < D ? Bk[((size_t)a * 2 + ii) * Dp + cp] : cx<float>(0.f, 0.f);   // B^i[a][c']
      // re row [Br, Bi] per i, im row [-Bi, Br] per i
      const int64_t o = row * 4 * Dk + col;
      split_store(ro == 0 ? (ri == 0 ? z.x : z.y) : (ri == 0 ? -z.y : z.x), a2 + o, a2_lo + o, true);
    }
  }
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
  const int64_t warps = (int64_t)4 * Dp * ((2 * D + 31) / 32) + (int64_t)2 * Dp * (4 * Dk / 32);
  const int grid = (int)std::min<int64_t>((warps + 7) / 8, 152 * 32);
  k_tc_site_operands<<<grid, 256, 0, st>>>(Bk, D, Dp, Dk, p.bt, p.bt_lo, p.a2, p.a2_lo);
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
