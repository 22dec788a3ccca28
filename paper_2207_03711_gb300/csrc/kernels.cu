// CUDA kernels of the MPS-VQE hot path for sm_103a (GB300).
//
//  k_reset        product-state reference (Sec. III-D: X gates on the occupied qubits).
//  k_renv_chain, k_renv_step   right identity environments R_k and B^_k = B_k R_{k+1}.
//  k_letter_blocks   per-letter right blocks, from which closing strings are evaluated.
//  k_level_fused, k_level_T/child   one level of the Pauli-string prefix trie (Eq. 11
//                 generalised) on the CUDA cores; env_tc.cu and env_fp64_tc.cu: larger bonds.
//  k_level_close  the strings that end at a level.
//  k_energy_sum   E = sum_i a_i <P_i> (Eq. 2) with Neumaier compensation in FP64.
#include <cfloat>
#include <cmath>
#include <cstdint>

#include <algorithm>
#include <type_traits>

#include "cx.cuh"
#include "gemm.cuh"
#include "kernels.cuh"
#include "smem_limit.cuh"

namespace mpsvqe {

// ------------------------------------------------------------------------- reset
template <class R>
__global__ void k_reset(DevMPS m, int slot0, const uint8_t* occ) {
  const int s = slot0 + blockIdx.x;
  Cx<R>* B = (Cx<R>*)m.B + (size_t)s * m.slot_elems;
  int* rank = m.rank + (size_t)s * (m.n + 1);
  double* lam = m.lam + (size_t)s * (m.n - 1) * m.chi;
  for (int k = threadIdx.x; k < m.n; k += blockDim.x) {
    const uint8_t o = occ[(size_t)blockIdx.x * m.n + k];
    Cx<R>* b = B + m.site_off[k];
    b[0] = cx<R>(o ? R(0) : R(1), R(0));
    b[1] = cx<R>(o ? R(1) : R(0), R(0));
  }
  for (int b = threadIdx.x; b <= m.n; b += blockDim.x) rank[b] = 1;
  for (int b = threadIdx.x; b < m.n - 1; b += blockDim.x) lam[(size_t)b * m.chi] = 1.0;
  if (threadIdx.x == 0) m.dw[s] = 0.0;
  if (threadIdx.x < kStatWords) m.stat[s * kStatWords + threadIdx.x] = (threadIdx.x == 2) ? 1 : 0;
}

cudaError_t launch_reset(const DevMPS& m, int prec, int slot0, int count, const uint8_t* occ,
                         cudaStream_t st) {
  if (prec == MPS_PREC_FP64)
    k_reset<double><<<count, 128, 0, st>>>(m, slot0, occ);
  else
    k_reset<float><<<count, 128, 0, st>>>(m, slot0, occ);
  return cudaGetLastError();
}

// ------------------------------------------------------------ small tiled GEMM
// C (Mdim x Ndim, ldc) = sum_t s_t opA_t(A_t) B_t with 256 threads and 64x64 tiles. opA: A
// stored Mdim x K (lda), or K x Mdim used as A^H (conjT). B stored K x Ndim (ldb).
template <class R>
struct GemmTerm {
  const Cx<R>* A;
  int lda;
  bool conjT;
  const Cx<R>* B;
  int ldb;
  Cx<R> s;
};

// One 64 x 64 output tile at (m0, n0).
template <class R>
__device__ void gemm_tile(int m0, int n0, int Mdim, int Ndim, int K, const GemmTerm<R>* terms, int nterm, Cx<R>* C,
                          int ldc, Cx<R> (*As)[17], Cx<R> (*Bs)[65]) {
  constexpr int NTH = 256, TY = NTH / 16, RPT = 64 / TY;
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  Cx<R> acc[RPT][4];
#pragma unroll
  for (int i = 0; i < RPT; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = cx<R>(0, 0);
  for (int t = 0; t < nterm; ++t) {
    const GemmTerm<R> T = terms[t];
    for (int k0 = 0; k0 < K; k0 += 16) {
      for (int e = threadIdx.x; e < 64 * 16; e += NTH) {
        const int r = e >> 4, cc = e & 15;
        const int gm = m0 + r, gk = k0 + cc;
        Cx<R> v = cx<R>(0, 0);
        if (gm < Mdim && gk < K) v = T.conjT ? conj(T.A[(size_t)gk * T.lda + gm]) : T.A[(size_t)gm * T.lda + gk];
        As[r][cc] = T.s * v;
      }
      for (int e = threadIdx.x; e < 16 * 64; e += NTH) {
        const int r = e >> 6, cc = e & 63;
        const int gk = k0 + r, gn = n0 + cc;
        Bs[r][cc] = gk < K && gn < Ndim ? T.B[(size_t)gk * T.ldb + gn] : cx<R>(0, 0);
      }
      __syncthreads();
#pragma unroll 4
      for (int kk = 0; kk < 16; ++kk) {
        Cx<R> a[RPT], b[4];
#pragma unroll
        for (int i = 0; i < RPT; ++i) a[i] = As[ty + TY * i][kk];
#pragma unroll
        for (int j = 0; j < 4; ++j) b[j] = Bs[kk][tx + 16 * j];
#pragma unroll
        for (int i = 0; i < RPT; ++i)
#pragma unroll
          for (int j = 0; j < 4; ++j) cmac(acc[i][j], a[i], b[j]);
      }
      __syncthreads();
    }
  }
#pragma unroll
  for (int i = 0; i < RPT; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int gm = m0 + ty + TY * i, gn = n0 + tx + 16 * j;
      if (gm < Mdim && gn < Ndim) C[(size_t)gm * ldc + gn] = acc[i][j];
    }
}

template <class R>
__device__ void block_gemm(int Mdim, int Ndim, int K, const GemmTerm<R>* terms, int nterm, Cx<R>* C, int ldc,
                           Cx<R> (*As)[17], Cx<R> (*Bs)[65]) {
  for (int m0 = 0; m0 < Mdim; m0 += 64)
    for (int n0 = 0; n0 < Ndim; n0 += 64) gemm_tile<R>(m0, n0, Mdim, Ndim, K, terms, nterm, C, ldc, As, Bs);
}

// --------------------------------------------------------- right environments
// R_n = [1]; Bhat_k^i = B_k^i R_{k+1} (same layout as B_k); R_k = sum_i Bhat_k^i (B_k^i)^+.
// A site is a chain of two products, both plain GEMMs on the stored layout: Bhat = (2 Dl x
// Dr) R and R_k = Bhat B^+ over (i, c) as one inner index. The per-letter blocks
//   Q_k^P = sum_ij conj(P_ij) Bhat_k^i (B_k^j)^+,  P = X, Y, Z
// (a string closing at site k with letter P has <P> = sum_ab L[a][b] conj(Q_k^P[a][b]),
// Eq. 11 with the right part contracted; no string closes with I) hang off the chain and
// run for all sites in one launch afterwards, from three sums over the four pairs of
// operand entries: G01 and G10 give X and Y, the difference of G00 and G11 gives Z.
template <class R, int NT>
__device__ __forceinline__ void renv_bhat(const Cx<R>* Bk, const Cx<R>* Rn, Cx<R>* Bh, int Dl, int Dr, int tile, int ntiles,
                                          unsigned char* smem) {
  // rows are dealt to blocks in slabs
  const int M = 2 * Dl, per = (M + ntiles - 1) / ntiles, m0 = min(M, per * tile), mn = min(per, M - m0);
  gate::tile_gemm<R, NT, false>(
      mn, Dr, Dr, [&](int i, int k) { return Bk[(size_t)(m0 + i) * Dr + k]; },
      [&](int k, int j) { return Rn ? gate::ldcg(Rn + (size_t)k * Dr + j) : cx<R>(R(1), R(0)); },   // R_n = [1]
      [&](int i, int j, Cx<R> v) { Bh[(size_t)(m0 + i) * Dr + j] = v; }, smem);
}
template <class R, int NT>
__device__ __forceinline__ void renv_close(const Cx<R>* Bk, const Cx<R>* Bh, Cx<R>* Rk, int Dl, int Dr, int tile, int ntiles,
                                           unsigned char* smem) {
  const int per = (Dl + ntiles - 1) / ntiles, m0 = min(Dl, per * tile), mn = min(per, Dl - m0);
  gate::tile_gemm<R, NT, true>(
      mn, Dl, 2 * Dr, [&](int i, int k) { return gate::ldcg(Bh + (size_t)(m0 + i) * 2 * Dr + k); },
      [&](int k, int j) { return conj(Bk[(size_t)j * 2 * Dr + k]); },
      [&](int i, int j, Cx<R> v) { Rk[(size_t)(m0 + i) * Dl + j] = v; }, smem);
}

// The whole chain by one cluster of C blocks (small bonds: a launch per product would cost
// more than the product).
template <class R, int C>
__global__ void __launch_bounds__(256) k_renv_chain(DevMPS m, int slot, Cx<R>* Renv, Cx<R>* Bhat) {
  extern __shared__ __align__(256) unsigned char smem[];
  const int* rank = m.rank + (size_t)slot * (m.n + 1);
  const Cx<R>* Bslot = (const Cx<R>*)m.B + (size_t)slot * m.slot_elems;
  const size_t chi2 = (size_t)m.chi * m.chi;
  const int c = (int)gate::crank<C>();
  for (int k = m.n - 1; k >= 0; --k) {
    const int Dl = rank[k], Dr = rank[k + 1];
    const Cx<R>* Bk = Bslot + m.site_off[k];
    Cx<R>* Bh = Bhat + m.site_off[k];
    renv_bhat<R, 256>(Bk, k == m.n - 1 ? nullptr : Renv + (size_t)(k + 1) * chi2, Bh, Dl, Dr, c, C, smem);
    gate::csync<C>();
    renv_close<R, 256>(Bk, Bh, Renv + (size_t)k * chi2, Dl, Dr, c, C, smem);
    gate::csync<C>();
  }
}
// One product of one site over a grid (large bonds): tiles of 16 rows and kRenvCols columns, the
// shortest time for a product of a serial chain. FP64 is bound by the FP64 lanes of the few
// SMs that have a tile, so its tiles are as small as the threads of a block allow (18 sites,
// chi = 64: 1.79 ms with 64 columns).
template <class R>
constexpr int kRenvCols = sizeof(R) == 4 ? 64 : 16;
template <class R>
__global__ void __launch_bounds__(256) k_renv_step(DevMPS m, int slot, int k, int stage, Cx<R>* Renv, Cx<R>* Bhat) {
  extern __shared__ __align__(256) unsigned char smem[];
  const int* rank = m.rank + (size_t)slot * (m.n + 1);
  const size_t chi2 = (size_t)m.chi * m.chi;
  const int Dl = rank[k], Dr = rank[k + 1];
  const Cx<R>* Bk = (const Cx<R>*)m.B + (size_t)slot * m.slot_elems + m.site_off[k];
  Cx<R>* Bh = Bhat + m.site_off[k];
  const int N = stage == 0 ? Dr : Dl, n0 = blockIdx.y * kRenvCols<R>, nn = min(kRenvCols<R>, N - n0);
  if (nn <= 0) return;
  const int M = stage == 0 ? 2 * Dl : Dl, per = (M + gridDim.x - 1) / gridDim.x, m0 = min(M, per * (int)blockIdx.x),
            mn = min(per, M - m0);
  const Cx<R>* Rn = k == m.n - 1 ? nullptr : Renv + (size_t)(k + 1) * chi2;
  Cx<R>* Rk = Renv + (size_t)k * chi2;
  if (stage == 0)
    gate::tile_gemm<R, 256, false>(
        mn, nn, Dr, [&](int i, int q) { return Bk[(size_t)(m0 + i) * Dr + q]; },
        [&](int q, int j) { return Rn ? gate::ldcg(Rn + (size_t)q * Dr + n0 + j) : cx<R>(R(1), R(0)); },
        [&](int i, int j, Cx<R> v) { Bh[(size_t)(m0 + i) * Dr + n0 + j] = v; }, smem);
  else
    gate::tile_gemm<R, 256, true>(
        mn, nn, 2 * Dr, [&](int i, int q) { return gate::ldcg(Bh + (size_t)(m0 + i) * 2 * Dr + q); },
        [&](int q, int j) { return conj(Bk[(size_t)(n0 + j) * 2 * Dr + q]); },
        [&](int i, int j, Cx<R> v) { Rk[(size_t)(m0 + i) * Dl + n0 + j] = v; }, smem);
}

// Q_k^X, Q_k^Y, Q_k^Z of all sites: output tiles of 16 TI x 16 TI, TI^2 outputs per thread
// and sum, 16-deep tiles of the four operands. Grid (tiles, sites). TI = 2 in FP32; 1 in
// FP64, whose tiles are worth more blocks.
template <class R, int TI>
__global__ void __launch_bounds__(256) k_letter_blocks(DevMPS m, int slot, const Cx<R>* Bhat, Cx<R>* Q) {
  __shared__ Cx<R> A[2][16 * TI][17];
  __shared__ Cx<R> B[2][16 * TI][17];
  const int k = blockIdx.y;
  const int* rank = m.rank + (size_t)slot * (m.n + 1);
  const int Dl = rank[k], Dr = rank[k + 1], TS = 16 * TI, nt = (Dl + TS - 1) / TS;
  if ((int)blockIdx.x >= nt * nt) return;
  const int m0 = blockIdx.x / nt * TS, n0 = blockIdx.x % nt * TS;
  const Cx<R>* Bk = (const Cx<R>*)m.B + (size_t)slot * m.slot_elems + m.site_off[k];
  const Cx<R>* Bh = Bhat + m.site_off[k];
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  Cx<R> g01[TI][TI], g10[TI][TI], gz[TI][TI];
#pragma unroll
  for (int i = 0; i < TI; ++i)
#pragma unroll
    for (int j = 0; j < TI; ++j) g01[i][j] = g10[i][j] = gz[i][j] = cx<R>(0, 0);
  for (int k0 = 0; k0 < Dr; k0 += 16) {
    __syncthreads();
    for (int e = tid; e < 2 * TS * 16; e += 256) {
      const int q = e & 15, r = (e >> 4) % TS, s = (e >> 4) / TS, c = k0 + q;
      A[s][r][q] = (m0 + r < Dl && c < Dr) ? Bh[((size_t)(m0 + r) * 2 + s) * Dr + c] : cx<R>(0, 0);
      B[s][r][q] = (n0 + r < Dl && c < Dr) ? Bk[((size_t)(n0 + r) * 2 + s) * Dr + c] : cx<R>(0, 0);
    }
    __syncthreads();
#pragma unroll 4
    for (int q = 0; q < 16; ++q) {
      Cx<R> a0[TI], a1[TI], b0[TI], b1[TI];
#pragma unroll
      for (int i = 0; i < TI; ++i) {
        a0[i] = A[0][ty + 16 * i][q];
        a1[i] = A[1][ty + 16 * i][q];
        b0[i] = B[0][tx + 16 * i][q];
        b1[i] = B[1][tx + 16 * i][q];
      }
#pragma unroll
      for (int i = 0; i < TI; ++i)
#pragma unroll
        for (int j = 0; j < TI; ++j) {
          cmac_bconj(g01[i][j], a0[i], b1[j]);
          cmac_bconj(g10[i][j], a1[i], b0[j]);
          cmac_bconj(gz[i][j], a0[i], b0[j]);
          cmac_bconj(gz[i][j], cx<R>(-a1[i].x, -a1[i].y), b1[j]);
        }
    }
  }
  const int ld = env_ld<R>(Dl);
  const size_t chi2 = (size_t)m.chi * env_ld<R>(m.chi);
  Cx<R>* q = Q + (size_t)k * 4 * chi2;
#pragma unroll
  for (int i = 0; i < TI; ++i)
#pragma unroll
    for (int j = 0; j < TI; ++j) {
      const int r = m0 + ty + 16 * i, c = n0 + tx + 16 * j;
      if (r < Dl && c < Dl) {
        const size_t o = (size_t)r * ld + c;
        if (c == Dl - 1 && ld > Dl) q[chi2 + o + 1] = q[2 * chi2 + o + 1] = q[3 * chi2 + o + 1] = cx<R>(0, 0);
        const Cx<R> d = g01[i][j] - g10[i][j];
        q[chi2 + o] = g01[i][j] + g10[i][j];
        q[2 * chi2 + o] = cx<R>(-d.y, d.x);   // i G01 - i G10
        q[3 * chi2 + o] = gz[i][j];
      }
    }
}

// Bonds up to this run the chain in one cluster launch. FP64 products of larger bonds are
// worth more SMs than a cluster has.
template <class R>
constexpr int kChainMax = sizeof(R) == 4 ? 64 : 32;

template <class R>
static cudaError_t right_envs_t(const DevMPS& m, int slot, const int* ranks, Cx<R>* Renv, Cx<R>* Bhat, Cx<R>* Q,
                                cudaStream_t st, int* launches) {
  const size_t smem = gate::gemm_tile_bytes<256>();
  int top = 1;
  for (int k = 0; k <= m.n; ++k) top = std::max(top, ranks[k]);
  if (top <= kChainMax<R>) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(8);
    cfg.blockDim = dim3(256);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = 8;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    cudaError_t e = cudaLaunchKernelEx(&cfg, k_renv_chain<R, 8>, m, slot, Renv, Bhat);
    if (e != cudaSuccess) return e;
    *launches += 1;
  } else {
    for (int k = m.n - 1; k >= 0; --k) {
      const int Dl = ranks[k], Dr = ranks[k + 1];
      constexpr int cw = kRenvCols<R>;
      k_renv_step<R><<<dim3((2 * Dl + 15) / 16, (Dr + cw - 1) / cw), 256, smem, st>>>(m, slot, k, 0, Renv, Bhat);
      k_renv_step<R><<<dim3((Dl + 15) / 16, (Dl + cw - 1) / cw), 256, smem, st>>>(m, slot, k, 1, Renv, Bhat);
    }
    *launches += 2 * m.n;
  }
  constexpr int TI = sizeof(R) == 4 ? 2 : 1;
  const int nt = (top + 16 * TI - 1) / (16 * TI);
  k_letter_blocks<R, TI><<<dim3(nt * nt, m.n), 256, 0, st>>>(m, slot, Bhat, Q);
  *launches += 1;
  return cudaGetLastError();
}

cudaError_t launch_right_envs(const DevMPS& m, int prec, int slot, const int* ranks, MeasDev& w, cudaStream_t st,
                              int* launches) {
  if (prec == MPS_PREC_FP64)
    return right_envs_t<double>(m, slot, ranks, (Cx<double>*)w.R, (Cx<double>*)w.Bhat, (Cx<double>*)w.Q, st, launches);
  return right_envs_t<float>(m, slot, ranks, (Cx<float>*)w.R, (Cx<float>*)w.Bhat, (Cx<float>*)w.Q, st, launches);
}

// ------------------------------------------------------------------ trie level
// Pauli letter -> the two (i, j, sigma_ij) entries of its 2x2 matrix.
template <class R>
__device__ __forceinline__ void letter_entries(uint8_t l, int* ii, int* jj, Cx<R>* s) {
  switch (l) {
    case 0: ii[0] = 0; jj[0] = 0; s[0] = cx<R>(1, 0); ii[1] = 1; jj[1] = 1; s[1] = cx<R>(1, 0); break;
    case 1: ii[0] = 0; jj[0] = 1; s[0] = cx<R>(1, 0); ii[1] = 1; jj[1] = 0; s[1] = cx<R>(1, 0); break;
    case 2: ii[0] = 0; jj[0] = 1; s[0] = cx<R>(0, -1); ii[1] = 1; jj[1] = 0; s[1] = cx<R>(0, 1); break;
    default: ii[0] = 0; jj[0] = 0; s[0] = cx<R>(1, 0); ii[1] = 1; jj[1] = 1; s[1] = cx<R>(-1, 0); break;
  }
}

// T_j[u] = L_k[u] B_k^j  (Dk x Dk)(Dk x Dk1), grid (nodes, 2)
template <class R>
__global__ void __launch_bounds__(256) k_level_T(DevMPS m, int slot, int k, const Cx<R>* Lin, Cx<R>* T,
                                                 const int32_t* cb) {
  __shared__ Cx<R> As[64][17];
  __shared__ Cx<R> Bs[16][65];
  const int u = blockIdx.x, j = blockIdx.y;
  if (cb[u] == cb[u + 1]) return;
  const int* rank = m.rank + (size_t)slot * (m.n + 1);
  const int Dk = rank[k], Dk1 = rank[k + 1];
  const Cx<R>* Bk = (const Cx<R>*)m.B + (size_t)slot * m.slot_elems + m.site_off[k];
  const int ld = env_ld<R>(Dk);
  GemmTerm<R> t{Lin + u * env_node<R>(Dk), ld, false, Bk + j * Dk1, 2 * Dk1, cx<R>(1, 0)};
  block_gemm<R>(Dk, Dk1, Dk, &t, 1, T + ((size_t)u * 2 + j) * Dk * Dk1, Dk1, As, Bs);
}

// L_{k+1}[c] = sum_ij sigma_ij (B_k^i)^+ T_j[parent(c)]
template <class R>
__global__ void __launch_bounds__(256) k_level_child(DevMPS m, int slot, int k, const int32_t* parent,
                                                     const uint8_t* edge, const Cx<R>* T, Cx<R>* Lout,
                                                     int node_base) {
  __shared__ Cx<R> As[64][17];
  __shared__ Cx<R> Bs[16][65];
  const int c = blockIdx.x;
  const int* rank = m.rank + (size_t)slot * (m.n + 1);
  const int Dk = rank[k], Dk1 = rank[k + 1];
  const Cx<R>* Bk = (const Cx<R>*)m.B + (size_t)slot * m.slot_elems + m.site_off[k];
  const int u = parent[c] - node_base;
  int ii[2], jj[2];
  Cx<R> sg[2];
  letter_entries<R>(edge[c], ii, jj, sg);
  GemmTerm<R> t[2];
  for (int e = 0; e < 2; ++e)
    t[e] = GemmTerm<R>{Bk + ii[e] * Dk1, 2 * Dk1, true, T + ((size_t)u * 2 + jj[e]) * Dk * Dk1, Dk1, sg[e]};
  const int ld = env_ld<R>(Dk1);
  Cx<R>* out = Lout + c * env_node<R>(Dk1);
  block_gemm<R>(Dk1, Dk1, Dk, t, 2, out, ld, As, Bs);
  for (int64_t e = threadIdx.x + (int64_t)Dk1 * ld; e < env_node<R>(Dk1); e += 256) out[e] = cx<R>(0, 0);
  if (ld > Dk1)
    for (int r = threadIdx.x; r < Dk1; r += 256) out[(size_t)r * ld + Dk1] = cx<R>(0, 0);
}

// Fused level for bonds up to 64: both T_j of a group of parents stay in shared memory and
// the group's children are formed from them at once, so T never travels through memory,
// nodes without children cost nothing but their rows, and small bonds share a block (64
// rows of L and 64 columns of children at a time, whatever D and D').
// Bound by the FP32 (FP64) lanes; what it saves is T's way through memory, the padding of
// small bonds to 64 x 64 tiles and a launch. Against a launch for T and one for the children:
// 24 qubits, chi = 64, mixed 13.5 -> 8.8 ms (all levels by this kernel), 18 qubits, chi = 64,
// FP64 93 -> 62 ms, 8 qubits, FP64 5.2 -> 0.34 ms (with the right environments in one launch).
// cb: first child of each node of the level (trie indices); children outside [c_lo, c_hi)
// are left to another launch; child c is written to Lout[c - c_lo].
struct LevelArgs {
  int slot, k;
  int u_lo, u_hi;           // parents (trie indices)
  int node_base;            // trie index of Lin's entry 0
  int c_lo, c_hi;
  const int32_t* cb;
  const int32_t* parent;
  const uint8_t* edge;
};

// FP32: site tensor, L rows and T in shared memory; 4 x JT outputs per thread for T, RM x 4
// for the children, DP: right bond rounded up to a power of two.
template <int DP>
__global__ void __launch_bounds__(256) k_level_fused(DevMPS m, LevelArgs g, const Cx<float>* Lin, Cx<float>* Lout) {
  extern __shared__ __align__(256) unsigned char smem[];
  constexpr int JT = DP >= 16 ? DP / 8 : 1, RM = DP >= 16 ? DP / 16 : 1;
  const int* rank = m.rank + (size_t)g.slot * (m.n + 1);
  const int D = rank[g.k], Dp = rank[g.k + 1], W = 2 * Dp;
  const int P = max(1, 64 / D), u0 = g.u_lo + blockIdx.x * P, u1 = min(u0 + P, g.u_hi);
  const int c0 = max(g.cb[u0], g.c_lo), c1 = min(g.cb[u1], g.c_hi);
  if (c0 >= c1) return;
  Cx<float>* Bs = (Cx<float>*)smem;             // [D][2 D'], as stored
  Cx<float>* Ls = Bs + D * W;                   // [rows][D + 1]
  Cx<float>* Ts = Ls + 64 * (D + 1);            // [rows][2 D']
  const Cx<float>* Bk = (const Cx<float>*)m.B + (size_t)g.slot * m.slot_elems + m.site_off[g.k];
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const int rows = (u1 - u0) * D, ld = env_ld<float>(D), ldp = env_ld<float>(Dp);
  const int64_t node = env_node<float>(D);
  const Cx<float>* Lu = Lin + (u0 - g.node_base) * node;
  for (int e = tid; e < D * W; e += 256) Bs[e] = Bk[e];
  for (int e = tid; e < rows * D; e += 256) {
    const int r = e / D, c = e - r * D;
    Ls[r * (D + 1) + c] = Lu[r / D * node + r % D * ld + c];
  }
  __syncthreads();
  {
    Cx<float> acc[4][JT];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < JT; ++j) acc[i][j] = cx<float>(0.f, 0.f);
    int ro[4], co[JT];
#pragma unroll
    for (int i = 0; i < 4; ++i) ro[i] = min(ty + 16 * i, rows - 1) * (D + 1);
#pragma unroll
    for (int j = 0; j < JT; ++j) co[j] = min(tx + 16 * j, W - 1);
#pragma unroll 2
    for (int q = 0; q < D; ++q) {
      Cx<float> a[4], b[JT];
#pragma unroll
      for (int i = 0; i < 4; ++i) a[i] = Ls[ro[i] + q];
#pragma unroll
      for (int j = 0; j < JT; ++j) b[j] = Bs[q * W + co[j]];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < JT; ++j) cmac(acc[i][j], a[i], b[j]);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < JT; ++j)
        if (ty + 16 * i < rows && tx + 16 * j < W) Ts[(ty + 16 * i) * W + tx + 16 * j] = acc[i][j];
  }
  __syncthreads();
  // children: columns (child, c) in turn, 64 at a time; out = s0 (B^0)^+ T_{j0} + s1 (B^1)^+ T_{j1}
  const int ncol = (c1 - c0) * Dp;
  for (int n0 = 0; n0 < ncol; n0 += 64) {
    Cx<float> acc[RM][4];
    int off[4], j0[4], ch[4], cc[4];
    uint8_t let[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int nn = min(n0 + tx + 16 * j, ncol - 1);
      ch[j] = nn / Dp;
      cc[j] = nn - ch[j] * Dp;
      let[j] = g.edge[c0 + ch[j]];
      off[j] = (g.parent[c0 + ch[j]] - u0) * D * W + cc[j];
      j0[j] = (let[j] == 1 || let[j] == 2) ? Dp : 0;   // X, Y swap the T_j
#pragma unroll
      for (int i = 0; i < RM; ++i) acc[i][j] = cx<float>(0.f, 0.f);
    }
    int bo[RM];
#pragma unroll
    for (int i = 0; i < RM; ++i) bo[i] = min(ty + 16 * i, Dp - 1);
#pragma unroll
    for (int half = 0; half < 2; ++half) {
#pragma unroll 2
      for (int q = 0; q < D; ++q) {
        Cx<float> a[RM], b[4];
#pragma unroll
        for (int i = 0; i < RM; ++i) a[i] = Bs[q * W + half * Dp + bo[i]];
#pragma unroll
        for (int j = 0; j < 4; ++j) b[j] = Ts[off[j] + (half ? Dp - j0[j] : j0[j]) + q * W];
#pragma unroll
        for (int i = 0; i < RM; ++i)
#pragma unroll
          for (int j = 0; j < 4; ++j) cmac_conj(acc[i][j], a[i], b[j]);
      }
      if (half == 0) {
        // s0 / s1 = 1 for I and X, -1 for Y (-i, i) and Z (1, -1)
#pragma unroll
        for (int j = 0; j < 4; ++j)
          if (let[j] >= 2) {
#pragma unroll
            for (int i = 0; i < RM; ++i) acc[i][j] = cx<float>(-acc[i][j].x, -acc[i][j].y);
          }
      }
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      if (n0 + tx + 16 * j >= ncol) continue;
      Cx<float>* o = Lout + (c0 + ch[j] - g.c_lo) * env_node<float>(Dp) + cc[j];
#pragma unroll
      for (int i = 0; i < RM; ++i) {
        const int r = ty + 16 * i;
        if (r >= env_rows(Dp)) continue;
        Cx<float> v = acc[i][j];
        if (let[j] == 2) v = cx<float>(-v.y, v.x);       // s1 = i
        if (let[j] == 3) v = cx<float>(-v.x, -v.y);      // s1 = -1
        if (r >= Dp) v = cx<float>(0.f, 0.f);
        o[(size_t)r * ldp] = v;
        if (ldp > Dp && cc[j] == Dp - 1) o[(size_t)r * ldp + 1] = cx<float>(0.f, 0.f);
      }
    }
  }
}

// FP64: what a block does is bound by the FP64 pipe (two lanes a clock), so the operands
// come through the tiled GEMM's staging; only T stays in shared memory.
__global__ void __launch_bounds__(256) k_level_fused64(DevMPS m, LevelArgs g, const Cx<double>* Lin, Cx<double>* Lout) {
  extern __shared__ __align__(256) unsigned char smem[];
  const int* rank = m.rank + (size_t)g.slot * (m.n + 1);
  const int D = rank[g.k], Dp = rank[g.k + 1], W = 2 * Dp;
  const int P = max(1, 16 / D), u0 = g.u_lo + blockIdx.x * P, u1 = min(u0 + P, g.u_hi);
  const int c0 = max(g.cb[u0], g.c_lo), c1 = min(g.cb[u1], g.c_hi);
  if (c0 >= c1) return;
  Cx<double>* Ts = (Cx<double>*)(smem + gate::gemm_tile_bytes<256>());   // [rows][2 D']
  const Cx<double>* Bk = (const Cx<double>*)m.B + (size_t)g.slot * m.slot_elems + m.site_off[g.k];
  const Cx<double>* Lu = Lin + (size_t)(u0 - g.node_base) * D * D;
  const int rows = (u1 - u0) * D;
  gate::tile_gemm<double, 256, false>(
      rows, W, D, [&](int i, int q) { return Lu[i * D + q]; }, [&](int q, int j) { return Bk[q * W + j]; },
      [&](int i, int j, Cx<double> v) { Ts[i * W + j] = v; }, smem);
  const int32_t* par = g.parent + c0;
  const uint8_t* ed = g.edge + c0;
  gate::tile_gemm<double, 256, false>(
      Dp, (c1 - c0) * Dp, 2 * D,
      [&](int i, int q) {
        const int h = q >= D;
        return conj(Bk[(q - h * D) * W + h * Dp + i]);
      },
      [&](int q, int n) {
        const int h = q >= D, ch = n / Dp, let = ed[ch];
        const int jj = (let == 1 || let == 2) ? 1 - h : h;
        const Cx<double> t = Ts[((par[ch] - u0) * D + q - h * D) * W + jj * Dp + n - ch * Dp];
        if (let == 2) return h ? cx<double>(-t.y, t.x) : cx<double>(t.y, -t.x);   // i T_0, -i T_1
        return let == 3 && h ? cx<double>(-t.x, -t.y) : t;
      },
      [&](int i, int n, Cx<double> v) {
        const int ch = n / Dp;
        Lout[((size_t)(c0 + ch - g.c_lo) * Dp + i) * Dp + n - ch * Dp] = v;
      },
      smem);
}

cudaError_t launch_level_fused(const DevMPS& m, int prec, int slot, int k, int D, int Dp, int u_lo, int u_hi,
                               int node_base, int c_lo, int c_hi, const int32_t* cb, const int32_t* parent,
                               const uint8_t* edge, const void* L, void* Lout, cudaStream_t st) {
  if (c_lo >= c_hi) return cudaSuccess;
  const LevelArgs g{slot, k, u_lo, u_hi, node_base, c_lo, c_hi, cb, parent, edge};
  const int nu = u_hi - u_lo;
  cudaError_t e;
  if (prec == MPS_PREC_FP64) {
    const int P = std::max(1, 16 / D), rows = std::min(nu, P) * D;
    const size_t smem = gate::gemm_tile_bytes<256>() + sizeof(Cx<double>) * (size_t)rows * 2 * Dp;
    if ((e = gate::raise_smem_limit<k_level_fused64>()) != cudaSuccess) return e;
    k_level_fused64<<<(nu + P - 1) / P, 256, smem, st>>>(m, g, (const Cx<double>*)L, (Cx<double>*)Lout);
    return cudaGetLastError();
  }
  const int P = std::max(1, 64 / D);
  const size_t smem = sizeof(Cx<float>) * ((size_t)D * 2 * Dp + 64 * (size_t)(D + 1) + 64 * (size_t)2 * Dp);
  auto go = [&](auto dp) {
    constexpr auto kern = k_level_fused<decltype(dp)::value>;
    cudaError_t r = gate::raise_smem_limit<kern>();
    if (r != cudaSuccess) return r;
    kern<<<(nu + P - 1) / P, 256, smem, st>>>(m, g, (const Cx<float>*)L, (Cx<float>*)Lout);
    return cudaGetLastError();
  };
  if (Dp <= 8) return go(std::integral_constant<int, 8>{});
  if (Dp <= 16) return go(std::integral_constant<int, 16>{});
  if (Dp <= 32) return go(std::integral_constant<int, 32>{});
  return go(std::integral_constant<int, 64>{});
}

// <P> (unnormalised) of a string closing at site k with letter P on node u:
// sum_ab L[u][a][b] conj(Q_k^P[a][b]), Q_k^P = sum_ij conj(P_ij) Bhat_k^i (B_k^j)^+ from the
// right-environment pass. This equals sum_ij P_ij <Bhat_k^i, L[u] B_k^j>_F (Eq. 11 with
// the right part contracted first) and reads one D x D block of the node instead of the
// two D x D' blocks of T. Both blocks are contiguous with leading dimension env_ld(D).
template <class R>
__global__ void __launch_bounds__(256) k_level_close(DevMPS m, int slot, int k, const int32_t* cnode,
                                                     const uint8_t* cletter, const int32_t* cterm,
                                                     const Cx<R>* L, const Cx<R>* Q, double* vals,
                                                     int node_base) {
  __shared__ double red[2][8];
  const int c = blockIdx.x;
  const int chi2 = m.chi * env_ld<R>(m.chi);
  const int* rank = m.rank + (size_t)slot * (m.n + 1);
  const int Dk = rank[k], ld = env_ld<R>(Dk);
  const Cx<R>* Lu = L + (cnode[c] - node_base) * env_node<R>(Dk);
  const Cx<R>* Qp = Q + ((size_t)k * 4 + (cletter[c] & 3)) * chi2;
  const int n = Dk * ld;
  double re = 0.0, im = 0.0;
  // R = float: FP32 products summed in FP32 over runs of 8 entries, the runs summed in
  // FP64. GB300's FP64 (and FP32 -> FP64 conversion) throughput is a small fraction of
  // its FP32 rate; one FP64 step per entry made the close a third of a chi = 256
  // measurement. A run's FP32 sum is off by at most ~8 ulps of its magnitudes, below the
  // ~2^-21 relative error of the tensor-core environments. R = double: FP64.
  int idx = threadIdx.x;
  for (; idx + 7 * 256 < n; idx += 8 * 256) {
    // a full run: its 16 loads are issued before the products that use them
    Cx<R> q[8], l[8];
#pragma unroll
    for (int t = 0; t < 8; ++t) {
      q[t] = Qp[idx + t * 256];
      l[t] = Lu[idx + t * 256];
    }
    R sr = 0, si = 0;
#pragma unroll
    for (int t = 0; t < 8; ++t) {
      // conj(q) * l
      sr += q[t].x * l[t].x + q[t].y * l[t].y;
      si += q[t].x * l[t].y - q[t].y * l[t].x;
    }
    re += (double)sr;
    im += (double)si;
  }
  if (idx < n) {
    R sr = 0, si = 0;
    for (; idx < n; idx += 256) {
      const Cx<R> q = Qp[idx], l = Lu[idx];
      sr += q.x * l.x + q.y * l.y;
      si += q.x * l.y - q.y * l.x;
    }
    re += (double)sr;
    im += (double)si;
  }
  for (int o = 16; o > 0; o >>= 1) {
    re += __shfl_xor_sync(0xffffffffu, re, o);
    im += __shfl_xor_sync(0xffffffffu, im, o);
  }
  if ((threadIdx.x & 31) == 0) {
    red[0][threadIdx.x >> 5] = re;
    red[1][threadIdx.x >> 5] = im;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double a = 0, b = 0;
    for (int w = 0; w < 8; ++w) {
      a += red[0][w];
      b += red[1][w];
    }
    vals[2 * (size_t)cterm[c]] = a;
    vals[2 * (size_t)cterm[c] + 1] = b;
  }
}

cudaError_t launch_env_T(const DevMPS& m, int prec, int slot, int k, const void* L, void* T, int n_nodes,
                         const int32_t* cb, cudaStream_t st) {
  if (n_nodes <= 0) return cudaSuccess;
  if (prec == MPS_PREC_FP64)
    k_level_T<double><<<dim3(n_nodes, 2), 256, 0, st>>>(m, slot, k, (const Cx<double>*)L, (Cx<double>*)T, cb);
  else
    k_level_T<float><<<dim3(n_nodes, 2), 256, 0, st>>>(m, slot, k, (const Cx<float>*)L, (Cx<float>*)T, cb);
  return cudaGetLastError();
}

cudaError_t launch_env_close(const DevMPS& m, int prec, int slot, int k, const void* L, const void* Q,
                             const int32_t* cnode, const uint8_t* cletter, const int32_t* cterm, int n_closes,
                             int node_base, double* vals, cudaStream_t st) {
  if (n_closes <= 0) return cudaSuccess;
  if (prec == MPS_PREC_FP64)
    k_level_close<double><<<n_closes, 256, 0, st>>>(m, slot, k, cnode, cletter, cterm, (const Cx<double>*)L,
                                                     (const Cx<double>*)Q, vals, node_base);
  else
    k_level_close<float><<<n_closes, 256, 0, st>>>(m, slot, k, cnode, cletter, cterm, (const Cx<float>*)L,
                                                    (const Cx<float>*)Q, vals, node_base);
  return cudaGetLastError();
}

cudaError_t launch_env_child(const DevMPS& m, int prec, int slot, int k, const void* T, const int32_t* parent,
                             const uint8_t* edge, int n_children, int node_base, void* Lout, cudaStream_t st) {
  if (n_children <= 0) return cudaSuccess;
  if (prec == MPS_PREC_FP64)
    k_level_child<double><<<n_children, 256, 0, st>>>(m, slot, k, parent, edge, (const Cx<double>*)T,
                                                       (Cx<double>*)Lout, node_base);
  else
    k_level_child<float><<<n_children, 256, 0, st>>>(m, slot, k, parent, edge, (const Cx<float>*)T,
                                                      (Cx<float>*)Lout, node_base);
  return cudaGetLastError();
}

// ------------------------------------------------------------------ energy sum
// E = sum_i a_i <P_i> in FP64, compensated throughout: each thread runs a Neumaier sum over
// its terms, pairs (sum, correction) are then merged by TwoSum in a fixed tree. A block
// covers 256 threads x kTermsPerThread terms; the block that finishes last merges the
// blocks' pairs in block order, so the result does not depend on the schedule.
constexpr int kTermsPerThread = 4;
__device__ __forceinline__ void neumaier_add(double& s, double& c, double v) {
  const double t = s + v;
  if (fabs(s) >= fabs(v))
    c += (s - t) + v;
  else
    c += (v - t) + s;
  s = t;
}
__device__ __forceinline__ void merge_pair(double& s, double& c, double s2, double c2) {
  const double t = s + s2, b = t - s;
  c = (c + c2) + ((s - (t - b)) + (s2 - b));
  s = t;
}
// The sum over a block's threads, in thread 0.
__device__ __forceinline__ void block_merge(double& s, double& c, double (*sh)[2]) {
  for (int o = 1; o < 32; o <<= 1) {
    const double s2 = __shfl_down_sync(0xffffffffu, s, o), c2 = __shfl_down_sync(0xffffffffu, c, o);
    merge_pair(s, c, s2, c2);
  }
  const int warp = threadIdx.x >> 5;
  if ((threadIdx.x & 31) == 0) {
    sh[warp][0] = s;
    sh[warp][1] = c;
  }
  __syncthreads();
  if (threadIdx.x == 0)
    for (int w = 1; w < 8; ++w) merge_pair(s, c, sh[w][0], sh[w][1]);
}

template <class R>
__global__ void __launch_bounds__(256) k_energy_sum(int64_t n_terms, const double* coeff, const double* vals,
                                                    const Cx<R>* R0, double id_coeff, int64_t id_term, double* part,
                                                    unsigned* done, double* out) {
  __shared__ double sh[8][2];
  __shared__ bool last;
  const double norm = (double)R0[0].x;
  const double2* v2 = reinterpret_cast<const double2*>(vals);
  double2* o2 = reinterpret_cast<double2*>(out + 4);
  double s = 0.0, c = 0.0;
#pragma unroll
  for (int i = 0; i < kTermsPerThread; ++i) {
    const int64_t t = ((int64_t)blockIdx.x * kTermsPerThread + i) * 256 + threadIdx.x;
    if (t < n_terms) {
      double2 v = make_double2(1.0, 0.0);
      if (t != id_term) {
        v = v2[t];
        v.x /= norm;
        v.y /= norm;
        neumaier_add(s, c, coeff[t] * v.x);
      }
      o2[t] = v;
    }
  }
  block_merge(s, c, sh);
  if (threadIdx.x == 0) {
    part[2 * blockIdx.x] = s;
    part[2 * blockIdx.x + 1] = c;
    __threadfence();
    last = atomicAdd(done, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  s = c = 0.0;
  const int per = (gridDim.x + 255) / 256;
  for (int i = 0; i < per; ++i) {
    const unsigned b = threadIdx.x * per + i;
    if (b < gridDim.x) merge_pair(s, c, __ldcg(part + 2 * b), __ldcg(part + 2 * b + 1));
  }
  __syncthreads();
  block_merge(s, c, sh);
  if (threadIdx.x == 0) {
    neumaier_add(s, c, id_coeff);
    out[0] = s + c;
    out[1] = norm;
    *done = 0;   // ready for the next measurement of this handle
  }
}

int64_t energy_sum_blocks(int64_t n_terms) {
  const int64_t per = 256 * kTermsPerThread;
  return n_terms > 0 ? (n_terms + per - 1) / per : 1;
}

cudaError_t launch_energy_sum(int prec, MeasDev& w, int64_t n_terms, const double* coeff_dev, double id_coeff,
                              int64_t id_term, cudaStream_t st) {
  const unsigned grid = (unsigned)energy_sum_blocks(n_terms);
  if (prec == MPS_PREC_FP64)
    k_energy_sum<double><<<grid, 256, 0, st>>>(n_terms, coeff_dev, w.vals, (const Cx<double>*)w.R, id_coeff, id_term,
                                               w.part, w.done, w.out);
  else
    k_energy_sum<float><<<grid, 256, 0, st>>>(n_terms, coeff_dev, w.vals, (const Cx<float>*)w.R, id_coeff, id_term,
                                              w.part, w.done, w.out);
  return cudaGetLastError();
}

}  // namespace mpsvqe

