// CUDA kernels of the MPS-VQE hot path for sm_103a (GB300).
//
//  k_reset        product-state reference (Sec. III-D: X gates on the occupied qubits).
//  k_right_envs   right identity environments R_k and B^_k = B_k R_{k+1}.
//  k_level_T/child/close   one level of the Pauli-string prefix trie (Eq. 11 generalised).
//  k_energy_sum   E = sum_i a_i <P_i> (Eq. 2) with Neumaier compensation in FP64.
#include <cfloat>
#include <cmath>
#include <cstdint>

#include "cx.cuh"
#include "kernels.cuh"

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
// C (Mdim x Ndim, ldc) = sum_t s_t opA_t(A_t) opB_t(B_t) with NTH threads (256 or 512)
// and 64x64 tiles. opA: A stored Mdim x K (lda), or K x Mdim used as A^H (conjT).
// opB: B stored K x Ndim (ldb), or Ndim x K used as B^T (transB); conjB conjugates the
// entries of B as they are loaded.
template <class R>
struct GemmTerm {
  const Cx<R>* A;
  int lda;
  bool conjT;
  const Cx<R>* B;
  int ldb;
  Cx<R> s;
  bool transB;
  bool conjB = false;
};

// One 64 x 64 output tile at (m0, n0).
template <class R, int NTH>
__device__ void gemm_tile(int m0, int n0, int Mdim, int Ndim, int K, const GemmTerm<R>* terms, int nterm, Cx<R>* C,
                          int ldc, Cx<R> (*As)[17], Cx<R> (*Bs)[65]) {
  constexpr int TY = NTH / 16, RPT = 64 / TY;
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
        const int r = T.transB ? (e & 15) : (e >> 6), cc = T.transB ? (e >> 4) : (e & 63);
        const int gk = k0 + r, gn = n0 + cc;
        Cx<R> v = cx<R>(0, 0);
        if (gk < K && gn < Ndim) v = T.transB ? T.B[(size_t)gn * T.ldb + gk] : T.B[(size_t)gk * T.ldb + gn];
        Bs[r][cc] = T.conjB ? conj(v) : v;
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

template <class R, int NTH>
__device__ void block_gemm(int Mdim, int Ndim, int K, const GemmTerm<R>* terms, int nterm, Cx<R>* C, int ldc,
                           Cx<R> (*As)[17], Cx<R> (*Bs)[65]) {
  for (int m0 = 0; m0 < Mdim; m0 += 64)
    for (int n0 = 0; n0 < Ndim; n0 += 64) gemm_tile<R, NTH>(m0, n0, Mdim, Ndim, K, terms, nterm, C, ldc, As, Bs);
}

// The same product spread over a grid: one 64 x 64 tile per thread block, blockIdx.z
// selecting one of up to four independent products.
template <class R>
struct GridGemm {
  GemmTerm<R> t[4][2];
  int nterm;
  Cx<R>* C[4];
  int ldc, M, N, K;
};

template <class R>
__global__ void __launch_bounds__(256) k_cgemm_grid(GridGemm<R> g) {
  __shared__ Cx<R> As[64][17];
  __shared__ Cx<R> Bs[16][65];
  const int z = blockIdx.z;
  gemm_tile<R, 256>(blockIdx.y * 64, blockIdx.x * 64, g.M, g.N, g.K, g.t[z], g.nterm, g.C[z], g.ldc, As, Bs);
}

// --------------------------------------------------------- right environments
// R_n = [1]; R_k = sum_i Bhat_k^i (B_k^i)^+ with Bhat_k^i = B_k^i R_{k+1} (same layout as
// B_k). Per site two grid launches (the two Bhat^i products side by side, then R_k), so
// large bond dimensions use many SMs. ranks: the slot's bond ranks on the host
// (ranks[k] = left dimension of site k).
template <class R>
static cudaError_t right_envs_t(const DevMPS& m, int slot, const int* ranks, const int64_t* site_off, Cx<R>* Renv,
                                Cx<R>* Bhat, Cx<R>* Q, cudaStream_t st) {
  const int n = m.n;
  const size_t chi2 = (size_t)m.chi * m.chi;
  const Cx<R>* Bslot = (const Cx<R>*)m.B + (size_t)slot * m.slot_elems;
  static const Cx<R> one = cx<R>(1, 0);
  cudaError_t e = cudaMemcpyAsync(Renv + (size_t)n * chi2, &one, sizeof(Cx<R>), cudaMemcpyHostToDevice, st);
  if (e != cudaSuccess) return e;
  for (int k = n - 1; k >= 0; --k) {
    const int Dl = ranks[k], Dr = ranks[k + 1];
    const Cx<R>* Bk = Bslot + site_off[k];
    Cx<R>* Bh = Bhat + site_off[k];
    const Cx<R>* Rn = Renv + (size_t)(k + 1) * chi2;
    GridGemm<R> g{};
    g.nterm = 1;
    g.ldc = 2 * Dr;
    g.M = Dl;
    g.N = Dr;
    g.K = Dr;
    for (int i = 0; i < 2; ++i) {   // Bhat^i = B^i R_{k+1}: (Dl x Dr)(Dr x Dr)
      g.t[i][0] = GemmTerm<R>{Bk + i * Dr, 2 * Dr, false, Rn, Dr, cx<R>(1, 0), false};
      g.C[i] = Bh + i * Dr;
    }
    k_cgemm_grid<R><<<dim3((Dr + 63) / 64, (Dl + 63) / 64, 2), 256, 0, st>>>(g);
    // R_k = sum_i Bhat^i (B^i)^+: B^i read as (Dl x Dr) transposed and conjugated
    GridGemm<R> h{};
    h.nterm = 2;
    h.ldc = Dl;
    h.M = Dl;
    h.N = Dl;
    h.K = Dr;
    for (int i = 0; i < 2; ++i) h.t[0][i] = GemmTerm<R>{Bh + i * Dr, 2 * Dr, false, Bk + i * Dr, 2 * Dr, cx<R>(1, 0), true, true};
    h.C[0] = Renv + (size_t)k * chi2;
    k_cgemm_grid<R><<<dim3((Dl + 63) / 64, (Dl + 63) / 64, 1), 256, 0, st>>>(h);
    // Q_k^P = sum over the letter's two entries (i, j, s) of conj(s) Bhat^i (B^j)^+, one
    // product per letter I, X, Y, Z: a string closing at site k with letter P has
    // <P> = sum_ab L[a][b] conj(Q_k^P[a][b]) (Eq. 11 with the right part contracted)
    GridGemm<R> q{};
    q.nterm = 2;
    q.ldc = Dl;
    q.M = Dl;
    q.N = Dl;
    q.K = Dr;
    for (int l = 0; l < 4; ++l) {
      const int ii[4][2] = {{0, 1}, {0, 1}, {0, 1}, {0, 1}};
      const int jj[4][2] = {{0, 1}, {1, 0}, {1, 0}, {0, 1}};
      // conj of the letter's entries: I (1, 1), X (1, 1), Y (-i, i) -> (i, -i), Z (1, -1)
      const Cx<R> cs[4][2] = {{cx<R>(1, 0), cx<R>(1, 0)},
                              {cx<R>(1, 0), cx<R>(1, 0)},
                              {cx<R>(0, 1), cx<R>(0, -1)},
                              {cx<R>(1, 0), cx<R>(-1, 0)}};
      for (int e = 0; e < 2; ++e)
        q.t[l][e] = GemmTerm<R>{Bh + ii[l][e] * Dr, 2 * Dr, false, Bk + jj[l][e] * Dr, 2 * Dr, cs[l][e], true, true};
      q.C[l] = Q + ((size_t)k * 4 + l) * chi2;
    }
    k_cgemm_grid<R><<<dim3((Dl + 63) / 64, (Dl + 63) / 64, 4), 256, 0, st>>>(q);
  }
  return cudaGetLastError();
}

cudaError_t launch_right_envs(const DevMPS& m, int prec, int slot, const int* ranks, const int64_t* site_off,
                              MeasDev& w, cudaStream_t st, int* launches) {
  *launches += 3 * m.n;
  if (prec == MPS_PREC_FP64)
    return right_envs_t<double>(m, slot, ranks, site_off, (Cx<double>*)w.R, (Cx<double>*)w.Bhat, (Cx<double>*)w.Q,
                                st);
  return right_envs_t<float>(m, slot, ranks, site_off, (Cx<float>*)w.R, (Cx<float>*)w.Bhat, (Cx<float>*)w.Q, st);
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

// Level buffers are dense: node u of level k holds L at u Dk^2 (leading dimension Dk)
// and, on the CUDA-core route, T_j at (2u + j) Dk Dk1 (leading dimension Dk1).
// T_j[u] = L_k[u] B_k^j  (Dk x Dk)(Dk x Dk1), grid (nodes, 2)
template <class R>
__global__ void __launch_bounds__(256) k_level_T(DevMPS m, int slot, int k, const Cx<R>* Lin, Cx<R>* T) {
  __shared__ Cx<R> As[64][17];
  __shared__ Cx<R> Bs[16][65];
  const int u = blockIdx.x, j = blockIdx.y;
  const int* rank = m.rank + (size_t)slot * (m.n + 1);
  const int Dk = rank[k], Dk1 = rank[k + 1];
  const Cx<R>* Bk = (const Cx<R>*)m.B + (size_t)slot * m.slot_elems + m.site_off[k];
  GemmTerm<R> t{Lin + (size_t)u * Dk * Dk, Dk, false, Bk + j * Dk1, 2 * Dk1, cx<R>(1, 0), false};
  block_gemm<R, 256>(Dk, Dk1, Dk, &t, 1, T + ((size_t)u * 2 + j) * Dk * Dk1, Dk1, As, Bs);
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
    t[e] = GemmTerm<R>{Bk + ii[e] * Dk1, 2 * Dk1, true, T + ((size_t)u * 2 + jj[e]) * Dk * Dk1, Dk1, sg[e], false};
  block_gemm<R, 256>(Dk1, Dk1, Dk, t, 2, Lout + (size_t)c * Dk1 * Dk1, Dk1, As, Bs);
}

// <P> (unnormalised) of a string closing at site k with letter P on node u:
// sum_ab L[u][a][b] conj(Q_k^P[a][b]), Q_k^P = sum_ij conj(P_ij) Bhat_k^i (B_k^j)^+ from the
// right-environment pass. This equals sum_ij P_ij <Bhat_k^i, L[u] B_k^j>_F (Eq. 11 with
// the right part contracted first) and reads one D x D block of the node instead of the
// two D x D' blocks of T. Both blocks are contiguous with leading dimension D.
template <class R>
__global__ void __launch_bounds__(256) k_level_close(DevMPS m, int slot, int k, const int32_t* cnode,
                                                     const uint8_t* cletter, const int32_t* cterm,
                                                     const Cx<R>* L, const Cx<R>* Q, double* vals,
                                                     int node_base) {
  __shared__ double red[2][8];
  const int c = blockIdx.x;
  const int chi2 = m.chi * m.chi;
  const int* rank = m.rank + (size_t)slot * (m.n + 1);
  const int Dk = rank[k];
  const Cx<R>* Lu = L + (size_t)(cnode[c] - node_base) * Dk * Dk;
  const Cx<R>* Qp = Q + ((size_t)k * 4 + (cletter[c] & 3)) * chi2;
  const int n = Dk * Dk;
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
                         cudaStream_t st) {
  if (n_nodes <= 0) return cudaSuccess;
  if (prec == MPS_PREC_FP64)
    k_level_T<double><<<dim3(n_nodes, 2), 256, 0, st>>>(m, slot, k, (const Cx<double>*)L, (Cx<double>*)T);
  else
    k_level_T<float><<<dim3(n_nodes, 2), 256, 0, st>>>(m, slot, k, (const Cx<float>*)L, (Cx<float>*)T);
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
__device__ __forceinline__ void neumaier_add(double& s, double& c, double v) {
  const double t = s + v;
  if (fabs(s) >= fabs(v))
    c += (s - t) + v;
  else
    c += (v - t) + s;
  s = t;
}

template <class R>
__global__ void __launch_bounds__(1024) k_energy_sum(int64_t n_terms, const double* coeff, const double* vals,
                                                     const Cx<R>* R0, double id_coeff, int64_t id_term,
                                                     double* out) {
  __shared__ double ps[1024], pc[1024];
  const double norm = (double)R0[0].x;
  const int64_t chunk = (n_terms + 1023) / 1024;
  const int64_t b = (int64_t)threadIdx.x * chunk, e = min(n_terms, b + chunk);
  double s = 0.0, c = 0.0;
  for (int64_t t = b; t < e; ++t) {
    double re, im;
    if (t == id_term) {
      re = 1.0;
      im = 0.0;
    } else {
      re = vals[2 * t] / norm;
      im = vals[2 * t + 1] / norm;
      neumaier_add(s, c, coeff[t] * re);
    }
    out[4 + 2 * t] = re;
    out[5 + 2 * t] = im;
  }
  ps[threadIdx.x] = s;
  pc[threadIdx.x] = c;
  __syncthreads();
  if (threadIdx.x == 0) {
    double S = 0.0, Cc = 0.0;
    for (int i = 0; i < 1024; ++i) {
      neumaier_add(S, Cc, ps[i]);
      neumaier_add(S, Cc, pc[i]);
    }
    neumaier_add(S, Cc, id_coeff);
    out[0] = S + Cc;
    out[1] = norm;
  }
}

cudaError_t launch_energy_sum(const DevMPS& m, int prec, int slot, MeasDev& w, int64_t n_terms,
                              const double* coeff_dev, double id_coeff, int64_t id_term, cudaStream_t st) {
  (void)m;
  (void)slot;
  if (prec == MPS_PREC_FP64)
    k_energy_sum<double><<<1, 1024, 0, st>>>(n_terms, coeff_dev, w.vals, (const Cx<double>*)w.R, id_coeff,
                                             id_term, w.out);
  else
    k_energy_sum<float><<<1, 1024, 0, st>>>(n_terms, coeff_dev, w.vals, (const Cx<float>*)w.R, id_coeff,
                                            id_term, w.out);
  return cudaGetLastError();
}

}  // namespace mpsvqe

