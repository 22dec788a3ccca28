// The gate engine: persistent kernel that applies a list of two-site gates to each MPS
// slot, one thread-block cluster per slot.
//
// Per gate: Eq. (7) contraction and 4x4 gate, Eq. (8) row scaling by lambda_{n-1}, Eq. (9)
// truncated SVD (bidiagonal route; one-sided Jacobi for spectra that stay degenerate),
// Eq. (10) updates. One evaluation's gate chain is serial, so what a gate costs is its own
// latency; a cluster of C blocks spreads every stage of it over C SMs, and keeps M' in
// distributed shared memory where one block's is too small. Where C depends on how many slots
// run together, C VG (virtual ranks: how the columns and the sums are dealt out) does not, so a
// slot's result does not depend on its company.
//
// A gate is bound by the latency of its serial stages, not by bandwidth or arithmetic. Time of a
// gate of a saturated circuit, with one block per slot before and now: FP64 chi = 16 1 000 and
// 115 us, chi = 64 16.8 and 1.6 ms; mixed chi = 16 60 and 38 us (one block still), chi = 33 280
// and 135, chi = 64 746 and 263 us, chi = 128 (M' in L2 before, in shared memory now) 6.5 and
// 0.74 ms, all with one slot; with many, see gate.cu.
#pragma once
#include <atomic>
#include <type_traits>

#include "gate.cuh"
#include "smem_limit.cuh"

namespace mpsvqe {

template <class R>
struct Eps;
template <>
struct Eps<double> {
  static constexpr double v = 2.220446049250313e-16;
};
template <>
struct Eps<float> {
  static constexpr float v = 1.1920929e-7f;
};

// Algorithmic real flops of one gate step, counted as the textbook dense algorithms:
// contraction theta = B_n B_{n+1} (2 rl x rm x 2 rr complex MACs), the 4x4 gate on
// (i, j), Golub-Reinsch SVD of the (m x n) complex M' computing singular values and
// right vectors (4 (4 m n^2 + 8 n^3) real flops for m >= n, roles swapped otherwise),
// and the site update B_n = M V^H (2 rl x 2 rr x k complex MACs). A complex MAC is 8.
__device__ __forceinline__ double flops_per_gate(int rl, int rm, int rr, int k) {
  const float m = 2.0f * rl, n = 2.0f * rr;   // products stay below 2^31: exact enough for a count
  const float big = m >= n ? m : n, small = m >= n ? n : m;
  const double contract = 8.0f * m * rm * n + 8.0f * 4.0f * m * n;
  const double svd = 4.0f * (4.0f * big * small * small + 8.0f * small * small * small);
  const double update = 8.0f * m * n * k;
  return contract + svd + update;
}

// Capacity of bond b (b = -1 and b = n-1 are the trivial outer bonds): the largest rank
// an n-site MPS with bond cap chi can have there, min(chi, 2^min(b+1, n-1-b)).
__device__ __forceinline__ int bond_cap(int b, int n, int chi) {
  if (b < 0 || b >= n - 1) return 1;
  const int e = min(min(b + 1, n - 1 - b), 30);
  return min(chi, 1 << e);
}

namespace gate {

// s + c += a b without rounding errors beyond c's: TwoProd by FMA and TwoSum (Knuth), the
// step of the compensated dot product "Dot2" (Ogita, Rump and Oishi, 2005). The _rn
// intrinsics keep the compiler from contracting the products into the sums.
__device__ __forceinline__ void dot2_acc(float a, float b, float& s, float& c) {
  const float p = __fmul_rn(a, b);
  const float ep = fmaf(a, b, -p);
  const float t = __fadd_rn(s, p);
  const float bv = __fsub_rn(t, s);
  const float et = __fadd_rn(__fsub_rn(s, __fsub_rn(t, bv)), __fsub_rn(p, bv));
  s = t;
  c = __fadd_rn(c, __fadd_rn(ep, et));
}

// Shared-memory plan of one block. Two areas have several tenants in turn:
//   exchange  GEMM tiles of the contraction | exchange buffers of the bidiagonalisation |
//             TGK arrays, its blocks, singular values, orderings
//   work      own columns of T | pivots of the twisted factorisations | chunks of W, V or
//             reflectors and the rows of E | GEMM tiles of the site update
// TG: T does not fit; as many columns as the rest of an SM's shared memory holds stay there.
template <class R, int NT, int C, int VG, bool TG>
struct Plan {
  static constexpr size_t kFixed = 3072;   // gate, record, reductions, ranks, site offsets
  static constexpr size_t kCap = 227 * 1024 - 1024;
  size_t fixed, exch, work, total;
  int mmax, cl, kc;
  int vb;   // vectors whose twisted factorisations are in shared memory together
  __host__ __device__ static size_t up(size_t b) { return (b + 255) & ~(size_t)255; }
  // leading dimension of T: 8 (mod 16) complex<float> entries, so that the two 8-lane
  // column walks of a half warp fall into different banks
  __host__ __device__ static int lead(int rows) { return sizeof(R) == 4 ? (rows + 15) / 16 * 16 + 8 : rows; }
  __host__ __device__ explicit Plan(int chi) {
    mmax = 2 * chi;
    cl = 2 * ((chi + C - 1) / C);
    kc = (chi + C - 1) / C;
    vb = kc;
    if (TG) {
      const int fit = (int)(96 * 1024 / (sizeof(R) * 2 * 2 * mmax));
      if (fit < vb) vb = fit;
    }
    fixed = up(kFixed + sizeof(R) * 2 * mmax + sizeof(Cx<R>) * 2 * mmax);
    const size_t bidiag = up(sizeof(Cx<R>) * ((size_t)2 * C * VG * mmax + 4 * (size_t)mmax + 4 * cl + 8) +
                             sizeof(R) * 2 * C * VG);
    const size_t post = up(sizeof(R) * (2 * 2 * (size_t)mmax + 2 * mmax) + sizeof(float) * 2 * mmax +
                           (8 + 2 * 4) * (size_t)mmax + 256 * sizeof(R) + 48 + sizeof(int) * (8 * (size_t)mmax + 4) +
                           sizeof(R) * 2 * vb * (2 * (size_t)mmax / SturmGroup<R>::v + 1));
    const size_t tiles = up(gemm_tile_bytes<NT>());
    exch = bidiag > post ? bidiag : post;
    if (tiles > exch) exch = tiles;
    const size_t t = TG ? 0 : up(sizeof(Cx<R>) * (size_t)cl * lead(mmax));
    const size_t twist = up(sizeof(R) * (size_t)vb * 2 * 2 * mmax);
    const size_t nsr = up(sizeof(R) * ((size_t)kc * chi + (size_t)chi * 33));
    const size_t nsc = sizeof(R) == 4 ? up(8 * (size_t)kc * chi + 16 * (size_t)chi * 33 + 16) : 0;
    const size_t ychunk = up(sizeof(Cx<R>) * 16 * (size_t)mmax);   // at least 16 reflectors
    work = t;
    for (size_t b : {twist, nsr, nsc, ychunk, tiles})
      if (b > work) work = b;
    total = fixed + exch + work;
    // room for the whole Jacobi matrix where a block has it, and for longer chunks
    const size_t want = up(sizeof(R) * (size_t)mmax * (mmax + 1));
    if (TG && total < kCap) {
      work = (kCap - fixed - exch) & ~(size_t)255;
      total = fixed + exch + work;
    } else if (want > work && fixed + exch + want <= kCap) {
      work = want;
      total = fixed + exch + work;
    }
  }
};

// Columns [q0, q0 + 32) of k rows (global, row length len) to shared memory, 33 entries a
// row, zeros beyond len. Eight loads are in flight per thread: one after the other, the
// trips to L2 took longer than the products made of them.
template <int NT, class V, class ST>
__device__ __forceinline__ int load_chunk(const V* X, int k, int len, int q0, ST store) {
  const int qn = min(32, len - q0);
  __syncthreads();
  const int q = threadIdx.x & 31, j0 = threadIdx.x >> 5;
  constexpr int RS = NT / 32;
  for (int j = j0; j < k; j += 8 * RS) {
    V v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      v[u] = V{};
      if (j + u * RS < k && q < qn) v[u] = ldcg(X + (size_t)(j + u * RS) * len + q0 + q);
    }
#pragma unroll
    for (int u = 0; u < 8; ++u)
      if (j + u * RS < k) store((j + u * RS) * 33 + q, v[u]);
  }
  __syncthreads();
  return qn;
}

// One Newton-Schulz step X <- X - (1/2) E X, E = X X^T - I, on the real rows w_0..w_{k-1}
// (length p) in global memory: this block's rows (t = rank + C i) of E, their largest
// absolute row sum, and (when asked) the updated rows.
template <class R, int NT, int C>
__device__ __forceinline__ R real_defect(const R* W, int k, int p, int kcv, unsigned rank, R* E, R* chunk, R* red) {
  const int tid = threadIdx.x;
  constexpr int QC = 32, LDC = 33, SP = C == 1 ? 16 : 8;
  const int npair = kcv * k;
  // once, but for many vectors in two or four blocks
  for (int e0 = tid; e0 - tid < (C == 2 || C == 4 ? npair : 1); e0 += SP * NT) {
    R acc[SP];
#pragma unroll
    for (int s = 0; s < SP; ++s) acc[s] = R(0);
    for (int q0 = 0; q0 < p; q0 += QC) {
      load_chunk<NT>(W, k, p, q0, [&](int at, R v) { chunk[at] = v; });
#pragma unroll
      for (int s = 0; s < SP; ++s) {
        const int e = e0 + s * NT;
        if (e < npair) {
          const int i = e / k, j = e - i * k;
          const R* wi = chunk + (rank + C * i) * LDC;
          const R* wj = chunk + j * LDC;
          R a = acc[s];
#pragma unroll 8
          for (int q = 0; q < QC; ++q) a = fma(wi[q], wj[q], a);
          acc[s] = a;
        }
      }
    }
    __syncthreads();
#pragma unroll
    for (int s = 0; s < SP; ++s) {
      const int e = e0 + s * NT;
      if (e < npair) {
        const int i = e / k, j = e - i * k;
        E[e] = acc[s] - (j == (int)rank + C * i ? R(1) : R(0));
      }
    }
  }
  __syncthreads();
  // largest row sum of |E|, as FP32 (it only steers the iteration)
  float worst = 0.f;
  const int warp = tid >> 5, lane = tid & 31;
  for (int i = warp; i < kcv; i += NT / 32) {
    float s = 0.f;
    for (int j = lane; j < k; j += 32) s += fabsf((float)E[i * k + j]);
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    worst = fmaxf(worst, s == s ? s : 3e38f);   // a NaN counts as a failure
  }
  if (lane == 0) red[warp] = (R)worst;
  __syncthreads();
  R m = R(0);
  for (int w = 0; w < NT / 32; ++w) m = fmax(m, red[w]);
  return m;
}

template <class R, int NT, int C>
__device__ __forceinline__ void real_update(const R* W, R* out, int k, int p, int kcv, unsigned rank, const R* E, R* chunk) {
  const int tid = threadIdx.x;
  constexpr int QC = 32, LDC = 33;
  for (int q0 = 0; q0 < p; q0 += QC) {
    const int qn = load_chunk<NT>(W, k, p, q0, [&](int at, R v) { chunk[at] = v; });
    for (int e = tid; e < kcv * QC; e += NT) {
      const int i = e / QC, q = e % QC;
      if (q >= qn) continue;
      R a = R(0);
#pragma unroll 4
      for (int j = 0; j < k; ++j) a = fma(E[i * k + j], chunk[j * LDC + q], a);
      const int t = rank + C * i;
      out[(size_t)t * p + q0 + q] = fma(R(-0.5), a, chunk[t * LDC + q]);
    }
  }
}

// Mixed precision: one Newton-Schulz step on the complex rows x_0..x_{k-1} of V (global,
// row length len) that the FP32 back-transformation leaves orthonormal only to a few
// 1e-7. E = X X^H - I is a few 1e-7 itself, so its Gram matrix has to be accurate far
// below FP32 resolution: the split products of the contractions give that (leading parts
// summed exactly, the rest 2^-12 times smaller) at four FMAs per real product, where a
// compensated (Dot2) sum takes eleven operations. One thread: column j of E and up to SP
// of this block's rows, so that a split entry of x_j serves them all.
template <int NT, int C>
__device__ __forceinline__ void newton_schulz_cluster(const Cx<float>* X, int k, int len, int kcv, unsigned rank,
                                                      Cx<float>* E, SplitF* chunk, Cx<float>* out, Cx<float>* site) {
  const int tid = threadIdx.x;
  constexpr int QC = 32, LDC = 33;
  const int jsh = row_shift(k), j = tid & ((1 << jsh) - 1), i0 = tid >> jsh, istep = NT >> jsh;
  const int ns = (kcv + istep - 1) / istep;   // rows per thread, uniform
  auto load = [&](int q0) {
    return load_chunk<NT>(X, k, len, q0, [&](int at, Cx<float> v) { chunk[at] = to_elem(v); });
  };
  auto gram = [&](auto sp, int r0) {   // rows r0 .. of each thread
    constexpr int NS = decltype(sp)::value;
    const int i1 = i0 + r0 * istep;
    SplitAcc acc[NS];
    const SplitF* row[NS];
#pragma unroll
    for (int s = 0; s < NS; ++s) {
      zero(acc[s]);
      row[s] = chunk + ((int)rank + C * max(min(i1 + s * istep, kcv - 1), 0)) * LDC;
    }
    for (int q0 = 0; q0 < len; q0 += QC) {
      load(q0);
      if (j < k) {
#pragma unroll 4
        for (int q = 0; q < QC; ++q) {
          SplitF b = chunk[j * LDC + q];
          b.v.z = -b.v.z;   // conj
          b.v.w = -b.v.w;
#pragma unroll
          for (int s = 0; s < NS; ++s) mac(acc[s], row[s][q], b);
        }
      }
    }
    __syncthreads();
    if (j < k) {
#pragma unroll
      for (int s = 0; s < NS; ++s) {
        const int i = i1 + s * istep;
        if (i < kcv) {
          const bool diag = j == (int)rank + C * i;
          E[i * k + j] = diag ? cx<float>(__fadd_rn(__fadd_rn(acc[s].hx, -1.0f), acc[s].lx), 0.f) : value(acc[s]);
        }
      }
    }
  };
  if (ns <= 1)
    gram(std::integral_constant<int, 1>{}, 0);
  else if (ns <= 2)
    gram(std::integral_constant<int, 2>{}, 0);
  else if (ns <= 4)
    gram(std::integral_constant<int, 4>{}, 0);
  else if (C == 8 || ns <= 8)
    gram(std::integral_constant<int, 8>{}, 0);
  else
    for (int r0 = 0; r0 < ns; r0 += 16) gram(std::integral_constant<int, C == 8 ? 8 : 16>{}, r0);
  for (int q0 = 0; q0 < len; q0 += QC) {
    const int qn = load(q0);
    for (int e = tid; e < kcv * QC; e += NT) {
      const int i = e / QC, q = e % QC;
      if (q >= qn) continue;
      Cx<float> a = cx<float>(0.f, 0.f), a2 = a;
      int jj = 0;
      for (; jj + 1 < k; jj += 2) {
        const SplitF x0 = chunk[jj * LDC + q], x1 = chunk[(jj + 1) * LDC + q];
        cmac(a, E[i * k + jj], cx<float>(x0.v.x + x0.v.y, x0.v.z + x0.v.w));
        cmac(a2, E[i * k + jj + 1], cx<float>(x1.v.x + x1.v.y, x1.v.z + x1.v.w));
      }
      if (jj < k) {
        const SplitF x0 = chunk[jj * LDC + q];
        cmac(a, E[i * k + jj], cx<float>(x0.v.x + x0.v.y, x0.v.z + x0.v.w));
      }
      a = a + a2;
      const int t = rank + C * i;
      const SplitF xs = chunk[t * LDC + q];
      const Cx<float> x = cx<float>(xs.v.x + xs.v.y, xs.v.z + xs.v.w);   // exact: the split parts add up to x
      const Cx<float> v = cx<float>(fmaf(-0.5f, a.x, x.x), fmaf(-0.5f, a.y, x.y));
      out[(size_t)t * len + q0 + q] = v;
      site[(size_t)t * len + q0 + q] = conj(v);
    }
  }
}

// Back-transformation x <- H_0 H_1 ... H_{nref-1} x of this block's vectors: GL lanes per
// vector, EL entries per lane, the reflectors staged from L2 in chunks of nch (even). Reflectors go in
// pairs: with c = h_q^H h_p the second product needs no pass of its own over the updated
// vector (h_q^H (x - f_p h_p) = h_q^H x - f_p c), which halves the chain of reductions.
template <class R, int NT, int C, int GL, int EL>
__device__ __forceinline__ void back_transform(const R* W, int p, int len, int nref, int kcv, unsigned rank, bool tall,
                                               int rr, const Cx<R>* Y, int ystride, const Cx<R>* tau, const Cx<R>* scl,
                                               Cx<R>* chunk, Cx<R>* cross, int nch, Cx<R>* out, Cx<R>* site) {
  const int tid = threadIdx.x, warp = tid >> 5, wl = tid & 31, lane = wl & (GL - 1);
  constexpr int NW = NT / 32, NGR = NT / GL;
  const int grp = tid / GL;
  for (int v0 = 0; v0 < kcv; v0 += NGR) {
    Cx<R> x[EL];
    const int i = v0 + grp, t = rank + C * i;
    const bool act = i < kcv;
#pragma unroll
    for (int e = 0; e < EL; ++e) {
      const int q = lane + GL * e;
      x[e] = cx<R>(act && q < p ? ldcg(W + (size_t)t * p + q) : R(0), R(0));
    }
    const bool warp_act = v0 + warp * (32 / GL) < kcv;   // uniform over the warp
    for (int hi = nref; hi > 0; hi -= nch) {
      const int lo = max(0, hi - nch), cnt = hi - lo;
      __syncthreads();
      // reflector hi - 1 - jj goes to row jj; an odd end is filled up with an identity
      for (int jj = warp; jj < ((cnt + 1) & ~1); jj += NW) {
        const int jr = hi - 1 - jj, start = tall ? jr + 1 : jr;
        const bool in = jj < cnt;
        const Cx<R> sc = in && tall ? scl[jr] : cx<R>(1, 0);
        const Cx<R>* y = Y + (size_t)max(jr, 0) * ystride;
        for (int q0 = 0; q0 < len; q0 += 128) {
          Cx<R> v[4];
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const int q = q0 + wl + 32 * e;
            v[e] = in && q > start && q < len ? ldcg(y + q) : cx<R>(0, 0);
          }
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const int q = q0 + wl + 32 * e;
            if (q < len) chunk[jj * len + q] = in && q == start ? cx<R>(1, 0) : (tall ? v[e] * sc : v[e]);
          }
        }
      }
      __syncthreads();
      for (int pr = warp; 2 * pr < cnt; pr += NW) {
        const Cx<R>*hp = chunk + 2 * pr * len, *hq = hp + len;
        Cx<R> c = cx<R>(0, 0);
        for (int q = wl; q < len; q += 32) cmac_conj(c, hq[q], hp[q]);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
          c.x += __shfl_xor_sync(0xffffffffu, c.x, o);
          c.y += __shfl_xor_sync(0xffffffffu, c.y, o);
        }
        if (wl == 0) cross[pr] = c;
      }
      __syncthreads();
      if (warp_act) {
        for (int jj = 0; jj < cnt; jj += 2) {
          const int jp = hi - 1 - jj, jq = jp - 1;
          const Cx<R>*hp = chunk + jj * len, *hq = hp + len;
          const int start = max(tall ? jq + 1 : jq, 0);
          // two sums per product: EL dependent steps would be the chain otherwise
          Cx<R> sp[2], sq[2];
          sp[0] = sp[1] = sq[0] = sq[1] = cx<R>(0, 0);
#pragma unroll
          for (int e = 0; e < EL; ++e) {
            if (GL * e + GL - 1 >= start) {   // uniform: whole rows of zeros are left out
              const int q = lane + GL * e;
              if (q < len) {
                cmac_conj(sp[e & 1], hp[q], x[e]);
                cmac_conj(sq[e & 1], hq[q], x[e]);
              }
            }
          }
          sp[0] = sp[0] + sp[1];
          sq[0] = sq[0] + sq[1];
#pragma unroll
          for (int o = GL / 2; o > 0; o >>= 1) {
            sp[0].x += __shfl_xor_sync(0xffffffffu, sp[0].x, o);
            sp[0].y += __shfl_xor_sync(0xffffffffu, sp[0].y, o);
            sq[0].x += __shfl_xor_sync(0xffffffffu, sq[0].x, o);
            sq[0].y += __shfl_xor_sync(0xffffffffu, sq[0].y, o);
          }
          const Cx<R> tp = tau[jp], tq = jq >= lo ? tau[jq] : cx<R>(0, 0), fp = tp * sp[0];
          cmsub(sq[0], fp, cross[jj >> 1]);
          const Cx<R> fq = tq * sq[0];
#pragma unroll
          for (int e = 0; e < EL; ++e)
            if (GL * e + GL - 1 >= start) {
              const int q = lane + GL * e;
              if (q < len) {
                cmsub(x[e], fp, hp[q]);
                cmsub(x[e], fq, hq[q]);
              }
            }
        }
      }
    }
    if (act) {
#pragma unroll
      for (int e = 0; e < EL; ++e) {
        const int q = lane + GL * e;
        if (q < len) {
          const int nat = tall ? (q & 1) * rr + (q >> 1) : q;
          out[(size_t)t * len + nat] = x[e];
          if (site) site[(size_t)t * len + nat] = conj(x[e]);
        }
      }
    }
  }
  __syncthreads();
}

// Site tensors of caller-owned memory (RAW) may lie on any 4-byte boundary: they are
// moved by component.
template <bool RAW, class R>
__device__ __forceinline__ Cx<R> ld_site(const Cx<R>* p) {
  if constexpr (RAW) {
    const R* q = reinterpret_cast<const R*>(p);
    return cx<R>(ldcg(q), ldcg(q + 1));
  } else {
    return ldcg(p);
  }
}
template <bool RAW, class R>
__device__ __forceinline__ void st_site(Cx<R>* p, Cx<R> v) {
  if constexpr (RAW) {
    R* q = reinterpret_cast<R*>(p);
    q[0] = v.x;
    q[1] = v.y;
  } else {
    *p = v;
  }
}

template <class R, int NT, int C, int VG, bool RAW, bool TG>
__global__ void __launch_bounds__(NT, 1) k_circuit(DevMPS m, CircDev c, int64_t g0, int64_t g1, int slot0,
                                                const double* theta, double cutoff, int max_sweeps) {
  extern __shared__ __align__(256) unsigned char smem[];
  constexpr bool kF64 = sizeof(R) == 8;
  constexpr int NW = NT / 32;
  using P = Plan<R, NT, C, VG, TG>;
  const P L(m.chi);
  const unsigned rank_c = crank<C>();
  const int blk = blockIdx.x / C, s = slot0 + blk;
  const int n = m.n, chi = m.chi, mmax = 2 * chi;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  Cx<R>* Bslot = (Cx<R>*)m.B + (size_t)s * m.slot_elems;
  double* lam = m.lam + (size_t)s * (n - 1) * chi;
  int* rank = m.rank + (size_t)s * (n + 1);
  Cx<R>* W = (Cx<R>*)m.work_M + (size_t)s * mmax * mmax;                 // unscaled M
  Cx<R>* Y = (Cx<R>*)m.work_X + (size_t)s * mmax * (mmax + 16);          // reflector vectors
  double* scratch = (double*)m.work_S + (size_t)s * 16 * chi * chi;      // chi^2 x 16 doubles:
  R* Wa = (R*)scratch;                                                   //   rows of W, twice
  R* Wb = (R*)(scratch + 2 * (size_t)chi * chi);
  Cx<R>* xout = (Cx<R>*)(scratch + 4 * (size_t)chi * chi);               //   rows of V, twice
  Cx<R>* xout2 = (Cx<R>*)(scratch + 8 * (size_t)chi * chi);

  // fixed part
  Cx<R>* Uh = (Cx<R>*)smem;                   // the gate matrix; FP32: leading parts,
  Cx<R>* Ul = (Cx<R>*)(smem + 256);           // and what they leave of the FP64 entries
  GateRec* rec = (GateRec*)(smem + 384);
  double* red = (double*)(smem + 512);        // 32 per-warp partials
  double* redc = red + 32;                    // per-block partials of the cluster (16)
  int* misc = (int*)(redc + 16);              // [0] k, [1] collapsed, [2] Jacobi caps, [3] splits
  int64_t* soff = (int64_t*)(smem + 1024);    // site offsets (128)
  int* ranks = (int*)(smem + 2048);           // bond ranks (129): every block keeps its own copy
  R* dd = (R*)(smem + P::kFixed);
  R* ee = dd + mmax;
  Cx<R>* tau = (Cx<R>*)(ee + mmax);
  Cx<R>* scl = tau + mmax;
  unsigned char* exch = smem + L.fixed;
  unsigned char* work = smem + L.fixed + L.exch;
  // exchange area, after the bidiagonalisation
  R* bn = (R*)exch;                           // TGK off-diagonals, scaled
  R* b2 = bn + 2 * mmax;
  R* sig = b2 + 2 * mmax;
  R* usig = sig + mmax;                       // the same before sorting
  double* sig2d = (double*)(((uintptr_t)(usig + mmax) + 15) & ~(uintptr_t)15);
  R* small = (R*)(sig2d + mmax);              // 256
  float* b2f = (float*)(small + 256);
  int* order = (int*)(b2f + 2 * mmax);        // 2 mmax
  int* bs = order + 2 * mmax;                 // block of each singular value: start, end
  int* be = bs + mmax;
  int* bstart = be + mmax;                    // unreduced blocks of the TGK: starts (2 mmax + 1),
  int* bpre = bstart + 2 * mmax + 1;          // values asked of the blocks before (2 mmax + 1)
  R* gscale = (R*)(((uintptr_t)(bpre + 2 * mmax + 1) + 15) & ~(uintptr_t)15);
  // columns of T: see Columns. Those in global memory lie where V comes later (12 chi^2 doubles
  // from there on; all columns of C blocks take less)
  const size_t gstride = (size_t)L.cl * P::lead(mmax);
  Columns<R> T;
  T.s = (Cx<R>*)work;
  T.g = TG ? xout + rank_c * gstride : nullptr;

  const double* th = theta + (size_t)blk * c.n_params;
  int st_max_iters = 0, st_max_rank = 1, st_bad = 0, st_nonfinite = 0, st_badarg = 0;
  if (tid == 0) misc[2] = 0;
  unsigned long long ph[8] = {0, 0, 0, 0, 0, 0, 0, 0};
  double alg_flops = 0.0, dw_acc = 0.0;
  long long t_mark = clock64();
#define PHASE(i)                                    \
  do {                                              \
    if (tid == 0) {                                 \
      const long long now_ = clock64();             \
      ph[i] += (unsigned long long)(now_ - t_mark); \
      t_mark = now_;                                \
    }                                               \
  } while (0)

  const int64_t g_first = c.start_gate ? max(g0, c.start_gate[blk]) : g0;
  const int64_t g_shift = c.shift_gate ? c.shift_gate[blk] : -1;
  const double phi_shift = c.shift_phi ? c.shift_phi[blk] : 0.0;
  for (int i = tid; i <= n; i += NT) ranks[i] = ldcg(rank + i);
  for (int i = tid; i < n; i += NT) soff[i] = m.site_off[i];
  // gate g by 16 lanes: fixed, or mats[m1] . Rz(phi) on one site . mats[m0]. Done for gate
  // g + 1 by a warp that idles while the twisted factorisations of gate g run.
  auto fetch_gate = [&](int64_t g, int l) {
    GateRec gr;
    if constexpr (RAW) {
      gr.bond = c.raw_bond[g];
      gr.param = -1;
      gr.m0 = (int32_t)g;
    } else {
      gr = c.gates[g];
    }
    const int i = l >> 2, j = l & 3;
    const double* A = c.mats + 32 * (size_t)gr.m0;
    Cx<double> u;
    if (gr.param < 0) {
      u = cx<double>(A[2 * l], A[2 * l + 1]);
    } else {
      const Cx<double>* Am = (const Cx<double>*)A;
      const Cx<double>* P = (const Cx<double>*)c.mats + 16 * (size_t)gr.m1;
      const double half = 0.5 * (gr.scale * th[gr.param] + (g == g_shift ? phi_shift : 0.0));
      double sn, cs;
      sincos(half, &sn, &cs);
      u = cx(0.0, 0.0);
      for (int k = 0; k < 4; ++k) {
        const int bit = gr.rz_site == 0 ? ((k >> 1) & 1) : (k & 1);
        const Cx<double> pz = cx(cs, bit ? sn : -sn);  // Rz = diag(e^{-i phi/2}, e^{i phi/2})
        u = u + (P[i * 4 + k] * pz) * Am[k * 4 + j];
      }
    }
    const Cx<R> h = cx<R>((R)u.x, (R)u.y);
    Uh[l] = h;
    if constexpr (!kF64) Ul[l] = cx<R>((R)(u.x - (double)h.x), (R)(u.y - (double)h.y));
    if (l == 0) rec->bond = gr.bond;
  };
  if (tid < 16 && g_first < g1) fetch_gate(g_first, tid);
  csync<C>();   // every block of the cluster runs before any touches a peer's shared memory
  for (int64_t g = g_first; g < g1; ++g) {
    const int bond = rec->bond;
    if constexpr (RAW) {
      // caller-owned device arrays: the bond and the three ranks it touches must lie
      // inside the site capacities before anything is indexed (uniform over the cluster)
      bool ok = bond >= 0 && bond <= n - 2;
      if (ok) {
        const int r0 = ranks[bond], r1 = ranks[bond + 1], r2 = ranks[bond + 2];
        ok = r0 >= 1 && r0 <= bond_cap(bond - 1, n, chi) && r1 >= 1 && r1 <= bond_cap(bond, n, chi) && r2 >= 1 &&
             r2 <= bond_cap(bond + 1, n, chi);
      }
      if (!ok) {
        if (tid == 0) st_badarg = 1;
        break;
      }
    }
    const int rl = ranks[bond], rm = ranks[bond + 1], rr = ranks[bond + 2];
    const int mrows = 2 * rl, ncol = 2 * rr;
    const bool tall = mrows >= ncol;
    const int tr = tall ? mrows : ncol, tp = tall ? ncol : mrows;
    T.ld = P::lead(tr);
    T.gc = 0;
    int gc0 = 0;
    if constexpr (TG) {
      const int fit = (int)(L.work / (sizeof(Cx<R>) * T.ld)) & ~1, np = tp >> 1;
      gc0 = max(0, 2 * ((np + C - 1) / C) - fit);
      T.gc = max(0, 2 * ((np + C - 1 - (int)rank_c) / C) - fit);
    }
    Cx<R>* Bn = Bslot + soff[bond];
    Cx<R>* Bn1 = Bslot + soff[bond + 1];
    const double* laml = bond > 0 ? lam + (size_t)(bond - 1) * chi : nullptr;
    // (2) Eq. (7): M[(a,i),(j,c)] = sum_{i'j'} U[ij,i'j'] sum_b B_n[a,i',b] B_{n+1}[b,j',c];
    //     W <- M; Eq. (8): M' = lambda_{n-1}[a] M. Each block contracts the columns of T it
    //     owns into place, then applies the gate and lambda to its (a, c) quads.
    const int nq = ((tall ? rr : rl) + C - 1 - (int)rank_c) / C;   // own c (tall) or a (wide)
    if (tall)
      tile_gemm<R, NT, false>(
          mrows, 2 * nq, rm, [&](int mi, int k) { return ld_site<RAW>(Bn + mi * rm + k); },
          [&](int k, int ni) { return ld_site<RAW>(Bn1 + k * ncol + (ni & 1) * rr + rank_c + C * (ni >> 1)); },
          [&](int mi, int ni, Cx<R> v) { T.template at<TG>(ni)[mi] = v; }, exch);
    else
      tile_gemm<R, NT, false>(
          2 * nq, ncol, rm,
          [&](int mi, int k) { return ld_site<RAW>(Bn + (2 * (rank_c + C * (mi >> 1)) + (mi & 1)) * rm + k); },
          [&](int k, int ni) { return ld_site<RAW>(Bn1 + k * ncol + ni); },
          [&](int mi, int ni, Cx<R> v) { T.template at<TG>(mi)[ni] = v; }, exch);
    double fro = 0.0;
    const int qfast = tall ? rl : rr;
    for (int it = tid; it < nq * qfast; it += NT) {
      const int o = it / qfast, f = it - o * qfast;
      const int a = tall ? f : (int)rank_c + C * o, cc = tall ? (int)rank_c + C * o : f;
      // entry (i, j) of the quad
      Cx<R>* e[4];
#pragma unroll
      for (int ij = 0; ij < 4; ++ij) {
        const int i = ij >> 1, j = ij & 1;
        e[ij] = tall ? T.template at<TG>(2 * o + j) + 2 * f + i : T.template at<TG>(2 * o + i) + j * rr + f;
      }
      const Cx<R> th4[4] = {*e[0], *e[1], *e[2], *e[3]};
      const R la = laml ? (R)__ldcg(laml + a) : R(1);
      R part = 0;
#pragma unroll
      for (int ij = 0; ij < 4; ++ij) {
        Cx<R> v = cx<R>(0, 0);
        if constexpr (kF64) {
#pragma unroll
          for (int kk = 0; kk < 4; ++kk) cmac(v, Uh[ij * 4 + kk], th4[kk]);
        } else {
          // one rounding per entry, against the matrix in 48 bits
          float cr = 0.f, ci = 0.f;
#pragma unroll
          for (int kk = 0; kk < 4; ++kk) {
            const Cx<float> u = Uh[ij * 4 + kk], l = Ul[ij * 4 + kk], t = th4[kk];
            dot2_acc(u.x, t.x, v.x, cr);
            dot2_acc(-u.y, t.y, v.x, cr);
            dot2_acc(u.x, t.y, v.y, ci);
            dot2_acc(u.y, t.x, v.y, ci);
            cr = fmaf(-l.y, t.y, fmaf(l.x, t.x, cr));
            ci = fmaf(l.y, t.x, fmaf(l.x, t.y, ci));
          }
          v = cx<float>(__fadd_rn(v.x, cr), __fadd_rn(v.y, ci));
        }
        W[(size_t)(2 * a + (ij >> 1)) * ncol + (ij & 1) * rr + cc] = v;
        const Cx<R> mv = la * v;
        *e[ij] = tall ? mv : conj(mv);
        part += norm2(mv);
      }
      fro += (double)part;
    }
    for (int o = 16; o > 0; o >>= 1) fro += __shfl_xor_sync(0xffffffffu, fro, o);
    if (lane == 0) red[warp] = fro;
    __syncthreads();
    if (tid < C) {
      double t = 0.0;
      for (int w = 0; w < NW; ++w) t += red[w];
      peer<C>(redc, tid)[rank_c] = t;
    }
    csync<C>();
    double total = 0.0;
#pragma unroll
    for (int w = 0; w < C; ++w) total += redc[w];
    // a NaN or Inf in M' (from corrupted inputs) would run through every later stage:
    // the gate is skipped, the state left as it was, and the host reports the count
    if (!(total <= DBL_MAX)) {
      if (tid == 0) ++st_nonfinite;
      if (tid < 16 && g + 1 < g1) fetch_gate(g + 1, tid);
      csync<C>();
      continue;
    }
    // a norm whose square is near the largest number: the reduction works on 2^-8 M' (its
    // reflectors take up to 4 times a squared norm, and the reciprocal estimate is 0 for the two
    // highest exponents)
    const bool huge = total >= (kF64 ? 0x1p1008 : 0x1p112);
    if (huge) {
      const int rows = tall ? mrows : ncol;
      for (int it = tid; it < 2 * nq * rows; it += NT) {
        Cx<R>* e = T.template at<TG>(it / rows) + it % rows;
        *e = R(0x1p-8) * *e;
      }
      csync<C>();
    }
    PHASE(0);
    // (3) Eq. (9): bidiagonalise T = Q B P^H (B real)
    {
      Bidiag<R> b;
      b.T = T;
      b.gc0 = gc0;
      b.gstride = gstride;
      b.zrows = mmax;
      b.zp = (Cx<R>*)exch;
      b.colp = b.zp + (size_t)2 * C * VG * mmax;
      b.xs = b.colp + 2 * mmax;
      b.us = b.xs + mmax;
      b.cs = (ColState<R>*)(b.us + mmax);
      b.sc = (Cx<R>*)(b.cs + L.cl);
      b.nrmp = (R*)(b.sc + 8);
      b.dd = dd;
      b.ee = ee;
      b.tau = tau;
      b.scl = scl;
      b.Y = Y;
      b.ystride = mmax;
      bidiagonalize_cluster<R, NT, C, VG, TG>(b, tr, tp, tall, rank_c);
    }
    PHASE(1);
    // Golub-Kahan tridiagonal off-diagonal (d0, e0, d1, e1, ..., d_{p-1}), scaled by a power
    // of two so that no singular value exceeds 1. Its squares also give ||M'||^2, against
    // which the kept part is measured (the rounding of the reduction then cancels, and the
    // sum has the same order for any number of blocks).
    const int N = 2 * tp;
    if (warp == 0) {
      R top = 0;
      double sq = 0.0;
      for (int i = lane; i < N; i += 32) {
        const R left = i > 0 ? rabs((i - 1) & 1 ? ee[(i - 1) >> 1] : dd[(i - 1) >> 1]) : R(0);
        const R right = i < N - 1 ? rabs(i & 1 ? ee[i >> 1] : dd[i >> 1]) : R(0);
        top = fmax(top, left + right);
        sq = fma((double)right, (double)right, sq);
      }
      for (int o = 16; o > 0; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
      if (lane == 0) red[0] = sq;
      for (int o = 16; o > 0; o >>= 1) top = fmax(top, __shfl_xor_sync(0xffffffffu, top, o));
      if (lane == 0) {
        small[0] = top;
        misc[1] = 0;
      }
    }
    __syncthreads();
    const R smax = small[0];
    total = red[0];
    int ex = 0;
    if (smax > R(0)) frexp(smax, &ex);        // smax = f 2^ex, f in [1/2, 1)
    ex = max(min(ex, kF64 ? 1000 : 120), kF64 ? -1000 : -120);
    const R down = ldexp(R(1), -ex), back = ldexp(R(1), ex), top = smax * down;
    // split the TGK where an off-diagonal is negligible (the perturbation is below 4 eps
    // ||B||): exact degeneracies, as symmetry sectors make them, live in different blocks
    for (int i = tid; i < N - 1; i += NT) {
      R v = ((i & 1) ? ee[i >> 1] : dd[i >> 1]) * down;
      if (rabs(v) <= R(4) * Eps<R>::v * top) v = R(0);
      bn[i] = v;
      b2[i] = v * v;
      if constexpr (kF64) b2f[i] = rabs(v) <= R(4) * (R)Eps<float>::v * top ? 0.f : (float)(v * v);   // FP32 range and resolution
    }
    if (tid == 0) {
      bn[N - 1] = R(0);
      b2[N - 1] = R(0);
      if constexpr (kF64) b2f[N - 1] = 0.f;
    }
    __syncthreads();
    const float* bf = kF64 ? b2f : (const float*)b2;
    const float topf = fminf((float)top * 1.001f, 1.01f);
    // sigma_0 >= top / 2, so values below this are dropped whatever they are exactly
    const float floor_f = 0.25f * (float)cutoff * (float)top;
    const int kk = min(chi, tp);
    int passes = 0;
    // Blocks, and how many of its values each has to give. A block of m indices has
    // floor(m / 2) positive values. If all blocks together have more than kk, those below
    // a bound under the kk-th value of the whole (with a margin far above rounding) are
    // left out. Every value is then asked of one block, so no two vectors can coincide.
    if (warp == 0) {
      int nb = 0;
      for (int i0 = 0; i0 < N; i0 += 32) {
        const int i = i0 + lane;
        const bool end = i < N && b2[i] == R(0);
        const unsigned mk = __ballot_sync(0xffffffffu, end);
        if (end) bstart[nb + 1 + __popc(mk & ((1u << lane) - 1u))] = i + 1;
        nb += __popc(mk);
      }
      float cut_at = 0.f;
      if (nb > 1) {
        int have = 0;
        __syncwarp();
        for (int i = lane; i < nb; i += 32) have += (bstart[i + 1] - (i ? bstart[i] : 0)) >> 1;
        for (int o = 16; o > 0; o >>= 1) have += __shfl_xor_sync(0xffffffffu, have, o);
        if (have > kk) {
          float a, b;
          half_bisect(bf, 0, N, kk - 1, true, topf, floor_f, 3, &a, &b);   // to 1 %: a bound is all it is for
          // values near the FP32 resolution are all asked for
          cut_at = a > 1e-5f * topf ? a * (1.0f - 1e-4f) : 0.f;
        }
      }
      if (lane == 0) {
        bstart[0] = 0;
        misc[3] = nb;
        small[1] = (R)cut_at;
      }
    }
    __syncthreads();
    const int nb = misc[3];
    {
      const float cut_at = (float)small[1];
      for (int i = tid; i < nb; i += NT) {
        const int s = bstart[i], e = bstart[i + 1];
        int cnt = nb == 1 ? kk : (e - s) >> 1;
        if (cut_at > 0.f && cnt > 0) cnt = min(cnt, sturm_ge1<float>(bf, s, e, cut_at));
        bpre[i + 1] = cnt;
      }
    }
    __syncthreads();
    if (warp == 0) {
      int base = 0;
      for (int i0 = 0; i0 < nb; i0 += 32) {
        const int i = i0 + lane;
        int v = i < nb ? bpre[i + 1] : 0;
        for (int o = 1; o < 32; o <<= 1) {
          const int y = __shfl_up_sync(0xffffffffu, v, o);
          if (lane >= o) v += y;
        }
        __syncwarp();
        if (i < nb) bpre[i + 1] = base + v;
        base += __shfl_sync(0xffffffffu, v, 31);
      }
      if (lane == 0) bpre[0] = 0;
    }
    __syncthreads();
    // value u (in block order) is the (u - bpre[block])-th of its block; this block of the
    // cluster finds u = rank + C i
    const int nval = bpre[nb], kco = (nval + C - 1 - (int)rank_c) / C;
    auto block_of = [&](int u) {
      int a = 0, b = nb;
      while (b - a > 1) {
        const int mid = (a + b) >> 1;
        if (bpre[mid] <= u) a = mid; else b = mid;
      }
      return a;
    };
    for (int i0 = 2 * warp; i0 < kco; i0 += 2 * NW) {
      const int i = i0 + lane / kBisectLanes;
      const bool act = i < kco;
      const int u = rank_c + C * (act ? i : i0), ib = block_of(u);
      float a, b;
      passes = max(passes, half_bisect(bf, bstart[ib], bstart[ib + 1], u - bpre[ib], act, topf, floor_f, 12, &a, &b));
      const int hl = lane & (kBisectLanes - 1);
      if constexpr (kF64) {
        // the bracket for the FP64 passes
        if (act && hl == 0) sig2d[i] = __hiloint2double(__float_as_int(b), __float_as_int(a));
      } else if (act && hl < C) {
        peer<C>(usig, hl)[u] = 0.5f * (a + b);
      }
    }
    if constexpr (kF64) {
      __syncthreads();
      for (int i0 = warp * 8; i0 < kco; i0 += NW * 8) {
        const int i = i0 + lane / 4;
        const bool act = i < kco;
        const int u = rank_c + C * (act ? i : i0), ib = block_of(u);
        const double pk = sig2d[act ? i : i0];
        double a, b;
        passes += lanes_bisect(b2, bstart[ib], bstart[ib + 1], u - bpre[ib], act, (double)top * 1.001, 0.25 * cutoff * (double)top,
                               __int_as_float(__double2loint(pk)), __int_as_float(__double2hiint(pk)), &a, &b);
        if (act)
          for (int cb = lane & 3; cb < C; cb += 4) peer<C>(usig, cb)[u] = 0.5 * (a + b);
      }
    }
    csync<C>();
    // descending order over all blocks
    for (int u = tid; u < nval; u += NT) {
      const R x = usig[u];
      int r = u;
      if (nb > 1) {
        r = 0;
        for (int w = 0; w < nval; ++w) {
          const R y = usig[w];
          r += (y > x) || (y == x && w < u);
        }
      }
      if (r < kk) {
        const int ib = block_of(u);
        sig[r] = x;
        bs[r] = bstart[ib];
        be[r] = bstart[ib + 1];
      }
    }
    __syncthreads();
    const int nsig = min(kk, nval);
    if (warp == 0) {
      // sig is descending: k = number of leading values above cutoff * sig_0
      const R s0 = nsig > 0 ? sig[0] : R(0), cut = (R)cutoff * s0;
      int cntk = 0;
      for (int t = lane; t < nsig; t += 32) cntk += (sig[t] > cut && sig[t] > R(0));
      for (int o = 16; o > 0; o >>= 1) cntk += __shfl_xor_sync(0xffffffffu, cntk, o);
      if (lane == 0) {
        misc[0] = cntk > 0 ? cntk : 1;
        if (nsig == 0) {   // M' = 0
          sig[0] = R(0);
          bs[0] = 0;
          be[0] = N;
        }
      }
    }
    __syncthreads();
    int k = misc[0];
    if (tid == 0) st_max_iters = max(st_max_iters, passes);
    PHASE(2);

    // (4) singular vectors of B from twisted factorisations of TGK - sigma. Leading minors
    // p_i from both ends by the division-free recurrence (one lane per vector and end: the
    // only serial chain, one multiply-add a step); the pivots' reciprocals p_{i-1} / p_i,
    // the twist where |gamma| is smallest and the ratios of neighbouring entries by whole
    // warps; then the running products of the ratios outward from the twist.
    int kcv = (k + C - 1 - (int)rank_c) / C;   // own vectors t = rank_c + C i
    {
      constexpr int STEP = SturmGroup<R>::v;
      const R big = kF64 ? R(1e300) : R(1e30);
      const int odd = tall ? 0 : 1;
      R* F = (R*)work;                       // [nv][2][N]: minors, then reciprocal pivots, ratios, entries
      const int ns = N / STEP + 1;
      R* S = gscale;                         // [kcv][2][ns]: scale of each group of steps
      int* rng = order;                      // [kcv][3]: block start, end, twist
      if (warp == NW - 1 && lane < 16 && g + 1 < g1) fetch_gate(g + 1, lane);
      const int v = tid >> 1, dir = tid & 1;
      // vectors v0 .. v0 + nv of the block at a time (all at once, but for large bonds in few blocks)
      for (int v0 = 0; v0 < (TG ? kcv : 1); v0 += TG ? L.vb : 1) {
        const int nv = TG ? min(kcv - v0, L.vb) : kcv;
        const bool act = v < nv;
        int s0 = 0, e0 = N;
        if (act) {
          const int t = rank_c + C * (v0 + v);
          const R x = sig[t];
          s0 = bs[t];
          e0 = be[t];
          if (dir == 0) {
            rng[3 * v] = s0;
            rng[3 * v + 1] = e0;
          }
          // entry q of the walk is index i0 + st q; its off-diagonal is b2[i0 + st q + bo]
          const int st = dir ? -1 : 1, i0 = dir ? e0 - 1 : s0, bo = dir ? 0 : -1, len = e0 - s0;
          R* f = F + (size_t)(2 * v + dir) * N;
          R* sg = S + (size_t)(2 * v + dir) * ns;
          R prev = R(1), cur = -x;
          f[i0] = cur;
          int q = 1, gi = 0;
          for (; q + STEP <= len; q += STEP) {
            R bb[STEP], o[STEP];
#pragma unroll
            for (int u = 0; u < STEP; ++u) bb[u] = b2[i0 + st * (q + u) + bo];
#pragma unroll
            for (int u = 0; u < STEP; ++u) {
              const R nxt = fma(-x, cur, -(bb[u] * prev));
              prev = cur;
              cur = nxt;
              o[u] = cur;
            }
            const R sc = rescale_factor(prev, cur);
            prev *= sc;
            cur *= sc;
            o[STEP - 1] = cur;   // the last of a group is kept scaled; the group's scale beside it
#pragma unroll
            for (int u = 0; u < STEP; ++u) f[i0 + st * (q + u)] = o[u];
            sg[gi++] = sc;
          }
          for (; q < len; ++q) {
            const R nxt = fma(-x, cur, -(b2[i0 + st * q + bo] * prev));
            prev = cur;
            cur = nxt;
            f[i0 + st * q] = cur;
          }
        }
        __syncthreads();
        for (int w = warp; w < nv; w += NW) {
          const int ws = rng[3 * w], we = rng[3 * w + 1];
          R* fu = F + (size_t)2 * w * N;
          R* fd = fu + N;
          // reciprocal pivots in place, walking against the recurrence so that the minor
          // before is still there: entry q needs entries q and q - 1 of its walk
          const int len = we - ws;
          for (int hi_q = len; hi_q > 0; hi_q -= 32) {
            const int q = hi_q - 1 - lane;
            R r0 = 0, r1 = 0;
            if (q >= 0) {
#pragma unroll
              for (int d = 0; d < 2; ++d) {
                const R* f = d ? fd : fu;
                const R* sg = S + (size_t)(2 * w + d) * ns;
                const int at = d ? we - 1 - q : ws + q, pv = d ? at + 1 : at - 1;
                R num = q > 0 ? f[pv] : R(1);
                // q closes group (q - 1) / STEP when q = STEP, 2 STEP, ..., if that group was whole
                if (q > 0 && q % STEP == 0) num *= sg[q / STEP - 1];
                const R den = f[at];
                R r = num * inverse(den);
                if (!(rabs(r) <= big)) r = -big;   // a zero pivot counts as a tiny negative one
                (d ? r1 : r0) = r;
              }
            }
            __syncwarp();
            if (q >= 0) {
              fu[ws + q] = r0;
              fd[we - 1 - q] = r1;
            }
            __syncwarp();
          }
          const R lw = sig[rank_c + C * (v0 + w)];
          R best = big;
          int at = we - 1;
          for (int i = ws + lane; i < we; i += 32) {
            // gamma_i = -lam - b_{i-1}^2 / dp_{i-1} - b_i^2 / dm_{i+1}
            R gm = -lw;
            if (i > ws) gm = fma(-b2[i - 1], fu[i - 1], gm);
            if (i < we - 1) gm = fma(-b2[i], fd[i + 1], gm);
            gm = rabs(gm);
            if (gm < best) {
              best = gm;
              at = i;
            }
          }
          for (int o = 16; o > 0; o >>= 1) {
            const R ob = __shfl_xor_sync(0xffffffffu, best, o);
            const int oa = __shfl_xor_sync(0xffffffffu, at, o);
            if (ob < best || (ob == best && oa < at)) {
              best = ob;
              at = oa;
            }
          }
          if (lane == 0) rng[3 * w + 2] = at;
          // ratios z_i / z_{i+1} = -b_i / dp_i above the twist, z_i / z_{i-1} = -b_{i-1} / dm_i below
          for (int i = lane; i < N; i += 32) {
            R r = 0;
            if (i >= ws && i < at) r = -bn[i] * fu[i];
            if (i > at && i < we) r = -bn[i - 1] * fd[i];
            if (i == at) r = R(1);
            fu[i] = r;
          }
        }
        __syncthreads();
        if (act) {
          const int at = rng[3 * v + 2], st = dir ? 1 : -1, len = dir ? e0 - 1 - at : at - s0;
          R* z = F + (size_t)2 * v * N + at;
          R zv = 1;
          int q = 1;
          for (; q + 7 <= len; q += 8) {
            R r[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) r[u] = z[st * (q + u)];
#pragma unroll
            for (int u = 0; u < 8; ++u) {
              zv *= r[u];
              z[st * (q + u)] = zv;
            }
          }
          for (; q <= len; ++q) {
            zv *= z[st * q];
            z[st * q] = zv;
          }
        }
        __syncthreads();
        for (int w = warp; w < nv; w += NW) {
          const R* z = F + (size_t)2 * w * N;
          R nrm = 0;
          for (int q = lane; q < tp; q += 32) {
            const R x = z[2 * q + odd];
            nrm = fma(x, x, nrm);
          }
          for (int o = 16; o > 0; o >>= 1) nrm += __shfl_xor_sync(0xffffffffu, nrm, o);
          const R inv = nrm > R(0) ? R(1) / sqrt(nrm) : R(0);
          const int t = rank_c + C * (v0 + w);
          for (int q = lane; q < tp; q += 32) Wa[(size_t)t * tp + q] = z[2 * q + odd] * inv;
        }
        if constexpr (TG) __syncthreads();
      }
    }
    csync<C>();
    PHASE(3);
    // (4b) the rows are orthonormal to about eps / (relative gap). Newton-Schulz steps pull
    // them together without the serial chain of a Gram-Schmidt (the span, and with it
    // B_n B_{n+1}, does not change); rows too far off go through block Gram-Schmidt, and
    // a collapse there to Jacobi. FP32 stops at 1e-4: the step on the final V, which works
    // from an accurate Gram matrix, squares that away.
    R *Wc = Wa, *Wn = Wb;
    {
      R* E = (R*)work;
      R* chunk = E + (size_t)L.kc * chi;
      const float tol = kF64 ? 1e-15f : 1e-4f;
      float pred = 2.f;
      bool slow = false;   // block Gram-Schmidt has been through
      for (int it = 0; it < 10 && pred > tol; ++it) {
        const R dmax = real_defect<R, NT, C>(Wc, k, tp, kcv, rank_c, E, chunk, small);
        if (tid < C) peer<C>(redc, tid)[rank_c] = (double)dmax;
        csync<C>();
        float defect = 0.f;
#pragma unroll
        for (int w = 0; w < C; ++w) defect = fmaxf(defect, (float)redc[w]);
        R* sw = Wc;
        if (!(defect <= 0.4f)) {
          if (slow) {
            if (tid == 0) misc[1] = 1;
            break;
          }
          slow = true;
          if (rank_c == 0) {
            for (int e = tid; e < k * tp; e += NT) Wn[e] = ldcg(Wc + e);
            __syncthreads();
            orthonormalize_rows_block<R, NT>(Wn, tp, k, tp, sig, (R*)work, small, &misc[1]);
            __syncthreads();
            if (tid < C) peer<C>(misc, tid)[1] = misc[1];
          }
          Wc = Wn;
          Wn = sw;
          csync<C>();
          if (misc[1] != 0) break;
          continue;
        }
        if (!kF64 && defect <= tol) break;
        real_update<R, NT, C>(Wc, Wn, k, tp, kcv, rank_c, E, chunk);
        Wc = Wn;
        Wn = sw;
        pred = defect * defect;
        csync<C>();
      }
      __syncthreads();
      if (misc[1] != 0) {
        // degenerate without a split: Jacobi on the bidiagonal by the first block. Columns of
        // B^T (tall) or B (wide) converge to sigma_t times the wanted vector.
        if (tid == 0) ++st_bad;
        Wc = Wn;
        if (rank_c == 0) {
          const int ldx = tp + 1;
          R* X = sizeof(R) * (size_t)tp * ldx <= L.work ? (R*)work : (R*)xout;
          for (int e = tid; e < tp * tp; e += NT) {
            const int c = e / tp, q = e - c * tp;   // entry q of column c: B[c][q] or B[q][c]
            R v = q == c ? dd[c] * down : R(0);
            if (tall && q == c + 1) v = ee[c] * down;
            if (!tall && q + 1 == c) v = ee[q] * down;
            X[(size_t)c * ldx + q] = v;
          }
          __syncthreads();
          const double zero2 = (double)Eps<R>::v * Eps<R>::v * 16.0 * total * (double)down * (double)down;
          jacobi_columns<R, NT, 8>(X, ldx, tp, zero2, max_sweeps, &misc[2]);
          for (int p = tid; p < tp; p += NT) {
            double acc = 0.0;
            for (int q = 0; q < tp; ++q) acc = fma((double)X[(size_t)p * ldx + q], (double)X[(size_t)p * ldx + q], acc);
            sig2d[p] = acc;
          }
          __syncthreads();
          for (int p = tid; p < tp; p += NT) {
            const double v = sig2d[p];
            int rk = 0;
            for (int q = 0; q < tp; ++q) {
              const double w = sig2d[q];
              rk += (w > v) || (w == v && q < p);
            }
            order[rk] = p;
          }
          __syncthreads();
          if (tid == 0) {
            const double s0 = sig2d[order[0]];
            int kj = 0;
            while (kj < kk && sig2d[order[kj]] > cutoff * cutoff * s0) ++kj;
            if (kj == 0) kj = 1;
            for (int cb = 0; cb < C; ++cb) peer<C>(misc, cb)[0] = kj;
          }
          __syncthreads();
          const int kj = misc[0];
          for (int t = tid; t < kj; t += NT) {
            const R v = (R)sqrt(sig2d[order[t]]);
            for (int cb = 0; cb < C; ++cb) peer<C>(sig, cb)[t] = v;
          }
          for (int e = tid; e < kj * tp; e += NT) {
            const int t = e / tp, q = e - t * tp, p = order[t];
            // M' = 0 (a gate that annihilates the state): any unit vector is its singular vector
            Wn[e] = sig2d[p] > 0.0 ? (R)((double)X[(size_t)p * ldx + q] / sqrt(sig2d[p])) : R(q == t ? 1 : 0);
          }
        }
        csync<C>();
        k = misc[0];
        kcv = (k + C - 1 - (int)rank_c) / C;
      }
      if (tid == 0) st_max_rank = max(st_max_rank, k);
    }
    PHASE(4);
    {
      // (5) back-transformation: x_t = P w_t (tall) or Q [w_t; 0] (wide) is the right
      //     singular vector v_t of M' (length ncol)
      const int nref = tall ? tp - 1 : tp;
      const int nch = max(2, min((nref + 1) & ~1, (int)(L.work / (sizeof(Cx<R>) * ncol)) & ~1));
      Cx<R>* site = kF64 ? Bn1 : nullptr;
      Cx<R>* cross = (Cx<R>*)sig2d;
      // half a warp a vector: fewer slots go to reductions than with a whole one, and two
      // vectors share the loads
      auto go = [&](auto el) {
        constexpr int EL = decltype(el)::value;
        back_transform<R, NT, C, 16, EL>(Wc, tp, ncol, nref, kcv, rank_c, tall, rr, Y, mmax, tau, scl, (Cx<R>*)work,
                                         cross, nch, xout, site);
      };
      if (ncol <= 32)
        go(std::integral_constant<int, 2>{});
      else if (ncol <= 64)
        go(std::integral_constant<int, 4>{});
      else if (ncol <= 128)
        go(std::integral_constant<int, 8>{});
      else if (C < 8 && ncol <= 160)   // one block, chi = 65: 166 k cycles a gate instead of 180 k
        go(std::integral_constant<int, C < 8 ? 10 : 16>{});
      else
        go(std::integral_constant<int, 16>{});
      if (rank_c == 0 && warp == 0) {
        double kept = 0.0;
        const double bk = (double)back;
        for (int t = lane; t < k; t += 32) kept += ((double)sig[t] * bk) * ((double)sig[t] * bk);
        for (int o = 16; o > 0; o >>= 1) kept += __shfl_xor_sync(0xffffffffu, kept, o);
        if (lane == 0 && total > 0.0) dw_acc += fmax(0.0, total - kept) / total;
        for (int t = lane; t < k; t += 32) lam[(size_t)bond * chi + t] = (double)(sig[t] * back) * (huge ? 256.0 : 1.0);
      }
    }
    csync<C>();
    Cx<R>* xv = xout;
    if constexpr (!kF64) {
      // (5b) mixed precision: over a long circuit the orthonormality defect of the FP32
      //      back-transformation, not the rounding of the stored tensors, dominates the
      //      energy error; one Newton-Schulz step brings it down to the storage rounding
      Cx<float>* E = (Cx<float>*)work;
      SplitF* chunk = (SplitF*)(E + ((size_t)L.kc * chi + 1) / 2 * 2);
      if constexpr (RAW) {
        newton_schulz_cluster<NT, C>(xout, k, ncol, kcv, rank_c, E, chunk, xout2, xout2);
        __syncthreads();
        // the caller's tensors take V by component; xout2 then holds conj(V) rows
        for (int i = 0; i < kcv; ++i) {
          const int t = rank_c + C * i;
          for (int q = tid; q < ncol; q += NT) {
            const Cx<R> v = xout2[(size_t)t * ncol + q];
            st_site<true>(Bn1 + (size_t)t * ncol + q, v);
            xout2[(size_t)t * ncol + q] = conj(v);
          }
        }
      } else {
        newton_schulz_cluster<NT, C>(xout, k, ncol, kcv, rank_c, E, chunk, xout2, Bn1);
      }
      xv = xout2;
      csync<C>();
    }
    PHASE(5);
    // (6) Eq. (10): B_{n+1} <- V (row t = v_t^H, written above), B_n <- M V^H (column t =
    //     M v_t), lambda_n <- sigma
    {
      const int mper = (mrows + C - 1) / C, m0 = min(mrows, mper * (int)rank_c), mn = min(mper, mrows - m0);
      tile_gemm<R, NT, true>(
          mn, k, ncol, [&](int mi, int q) { return ldcg(W + (m0 + mi) * ncol + q); },
          [&](int q, int t) { return ldcg(xv + t * ncol + q); },
          [&](int mi, int t, Cx<R> v) { st_site<RAW>(Bn + (m0 + mi) * k + t, v); }, work);
    }
    if (tid == 0) {
      ranks[bond + 1] = k;
      if (rank_c == 0) rank[bond + 1] = k;
    }
    csync<C>();
    PHASE(6);
    if (tid == 0) alg_flops += flops_per_gate(rl, rm, rr, k);
  }
#undef PHASE
  if (rank_c == 0 && tid == 0) {
    for (int i = 0; i < 7; ++i) m.prof[s * 8 + i] += ph[i];
    m.prof[s * 8 + 7] = __double_as_longlong(__longlong_as_double(m.prof[s * 8 + 7]) + alg_flops);
    m.dw[s] += dw_acc;
    int* stt = m.stat + s * kStatWords;
    stt[0] = max(stt[0], st_max_iters);
    stt[1] += misc[2];
    stt[3] += st_bad;
    stt[2] = max(stt[2], st_max_rank);
    stt[4] += st_nonfinite;
    stt[5] |= st_badarg;
  }
  csync<C>();   // no block leaves while a peer may still reach its shared memory
}

}  // namespace gate

// One translation unit instantiates each (they compile side by side): see gate_*.cu.
template <class R, int NT, int C, int VG, bool RAW, bool TG>
static cudaError_t cluster_config(int chi, cudaLaunchConfig_t* cfg, cudaLaunchAttribute* at) {
  const gate::Plan<R, NT, C, VG, TG> L(chi);
  if (L.total > L.kCap) return cudaErrorInvalidValue;
  *cfg = cudaLaunchConfig_t{};
  cfg->blockDim = dim3(NT);
  cfg->dynamicSmemBytes = L.total;
  at->id = cudaLaunchAttributeClusterDimension;
  at->val.clusterDim.x = C;
  at->val.clusterDim.y = 1;
  at->val.clusterDim.z = 1;
  cfg->attrs = at;
  cfg->numAttrs = C > 1 ? 1 : 0;
  return gate::raise_smem_limit<gate::k_circuit<R, NT, C, VG, RAW, TG>>();
}

template <class R, int NT, int C, int VG, bool RAW, bool TG>
cudaError_t launch_cluster(const DevMPS& m, const CircDev& c, int64_t g0, int64_t g1, int slot0, int count,
                           const double* theta, double cutoff, int max_sweeps, cudaStream_t st) {
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute at[1];
  cudaError_t e = cluster_config<R, NT, C, VG, RAW, TG>(m.chi, &cfg, at);
  if (e != cudaSuccess) return e;
  cfg.gridDim = dim3((unsigned)(count * C));
  cfg.stream = st;
  return cudaLaunchKernelEx(&cfg, gate::k_circuit<R, NT, C, VG, RAW, TG>, m, c, g0, g1, slot0, theta, cutoff, max_sweeps);
}

// 0 where the bond cap does not fit. The registers of one block fill an SM, so else the answer
// does not depend on chi and is asked for once per device; 0 too (then other instances are
// taken) where it cannot be had.
template <class R, int NT, int C, int VG, bool RAW, bool TG>
int max_clusters(int chi) {
  static std::atomic<int> known[64];
  int dev = 0;
  if (gate::Plan<R, NT, C, VG, TG>(chi).total > gate::Plan<R, NT, C, VG, TG>::kCap) return 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
  int n = known[dev].load();
  if (C == 1 && n == 0) {
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 0;
    known[dev].store(n);
  }
  if (n == 0) {
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute at[1];
    if (cluster_config<R, NT, C, VG, RAW, TG>(chi, &cfg, at) != cudaSuccess) return 0;
    cfg.gridDim = dim3(C);
    if (cudaOccupancyMaxActiveClusters(&n, gate::k_circuit<R, NT, C, VG, RAW, TG>, &cfg) != cudaSuccess) return 0;
    known[dev].store(n);
  }
  return n;
}

}  // namespace mpsvqe
