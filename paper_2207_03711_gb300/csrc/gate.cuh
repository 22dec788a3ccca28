// Device code of the gate engine: one two-site gate (Eqs. 7-10) by a thread-block cluster
// of C blocks (C = 1: one block). See gate.cu for the kernel that strings these together.
//
// M' (tall orientation: T = M' or M'^H, tr x tp, tr >= tp) is spread over the cluster by
// columns: column q belongs to block (q / 2) mod C and stays in that block's shared memory
// at local index 2 ((q / 2) / C) + (q & 1). Columns leave the bidiagonalisation in order of
// q, so the cyclic spread keeps the blocks evenly loaded to the end.
//
// Order of the columns q: tall (T = M'): q = 2 c + j for column j r_r + c of M', tall rows
// = rows of M'; wide (T = M'^H): q = row of M' (2 a + i), rows = columns of M'. Either way
// the four entries of one (a, c) quad lie in one block, which applies the 4 x 4 gate there.
#pragma once
#include <cooperative_groups.h>

#include <cfloat>
#include <cmath>
#include <cstdint>

#include "cx.cuh"
#include "kernels.cuh"
#include "svd.cuh"

namespace mpsvqe {
namespace gate {

namespace cg = cooperative_groups;

// ------------------------------------------------------------------ cluster primitives
template <int C>
__device__ __forceinline__ void csync() {
  if constexpr (C == 1) {
    __syncthreads();
  } else {
    // release / acquire at cluster scope: covers shared and global memory of the blocks
    asm volatile("barrier.cluster.arrive.release.aligned;\n barrier.cluster.wait.acquire.aligned;" ::: "memory");
  }
}

template <int C>
__device__ __forceinline__ unsigned crank() {
  if constexpr (C == 1) return 0;
  unsigned r;
  asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}

// The same shared-memory variable of block `rank` of the cluster.
template <int C, class T>
__device__ __forceinline__ T* peer(T* p, unsigned rank) {
  if constexpr (C == 1) {
    return p;
  } else {
    return cg::this_cluster().map_shared_rank(p, rank);
  }
}

// Data that other blocks of the cluster wrote to global memory is read past L1.
__device__ __forceinline__ Cx<float> ldcg(const Cx<float>* p) {
  const float2 v = __ldcg(reinterpret_cast<const float2*>(p));
  return cx<float>(v.x, v.y);
}
__device__ __forceinline__ Cx<double> ldcg(const Cx<double>* p) {
  const double2 v = __ldcg(reinterpret_cast<const double2*>(p));
  return cx<double>(v.x, v.y);
}
__device__ __forceinline__ float ldcg(const float* p) { return __ldcg(p); }
__device__ __forceinline__ double ldcg(const double* p) { return __ldcg(p); }
__device__ __forceinline__ int ldcg(const int* p) { return __ldcg(p); }

// ------------------------------------------------------------------------- tiled GEMM
// out(m, n) = sum_k a(m, k) b(k, n) for m < M, n < N by one block: NT / 16 rows x 64
// columns per tile, 32-deep K tiles in shared memory, four columns per thread. The
// operands come from L2 through functors, so orientation, conjugation and the cyclic
// column spread cost nothing extra. As: (NT / 16) x 33, Bs: 32 x 65.
template <class R, int NT>
struct GemmTiles {
  static constexpr int TM = NT / 16, KT = 32;
  static constexpr size_t bytes = sizeof(Cx<R>) * (TM * (KT + 1) + KT * 65);
};

template <class R, int NT, class FA, class FB, class FC>
__device__ __forceinline__ void tile_gemm(int M, int N, int K, FA fa, FB fb, FC fc, unsigned char* smem) {
  constexpr int TM = GemmTiles<R, NT>::TM, KT = GemmTiles<R, NT>::KT;
  Cx<R>(*As)[KT + 1] = reinterpret_cast<Cx<R>(*)[KT + 1]>(smem);
  Cx<R>(*Bs)[65] = reinterpret_cast<Cx<R>(*)[65]>(smem + sizeof(Cx<R>) * TM * (KT + 1));
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  for (int m0 = 0; m0 < M; m0 += TM)
    for (int n0 = 0; n0 < N; n0 += 64) {
      Cx<R> acc[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) acc[j] = cx<R>(0, 0);
      const int jn = (min(64, N - n0) + 15) >> 4;
      for (int k0 = 0; k0 < K; k0 += KT) {
        const int kt = min(KT, K - k0);
        __syncthreads();
        for (int e = tid; e < TM * KT; e += NT) {
          const int r = e / KT, kk = e % KT;
          As[r][kk] = (m0 + r < M && kk < kt) ? fa(m0 + r, k0 + kk) : cx<R>(0, 0);
        }
        for (int e = tid; e < KT * 64; e += NT) {
          const int kk = fb.k_fast ? e % KT : e >> 6, n = fb.k_fast ? e / KT : e & 63;
          Bs[kk][n] = (n0 + n < N && kk < kt) ? fb(k0 + kk, n0 + n) : cx<R>(0, 0);
        }
        __syncthreads();
        if (m0 + ty < M) {
          if (jn == 4) {
#pragma unroll 8
            for (int kk = 0; kk < kt; ++kk) {
              const Cx<R> a = As[ty][kk];
#pragma unroll
              for (int j = 0; j < 4; ++j) cmac(acc[j], a, Bs[kk][tx + 16 * j]);
            }
          } else {
            for (int kk = 0; kk < kt; ++kk) {
              const Cx<R> a = As[ty][kk];
#pragma unroll
              for (int j = 0; j < 4; ++j)
                if (j < jn) cmac(acc[j], a, Bs[kk][tx + 16 * j]);
            }
          }
        }
      }
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if (m0 + ty < M && n0 + tx + 16 * j < N) fc(m0 + ty, n0 + tx + 16 * j, acc[j]);
    }
  __syncthreads();
}

// -------------------------------------------------------------------- bidiagonalisation
// T = Q B P^H (LAPACK reflector conventions, svd.cuh) with a single cluster barrier per
// step: the updates by right reflector k-1 and left reflector k go over the trailing
// columns together, the next row comes out of that pass, and the product z with the next
// right reflector is formed from the unscaled row (its norm, hence its scale, is known one
// barrier later). Every block then forms the next column and its left reflector for itself
// from the exchanged sums, so no block waits for another inside a step. Exchanged per step:
// z partials, the next column before its right update, the partial norms of the row.
// The trailing matrix is read twice and written once per step, where two separate half
// steps read and write it twice.
template <class R>
struct Bidiag {
  Cx<R>* T;            // own columns, leading dimension ld (>= r)
  int ld;
  int zrows;
  Cx<R>* zp;           // [2][C][GMAX][zrows] z partials
  Cx<R>* colp;         // [2][zrows] next column before its right update
  Cx<R>* sc;           // [2] row entry of the next column, [2]: X of the leading row, [3..6]: scalars
  R* nrmp;             // [2][C] partial |row|^2
  Cx<R>*xs, *us;       // [zrows] X conj(right scale), the column (unscaled left reflector)
  Cx<R>*rj, *fj;       // [2][own] row entries, [own] factors of the left update
  R* part;             // [24] per-warp partial sums
  R *dd, *ee;
  Cx<R>*tau, *scl;     // factor and scale per reflector of the side the back-transformation needs
  Cx<R>* Y;            // global [.][ystride]: the reflector vectors of that side
  int ystride;
};

// Smallest power of two >= rows, at least a warp.
__device__ __forceinline__ int pow2_rows(int rows) {
  return rows <= 32 ? 32 : 1 << (32 - __clz(rows - 1));
}

template <class R, int NT, int C, int GMAX>
__device__ __noinline__ void bidiagonalize_cluster(const Bidiag<R>& b, int r, int p, bool right_side, unsigned rank) {
  const int tid = threadIdx.x;
  // On this chip a SM does two FP64 operations a clock: scalar work in FP64 runs in one
  // warp and is passed on through shared memory. In FP32 every warp does it for itself,
  // which saves the barrier.
  constexpr bool kOneWarp = sizeof(R) == 8;
  constexpr int GL = 16, NG = NT / GL;   // lanes per column, columns at a time
  const int own = 2 * (((p >> 1) + C - 1 - (int)rank) / C);   // p is even: pairs are never split
  Cx<R> tauR = cx<R>(0, 0), scR = cx<R>(0, 0);
  for (int i = tid; i < 2 * own; i += NT) b.rj[i] = cx<R>(0, 0);
  for (int k = 0; k < p; ++k) {
    const int par = k & 1, rows = r - k;
    const bool have_old = k > 0;
    // ---- the next column and the right-update vector X, one thread per row
    const int rp = pow2_rows(rows);
    if (tid < rp) {
      R pn = 0;
      Cx<R> pd = cx<R>(0, 0);
      if (tid < rows) {
        Cx<R> col, X = cx<R>(0, 0);
        if (!have_old) {
          col = peer<C>(b.T, 0)[tid];
        } else {
          const int groups = min(GMAX, NT / rp);
          Cx<R> z = cx<R>(0, 0);
          const Cx<R>* zq = b.zp + (size_t)par * C * GMAX * b.zrows + tid;
#pragma unroll
          for (int c = 0; c < C; ++c) {
#pragma unroll
            for (int g = 0; g < GMAX; ++g)
              if (g < groups) z = z + zq[(c * GMAX + g) * b.zrows];
          }
          const Cx<R> a = b.colp[par * b.zrows + tid];
          X = tauR * (a + scR * z);
          col = a - X;
          b.xs[tid] = X * conj(scR);
        }
        b.us[tid] = col;
        if (tid > 0) {
          pn = norm2(col);
          cmac_conj(pd, col, X);
        } else {
          b.sc[2] = X;
        }
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        pn += __shfl_xor_sync(0xffffffffu, pn, o);
        pd.x += __shfl_xor_sync(0xffffffffu, pd.x, o);
        pd.y += __shfl_xor_sync(0xffffffffu, pd.y, o);
      }
      if ((tid & 31) == 0) {
        b.part[tid >> 5] = pn;
        b.part[8 + (tid >> 5)] = pd.x;
        b.part[16 + (tid >> 5)] = pd.y;
      }
    }
    __syncthreads();
    // ---- left reflector u = (1, col scL) of that column; g = u^H (X conj(scR))
    Cx<R> scL, ct, g;
    if (!kOneWarp || tid < 32) {
      R xn2 = 0, betaL;
      Cx<R> dot = cx<R>(0, 0), tauL;
      for (int w = 0; w < rp / 32; ++w) {
        xn2 += b.part[w];
        dot.x += b.part[8 + w];
        dot.y += b.part[16 + w];
      }
      make_reflector(b.us[0], xn2, &tauL, &betaL, &scL);
      g = have_old ? (b.sc[2] + conj(scL) * dot) * conj(scR) : cx<R>(0, 0);
      ct = conj(tauL);
      if (tid == 0) {
        b.dd[k] = betaL;
        if (!right_side) {
          b.tau[k] = tauL;
          b.scl[k] = cx<R>(1, 0);
        }
        if (kOneWarp) {
          b.sc[3] = scL;
          b.sc[4] = ct;
          b.sc[5] = g;
        }
      }
    }
    if (kOneWarp) {
      __syncthreads();
      scL = b.sc[3];
      ct = b.sc[4];
      g = b.sc[5];
    }
    if (!right_side && (k % C) == (int)rank)
      for (int i = tid; i < rows; i += NT) b.Y[(size_t)k * b.ystride + k + i] = i == 0 ? cx<R>(1, 0) : b.us[i] * scL;
    if (k + 1 >= p) break;
    // ---- pass 1: s_j = u^H a_j of the own trailing columns; then the left factor f_j and
    // the new row entry r_j, both with the pending right update taken into account
    const int l0 = 2 * ((((k + 1) >> 1) + C - 1 - (int)rank) / C);   // own pairs from column k (or k + 1) on
    const int first = 2 * (C * (l0 >> 1) + (int)rank) > k ? l0 : l0 + 1;   // own columns after k
    const int lane = tid & (GL - 1), grp = tid / GL;
    const Cx<R>* rold = b.rj + (par ^ 1) * own;
    Cx<R>* rnew = b.rj + par * own;
    auto finish = [&](int lc, Cx<R> s) {
      const Cx<R> a0 = b.T[(size_t)lc * b.ld + k];
      s = a0 + conj(scL) * s;
      Cx<R> rn = a0;
      if (have_old) {
        const Cx<R> ro = rold[lc];
        cmsub(s, g, ro);
        cmsub(rn, b.xs[0], ro);
      }
      const Cx<R> f = ct * s;
      rn = rn - f;
      b.fj[lc] = f;
      rnew[lc] = rn;
      if (right_side) b.Y[(size_t)k * b.ystride + 2 * (C * (lc >> 1) + (int)rank) + (lc & 1)] = conj(rn);
    };
    for (int base = first; base < own; base += NG) {
      const int lc = base + grp;
      const bool act = lc < own;
      Cx<R> s = cx<R>(0, 0);
      if (act) {
        const Cx<R>* a = b.T + (size_t)lc * b.ld + k;
#pragma unroll 4
        for (int i = lane == 0 ? GL : lane; i < rows; i += GL) cmac_conj(s, b.us[i], a[i]);
      }
#pragma unroll
      for (int o = 1; o < GL; o <<= 1) {
        s.x += __shfl_xor_sync(0xffffffffu, s.x, o, GL);
        s.y += __shfl_xor_sync(0xffffffffu, s.y, o, GL);
      }
      if (act && lane == 0) {
        if constexpr (kOneWarp)
          b.fj[lc] = s;
        else
          finish(lc, s);
      }
    }
    __syncthreads();
    if constexpr (kOneWarp) {
      for (int lc = first + tid; lc < own; lc += NT) finish(lc, b.fj[lc]);
      __syncthreads();
    }
    // ---- pass 2: both updates, one thread per row and column group; z = sum a_j conj(r_j)
    // over the columns after k + 1; column k + 1 goes out whole
    const int nrow = rows - 1, rp2 = pow2_rows(nrow), groups = min(GMAX, NT / rp2);
    const int row = tid & (rp2 - 1), cgp = tid / rp2, npar = par ^ 1;
    const int lnext = ((k + 1) >> 1) % C == (int)rank ? 2 * (((k + 1) >> 1) / C) + ((k + 1) & 1) : -1;
    if (cgp < groups && row < nrow) {
      Cx<R> z = cx<R>(0, 0);
      const Cx<R> u = b.us[row + 1] * scL;
      const Cx<R> x = have_old ? b.xs[row + 1] : cx<R>(0, 0);
      int lc = first + cgp;
      Cx<R>* a = b.T + (size_t)lc * b.ld + k + 1 + row;
      if (lc == lnext) {   // first own column: only group 0 can meet it
        Cx<R> v = *a;
        cmsub(v, x, rold[lc]);
        cmsub(v, b.fj[lc], u);
#pragma unroll
        for (int c = 0; c < C; ++c) peer<C>(b.colp, c)[npar * b.zrows + row] = v;
        lc += groups;
        a += (size_t)groups * b.ld;
      }
#pragma unroll 2
      for (; lc < own; lc += groups, a += (size_t)groups * b.ld) {
        Cx<R> v = *a;
        cmsub(v, x, rold[lc]);
        cmsub(v, b.fj[lc], u);
        *a = v;
        cmac_bconj(z, v, rnew[lc]);
      }
#pragma unroll
      for (int c = 0; c < C; ++c)
        peer<C>(b.zp, c)[(size_t)((npar * C + (int)rank) * GMAX + cgp) * b.zrows + row] = z;
    }
    // partial norm of the new row (columns after k + 1) and its leading entry
    if (tid >= NT - 32) {
      const int l = tid & 31;
      R nn = 0;
      for (int lc = first + l; lc < own; lc += 32)
        if (lc != lnext) nn += norm2(rnew[lc]);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) nn += __shfl_xor_sync(0xffffffffu, nn, o);
      if (l < C) {
        peer<C>(b.nrmp, l)[npar * C + (int)rank] = nn;
        if (lnext >= 0) peer<C>(b.sc, l)[npar] = rnew[lnext];
      }
    }
    csync<C>();
    // ---- right reflector of the new row
    if (!kOneWarp || tid < 32) {
      R rn2 = 0, betaR;
#pragma unroll
      for (int c = 0; c < C; ++c) rn2 += b.nrmp[npar * C + c];
      make_reflector(conj(b.sc[npar]), rn2, &tauR, &betaR, &scR);
      if (tid == 0) {
        b.ee[k] = betaR;
        if (right_side) {
          b.tau[k] = tauR;
          b.scl[k] = scR;
        }
        if (kOneWarp) {
          b.sc[6] = tauR;
          b.sc[7] = scR;
        }
      }
    }
    if (kOneWarp) {
      __syncthreads();
      tauR = b.sc[6];
      scR = b.sc[7];
    }
  }
  csync<C>();
}

// ---------------------------------------------------------------------- Sturm counts
// Sign changes of the leading principal minors p_i of TGK - x I over indices [s, e):
// p_{i+1} = -x p_i - b_i^2 p_{i-1}. The three-term recurrence needs no division (a FP64
// division costs ~10 DFMA, and its latency was the chain of the earlier quotient form);
// the pair is rescaled by a power of two every few steps, so that nothing leaves the
// range: entries are scaled to |b| <= 1 and split off below 4 eps, so two steps shrink
// the larger of a pair by at most (4 eps)^2. An exact zero counts once either way, because
// its neighbours have opposite signs. Returns the number of eigenvalues >= x.
template <class R>
__device__ __forceinline__ int sturm_ge(const R* b2, int s, int e, R x);

template <>
__device__ __forceinline__ int sturm_ge<float>(const float* b2, int s, int e, float x) {
  float prev = 1.f, cur = -x;
  unsigned neg = __float_as_uint(cur) >> 31;
  int i = s + 1;
#pragma unroll 2
  for (; i + 3 < e; i += 4) {
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const float nxt = fmaf(-x, cur, -(b2[i + u - 1] * prev));
      neg += (__float_as_uint(nxt) ^ __float_as_uint(cur)) >> 31;
      prev = cur;
      cur = nxt;
    }
    const unsigned m = max((__float_as_uint(prev) >> 23) & 255u, (__float_as_uint(cur) >> 23) & 255u);
    const float sc = __uint_as_float((254u - min(m, 253u)) << 23);
    prev *= sc;
    cur *= sc;
  }
  for (; i < e; ++i) {
    const float nxt = fmaf(-x, cur, -(b2[i - 1] * prev));
    neg += (__float_as_uint(nxt) ^ __float_as_uint(cur)) >> 31;
    prev = cur;
    cur = nxt;
  }
  return (e - s) - (int)neg;
}

template <>
__device__ __forceinline__ int sturm_ge<double>(const double* b2, int s, int e, double x) {
  double prev = 1.0, cur = -x;
  unsigned neg = (unsigned)__double2hiint(cur) >> 31;
  int i = s + 1;
  for (; i + 7 < e; i += 8) {
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const double nxt = fma(-x, cur, -(b2[i + u - 1] * prev));
      neg += (unsigned)(__double2hiint(nxt) ^ __double2hiint(cur)) >> 31;
      prev = cur;
      cur = nxt;
    }
    const unsigned m = max(((unsigned)__double2hiint(prev) >> 20) & 2047u, ((unsigned)__double2hiint(cur) >> 20) & 2047u);
    const double sc = __hiloint2double((int)((2046u - min(m, 2045u)) << 20), 0);
    prev *= sc;
    cur *= sc;
  }
  for (; i < e; ++i) {
    const double nxt = fma(-x, cur, -(b2[i - 1] * prev));
    neg += (unsigned)(__double2hiint(nxt) ^ __double2hiint(cur)) >> 31;
    prev = cur;
    cur = nxt;
  }
  return (e - s) - (int)neg;
}

// Singular value t (0-based, descending) in FP32 by one warp: 32 shifts per pass, each
// pass narrows the bracket 33-fold. First pass on a log grid over eight decades, then
// linear to the working precision. lo/hi bracket the value (scaled to smax ~ 1).
__device__ __forceinline__ int warp_bisect(const float* b2, int N, int t, float top, float* lo_out, float* hi_out) {
  const int lane = threadIdx.x & 31;
  float lo = 0.f, hi = top;
  int passes = 0;
  for (int it = 0; it < 9; ++it) {
    float x;
    if (it == 0) {
      x = top * exp10f(-8.0f * (float)(32 - lane) / 32.0f);
    } else {
      x = fmaf(hi - lo, (float)(lane + 1) / 33.0f, lo);
    }
    const unsigned ge = __ballot_sync(0xffffffffu, sturm_ge<float>(b2, 0, N, x) >= t + 1);
    // counts fall with x: the number of shifts below the value locates it
    const int m = __popc(ge);
    const float nlo = __shfl_sync(0xffffffffu, x, max(m - 1, 0)), nhi = __shfl_sync(0xffffffffu, x, min(m, 31));
    if (m > 0) lo = nlo;
    if (m < 32) hi = nhi;
    ++passes;
    if (hi - lo <= 1.2e-7f * hi) break;   // the bracket is two neighbours of the working precision
  }
  *lo_out = lo;
  *hi_out = hi;
  return passes;
}

// The same in FP64 from the FP32 bracket: LT lanes per value (LT = 4: on this chip FP64
// runs at two lanes a clock per SM, and few shifts per pass cost the least per bit), the
// bracket first checked with FP64 counts and opened up if it does not hold. Stops at the
// working precision relative to the value, or at 2^-60 of the largest one.
template <int LT>
__device__ __forceinline__ int lanes_bisect(const double* b2, int N, int t, bool act, double top, float lo_f,
                                            float hi_f, double* lo_out, double* hi_out) {
  const int lane = threadIdx.x & (LT - 1);
  double lo = (double)lo_f * (1.0 - 4e-6), hi = fmin(top, (double)hi_f * (1.0 + 4e-6) + 1e-30);
  bool done = !act;
  int passes = 0;
  for (int it = 0; it < 64; ++it) {
    // pass 0 checks the bracket: lane 0 its lower end, the last lane its upper end
    double x;
    if (it == 0)
      x = lane == 0 ? lo : hi;
    else
      x = fma(hi - lo, (double)(lane + 1) / (double)(LT + 1), lo);
    const int ge = sturm_ge<double>(b2, 0, N, x) >= t + 1;
    const unsigned mask = __ballot_sync(0xffffffffu, ge) >> ((threadIdx.x & 31) & ~(LT - 1)) & ((1u << LT) - 1u);
    ++passes;
    if (it == 0) {
      if (!(mask & 1u)) {
        hi = lo;    // value below the bracket
        lo = 0.0;
      } else if (mask >> (LT - 1)) {
        lo = hi;    // value at or above it
        hi = top;
      }
    } else {
      const int m = __popc(mask);
      const int base = (threadIdx.x & 31) & ~(LT - 1);
      const double nlo = __shfl_sync(0xffffffffu, x, base + max(m - 1, 0));
      const double nhi = __shfl_sync(0xffffffffu, x, base + min(m, LT - 1));
      if (!done) {
        if (m > 0) lo = nlo;
        if (m < LT) hi = nhi;
      }
    }
    done = done || hi - lo <= fmax(2.3e-16 * hi, 8.7e-19);
    if (__all_sync(0xffffffffu, done)) break;
  }
  *lo_out = lo;
  *hi_out = hi;
  return passes;
}

// ------------------------------------------------------------------ twisted vectors
// 1 / d for the pivots: FP32 the fast reciprocal; FP64 the hardware estimate and two
// Newton-Raphson steps r <- r + r (1 - d r), which square the relative error each time.
__device__ __forceinline__ float pivot_rcp(float d) { return __fdividef(1.f, d); }
__device__ __forceinline__ double pivot_rcp(double d) {
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(d));
  r = fma(r, fma(-d, r, 1.0), r);
  r = fma(r, fma(-d, r, 1.0), r);
  return r;
}

// Block [s, e) of the split TGK that owns target t (see svd.cuh owning_block), by counts
// without divisions. lam, delta in the units of b2.
template <class R>
__device__ void owning_range(const R* b2, int N, const R* sig, int t, R delta, int* s_out, int* e_out) {
  const R lam = sig[t];
  int m = 0;
  for (int u = 0; u < t; ++u) m += rabs(sig[u] - lam) <= delta;
  int occ = 0, bs = 0;
  *s_out = 0;
  *e_out = N;
  for (int i = 0; i < N; ++i) {
    const bool end = (i == N - 1) || (b2[i] == R(0));
    if (!end) continue;
    const int e = i + 1;
    const int inwin = sturm_ge<R>(b2, bs, e, lam - delta) - sturm_ge<R>(b2, bs, e, lam + delta);
    if (inwin > 0 && occ + inwin > m) {
      *s_out = bs;
      *e_out = e;
      return;
    }
    occ += inwin;
    bs = e;
  }
}

}  // namespace gate
}  // namespace mpsvqe
