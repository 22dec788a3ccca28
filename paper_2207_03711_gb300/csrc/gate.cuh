// Device code of the gate engine: one two-site gate (Eqs. 7-10) by a thread-block cluster
// of C blocks (C = 1: one block). See gate_kernel.cuh for the kernel that strings these together.
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
#include <cfloat>
#include <cmath>
#include <cstdint>

#include "cx.cuh"
#include "gemm.cuh"
#include "kernels.cuh"
#include "svd.cuh"

namespace mpsvqe {
namespace gate {

// -------------------------------------------------------------------- bidiagonalisation
// T = Q B P^H (LAPACK reflector conventions) with one exposed cluster barrier per
// step: the updates by right reflector k-1 and left reflector k go over the trailing
// columns together, the next row comes out of that pass, and the product z with the next
// right reflector is formed from the unscaled row (its norm, hence its scale, is known one
// barrier later). Every block then forms the next column and its left reflector for itself
// from the exchanged sums, so no block waits for another inside a step. Exchanged per step:
// z partials, the next column before its right update, the partial norms of the row.
// The trailing matrix is read twice and written once per step, where two separate half
// steps read and write it twice.
// chi = 64 in mixed precision (128 steps): 667 k cycles in one block with two barriers a step, 311 k
// so on eight; chi = 128: 8.1 M cycles in one block from L2, 0.7 M; FP64 chi = 64: 12.4 M, 1.8 M.
// LAPACK-style reflector H = I - tau v v^H, v_0 = 1, for x = (alpha, tail) with ||tail||^2 =
// xn2: H^H x = beta e_1 with beta real, v = scale tail. A vector whose squared norm is
// within 16x of the smallest normal number counts as zero: the squares that make up that
// norm have lost their bits to underflow (entries below ~5e-19 in FP32, ~6e-154 in FP64),
// so the norm could come out as 0 while alpha is not, and 1 / (alpha - beta) would be a
// division by zero. The identity is taken there and the entries (absolutely that small)
// are dropped from the bidiagonal. The root and the reciprocals are the hardware estimates
// with a Newton-Raphson step, whose dependent chain is a quarter of a library square root's
// and four divisions': it runs twice per step of a serial recurrence.
// FP64 takes one step of third order (Chebyshev's iteration: the binomial series of
// (1 - e)^(-1/2) and (1 - e)^-1 in the residual e, up to e^2) from estimates of 20 bits, which is
// shorter in dependent operations than two Newton-Raphson steps; FP64 latency is what it costs.
// Both are within one and a half units of the last place over the range used.
__device__ __forceinline__ void root_and_inverse(float x, float* root, float* inv) {
  const float y = rsqrtf(x);
  float r = x * y;
  r = fmaf(0.5f * y, fmaf(-r, r, x), r);
  *root = r;
  *inv = fmaf(y, fmaf(-r, y, 1.0f), y);
}
__device__ __forceinline__ void root_and_inverse(double x, double* root, double* inv) {
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double e = fma(-x * y, y, 1.0);
  y = fma(y * e, fma(0.375, e, 0.5), y);
  *root = x * y;
  *inv = y;
}
__device__ __forceinline__ float inverse(float d) {
  const float r = __fdividef(1.0f, d);
  return fmaf(r, fmaf(-d, r, 1.0f), r);
}
__device__ __forceinline__ double inverse(double d) {
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(d));
  const double e = fma(-d, r, 1.0);
  return fma(r, fma(e, e, e), r);
}
template <class R>
__device__ __forceinline__ void reflector(Cx<R> alpha, R xn2, Cx<R>* tau, R* beta, Cx<R>* scale) {
  constexpr R kTiny2 = R(16) * (sizeof(R) == 4 ? R(FLT_MIN) : R(DBL_MIN));
  const R n2 = alpha.x * alpha.x + alpha.y * alpha.y + xn2;
  if ((xn2 == R(0) && alpha.y == R(0)) || !(n2 > kTiny2)) {
    *tau = cx<R>(0, 0);
    *beta = alpha.x;
    *scale = cx<R>(0, 0);
    return;
  }
  R nrm, inv;
  root_and_inverse(n2, &nrm, &inv);
  // |alpha - beta|^2 = |alpha|^2 + nrm^2 + 2 |Re alpha| nrm, without waiting for alpha - beta
  const R ax = alpha.x >= R(0) ? alpha.x : -alpha.x;
  const R rd = inverse(fma(R(2) * ax, nrm, R(2) * n2 - xn2));
  const R b = alpha.x >= R(0) ? -nrm : nrm, rb = alpha.x >= R(0) ? -inv : inv;
  *beta = b;
  *tau = cx<R>((b - alpha.x) * rb, -alpha.y * rb);
  *scale = cx<R>((alpha.x - b) * rd, -alpha.y * rd);
}

// Per own column: left factor, pending and new row entry (the pending right update uses
// the row entry of the step before).
template <class R>
struct alignas(16) ColState {
  Cx<R> f, ro, rn, pad;
};

// Own columns of T by local index, leading dimension ld (>= r): in shared memory, the first gc
// (even) of them in global memory where a block's shared memory does not hold them all. The
// columns leave the reduction in order, so the ones in global memory are read the least.
template <class R>
struct Columns {
  Cx<R>*s, *g;   // g: null where all fit (known at compile time: the engine's TG)
  int ld, gc;
  template <bool TG>
  __device__ __forceinline__ Cx<R>* at(int lc) const {
    if constexpr (!TG) return s + lc * ld;
    return lc < gc ? g + lc * ld : s + (lc - gc) * ld;
  }
};

template <class R>
struct Bidiag {
  Columns<R> T;        // own columns
  int gc0;             // columns of block 0 in global memory,
  size_t gstride;      // and from one block's to the next
  int zrows;
  Cx<R>* zp;           // [2][C VG][zrows] z partials, one per virtual rank
  Cx<R>* colp;         // [2][zrows] next column before its right update
  Cx<R>* sc;           // [0..1] row entry of the next column, [3..7]: scalars
  R* nrmp;             // [2][C VG] partial |row|^2
  Cx<R>*xs, *us;       // [zrows] X conj(right scale), the column (unscaled left reflector)
  ColState<R>* cs;     // [own]
  R *dd, *ee;
  Cx<R>*tau, *scl;     // factor and scale per reflector of the side the back-transformation needs
  Cx<R>* Y;            // global [.][ystride]: the reflector vectors of that side
  int ystride;
};

// log2 of the smallest power of two >= rows, at least a warp's.
__device__ __forceinline__ int row_shift(int rows) { return rows <= 32 ? 5 : 32 - __clz(rows - 1); }

// Virtual ranks: pair pi of columns belongs to rank pi mod (C VG), of which block pi mod C
// holds VG. Sums over columns are formed per virtual rank and added in a fixed tree, so the
// result has the same bits for every C with the same C VG: how many blocks a slot gets can
// follow from how many slots run.
template <class R, int NT, int C, int VG, bool TG>
__device__ __forceinline__ void bidiagonalize_cluster(const Bidiag<R> b, const int r, const int p,
                                                      const bool right_side, const unsigned rank) {
  const int tid = threadIdx.x;
  constexpr int GL = 8;                  // lanes per column in pass 1
  constexpr int NG = (NT - 64) / GL;     // columns at a time: all warps but two
  constexpr int NV = C * VG;             // virtual ranks
  const int own = 2 * (((p >> 1) + C - 1 - (int)rank) / C);   // p is even: pairs are never split
  for (int i = tid; i < own; i += NT) b.cs[i].rn = cx<R>(0, 0);
  // The right reflector of a row waits for the blocks' partial norms. One block, and FP64,
  // form it during pass 2 (with a cluster barrier of its own, hidden there); in FP32 that
  // barrier costs more than the reflector, which goes beside the sums of z after the step's
  // one barrier (chi = 64: 322 k cycles per gate against 345 k; FP64 1 861 k against 1 807 k).
  constexpr bool kEarly = C == 1 || sizeof(R) == 8;
  const bool last_warp = tid >= NT - 32;
  auto send_norm = [&](int first, int lnext, int npar) {
    // lane pairs over the pairs of one virtual rank, in the order of its columns
    const int l = tid & 31;
    R nn[VG];
#pragma unroll
    for (int g = 0; g < VG; ++g) {
      nn[g] = 0;
      // columns of virtual rank g at or after `first`: pairs lp = g mod VG
      const int lp0 = (first >> 1) + ((g - (first >> 1)) % VG + VG) % VG;
      for (int lc = 2 * (lp0 + (l >> 1) * VG) + (l & 1); lc < own; lc += 32 * VG)
        if (lc >= first && lc != lnext) nn[g] += norm2(b.cs[lc].rn);
    }
    // side by side: one after the other, VG chains of five shuffles were the longest of a step
    // in one block
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
      for (int g = 0; g < VG; ++g) nn[g] += __shfl_xor_sync(0xffffffffu, nn[g], o);
#pragma unroll
    for (int g = 0; g < VG; ++g)
      if (l < C) peer<C>(b.nrmp, l)[npar * NV + (int)rank + C * g] = nn[g];
    if (l < C && lnext >= 0) peer<C>(b.sc, l)[npar] = b.cs[lnext].rn;
    __syncwarp();
  };
  auto right_reflector = [&](int k, int npar) {
    Cx<R> tauR, scR;
    R betaR, rc[NV];
#pragma unroll
    for (int c = 0; c < NV; ++c) rc[c] = b.nrmp[npar * NV + c];
#pragma unroll
    for (int h = NV / 2; h > 0; h >>= 1)
#pragma unroll
      for (int c = 0; c < h; ++c) rc[c] += rc[c + h];
    reflector(conj(b.sc[npar]), rc[0], &tauR, &betaR, &scR);
    if (tid == NT - 32) {
      b.sc[6] = tauR;
      b.sc[7] = scR;
      b.ee[k] = betaR;
      if (right_side) {
        b.tau[k] = tauR;
        b.scl[k] = scR;
      }
    }
  };
  for (int k = 0; k < p; ++k) {
    const int par = k & 1, npar = par ^ 1, rows = r - k;
    const bool have_old = k > 0;
    // conj(col) X and |col|^2 per row, in place of the first two z partials of that row, which
    // its own thread has read by then (the peers write that buffer again after the next
    // cluster barrier)
    Cx<R>* pd = b.zp + par * NV * b.zrows;
    Cx<R>* pn = pd + b.zrows;
    // ---- sums of z, the right-update vector X and the next column, one thread per row
    Cx<R> a = cx<R>(0, 0), z = a;
    if (have_old) {
      if (!kEarly && last_warp) right_reflector(k - 1, par);
      if (tid < rows) {
        const Cx<R>* zq = b.zp + par * NV * b.zrows + tid;
        a = b.colp[par * b.zrows + tid];
        Cx<R> zc[NV];
#pragma unroll
        for (int c = 0; c < NV; ++c) zc[c] = zq[c * b.zrows];
#pragma unroll
        for (int h = NV / 2; h > 0; h >>= 1)
#pragma unroll
          for (int c = 0; c < h; ++c) zc[c] = zc[c] + zc[c + h];
        z = zc[0];
      }
      if (!kEarly) __syncthreads();
    }
    if (tid < rows) {
      Cx<R> X = cx<R>(0, 0), col;
      if (have_old) {
        const Cx<R> scR = b.sc[7];
        X = b.sc[6] * (a + scR * z);
        col = a - X;
        b.xs[tid] = X * conj(scR);
      } else {
        // column 0 is block 0's
        col = TG && b.gc0 ? ldcg(b.T.g - (size_t)rank * b.gstride + tid) : peer<C>(b.T.s, 0)[tid];
      }
      b.us[tid] = col;
      Cx<R> d = cx<R>(0, 0);
      cmac_conj(d, col, X);
      pn[tid].x = tid > 0 ? norm2(col) : R(0);
      pd[tid] = tid > 0 ? d : cx<R>(0, 0);
    }
    __syncthreads();
    // ---- first warp: left reflector u = (1, col scL) of that column; second warp: col^H X;
    // the others: pass 1, s_j = col^H a_j of the own trailing columns, which needs neither.
    // (Scalars go through one warp: they would cost every warp the same instructions, and
    // FP64 runs at two lanes a clock whatever the lanes hold.)
    const int l0 = 2 * ((((k + 1) >> 1) + C - 1 - (int)rank) / C);   // own pairs from column k (or k + 1) on
    const int first = 2 * (C * (l0 >> 1) + (int)rank) > k ? l0 : l0 + 1;   // own columns after k
    if (tid < 32) {
      R v = 0;
#pragma unroll
      for (int i = 0; i < 8; ++i)
        if (tid + 32 * i < rows) v += pn[tid + 32 * i].x;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
      Cx<R> tauL, scL;
      R betaL;
      reflector(b.us[0], v, &tauL, &betaL, &scL);
      if (tid == 0) {
        b.dd[k] = betaL;
        if (!right_side) {
          b.tau[k] = tauL;
          b.scl[k] = cx<R>(1, 0);
        }
        b.sc[3] = scL;
        b.sc[4] = conj(tauL);
      }
    } else if (tid < 64) {
      if (have_old) {
        Cx<R> v = cx<R>(0, 0);
#pragma unroll
        for (int i = 0; i < 8; ++i)
          if (tid - 32 + 32 * i < rows) v = v + pd[tid - 32 + 32 * i];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
          v.x += __shfl_xor_sync(0xffffffffu, v.x, o);
          v.y += __shfl_xor_sync(0xffffffffu, v.y, o);
        }
        if (tid == 32) b.sc[5] = v * conj(b.sc[7]);
      }
    } else if (k + 1 < p) {
      const int lane = tid & (GL - 1), grp = (tid - 64) / GL;
      for (int base = first; base < own; base += NG) {
        const int lc = base + grp;
        const bool act = lc < own;
        Cx<R> s = cx<R>(0, 0);
        if (act) {
          // four partial sums: the dependent chain, not the arithmetic, is what this costs
          auto dot = [&](const Cx<R>* t) {
            Cx<R> sp[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) sp[e] = cx<R>(0, 0);
            int i = lane == 0 ? GL : lane;
            for (; i + 3 * GL < rows; i += 4 * GL) {
              Cx<R> av[4], uv[4];
#pragma unroll
              for (int e = 0; e < 4; ++e) {
                av[e] = t[i + e * GL];
                uv[e] = b.us[i + e * GL];
              }
#pragma unroll
              for (int e = 0; e < 4; ++e) cmac_conj(sp[e], uv[e], av[e]);
            }
#pragma unroll
            for (int e = 0; e < 3; ++e)
              if (i + e * GL < rows) cmac_conj(sp[e], b.us[i + e * GL], t[i + e * GL]);
            return (sp[0] + sp[1]) + (sp[2] + sp[3]);
          };
          if (TG && lc < b.T.gc)
            s = dot(b.T.g + lc * b.T.ld + k);
          else
            s = dot(b.T.s + (TG ? lc - b.T.gc : lc) * b.T.ld + k);
        }
#pragma unroll
        for (int o = 1; o < GL; o <<= 1) {
          s.x += __shfl_xor_sync(0xffffffffu, s.x, o, GL);
          s.y += __shfl_xor_sync(0xffffffffu, s.y, o, GL);
        }
        if (act && lane == 0) b.cs[lc].f = s;
      }
    }
    __syncthreads();
    const Cx<R> scL = b.sc[3];
    if (!right_side && (k % C) == (int)rank)
      for (int i = tid; i < rows; i += NT) b.Y[(size_t)k * b.ystride + k + i] = i == 0 ? cx<R>(1, 0) : b.us[i] * scL;
    if (k + 1 >= p) break;
    // ---- the left factor f_j and the new row entry r_j, with the pending right update taken
    // into account: u^H (a_j - X conj(scR) r_j') = (a_j - X conj(scR) r_j')_0 + conj(scL)
    // (col^H a_j - col^H X conj(scR) r_j')
    for (int lc = first + tid; lc < own; lc += NT) {
      Cx<R> rn = b.T.template at<TG>(lc)[k], t = b.cs[lc].f;
      const Cx<R> ro = b.cs[lc].rn;
      if (have_old) {
        cmsub(rn, b.xs[0], ro);
        cmsub(t, b.sc[5], ro);
      }
      Cx<R> s = rn;
      cmac_conj(s, scL, t);
      const Cx<R> f = b.sc[4] * s;
      rn = rn - f;
      b.cs[lc].f = f;
      b.cs[lc].ro = ro;
      b.cs[lc].rn = rn;
      if (right_side) b.Y[(size_t)k * b.ystride + 2 * (C * (lc >> 1) + (int)rank) + (lc & 1)] = conj(rn);
    }
    __syncthreads();
    const int lnext = ((k + 1) >> 1) % C == (int)rank ? 2 * (((k + 1) >> 1) / C) + ((k + 1) & 1) : -1;
    // ---- last warp: partial norm of the new row (columns after k + 1) and its leading entry
    // to all blocks
    const int nrow = rows - 1, rsh2 = row_shift(nrow), groups = min(VG, NT >> rsh2);
    const bool last_busy = (groups << rsh2) > NT - 32;   // it has rows of its own in pass 2
    if (last_warp && (kEarly || !last_busy)) send_norm(first, lnext, npar);
    if constexpr (kEarly) {
      csync_arrive<C>();
      if (last_warp && !last_busy) {
        csync_wait<C>();
        right_reflector(k, npar);
      }
    }
    // ---- pass 2: both updates, one thread per row and column group; z = sum a_j conj(r_j)
    // over the columns after k + 1; column k + 1 goes out whole
    const int row = tid & ((1 << rsh2) - 1), cgp = tid >> rsh2;
    if (cgp < groups && row < nrow) {
      const Cx<R> u = b.us[row + 1] * scL;
      const Cx<R> x = have_old ? b.xs[row + 1] : cx<R>(0, 0);
      Cx<R>* col0 = b.T.s + k + 1 + row - (TG ? b.T.gc * b.T.ld : 0);   // of the columns in shared memory
      auto update = [&](Cx<R> v, const ColState<R>& q) {
        cmsub(v, x, q.ro);
        cmsub(v, q.f, u);
        return v;
      };
      auto entry = [&](int lc) { return TG ? b.T.template at<TG>(lc) + k + 1 + row : col0 + lc * b.T.ld; };
      for (int g = cgp; g < VG; g += groups) {
        Cx<R> z1 = cx<R>(0, 0), z2 = cx<R>(0, 0);   // even and odd columns of the pairs
        const int lf = first >> 1;
        int lp = VG == 1 ? lf : lf + ((g - lf) % VG + VG) % VG;
        if (lp == lf) {
          // the first pair: its even column may be gone, or one of them be column k + 1
          const int lc = 2 * lp;
          if (lc >= first && lc < own) {
            const ColState<R> q = b.cs[lc];
            Cx<R>* at = entry(lc);
            const Cx<R> v = update(*at, q);
            if (lc == lnext) {
#pragma unroll
              for (int c = 0; c < C; ++c) peer<C>(b.colp, c)[npar * b.zrows + row] = v;
            } else {
              *at = v;
              cmac_bconj(z1, v, q.rn);
            }
          }
          if (lc + 1 < own) {
            const ColState<R> q = b.cs[lc + 1];
            Cx<R>* at = entry(lc + 1);
            const Cx<R> v = update(*at, q);
            if (lc + 1 == lnext) {
#pragma unroll
              for (int c = 0; c < C; ++c) peer<C>(b.colp, c)[npar * b.zrows + row] = v;
            } else {
              *at = v;
              cmac_bconj(z2, v, q.rn);
            }
          }
          lp += VG;
        }
        if constexpr (TG) {
          // columns in global memory: those of two pairs on their way at a time
          Cx<R>* cg = b.T.g + k + 1 + row;
          const int ge = min(b.T.gc, own);
          while (2 * lp < ge) {
            const bool two = 2 * (lp + VG) < ge;
            Cx<R> in[4];
#pragma unroll
            for (int e = 0; e < 4; ++e)
              if (e < 2 || two) in[e] = cg[(2 * (lp + e / 2 * VG) + (e & 1)) * b.T.ld];
#pragma unroll
            for (int e = 0; e < 2; ++e)
              if (e == 0 || two) {
                const int lc = 2 * (lp + e * VG);
                const ColState<R> q = b.cs[lc], q2 = b.cs[lc + 1];
                const Cx<R> v = update(in[2 * e], q), v2 = update(in[2 * e + 1], q2);
                cg[lc * b.T.ld] = v;
                cg[(lc + 1) * b.T.ld] = v2;
                cmac_bconj(z1, v, q.rn);
                cmac_bconj(z2, v2, q2.rn);
              }
            lp += two ? 2 * VG : VG;
          }
        }
        for (int lc = 2 * lp; lc < own; lc += 2 * VG) {
          const ColState<R> q = b.cs[lc], q2 = b.cs[lc + 1];
          const Cx<R> v = update(col0[lc * b.T.ld], q), v2 = update(col0[(lc + 1) * b.T.ld], q2);
          col0[lc * b.T.ld] = v;
          col0[(lc + 1) * b.T.ld] = v2;
          cmac_bconj(z1, v, q.rn);
          cmac_bconj(z2, v2, q2.rn);
        }
        z1 = z1 + z2;
#pragma unroll
        for (int c = 0; c < C; ++c)
          peer<C>(b.zp, c)[(npar * NV + (int)rank + C * g) * b.zrows + row] = z1;
      }
    }
    if constexpr (kEarly) {
      if (!last_warp) {
        csync_wait<C>();
      } else if (last_busy) {
        csync_wait<C>();
        right_reflector(k, npar);
      }
    } else if (last_warp && last_busy) {
      send_norm(first, lnext, npar);
    }
    csync<C>();
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
__device__ __forceinline__ float rescale_factor(float a, float b) {
  const unsigned m = max((__float_as_uint(a) >> 23) & 255u, (__float_as_uint(b) >> 23) & 255u);
  return __uint_as_float((254u - min(m, 253u)) << 23);
}
__device__ __forceinline__ double rescale_factor(double a, double b) {
  const unsigned m = max(((unsigned)__double2hiint(a) >> 20) & 2047u, ((unsigned)__double2hiint(b) >> 20) & 2047u);
  return __hiloint2double((int)((2046u - min(m, 2045u)) << 20), 0);
}
__device__ __forceinline__ unsigned sign_bits(float a, float b) { return (__float_as_uint(a) ^ __float_as_uint(b)) >> 31; }
__device__ __forceinline__ unsigned sign_bits(double a, double b) {
  return (unsigned)(__double2hiint(a) ^ __double2hiint(b)) >> 31;
}
template <class R>
struct SturmGroup;   // steps between rescalings
template <>
struct SturmGroup<float> {
  static constexpr int v = 4;
};
template <>
struct SturmGroup<double> {
  static constexpr int v = 8;
};
// V shifts at once, for as many independent chains. last (optional): p_e with its binary
// exponent, for interpolation.
template <class R, int V>
__device__ __forceinline__ void sturm_ge(const R* b2, int s, int e, const R* x, int* ge, R* last = nullptr,
                                         int* last_exp = nullptr) {
  constexpr int GRP = SturmGroup<R>::v;
  R prev[V], cur[V];
  unsigned neg[V];
  int ex[V];
#pragma unroll
  for (int v = 0; v < V; ++v) {
    prev[v] = R(1);
    cur[v] = -x[v];
    neg[v] = sign_bits(cur[v], prev[v]);
    ex[v] = 0;
  }
  int i = s + 1;
  for (; i + GRP <= e; i += GRP) {
    R bb[GRP];
#pragma unroll
    for (int u = 0; u < GRP; ++u) bb[u] = b2[i + u - 1];
#pragma unroll
    for (int u = 0; u < GRP; ++u)
#pragma unroll
      for (int v = 0; v < V; ++v) {
        const R nxt = fma(-x[v], cur[v], -(bb[u] * prev[v]));
        neg[v] += sign_bits(nxt, cur[v]);
        prev[v] = cur[v];
        cur[v] = nxt;
      }
#pragma unroll
    for (int v = 0; v < V; ++v) {
      const R sc = rescale_factor(prev[v], cur[v]);
      prev[v] *= sc;
      cur[v] *= sc;
      if (last) ex[v] += 1023 - (int)(((unsigned)__double2hiint((double)sc) >> 20) & 2047u);
    }
  }
  for (; i < e; ++i) {
    const R bi = b2[i - 1];
#pragma unroll
    for (int v = 0; v < V; ++v) {
      const R nxt = fma(-x[v], cur[v], -(bi * prev[v]));
      neg[v] += sign_bits(nxt, cur[v]);
      prev[v] = cur[v];
      cur[v] = nxt;
    }
  }
#pragma unroll
  for (int v = 0; v < V; ++v) {
    ge[v] = (e - s) - (int)neg[v];
    if (last) {
      last[v] = cur[v];
      last_exp[v] = ex[v];
    }
  }
}
template <class R>
__device__ __forceinline__ int sturm_ge1(const R* b2, int s, int e, R x) {
  int ge;
  sturm_ge<R, 1>(b2, s, e, &x, &ge);
  return ge;
}

// Singular value t (0-based, descending) of the TGK block [s, e) in FP32 by half a warp: 16
// shifts a pass, each pass narrows the bracket 17-fold. First pass on a log grid over
// eight decades, then linear to the working precision or `passes` passes. lo/hi bracket
// the value; one found to lie below `floor` is left there. Always 16 lanes, so that the
// shifts, and with them the last bits, do not depend on how many values a block has.
constexpr int kBisectLanes = 16;
__device__ __forceinline__ int half_bisect(const float* b2, int s, int e, int t, bool act, float top, float floor,
                                           int passes, float* lo_out, float* hi_out) {
  constexpr int LP = kBisectLanes;
  const int wl = threadIdx.x & 31, lane = wl & (LP - 1), base = wl & ~(LP - 1);
  float lo = 0.f, hi = top;
  int it = 0;
  bool open = act;
  while (it < passes) {
    const float x = it == 0 ? top * exp10f(-8.0f * (float)(LP - lane) / (float)(LP + 1))
                            : fmaf(hi - lo, (float)(lane + 1) / (float)(LP + 1), lo);
    const bool above = sturm_ge1<float>(b2, s, e, x) >= t + 1;
    // counts fall with x: the number of shifts below the value locates it
    const int m = __popc((__ballot_sync(0xffffffffu, above) >> base) & ((1u << LP) - 1u));
    const float nlo = __shfl_sync(0xffffffffu, x, base + max(m - 1, 0));
    const float nhi = __shfl_sync(0xffffffffu, x, base + min(m, LP - 1));
    if (open) {
      if (m > 0) lo = nlo;
      if (m < LP) hi = nhi;
    }
    // not yet two neighbours of the working precision, and not below what is kept
    open = open && hi - lo > 1.2e-7f * hi && hi > floor;
    ++it;
    if (!__any_sync(0xffffffffu, open)) break;
  }
  *lo_out = lo;
  *hi_out = hi;
  return it;
}

// Value t of block [s, e) in FP64 from the FP32 bracket, LT = 4 lanes per value (a warp's FP64 operation
// takes 16 clocks whatever the lanes do, so few shifts per pass cost the least). The
// bracket is checked with FP64 counts first and opened up if it does not hold. Then every
// other way of placing the shifts: two on either side of the secant estimate of the root
// of p_N inside the bracket (w 2^-16 and w 2^-6 away; a simple root gains 5 to 15 bits a
// pass), or, when that gained less than a plain section would, evenly. The bracket itself
// always moves by counts, so a wrong estimate costs a pass and nothing else. Stops at the
// working precision relative to the value, or at 2^-60 of the largest one.
__device__ __forceinline__ int lanes_bisect(const double* b2, int s, int e, int t, bool act, double top, double floor,
                                            float lo_f, float hi_f, double* lo_out, double* hi_out) {
  constexpr int LT = 4;
  const int wl = threadIdx.x & 31, lane = wl & (LT - 1), base = wl & ~(LT - 1);
  double lo = (double)lo_f * (1.0 - 4e-6), hi = fmin(top, (double)hi_f * (1.0 + 4e-6) + 1e-30);
  double flo = 0.0, fhi = 0.0;   // p_N at the ends, in a common scale; 0: not known
  bool done = !act, even = false;
  int passes = 0;
  for (int it = 0; it < 64; ++it) {
    const double w = hi - lo;
    double x;
    // secant estimate; both ends have to be known and of opposite sign
    const bool secant = it > 0 && flo * fhi < 0.0 && !even;
    if (it == 0) {
      x = lane == 0 ? lo : hi;
    } else if (secant) {
      const double off = lane == 0 ? -0x1p-6 : lane == 1 ? -0x1p-16 : lane == 2 ? 0x1p-16 : 0x1p-6;
      x = fma(w, fmin(fmax(fma(flo, inverse(flo - fhi), off), 0x1p-30), 1.0 - 0x1p-30), lo);
    } else {
      x = fma(w, (double)(lane + 1) * 0.2, lo);
    }
    int ge1, ex;
    double f;
    sturm_ge<double, 1>(b2, s, e, &x, &ge1, &f, &ex);
    const unsigned mask = (__ballot_sync(0xffffffffu, ge1 >= t + 1) >> base) & 15u;
    ++passes;
    int il, ih;   // lanes that become the new ends (-1: the old one stays)
    bool reopen = false;
    if (it == 0) {
      il = 0;
      ih = LT - 1;
      if (!(mask & 1u) || (mask >> (LT - 1))) reopen = true;
    } else {
      const int m = __popc(mask);
      il = m > 0 ? m - 1 : -1;
      ih = m < LT ? m : -1;
    }
    const double xl = __shfl_sync(0xffffffffu, x, base + max(il, 0)), xh = __shfl_sync(0xffffffffu, x, base + max(ih, 0));
    const double fl = __shfl_sync(0xffffffffu, f, base + max(il, 0)), fh = __shfl_sync(0xffffffffu, f, base + max(ih, 0));
    const int el = __shfl_sync(0xffffffffu, ex, base + max(il, 0)), eh = __shfl_sync(0xffffffffu, ex, base + max(ih, 0));
    if (!done) {
      if (reopen) {
        if (!(mask & 1u)) {
          hi = lo;    // value below the bracket
          lo = 0.0;
        } else {
          lo = hi;    // value at or above it
          hi = top;
        }
        flo = fhi = 0.0;
      } else {
        // an end that stays keeps no usable scale next to a new one: the estimate then
        // waits for the next pass
        if (il >= 0) lo = xl;
        if (ih >= 0) hi = xh;
        if (il >= 0 && ih >= 0) {
          const int d = max(-900, min(900, el - eh));
          flo = ldexp(fl, d > 0 ? 0 : d);
          fhi = ldexp(fh, d > 0 ? -d : 0);
        } else {
          flo = fhi = 0.0;
        }
        even = secant && !(hi - lo < 0.2 * w);
      }
    }
    done = done || hi - lo <= fmax(2.3e-16 * hi, 8.7e-19) || hi <= floor;
    if (__all_sync(0xffffffffu, done)) break;
  }
  *lo_out = lo;
  *hi_out = hi;
  return passes;
}

}  // namespace gate
}  // namespace mpsvqe
