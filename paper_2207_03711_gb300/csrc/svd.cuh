// The two fallbacks of a gate's truncated SVD (Eq. 9 of the paper), run by one thread
// block: block Gram-Schmidt for singular vectors of the bidiagonal that are too far from
// orthonormal for Newton-Schulz steps, and one-sided Jacobi where even that collapses
// (numerically degenerate singular values without a split). The main route is gate.cuh's.
#pragma once
#include <cfloat>
#include "cx.cuh"

namespace mpsvqe {

template <class R>
__device__ __forceinline__ R rabs(R x) {
  return x < R(0) ? -x : x;
}
// Block classical Gram-Schmidt twice (BCGS2) over the rows of W (k x p, row stride
// ldw), in blocks of 8 rows. Each of the two repetitions projects the block out of all
// earlier rows and then orthonormalises it internally by Cholesky QR (G = W_b W_b^T =
// L L^T, W_b <- L^{-1} W_b). Row t of the result depends only on rows 0..t, so the
// leading singular vectors keep their directions. The rows come in with unit norm. A row of
// which only theta is left beside the rows before it keeps theta of its own direction
// against eps of rounding, so eps / theta of sigma / sigma_0 is what M' loses by it: a
// squared theta below collapse_limit counts as a collapse. coef: >= 8 k shared scratch (used
// once k > 8); small: >= 128 shared.
template <class R>
__device__ __forceinline__ R collapse_limit(R sigma, R sigma0) {
  const R t = sigma0 > R(0) ? sigma / sigma0 : R(1);
  const R lim = sizeof(R) == 4 ? R(0.36) * t * t : R(0.01) * t * t;
  return fmin(R(1e-6), fmax(sizeof(R) == 4 ? R(1e-11) : R(1e-26), lim));
}
template <class R, int NT>
__device__ void orthonormalize_rows_block(R* W, int ldw, int k, int p, const R* sig, R* coef, R* small,
                                          int* collapsed) {
  const int tid = threadIdx.x;
  for (int b0 = 0; b0 < k; b0 += 8) {
    const int nb = min(8, k - b0);
    for (int rep = 0; rep < 2; ++rep) {
      if (b0 > 0) {
        // coef[u * 8 + j] = <w_u, w_{b0+j}>, 8 lanes per dot
        const int nd = b0 * nb;
        for (int base = 0; base < nd * 8; base += NT) {
          const int d = (base + tid) >> 3, l = tid & 7;
          const bool act = d < nd;
          const int u = act ? d / nb : 0, j = act ? d - u * nb : 0;
          R acc = 0;
          if (act)
            for (int q = l; q < p; q += 8) acc += W[(size_t)u * ldw + q] * W[(size_t)(b0 + j) * ldw + q];
          for (int o = 1; o < 8; o <<= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
          if (act && l == 0) coef[u * 8 + j] = acc;
        }
        __syncthreads();
        for (int it = tid; it < nb * p; it += NT) {
          const int j = it / p, q = it - j * p;
          R v = W[(size_t)(b0 + j) * ldw + q];
          for (int u = 0; u < b0; ++u) v -= coef[u * 8 + j] * W[(size_t)u * ldw + q];
          W[(size_t)(b0 + j) * ldw + q] = v;
        }
        __syncthreads();
      }
      // Gram matrix of the block (lower triangle): small[i * 8 + j], j <= i
      const int ng = nb * (nb + 1) / 2;
      for (int base = 0; base < ng * 8; base += NT) {
        const int d = (base + tid) >> 3, l = tid & 7;
        const bool act = d < ng;
        int i = 0;
        while ((i + 1) * (i + 2) / 2 <= d && i < 7) ++i;
        const int j = d - i * (i + 1) / 2;
        R acc = 0;
        if (act)
          for (int q = l; q < p; q += 8) acc += W[(size_t)(b0 + i) * ldw + q] * W[(size_t)(b0 + j) * ldw + q];
        for (int o = 1; o < 8; o <<= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        if (act && l == 0) small[i * 8 + j] = acc;
      }
      __syncthreads();
      // Cholesky factor L and its inverse X = L^{-1} (written to small + 64); one thread,
      // the 8 x 8 factor kept in registers (all indices compile-time)
      if (tid == 0) {
        R Lm[8][8], Xm[8][8];
#pragma unroll
        for (int i = 0; i < 8; ++i)
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            Lm[i][j] = (j <= i && i < nb) ? small[i * 8 + j] : R(0);
            Xm[i][j] = R(0);
          }
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          if (j < nb) {
            const R gjj = Lm[j][j];
            R d = gjj;
#pragma unroll
            for (int u = 0; u < j; ++u) d -= Lm[j][u] * Lm[j][u];
            if (!(d > (rep == 0 ? collapse_limit(sig[b0 + j], sig[0]) : R(1e-6) * gjj))) {
              ++*collapsed;
              d = gjj > R(0) ? gjj * R(1e-30) : R(1e-30);
            }
            const R ljj = sqrt(d), inv = R(1) / ljj;
            Lm[j][j] = ljj;
#pragma unroll
            for (int i = j + 1; i < 8; ++i) {
              R v = Lm[i][j];
#pragma unroll
              for (int u = 0; u < j; ++u) v -= Lm[i][u] * Lm[j][u];
              Lm[i][j] = v * inv;
            }
          }
        }
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          Xm[j][j] = R(1) / Lm[j][j];
#pragma unroll
          for (int i = j + 1; i < 8; ++i) {
            R v = 0;
#pragma unroll
            for (int u = j; u < i; ++u) v += Lm[i][u] * Xm[u][j];
            Xm[i][j] = -v / Lm[i][i];
          }
        }
#pragma unroll
        for (int i = 0; i < 8; ++i)
#pragma unroll
          for (int j = 0; j < 8; ++j) small[64 + i * 8 + j] = Xm[i][j];
      }
      __syncthreads();
      // W_b <- X W_b, one thread per column
      for (int q = tid; q < p; q += NT) {
        R x[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) x[i] = i < nb ? W[(size_t)(b0 + i) * ldw + q] : R(0);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          if (i < nb) {
            R y = 0;
#pragma unroll
            for (int u = 0; u <= i; ++u) y += small[64 + i * 8 + u] * x[u];
            W[(size_t)(b0 + i) * ldw + q] = y;
          }
        }
      }
      __syncthreads();
    }
  }
}

// One-sided (Hestenes) Jacobi on the n columns of the real n x n matrix X (column stride
// ldx), used when Gram-Schmidt reports a collapsed vector (numerically degenerate singular
// values without a split). It runs on the bidiagonal factor, not on the complex M': a
// quarter of the arithmetic, and the back-transformation takes its vectors like any
// others. Columns converge to sigma_p times a singular vector; columns below sqrt(zero2)
// are numerically zero. n <= 32 MAXE.
template <class R, int NT, int MAXE>
__device__ void jacobi_columns(R* X, int ldx, int n, double zero2, int max_sweeps, int* noconv) {
  int G = 1;
  while (G < 32 && G * MAXE < n) G <<= 1;
  const int npairs = (n + 1) >> 1;
  // (as for 256 threads, whatever NT: the lanes of a dot product fix its last bits)
  while (G < 32 && G < n && (256 / (2 * G)) >= npairs) G <<= 1;
  const int ept = (n + G - 1) / G;
  const int ngroups = NT / G, grp = threadIdx.x / G, lane = threadIdx.x - grp * G;
  const R tol = R(2) * (sizeof(R) == 8 ? R(2.220446049250313e-16) : R(1.1920929e-7)) * sqrt((R)n);
  const int mm = n + (n & 1);  // even number of players; index n is a dummy
  bool converged = n <= 1;
  int sweep = 0;
  for (; sweep < max_sweeps && !converged; ++sweep) {
    int rotated = 0;
    for (int r = 0; r < mm - 1; ++r) {
      for (int base = 0; base < mm / 2; base += ngroups) {
        const int pi = base + grp;
        int p = 0, q = 1;
        if (pi == 0) {
          p = r;
          q = mm - 1;
        } else if (pi < mm / 2) {
          p = r + pi;
          if (p >= mm - 1) p -= mm - 1;
          q = r - pi;
          if (q < 0) q += mm - 1;
        }
        const bool active = pi < mm / 2 && p < n && q < n;
        R* xp = X + (size_t)p * ldx;
        R* xq = X + (size_t)q * ldx;
        R vp[MAXE], vq[MAXE];
        R al = 0, be = 0, ga = 0;
#pragma unroll
        for (int e = 0; e < MAXE; ++e) {
          const int idx = lane + e * G;
          const bool in = active && e < ept && idx < n;
          vp[e] = in ? xp[idx] : R(0);
          vq[e] = in ? xq[idx] : R(0);
          al = fma(vp[e], vp[e], al);
          be = fma(vq[e], vq[e], be);
          ga = fma(vp[e], vq[e], ga);
        }
        for (int o = G >> 1; o > 0; o >>= 1) {
          al += __shfl_xor_sync(0xffffffffu, al, o, G);
          be += __shfl_xor_sync(0xffffffffu, be, o, G);
          ga += __shfl_xor_sync(0xffffffffu, ga, o, G);
        }
        const R ag = rabs(ga);
        if (active && ag > R(0) && (double)fmin(al, be) > zero2 && ag > tol * sqrt(al) * sqrt(be)) {
          const R zeta = (be - al) / (R(2) * ga);
          const R az = rabs(zeta);
          const R t = az > R(1e15) ? R(0.5) / zeta : copysign(R(1), zeta) / (az + sqrt(R(1) + zeta * zeta));
          if (t != R(0)) {
            const R cs = R(1) / sqrt(R(1) + t * t), sn = cs * t;
#pragma unroll
            for (int e = 0; e < MAXE; ++e) {
              const int idx = lane + e * G;
              if (e < ept && idx < n) {
                const R a = vp[e], b = vq[e];
                xp[idx] = cs * a - sn * b;
                xq[idx] = sn * a + cs * b;
              }
            }
            rotated = 1;
          }
        }
      }
      __syncthreads();
    }
    converged = !__syncthreads_or(rotated);
  }
  if (threadIdx.x == 0 && !converged) ++*noconv;
}

}  // namespace mpsvqe
