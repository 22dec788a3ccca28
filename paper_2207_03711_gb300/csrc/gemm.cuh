// Device helpers shared by the gate engine and the measurement: thread-block clusters and
// a tiled complex GEMM for one thread block.
#pragma once
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <cstdint>

#include "cx.cuh"

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

// The two halves of a cluster barrier, for work in between; whole warps, every warp both.
template <int C>
__device__ __forceinline__ void csync_arrive() {
  if constexpr (C > 1) asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
template <int C>
__device__ __forceinline__ void csync_wait() {
  if constexpr (C > 1) asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
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
// Operand entries in shared memory and their accumulators. FP32: an entry is split into a
// multiple of 2^-11 and a rest; products of two leading parts are multiples of 2^-22 and,
// with rows and columns of norm <= 1 (isometries), their partial sums stay below 4, so FP32
// adds them exactly, while the three products with a rest are 2^-12 times smaller and so
// are their rounding errors. The sum comes out rounded once, at the price of four FMAs per
// real product; larger entries only lose the exactness, not the value. These contractions
// are a few per cent of a gate, and their plain FP32 rounding was the largest part of a
// mixed-precision energy's error after the truncation itself.
struct SplitF {
  float4 v;   // x leading, x rest, y leading, y rest
};
struct SplitAcc {
  float hx, hy, lx, ly;
};
__device__ __forceinline__ float lead11(float x) {
  constexpr float kMagic = 6144.0f;   // 1.5 2^12: adding it rounds to a multiple of 2^-11
  return __fadd_rn(__fadd_rn(x, kMagic), -kMagic);
}
__device__ __forceinline__ SplitF to_elem(Cx<float> a) {
  const float hx = lead11(a.x), hy = lead11(a.y);
  return SplitF{make_float4(hx, __fadd_rn(a.x, -hx), hy, __fadd_rn(a.y, -hy))};
}
__device__ __forceinline__ void zero(SplitAcc& a) { a.hx = a.hy = a.lx = a.ly = 0.f; }
__device__ __forceinline__ void zero(Cx<double>& a) { a = cx<double>(0, 0); }
// acc += a b
__device__ __forceinline__ void mac(SplitAcc& c, const SplitF& a, const SplitF& b) {
  c.hx = fmaf(-a.v.z, b.v.z, fmaf(a.v.x, b.v.x, c.hx));
  c.hy = fmaf(a.v.z, b.v.x, fmaf(a.v.x, b.v.z, c.hy));
  c.lx = fmaf(a.v.y, b.v.x, fmaf(a.v.x, b.v.y, c.lx));
  c.ly = fmaf(a.v.y, b.v.z, fmaf(a.v.x, b.v.w, c.ly));
  c.lx = fmaf(-a.v.w, b.v.z, fmaf(-a.v.z, b.v.w, c.lx));
  c.ly = fmaf(a.v.w, b.v.x, fmaf(a.v.z, b.v.y, c.ly));
  c.lx = fmaf(-a.v.w, b.v.w, fmaf(a.v.y, b.v.y, c.lx));
  c.ly = fmaf(a.v.w, b.v.y, fmaf(a.v.y, b.v.w, c.ly));
}
__device__ __forceinline__ void mac(Cx<double>& c, const Cx<double>& a, const Cx<double>& b) { cmac(c, a, b); }
__device__ __forceinline__ Cx<float> value(const SplitAcc& a) {
  return cx<float>(__fadd_rn(a.hx, a.lx), __fadd_rn(a.hy, a.ly));
}
__device__ __forceinline__ Cx<double> value(const Cx<double>& a) { return a; }
template <class R>
struct Gemm {
  using E = Cx<R>;
  using A = Cx<R>;
  static __device__ __forceinline__ E elem(Cx<R> a) { return a; }
};
template <>
struct Gemm<float> {
  using E = SplitF;
  using A = SplitAcc;
  static __device__ __forceinline__ E elem(Cx<float> a) { return to_elem(a); }
};

// out(m, n) = sum_k a(m, k) b(k, n) for m < M, n < N by one block. The operands come from
// L2 through functors, so orientation, conjugation and the cyclic column spread cost
// nothing extra. RM x JN outputs per thread: tiles of (NT / 16) RM rows by 16 JN columns,
// KT deep, the next K tile loaded to registers while the present one is used. KF: b's k
// index runs fastest in memory.
constexpr int kKT = 16;
template <int NT>
__host__ __device__ constexpr size_t gemm_tile_bytes() {   // of the largest tile shape below; entries are 16 bytes
  constexpr int TY = NT / 16;
  return 16 * (size_t)((4 * TY) * (kKT + 1) + kKT * (64 + 1));
}
template <class R, int NT, int RM, int JN, bool KF, class FA, class FB, class FC>
__device__ __forceinline__ void tile_gemm_shape(int M, int N, int K, FA fa, FB fb, FC fc, unsigned char* smem) {
  using G = Gemm<R>;
  using E = typename G::E;
  constexpr int TY = NT / 16, TM = TY * RM, TN = 16 * JN, KT = kKT;
  constexpr int NA = TM * KT / NT, NB = KT * TN / NT > 0 ? KT * TN / NT : 1;
  E(*As)[KT + 1] = reinterpret_cast<E(*)[KT + 1]>(smem);
  E(*Bs)[TN + 1] = reinterpret_cast<E(*)[TN + 1]>(smem + sizeof(E) * TM * (KT + 1));
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  for (int m0 = 0; m0 < M; m0 += TM)
    for (int n0 = 0; n0 < N; n0 += TN) {
      typename G::A acc[RM][JN];
#pragma unroll
      for (int i = 0; i < RM; ++i)
#pragma unroll
        for (int j = 0; j < JN; ++j) zero(acc[i][j]);
      Cx<R> ra[NA], rb[NB];
      auto fetch = [&](int k0) {
#pragma unroll
        for (int e = 0; e < NA; ++e) {
          const int x = tid + e * NT, r = x / KT, kk = x % KT;
          ra[e] = (m0 + r < M && k0 + kk < K) ? fa(m0 + r, k0 + kk) : cx<R>(0, 0);
        }
#pragma unroll
        for (int e = 0; e < NB; ++e) {
          const int x = tid + e * NT, kk = KF ? x % KT : x / TN, n = KF ? x / KT : x % TN;
          rb[e] = (x < KT * TN && n0 + n < N && k0 + kk < K) ? fb(k0 + kk, n0 + n) : cx<R>(0, 0);
        }
      };
      fetch(0);
      for (int k0 = 0; k0 < K; k0 += KT) {
        __syncthreads();
#pragma unroll
        for (int e = 0; e < NA; ++e) {
          const int x = tid + e * NT;
          As[x / KT][x % KT] = G::elem(ra[e]);
        }
#pragma unroll
        for (int e = 0; e < NB; ++e) {
          const int x = tid + e * NT, kk = KF ? x % KT : x / TN, n = KF ? x / KT : x % TN;
          if (x < KT * TN) Bs[kk][n] = G::elem(rb[e]);
        }
        __syncthreads();
        if (k0 + KT < K) fetch(k0 + KT);
        const int kt = min(KT, K - k0);
        if (kt == KT) {
#pragma unroll 4
          for (int kk = 0; kk < KT; ++kk) {
            E a[RM], b[JN];
#pragma unroll
            for (int i = 0; i < RM; ++i) a[i] = As[ty + TY * i][kk];
#pragma unroll
            for (int j = 0; j < JN; ++j) b[j] = Bs[kk][tx + 16 * j];
#pragma unroll
            for (int i = 0; i < RM; ++i)
#pragma unroll
              for (int j = 0; j < JN; ++j) mac(acc[i][j], a[i], b[j]);
          }
        } else {
          for (int kk = 0; kk < kt; ++kk) {
            E a[RM], b[JN];
#pragma unroll
            for (int i = 0; i < RM; ++i) a[i] = As[ty + TY * i][kk];
#pragma unroll
            for (int j = 0; j < JN; ++j) b[j] = Bs[kk][tx + 16 * j];
#pragma unroll
            for (int i = 0; i < RM; ++i)
#pragma unroll
              for (int j = 0; j < JN; ++j) mac(acc[i][j], a[i], b[j]);
          }
        }
      }
#pragma unroll
      for (int i = 0; i < RM; ++i)
#pragma unroll
        for (int j = 0; j < JN; ++j) {
          const int mi = m0 + ty + TY * i, ni = n0 + tx + 16 * j;
          if (mi < M && ni < N) fc(mi, ni, value(acc[i][j]));
        }
    }
  __syncthreads();
}

// Shape by the narrow side: what one thread computes is kept at four outputs where the
// product has them, and small products spread over all threads.
template <class R, int NT, bool KF, class FA, class FB, class FC>
__device__ __forceinline__ void tile_gemm(int M, int N, int K, FA fa, FB fb, FC fc, unsigned char* smem) {
  constexpr int TY = NT / 16;
  if (N <= 16) {
    if (M <= TY)
      tile_gemm_shape<R, NT, 1, 1, KF>(M, N, K, fa, fb, fc, smem);
    else
      tile_gemm_shape<R, NT, 4, 1, KF>(M, N, K, fa, fb, fc, smem);
  } else if (N <= 32 && M > TY) {
    tile_gemm_shape<R, NT, 2, 2, KF>(M, N, K, fa, fb, fc, smem);
  } else {
    tile_gemm_shape<R, NT, 1, 4, KF>(M, N, K, fa, fb, fc, smem);
  }
}

}  // namespace gate
}  // namespace mpsvqe
