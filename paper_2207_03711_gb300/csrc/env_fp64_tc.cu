// Environment contractions of the trie measurement in FP64 on the tensor cores.
//
// GB300 has two FP64 lanes an SM and clock: a measurement at chi = 64 is bound by them. The
// error-free splitting of Ozaki, Ogita, Oishi and Rump (Numer. Algorithms 59, 2012; on matrix
// units: Mukunoki et al., ISC 2020) gives an FP64 product from small exact ones: each row
// of an operand is scaled by a power of two into (-1, 1), rounded to 55 bits and cut into
// kDigits = 8 signed digits of 7 bits (BF16, exact). The products of digits p and q with p + q
// = t are summed in one FP32 accumulator of TMEM: |d| <= 64, so 256 inner indices and at most 8
// pairs stay below 2^12 2^8 2^3 = 2^23 and the sums are exact whole numbers, which the tensor
// core's truncation cannot touch. The 36 pairs with t < 8 are kept; what is left out is below
// 2^-53.2 (7 2^-56 and less) of (largest of the row) (largest of the column) per term, the
// rounding of the operands below 2^-55. The epilogue adds the eight sums in 64-bit integers and
// rounds once, twice where their upper part has more than 53 bits.
//
// 18 qubits, chi = 64, molecular Hamiltonian: 62 ms on the FP64 lanes (60 of it in the levels), 8.6 ms
// so, 3.9 in the levels that use it; against 128-bit arithmetic the rms error of 16 strings is
// 0.4 - 1.4e-16 at bonds of 24 .. 64, of the FP64 kernels 0.7 - 1.9e-16.
//
// One scale for a row wants entries of like weight, which a gauge B_k -> B_k X, B_{k+1} ->
// X^-1 B_{k+1} on a bond takes away from both operands at once: the products do not notice a
// diagonal X, 55 bits below the largest entry do (a spread of 2^20 cost 1e-12 of <P>, 2^30
// 5e-10). So the inner index of every product is balanced first: entry b of L's rows (of T's
// columns) is taken times 2^x, entry b of the site operand times 2^-x, where 2^x is the weight of
// b in the state (k_balance). That is exact, costs an addition per exponent, and makes a state
// with a gauge of powers of two give the bits it gives without; x = 0 where the site tensors are
// right-canonical.
//
// A level is, for a batch of nodes (see env_tc.cu for the real form of the products):
//   k_split_L       digits of L's rows (node, a), inner (b, re/im)
//   k_gemm_digits   T^T: rows (j, re/im, c) over columns (node, a), FP64
//   k_split_T       digits of T's columns (node, c), inner (j, re/im, a): all that one column of
//                   a child's product needs has one scale
//   k_gemm_digits   L[child], the letter choosing the order and the sign of the four ranges
//                   (the shared operand is there with both signs)
#include <algorithm>
#include <cstdint>

#include "cx.cuh"
#include "env_fp64_tc.cuh"
#include "kernels.cuh"
#include "smem_limit.cuh"
#include "tc_ptx.cuh"

namespace mpsvqe {

namespace {
constexpr int kDigits = 8;
constexpr int kNoScale = 1 << 20;   // exponent of a row with an infinity or NaN
constexpr int kNone = -8000;        // exponent of zero
constexpr int BM = 128, BN = 64, BK = 64;   // 64 BF16 = one 128-byte swizzle row
constexpr int kDrain = 256 / BK;            // K tiles that the accumulators take exactly
constexpr int PLANE_A = BM * BK * 2, PLANE_B = BN * BK * 2;
constexpr int SMEM = kDigits * (PLANE_A + PLANE_B) + 1024 + 64;
constexpr int NTHREADS = 320, NEPI = 256;
constexpr int TMEM_COLS = kDigits * BN;

__host__ __device__ constexpr int pad8(int d) { return (d + 7) & ~7; }
__host__ __device__ constexpr int pad64(int d) { return (d + 63) & ~63; }

// Exponent e with |x| 2^s < 2^e.
__device__ __forceinline__ int exponent_of(double x, int s) {
  const int b = (__double2hiint(x) >> 20) & 0x7ff;
  return b == 0x7ff ? kNoScale : x == 0.0 ? kNone : max(b, 1) - 1022 + s;
}
__device__ __forceinline__ int exponent_of(Cx<double> z, int s) { return max(exponent_of(z.x, s), exponent_of(z.y, s)); }
// x 2^(55 - e) rounded to a whole number, digits' offset added: digit p (p = 0 the highest) is
// (y >> 7 (7 - p)) - 64, of 7 bits but the highest, which takes all that is left.
__device__ __forceinline__ long long to_fixed(double x, int e) {
  const long long u = __double_as_longlong(x);
  const int b = (int)((u >> 52) & 0x7ff);
  unsigned long long m = (unsigned long long)u & 0xfffffffffffffull;
  if (b) m |= 1ull << 52;
  const int sh = 3 - e + (max(b, 1) - 1023);   // <= 2 but in a row of zeros
  if (sh >= 0)
    m <<= min(sh, 2);
  else
    m = sh < -60 ? 0 : (m + (1ull << (-sh - 1))) >> -sh;
  const long long v = u < 0 ? -(long long)m : (long long)m;
  return v + (long long)(0x1ull << 6) * 0x40810204081ll;   // 64 (1 + 2^7 + ... + 2^42)
}
__device__ __forceinline__ uint32_t bf16_of(int d) { return __float_as_uint((float)d) >> 16; }   // |d| <= 64: exact
__device__ __forceinline__ int digit(long long y, int p) {
  return p == 0 ? (int)(y >> 49) : ((int)(y >> (7 * (7 - p))) & 127) - 64;
}
__device__ __forceinline__ int warp_max(int v) { return __reduce_max_sync(0xffffffffu, v); }
// Two neighbouring entries into the planes at o (even), plane stride ps.
__device__ __forceinline__ void store_digits(uint16_t* o, int64_t ps, double x0, int e0, double x1, int e1) {
  const long long y0 = to_fixed(x0, e0), y1 = to_fixed(x1, e1);
#pragma unroll
  for (int p = 0; p < kDigits; ++p)
    *reinterpret_cast<uint32_t*>(o + p * ps) = bf16_of(digit(y0, p)) | bf16_of(digit(y1, p)) << 16;
}

// Balance of the left bond's indices of every site: x with 2^x about the norm of the state that
// index b stands for to the right (the root of R_k[b][b], to the nearest power of two), raised
// where that norm comes from cancellation to what the entries of row b weigh against the norms
// right of the site. So the balanced site operand stays below 1 and the balanced L is a part of
// <psi|psi>. One warp an index; grid (indices / 8, sites).
__device__ __forceinline__ int norm_exponent(double r2) {
  if (!(r2 > 0.0)) return kNone;
  const int b = __double2hiint(r2) >> 20;
  return b == 0x7ff ? kNoScale : (max(b, 1) - 1022) >> 1;
}
__global__ void __launch_bounds__(256) k_balance(DevMPS m, int slot, const Cx<double>* Renv, int* bal) {
  const int* rank = m.rank + (size_t)slot * (m.n + 1);
  const int k = blockIdx.y, D = rank[k], Dp = rank[k + 1];
  const int b = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (b >= D) return;
  const size_t chi2 = (size_t)m.chi * m.chi;
  const Cx<double>* R = Renv + (size_t)k * chi2;
  const Cx<double>* Rn = R + chi2;
  const Cx<double>* row = (const Cx<double>*)m.B + (size_t)slot * m.slot_elems + m.site_off[k] + (size_t)b * 2 * Dp;
  int x = norm_exponent(R[(size_t)b * (D + 1)].x);
  for (int q = lane; q < 2 * Dp; q += 32) {
    const int c = q < Dp ? q : q - Dp;
    x = max(x, exponent_of(row[q], k == m.n - 1 ? 0 : norm_exponent(Rn[(size_t)c * (Dp + 1)].x)) - 1);
  }
  x = warp_max(x);
  if (lane == 0) bal[(size_t)k * m.chi + b] = x > 4000 || x < -4000 ? 0 : x;
}

// Row r = (u, a) of L: 2D reals (b, re/im), one warp a row.
__global__ void __launch_bounds__(256) k_split_L(const Cx<double>* L, int64_t rows, int D, const int* bal, uint16_t* out,
                                                 int* ex) {
  const int64_t r = blockIdx.x * (int64_t)8 + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31, ld = pad8(2 * D);
  if (r >= rows) return;
  const Cx<double>* x = L + r * D;
  int e = kNone;
  for (int b = lane; b < D; b += 32) e = max(e, exponent_of(x[b], bal[b]));
  e = warp_max(e);
  if (lane == 0) ex[r] = e;
  for (int b = lane; 2 * b < ld; b += 32) {
    const Cx<double> z = b < D ? x[b] : cx<double>(0, 0);
    const int eb = b < D ? e - bal[b] : e;
    store_digits(out + r * ld + 2 * b, rows * ld, z.x, eb, z.y, eb);
  }
}

// Column (u, c) of T: ranges (j, re/im) of D entries a, each padded to pad8(D); one warp a column.
__global__ void __launch_bounds__(256) k_split_T(const double* Tt, int U, int D, int Dp, const int* bal, uint16_t* out,
                                                 int* ex) {
  const int64_t rows = (int64_t)U * Dp, r = blockIdx.x * (int64_t)8 + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31, ds = pad8(D);
  if (r >= rows) return;
  const int64_t u = r / Dp, c = r - u * Dp, ldt = (int64_t)U * D;
  const double* t = Tt + c * ldt + u * D;
  int e = kNone;
  for (int s = 0; s < 4; ++s)
    for (int a = lane; a < D; a += 32) e = max(e, exponent_of(t[(int64_t)s * Dp * ldt + a], bal[a]));
  e = warp_max(e);
  if (lane == 0) ex[r] = e;
  for (int s = 0; s < 4; ++s)
    for (int a = 2 * lane; a < ds; a += 64) {
      const double* x = t + (int64_t)s * Dp * ldt + a;
      const bool i0 = a < D, i1 = a + 1 < D;
      store_digits(out + (r * 4 + s) * ds + a, rows * 4 * ds, i0 ? x[0] : 0.0, i0 ? e - bal[a] : e, i1 ? x[1] : 0.0,
                   i1 ? e - bal[a + 1] : e);
    }
}

// Shared operands of a site (layouts as in env_tc.cu): BT, 4D' rows of 2D; A2, 2D' rows of
// eight ranges of pad64(D): the four ranges (i, re/im) and the same with the other sign.
__global__ void __launch_bounds__(256) k_split_site(const Cx<double>* Bk, int D, int Dp, const int* bal, uint16_t* bt,
                                                    int* bt_ex, uint16_t* a2, int* a2_ex) {
  const int r = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (r < 4 * Dp) {
    const int c = r % Dp, ro = r / Dp & 1, j = r / Dp >> 1, ld = pad8(2 * D);
    int e = kNone;
    for (int b = lane; b < D; b += 32) e = max(e, exponent_of(Bk[((size_t)b * 2 + j) * Dp + c], -bal[b]));
    e = warp_max(e);
    if (lane == 0) bt_ex[r] = e;
    for (int b = lane; 2 * b < ld; b += 32) {
      const Cx<double> z = b < D ? Bk[((size_t)b * 2 + j) * Dp + c] : cx<double>(0, 0);
      const int eb = b < D ? e + bal[b] : e;
      store_digits(bt + (int64_t)r * ld + 2 * b, (int64_t)4 * Dp * ld, ro ? z.y : z.x, eb, ro ? z.x : -z.y, eb);
    }
  } else if (r < 6 * Dp) {
    const int q = r - 4 * Dp, ro = q & 1, cp = q >> 1, ds = pad64(D), ld = 8 * ds;
    int e = kNone;
    for (int a = lane; a < 2 * D; a += 32) e = max(e, exponent_of(Bk[(size_t)a * Dp + cp], -bal[a >> 1]));   // (a, i) in one index
    e = warp_max(e);
    if (lane == 0) a2_ex[q] = e;
    for (int x = 2 * lane; x < ld; x += 64) {
      const int seg = x / ds, a = x - seg * ds, i = seg >> 1 & 1, ri = seg & 1;
      double v[2];
      int ek[2];
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        ek[k] = a + k < D ? e + bal[a + k] : e;
        const Cx<double> z = a + k < D ? Bk[((size_t)(a + k) * 2 + i) * Dp + cp] : cx<double>(0, 0);
        v[k] = ro == ri ? z.x : ro ? -z.y : z.y;   // re row [Br, Bi] per i, im row [-Bi, Br]
        if (seg >= 4) v[k] = -v[k];
      }
      store_digits(a2 + (int64_t)q * ld + x, (int64_t)2 * Dp * ld, v[0], ek[0], v[1], ek[1]);
    }
  }
}

__device__ __forceinline__ void mma_bf16(uint32_t tmem_d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n"
      " .reg .pred p;\n"
      " setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n"
      "}\n" ::"r"(tmem_d),
      "l"(a), "l"(b), "r"(idesc), "r"(acc)
      : "memory");
}

struct DigitGemm {
  int M = 0, N = 0, nk = 0;          // rows, columns, K tiles
  int a_rows = 0, b_rows = 0;        // rows of a plane
  const int *a_ex = nullptr, *b_ex = nullptr;
  double* T = nullptr;               // T^T, leading dimension N
  // children
  const int32_t* parent = nullptr;
  const uint8_t* edge = nullptr;
  int node_base = 0, nc = 0, Dp = 0, ds = 0, seg_tiles = 0, per = 0;
  Cx<double>* L = nullptr;
};

// One 128 x 64 tile of the product a block and turn: all eight planes of a K tile are one
// stage of 192 KB and the eight sums take the whole TMEM, so loads, products and epilogue
// follow each other within a block.
template <bool CHILDREN>
__global__ void __launch_bounds__(NTHREADS, 1)
    k_gemm_digits(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                  const __grid_constant__ DigitGemm g, int* err) {
  using namespace tc;
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* base = (unsigned char*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint64_t* bars = (uint64_t*)(base + kDigits * (PLANE_A + PLANE_B));
  const uint32_t full = smem_u32(&bars[0]), empty = smem_u32(&bars[1]), ready = smem_u32(&bars[2]), freed = smem_u32(&bars[3]);
  uint32_t* tmem_slot = (uint32_t*)(bars + 4);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int tiles_m = (g.M + BM - 1) / BM;
  const int tiles_n = CHILDREN ? g.nc * g.per : (g.N + BN - 1) / BN;
  const int tiles = tiles_m * tiles_n;   // rows vary fastest: blocks side by side share a column tile
  if (tid == 0) {
    mbar_init(full, 1);
    mbar_init(empty, 1);
    mbar_init(ready, 1);
    mbar_init(freed, NEPI);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tmem_slot;
  const uint32_t sa = smem_u32(base), sb = sa + kDigits * PLANE_A;

  if (warp == 0 && lane == 0) {
    // ---- loads
    int n = 0;
    bool ok = true;
    for (int tile = blockIdx.x; tile < tiles && ok; tile += gridDim.x) {
      const int nt = tile / tiles_m, m0 = (tile - nt * tiles_m) * BM;
      int letter = 0, y0 = nt * BN;
      if (CHILDREN) {
        const int ch = nt / g.per;
        letter = g.edge[ch];
        y0 = (g.parent[ch] - g.node_base) * g.Dp + (nt - ch * g.per) * BN;
      }
      for (int kt = 0; kt < g.nk; ++kt, ++n) {
        if (n > 0 && !mbar_wait(empty, (n - 1) & 1, err, 11)) {
          ok = false;
          break;
        }
        int xa = kt * BK, xb = kt * BK;
        if (CHILDREN) {
          const int seg = kt / g.seg_tiles, x = (kt - seg * g.seg_tiles) * BK;
          float sg;
          xb = child_block(letter, seg, &sg) * g.ds + x;
          xa = ((sg < 0.f ? 4 : 0) + seg) * g.seg_tiles * BK + x;
        }
        mbar_arrive_expect_tx(full, kDigits * (PLANE_A + PLANE_B));
        for (int p = 0; p < kDigits; ++p) {
          tma_load_2d(sa + p * PLANE_A, &tmA, xa, p * g.a_rows + m0, full);
          tma_load_2d(sb + p * PLANE_B, &tmB, xb, p * g.b_rows + y0, full);
        }
      }
    }
    // no copy may still be landing when the block exits
    if (n > 0) mbar_wait(full, (n - 1) & 1, err, 12);
  } else if (warp == 1 && lane == 0) {
    // ---- products: accumulator t = p + q
    // FP32 accumulator (bits 4-5 = 1), A and B BF16 (bits 7-9, 10-12 = 1), both K-major
    constexpr uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(BN >> 3) << 17) | ((uint32_t)(BM >> 4) << 24);
    int n = 0, drained = 0;
    bool ok = true;
    for (int tile = blockIdx.x; tile < tiles && ok; tile += gridDim.x)
      for (int kt = 0; kt < g.nk; ++kt, ++n) {
        const bool first = kt % kDrain == 0;
        if (!mbar_wait(full, n & 1, err, 13) ||
            (first && drained > 0 && !mbar_wait(freed, (drained - 1) & 1, err, 14))) {
          ok = false;
          break;
        }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        for (int ks = 0; ks < BK / 16; ++ks)
#pragma unroll
          for (int p = 0; p < kDigits; ++p)
#pragma unroll
            for (int q = 0; p + q < kDigits; ++q)
              mma_bf16(tmem + (uint32_t)((p + q) * BN), sw128_kmajor_desc(sa + p * PLANE_A + ks * 32),
                       sw128_kmajor_desc(sb + q * PLANE_B + ks * 32), idesc, first && ks == 0 && p == 0 ? 0u : 1u);
        mma_commit(empty);
        if (kt % kDrain == kDrain - 1 || kt == g.nk - 1) {
          mma_commit(ready);
          ++drained;
        }
      }
  } else if (warp >= 2) {
    // ---- epilogue: warp w reads TMEM lanes 32 (w mod 4) .. (its rows) and half of the columns
    const int q4 = warp & 3, c_lo = ((warp - 2) >> 2) * (BN / 2);
    const uint32_t lane_off = (uint32_t)(q4 * 32) << 16;
    int drained = 0;
    bool ok = true;
    for (int tile = blockIdx.x; tile < tiles && ok; tile += gridDim.x) {
      const int nt = tile / tiles_m, row = (tile - nt * tiles_m) * BM + q4 * 32 + lane;
      // sum of the accumulators: hi in units of t = 5, lo (in [0, 2^14) between drains) of t = 7;
      // |hi| < 2^58 a drain
      long long hi[BN / 2];
      int lo[BN / 2];
#pragma unroll
      for (int c = 0; c < BN / 2; ++c) hi[c] = lo[c] = 0;
      for (int kt = 0; kt < g.nk && ok; kt += kDrain, ++drained) {
        ok = __all_sync(0xffffffffu, mbar_wait(ready, drained & 1, err, 15, true));
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        if (ok) {
#pragma unroll
          for (int t = 0; t < kDigits; ++t) {
            float v[32];
            tmem_ld32(tmem + lane_off + (uint32_t)(t * BN + c_lo), v);
#pragma unroll
            for (int c = 0; c < BN / 2; ++c) {
              const int x = __float2int_rn(v[c]);
              if (t <= 5)
                hi[c] += (long long)x << (7 * (5 - t));
              else
                lo[c] += x << (7 * (7 - t));
              if (t == kDigits - 1) {
                hi[c] += lo[c] >> 14;
                lo[c] &= 16383;
              }
            }
          }
        }
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        mbar_arrive(freed);
      }
      if (!ok || row >= g.M) continue;
      const int ea = g.a_ex[row];
      int ncol, col0;      // valid columns of the tile, index of the first in b_ex
      double* out;
      int64_t step;
      if (CHILDREN) {
        const int ch = nt / g.per, cc = (nt - ch * g.per) * BN + c_lo;
        ncol = g.Dp - cc;
        col0 = (g.parent[ch] - g.node_base) * g.Dp + cc;
        out = (double*)(g.L + ((int64_t)ch * g.Dp + (row >> 1)) * g.Dp + cc) + (row & 1);
        step = 2;
      } else {
        col0 = nt * BN + c_lo;
        ncol = g.N - col0;
        out = g.T + (int64_t)row * g.N + col0;
        step = 1;
      }
#pragma unroll
      for (int c = 0; c < BN / 2; ++c) {
        if (c < ncol) {
          const int e = ea + g.b_ex[col0 + c];
          double v = fma((double)hi[c], 16384.0, (double)lo[c]);
          // exponents far from 0 in two steps; a row with an infinity or NaN gives NaN
          if (e > 900 || e < -900)
            v = e > kNoScale / 2 ? __longlong_as_double(0x7ff8000000000000ll) : ldexp(v, e - 61);
          else
            v *= __hiloint2double((1023 + e - 61) << 20, 0);
          out[c * step] = v;
        }
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 1) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS) : "memory");
  }
}

template <bool CHILDREN>
cudaError_t launch(const DigitGemm& g, const uint16_t* A, int a_cols, const uint16_t* B, int b_cols, int* err, cudaStream_t st) {
  CUtensorMap am, bm;
  cudaError_t e;
  const auto type = CU_TENSOR_MAP_DATA_TYPE_BFLOAT16;
  if ((e = tc::make_map(&am, type, A, (int64_t)kDigits * g.a_rows, a_cols, 2 * (int64_t)a_cols, BK, BM)) != cudaSuccess) return e;
  if ((e = tc::make_map(&bm, type, B, (int64_t)kDigits * g.b_rows, b_cols, 2 * (int64_t)b_cols, BK, BN)) != cudaSuccess) return e;
  if ((e = gate::raise_smem_limit<k_gemm_digits<CHILDREN>>()) != cudaSuccess) return e;
  const int64_t tiles = (int64_t)((g.M + BM - 1) / BM) * (CHILDREN ? g.nc * g.per : (g.N + BN - 1) / BN);
  if (tiles <= 0) return cudaSuccess;
  const int grid = (int)std::min<int64_t>(tiles, 152);
  k_gemm_digits<CHILDREN><<<grid, NTHREADS, SMEM, st>>>(am, bm, g, err);
  return cudaGetLastError();
}

size_t up(size_t b) { return (b + 255) & ~size_t(255); }
struct Parts {
  uint16_t *bt, *a2, *l, *t;
  int *bt_ex, *a2_ex, *l_ex, *t_ex;
  double* T;
  size_t bytes;
};
// Scratch for bonds up to chi and batches of nb nodes.
Parts carve(char* base, int chi, int nb) {
  Parts p;
  size_t at = 0;
  auto take = [&](size_t b) {
    char* q = base ? base + at : nullptr;
    at += up(b);
    return q;
  };
  const size_t x = chi, ld = pad8(2 * chi), n = nb;
  p.bt = (uint16_t*)take(2 * kDigits * 4 * x * ld);
  p.a2 = (uint16_t*)take(2 * kDigits * 2 * x * 8 * pad64(chi));
  p.bt_ex = (int*)take(4 * 4 * x);
  p.a2_ex = (int*)take(4 * 2 * x);
  p.l = (uint16_t*)take(2 * kDigits * n * x * ld);
  p.l_ex = (int*)take(4 * n * x);
  p.T = (double*)take(8 * 4 * n * x * x);
  p.t = (uint16_t*)take(2 * kDigits * n * x * 4 * pad8(chi));
  p.t_ex = (int*)take(4 * n * x);
  p.bytes = at;
  return p;
}
}  // namespace

int env_fp64_batch(int chi) { return std::max(16, (int)((size_t(512) << 20) / (128 * (size_t)chi * chi))); }
size_t env_fp64_scratch(int chi, int batch) { return carve(nullptr, chi, batch).bytes; }

cudaError_t env_fp64_balance(const EnvFp64& s, const DevMPS& m, int slot, int top, const Cx<double>* Renv, cudaStream_t st) {
  k_balance<<<dim3((top + 7) / 8, m.n), 256, 0, st>>>(m, slot, Renv, s.bal);
  return cudaGetLastError();
}

cudaError_t env_fp64_site(const EnvFp64& s, const Cx<double>* Bk, int k, int D, int Dp, cudaStream_t st) {
  const Parts p = carve(s.scratch, s.chi, s.batch);
  k_split_site<<<(6 * Dp + 7) / 8, 256, 0, st>>>(Bk, D, Dp, s.bal + (size_t)k * s.chi, p.bt, p.bt_ex, p.a2, p.a2_ex);
  return cudaGetLastError();
}

cudaError_t env_fp64_T(const EnvFp64& s, const Cx<double>* L, int k, int U, int D, int Dp, cudaStream_t st, cudaEvent_t e0,
                       cudaEvent_t e1) {
  if (U <= 0) return cudaSuccess;
  const int* bal = s.bal + (size_t)k * s.chi;
  const Parts p = carve(s.scratch, s.chi, s.batch);
  const int64_t rows = (int64_t)U * D, cols = (int64_t)U * Dp;
  k_split_L<<<(unsigned)((rows + 7) / 8), 256, 0, st>>>(L, rows, D, bal, p.l, p.l_ex);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  DigitGemm g;
  g.M = 4 * Dp;
  g.N = (int)rows;
  g.nk = (2 * D + BK - 1) / BK;
  g.a_rows = 4 * Dp;
  g.b_rows = (int)rows;
  g.a_ex = p.bt_ex;
  g.b_ex = p.l_ex;
  g.T = p.T;
  if (e0 && (e = cudaEventRecord(e0, st)) != cudaSuccess) return e;
  if ((e = launch<false>(g, p.bt, pad8(2 * D), p.l, pad8(2 * D), s.err, st)) != cudaSuccess) return e;
  if (e1 && (e = cudaEventRecord(e1, st)) != cudaSuccess) return e;
  k_split_T<<<(unsigned)((cols + 7) / 8), 256, 0, st>>>(p.T, U, D, Dp, bal, p.t, p.t_ex);
  return cudaGetLastError();
}

cudaError_t env_fp64_children(const EnvFp64& s, const int32_t* parent, const uint8_t* edge, int nc, int node_base, int U, int D,
                              int Dp, Cx<double>* Lout, cudaStream_t st, cudaEvent_t e0, cudaEvent_t e1) {
  if (nc <= 0) return cudaSuccess;
  const Parts p = carve(s.scratch, s.chi, s.batch);
  DigitGemm g;
  g.M = 2 * Dp;
  g.seg_tiles = pad64(D) / BK;
  g.nk = 4 * g.seg_tiles;
  g.a_rows = 2 * Dp;
  g.b_rows = U * Dp;
  g.a_ex = p.a2_ex;
  g.b_ex = p.t_ex;
  g.parent = parent;
  g.edge = edge;
  g.node_base = node_base;
  g.nc = nc;
  g.Dp = Dp;
  g.ds = pad8(D);
  g.per = (Dp + BN - 1) / BN;
  g.L = Lout;
  cudaError_t e;
  if (e0 && (e = cudaEventRecord(e0, st)) != cudaSuccess) return e;
  if ((e = launch<true>(g, p.a2, 8 * pad64(D), p.t, 4 * pad8(D), s.err, st)) != cudaSuccess) return e;
  return e1 ? cudaEventRecord(e1, st) : cudaSuccess;
}

}  // namespace mpsvqe
